"""Meshes on either side of the line where DG_FACES_AUTO takes the faces inline: the same bits as the
face pass for steps, right-hand sides and the fall-out, in every precision form."""
import numpy as np
import pytest

from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import library_context, oracle_problem, perturbed_state, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dim,n,order", [
    (dm.DG_FP64, 2, (25, 32), 3), (dm.DG_FP64, 2, (27, 30), 3), (dm.DG_FP64, 2, (3, 2), 5),
    (dm.DG_FP64_FFC, 2, (5, 4), 2), (dm.DG_FP64, 3, (2, 2, 2), 1),
    (dm.DG_FP32_BULK, 3, (8, 8, 9), 4), (dm.DG_FP32_BULK, 3, (8, 8, 10), 4),
    (dm.DG_FP32_PERT, 2, (38, 32), 3), (dm.DG_FP32_PERT, 2, (1, 1), 1)])
def test_auto_equals_face_pass(precision, dim, n, order):
    import torch
    real = torch.float32 if precision in (dm.DG_FP32_BULK, dm.DG_FP32_PERT) else torch.float64
    prob, _ = oracle_problem(dim, n, (8e3,) * (dim - 1) + (6e3,), order, (True,) * (dim - 1) + (False,), True)
    U = to_device(perturbed_state(prob, seed=400 + order), real)
    got = []
    for faces in (dm.DG_FACES_AUTO, dm.DG_FACES_PASS):
        ctx = library_context(prob, precision, faces=faces)
        try:
            R, V = torch.empty_like(U), torch.empty_like(U)
            dm.dg_rhs(ctx, U, R)
            dm.dg_set_state(ctx, U, dm.DG_DEVICE)
            dm.dg_step(ctx, 0.02, 2)
            dm.dg_get_state(ctx, V, dm.DG_DEVICE)
            H = np.empty(tuple(U.shape), dtype=np.float32 if real == torch.float32 else np.float64)
            dm.dg_step_to_host(ctx, 0.02, 1, H)
            got.append((R.cpu().numpy(), V.cpu().numpy(), H, dm.dg_reduce(ctx)[8]))
        finally:
            dm.dg_free(ctx)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
