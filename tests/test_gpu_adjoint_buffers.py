"""What the adjoint entry points do to the caller's buffers and the context's memory."""
import numpy as np
import pytest

from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import library_context, oracle_problem, perturbed_state, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _problem(dim=2, n=(7, 5), order=3):
    L = (8e3,) * (dim - 1) + (6e3,)
    return oracle_problem(dim, n, L, order, (True,) * (dim - 1) + (False,), True)[0]


@pytest.mark.parametrize("dim,n,order", [(2, (7, 5), 3), (3, (3, 2, 3), 2)])
def test_cloud_functional_in_place(dim, n, order):
    """dJ/dU written over U itself: the same bits as into a buffer of its own."""
    prob = _problem(dim, n, order)
    U = to_device(perturbed_state(prob, seed=41), torch.float64)
    ctx = library_context(prob)
    try:
        g, V = torch.empty_like(U), U.clone()
        J = dm.dg_cloud_functional(ctx, U, g)
        assert dm.dg_cloud_functional(ctx, V, V) == J
        assert np.array_equal(V.cpu().numpy(), g.cpu().numpy())
    finally:
        dm.dg_free(ctx)
