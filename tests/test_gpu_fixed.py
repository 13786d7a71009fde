"""Float64 contractions in fixed point (csrc/dg_fixed.cuh) where they can go wrong: every order and
dimension on ragged tiles, fields that vanish or vary over many decades, and values outside the
fixed-point range, against the oracle."""
import numpy as np
import pytest

from oracle import dg
from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import flux_scale, library_context, oracle_problem, perturbed_state, to_device

pytestmark = pytest.mark.gpu


def _rhs(prob, U):
    import torch
    ctx = library_context(prob)
    try:
        R = torch.empty(U.shape, dtype=torch.float64, device="cuda")
        dm.dg_rhs(ctx, to_device(U, torch.float64), R)
        return R.cpu().numpy()
    finally:
        dm.dg_free(ctx)


def _problem(dim, order, rain, periodic=True):
    n = (7, 3) if dim == 2 else (3, 2, 3)
    L = (7e3, 3e3) if dim == 2 else (3e3, 2.5e3, 3e3)
    prob, _ = oracle_problem(dim, n, L, order, (periodic,) * (dim - 1) + (False,), rain)
    return prob


@pytest.mark.parametrize("dim,order", [(d, k) for d in (2, 3) for k in (1, 2, 3, 4, 5)])
@pytest.mark.parametrize("rain", [False, True])
def test_rhs_every_order(dim, order, rain):
    """Within 1e-12 of the flux scale, the bar of every float64 right-hand side."""
    prob = _problem(dim, order, rain, periodic=not rain)
    U = perturbed_state(prob, seed=300 + order)
    R, Ro = _rhs(prob, U), dg.rhs(prob, U)
    err = np.abs(R - Ro).reshape(prob.nf, -1).max(axis=1)
    assert np.all(err <= 1e-12 * flux_scale(prob, U)), err


def test_rain_edge_keeps_relative_accuracy():
    """Rain that decays over 60 decades within a tile and vanishes beyond: its tendency has to carry the
    sign and size of the small values (v_r ~ rho_r^(1/8)), so it is compared node by node with the
    magnitude of its own terms: 1e-12 of (k+1)^2 2/h times the largest flux along the node's lines."""
    prob = _problem(2, 3, True)
    U = perturbed_state(prob, seed=310)
    x = prob.mesh.node_coords()[0]
    U[prob.i_rr] = np.where(x < 5e3, 1e-4 * 10.0 ** (-60.0 * x / 5e3), 0.0)
    R, Ro = _rhs(prob, U), dg.rhs(prob, U)
    wet = U[prob.i_rr].reshape(prob.mesh.Ne, -1).max(axis=1)
    nb = np.stack([wet] + [wet[np.maximum(prob.mesh.neighbour(np.arange(prob.mesh.Ne), j, s), 0)]
                           for j in range(2) for s in (-1, 1)]).max(axis=0)
    # sources turn cloud into rain everywhere; the bound adds their size (0.001 rho_c, 1.72 rho_c rho_r^(7/8))
    scale = (prob.mesh.k + 1) ** 2 * max(2.0 / h for h in prob.mesh.h) * 400.0 * nb[:, None] + 1e-5
    assert np.all(np.abs(R[prob.i_rr] - Ro[prob.i_rr]) <= 1e-12 * scale)


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e300])
def test_values_outside_the_range_stay_local(bad):
    """One node's energy out of the fixed-point range: the right-hand side is not finite only where the
    oracle's is not (the node's lines and the neighbours across them), and unchanged elsewhere."""
    prob = _problem(3, 2, False)
    U = perturbed_state(prob, seed=320)
    good = _rhs(prob, U)
    U[prob.i_E, 4, 13] = bad
    R = _rhs(prob, U)
    reach = np.zeros(U.shape[1:], dtype=bool)
    reach[4] = True
    for j in range(3):
        for s in (-1, 1):
            nb = int(prob.mesh.neighbour(np.array([4]), j, s)[0])
            if nb >= 0:
                reach[nb] = True
    far = ~reach
    scale = flux_scale(prob, np.where(np.isfinite(U) & (np.abs(U) < 1e200), U, 0.0))
    assert np.all(np.isfinite(R[:, far]))
    assert np.all(np.abs(R - good)[:, far].max(axis=1) <= 1e-12 * scale)
    # inside the element only the three lines through the node (middle of 3^3) are touched for a node
    # that spoils its flux alone; the corners of element 4 lie on none of them nor on its faces' points
    corner = [0, 2, 6, 8, 18, 20, 24, 26]
    assert np.all(np.isfinite(R[:, 4][:, corner]))
