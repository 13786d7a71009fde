"""Rain over many decades inside one float64 tile (rain_sum, csrc/dg_stage64.cuh): v_r ~ rho_r^(1/8)
makes the sign and the size of the smallest rain matter, so its tendency has to be right against the
terms of its own node, whatever the rest of the tile holds.  The bound has no floor: it is also applied
(on the CPU) to the oracle's tendency with the error of a scale shared by the tile planted in it."""
import numpy as np
import pytest

from oracle import dg, thermo
from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import library_context, oracle_problem, perturbed_state, to_device

DECADES = 60.0


def _state(dim, order):
    """Unsaturated moist air with waves and rain that falls off by DECADES along x, none beyond."""
    n, L = ((7, 3), (7e3, 3e3)) if dim == 2 else ((5, 2, 2), (5e3, 2e3, 3e3))
    prob, _ = oracle_problem(dim, n, L, order, (True,) * (dim - 1) + (False,), True, qt0=0.002)
    U = perturbed_state(prob, seed=370)
    smooth = U[prob.i_E] * 1e-4
    U[prob.i_rd] = U[prob.i_rm] = 0.0
    U[prob.i_E] = smooth
    x = prob.mesh.node_coords()[0]
    edge = 0.8 * L[0]
    U[prob.i_rr] = np.where(x < edge, 1e-4 * 10.0 ** (-DECADES * x / edge), 0.0)
    return prob, U


def _bound(prob, U):
    """1e-12 of each node's own terms: the derivative factor (k+1)^2 2/h times 400 m/s (flow, fall and
    dissipation) times the largest rain on the node's lines and on the neighbours' lines across the faces
    that they end on, and the source terms with rho_vs in the place of the evaporation deficit rho_vs -
    rho_v, a difference that is itself rounded (no node is saturated, so there is no cloud)."""
    mesh = prob.mesh
    el = np.arange(mesh.Ne)
    T, rv, _, _ = dg.nodal_derived(prob, U, el)
    rm = prob.base_node["rho_m"][mesh.node_level_index()] + U[prob.i_rm]
    assert np.all(rv == rm)
    s_ev, _, _ = thermo.sources(T, rv, rm - rv, U[prob.i_rr])
    rvs = thermo.saturation_vapour_density(T)
    terms = np.abs(s_ev) * rvs / (rvs - rv)
    p1 = mesh.k + 1
    rr = np.abs(U[prob.i_rr]).reshape((mesh.Ne,) + (p1,) * mesh.dim)      # nodes (.., y, x)
    for j in range(mesh.dim):
        line = rr.max(axis=mesh.dim - j, keepdims=True)
        own = line
        for s in (-1, 1):
            nb = mesh.neighbour(el, j, s)
            own = np.maximum(own, np.where((nb >= 0).reshape((-1,) + (1,) * mesh.dim), line[np.maximum(nb, 0)], 0.0))
        terms = terms + p1 ** 2 * 2.0 / mesh.h[j] * 400.0 * np.broadcast_to(own, rr.shape).reshape(mesh.Ne, -1)
    return 1e-12 * terms


CASES = [(2, 3), (2, 5), (3, 2)]


@pytest.mark.parametrize("dim,order", CASES)
def test_bound_rejects_a_shared_scale(dim, order):
    """A sum truncated at 2^-57 of the whole state's largest term (one scale for a tile) exceeds the
    bound over much of the range; the oracle in another order of summation would not."""
    prob, U = _state(dim, order)
    bound = _bound(prob, U)
    p1 = order + 1
    unit = 2.0 ** -57 * p1 ** 2 * max(2.0 / h for h in prob.mesh.h) * np.abs(U[prob.i_rr]).max()
    wet = U[prob.i_rr] > 0.0
    assert np.mean(unit > bound[wet]) > 0.4
    assert bound[wet].min() < 1e-40


@pytest.mark.gpu
@pytest.mark.parametrize("dim,order", CASES)
def test_rain_tendency_against_its_own_terms(dim, order):
    torch = pytest.importorskip("torch")
    prob, U = _state(dim, order)
    ctx = library_context(prob)
    try:
        out = torch.empty(U.shape, dtype=torch.float64, device="cuda")
        dm.dg_rhs(ctx, to_device(U, torch.float64), out)
        R = out.cpu().numpy()
    finally:
        dm.dg_free(ctx)
    err = np.abs(R - dg.rhs(prob, U))[prob.i_rr]
    assert np.all(err <= _bound(prob, U)), np.max(err / np.maximum(_bound(prob, U), 1e-300))


@pytest.mark.gpu
def test_rain_shaft_edge_after_two_steps():
    """Rain that ends inside a tile: the rain field after two steps to 1e-12 of its norm (a scale shared
    by the tile left 2e-9)."""
    torch = pytest.importorskip("torch")
    prob, _ = oracle_problem(2, (6, 4), (6e3, 4e3), 4, (True, False), True)
    U = perturbed_state(prob, seed=380)
    x, z = prob.mesh.node_coords()[:2]
    r = np.minimum(np.sqrt(((x - 3e3) / 1.6e3) ** 2 + ((z - 2e3) / 1.2e3) ** 2), 1.0)
    U[prob.i_rr] = 1e-4 * np.cos(0.5 * np.pi * r) ** 2 * (r < 1.0)
    dt = 0.05 * min(prob.mesh.h) / 380.0
    ctx = library_context(prob)
    try:
        dm.dg_set_state(ctx, to_device(U, torch.float64), dm.DG_DEVICE)
        dm.dg_step(ctx, dt, 2)
        V = torch.empty(U.shape, dtype=torch.float64, device="cuda")
        dm.dg_get_state(ctx, V, dm.DG_DEVICE)
        V = V.cpu().numpy()
    finally:
        dm.dg_free(ctx)
    W = U
    for _ in range(2):
        W = dg.ssprk43_step(lambda X: dg.rhs(prob, X), W, dt)
    assert np.linalg.norm((V - W)[prob.i_rr]) <= 1e-12 * np.linalg.norm(W[prob.i_rr])
