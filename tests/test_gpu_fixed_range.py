"""A value far above anything physical, finite and below the top of the fixed-point range, in a float64
tile (csrc/dg_stage64.cuh): as with float64 sums, it reaches only its own lines and the neighbours
across them, not the other elements of its tile nor the other nodes of its element."""
import numpy as np
import pytest

from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import flux_scale, library_context, oracle_problem, perturbed_state, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# dimension, mesh, order, element, its middle node
MESHES = [(2, (7, 5), 2, 3, 4), (2, (6, 4), 4, 1, 12), (3, (3, 2, 3), 2, 4, 13)]


@pytest.mark.parametrize("dim,n,order,elem,node", MESHES)
@pytest.mark.parametrize("field,value", [("E", v) for v in (1e7, 1e12, 1e20, 1e60, 1e150, 1e250)] +
                         [("rho_d", 1e5), ("rho_d", 1e20), ("m", 1e9), ("m", 1e20)])
@pytest.mark.parametrize("rain,gamma", [(True, 0.0), (False, 0.06)])
def test_blown_up_node_stays_local(dim, n, order, elem, node, field, value, rain, gamma):
    """The right-hand side off the node's lines agrees with that of the unspoilt state to 1e-12 of its
    flux scale, the bar of every float64 right-hand side."""
    if gamma and field == "m":
        pytest.skip("the diffusion coefficient of the element follows its velocity: not local by itself")
    L = (7e3, 3e3) if dim == 2 else (3e3, 2.5e3, 3e3)
    prob, _ = oracle_problem(dim, n, L, order, (True,) * (dim - 1) + (False,), rain)
    U = perturbed_state(prob, seed=330)
    V = U.copy()
    V[{"E": prob.i_E, "rho_d": prob.i_rd, "m": prob.i_m[0]}[field], elem, node] = value
    ctx = library_context(prob)
    try:
        if gamma:
            dm.dg_set_stabilisation(ctx, gamma, 10.0)
        R = []
        for X in (U, V):
            out = torch.empty(U.shape, dtype=torch.float64, device="cuda")
            dm.dg_rhs(ctx, to_device(X, torch.float64), out)
            R.append(out.cpu().numpy())
        per_tile = dm.dg_get_info(ctx).elems_per_block
    finally:
        dm.dg_free(ctx)
    near = {elem} | {int(prob.mesh.neighbour(np.array([elem]), j, s)[0]) for j in range(dim) for s in (-1, 1)}
    if gamma and field == "rho_d":
        # alpha_K and its vertex means follow the element's velocity: every element at its corners
        idx = np.array(np.unravel_index(np.arange(prob.mesh.Ne), n, order="F"))
        gap = np.abs(idx - idx[:, [elem]])
        gap = np.minimum(gap, np.array(n)[:, None] - gap)
        near |= set(np.nonzero((gap <= 1).all(axis=0))[0])
    far = np.array([e not in near for e in range(prob.mesh.Ne)])
    tile = np.arange(prob.mesh.Ne) // per_tile == elem // per_tile
    assert per_tile == 1 or (far & tile).any() or (gamma and field == "rho_d")
    bound = 1e-12 * flux_scale(prob, U)
    if far.any():
        assert np.all(np.abs(R[1] - R[0])[:, far].max(axis=(1, 2)) <= bound)
    if not (gamma and field == "rho_d"):
        p1 = order + 1
        corner = [int(sum(c * order * p1 ** j for j, c in enumerate(b))) for b in np.ndindex(*(2,) * dim)]
        assert np.all(np.abs(R[1] - R[0])[:, elem][:, corner].max(axis=1) <= bound)
