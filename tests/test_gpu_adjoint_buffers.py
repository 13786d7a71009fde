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


def test_cloud_functional_refuses_its_own_state():
    """dJ/dU over U itself is refused, and the state is left as it was."""
    prob = _problem()
    U = to_device(perturbed_state(prob, seed=41), torch.float64)
    V = U.clone()
    ctx = library_context(prob)
    try:
        with pytest.raises(dm.DGError):
            dm.dg_cloud_functional(ctx, U, U)
        assert np.array_equal(V.cpu().numpy(), U.cpu().numpy())
    finally:
        dm.dg_free(ctx)


def _scratch(prob):
    """Bytes of dg_rhs_adjoint's scratch: six states, the traces and n_f + 3 values per node."""
    mesh = prob.mesh
    nodes, ntr = mesh.Ne * (mesh.k + 1) ** mesh.dim, prob.nf + 3
    trace = 2 * mesh.dim * mesh.Ne * (mesh.k + 1) ** (mesh.dim - 1) * ntr
    return 8 * (6 * prob.nf * nodes + trace + ntr * nodes)


@pytest.mark.parametrize("dim,n,order", [(2, (7, 5), 3), (3, (3, 2, 3), 4)])
def test_adjoint_step_with_and_without_kept_states(dim, n, order):
    """Only dg_adjoint_step holds the intermediate states' split and traces, gives them back when told
    to, and without them returns the same adjoint: within 1e-12 of each field's norm, twelve times the
    8e-14 that either lies off the adjoint in exact arithmetic (the split's rounding is all that differs)."""
    prob = _problem(dim, n, order)
    U = to_device(perturbed_state(prob, seed=43), torch.float64)
    g = torch.Generator().manual_seed(7)
    lam = torch.randn(U.shape, generator=g, dtype=torch.float64).cuda()
    ctx = library_context(prob)
    try:
        held = dm.dg_get_info(ctx).device_bytes
        out = [torch.empty_like(U) for _ in range(4)]
        dm.dg_rhs_adjoint(ctx, U, lam, out[3])
        assert dm.dg_get_info(ctx).device_bytes - held == _scratch(prob)
        held += _scratch(prob)
        dm.dg_set_adjoint_memory(ctx, 0)
        dm.dg_adjoint_step(ctx, 0.02, U, lam, out[0])
        assert dm.dg_get_info(ctx).device_bytes == held
        dm.dg_set_adjoint_memory(ctx, 1)
        dm.dg_adjoint_step(ctx, 0.02, U, lam, out[1])
        assert dm.dg_get_info(ctx).device_bytes > held
        dm.dg_set_adjoint_memory(ctx, 0)
        assert dm.dg_get_info(ctx).device_bytes == held
        dm.dg_adjoint_step(ctx, 0.02, U, lam, out[2])
        a, b, c = (o.cpu().numpy().reshape(prob.nf, -1) for o in out[:3])
    finally:
        dm.dg_free(ctx)
    assert np.array_equal(a, c)
    assert np.all(np.linalg.norm(a - b, axis=1) <= 1e-12 * np.linalg.norm(a, axis=1))


@pytest.mark.parametrize("keep", [0, 1])
def test_adjoint_step_counts_do_not_depend_on_its_memory(keep):
    """One overheated node (finite, above 1000 K) in each of the four stage states of a vanishing step:
    counted twice per state, for the stage's split and the reversal's, whether the second is made or not."""
    prob = _problem()
    U = perturbed_state(prob, seed=45)
    U[prob.i_E, 4, 5] = 2e6
    ctx = library_context(prob)
    try:
        dm.dg_set_adjoint_memory(ctx, keep)
        Ud = to_device(U, torch.float64)
        out = torch.empty_like(Ud)
        dm.dg_adjoint_step(ctx, 1e-12, Ud, torch.ones_like(Ud), out)
        st, counts = dm.dg_check_status(ctx)
        assert st == dm.DG_ENONPHYS and list(counts) == [0, 8]
    finally:
        dm.dg_free(ctx)


def test_adjoint_step_captured_before_its_first_use():
    """A first reversed step inside a stream capture, after dg_rhs_adjoint has made the common scratch:
    it allocates nothing, and a replay gives the eager step without kept states, bit by bit."""
    prob = _problem()
    U = to_device(perturbed_state(prob, seed=47), torch.float64)
    g = torch.Generator().manual_seed(9)
    lam = torch.randn(U.shape, generator=g, dtype=torch.float64).cuda()
    a, b, r = (torch.empty_like(U) for _ in range(3))
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = library_context(prob, stream=stream)
    try:
        dm.dg_rhs_adjoint(ctx, U, lam, r)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            graph.capture_begin()
            dm.dg_adjoint_step(ctx, 0.02, U, lam, a)
            graph.capture_end()
            graph.replay()
        stream.synchronize()
        dm.dg_set_adjoint_memory(ctx, 0)
        dm.dg_adjoint_step(ctx, 0.02, U, lam, b)
        stream.synchronize()
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
    finally:
        dm.dg_free(ctx)
