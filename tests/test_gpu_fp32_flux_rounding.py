"""The rounding of the float32 Lax-Friedrichs flux (csrc/dg_device.cuh, lf_flux)."""
import numpy as np
import pytest

from oracle import dg
from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import library_context, oracle_problem, perturbed_state, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rhs_errors(precision):
    """Relative L2 error of the mass and energy tendencies of a fixed float32 state: 4096 elements high,
    since the rounding of the base state's totals, the largest part, is one sample per level."""
    prob, _ = oracle_problem(2, (2, 4096), (2e3, 10e3), 3, (True, False), True)
    U = perturbed_state(prob, seed=360).astype(np.float32).astype(np.float64)
    ctx = library_context(prob, precision)
    try:
        out = torch.empty(U.shape, dtype=torch.float32, device="cuda")
        dm.dg_rhs(ctx, to_device(U, torch.float32), out)
        R = out.cpu().numpy().astype(np.float64)
    finally:
        dm.dg_free(ctx)
    Ro = dg.rhs(prob, U)
    return [float(np.linalg.norm(R[f] - Ro[f]) / np.linalg.norm(Ro[f])) for f in (prob.i_rd, prob.i_rm, prob.i_E)]


@pytest.mark.parametrize("precision", [dm.DG_FP32_BULK, dm.DG_FP32_PERT])
def test_flux_rounds_no_more_than_the_two_fluxes(precision):
    """The flux written on the jumps is no further from the exact tendencies of rho_d', rho_m' and E' than
    the average of the two sides' fluxes was on this state (4.726e-6, 4.807e-6, 6.041e-6), up to the 1 % by
    which an error over 4097 levels of faces scatters."""
    assert np.all(np.array(rhs_errors(precision)) <= 1.01 * np.array([4.726e-6, 4.807e-6, 6.041e-6]))
