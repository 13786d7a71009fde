"""A trace of rain in dry air in the float32 forms: rho_w = rho_m + rho_r is then as small as the rain
itself, down to float32's subnormal numbers, and the fall speed depends on their ratio alone."""
import numpy as np
import pytest

from paper_2305_13847_gb300 import dgmoist as dm
from tests.gpu_helpers import flux_scale, library_context, oracle_problem, perturbed_state, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", [dm.DG_FP32_BULK, dm.DG_FP32_PERT])
@pytest.mark.parametrize("rain", [1e-38, 6e-39, 2e-39, 1e-40, 1e-44])
def test_trace_of_rain_in_dry_air(precision, rain):
    """The tendencies of the fields that are not water are those with 1e-30 kg/m^3 of rain, whose fall
    speed is the same (rho_r / rho_w = 1), to 2e-6 of the flux scale, the bar of the float32 right-hand
    sides; those of the water itself, of the rain's own size, are finite."""
    prob, _ = oracle_problem(2, (5, 4), (8e3, 6e3), 3, (True, False), True, qt0=0.0)
    assert np.all(prob.base_node["rho_m"] == 0.0)
    U = perturbed_state(prob, seed=350)
    U[prob.i_rm] = 0.0
    R = []
    ctx = library_context(prob, precision)
    try:
        for r in (1e-30, rain):
            U[prob.i_rr] = r
            out = torch.empty(U.shape, dtype=torch.float32, device="cuda")
            dm.dg_rhs(ctx, to_device(U, torch.float32), out)
            R.append(out.cpu().numpy().astype(np.float64))
    finally:
        dm.dg_free(ctx)
    assert np.all(np.isfinite(R[1]))
    dry = [f for f in range(prob.nf) if f not in (prob.i_rm, prob.i_rr)]
    assert np.all(np.abs(R[1] - R[0])[dry].max(axis=(1, 2)) <= 2e-6 * flux_scale(prob, U)[dry])
