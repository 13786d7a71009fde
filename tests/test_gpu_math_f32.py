"""The float32 kernels' elementary functions and the fixed-point words of the float64 contractions
(csrc/dg_math.cuh, csrc/dg_fixed.cuh) through dg_selftest_math.

Bars, in units of the last place of float32 (the exact value is the float64 function of the same float32
argument, rounded 2^-29 below one such unit):
  * frcp: the Newton step from a 1-ulp estimate leaves its square, 2^-46, and the last rounding: 0.51;
  * rsqrt_nr: half an ulp of the last fma and half the rounding of x y, 2^-25: 1.05;
  * log1p_small, |x| <= 1/16: x (1 + x p) with |x p| < 1/30 carrying two roundings: 0.57, the library's
    (2 allowed) beyond; expm1_small, |x| <= 0.35, |x p| < 0.21: 0.85, the library's beyond;
  * fixed point: exact while the group's exponent is at most 4 above the value's (57 bits hold its 53),
    then truncated towards zero below 2^-57 of the group's scale."""
import numpy as np
import pytest

from paper_2305_13847_gb300 import dgmoist as dm
from paper_2305_13847_gb300 import inputs
from tests.gpu_helpers import library_context, oracle_problem

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N = 200000


def _run(fn, x):
    prob, _ = oracle_problem(2, (2, 2), (2e3, 2e3), 1, (True, False), False)
    ctx = library_context(prob)
    try:
        xd = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        out = torch.empty(4 * xd.numel(), dtype=torch.float64, device="cuda")
        dm.dg_selftest_math(ctx, fn, xd, out)
        o = out.cpu().numpy().reshape(4, -1)
        return o[0], o[1]
    finally:
        dm.dg_free(ctx)


def _signed_log(seed, lo, hi):
    u = inputs.uniform(seed, np.arange(2 * N))
    return np.where(u[N:] < 0.5, -1.0, 1.0) * np.exp2(lo + (hi - lo) * u[:N])


@pytest.mark.parametrize("fn,lo,hi,bar", [
    ("recip_f32", -126.0, 125.99, 0.51), ("rsqrt_f32", -126.0, 127.99, 1.05),
    ("log1p_f32", -60.0, -4.0, 0.57), ("log1p_f32", -4.0, -0.1, 2.0),
    ("expm1_f32", -60.0, -1.52, 0.85), ("expm1_f32", -1.51, 4.0, 2.0)])
def test_float32_functions(fn, lo, hi, bar):
    x = _signed_log(90 + len(fn), lo, hi)
    if fn == "rsqrt_f32":
        x = np.abs(x)
    ours, ref = _run(fn, x)
    unit = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    # a result that rounds up to a power of two counts in the smaller unit below it
    below = np.abs(ref) < np.abs(ref).astype(np.float32)
    unit = np.where(below, np.spacing(np.nextafter(np.abs(ref).astype(np.float32), np.float32(0.0))), unit)
    assert np.max(np.abs(ours - ref) / unit) <= bar


def test_fixed_point_words():
    x = _signed_log(97, -300.0, 60.0)
    x[:8] = [1.0, -1.0, np.nextafter(2.0, 0.0), -np.nextafter(2.0, 0.0), 1.0 + 2.0 ** -52, 2.0 ** -300, 0.0, -0.0]
    x[8:4096] = 1.0 + 2.0 ** -52 * np.arange(4088)                 # carries of the truncated mantissa
    ours, ref = _run("fixed", x)
    d = np.arange(N) & 63
    top = np.exp2(np.floor(np.log2(np.where(ref == 0.0, 1.0, np.abs(ref)))) + 1 + d)   # 2^(E - 1022)
    assert np.array_equal(ours[d <= 4], ref[d <= 4])
    assert np.all(np.abs(ours) <= np.abs(ref)) and np.all(ours * ref >= 0.0)
    assert np.all(np.abs(ours - ref) < top * 2.0 ** -57)
    big = d >= 58
    assert np.all(ours[big] == 0.0)
