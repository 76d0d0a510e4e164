"""The subtraction (csrc/subtract.cu) where a fit's kernel values fill shared
memory: kept once instead of as two pairs, and segments of the columns halved
until they fit beside them.

Tolerance: an output sums N = n_K (2 w0 + 1) (2 w1 + 1) products whose partial sums
stay within a few times the largest output; N independent roundings of
relative size u (half an ulp) give u sqrt(N) of that, taken times 8."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from synth import coefficient_draw, random_field  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    # n0, w0, precision (37 B-spline terms, n1 = 16, w1 = 0)
    (1000, 172, "mixed"),  # the last half-width whose values fit as two pairs
    (1000, 176, "mixed"),  # kept once
    (1500, 340, "mixed"),  # and shorter segments
    (681, 170, "fp64"),    # FP64: shorter segments
]


@pytest.mark.parametrize("n0,w0,precision", CASES)
def test_wide_kernel_against_oracle(n0, w0, precision):
    from paper_2109_09334_gb300 import SfftPlan
    n1 = 16
    dt = np.float64 if precision == "fp64" else np.float32
    R, S = (random_field(n0, n1, k).astype(dt) for k in (1, 2))
    plan = SfftPlan(n0, n1, w0, 0, 0, 0, True, dtype=np.dtype(dt).name, precision=precision, spline=(2, 3, 0, 0))
    try:
        x = coefficient_draw(plan.n, 7, 0.02)
        D = plan.subtract(*(torch.from_numpy(v).cuda() for v in (R, S, x))).double().cpu().numpy()
    finally:
        plan.close()
    c = oracle.OracleConfig(n0, n1, w0, 0, 0, 0, True, "bspline", 2, 3, 0, 0)
    Do = oracle.subtract(R.astype(np.float64), S.astype(np.float64), x, c)
    u = 2.0 ** (-53 if precision == "fp64" else -24)
    err = np.abs(D - Do)
    top = np.abs(Do).max()
    assert np.sqrt(np.mean(err ** 2)) <= 8 * u * np.sqrt(37 * (2 * w0 + 1)) * top
    assert err.max() <= 8 * 8 * u * np.sqrt(37 * (2 * w0 + 1)) * top
