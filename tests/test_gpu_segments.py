"""The overlap-save transforms (csrc/segment.cu) against the oracle at the
edges of their segments: lag sums along x over segments of 128 - 4 w0 samples
taken four (six terms, three terms) or sixteen (one term) at a time, and row
transforms over segments of at most 256 - 4 w1 pixels.  The system is compared
with the oracle's and the subtraction is applied to given coefficients, with
the tolerances of test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from synth import coefficient_draw, random_field  # noqa: E402
from test_gpu_parity import SIGMA, check_system  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    # n0, n1, w0, w1, dk, db, cpr, masked
    (96, 225, 8, 8, 1, 1, 1, False),   # one whole segment along x; two row segments
    (97, 449, 8, 8, 1, 1, 0, True),    # a last segment of one sample; three row segments
    (385, 30, 8, 2, 2, 0, 1, False),   # a batch of four segments and one sample; the row window wraps the row
    (21, 700, 2, 16, 1, 1, 1, True),   # the window along x wraps the image; the widest row halo
    (70, 67, 16, 16, 0, 0, 1, False),  # the largest lags, 32
    (513, 33, 0, 1, 2, 1, 0, False),   # no halo: segments of 128
    (2049, 20, 0, 0, 0, 1, 1, False),  # one term: a batch of sixteen segments and one sample
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}w{c[2]}" for c in CASES])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_segment_edges_against_oracle(case, precision):
    from paper_2109_09334_gb300 import SfftPlan
    n0, n1, w0, w1, dk, db, cpr, masked = case
    dt = np.float64 if precision == "fp64" else np.float32
    R = random_field(n0, n1, 3 + n0).astype(dt).astype(np.float64)
    S = (0.9 * np.roll(R, (1, 2), axis=(0, 1)) + 0.2 * random_field(n0, n1, 5 + n1)).astype(dt).astype(np.float64)
    mask = (np.random.default_rng(n0).random((n0, n1)) > 0.15).astype(np.uint8) if masked else None
    c = oracle.OracleConfig(n0, n1, w0, w1, dk, db, bool(cpr))
    Mo, ro = oracle.build_system(R, S, c, mask=mask)
    plan = SfftPlan(n0, n1, w0, w1, dk, db, cpr, dtype=np.dtype(dt).name, precision=precision)
    try:
        Rt, St = (torch.from_numpy(v.astype(dt)).cuda() for v in (R, S))
        M, rhs = plan.build_system(Rt, St, None if mask is None else torch.from_numpy(mask).cuda())
        tol = (1e-10, 1e-9) if precision == "fp64" else (1e-5, 1e-4)
        check_system(M.cpu().numpy(), rhs.cpu().numpy(), Mo, ro, c, S, mask, *tol)
        x = coefficient_draw(plan.n, 7, 0.02)
        D = plan.subtract(Rt, St, torch.from_numpy(x).cuda()).double().cpu().numpy()
        Do = oracle.subtract(R, S, x, c)
        scale = max(1.0, np.abs(Do).max() / (100 * SIGMA))  # large coefficients: relative to the model's range
        rms, top = (1e-6, 1e-5) if precision == "fp64" else (1e-3, 1e-2)
        assert np.sqrt(np.mean((D - Do) ** 2)) <= rms * SIGMA * scale
        assert np.max(np.abs(D - Do)) <= top * SIGMA * scale
    finally:
        plan.close()
