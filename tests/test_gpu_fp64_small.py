"""FP64 builds at the borders of their routes: columns of fewer windows than a
batch of the lag sums (their transforms packed into warps), the column FFT on
both sides of its limits, and rows by Bluestein or by segments.  Against the
oracle with the tolerances of test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from test_gpu_parity import check_against_oracle, gpu_run, small_pair  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    # n0, n1, w0, w1, dk, db, cpr, masked
    (96, 64, 8, 2, 2, 1, 1, False),     # one window (of 96 samples)
    (97, 64, 8, 2, 2, 1, 1, True),      # two, the last of one sample
    (200, 32, 8, 2, 1, 1, 0, False),    # three
    (384, 32, 8, 1, 2, 0, 1, False),    # a whole batch
    (385, 32, 8, 1, 1, 0, 1, False),    # and one more
    (300, 40, 8, 2, 0, 1, 1, True),     # one term: four of a batch of sixteen
    (2040, 17, 0, 1, 0, 0, 1, False),   # all sixteen
    (16, 513, 1, 1, 2, 1, 1, False),    # rows by segments, one window
    (16, 512, 1, 1, 2, 1, 1, False),    # the last row length without the column FFT
    (16, 1024, 1, 2, 2, 1, 1, True),    # column FFT
    (512, 1024, 1, 1, 1, 0, 1, False),  # column FFT, three terms
    (512, 1024, 1, 1, 0, 0, 1, False),  # windows
    (64, 64, 2, 2, 1, 1, 1, False),
    (64, 63, 2, 2, 1, 1, 1, False),     # three terms: Bluestein rows of 128
    (64, 65, 2, 2, 1, 1, 1, False),     # segments
    (64, 127, 2, 2, 2, 1, 1, False),    # six terms: Bluestein rows of 256
    (64, 129, 2, 2, 2, 1, 1, False),    # segments
    (64, 31, 2, 2, 0, 1, 1, False),     # one term: Bluestein rows of 64
    (64, 33, 2, 2, 0, 1, 1, False),     # segments
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}w{c[2]}d{c[4]}" for c in CASES])
def test_fp64_routes(case):
    n0, n1, w0, w1, dk, db, cpr, masked = case
    R, S = small_pair(n0, n1, seed=n0 + 3 * n1 + w0)
    mask = (np.random.default_rng(n0).random((n0, n1)) > 0.15).astype(np.uint8) if masked else None
    c = oracle.OracleConfig(n0, n1, w0, w1, dk, db, bool(cpr))
    g = gpu_run(R, S, w0, w1, dk, db, cpr, "fp64", "float64", mask)
    check_against_oracle(R, S, c, "fp64", mask, g)
    g["plan"].close()
