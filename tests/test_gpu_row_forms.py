"""Plans whose builds take Bluestein rows and whose own subtractions take
segments: a masked pair (rows of both forms in one call) against the oracle, and
a subtraction alone against the pair's, with the tolerances of
test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from test_gpu_parity import SIGMA, check_against_oracle, gpu_run, small_pair  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    # n0, n1, w0, w1, dk, db, precision
    (60, 90, 2, 2, 1, 1, "mixed"),
    (64, 300, 3, 3, 2, 1, "mixed"),    # two segments
    (45, 511, 2, 16, 1, 0, "mixed"),   # the longest, the widest halo
    (60, 100, 2, 2, 2, 1, "fp64"),
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}{c[6]}" for c in CASES])
@pytest.mark.parametrize("masked", [True, False])
def test_both_forms(case, masked):
    n0, n1, w0, w1, dk, db, precision = case
    dtype = "float64" if precision == "fp64" else "float32"
    R, S = small_pair(n0, n1, seed=n0 + n1)
    mask = (np.random.default_rng(n0).random((n0, n1)) > 0.15).astype(np.uint8) if masked else None
    g = gpu_run(R, S, w0, w1, dk, db, 1, precision, dtype, mask)
    try:
        check_against_oracle(R, S, oracle.OracleConfig(n0, n1, w0, w1, dk, db, True), precision, mask, g)
        D = g["plan"].subtract(g["R"], g["S"], torch.from_numpy(g["x"]).cuda()).double().cpu().numpy()
        if masked:  # the same kernels on the same rows
            assert np.array_equal(D, g["D"])
        else:
            rms, top = (1e-6, 1e-5) if precision == "fp64" else (1e-3, 1e-2)
            assert np.sqrt(np.mean((D - g["D"]) ** 2)) <= rms * SIGMA
            assert np.max(np.abs(D - g["D"])) <= top * SIGMA
    finally:
        g["plan"].close()
