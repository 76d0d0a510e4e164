"""Error of a mixed-precision pair's difference image against 64 bits, where the
lag sums along x and the row segments set it: rows or columns of other lengths
than powers of two.  Limits: 1.4 times the mean error over these seeds of the
transforms that the windows took the place of (direct lag sums along x in FP32
with compensated sums, and Bluestein rows): 1.92e-6, 1.17e-6 and 4.79e-6; single
seeds spread by a tenth of that.  (Windows with rounded twiddles and an FP32
inverse, and segments on short rows, came to 3.9e-6, 3.2e-6 and 1.0e-5.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from perf import cases  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,n1,w,dk,db,was", [(1501, 512, 5, 2, 1, 1.92e-6), (1100, 240, 5, 1, 1, 1.17e-6),
                                               (1100, 260, 8, 2, 2, 4.79e-6)])
def test_error_of_difference(n0, n1, w, dk, db, was):
    case = {"kind": "pair", "n0": n0, "n1": n1, "w": w, "dk": dk, "db": db, "const": True, "precision": "mixed",
            "spline": "", "masked": False, "count": 1}
    err = []
    for seed in (11, 12, 13, 14):
        state = cases.prepare(case, seed)
        D = cases.run(state)["D"]
        torch.cuda.synchronize()
        want = cases.exact(case, seed)["D"]
        err.append(float((D.double() - want).norm() / want.norm()))
        state["plan"].close()
    assert np.mean(err) <= 1.4 * was, err
