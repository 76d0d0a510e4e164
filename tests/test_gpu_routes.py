"""The fits that keep the column transforms, the direct lag sums or the
Bluestein rows (polynomial degree 3, half-widths above 16, B-splines): parity
with the oracle where the row count is no power of two, launch shapes, and
stream capture."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from synth import random_field  # noqa: E402
from test_gpu_parity import check_against_oracle, gpu_run, small_pair  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    # n0, n1, w0, w1, dk, db, cpr, masked
    (48, 40, 2, 2, 3, 1, 1, False),   # ten terms, neither axis a power of two
    (50, 64, 2, 1, 3, 3, 0, True),    # ten terms, rows a power of two
    (64, 41, 1, 2, 3, 0, 1, False),   # ten terms, columns a power of two, Bluestein rows
    (75, 41, 17, 2, 1, 1, 1, False),  # half-width above 16 along x
    (72, 96, 2, 20, 2, 1, 1, True),   # and along y
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}w{c[2]},{c[3]}d{c[4]}" for c in CASES])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_parity(case, precision):
    n0, n1, w0, w1, dk, db, cpr, masked = case
    R, S = small_pair(n0, n1, seed=n0 + 3 * n1 + w0)
    mask = (np.random.default_rng(n0).random((n0, n1)) > 0.15).astype(np.uint8) if masked else None
    c = oracle.OracleConfig(n0, n1, w0, w1, dk, db, bool(cpr))
    g = gpu_run(R, S, w0, w1, dk, db, cpr, precision, "float64" if precision == "fp64" else "float32", mask)
    check_against_oracle(R, S, c, precision, mask, g)
    g["plan"].close()


@pytest.mark.parametrize("dk,spline", [(3, None), (0, (2, 0, 1, 1))])
@pytest.mark.parametrize("shape", [(256, 64), (64, 48)])
def test_images_per_block(dk, spline, shape):
    """Every number of images per block of the column FFT gives the built-in choice's results."""
    from paper_2109_09334_gb300 import SfftPlan, binding as B
    n0, n1 = shape
    R, S = (torch.from_numpy(v).float().cuda() for v in small_pair(n0, n1, 5))
    plan = SfftPlan(n0, n1, 2, 2, dk, 0, 1, spline=spline)
    was = B.sfft_plan_tuning(plan.handle)
    try:
        want = None
        for shapes in ([0, 0, 0, 0, 0], [1, 1, 1, 0, 0], [2, 2, 2, 0, 0], [4, 3, 1, 0, 0], [16, 4, 4, 0, 0]):
            B.sfft_plan_set_tuning(plan.handle, shapes)
            D, x, _, M, _ = plan.run_pair(R, S, keep_system=True)
            torch.cuda.synchronize()
            got = [v.cpu().numpy() for v in (M, x, D)]
            want = want or got
            assert all(np.array_equal(a, b) for a, b in zip(got, want)), shapes
        B.sfft_plan_set_tuning(plan.handle, [0, 0, 0, 0, 0])
        shapes = plan.autotune(R, S)
        D, x, _, M, _ = plan.run_pair(R, S, keep_system=True)
        torch.cuda.synchronize()
        assert all(np.array_equal(v.cpu().numpy(), w) for v, w in zip((M, x, D), want)), shapes
    finally:
        B.sfft_plan_set_tuning(plan.handle, was)
        plan.close()


@pytest.mark.parametrize("n0", [64, 70])  # column FFT and gather; direct lag sums
def test_captured_masked_bspline_pair(n0):
    """The unmasked rows overwrite the masked ones beside the lag sums' second
    stage: a captured pair replays to the eager call's results on new images."""
    from paper_2109_09334_gb300 import SfftPlan, binding as B
    n1 = 48
    make = lambda k: torch.from_numpy(random_field(n0, n1, k).astype(np.float32)).cuda()  # noqa: E731
    R, S = make(1), make(2)
    mask = torch.from_numpy((np.random.default_rng(3).random((n0, n1)) > 0.1).astype(np.uint8)).cuda()
    plan = SfftPlan(n0, n1, 2, 2, 0, 0, True, spline=(1, 1, 1, 0))
    out = [(torch.zeros((n0, n1), device="cuda"), torch.zeros(plan.n, dtype=torch.float64, device="cuda"))
           for _ in range(2)]

    def run(k, stream):
        B.sfft_run_pair(plan.handle, R, S, mask, None, None, out[k][1], None, out[k][0], stream)

    try:
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            run(0, torch.cuda.current_stream().cuda_stream)
        for k in range(3):
            g.replay()
            torch.cuda.synchronize()
            run(1, torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
            assert float(out[1][0].abs().max()) > 0
            R.copy_(make(10 + k))
            S.copy_(make(20 + k))
            torch.cuda.synchronize()
    finally:
        plan.close()
