"""The kernels that run beside the caller's stream (the moments, the unmasked
rows of a masked pair, the lanes of a set of pairs) under stream capture: a
captured call replays to the eager call's results bit for bit, on new inputs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import random_field  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,n1,masked", [(64, 64, False), (70, 90, True), (128, 64, True)])
def test_captured_pair_equals_eager(n0, n1, masked):
    from paper_2109_09334_gb300 import SfftPlan, binding as B
    make = lambda k: torch.from_numpy(random_field(n0, n1, k).astype(np.float32)).cuda()  # noqa: E731
    R, S = make(1), make(2)
    mask = torch.from_numpy((np.random.default_rng(3).random((n0, n1)) > 0.1).astype(np.uint8)).cuda() if masked else None
    plan = SfftPlan(n0, n1, 2, 2, 1, 1, True)
    out = {}
    for name in ("graph", "eager"):
        out[name] = (torch.zeros((n0, n1), device="cuda"), torch.zeros(plan.n, dtype=torch.float64, device="cuda"))

    def run(name, stream):
        D, x = out[name]
        B.sfft_run_pair(plan.handle, R, S, mask, None, None, x, None, D, stream)

    try:
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            run("graph", torch.cuda.current_stream().cuda_stream)
        for k in range(2):  # the second replay on new images
            g.replay()
            torch.cuda.synchronize()
            run("eager", torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            assert torch.equal(out["graph"][0], out["eager"][0]) and torch.equal(out["graph"][1], out["eager"][1])
            assert float(out["eager"][0].abs().max()) > 0
            R.copy_(make(10 + k))
            S.copy_(make(20 + k))
            torch.cuda.synchronize()
    finally:
        plan.close()
