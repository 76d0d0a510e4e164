"""sfft_run_pairs and captured batches whose pairs share a buffer that one of
them writes: the results of one stream's order (every build, every solve, the
subtractions as listed), as sfft_run_pair gives them on the images as they were
at the start."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import random_field  # noqa: E402

pytestmark = pytest.mark.gpu

COUNT = 10  # two launches of the solve, on four streams where nothing is shared


@pytest.mark.parametrize("captured", [False, True])
def test_difference_over_another_pairs_reference(captured):
    from paper_2109_09334_gb300 import SfftBatch, SfftPlan, run_pairs
    sizes = [(64, 64) if k < COUNT - 1 else (512, 512) for k in range(COUNT)]  # the last build is the longest
    plans = [SfftPlan(a, b, 2, 2, 1, 1, True) for a, b in sizes]
    R = [torch.from_numpy(random_field(a, b, k).astype(np.float32)).cuda() for k, (a, b) in enumerate(sizes)]
    S = [torch.from_numpy(random_field(a, b, 50 + k).astype(np.float32)).cuda() for k, (a, b) in enumerate(sizes)]
    try:
        want = [p.run_pair(r, s)[0].clone() for p, r, s in zip(plans, R, S)]
        torch.cuda.synchronize()
        outs = [torch.empty_like(r) for r in R]
        outs[0] = R[COUNT - 1].view(-1)[:64 * 64].view(64, 64)  # over pixels that the last build reads
        outs[3] = outs[5]  # the later pair's stays
        if captured:
            batch = SfftBatch(plans, R, S, outs=outs, solve_group=3)
            batch.launch()
        else:
            run_pairs(plans, R, S, outs=outs)
        torch.cuda.synchronize()
        for k in range(COUNT):
            if k != 3:
                assert torch.equal(outs[k], want[k]), k
        if captured:
            batch.close()
    finally:
        for p in plans:
            p.close()
