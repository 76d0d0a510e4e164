"""Launch shapes of plans whose rows are transformed by segments: their kernels
have one shape, so the autotuner leaves the row shapes alone, and plans whose
transforms are other kernels do not inherit theirs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import random_field  # noqa: E402

pytestmark = pytest.mark.gpu


def test_shapes_of_kernels_not_run_stay():
    from paper_2109_09334_gb300 import SfftPlan, binding as B
    n0, n1 = 96, 600
    R, S = (torch.from_numpy(random_field(n0, n1, k)).float().cuda() for k in (1, 2))
    seg, blu = SfftPlan(n0, n1, 3, 3, 1, 1, 1), None
    was = B.sfft_plan_tuning(seg.handle)
    try:
        for v in (0, 1):
            B.sfft_plan_set_tuning(seg.handle, [v, v, v, 0, 0])
            for _ in range(3):
                assert list(seg.autotune(R, S).values()) == [v, v, v, 0, 0]
        other = SfftPlan(n0, n1, 2, 2, 1, 1, 1)  # the same kernels
        assert list(B.sfft_plan_tuning(other.handle).values()) == [1, 1, 1, 0, 0]
        other.close()
        blu = SfftPlan(n0, n1, 3, 20, 1, 1, 1)  # half-width above 16: Bluestein rows
        assert list(B.sfft_plan_tuning(blu.handle).values()) == [0, 0, 0, 0, 0]
        D0 = blu.run_pair(R, S)[0].cpu().numpy()
        blu.autotune(R, S)
        assert np.array_equal(blu.run_pair(R, S)[0].cpu().numpy(), D0)
    finally:
        B.sfft_plan_set_tuning(seg.handle, was)
        for p in (seg, blu):
            if p is not None:
                p.close()
