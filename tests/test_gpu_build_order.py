"""A build's kernels beside the transforms (its own stream) leave the time of
the direct lag sums alone: these keep few long blocks, whose placement the other
kernels disturbed.  The build may take no more than the sum of its stages, each
replayed alone, and a fifth (it took 1.5 to 2.2 times that)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,n1", [(300, 256), (300, 280)])
def test_build_takes_its_stages_time(n0, n1):
    from paper_2109_09334_gb300 import SfftPlan, binding as B
    g = torch.Generator(device="cuda").manual_seed(1)
    R, S = (100 + 5 * torch.randn((n0, n1), device="cuda", dtype=torch.float64, generator=g) for _ in range(2))
    plan = SfftPlan(n0, n1, 4, 4, 0, 0, True, dtype="float64", precision="fp64", spline=(2, 1, 1, 0))
    try:
        plan.run_pair(R, S)
        M, rhs = plan.build_system(R, S)

        def ms(f):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            best = float("inf")
            for _ in range(5):
                a.record()
                f()
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            return best

        stages = sum(ms(lambda: B.sfft_replay_stage(plan.handle, k, plan.stream)) for k in range(4))
        build = ms(lambda: B.sfft_build_system(plan.handle, R, S, None, M, rhs, plan.stream))
        assert build <= 1.2 * stages, (build, stages)
    finally:
        plan.close()
