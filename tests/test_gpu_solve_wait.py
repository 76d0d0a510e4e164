"""The bounded waits of the solve's grid barrier (csrc/solve.cu): a wait that
runs out ends the launch in every block, with a status, and leaves the plan
usable.  The limit is set to 0 cycles, so that the first block that has to wait
gives up; nothing is made to hang."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


def test_hook_checks_its_plan():
    from paper_2109_09334_gb300 import binding as B
    from paper_2109_09334_gb300.build import build
    build()
    assert B.library().sfft_plan_debug_solve_wait(None, 0) == B.SFFT_ERR_INVALID


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tensor_cores", [("fp64", 0), ("mixed", 0), ("mixed", 2)])
@pytest.mark.parametrize("count", [1, 3])
def test_wait_that_runs_out(precision, tensor_cores, count):
    from paper_2109_09334_gb300 import SfftPlan, binding as B, info_from_bytes
    plans, M, rhs = [], [], []
    for k in range(count):
        p = SfftPlan(64, 64, 3 + k, 3, 1, 1, True, dtype="float64" if precision == "fp64" else "float32",
                     precision=precision)
        was = B.sfft_plan_tuning(p.handle)
        B.sfft_plan_set_tuning(p.handle, [0, 0, 0, 0, tensor_cores])
        G = np.random.default_rng(k).standard_normal((p.n, 4 * p.n))
        plans.append(p)
        M.append(torch.from_numpy(G @ G.T).cuda())
        rhs.append(torch.from_numpy(G[:, 0].copy()).cuda())

    def solve():
        x = [torch.full((p.n,), float("nan"), dtype=torch.float64, device="cuda") for p in plans]
        info = [torch.zeros(24, dtype=torch.uint8, device="cuda") for _ in plans]
        B.sfft_solve_batch([p.handle for p in plans], M, rhs, x, info, torch.cuda.current_stream())
        torch.cuda.synchronize()
        return [v.cpu().numpy() for v in x], [info_from_bytes(v.cpu().numpy())["status"] for v in info]

    try:
        before, status = solve()
        assert status == [B.SFFT_OK] * count
        for _ in range(3):
            B.sfft_plan_debug_solve_wait(plans[0].handle, 0)
            x, status = solve()
            assert status == [B.SFFT_ERR_TIMEOUT] * count
            assert all(not v.any() for v in x)
            B.sfft_plan_debug_solve_wait(plans[0].handle, -1)
            x, status = solve()
            assert status == [B.SFFT_OK] * count
            assert all(np.array_equal(a, b) for a, b in zip(x, before))
    finally:
        B.sfft_plan_set_tuning(plans[0].handle, was)
        for p in plans:
            p.close()
