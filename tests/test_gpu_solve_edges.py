"""The solve (csrc/solve.cu) at the edges of its tiles (64 unknowns in FP32, 32
in FP64) and of the 32-wide blocks inside them, through sfft_solve_static: the
refinement's tolerance on the FP64 residual, the solution against numpy's, and
a system whose Cholesky fails in a given block."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def solve(M, rhs, precision):
    from paper_2109_09334_gb300 import binding as B, info_from_bytes
    n = len(rhs)
    x = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    info = torch.zeros(ctypes.sizeof(B.sfft_solve_info), dtype=torch.uint8, device="cuda")
    B.sfft_solve_static(torch.from_numpy(M).cuda(), torch.from_numpy(rhs).cuda(), n, precision, x, info,
                        torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return x.cpu().numpy(), info_from_bytes(info.cpu().numpy())


def system(n, seed):
    """Wishart matrix of 4 n samples (condition number near 9) with scales over four decades."""
    rng = np.random.default_rng(seed)
    G = rng.standard_normal((n, 4 * n)) * 10.0 ** rng.uniform(-2, 2, n)[:, None]
    return G @ G.T, rng.standard_normal(n)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 193, 321, 1023, 1024])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solve_sizes(n, precision):
    from paper_2109_09334_gb300 import binding as B
    M, rhs = system(n, n)
    x, info = solve(M, rhs, precision)
    assert info["status"] == B.SFFT_OK
    # 1e-12 is the solver's stopping rule; the residual's own rounding here is
    # below n eps ||M|| ||x|| / ||rhs||
    own = n * 2.3e-16 * np.linalg.norm(M, 2) * np.linalg.norm(x) / np.linalg.norm(rhs)
    assert np.linalg.norm(rhs - M @ x) <= (1e-12 + 2 * own) * np.linalg.norm(rhs)
    d = 1 / np.sqrt(np.diag(M))
    A = d[:, None] * M * d[None, :]
    xs, want = x / d, np.linalg.solve(A, d * rhs)
    # scaled, ||A^-1|| times the scaled residual
    bound = np.linalg.norm(np.linalg.inv(A), 2) * (np.linalg.norm(d * (rhs - M @ x)) + n * 2.3e-16 * np.linalg.norm(d * rhs))
    assert np.linalg.norm(xs - want) <= 2 * bound + 1e-14 * np.linalg.norm(want)


@pytest.mark.parametrize("at", [0, 31, 32, 63, 64, 100, 149])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solve_reports_a_bad_pivot(at, precision):
    from paper_2109_09334_gb300 import binding as B
    M, rhs = system(150, 7)
    M[at, at] *= 1e-3 if at else -1.0  # far below the Schur complement's need
    _, info = solve(M, rhs, precision)
    assert info["status"] == B.SFFT_ERR_SINGULAR
