"""The saturation mask (csrc/mask.cu) at the edges of its tiles, for every tile
height (64, 32, 16 and 8 rows, by image size and halo), bit for bit against the
oracle: clusters of saturated pixels at word and tile borders, images smaller
than a word, a tile or the halo, and NaN and infinite pixels."""
import numpy as np
import pytest

from oracle import masking

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # n0, n1, grow
    (1, 1, 16), (3, 33, 16), (8, 256, 0), (9, 257, 1), (17, 31, 5), (40, 700, 16),  # 8 rows
    (1601, 300, 0), (1617, 512, 5), (900, 513, 16),                                 # 16 rows
    (1700, 1000, 0), (1000, 1793, 5), (2050, 260, 16),                              # 32 rows
    (1665, 2049, 0), (4097, 770, 5), (3300, 700, 16),                               # 64 rows
]


@pytest.mark.parametrize("n0,n1,grow", CASES)
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_tiles_match_oracle(n0, n1, grow, dtype):
    from paper_2109_09334_gb300 import binding as B
    rng = np.random.default_rng(n0 + 7 * n1 + grow)
    R, S = (rng.uniform(0, 100, (n0, n1)).astype(dtype) for _ in range(2))
    sat = 1e3
    for img in (R, S):  # sparse, so that most of the dilated area is the halo's
        for x, y in zip(rng.integers(0, n0, 12), rng.integers(0, n1, 12)):
            img[x, y] = sat
        for x in range(0, n0, 64):
            img[x, rng.choice([0, 31, 32, 255, 256, n1 - 1]) % n1] = sat
        img[rng.integers(0, n0), rng.integers(0, n1)] = np.inf
        img[rng.integers(0, n0), rng.integers(0, n1)] = np.nan
    m = torch.from_numpy((rng.random((n0, n1)) > 0.05).astype(np.uint8)).cuda()
    want = masking.saturation_mask(R.astype(np.float64), S.astype(np.float64), sat, sat, grow, m.cpu().numpy())
    B.sfft_saturation_mask(torch.from_numpy(R).cuda(), torch.from_numpy(S).cuda(), sat, sat, grow, m, d_mask_in=m)
    torch.cuda.synchronize()
    assert np.array_equal(m.cpu().numpy(), want)


@pytest.mark.parametrize("dtype,small,large", [("float32", (3500, 4000), (4096, 4096)),
                                               ("float64", (3001, 2048), (3500, 4000))])
def test_time_grows_no_faster_than_pixels(dtype, small, large):
    """The larger image's tiles run in one wave too (1024 of 64 rows in FP32, 880
    in FP64): its time against the smaller's is at most their pixels', and a
    tenth for noise.  With fewer resident blocks its last tiles took a wave of
    their own: 1.38 times for 1.20 times the pixels, 2.65 for 2.28."""
    from paper_2109_09334_gb300 import binding as B

    def best(n0, n1):
        R, S = (torch.rand((n0, n1), device="cuda", dtype=getattr(torch, dtype)) for _ in range(2))
        m = torch.empty((n0, n1), dtype=torch.uint8, device="cuda")
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        times = []
        for _ in range(8):
            ev[0].record()
            for _ in range(20):
                B.sfft_saturation_mask(R, S, 0.999, 0.999, 0, m)
            ev[1].record()
            torch.cuda.synchronize()
            times.append(ev[0].elapsed_time(ev[1]))
        return min(times)

    pixels = large[0] * large[1] / (small[0] * small[1])
    assert best(*large) <= 1.1 * pixels * best(*small)
