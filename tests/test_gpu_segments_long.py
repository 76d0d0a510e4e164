"""The edges of test_gpu_segments.py on rows long enough for segments in mixed
precision too (above 512 pixels), with its checks and tolerances."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_segments as edges  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [
    # n0, n1, w0, w1, dk, db, cpr, masked
    (96, 513, 8, 16, 1, 1, 1, False),  # one whole segment along x; three row segments, the widest halo
    (97, 672, 8, 8, 1, 1, 0, True),    # a last segment of one sample; three whole row segments
    (385, 673, 8, 8, 0, 0, 1, False),  # four segments and one sample; a row segment more, all shorter
    (21, 767, 2, 0, 2, 1, 1, True),    # the window along x wraps the image; no row halo, a last row segment of 255
    (70, 1000, 16, 1, 1, 0, 1, False), # the largest lags
    (513, 600, 0, 1, 2, 0, 0, False),  # no halo along x
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}w{c[2]}" for c in CASES])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_long_rows(case, precision):
    edges.test_segment_edges_against_oracle(case, precision)
