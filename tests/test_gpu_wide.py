"""The wide-rank kernel (65 to 128 ranks, up to 16 tokens), forced, at the edges of its tiles: rows around 32 and 128,
columns around 64 and 128, ranks that are and are not 16-byte rows, and every way of splitting the columns over a cluster."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer, check_against_oracle

pytestmark = pytest.mark.gpu

SHAPES = [
    # bits, m, n, r, M, mixed
    (4, 1, 32, 65, 1, False),
    (4, 128, 128, 128, 1, False),        # one strip
    (4, 127, 160, 72, 8, True),
    (4, 129, 1056, 127, 9, True),
    (4, 4096, 192, 96, 16, False),       # many row tiles, few strips
    (3, 130, 128, 66, 2, True),
    (3, 257, 4096, 128, 16, True),
    (3, 96, 384, 100, 7, False),
    (2, 144, 64, 112, 1, True),
    (2, 200, 1088, 80, 15, False),
    (2, 33, 192, 128, 4, False),
]


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_set_option("splitk", "0")
    binding.lords_shutdown()


def _forward(lords, lay, split=0):
    lords.lords_set_option("path", "wide")
    lords.lords_set_option("splitk", str(split))
    try:
        dl = DeviceLayer(lay)
        y32, ybf = dl.forward()
        again = dl.forward()
        assert lords.lords_last_launch_count() == 1
    finally:
        lords.lords_set_option("path", "auto")
        lords.lords_set_option("splitk", "0")
    assert np.array_equal(y32, again[0]) and np.array_equal(ybf, again[1])
    return dl, y32, ybf


@pytest.mark.parametrize("bits,m,n,r,M,mixed", SHAPES)
def test_wide_kernel_shapes(lords, bits, m, n, r, M, mixed):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r + M, mixed_sign=mixed)
    dl, y32, ybf = _forward(lords, lay)
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


@pytest.mark.parametrize("split", [1, 2, 3, 7, 14, 16])
def test_wide_kernel_cluster_splits(lords, split):
    lay = gen.make_integer_layer(300, 2112, 90, 5, bits=4, seed=split)
    dl, y32, ybf = _forward(lords, lay, split)
    want = oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, 4)
    assert np.array_equal(y32.astype(np.float64), want)
