"""The direct kernel (weights formed in registers and multiplied there), forced, at the edges of its tiles: rows
around 16 and 128, columns around 64 and off every alignment, ranks at and past each fragment count, both token
groups and several of them, and every way of splitting the columns over a cluster."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer, check_against_oracle

pytestmark = pytest.mark.gpu

SHAPES = [
    # bits, m, n, r, M, mixed
    (4, 1, 2, 1, 1, False),
    (4, 128, 64, 4, 1, False),          # one strip
    (4, 127, 66, 32, 8, True),
    (4, 129, 1000, 33, 9, True),
    (4, 256, 2730, 10, 16, False),
    (4, 300, 4096, 128, 3, True),
    (4, 4096, 192, 17, 8, False),       # many row tiles, few strips
    (3, 130, 64, 5, 2, True),
    (3, 257, 352, 48, 16, True),
    (3, 96, 1056, 65, 7, False),
    (3, 640, 4096, 96, 8, True),
    (2, 144, 132, 16, 1, True),
    (2, 200, 1028, 64, 15, False),
    (2, 384, 2048, 100, 16, True),
    (2, 16, 4, 2, 4, False),
    (4, 200, 1000, 10, 17, True),       # more than one token group
    (3, 130, 352, 48, 40, False),
    (4, 1000, 2730, 10, 37, False),
    (2, 140, 260, 70, 128, True),
    # the form with fp16 operands (n a multiple of 64 or 128, ranks up to 64, three tokens and more; the others are computed in fp32)
    (4, 130, 128, 33, 9, True),
    (4, 129, 64, 5, 17, False),
    (3, 127, 128, 16, 3, True),
    (3, 300, 1024, 64, 16, False),
    (2, 300, 192, 48, 8, True),
]
# groups of up to 24 and 32 tokens, their remainders and several of them; ranks in one fragment and past it; codes in asynchronous copies (n a
# multiple of 32) and through registers
GROUP_SHAPES = [(bits, m, n, r, M, M % 2 == 0) for (bits, m, n, r) in
                ((4, 2700, 2080, 16), (4, 2700, 1002, 17), (3, 2700, 1056, 33), (2, 2700, 1004, 64))
                for M in (17, 24, 25, 32, 33, 48, 49, 65, 128)]


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_set_option("splitk", "0")
    binding.lords_shutdown()


def _forward(lords, lay, split=0):
    lords.lords_set_option("path", "direct")
    lords.lords_set_option("splitk", str(split))
    try:
        dl = DeviceLayer(lay)
        y32, ybf = dl.forward()
        again = dl.forward()
        assert lords.lords_last_path() == "direct" and lords.lords_last_launch_count() == 1
    finally:
        lords.lords_set_option("path", "auto")
        lords.lords_set_option("splitk", "0")
    assert np.array_equal(y32, again[0]) and np.array_equal(ybf, again[1])
    return dl, y32, ybf


@pytest.mark.parametrize("bits,m,n,r,M,mixed", SHAPES + GROUP_SHAPES)
def test_direct_kernel_shapes(lords, bits, m, n, r, M, mixed):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r + M, mixed_sign=mixed)
    dl, y32, ybf = _forward(lords, lay)
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


@pytest.mark.parametrize("split", [1, 2, 3, 7, 14, 16])
def test_direct_kernel_cluster_splits(lords, split):
    lay = gen.make_integer_layer(300, 1100, 9, 5, bits=4, seed=split)
    dl, y32, ybf = _forward(lords, lay, split)
    want = oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, 4)
    assert np.array_equal(y32.astype(np.float64), want)


# Under a forced split the fewest groups win and of those the narrowest: groups of 24 tokens, 24, 32, 32, two of 24, two of 32; 16 with ranks
# above 64 and with fp16 operands
@pytest.mark.parametrize("bits,m,n,r", [(4, 300, 1100, 9), (3, 260, 1056, 30), (2, 200, 1000, 60), (4, 257, 1152, 40), (4, 200, 1100, 70)])
@pytest.mark.parametrize("M", [17, 24, 25, 32, 47, 63])
@pytest.mark.parametrize("split", [1, 3])
def test_direct_kernel_group_widths(lords, bits, m, n, r, M, split):
    lay = gen.make_integer_layer(m, n, r, M, bits=bits, seed=M + split)
    dl, y32, ybf = _forward(lords, lay, split)
    want = oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits)
    assert np.array_equal(y32.astype(np.float64), want)
