"""The scale-MMA kernel on CTA pairs at the edges of its tiles: rows around 128 and 256, columns around
a step of 128, token counts around whole and uneven token tiles, ranks that are and are not 16-byte rows,
one piece per tile and several."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer, check_against_oracle

pytestmark = pytest.mark.gpu

SHAPES = [
    # bits, m, n, r, M, mixed
    (4, 300, 256, 16, 1, True),          # one token in a tile of 32
    (2, 260, 512, 32, 40, False),
    (4, 130, 64, 1, 129, False),         # half a step
    (4, 128, 128, 16, 160, False),       # one step
    (4, 129, 192, 5, 161, True),         # padded copy of B
    (4, 256, 320, 20, 256, False),
    (4, 257, 1024, 64, 257, True),       # two token tiles, uneven
    (4, 300, 4096, 33, 300, False),      # many pieces to a tile
    (4, 5000, 512, 32, 1100, False),     # whole waves and pieces
    (3, 127, 128, 8, 129, True),
    (3, 255, 384, 48, 512, False),
    (3, 1024, 2048, 7, 513, True),
    (2, 64, 64, 4, 144, True),
    (2, 384, 704, 40, 200, False),
    (2, 700, 1024, 64, 290, False),
]


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_shutdown()


@pytest.mark.parametrize("bits,m,n,r,M,mixed", SHAPES)
def test_pair_kernel_shapes(lords, bits, m, n, r, M, mixed):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r + M, mixed_sign=mixed)
    lords.lords_set_option("path", "pair")
    try:
        dl = DeviceLayer(lay)
        y32, ybf = dl.forward()
        again = dl.forward()
        assert lords.lords_last_launch_count() == 2
    finally:
        lords.lords_set_option("path", "auto")
    assert np.array_equal(y32, again[0]) and np.array_equal(ybf, again[1])
    assert lords.lords_poll_status() == 0
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


@pytest.mark.parametrize("path", ["pair", "dense"])
@pytest.mark.parametrize("bits,m,n,r,M", [
    (4, 5000, 512, 32, 1100),       # two waves of whole tiles, the last one partial
    (3, 5000, 4224, 8, 1100),       # a whole wave, the tiles left over cut
    (4, 4700, 2880, 16, 1000),      # few tiles more than a wave: all of them cut
])
def test_division_of_tiles(lords, path, bits, m, n, r, M):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r + M)
    lords.lords_set_option("path", path)
    try:
        dl = DeviceLayer(lay)
        y32, ybf = dl.forward()
    finally:
        lords.lords_set_option("path", "auto")
    assert lords.lords_poll_status() == 0
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))
