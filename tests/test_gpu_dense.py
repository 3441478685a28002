"""The two-phase path (weights expanded to scratch, then a dense product on CTA pairs), forced, at the edges of
its tiles: rows around 128 / 256, columns around 64 and off every alignment, ranks at and past each fragment
count, token counts around each token tile, split tiles (few tiles, many k-steps) and whole waves."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer, check_against_oracle

pytestmark = pytest.mark.gpu

SHAPES = [
    # bits, m, n, r, M, mixed
    (4, 256, 64, 4, 1, False),          # one k-step
    (4, 1, 2, 1, 1, False),
    (4, 255, 66, 5, 3, True),
    (4, 257, 1000, 32, 31, True),
    (2, 128, 130 * 4, 33, 32, False),
    (3, 129, 352, 64, 33, True),
    (4, 300, 1022, 65, 64, False),
    (2, 513, 1028, 128, 65, True),
    (3, 640, 2048, 16, 128, False),     # few tiles: k-ranges split over several pairs
    (4, 256, 8192, 17, 129, True),
    (4, 1000, 2730, 10, 37, False),
    (4, 384, 1536, 100, 255, False),
    (3, 384, 96, 48, 257, True),
    (4, 2100, 512, 8, 2300, False),     # more tiles than pairs: whole waves and a shared rest
    (2, 5000, 192, 12, 600, True),
]


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_shutdown()


def _forward(lords, lay):
    lords.lords_set_option("path", "dense")
    try:
        dl = DeviceLayer(lay)
        y32, ybf = dl.forward()
        again = dl.forward()
    finally:
        lords.lords_set_option("path", "auto")
    assert np.array_equal(y32, again[0]) and np.array_equal(ybf, again[1])      # pieces are added in a fixed order
    return dl, y32, ybf


@pytest.mark.parametrize("bits,m,n,r,M,mixed", SHAPES)
def test_dense_path_shapes(lords, bits, m, n, r, M, mixed):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r + M, mixed_sign=mixed)
    dl, y32, ybf = _forward(lords, lay)
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


@pytest.mark.parametrize("bits,m,n,r,M", [(4, 300, 1030, 9, 40), (3, 260, 4096, 128, 5), (2, 700, 516, 40, 300)])
def test_dense_path_integer_case_is_bit_exact(lords, bits, m, n, r, M):
    lay = gen.make_integer_layer(m, n, r, M, bits=bits, seed=bits + m)
    dl, y32, ybf = _forward(lords, lay)
    assert np.array_equal(y32.astype(np.float64), oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


def test_dense_path_in_row_chunks(lords):
    """A workspace that holds only some row tiles of W^: the layer runs chunk by chunk."""
    lay = gen.make_layer(1300, 1024, 24, 20, bits=4, seed=5, mixed_sign=True)
    lords.lords_init(0, 4 << 20)
    try:
        _, small, _ = _forward(lords, lay)
        assert lords.lords_last_launch_count() > 2
    finally:
        lords.lords_init(0, 0)
    dl, y32, ybf = _forward(lords, lay)
    assert lords.lords_last_launch_count() == 2
    want = oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, 4)
    check_against_oracle(y32, ybf, want)
    assert np.linalg.norm(small - want) <= 1e-3 * np.linalg.norm(want)
