"""The scale-MMA kernels.  Where the two CTAs of a cluster share a tile's columns and exchange halves of its tokens: every token tile, token
counts around its half and its whole, ragged rows; sums of small integers are exact in any order.  And what the dispatch chooses by its
estimates: the kernel on CTA pairs from 17 tokens on, and small and large token tiles."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer, check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_set_option("bn", "0")
    binding.lords_shutdown()


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("bn,M", [(bn, M) for bn in (32, 64, 128, 256) for M in (bn // 2 - 1, bn // 2 + 1, bn, bn + 1)])
def test_halves_of_the_tokens(lords, bits, bn, M):
    lay = gen.make_integer_layer(130, 1152, 8, M, bits=bits, seed=bn + M)
    lords.lords_set_option("path", "umma")
    lords.lords_set_option("bn", str(bn))
    try:
        dl = DeviceLayer(lay)
        y32, _ = dl.forward()
        assert lords.lords_last_path() == "umma"
    finally:
        lords.lords_set_option("path", "auto")
        lords.lords_set_option("bn", "0")
    assert np.array_equal(y32.astype(np.float64), oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


@pytest.mark.parametrize("bits,m,n,r,M", [(4, 500, 8192, 20, 17), (3, 512, 8192, 48, 32), (4, 640, 1024, 8, 256), (2, 1100, 1536, 32, 140), (4, 390, 768, 16, 300)])
def test_estimates_choose(lords, bits, m, n, r, M):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + M)
    dl = DeviceLayer(lay)
    y32, ybf = dl.forward()
    assert lords.lords_last_path() == "umma"
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))


# m, n, r, M and the scratch beyond the fp16 activations: too little for the pieces that the preferred tile's or kernel's CTAs exchange
@pytest.mark.parametrize("m,n,r,M,room", [(2560, 1024, 32, 512, 1 << 20), (512, 8192, 48, 300, 700 << 10)])
def test_tight_scratch_keeps_the_path(lords, m, n, r, M, room):
    lay = gen.make_layer(m, n, r, M, bits=4, seed=m + M)
    dl = DeviceLayer(lay)
    lords.lords_init(0, M * n * 2 + room)
    try:
        y32, ybf = dl.forward()
        assert lords.lords_last_path() == "umma"
    finally:
        lords.lords_init(0, 0)
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, 4))
