"""The scale-MMA kernel where the two CTAs of a cluster share a tile's columns and exchange halves of its tokens: every token tile, token
counts around its half and its whole, ragged rows.  Sums of small integers are exact in any order."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer

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
