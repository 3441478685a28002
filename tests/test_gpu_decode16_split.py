"""The 16-token kernel with its columns split over a cluster whose CTAs add up the tokens between them: fewer tokens than CTAs, as many,
and counts that leave the last of them with fewer.  Sums of small integers are exact in any order."""
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
    binding.lords_set_option("splitk", "0")
    binding.lords_shutdown()


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("split", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("M", [1, 3, 7, 8, 13, 16])
def test_tokens_over_the_cluster(lords, bits, split, M):
    lay = gen.make_integer_layer(130, 1280, 8, M, bits=bits, seed=16 * split + M)
    lords.lords_set_option("path", "decode16")
    lords.lords_set_option("splitk", str(split))
    try:
        dl = DeviceLayer(lay)
        y32, _ = dl.forward()
        assert lords.lords_last_path() == "decode16"
    finally:
        lords.lords_set_option("path", "auto")
        lords.lords_set_option("splitk", "0")
    assert np.array_equal(y32.astype(np.float64), oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))
