"""The scale-MMA kernels.  Where the two CTAs of a cluster share a tile's columns and exchange halves of its tokens: every token tile, token
counts around its half and its whole, ragged rows; sums of small integers are exact in any order.  And what the dispatch chooses by its
estimates: the direct kernel and the one on CTA pairs from 17 tokens on, token tiles, and other ones where scratch is short."""
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


KERNELS = {"direct": ("direct", "0"), "pair": ("pair", "0"), 32: ("umma", "32"), 64: ("umma", "64"), 128: ("umma", "128"), 256: ("umma", "256")}


# What tells the kernels apart: the number of launches, and the fp32 sums' last bits, which depend on how a kernel or tile splits the columns.  Token
# tiles that split them alike (or not at all) have the same bits: `chosen` are those that the call may have taken.
@pytest.mark.parametrize("bits,m,n,r,M,chosen", [
    (4, 500, 8192, 20, 17, {"direct"}),
    (3, 512, 8192, 48, 32, {"direct"}),
    (3, 2048, 8192, 48, 20, {"pair"}),
    (4, 4096, 14336, 32, 32, {"pair"}),
    (4, 2600, 1024, 40, 500, {256}),
    (2, 4096, 1024, 16, 130, {128, 256}),
    (4, 1024, 4096, 32, 512, {64, 128, 256}),
    (4, 390, 768, 16, 300, {32, 64, 128, 256}),
])
def test_estimates_choose(lords, bits, m, n, r, M, chosen):
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + M)
    dl = DeviceLayer(lay)
    y32, ybf = dl.forward()
    launches = lords.lords_last_launch_count()
    assert lords.lords_last_path() == "umma"
    check_against_oracle(y32, ybf, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))
    same = set()
    try:
        for kernel, (path, bn) in KERNELS.items():
            if kernel == "direct" and M > 128:
                continue
            lords.lords_set_option("path", path)
            lords.lords_set_option("bn", bn)
            if np.array_equal(dl.forward()[0], y32) and lords.lords_last_launch_count() == launches:
                same.add(kernel)
    finally:
        lords.lords_set_option("path", "auto")
        lords.lords_set_option("bn", "0")
    assert same == chosen


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
