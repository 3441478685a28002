"""The quantisation step on the tensor-core path beyond 64 ranks and off the 64-column grid (padded copies, partial code
groups), and with ascending tables whose midpoints lie too close together for buckets."""
import dataclasses

import numpy as np
import pytest

from paper_2601_22716_b200 import inputs as gen
from test_gpu_quantize import _check_codes, _quantize_on_gpu, lords  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,m,n,r", [(4, 1024, 2048, 128), (4, 1200, 1110, 33), (4, 1201, 1096, 72), (3, 1400, 992, 65), (2, 1536, 1028, 100),
                                        (2, 2600, 516, 7)])
def test_quantize_ragged_rows_and_large_ranks(lords, bits, m, n, r):  # noqa: F811
    lay = gen.make_layer(m, n, r, 1, bits=bits, seed=m + n)
    Wb = gen.make_weight(m, n, seed=m, sigma=0.05 * (r / 32.0))
    Q, used = _quantize_on_gpu(lords, Wb, lay)
    assert used == "quantize"
    _check_codes(lords, Q, Wb, lay)


@pytest.mark.parametrize("bits", [4, 3, 2])
@pytest.mark.parametrize("gap", [1e-3, 3e-7])
def test_quantize_with_crowded_levels(lords, bits, gap):  # noqa: F811
    lay = gen.make_layer(200, 320, 16, 1, bits=bits, seed=bits, mixed_sign=True)
    cb = lay.codebook.copy()
    cb[2] = cb[1] + np.float32(gap)                  # two midpoints in one bucket
    lay = dataclasses.replace(lay, codebook=cb)
    Wb = gen.make_weight(200, 320, seed=bits, sigma=0.025)
    Q, used = _quantize_on_gpu(lords, Wb, lay)
    assert used == "quantize"
    from test_gpu_quantize import oracle
    packed = Q.cpu().numpy().reshape(200, -1)
    got = oracle.unpack_codes(packed, 200, 320, bits)
    want, _, g, mag = oracle.quantize(Wb, lay.B, lay.A, lay.codebook, bits, details=True)
    clear = g > 8.0 * (lay.r + 2) * 2.0 ** -24 * mag
    assert np.array_equal(got[clear], want[clear])
