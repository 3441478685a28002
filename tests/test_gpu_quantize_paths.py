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


@pytest.mark.parametrize("bits,m,n,r,mixed", [(4, 5472, 10524, 6, False), (3, 4800, 3392, 91, False), (4, 1200, 1280, 128, True), (2, 3000, 1412, 30, True)])
def test_close_decisions_are_exact(lords, bits, m, n, r, mixed):  # noqa: F811
    """Ragged rows and ranks above 64: every code is that of the oracle, also where the two nearest levels are equally far to within
    fp32 rounding (of the first case's weights some ten are)."""
    from test_gpu_quantize import oracle
    lay = gen.make_layer(m, n, r, 1, bits=bits, seed=r, mixed_sign=mixed)
    Wb = gen.make_weight(m, n, seed=m, sigma=0.05 * (r / 32.0))
    Wb[::7, ::5] = 0x8000                             # negative zeros: ties of a table that is symmetric around zero
    Wb[1, 2], Wb[3, 4], Wb[5, 6] = 0x7F80, 0xFF80, 0x7FC0
    lay.B[9, :] = 0                                   # S = 0: every level equally good
    Q, used = _quantize_on_gpu(lords, Wb, lay)
    assert used == "quantize"
    got = oracle.unpack_codes(Q.cpu().numpy().reshape(m, -1), m, n, bits)
    assert np.array_equal(got, oracle.quantize(Wb, lay.B, lay.A, lay.codebook, bits))
    assert not got[9].any()


def test_exact_ties_take_the_lower_code(lords):  # noqa: F811
    """Integer factors and levels, weights on the midpoints: nothing is rounded anywhere."""
    import torch
    from test_gpu_quantize import oracle
    m, n, r = 1300, 1050, 9
    lay = gen.make_integer_layer(m, n, r, 1, bits=4, seed=9)
    S = gen.bf16_to_f32(lay.B) @ gen.bf16_to_f32(lay.A)
    W = S * (lay.codebook[lay.codes] + np.float32(0.5))
    Wb = gen.bf16_bits(torch.from_numpy(W.astype(np.float32)))
    Q, used = _quantize_on_gpu(lords, Wb, lay)
    assert used == "quantize"
    assert np.array_equal(oracle.unpack_codes(Q.cpu().numpy().reshape(m, -1), m, n, 4), np.minimum(lay.codes, 15))
