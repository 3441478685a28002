"""Layers whose operands are held in 32 bits (include/lords.h): rows that are no multiples of the aligned kernels' steps, ranks
above 64, and one or two tokens of a small layer.  Precision, range, and infinities and NaNs as on the CUDA cores."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer, error_metrics

pytestmark = pytest.mark.gpu

# fp32 arithmetic: unit roundoff 6e-8, products of bf16 exact, sums of r and of n terms in many short chains; the CUDA-core path
# measures 1e-7 to 4e-7 on these sizes.  One operand rounded to fp16 gives 2e-4.
FP32_TOL = 1e-6

DIRECT = [
    # bits, m, n, r, M: what the direct kernel takes
    (4, 384, 1024, 32, 1),       # aligned, one and two tokens: stands in for the reassociated form
    (3, 256, 256, 17, 2),
    (4, 1000, 2730, 10, 37),     # ragged, several token groups
    (2, 333, 1028, 64, 9),
    (3, 130, 352, 33, 16),
    (4, 500, 1000, 128, 16),     # wide and ragged
    (4, 512, 640, 128, 5),       # wide, small
]
WIDE = [
    # ranks above 64: more than a million weights, up to 16 tokens; three and four sums of 32 ranks, with and without a rest
    (4, 1030, 1056, 65, 1),
    (3, 520, 2176, 96, 9),
    (2, 530, 2112, 97, 16),
    (4, 300, 4096, 128, 8),
]
DENSE = [
    # more than 128 tokens: every part of W^ through scratch; one and several token tiles, cut and whole tiles
    (4, 300, 1030, 9, 130),
    (3, 270, 2080, 100, 257),
    (2, 700, 516, 40, 300),
]
SHAPES = DIRECT + WIDE + DENSE


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_shutdown()


def _scaled(bits, words, factor):
    import torch
    return gen.bf16_bits(torch.from_numpy(gen.bf16_to_f32(words) * np.float32(factor)))


@pytest.mark.parametrize("bits,m,n,r,M", SHAPES)
@pytest.mark.parametrize("xs,bs", [(1.0, 1.0), (2.0**30, 2.0**-20), (2.0**-30, 2.0**-30), (2.0**-20, 2.0**40), (2.0**-129, 2.0**60)])
def test_precision_and_range(lords, bits, m, n, r, M, xs, bs):
    """x to 2^30 and factors from 2^-30 to 2^60, subnormal x: far outside fp16, with the precision of fp32."""
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r + M, mixed_sign=True)
    lay.x, lay.B = _scaled(bits, lay.x, xs), _scaled(bits, lay.B, bs)
    dl = DeviceLayer(lay)
    y32, _ = dl.forward()
    shape = (bits, m, n, r, M)
    assert (lords.lords_last_path() == "wide", lords.lords_last_path() == "dense") == (shape in WIDE, shape in DENSE)
    normwise, _ = error_metrics(y32, oracle.forward(lay.x, dl.packed_host, lay.B, lay.A, lay.codebook, bits))
    assert normwise <= FP32_TOL


@pytest.mark.parametrize("bits,m,n,r,M", SHAPES)
def test_infinities_and_nans_as_on_the_cuda_cores(lords, bits, m, n, r, M):
    """One infinite, one NaN activation, a row of infinite weights and one of NaNs.  Integer data: most weights have lower parts that
    are exactly zero, which must not meet an infinity.  Products that overflow a float are infinite as well."""
    lay = gen.make_integer_layer(m, n, r, M, bits=bits, seed=m + M)
    x, B = lay.x.copy(), lay.B.copy()
    if M > 1:                        # one token stays finite
        x[0, n // 2] = 0x7F80
    if M > 2:
        x[1, 1] = 0xFF80
        x[2, n - 1] = 0x7FC0
    B[m // 2, 0] = 0x7F80
    B[m - 1, r - 1] = 0x7FC0
    B[0, :] = 0x7F00                 # 1.7e38: S overflows
    lay.x, lay.B = x, B
    dl = DeviceLayer(lay)
    got, _ = dl.forward()
    lords.lords_set_option("path", "simt")
    try:
        want, _ = dl.forward()
    finally:
        lords.lords_set_option("path", "auto")
    assert np.array_equal(got, want, equal_nan=True)
    assert np.isnan(want).any() and np.isfinite(want).any() and (M == 1 or np.isinf(want).any())
