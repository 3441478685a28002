"""Factor and QAT gradients where a CTA's run of tiles crosses from one row block into the next, including runs of several row
blocks of one column tile each, with and without room for two accumulators of the folds, and ranks whose B tile is built
element by element; and where rows that are no 16-byte multiples are copied first."""
import numpy as np
import pytest

import oracle
from paper_2601_22716_b200 import inputs as gen
from _util import error_metrics
from test_gpu_quantize import lords  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,m,n,r,M", [(4, 2048, 2560, 32, 72), (4, 1920, 2304, 64, 40), (4, 19200, 128, 16, 33), (3, 1664, 3200, 24, 64),
                                          (2, 2304, 1664, 128, 20), (4, 1408, 2816, 7, 48), (4, 38400, 64, 40, 16),
                                          # rows of g, x, A, W or the codes that begin anywhere
                                          (4, 1030, 2050, 32, 65), (4, 258, 16386, 20, 40), (2, 1028, 1988, 9, 50), (2, 136, 1096, 24, 20), (3, 1024, 2080, 33, 129)])
def test_gradients_over_several_row_blocks(lords, bits, m, n, r, M):  # noqa: F811
    import torch
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n + r)
    packed = oracle.pack_codes(lay.codes, bits)
    g = gen.bf16_bits(torch.randn(M, m, generator=torch.Generator().manual_seed(r)))
    Wb = gen.make_weight(m, n, seed=r)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).to("cuda:0")  # noqa: E731
    q = torch.from_numpy(packed).to("cuda:0")
    new = lambda *shape: torch.full(shape, float("nan"), dtype=torch.float32, device="cuda:0")  # noqa: E731
    dB, dA, dW, dBq, dAq = new(m, r), new(r, n), new(m, n), new(m, r), new(r, n)
    args = (q, dev(lay.B), dev(lay.A), lay.codebook, bits, M, m, n, r)
    gd, xd = dev(g), dev(lay.x)
    lords.lords_linear_backward_factors(gd, xd, *args, dB, dA)
    assert lords.lords_last_path() == "backward_tensor"
    lords.lords_linear_backward_qat(gd, xd, dev(Wb), *args, dW, dBq, dAq)
    assert lords.lords_last_path() == "backward_qat_tensor"
    torch.cuda.synchronize()
    assert lords.lords_poll_status() == 0
    _, dB64, dA64 = oracle.backward(g, lay.x, packed, lay.B, lay.A, lay.codebook, bits)
    dW64, dBq64, dAq64 = oracle.backward_qat(g, lay.x, Wb, packed, lay.B, lay.A, lay.codebook, bits)
    for name, got, want in (("dB", dB, dB64), ("dA", dA, dA64), ("dW", dW, dW64), ("dBq", dBq, dBq64), ("dAq", dAq, dAq64)):
        nw, el = error_metrics(got.cpu().numpy(), want)
        assert nw <= 1e-4 and el <= 1e-3, (name, nw, el)


@pytest.mark.parametrize("bits,m,n,r,M,tol", [(4, 640, 4096, 32, 512, 4.5e-7), (4, 512, 8190, 32, 64, 3e-7), (4, 1026, 1030, 10, 1000, 3e-7), (4, 260, 4100, 100, 300, 3e-7)])
def test_gradients_keep_the_precision_of_fp32_sums(lords, bits, m, n, r, M, tol):  # noqa: F811
    """The tensor cores cut sums off (about 1.5e-8 an MMA of 16 tokens, 1e-7 a fold of 128 columns), so long sums are taken apart: at most half
    of the tokens on a layer with 16-byte rows, 64 tokens otherwise (those layers' sums were rounded to nearest before), one tile in
    the folds.  In one piece each they are off by 1.2e-6 to 5e-6.  QAT's factors carry the quotient's rounding as well."""
    import torch
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + r)
    packed = oracle.pack_codes(lay.codes, bits)
    g = gen.bf16_bits(torch.randn(M, m, generator=torch.Generator().manual_seed(r)))
    Wb = gen.make_weight(m, n, seed=r)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).to("cuda:0")  # noqa: E731
    new = lambda *shape: torch.full(shape, float("nan"), dtype=torch.float32, device="cuda:0")  # noqa: E731
    dB, dA, dW, dBq, dAq = new(m, r), new(r, n), new(m, n), new(m, r), new(r, n)
    args = (torch.from_numpy(packed).to("cuda:0"), dev(lay.B), dev(lay.A), lay.codebook, bits, M, m, n, r)
    gd, xd = dev(g), dev(lay.x)
    lords.lords_linear_backward_factors(gd, xd, *args, dB, dA)
    lords.lords_linear_backward_qat(gd, xd, dev(Wb), *args, dW, dBq, dAq)
    assert lords.lords_last_path() == "backward_qat_tensor"
    torch.cuda.synchronize()
    assert lords.lords_poll_status() == 0
    _, dB64, dA64 = oracle.backward(g, lay.x, packed, lay.B, lay.A, lay.codebook, bits)
    dW64, dBq64, dAq64 = oracle.backward_qat(g, lay.x, Wb, packed, lay.B, lay.A, lay.codebook, bits)
    for name, got, want, bound in (("dB", dB, dB64, tol), ("dA", dA, dA64, tol), ("dW", dW, dW64, tol), ("dBq", dBq, dBq64, 2 * tol), ("dAq", dAq, dAq64, 2 * tol)):
        nw, _ = error_metrics(got.cpu().numpy(), want)
        assert nw <= bound, (name, nw)
