"""Transposition of packed codes at the edges of its 64 x 128 tiles and of 32-code words, against the oracle's reader of the layout."""
import numpy as np
import pytest

import oracle
from test_gpu_quantize import lords  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,m,n", [(4, 2, 2), (4, 64, 128), (4, 66, 130), (4, 4098, 62), (4, 96, 392), (3, 32, 32), (3, 96, 160), (3, 64, 128), (3, 1056, 2080),
                                      (2, 4, 4), (2, 68, 132), (2, 128, 256), (2, 32, 100), (2, 1000, 1004)])
def test_transpose_codes(lords, bits, m, n):  # noqa: F811
    import torch
    rng = np.random.default_rng(m * 7 + n)
    q = rng.integers(0, 256, size=lords.lords_packed_bytes(m, n, bits), dtype=np.uint8)
    out = torch.full((q.size,), 0xA5, dtype=torch.uint8, device="cuda:0")
    lords.lords_transpose_codes(torch.from_numpy(q).to("cuda:0"), bits, m, n, out)
    torch.cuda.synchronize()
    got = oracle.unpack_codes(out.cpu().numpy().reshape(n, -1), n, m, bits)
    assert np.array_equal(got, oracle.unpack_codes(q.reshape(m, -1), m, n, bits).T)
