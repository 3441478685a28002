"""Weights written on the stream right before a call: layers off the aligned kernels' grid and ranks above 64 need no synchronisation
in between (include/lords.h)."""
import numpy as np
import pytest

from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_shutdown()


@pytest.mark.parametrize("bits,m,n,r,M,path", [(4, 1000, 2730, 10, 37, "direct"), (3, 1100, 1056, 33, 5, "direct"), (4, 1024, 2048, 128, 16, "wide"),
                                               (4, 1030, 1056, 65, 3, "wide"), (2, 700, 1028, 40, 300, "dense")])
def test_weights_written_just_before_the_call(lords, bits, m, n, r, M, path):
    import torch
    layers = [DeviceLayer(gen.make_layer(m, n, r, M, bits=bits, seed=s, mixed_sign=True)) for s in (1, 2)]
    want = []
    for L in layers:                                  # with a synchronisation between the upload and the call
        torch.cuda.synchronize()
        want.append(L.forward()[0])
    assert lords.lords_last_path() == path
    q, B, A = (torch.empty_like(t) for t in (layers[0].q, layers[0].B, layers[0].A))
    got = [torch.empty(M, m, dtype=torch.float32, device="cuda") for _ in range(20)]
    for k, y in enumerate(got):                       # weights and call by turns, all in flight
        L = layers[k & 1]
        q.copy_(L.q)
        B.copy_(L.B)
        A.copy_(L.A)
        lords.lords_linear_forward_f32(L.x, q, B, A, L.lay.codebook, bits, M, m, n, r, y)
    torch.cuda.synchronize()
    assert lords.lords_poll_status() == 0
    for k, y in enumerate(got):
        assert np.array_equal(y.cpu().numpy(), want[k & 1])
