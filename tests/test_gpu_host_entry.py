"""The host-buffer entry where the way x travels changes: launch parameters up to 30 KiB (three sizes of parameter
block), a fetch kernel above that and during stream capture."""
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


@pytest.mark.parametrize("M", [1, 2, 4, 5, 15, 16])      # 2, 4, 8 KiB of x (block edges), 10, 30 and 32 KiB
def test_x_by_parameters_by_fetch_and_in_a_graph(lords, M):
    import torch
    lay = gen.make_layer(192, 1024, 8, M, bits=4, seed=70 + M)
    dl = DeviceLayer(lay)
    _, want = dl.forward()
    args = (dl.q, dl.B, dl.A, lay.codebook, 4, M, lay.m, lay.n, lay.r)
    xh = torch.from_numpy(lay.x.view(np.int16)).pin_memory()
    yh = torch.full((M, lay.m), 0x7FC0, dtype=torch.int16).pin_memory()
    lords.lords_linear_forward_host(xh, *args, yh)
    torch.cuda.synchronize()
    assert np.array_equal(yh.numpy().view(np.uint16), want)
    # a captured call reads the host buffer at every replay
    xg = torch.zeros_like(xh).pin_memory()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        lords.lords_linear_forward_host(xg, *args, yh)
    xg.copy_(xh)
    yh.fill_(0x7FC0)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(yh.numpy().view(np.uint16), want)
    assert lords.lords_poll_status() == 0


@pytest.mark.parametrize("m,n,M", [(193, 258, 1), (195, 514, 3), (250, 5122, 3), (97, 6002, 7)])       # rows that are no 16-byte multiples; the last two: by fetch
def test_ragged_lengths(lords, m, n, M):
    import torch
    lay = gen.make_layer(m, n, 8, M, bits=4, seed=m)
    dl = DeviceLayer(lay)
    _, want = dl.forward()
    xh = torch.from_numpy(lay.x.view(np.int16)).pin_memory()
    room = torch.full((M * m + 8,), 0x7FC0, dtype=torch.int16).pin_memory()
    yh = room[:M * m].view(M, m)
    lords.lords_linear_forward_host(xh, dl.q, dl.B, dl.A, lay.codebook, 4, M, lay.m, lay.n, lay.r, yh)
    torch.cuda.synchronize()
    assert np.array_equal(yh.numpy().view(np.uint16), want)
    assert bool((room[M * m:] == 0x7FC0).all())
    assert lords.lords_poll_status() == 0
