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


@pytest.mark.parametrize("bits,m,n,r,M", [(4, 1024, 4096, 32, 1), (4, 4096, 2048, 20, 2), (3, 1300, 1152, 48, 1), (2, 3000, 1088, 16, 2), (4, 16500, 32, 8, 1),
                                          (4, 140, 4064, 64, 1)])
def test_x_carried_by_the_decode_launch(lords, bits, m, n, r, M):
    """One or two tokens, up to 8 KiB: x travels with the decode launch, back to back calls keep their order."""
    import torch
    lay = gen.make_layer(m, n, r, M, bits=bits, seed=m + n)
    dl = DeviceLayer(lay)
    _, want = dl.forward()
    args = (dl.q, dl.B, dl.A, lay.codebook, bits, M, lay.m, lay.n, lay.r)
    xh = torch.from_numpy(lay.x.view(np.int16)).pin_memory()
    zero = torch.zeros_like(xh).pin_memory()
    yh = torch.full((M, lay.m), 0x7FC0, dtype=torch.int16).pin_memory()
    for _ in range(20):                                   # the last call's y stays
        lords.lords_linear_forward_host(zero, *args, yh)
        lords.lords_linear_forward_host(xh, *args, yh)
    assert lords.lords_last_path() == "decode" and lords.lords_last_launch_count() == 1
    torch.cuda.synchronize()
    assert np.array_equal(yh.numpy().view(np.uint16), want)
    assert lords.lords_poll_status() == 0
