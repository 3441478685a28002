"""Calls behind a launch that lets its dependents begin early and then works longer than the 50 ms that a device-side wait may take: no
wait of theirs may run while that launch does.  The launch is the direct kernel on one CTA, with one column split for millions of columns."""
import numpy as np
import pytest

from paper_2601_22716_b200 import inputs as gen
from _util import DeviceLayer

pytestmark = pytest.mark.gpu

LONG = (8, 64 * 160000, 4, 16)      # m, n, r, M


@pytest.fixture(scope="module")
def lords():
    from paper_2601_22716_b200 import binding
    binding.lords_init(0, 0)
    yield binding
    binding.lords_set_option("path", "auto")
    binding.lords_set_option("splitk", "0")
    binding.lords_shutdown()


@pytest.fixture(scope="module")
def long_launch(lords):
    import torch
    m, n, r, M = LONG
    q = torch.zeros(m, n // 2, dtype=torch.uint8, device="cuda")
    B, A, x, y = (torch.zeros(s, dtype=torch.bfloat16, device="cuda") for s in ((m, r), (r, n), (M, n), (M, m)))
    book = gen.nf_codebook(4)
    torch.cuda.synchronize()

    def run():
        lords.lords_set_option("path", "direct")
        lords.lords_set_option("splitk", "1")
        lords.lords_linear_forward_bits(x, q, B, A, book, 4, M, m, n, r, y)
        lords.lords_set_option("path", "auto")
        lords.lords_set_option("splitk", "0")

    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    run()
    start.record()
    run()
    end.record()
    torch.cuda.synchronize()
    assert start.elapsed_time(end) > 60.0, "the launch does not outlast the waits' limit"
    return run


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("kernel", ["blockscale16", "decode16"])
def test_no_wait_runs_out_behind_a_long_launch(lords, long_launch, kernel, bits):
    import torch
    m, n, blk, M = 128, 2048, 128, 5                  # 16 steps for one CTA: more than any ring holds
    lay, s = gen.make_blockwise_layer(m, n, blk, M, bits=bits, seed=bits)
    dl = DeviceLayer(lay)
    scales = torch.from_numpy(s.view(np.int16)).to("cuda")

    def call(y):
        lords.lords_set_option("splitk", "1")
        if kernel == "blockscale16":
            lords.lords_blockscale_forward(dl.x, dl.q, scales, lay.codebook, bits, blk, M, m, n, y, f32=True)
        else:
            lords.lords_set_option("path", kernel)
            lords.lords_linear_forward_f32(dl.x, dl.q, dl.B, dl.A, lay.codebook, bits, M, m, n, lay.r, y)
            lords.lords_set_option("path", "auto")
        lords.lords_set_option("splitk", "0")
        assert lords.lords_last_path() == kernel

    want, got = (torch.full((M, m), float("nan"), device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    call(want)
    torch.cuda.synchronize()
    long_launch()
    call(got)
    assert lords.lords_poll_status() == 0
    assert torch.equal(got, want)
