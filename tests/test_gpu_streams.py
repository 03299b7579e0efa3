"""Which stream Plan.execute runs on, and that a plan's overlapping launches keep
its order there."""
import pytest
import torch

from paper_1904_10119_gb300 import fft3, synth
from tests.gpu_util import assert_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("raw", [True, False])
def test_execute_takes_the_current_stream(raw, monkeypatch):
    """The current stream, with or without torch's call for its raw handle."""
    if not raw:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    shape = (48, 60, 64)
    x = synth.uniform_c64((1, *shape[::-1]), 1)
    xt, out = torch.zeros(x.shape, dtype=torch.complex64, device="cuda"), torch.zeros(x.shape, dtype=torch.complex64, device="cuda")
    src = torch.from_numpy(x).pin_memory()
    plan = fft3.Plan(*shape)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)  # the stream is busy when the copy and the transform are queued
        xt.copy_(src, non_blocking=True)
        plan.execute(xt, out)
    s.synchronize()
    assert_parity(x, out.cpu().numpy(), shape)
    plan.close()
