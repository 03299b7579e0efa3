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


@pytest.mark.parametrize("shape,decomposition,dtype", [
    ((64, 64, 64), fft3.FFT3_PENCIL3, fft3.FFT3_C64_FP32), ((40, 512, 48), fft3.FFT3_AUTO, fft3.FFT3_C64_FP32),
    ((32, 32, 16), fft3.FFT3_SLAB_PENCIL, fft3.FFT3_C64_FP32), ((48, 128, 64), fft3.FFT3_VOLUMETRIC, fft3.FFT3_C64_FP32),
    ((60, 45, 50), fft3.FFT3_AUTO, fft3.FFT3_C64_FP32), ((60, 64, 54), fft3.FFT3_AUTO, fft3.FFT3_C128_FP64)])
def test_overlapping_passes_under_capture_and_back_to_back(shape, decomposition, dtype):
    """A captured execution behind a writer of its input, replayed on changing inputs;
    executions back to back into one output, the last of them with other values."""
    c = torch.complex128 if dtype == fft3.FFT3_C128_FP64 else torch.complex64
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    xs = [torch.randn(*shape[::-1], dtype=c, device="cuda", generator=g) for _ in range(3)]
    plan = fft3.Plan(*shape, decomposition=decomposition, dtype=dtype)
    alone = []
    for x in xs:
        out = torch.empty_like(x)
        plan.execute(x, out)
        torch.cuda.synchronize()
        alone.append(out)
    ref = torch.fft.fftn(xs[0].to(torch.complex128))
    assert (alone[0] - ref).norm() <= 1e-5 * ref.norm()
    s = torch.cuda.Stream()
    src, x, out = xs[0].clone(), torch.empty_like(xs[0]), torch.empty_like(xs[0])
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        x.copy_(src)
        plan.execute(x, out)
        x.zero_()  # a later writer of the input waits for the passes
    for k in (1, 2, 0):
        src.copy_(xs[k])
        out.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, alone[k])
    with torch.cuda.stream(s):
        for _ in range(20):
            plan.execute(xs[1], out)
            plan.execute(xs[2], out)
    s.synchronize()
    assert torch.equal(out, alone[2])
    assert plan.check() == 0, fft3.last_error()
    plan.close()
