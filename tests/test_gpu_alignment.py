"""Buffers aligned to 8 bytes only (a tensor that starts one value into an
allocation): plans without TMA run on them, among them those whose streamed
passes took the place of kernels with plain loads (volumetric splits of 64 to 256
points, y lines of slabs that fit a block's shared memory); plans that stream
512- and 1024-point lines by TMA refuse them."""
import numpy as np
import pytest
import torch

from paper_1904_10119_gb300 import fft3, synth
from tests.gpu_util import assert_parity

pytestmark = pytest.mark.gpu


def _run(shape, decomposition, direction=fft3.FFT3_FORWARD, **opts):
    n0, n1, n2 = shape
    x = synth.uniform_c64((1, n2, n1, n0), 3)
    buf = torch.empty(2 * x.size + 2, dtype=torch.complex64, device="cuda")
    off = 1 if buf.data_ptr() % 16 == 0 else 0
    xt, out = (buf[off + k * (x.size + x.size % 2):][:x.size].view(x.shape) for k in range(2))
    xt.copy_(torch.from_numpy(x))
    assert xt.data_ptr() % 16 == 8 and out.data_ptr() % 16 == 8
    plan = fft3.Plan(n0, n1, n2, decomposition=decomposition, direction=direction, **opts)
    kinds = [p["kind"] for p in plan.describe()["passes"]]
    plan.execute(xt, out)
    torch.cuda.synchronize()
    assert plan.check() == 0, fft3.last_error()
    assert_parity(x, out.cpu().numpy(), shape, 1, direction)
    plan.close()
    return kinds


@pytest.mark.parametrize("shape,decomposition,opts", [
    ((64, 64, 64), fft3.FFT3_VOLUMETRIC, {}), ((40, 128, 256), fft3.FFT3_VOLUMETRIC, {}),
    ((6, 256, 128), fft3.FFT3_VOLUMETRIC, {"mesh": (0, 2, 2)}), ((16, 512, 20), fft3.FFT3_AUTO, {}),
    ((8, 1024, 9), fft3.FFT3_AUTO, {}), ((24, 512, 30), fft3.FFT3_SLAB_PENCIL, {})])
@pytest.mark.parametrize("direction", [fft3.FFT3_FORWARD, fft3.FFT3_INVERSE])
def test_streamed_passes_keep_eight_byte_buffers(shape, decomposition, opts, direction):
    assert any("stream" in k for k in _run(shape, decomposition, direction, **opts))


def test_plain_and_streamed_plans_as_before():
    _run((60, 45, 50), fft3.FFT3_AUTO)
    _run((32, 64, 8), fft3.FFT3_SLAB_PENCIL, slab_mode=1)
    for shape, decomposition in (((16, 512, 20), fft3.FFT3_PENCIL3), ((64, 512, 512), fft3.FFT3_VOLUMETRIC)):
        with pytest.raises(fft3.Fft3Error, match="16-byte aligned"):
            _run(shape, decomposition)
