"""FFT3_AUTO without room for the blocked intermediate's workspace plans the natural
order instead of failing; a blocked plan that was asked for still reports it."""
import pytest
import torch

from paper_1904_10119_gb300 import fft3, synth
from tests.gpu_util import assert_parity

pytestmark = pytest.mark.gpu


def test_automatic_plan_falls_back_to_natural_order():
    shape = (64, 512, 1024)  # 256 MiB, where FFT3_AUTO takes the blocked intermediate
    n0, n1, n2 = shape
    x = synth.uniform_c64((1, n2, n1, n0), 5)
    xt = torch.from_numpy(x).cuda()
    out = torch.empty_like(xt)
    for decomposition in (fft3.FFT3_AUTO, fft3.FFT3_PENCIL3):  # loads every kernel used below
        plan = fft3.Plan(*shape, decomposition=decomposition)
        assert (plan.describe()["workspace_bytes"] > 0) == (decomposition == fft3.FFT3_AUTO)
        plan.execute(xt, out)
        torch.cuda.synchronize()
        plan.close()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(fft3.Fft3Error, match="OOM"):
            fft3.Plan(*shape, decomposition=fft3.FFT3_PENCIL3, variant=fft3.FFT3_PPP_BLOCKED)
        plan = fft3.Plan(*shape, decomposition=fft3.FFT3_AUTO)
        assert plan.describe()["workspace_bytes"] == 0
        plan.execute(xt, out)
        torch.cuda.synchronize()
        assert plan.check() == 0, fft3.last_error()
        plan.close()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert_parity(x, out.cpu().numpy(), shape)
