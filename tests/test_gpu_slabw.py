"""The slab pass with compile-time warp-register lines (k_slab_warp): every length
of its list as rows and as columns, several slabs per block, both directions."""
import numpy as np
import pytest
import torch

import oracle
from paper_1904_10119_gb300 import fft3, synth
from tests.gpu_util import MAXABS_TOL, REL_L2_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,n1,n2,batch,direction", [
    (8, 128, 3, 2, fft3.FFT3_FORWARD), (128, 8, 1, 1, fft3.FFT3_INVERSE), (16, 96, 5, 1, fft3.FFT3_INVERSE),
    (96, 16, 2, 3, fft3.FFT3_FORWARD), (24, 80, 4, 1, fft3.FFT3_FORWARD), (80, 24, 4, 1, fft3.FFT3_INVERSE),
    (32, 64, 1000, 1, fft3.FFT3_FORWARD), (64, 32, 3, 1, fft3.FFT3_INVERSE), (40, 48, 2, 1, fft3.FFT3_FORWARD),
    (48, 40, 2, 1, fft3.FFT3_INVERSE), (128, 96, 2, 1, fft3.FFT3_FORWARD)])
def test_warp_slab_matches_oracle(n0, n1, n2, batch, direction):
    x = synth.uniform_c64((batch, n2, n1, n0), n0 + n1)
    xt = torch.from_numpy(x).cuda()
    out = torch.full_like(xt, complex(float("nan"), 0.0))
    plan = fft3.Plan(n0, n1, n2, batch, decomposition=fft3.FFT3_SLAB_PENCIL, direction=direction, slab_mode=1)
    first = plan.describe()["passes"][0]
    assert first["kind"] == "slab_smem" and first.get("compiled")
    plan.execute(xt, out)
    torch.cuda.synchronize()
    ref = oracle.fft3(x.ravel(), n0, n1, n2, batch, sign=direction)
    got = out.cpu().numpy()
    assert oracle.rel_l2(got, ref) <= REL_L2_TOL and oracle.max_abs_ratio(got, ref) <= MAXABS_TOL
    plan.close()
