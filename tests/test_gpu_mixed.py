"""Compile-time mixed-radix line passes (lengths 2^a 3^b 5^c up to 1024 that are
not powers of two) against the FP64 oracle: every plan, contiguous and strided
lines, ragged tiles, both directions."""
import numpy as np
import pytest
import torch

import oracle
from paper_1904_10119_gb300 import fft3, synth

pytestmark = pytest.mark.gpu

LENGTHS = [n for n in synth.smooth_sizes(3, 1024) if n & (n - 1)]
# A value passes at most ten radix-2 levels' worth of additions and four twiddle
# products, each rounding by at most 2^-24 of the value's size with random signs:
# rms sqrt(2 * 10 + 3 * 4) * 2^-24 = 3.4e-7; twice that for the butterflies'
# constants, themselves rounded to 2^-24.
TOL = 7e-7


@pytest.mark.parametrize("n", LENGTHS)
def test_mixed_plan_matches_oracle(n):
    for shape, batch, direction, dim in (((n, 3, 1), 2, fft3.FFT3_FORWARD, 0), ((27, n, 2), 1, fft3.FFT3_INVERSE, 1)):
        x = synth.uniform_c64((batch, shape[2], shape[1], shape[0]), n)
        xt = torch.from_numpy(x).cuda()
        out = torch.full_like(xt, complex(float("nan"), float("nan")))
        plan = fft3.Plan(*shape, batch, decomposition=fft3.FFT3_PENCIL3, direction=direction)
        assert any(p["dim"] == dim and p.get("compiled") and p["line"]["n"] == n for p in plan.describe()["passes"])
        plan.execute(xt, out)
        torch.cuda.synchronize()
        ref = oracle.fft3(x.ravel(), *shape, batch, sign=direction)
        assert oracle.rel_l2(out.cpu().numpy(), ref) <= TOL
        plan.close()
