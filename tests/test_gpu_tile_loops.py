"""Persistent tile loops past their first tile: more tiles than resident blocks
several times over, the last one ragged, so that a block reuses its shared buffer
and its per-line words; and the ragged last tile of volumetric cluster pairs."""
import pytest
import torch

from paper_1904_10119_gb300 import fft3
from tests.gpu_util import assert_parity, run_plan

pytestmark = pytest.mark.gpu


def _pass(x, strided, dtype):
    """The lines x[b, j, c] along j, as strided columns, or x[b, c, j] as contiguous lines:
    (result of that one pass, its description)."""
    b, n1, n0 = x.shape
    plan = fft3.Plan(n0, n1, 1, b, dtype=dtype, decomposition=fft3.FFT3_PENCIL3)
    k = 1 if strided else 0
    out = x.clone()
    fft3.fft3_plan_execute_pass(plan.handle, k, x.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    assert plan.check() == 0, fft3.last_error()
    desc = plan.describe()["passes"][k]
    plan.close()
    return out, desc


def _randn(shape, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, dtype=torch.complex128 if dtype == fft3.FFT3_C128_FP64 else torch.complex64, device="cuda",
                       generator=g)


@pytest.mark.parametrize("dtype", [fft3.FFT3_C64_FP32, fft3.FFT3_C128_FP64])
@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("n", [15, 60, 125, 240, 375, 500, 64, 512, 1024])
def test_many_tiles_per_block(n, strided, dtype):
    # columns: 20 a tile row, the second tile of 16 (complex64) or the third of 8 ragged; lines: 3 x an odd
    # number of them in one run
    b = (1 << 25) // (20 * n) + 1 if strided else (1 << 25) // (3 * n) | 1
    x = _randn((b, n, 20) if strided else (b, 3, n), dtype, n)
    out, p = _pass(x, strided, dtype)
    assert p["tiles"] > 3 * 152 * min(32, 2048 // p["threads"], (227 << 10) // p["smem"])
    ref = torch.fft.fft(x.to(torch.complex128), dim=1 if strided else 2)
    err = (out - ref).norm(dim=1 if strided else 2) / ref.norm(dim=1 if strided else 2)
    # FP32: about 40 roundings of at most 2^-24 of a value, with random signs; FP64: both within 4e-16
    assert err.max() <= (1e-15 if dtype == fft3.FFT3_C128_FP64 else 40 ** 0.5 * 2.0 ** -24), float(err.max())


@pytest.mark.parametrize("strided", [False, True])
@pytest.mark.parametrize("n", [60, 256, 375, 512, 1500])
def test_fp64_lines_between_fixed_point_tiles(n, strided):
    """Every 97th line goes to the FP64 stages (an infinity; imaginary parts far below
    the real ones), the tiles before and after it in the same block do not."""
    b = (1 << 24) // (20 * n) + 1
    x = _randn((b * 20, n), fft3.FFT3_C128_FP64, n)
    x[::97] = torch.complex(x[::97].real, 1e-9 * x[::97].imag)
    x[5 * 97, n // 2] = float("inf")
    keep = torch.ones(b * 20, dtype=torch.bool, device="cuda")
    keep[5 * 97] = False
    xt = x.view(b, 20, n)
    out, _ = _pass(xt.transpose(1, 2).contiguous() if strided else xt, strided, fft3.FFT3_C128_FP64)
    got = (out.transpose(1, 2) if strided else out).reshape(b * 20, n)
    assert not torch.isfinite(torch.view_as_real(got[5 * 97])).all(dim=1).any()
    ref = torch.fft.fft(x[keep], dim=1)
    err = (got[keep] - ref).norm(dim=1) / ref.norm(dim=1)
    assert err.max() <= 1e-15, float(err.max())  # both transforms in FP64, each within 4e-16


@pytest.mark.parametrize("direction", [fft3.FFT3_FORWARD, fft3.FFT3_INVERSE])
@pytest.mark.parametrize("shape", [(36, 128, 256), (6, 256, 128), (50, 64, 64), (80, 512, 64), (2, 64, 256), (90, 256, 9)])
def test_volumetric_pairs_with_a_ragged_tile(shape, direction):
    """Lines of 64 to 512 points over a cluster pair, y and z, the last tile of 32 columns ragged."""
    x, got, plan = run_plan(shape, 1, fft3.FFT3_VOLUMETRIC, direction)
    pairs = [p for p in plan.describe()["passes"] if p.get("p") == 2 and p["kind"] == "line_strided_stream"]
    assert pairs and any(p["geom"]["C"] % 32 for p in pairs)
    assert_parity(x, got, shape, 1, direction)
    plan.close()
