"""complex128 passes in 64-bit block fixed point: accuracy against an extended
precision reference, the inputs that make a fixed point hard (spikes, values
over 24 decades, lines of very different size), and the lines it leaves to FP64
(infinities, NaN, subnormals, the ends of the exponent range)."""
import numpy as np
import pytest
import torch

from paper_1904_10119_gb300 import fft3, synth

pytestmark = pytest.mark.gpu


def _passes(z, **opts):
    """The rows of z as contiguous lines (pass 0 of n x lines) and as strided
    columns (pass 1 of lines x n, in place on the output), one pass alone."""
    lines, n = z.shape
    res = []
    for dims, k, a in (((n, lines, 1), 0, z), ((lines, n, 1), 1, z.T)):
        x = torch.from_numpy(np.ascontiguousarray(a)).cuda()
        out = torch.full_like(x, complex(float("nan"), float("nan"))) if k == 0 else x.clone()
        plan = fft3.Plan(*dims, dtype=fft3.FFT3_C128_FP64, **opts)
        fft3.fft3_plan_execute_pass(plan.handle, k, x.data_ptr(), out.data_ptr())
        torch.cuda.synchronize()
        assert plan.check() == 0, fft3.last_error()
        plan.close()
        got = out.cpu().numpy()
        res.append(got if k == 0 else got.T)
    return res


def _lines(kind, n, lines, rng):
    z = rng.uniform(-1, 1, (lines, n)) + 1j * rng.uniform(-1, 1, (lines, n))
    if kind == "spike":
        z = np.zeros((lines, n), complex)
        z[np.arange(lines), rng.integers(0, n, lines)] = rng.normal(size=lines) + 0.3j
    elif kind == "decades":
        z = 10 ** rng.uniform(-12, 12, (lines, n)) * np.exp(2j * np.pi * rng.uniform(size=(lines, n)))
    elif kind == "scales":  # neighbouring lines 400 decades apart, one of them zero
        z *= 10.0 ** rng.integers(-200, 200, (lines, 1))
        z[1] = 0
    return z


@pytest.mark.parametrize("n", [4, 16, 32, 60, 64, 128, 256, 375, 512, 960, 1024, 2025, 2048, 4096])
@pytest.mark.parametrize("kind", ["uniform", "spike", "decades", "scales"])
def test_one_pass_is_rounded_once(n, kind):
    """Contiguous and strided lines, each line against its own norm.  A result
    is rounded once to FP64 (rms 2^-53 / sqrt(3) = 6.4e-17 of the values' size
    at most) after integer stages whose error is at most about twice that in
    the hardest line (one spike that stays one through the first stage)."""
    rng = np.random.default_rng(n)
    z = _lines(kind, n, 9, rng)
    sc = np.abs(z).max(axis=1, keepdims=True)
    sc[sc == 0] = 1
    ref = np.fft.fft((z.astype(np.clongdouble) / sc), axis=1)
    for got in _passes(z):
        err = np.abs(got.astype(np.clongdouble) / sc - ref)
        norm = np.sqrt((np.abs(ref) ** 2).sum(axis=1))
        rel = np.sqrt((err ** 2).sum(axis=1)) / np.where(norm == 0, 1, norm)
        assert rel.max() <= 2e-16, (kind, float(rel.max()))
        if kind == "scales":
            assert not got[1].any()


@pytest.mark.parametrize("n", [n for n in synth.smooth_sizes(3, 512) if n & (n - 1)])
def test_mixed_plans_are_rounded_once(n):
    """Every mixed-radix plan (contiguous and strided), on values over 24 decades:
    the bound of the test above."""
    z = _lines("decades", n, 9, np.random.default_rng(n))
    sc = np.abs(z).max(axis=1, keepdims=True)
    ref = np.fft.fft(z.astype(np.clongdouble) / sc, axis=1)
    for k, dims in ((0, (n, 9, 1)), (1, (9, n, 1))):
        p = fft3.fft3_plan_schedule(*dims, 1, fft3.FFT3_C128_FP64)["passes"][k]
        assert p.get("compiled") and p["line"]["n"] == n
    for got in _passes(z):
        err = np.abs(got.astype(np.clongdouble) / sc - ref)
        rel = np.sqrt((err ** 2).sum(axis=1) / (np.abs(ref) ** 2).sum(axis=1))
        assert rel.max() <= 2e-16, float(rel.max())


@pytest.mark.parametrize("n", [8, 60, 256, 1024, 1500])
def test_lines_left_to_fp64(n):
    """A tile holding such a line still gives every other line its result."""
    rng = np.random.default_rng(n)
    z = rng.uniform(-1, 1, (9, n)) + 1j * rng.uniform(-1, 1, (9, n))
    z[2, n // 3] = complex(np.inf, 0)
    z[4, 1] = complex(0.5, np.nan)
    z[5] *= 1e-310
    z[6] *= 1e305
    ref = np.fft.fft(np.delete(z, (2, 4), 0), axis=1)
    for got in _passes(z):
        assert not np.isfinite(got[2]).any() and not np.isfinite(got[4]).any()
        g = np.delete(got, (2, 4), 0)
        for a, b in zip(g, ref):
            # 1e-310 is held to 2^-1074 only: 4e-324 * sqrt(n) of absolute error
            assert np.linalg.norm((a - b) * 2.0 ** -60) <= 1e-15 * np.linalg.norm(b * 2.0 ** -60) or \
                np.abs(a - b).max() <= 5e-324 * 4 * n


@pytest.mark.parametrize("order", range(5))
@pytest.mark.parametrize("n", [48, 64, 120, 128, 256, 375, 512, 600, 1024, 2048, 2560])
def test_dominated_lines_keep_fp64_accuracy(n, order):
    """One value just above a power of two over a small background, and its
    transform (a constant with noise), under every radix order: no further off
    than FP64 stages, at most 33 roundings of 2^-53 / sqrt(3) (log2 n levels of two
    additions, three products per twiddle), each of the value's size at most."""
    rng = np.random.default_rng(n)
    noise = rng.uniform(-1, 1, (9, n)) + 1j * rng.uniform(-1, 1, (9, n))
    for bg in (0.1, 1e-3, 1e-12):
        for dc in (False, True):
            z = bg * noise
            if dc:
                z += 1.01 + 0.7j
            else:
                z[np.arange(9), rng.integers(0, n, 9)] = 1.01 + 0.3j
            ref = np.fft.fft(z.astype(np.clongdouble), axis=1)
            for got in _passes(z, radix_order=order):
                err = np.sqrt((np.abs(got.astype(np.clongdouble) - ref) ** 2).sum(axis=1) / (np.abs(ref) ** 2).sum(axis=1))
                assert err.max() <= 3.7e-16, (bg, dc, float(err.max()))


@pytest.mark.parametrize("n", [2, 3, 4, 16, 60, 64, 256, 375, 512, 1024, 1500])
def test_small_parts_beside_large_ones_are_kept(n):
    """What FP64 additions keep apart: a single complex value at index 0 is the
    transform's every value; a tiny imaginary background beside a real value
    there keeps its own relative accuracy."""
    rng = np.random.default_rng(n)
    z = np.zeros((9, n), complex)
    z[:, 0] = rng.normal(size=9) + 1e-9j * rng.normal(size=9)
    for got in _passes(z):
        assert (got == z[:, :1]).all()
    z = 1e-12 * (rng.uniform(-1, 1, (9, n)) + 1j * rng.uniform(-1, 1, (9, n)))
    z[:, 0] = 1.0
    ref = np.fft.fft(z.astype(np.clongdouble), axis=1).imag
    for got in _passes(z):
        err = np.sqrt(((got.imag.astype(np.longdouble) - ref) ** 2).sum(axis=1) / (ref ** 2).sum(axis=1))
        assert err.max() <= 1e-15, float(err.max())
