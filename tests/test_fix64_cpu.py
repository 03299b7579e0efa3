"""Which complex128 lines the integer stages take, and their error against the FP64
stages on the same lines (both on the host, against long double): over every radix
list that the planner gives a complex128 line, lines taken are at least as close."""
import os
import shutil
import subprocess

import pytest

from paper_1904_10119_gb300 import fft3, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _lists():
    """(kernel, n, radices) of contiguous and strided lines under every radix order."""
    out = set()
    for n in [n for n in synth.smooth_sizes(3, 512) if n != 4] + [540, 768, 1024, 1500, 2025, 2048, 2560, 4000, 4096]:
        for order in range(5):
            for k, dims in ((0, (n, 9, 1)), (1, (9, n, 1))):
                s = fft3.fft3_plan_schedule(*dims, 1, fft3.FFT3_C128_FP64, fft3.FFT3_PENCIL3,
                                            opts=fft3.make_options(radix_order=order))
                p = s["passes"][k]
                runtime = p["kind"] == "line_runtime_fp64" and not p.get("compiled")
                out.add(("g" if runtime else "c", n, tuple(p["line"]["radices"])))
    return sorted(out)


def test_integer_stages_are_no_further_off_than_fp64(tmp_path):
    cxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "fix64_host")
    subprocess.run([cxx, "-O2", "-std=gnu++17", "-w", "-I", os.path.join(ROOT, "paper_1904_10119_gb300", "csrc"), "-I", cuda,
                    os.path.join(ROOT, "tests", "fix64_host.cpp"), "-o", exe], check=True)
    lists = "".join(f"{k} {n} {' '.join(map(str, r))}\n" for k, n, r in _lists())
    rows = [r.split() for r in subprocess.run([exe], input=lists, text=True, capture_output=True, check=True).stdout.split("\n") if r]
    assert len(rows) > 1000
    taken = {}
    for n, kind, count, fix, fp64 in rows:
        n, count, fix, fp64 = int(n), int(count), float(fix), float(fp64)
        taken.setdefault(kind, []).append(count)
        # a line of three or six points is rounded once either way: equal within the sampling of the
        # rounding errors of its 96 components and more
        assert count == 0 or fix <= (1.06 if n <= 6 else 1) * fp64, (n, kind, fix, fp64)
    # flat lines are taken, lines whose real and imaginary parts differ by more than 2^5 are not
    for kind in ("uniform", "real", "dc-3"):
        assert sum(taken[kind]) >= 0.98 * 16 * len(taken[kind]), kind
    for kind in ("im-12",):
        assert not any(taken[kind]), kind
