"""The row-block matvec's layout and sign algebra on the CPU (tests/host/row_block_check.cu): 8 and 32
rows per thread, with and without low bits, 1 to 5 states, tiles dealt to 1, 3 and 8 CTAs, both
sectors, N = 12 to 20.

Bound: a row is a sum of at most 256 masks (N = 20) in FP32, with random signs about sqrt(256) / 2
roundings of 2^-24 of it: 5e-7.  2e-6 leaves a factor of four; a wrong sign or table entry gives 1e-2
and more."""
import os
import subprocess

from paper_2002_05725_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_layout_and_signs(tmp_path):
    lib = build.build()
    exe = str(tmp_path / "row_block_check")
    cmd = [build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "--expt-extended-lambda",
           "-I", build.CSRC, "-I", os.path.join(ROOT, "include"), "-o", exe,
           os.path.join(ROOT, "tests", "host", "row_block_check.cu"), lib, "-lcudart",
           "-Xlinker", "-rpath," + os.path.dirname(lib)]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:]
    assert "shapes" in r.stdout, r.stdout
