"""The residue arithmetic of the FP64-accurate products, on the host.

csrc/crt_scheme.cuh is compiled with the host compiler and its functions (the
ones the kernels run) are compared with 128-bit integers: the moduli's
conditions, the reduction at every quotient boundary, FP64 bits to scaled
integers, and the recombination over the whole range below M / 2.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_residue_arithmetic_against_128_bit_integers(tmp_path):
    exe = str(tmp_path / "crt_scheme_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2403_06937_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "crt_scheme_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
