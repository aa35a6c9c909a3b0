"""The residue step of the operand kernels (crt.h): congruent, and within 128 of zero, for every modulus."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_residue_step(tmp_path):
    exe = str(tmp_path / "crt_residue_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2404_19163_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "native", "crt_residue_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
