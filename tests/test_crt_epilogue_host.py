"""The residue products' epilogue arithmetic (crt.h: crt_step, the packed sums, crt_digit_sum) against integers."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_epilogue_residues_exact(tmp_path):
    exe = str(tmp_path / "crt_epilogue_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2404_19163_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "native", "crt_epilogue_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
