"""The CRT reconstruction's table is read inside its bounds whatever the digits hold (crt_combine.h)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_table_index(tmp_path):
    exe = str(tmp_path / "crt_unwritten_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2404_19163_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "native", "crt_unwritten_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
