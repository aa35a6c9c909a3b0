"""The epilogue's packed residue sums through their folds, up to 64 sub-chunks (crt.h)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sums_through_folds(tmp_path):
    exe = str(tmp_path / "crt_fold_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2404_19163_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "native", "crt_fold_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
