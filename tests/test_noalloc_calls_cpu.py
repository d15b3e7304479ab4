"""The host side of the allocation-free residual's calls (which words they share), compiled without CUDA."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_calls_share_no_word(tmp_path):
    exe = tmp_path / "noalloc_calls"
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2309_11488_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "c", "noalloc_calls.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stdout
