"""The task lists' device array after a failed allocation (host only: the allocator is the test's)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_failed_growth_leaves_an_empty_array(tmp_path):
    exe = str(tmp_path / "regrow_check")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"),
                        "-I", os.path.join(ROOT, "paper_2407_19614_gb300", "csrc"), "-x", "c++",
                        os.path.join(ROOT, "tests", "regrow_check.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.strip() == "OK", out.stdout
