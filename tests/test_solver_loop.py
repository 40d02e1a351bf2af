"""The solver's loop over graph iterations on the host: it ends after its
segment for every value of the graph's handles, zero among them.  No GPU
needed."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_segments_end_for_every_handle_value(tmp_path):
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = cand if os.path.exists(cand) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = tmp_path / "solver_loop_check"
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_1311_4521_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(HERE, "host", "solver_loop_check.cu"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and "0 failures" in out.stdout, out.stdout + out.stderr
