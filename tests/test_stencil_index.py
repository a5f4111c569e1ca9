"""Index arithmetic of the stored-stencil product near the largest number of
unknowns, compiled and run on the host (tests/stencil_index.cu)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_2106_06404_gb300")


def test_stencil_neighbours_stay_in_range(tmp_path):
    exe = str(tmp_path / "stencil_index")
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    subprocess.check_call([nvcc if os.path.exists(nvcc) else "nvcc", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-std=c++17", "-I", os.path.join(PKG, "csrc"),
                           "-I", os.path.join(os.path.dirname(HERE), "include"),
                           os.path.join(HERE, "stencil_index.cu"), "-o", exe])
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "0"
