"""spmv_stokes as a warp sees it, on the CPU (spmv_stokes_host.cpp): every lane
of a warp that holds velocity nodes and pressure rows takes part in every
full-mask shuffle, with 4 to 32 lanes per group, in 2D and 3D, and the rows'
sums agree with sums in double to 2^-24 times their length (at most 3 * 70
products and the residual's own term)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_lanes_and_sums(tmp_path):
    src = open(os.path.join(ROOT, "paper_2407_07253_gb300", "csrc", "kernels.cuh")).read()
    at = src.rindex("template <int LANES, int MODE, int D>", 0, src.index(" spmv_stokes("))
    (tmp_path / "kernel.inc").write_text(src[at:src.index("\n}\n", at) + 3])
    exe = str(tmp_path / "spmv")
    subprocess.run(["g++", "-O1", "-std=c++20", "-pthread", "-I", str(tmp_path), "-o", exe,
                    os.path.join(ROOT, "tests", "spmv_stokes_host.cpp")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, "lanes of a warp skip a shuffle: " + r.stdout
    assert float(r.stdout) <= 211 * 2.0**-24
