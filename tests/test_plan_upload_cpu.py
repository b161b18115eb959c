"""Plans that live within one call (circuits, remaps, layout restores) keep the host image of their upload until
the stream has been waited for: the library's host code on a CUDA stand-in with late copies
(plan_upload_host.cpp), no GPU."""
import os
import subprocess

from paper_2406_14084_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_upload_source_outlives_its_copy(tmp_path):
    exe = str(tmp_path / "plan_upload_host")
    cuda = os.path.join(build._cuda_home(build._nvcc()), "include")
    src = [os.path.join(build.CSRC, f) for f in ("api.cpp", "planner.cpp", "lower.cpp")]
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", build.INCLUDE, "-I", build.CSRC, "-I", cuda,
                    os.path.join(HERE, "plan_upload_host.cpp"), *src, "-o", exe, "-Wl,--unresolved-symbols=ignore-all"],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
