"""Host check of the streamed triangle kernels' work division (csrc/tri_plan.h): compiled
with the host compiler, it walks every share of a grid of plans as the kernel does."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_unit_in_exactly_one_share(tmp_path):
    exe = str(tmp_path / "tri_plan_host")
    subprocess.run(["g++", "-O2", "-std=c++17",
                    "-I" + os.path.join(ROOT, "paper_0706_3060_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "tri_plan_host.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.startswith("ok "), out.stdout + out.stderr
