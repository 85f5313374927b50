"""Host check of the streamed triangle kernels' work division at large sizes (csrc/tri_plan.h)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_shares_of_large_systems(tmp_path):
    exe = str(tmp_path / "tri_plan_large_host")
    subprocess.run(["g++", "-O2", "-std=c++17",
                    "-I" + os.path.join(ROOT, "paper_0706_3060_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "tri_plan_large_host.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.startswith("ok "), out.stdout + out.stderr
