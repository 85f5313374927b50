"""Host check of the batched streamed triangle kernel's work division
(csrc/tri_batch_plan.h), compiled with the host compiler."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_unit_of_every_system_in_one_segment(tmp_path):
    exe = str(tmp_path / "tri_batch_plan_host")
    subprocess.run(["g++", "-O2", "-std=c++17",
                    "-I" + os.path.join(ROOT, "paper_0706_3060_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "tri_batch_plan_host.cpp"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.startswith("ok "), out.stdout + out.stderr
