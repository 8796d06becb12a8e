"""Host check of repeat_step (qp_df.h), the photons' equal moves of a fused
window: the bits of the moves taken one by one."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_equal_steps_have_the_bits_of_single_ones(tmp_path):
    exe = tmp_path / "repeat_step_check"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1311_1107_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "repeat_step_check.cpp"), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    n = {line.split()[0]: line.split()[1] for line in out.splitlines() if line[0] != "#"}
    assert int(n["checked"]) > 1_000_000 and int(n["wrong"]) == 0, out
