"""Host check that the mixed path's conversions keep infinities and NaN
(qp_df.h): a fault in a particle's state must stay visible in it."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_conversions_keep_infinities_and_nan(tmp_path):
    exe = tmp_path / "df_special_check"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1311_1107_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "df_special_check.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    results = {line.split()[0]: int(line.split()[1]) for line in out.splitlines()}
    assert set(results) == {"f_to_d", "merge", "add_fd", "depth"}
    assert all(v == 0 for v in results.values()), out
