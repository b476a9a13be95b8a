"""Packed mask tables and zero couplings of the run-time operator bodies
(csrc/kuhn_weights.hpp): every entry unpacks to the weight that it was packed from, and a
coupling is left out exactly where no mask gives it a weight."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tables_hold_the_weights(tmp_path):
    exe = str(tmp_path / "tables")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2007_02082_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "mask_tables_probe.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    rows = {ln.split()[0]: [int(v) for v in ln.split()[1:]] for ln in out if ln}
    assert set(rows) == {"mass", "trans", "couples", "coupled"}
    for name, (n, bad) in rows.items():
        assert n > 0 and bad == 0, name
