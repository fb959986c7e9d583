"""The fixed-point pair arithmetic at every small distance, on the host: such pairs are left to the native loop."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_04801_gb300", "csrc")


def test_close_pairs_are_recognised(tmp_path):
    out = str(tmp_path / "pair_fx_close_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", out, os.path.join(HERE, "pair_fx_close_host.cpp")],
                   check=True)
    r = subprocess.run([out, "2000000", "5"], check=True, text=True, capture_output=True)
    assert r.stdout.split() == ["0", "0"]
