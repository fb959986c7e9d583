"""The fixed-point pair arithmetic of the FP64 near sums, on the host."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_04801_gb300", "csrc")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fx") / "pair_fx_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", out, os.path.join(HERE, "pair_fx_host.cpp")],
                   check=True)
    return out


# Bounds from the formats, with r <= 2.4 in scaled units.  Potential: e to one
# unit of 2^-52 (half of it reaches 1/r), its correction to 2^-27 2^-22, the
# rounding of the result: 2^-50.  Field: 3/2 of e and the correction's rounding
# (2^-51), V to half of 2^-51 times r^2 |d| <= 2.4^3 (2^-48.2), V dl in FP32.
@pytest.mark.parametrize("mode,count", [(0, 200000), (1, 200000), (2, 2000), (3, 20000)])
def test_pair_against_long_double(exe, mode, count):
    pot, field, e = (float(v) for v in subprocess.run([exe, str(mode), str(count), "11"], check=True, text=True,
                                                      capture_output=True).stdout.split())
    assert e < 2.0**-21.6  # what the 64-bit product holds
    assert pot < 2.0**-50
    assert field < 2.0**-47
