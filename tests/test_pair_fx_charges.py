"""The fixed-point pair arithmetic where the charges of a tile differ, on the host: it is taken only where a target
that skips the largest charge keeps FP64 accuracy on the others."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_04801_gb300", "csrc")
TILES = 400


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fx") / "pair_fx_charges_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", out, os.path.join(HERE, "pair_fx_charges_host.cpp")],
                   check=True)

    def call(dist, n, par):
        o = subprocess.run([out, dist, str(n), str(par), str(TILES), "17"], check=True, text=True, capture_output=True)
        return [float(v) for v in o.stdout.split()]

    return call


# taken: at least this share of the tiles are summed in fixed point, at most that share.
#
# Worst case of a pair, in units of the charge 1, with 1/r >= 1/2.4 here: potential 2^-50.6 (the correction's charge
# to 2^-28, times 2^-21, a third of it), field 2^-49 y + 2^-52 / y.  The others' mean |q| is at least 1/12: 12 x 2.4 x
# 2^-50.6 = 2^-45.7 of |q|/r, 12 (2.4 x 2^-49 + 2.4^3 2^-52) = 2^-43.3 of |q|/r^2, and the bounds of equal charges
# (2^-50, 2^-47) with them.  Rms: as the FP64 loop over the same sources; half again at most where the charges are
# the widest that are taken.
@pytest.mark.parametrize("dist,n,par,taken", [
    ("normal", 256, 1.0, (0.95, 1.0)), ("normal", 256, 1.2e-19, (0.95, 1.0)), ("normal", 200, 1.7, (0.95, 1.0)),
    ("ions", 256, 1.0, (1.0, 1.0)), ("ions", 40, 3.0, (1.0, 1.0)), ("zeros", 256, 0.3, (1.0, 1.0)),
    ("heavy", 256, 0.5, (1.0, 1.0)), ("heavy", 256, 0.25, (1.0, 1.0)), ("lognormal", 256, 0.5, (0.9, 1.0)),
    ("lognormal", 256, 1.0, (0.0, 1.0)), ("normal", 16, 1.0, (0.0, 0.3)), ("ions", 2, 1.0, (1.0, 1.0)),
    ("ions", 13, 1.0, (1.0, 1.0)), ("uniform", 8, 1.0, (0.0, 1.0)), ("zeros", 60, 0.3, (1.0, 1.0)),
    ("heavy", 256, 2.0**-4, (0.0, 0.0)), ("heavy", 256, 2.0**-10, (0.0, 0.0)), ("heavy", 256, 2.0**-19, (0.0, 0.0)),
    ("heavy", 12, 0.25, (0.0, 0.0)), ("lognormal", 256, 4.0, (0.0, 0.0))])
def test_target_that_skips_the_largest_charge(run, dist, n, par, taken):
    accepted, rms_p, rms_f, pot, field = run(dist, n, par)
    assert taken[0] <= accepted / TILES <= taken[1]
    assert rms_p <= 1.5 and rms_f <= 1.5
    assert pot < 2.0**-45.6 and field < 2.0**-43.2
