"""The scale of the FP64 direct sums for sources and targets in boxes of their own, on the host: as accurate as an FP64
loop at targets away from the sources, and no more near pairs than a cube of both has."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1806_04801_gb300", "csrc")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fx") / "pair_fx_boxes_host")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", out, os.path.join(HERE, "pair_fx_boxes_host.cpp")],
                   check=True)
    return out


# Sides of the sources' box, of the targets', the targets' offset; halvings.  Halved sets have at most 0.2% near pairs
# (half again for scatter).  Rms errors as the FP64 loop's (256 charges +-1 and 400 targets: half again for scatter).
@pytest.mark.parametrize("side,tside,off,halvings", [
    ((1, 1, 1), (1, 1, 1), (0, 0, 0), 0), ((0.9999,) * 3, (0.9999,) * 3, (0, 0, 0), 0),
    ((1.9, 1.9, 1.9), (1.9, 1.9, 1.9), (0, 0, 0), 0),
    ((7.3, 7.3, 7.3), (7.3, 7.3, 7.3), (0, 0, 0), 0), ((1, 1, 1), (0.1, 0.1, 0.1), (0.4, 0.4, 0.4), 0),
    ((1, 1, 1), (1, 1, 1), (1, 1, 1), None), ((1, 1, 1), (1, 1, 1), (0.99, 0.99, 0.99), 1),
    ((1, 1, 1), (1, 1, 1), (0.5, 0.5, 0.5), None),
    ((1, 1, 1), (1, 1, 1), (0, 0, 2), None), ((1, 1, 1), (1, 1, 1), (20, 0, 0), None),
    ((1, 1, 1), (1, 1, 1), (20, 20, 20), None), ((1, 1, 1), (0, 0, 0), (3, 3, 3), None),
    ((1e-9, 1e-9, 1e-9), (1e-9, 1e-9, 1e-9), (2e-8, 2e-8, 2e-8), None), ((1, 1, 0), (1, 1, 0), (5, 0, 0.5), None),
    ((1, 2, 40), (1, 2, 40), (1.5, 0, 0), None), ((0.1, 0.1, 0.1), (3, 3, 3), (0, 0, 0), None)])
def test_scale_of_two_boxes(exe, side, tside, off, halvings):
    r = subprocess.run([exe] + [str(v) for v in (*side, *tside, *off)] + ["400", "3"], check=True, text=True,
                       capture_output=True)
    k, near, pot, field = (float(v) for v in r.stdout.split())
    if halvings is not None:
        assert k == halvings
    assert k == 0 or near <= 0.003
    assert pot <= 1.5 and field <= 1.5
