"""Harmonic basis: a row's values do not depend on how many points the call has.

The number of points and the order decide how many groups of 32 points a block holds and how many warps share a
group's orders.  Every value goes through the same operations in each of these shapes, so the rows of a small call
are those of a large one bit for bit; tests/test_gpu_parity.py compares the values themselves with the oracle.
"""
import numpy as np
import pytest
import torch

hsma = pytest.importorskip("paper_1806_04801_gb300.hsma")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("p", [0, 1, 2, 3, 5, 8, 12, 17, 25, 40])
def test_rows_do_not_depend_on_the_number_of_points(p, precision):
    rng = np.random.default_rng(90 + p)
    big = min(150_001, 60_000_000 // (p + 1) ** 2)
    x = rng.uniform(-0.9, 0.9, (big, 3))
    x[:4] = [[0.0, 0.0, 0.0], [1e-12, -3e-14, 2e-13], [0.5, 0.0, 0.0], [0.0, 0.0, -1.0]]
    x = torch.from_numpy(x).cuda()
    full = hsma.basis(x, p, 1.5, precision=precision)
    for n in (1, 31, 33, 1003, 5000, 20011, 33333):
        if n > big:
            break
        part = hsma.basis(x[:n].contiguous(), p, 1.5, precision=precision)
        assert torch.equal(part.view(torch.int64), full[:n].contiguous().view(torch.int64)), n
