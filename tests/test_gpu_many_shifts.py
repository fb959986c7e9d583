"""Small systems in a sphere many boxes wide: the in-set has more counts (one per shift and 256 particles) than its
scatter adds up by itself."""
import numpy as np
import pytest

from oracle import hsma as oh
from paper_1806_04801_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# 17^3 = 4913 shifts: 29478 counts with six blocks, 34391 with seven.  FP64 against the oracle's FP64: 2 m 2^-53 of
# the sums' terms is 1e-9 for m = 4e6, the difference of two summation orders far below it.
def test_inset_on_both_sides_of_the_limit():
    from paper_1806_04801_gb300 import hsma

    box, R = (1.0, 1.0, 1.0), 8.4
    launches = {}
    with hsma.Plan(box, I.PERIODIC, 4, R, 540, 100, precision="fp64") as p:
        plan = oh.make_plan(box, I.PERIODIC, 4, R, 100, 89)
        for n in (40, 1536, 1537):
            g = np.random.default_rng(n)
            xyz, q = g.random((n, 3)), g.standard_normal(n)
            q -= q.mean()
            U, F, _, ns = p.energy_forces(xyz, q)
            before = hsma.kernel_launches()
            U2, F2, _, _ = p.energy_forces(xyz, q)
            launches[n] = hsma.kernel_launches() - before
            assert U == U2 and np.array_equal(F, F2)
            ref = oh.energy_forces(xyz, q, plan, nthreads=16)
            assert ns == ref["n_inset"]
            assert abs(U - ref["energy"]) <= 1e-9 * np.abs(q * ref["pot"]).sum()
            assert np.abs(F - ref["forces"]).max() <= 1e-9 * np.abs(ref["forces"]).max()
    # beyond the limit the counts are scanned by a kernel of its own
    assert launches[40] == launches[1536] == launches[1537] - 1
