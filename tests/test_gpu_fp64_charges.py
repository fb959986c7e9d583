"""FP64 sums at a target that sits on a charge far above its neighbours (a macro-ion among counter-ions): the sum leaves
that charge out, so its error is measured against the small charges alone."""
import numpy as np
import pytest

from oracle import hsma as oh
from paper_1806_04801_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _sums(s, q, t):
    """Potential and field at t in extended precision, and the sums of |q|/r and |q|/r^2; a source at t is left out."""
    d = t.astype(np.longdouble) - s
    r2 = (d * d).sum(1)
    ri = np.where(r2 > 0, 1 / np.sqrt(np.where(r2 > 0, r2, 1)), 0)
    return (ri * q).sum(), (d * (ri**3 * q)[:, None]).sum(0), (ri * np.abs(q)).sum(), (ri**2 * np.abs(q)).sum()


# An FP64 sum of m terms rounds its running sum m times: 2^-53 sqrt(m) sum |q|/r in the mean square; twice that.
@pytest.mark.parametrize("ratio", [2.0**3, 2.0**5, 2.0**12, 2.0**17, 2.0**19, 2.0**25])
@pytest.mark.parametrize("ns", [200, 1021])
def test_direct_sum_on_a_heavy_source(ns, ratio):
    import torch

    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(ns)
    s, q, t = g.random((ns, 3)), np.where(g.random(ns) < 0.5, -1.0, 1.0), g.random((5, 3))
    q[17] = ratio
    t[2] = s[17]
    src = torch.as_tensor(np.concatenate([s, q[:, None]], 1)).cuda()
    pot, fld = hsma.coulomb_sum(src, torch.as_tensor(t).cuda(), field=True, precision="fp64")
    phi, e, ap, ae = _sums(s, q, t[2])
    bound = 2 * np.sqrt(ns) * 2.0**-53
    assert abs(pot[2].item() - phi) <= bound * ap
    assert np.all(np.abs(fld[2].cpu().numpy() - e) <= bound * ae)


# In a plan: the charge at the box's centre and a sphere that holds none of its images.
@pytest.mark.parametrize("ratio", [2.0**5, 2.0**12, 2.0**19])
@pytest.mark.parametrize("n", [100, 700])
def test_near_sums_on_a_heavy_particle(n, ratio):
    from paper_1806_04801_gb300 import hsma

    box, bc, rs = (1.0, 1.0, 1.0), I.GROUNDED, 0.95
    g = np.random.default_rng(n)
    xyz, q = 0.02 + 0.96 * g.random((n, 3)), np.where(g.random(n) < 0.5, -1.0, 1.0)
    xyz[7], q[7] = 0.5, ratio
    c = oh.centre_positions(xyz, box, bc)
    s, sq, _, _ = oh.inset(c, q, np.array(box), bc, rs)
    assert (np.abs(sq) == ratio).sum() == 1
    phi, e, ap, ae = _sums(s, sq, c[7])
    with hsma.Plan(box, bc, 4, rs, 540, 100, precision="fp64") as p:
        own, gphi, ge, _ = p.shard_near(xyz, q, 0, 1)
    at = int(np.flatnonzero(own == 7)[0])
    bound = 2 * np.sqrt(len(sq)) * 2.0**-53
    assert abs(gphi[at] - phi) <= bound * ap
    assert np.all(np.abs(ge[at] - e) <= bound * ae)
