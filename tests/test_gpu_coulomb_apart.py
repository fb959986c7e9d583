"""FP64 direct sums at targets away from the sources, where neutral charges nearly cancel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# An FP64 loop makes some four roundings of each of the n terms (2^-53 of it each, independent: 4 sqrt(n)) and rounds
# its running sum, of the size of sqrt(n) terms, n times (sqrt(n) sqrt(n) / 2): in the root mean square over the
# targets, in units of 2^-53 of a term.
@pytest.mark.parametrize("away", [(0.0, 0.0, 2.0), (1.0, 1.0, 1.0), (6.0, 6.0, 6.0), (40.0, 3.0, 0.0)])
@pytest.mark.parametrize("n", [40, 256, 1500])
def test_fields_of_neutral_charges_from_afar(n, away):
    import torch

    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(n)
    s, q = g.random((n, 3)), g.permutation(np.where(np.arange(n) % 2, -1.0, 1.0))
    t = g.random((130, 3)) + away
    src = np.concatenate([s, q[:, None]], 1)
    pot, fld = hsma.coulomb_sum(torch.as_tensor(src).cuda(), torch.as_tensor(t).cuda(), field=True, precision="fp64")
    k = slice(0, 60)
    d = t[k, None].astype(np.longdouble) - s[None]
    ri = 1 / np.sqrt((d * d).sum(2))
    ep = pot[k].cpu().numpy() - (ri * q).sum(1)
    ef = fld[k].cpu().numpy() - (d * (ri**3 * q)[:, :, None]).sum(1)
    rms = lambda v: float(np.sqrt(np.mean(v * v)))  # noqa: E731
    units = (4 * np.sqrt(n) + n / 2) * 2.0**-53
    assert rms(ep) <= units * rms(ri)
    assert rms(ef) <= units * rms(ri**2)
