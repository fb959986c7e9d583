"""FP64 sums of particles that nearly coincide: distances below the units of the fixed-point words."""
import numpy as np
import pytest

from paper_1806_04801_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# The pair's own term is 1/d with d as the caller's coordinates give it, and the largest by far; the others' sum has
# the rounding of m = 400 FP64 terms (2 sqrt(m) 2^-53 of sum |q|/r), added to it once (2^-53 of 1/d) like the pair's
# own roundings (a few 2^-53).
@pytest.mark.parametrize("exponent", [-50, -40, -34, -33, -32, -31, -30, -29, -28, -20, -10])
def test_direct_sum_next_to_a_source(exponent):
    import torch

    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(60 - exponent)
    s, q, t = g.random((400, 3)), np.where(g.random(400) < 0.5, -1.0, 1.0), g.random((64, 3))
    s[:64] = (np.floor(s[:64] * 2.0**30) + 0.5) * 2.0**-30  # between two values of the high word
    t = s[:64] + 2.0**exponent * g.uniform(-1.0, 1.0, (64, 3))
    src = torch.as_tensor(np.concatenate([s, q[:, None]], 1)).cuda()
    pot, fld = hsma.coulomb_sum(src, torch.as_tensor(t).cuda(), field=True, precision="fp64")
    d = t[:, None].astype(np.longdouble) - s[None]
    r2 = (d * d).sum(2)
    ri = np.where(r2 > 0, 1 / np.sqrt(np.where(r2 > 0, r2, 1)), 0)
    bound = (2 * np.sqrt(400) + 8) * 2.0**-53
    assert np.all(np.abs(pot.cpu().numpy() - (ri * q).sum(1)) <= bound * ri.sum(1))
    e = (d * (ri**3 * q)[:, :, None]).sum(1)
    assert np.all(np.abs(fld.cpu().numpy() - e) <= bound * (ri**2).sum(1)[:, None])


# Two particles of a plan at distances down to 2^-40: the energy is q q'/d and a smooth rest.
@pytest.mark.parametrize("exponent", [-40, -33, -32, -31, -30, -25])
def test_step_with_two_particles_that_nearly_coincide(exponent):
    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(5)
    n = 64
    xyz, q = 0.05 + 0.9 * g.random((n, 3)), np.where(np.arange(n) % 2, -1.0, 1.0)
    with hsma.Plan((1.0, 1.0, 1.0), I.PERIODIC, 6, 1.5, 540, 200, precision="fp64") as p:
        for k in range(8):
            xyz[0] = 0.25 + 0.5 * g.random(3)
            xyz[0] = (np.floor(xyz[0] * 2.0**30) + 0.5) * 2.0**-30
            xyz[1] = xyz[0] + 2.0**exponent * g.uniform(-1.0, 1.0, 3)
            # the centred coordinates that both particles' sums start from
            d = np.linalg.norm((xyz[1] - 0.5) - (xyz[0] - 0.5))
            U = p.energy_forces(xyz, q)[0]
            assert abs(U * d + 1.0) <= 1e-12 + 1e5 * d
