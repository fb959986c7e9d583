"""The FP64 near sums and the FP64 surface sums at the edges of their forms."""
import numpy as np
import pytest

from oracle import hsma as oh
from paper_1806_04801_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BOX = (1.0, 1.0, 1.0)


def _case(name, n, seed=3):
    g = np.random.default_rng(seed + n)
    xyz, q = g.random((n, 3)), g.standard_normal(n)
    if name == "cluster":  # every pair of the box is a near pair: native FP64, tile by tile
        xyz = 0.5 + 0.02 * (xyz - 0.5)
    elif name == "wide charges":  # tiles whose charges span more than the formats keep
        q *= 10.0 ** g.integers(-9, 9, n)
    elif name == "tiny units":
        q *= 1.6e-19
    elif name == "zeros":
        q[::2] = 0.0
    elif name == "walls":  # coordinates on and next to the box's faces
        xyz[: n // 2, 0] = np.where(np.arange(n // 2) % 2, 0.0, 1.0 - 2.0**-53)
    q -= q.mean() if name not in ("wide charges", "zeros") else 0.0
    if name == "zeros" and n > 1:
        q[1::2] -= q[1::2].mean()
    return xyz, q


# Both sides sum up to m terms in FP64-like precision, in different orders:
# |difference| <= 2 m 2^-53 sum |q|/r (potential; the field likewise with
# |q|/r^2), m the in-set size.
@pytest.mark.parametrize("name", ["plain", "cluster", "wide charges", "tiny units", "zeros", "walls"])
@pytest.mark.parametrize("n", [2, 129, 256, 301, 700])
def test_near_sums_against_the_oracle(name, n):
    from paper_1806_04801_gb300 import hsma

    xyz, q = _case(name, n)
    if name == "wide charges":
        bc = I.GROUNDED  # no neutrality to keep
        xyz = 0.05 + 0.9 * xyz
    else:
        bc = I.PERIODIC
    plan = oh.make_plan(BOX, bc, 4, 1.5, 100, 89)
    c = oh.centre_positions(xyz, BOX, bc)
    s_xyz, s_q, _, _ = oh.inset(c, q, plan.box, bc, 1.5)
    idx = np.arange(n)
    phi, e = oh.coulomb(s_xyz, s_q, c, tskip=idx, field=True)
    pa, _ = oh.coulomb(s_xyz, np.abs(s_q), c, tskip=idx, field=True)
    d = c[:, None] - s_xyz[None]
    r2 = (d * d).sum(2)
    r2[idx, idx] = np.inf
    ea = (np.abs(s_q) / r2).sum(1)
    with hsma.Plan(BOX, bc, 4, 1.5, 540, 100, precision="fp64") as p:
        own, gphi, ge, gmon = p.shard_near(xyz, q, 0, 1)
    bound = 2 * len(s_q) * 2.0**-53
    assert np.all(np.abs(gphi - phi[own]) <= bound * pa[own])
    assert np.all(np.abs(ge - e[own]) <= bound * ea[own][:, None])


def test_non_finite_and_coincident_inputs_still_error():
    from paper_1806_04801_gb300 import hsma

    with hsma.Plan(BOX, I.PERIODIC, 4, 1.5, 540, 100, precision="fp64") as p:
        for bad in ("coincident", "nan position", "inf charge"):
            xyz, q = _case("plain", 300)
            if bad == "coincident":
                xyz[7] = xyz[200]
            elif bad == "nan position":
                xyz[5, 1] = np.nan
            else:
                q[9] = np.inf
            with pytest.raises(hsma.HsmaError):
                p.energy_forces(xyz, q)


# Thin layers take the point-dipole series, thick ones the literal images;
# the line is h = 6.4e-4 (Rs - R0).  The oracle sums the literal images: its
# rounding is 2^-53 Rs/dr of the dipole terms, 2e-11 at the thinnest layer.
@pytest.mark.parametrize("dr_rel", [1e-5, 1e-4, 5.3e-4, 5.5e-4, 5e-3])
@pytest.mark.parametrize("n", [1, 63, 65, 200])
def test_surface_sums_at_every_layer_thickness(dr_rel, n):
    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(n)
    xyz, q = 0.05 + 0.9 * g.random((n, 3)), g.standard_normal(n) * 1e-17
    F2, _ = oh.fib_from_points(540)
    ref = oh.energy_forces(xyz, q, oh.make_plan(BOX, I.GROUNDED, 6, 1.5, 300, F2, dr_rel))
    with hsma.Plan(BOX, I.GROUNDED, 6, 1.5, 540, 300, precision="fp64", dr_rel=dr_rel) as p:
        _, f, pot, _ = p.energy_forces(xyz, q, potentials=True)
    scale = np.abs(ref["phi_out"]).max()
    assert np.abs(pot - ref["pot"]).max() <= 1e-10 * max(scale, np.abs(ref["pot"]).max())
    assert np.abs(f - ref["forces"]).max() <= 1e-10 * max(np.abs(ref["forces"]).max(),
                                                          np.abs(q).max() * np.abs(ref["e_out"]).max())
