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


# The direct sum finds its scale from the coordinates: boxes off the origin,
# flat and clustered sets, targets outside the sources' box, a target on a
# source (skipped), and sets whose offset leaves the formats (native FP64).
@pytest.mark.parametrize("field", [True, False])
@pytest.mark.parametrize("shape", ["unit", "offset", "far offset", "flat", "cluster and one far", "small units",
                                   "one point"])
@pytest.mark.parametrize("ns,nt", [(1, 1), (255, 257), (1021, 130)])
def test_direct_sum_at_every_scale(shape, ns, nt, field):
    import torch

    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(ns)
    s, t, q = g.random((ns, 3)), 1.5 * g.random((nt, 3)) - 0.2, g.standard_normal(ns)
    if shape == "offset":
        s, t = s + [100.0, -7.0, 0.0], t + [100.0, -7.0, 0.0]
    elif shape == "far offset":
        s, t = s + 3e7, t + 3e7
    elif shape == "flat":
        s[:, 2], t[:, 2] = 0.25, 0.25
    elif shape == "cluster and one far":
        s, t = 1e-5 * s, 1e-5 * t
        t[0] = 1.0
    elif shape == "small units":
        s, t, q = 1e-9 * s, 1e-9 * t, 1.6e-19 * q
    elif shape == "one point":
        s[:], t[:] = 0.5, 0.5
    t[nt // 2] = s[ns // 2]
    src = np.concatenate([s, q[:, None]], 1)
    pot, fld = hsma.coulomb_sum(torch.as_tensor(src).cuda(), torch.as_tensor(t).cuda(), field=field,
                                precision="fp64")
    d = t[:, None].astype(np.longdouble) - s[None]
    r2 = (d * d).sum(2)
    ri = np.where(r2 > 0, 1 / np.sqrt(np.where(r2 > 0, r2, 1)), 0)
    bound = (2 * ns + 30) * 2.0**-53
    assert np.all(np.abs(pot.cpu().numpy() - (ri * q).sum(1)) <= bound * (ri * np.abs(q)).sum(1))
    if field:
        e = (d * (ri**3 * q)[:, :, None]).sum(1)
        assert np.all(np.abs(fld.cpu().numpy() - e) <= bound * (ri**2 * np.abs(q)).sum(1)[:, None])
    else:
        assert fld is None
