"""The paths that systems take by their size: the one-block spatial order up to 4096 particles, the surface and fit
kernels' splits, against the oracle on both sides of each line."""
import numpy as np
import pytest

from oracle import hsma as oh
from paper_1806_04801_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BOX = (1.0, 1.0, 1.0)


def _system(n, bc, seed=5):
    g = np.random.default_rng(seed + n)
    xyz, q = 0.02 + 0.96 * g.random((n, 3)), g.standard_normal(n)
    if n > 8:  # several particles in one Morton cell: ties keep the caller's order
        xyz[n // 2: n // 2 + 4] = 0.3 + 1e-3 * g.random((4, 3))
    return xyz, q - (q.mean() if bc == I.PERIODIC else 0.0)


# FP64 against the oracle's FP64: both sum up to m = 15 n terms, 2 m 2^-53 of
# sum |q|/r <= 1e-11 of the energy's terms at these sizes.
@pytest.mark.parametrize("n", [2, 63, 64, 65, 1023, 1025, 4095, 4096, 4097])
def test_order_and_inset_around_the_small_limit(n):
    from paper_1806_04801_gb300 import hsma

    xyz, q = _system(n, I.PERIODIC)
    ref = oh.energy_forces(xyz, q, oh.make_plan(BOX, I.PERIODIC, 4, 1.5, 100, 89), nthreads=16)
    with hsma.Plan(BOX, I.PERIODIC, 4, 1.5, 540, 100, precision="fp64") as p:
        U, F, pot, ns = p.energy_forces(xyz, q, potentials=True)
        b = [_system(m, I.PERIODIC) for m in (n, 17)]  # and in a batch with a smaller one
        off = [0, n, n + 17]
        E2, F2, _, _ = p.energy_forces_batched(np.concatenate([v[0] for v in b]), np.concatenate([v[1] for v in b]),
                                               off)
    assert ns == ref["n_inset"]
    scale = np.abs(ref["pot"]).max()
    assert np.abs(pot - ref["pot"]).max() <= 1e-10 * scale
    assert np.abs(F - ref["forces"]).max() <= 1e-10 * np.abs(ref["forces"]).max()
    assert abs(U - ref["energy"]) <= 1e-10 * scale * np.abs(q).sum()
    assert abs(E2[0] - U) <= 1e-10 * scale * np.abs(q).sum()
    assert np.abs(F2[:n] - F).max() <= 1e-10 * np.abs(F).max()


# FP32 surface sums: thin layers without and with the h^2 terms, thick ones
# literally (lines at h = 3e-5 and 5e-3 of Rs - R0), a batch with more blocks
# than the split to 8 particles takes.  The forces' stated bound is 1e-5 RMS.
@pytest.mark.parametrize("dr_rel", [1e-5, 2e-4, 3e-3, 6e-3])
@pytest.mark.parametrize("n", [1, 9, 65, 300])
def test_fp32_surface_sums_at_every_layer_thickness(dr_rel, n):
    from paper_1806_04801_gb300 import hsma

    xyz, q = _system(n, I.GROUNDED)
    F2, _ = oh.fib_from_points(540)
    ref = oh.energy_forces(xyz, q, oh.make_plan(BOX, I.GROUNDED, 6, 1.5, 300, F2, dr_rel))
    with hsma.Plan(BOX, I.GROUNDED, 6, 1.5, 540, 300, precision="fp32", dr_rel=dr_rel) as p:
        _, _, pot, _ = p.energy_forces(xyz, q, potentials=True)
        reps = -(-65 * 300 // n) if n >= 65 else 2
        xs, qs = np.tile(xyz, (reps, 1)), np.tile(q, reps)
        _, fb, _, _ = p.energy_forces_batched(xs, qs, np.arange(reps + 1) * n)
    assert np.abs(pot - ref["pot"]).max() <= 2e-6 * max(np.abs(ref["pot"]).max(), np.abs(ref["phi_out"]).max())
    rms = lambda v: np.sqrt(np.mean(v * v))  # noqa: E731
    fr = np.tile(ref["forces"], (reps, 1))
    assert rms(fb - fr) <= 1e-5 * rms(np.abs(fr) + np.abs(qs[:, None]) * np.abs(ref["e_out"]).max())
