"""In-set reuse on one plan whose skin, or number of particles, changes between steps."""
import numpy as np
import pytest

from paper_1806_04801_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BOX = (1.0, 1.0, 1.0)


def _plan(R, precision):
    from paper_1806_04801_gb300 import hsma
    return hsma.Plan(BOX, I.PERIODIC, 8, R, 2000, 600, precision=precision)


def _check(ref, pl, xyz, q, precision, what):
    import torch
    from gpu_common import TOL, assert_within, errors, rel_energy_err
    dx, dq = torch.as_tensor(xyz).cuda(), torch.as_tensor(q).cuda()
    U0, F0, _, _ = ref.energy_forces(dx, dq)
    U1, F1, _, _ = pl.energy_forces(dx, dq)
    assert_within(errors(F1.cpu().numpy(), F0.cpu().numpy()), precision, what)
    assert rel_energy_err(U1, U0, q) <= TOL[precision]["energy"], what


# R = 1.45: the candidates of a skin of 0.1 need a shell of images more than those of 0.01 and 0.04 (1.45 + 0.1 above
# 1.5 box lengths); R = 1.5: all skins need the same shells.
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("R", [1.45, 1.5])
def test_steps_across_changes_of_the_skin(R, precision):
    xyz, q = I.uniform_pm1(2500, BOX, seed_offset=434)
    g = np.random.default_rng(435)
    with _plan(R, precision) as ref, _plan(R, precision) as pl:
        expect = {"builds": 0, "reuses": 0, "stale": 0}
        for skin in (0.01, 0.1, 0.01, 0.04, 0.0, 0.1):
            pl.set_inset_skin(skin)
            d = g.standard_normal(xyz.shape)
            d *= 0.9 * skin / np.linalg.norm(d, axis=1)[:, None]
            for k in range(3):
                _check(ref, pl, np.mod(xyz + 0.5 * k * d, 1.0), q, precision, f"skin {skin}, step {k}")
            expect["builds"] += skin > 0.0
            expect["reuses"] += 2 * (skin > 0.0)
            assert pl.inset_stats() == expect


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_steps_of_several_sizes_with_one_skin(precision):
    skin, g = 0.05, np.random.default_rng(436)
    with _plan(1.5, precision) as ref, _plan(1.5, precision) as pl:
        pl.set_inset_skin(skin)
        for i, n in enumerate((2500, 700, 1801, 2500)):
            xyz, q = I.uniform_pm1(n, BOX, seed_offset=437)
            d = g.standard_normal(xyz.shape)
            d *= 0.9 * skin / np.linalg.norm(d, axis=1)[:, None]
            for k in range(3):
                _check(ref, pl, np.mod(xyz + 0.5 * k * d, 1.0), q, precision, f"n {n}, step {k}")
            assert pl.inset_stats() == {"builds": i + 1, "reuses": 2 * i + 2, "stale": 0}
