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
    from gpu_common import assert_within, errors
    dx, dq = torch.as_tensor(xyz).cuda(), torch.as_tensor(q).cuda()
    U0, F0, _, _ = ref.energy_forces(dx, dq)
    U1, F1, _, _ = pl.energy_forces(dx, dq)
    assert_within(errors(F1.cpu().numpy(), F0.cpu().numpy(), U1, U0), "fp64" if precision == "fp64" else "fp32", what)


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
