"""FP32 direct sums of a salt listed pair by pair: the packed loop's lanes do not split it by sign."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# Each FP32 partial sum rounds at its own size.  Charges of alternating sign keep those sums at a few terms, random
# signs at the square root of their number; so the alternating order's error is no larger than a random order's (half
# again for the scatter of 300 targets).  The targets are away from the sources: beside them a few closest pairs, the
# same in every order, make up most of the field's error.
@pytest.mark.parametrize("away", [2.0, 20.0])
@pytest.mark.parametrize("n", [64, 250, 2000, 20001])
def test_alternating_charges_are_summed_as_well_as_random_ones(n, away):
    import torch

    from paper_1806_04801_gb300 import hsma

    g = np.random.default_rng(n)
    s, q = g.random((n, 3)), np.where(np.arange(n) % 2, -1.0, 1.0)
    t = torch.as_tensor(g.random((300, 3)) + [away, 0.0, 0.0]).cuda()
    mixed = g.permutation(n)
    err = {}
    for name, order in (("alternating", np.arange(n)), ("random", mixed)):
        src = torch.as_tensor(np.concatenate([s, q[:, None]], 1)[order]).cuda()
        pot, fld = hsma.coulomb_sum(src, t, field=True, precision="fp32")
        pot64, fld64 = hsma.coulomb_sum(src, t, field=True, precision="fp64")
        err[name] = ((pot - pot64).norm().item(), (fld - fld64).norm().item())
    assert err["alternating"][0] <= 1.5 * err["random"][0]
    assert err["alternating"][1] <= 1.5 * err["random"][1]
