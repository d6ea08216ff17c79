"""Radius groups: on small grids one launch covers several radii and keeps the
running maximum in a packed word.  A plan with velocities never groups, and
its F_max and index are computed by the same arithmetic one radius at a time,
so the two agree bit for bit, whatever the number and order of the radii."""
import numpy as np
import pytest

from tests.test_gpu_noncubic import _field

pytestmark = pytest.mark.gpu


def _both(shape, radii, delta, batch=1, correction=1):
    import torch
    from paper_1305_1505_gb300 import pin
    out = []
    for vel in (False, True):
        plan = pin.Plan(shape, 2.0 * shape[0], radii, batch=batch, velocities=vel, correction=correction)
        plan.set_ic(torch.from_numpy(delta).cuda())
        plan.collapse_times()
        out.append([t.clone() for t in plan.collapse_times()])  # a second call on the same buffers
        out[-1].append(pin.pin_kernels_per_call(plan.handle))
        plan.close()
    return out


@pytest.mark.parametrize("shape,counts", [((16, 16, 16), (1, 15, 16, 17, 64)), ((64, 64, 64), (5, 6, 7, 20)),
                                          ((8, 128, 48), (2, 33)), ((96, 96, 96), (3, 4)), ((48, 32, 64), (11,))])
def test_groups_match_single_radii(shape, counts):
    import torch
    d32, _ = _field(shape, 2.0 * shape[0], 61)
    for s in counts:
        radii = np.geomspace(2.0, max(2.0, 0.5 * min(shape)), s)
        np.random.default_rng(s).shuffle(radii)
        radii[s // 2] = radii[0]  # a tie: the lower index wins
        (F, I, k), (Fv, Iv, kv) = _both(shape, radii, d32, correction=s % 2)
        assert torch.equal(F, Fv) and torch.equal(I, Iv)
        assert (I >= 0).float().mean() > 0.5
        assert kv == 4 * s and (s == 1 or k < kv)


def test_groups_of_a_batch_and_of_degenerate_fields():
    import torch
    shape, radii = (16, 32, 24 * 2), np.geomspace(2.0, 8.0, 9)
    d = np.stack([_field(shape, 32.0, 70 + b)[0] for b in range(5)])
    (F, I, _), (Fv, Iv, _) = _both(shape, radii, d, batch=5)
    assert torch.equal(F, Fv) and torch.equal(I, Iv)
    for fill in (0.0, np.nan, np.inf):  # every particle near-degenerate; nothing finite
        (F, I, _), (Fv, Iv, _) = _both(shape, radii, np.full_like(d[0], fill))
        assert torch.equal(F, Fv) and torch.equal(I, Iv)
        assert (F == 0).all() and (I == -1).all()
