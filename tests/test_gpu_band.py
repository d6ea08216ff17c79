"""Modes that the filter takes to exactly zero are neither loaded nor
transformed: the tensor at radii from nothing filtered to everything filtered,
on lines whose bands end inside, at and next to a box of rows, against the
oracle; and a field that is not finite still spreads over the whole grid."""
import numpy as np
import pytest

import oracle
from paper_1305_1505_gb300 import ic
from tests.test_gpu_noncubic import _field

pytestmark = pytest.mark.gpu

RADII = (0.0, 2.0, 9.0, 11.0, 13.5, 17.0, 23.0, 37.0, 60.0, 110.0, 3000.0)
SHAPES = [((64, 64, 64), None, False), ((32, 96, 192), (32, 8), True), ((48, 16, 128), (0, 8), False),
          ((384, 8, 64), None, True), ((16, 384, 48), None, False), ((8, 32, 512), None, False)]


@pytest.mark.parametrize("radix", [0, 1])
@pytest.mark.parametrize("shape,tiles,vel", SHAPES)
def test_tensor_at_every_band(shape, tiles, vel, radix):
    import torch
    from paper_1305_1505_gb300 import pin
    box = 4.0 * shape[0]
    d32, d64 = _field(shape, box, 7)
    plan = pin.Plan(shape, box, RADII, velocities=vel)
    plan.set_radix(radix, radix)
    if tiles:
        plan.set_tiles(*(t if t in pin.pin_tile_options_radix(n, radix) else 0 for t, n in zip(tiles, shape)))
    # the workspaces start out full of NaN: nothing outside a band may be read
    nan = np.full_like(d32, np.nan)
    plan.set_ic(torch.from_numpy(nan).cuda())
    F, I = plan.collapse_times()
    assert (F == 0).all() and (I == -1).all()
    plan.set_ic(torch.from_numpy(d32).cuda())
    for s in reversed(range(len(RADII))):
        h = plan.hessian(s).double().cpu().numpy()
        ref, _ = oracle.hessian(d64, box, RADII[s])
        # FP32 transforms: 2e-5 of the rms; factors below 1e-38 are denormal
        assert np.abs(h - ref).max() <= 2e-5 * np.sqrt(np.mean(ref ** 2)) + 1e-30, RADII[s]
    plan.close()


def test_one_infinite_mode_spreads_at_every_radius():
    """A mode whose filter factor is zero at the larger radii: 0 x inf is NaN
    there too, and no particle collapses."""
    import torch
    from paper_1305_1505_gb300 import pin
    n, box = 64, 256.0
    d32, _ = _field((n, n, n), box, 9)
    d32[20, 21, 22] = np.inf
    plan = pin.Plan(n, box, [60.0, 30.0, 4.0])
    plan.set_ic(torch.from_numpy(d32).cuda())
    F, I = plan.collapse_times()
    assert (F == 0).all() and (I == -1).all()
    assert torch.isnan(plan.hessian(0)).all()
    plan.close()
