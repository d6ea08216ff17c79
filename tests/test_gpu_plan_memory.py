"""A device that has no room for the spectra of a group of radii: the plan runs
one radius at a time, as every plan did that fitted there, with the same bits."""
import numpy as np
import pytest

from paper_1305_1505_gb300 import ic
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,left_mb", [(128, 240), (96, 160)])  # a group takes 372 and 347 MB, one radius 108 and 48
def test_a_full_device_takes_one_radius_at_a_time(n, left_mb):
    import torch
    from paper_1305_1505_gb300 import pin
    radii = ic.log_radii(2.0, 30.0, 12)
    dk = torch.from_numpy(parity.inputs(n, 2.0 * n, 11)[0]).cuda()

    def run():
        plan = pin.Plan(n, 2.0 * n, radii)
        try:
            plan.set_ic(dk)
            F, I = plan.collapse_times()
            o, c = plan.fragment_order()
            return F, I, o, c, pin.pin_kernels_per_call(plan.handle)
        finally:
            plan.close()

    ref = run()
    assert ref[4] < 4 * len(radii)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - (left_mb << 20), dtype=torch.uint8, device="cuda")
    try:
        left, _ = torch.cuda.mem_get_info()
        assert left < pin.pin_footprint_bytes(pin.make_desc(n, 2.0 * n, radii))
        got = run()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert got[4] == 4 * len(radii)
    assert all(torch.equal(a, b) for a, b in zip(got[:4], ref[:4]))
    assert (ref[1] >= 0).float().mean() > 0.05 and np.isfinite(ref[0].cpu().numpy()).all()
