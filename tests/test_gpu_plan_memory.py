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


@pytest.mark.parametrize("n", [64, 128])
def test_fp64_plans_hold_only_what_their_loop_uses(n):
    import torch
    from paper_1305_1505_gb300 import pin
    pin.Plan(n, 2.0 * n, [4.0, 2.0], precision=pin.PIN_FP64).close()  # loads the kernels
    desc = pin.make_desc(n, 2.0 * n, [4.0, 2.0], precision=pin.PIN_FP64)
    need = pin.pin_footprint_within(desc, 0)
    single = pin.pin_footprint_within(pin.make_desc(n, 2.0 * n, [4.0, 2.0]), 0)
    # half-spectrum, twiddles, tensor, F_max
    assert need == single + 16 * (n * n * (n // 2 + 1) + 3 * n) + 56 * n ** 3
    assert need == pin.pin_footprint_within(desc, 1 << 62) < pin.pin_footprint_bytes(desc)
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    plan = pin.Plan(n, 2.0 * n, [4.0, 2.0], precision=pin.PIN_FP64)
    free1, _ = torch.cuda.mem_get_info()
    plan.close()
    assert free0 - free1 <= need + 15 * (2 << 20)  # fifteen arrays, each at most 2 MB over
