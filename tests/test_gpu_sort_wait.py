"""The particle order when its blocks' waits for one another run out: the
failure is reported once, the outputs stay inside their buffers, and the plan
gives the right order again afterwards."""
import numpy as np
import pytest

from paper_1305_1505_gb300 import ic
from tests import parity

pytestmark = pytest.mark.gpu

GUARD = 4096


@pytest.mark.parametrize("n", [32, 128])  # 4 tiles, and 256 on as many blocks at once
def test_waits_run_out_and_the_plan_recovers(n):
    import torch
    from paper_1305_1505_gb300 import pin
    plan = pin.Plan(n, 2.0 * n, ic.log_radii(2.0, 20.0, 6), stream=torch.cuda.Stream())
    plan.set_ic(torch.from_numpy(parity.inputs(n, 2.0 * n, 5)[0]).cuda())
    F, _ = plan.collapse_times()
    ref, _ = plan.fragment_order()
    out = torch.empty(n ** 3 + 2 * GUARD, dtype=torch.int32, device="cuda")
    gave_up = 0
    pin.pin_set_wait_budget(plan.handle, 1)  # no poll after the first look
    for _ in range(8):
        out.fill_(-7)
        torch.cuda.synchronize()
        pin.pin_fragment_order(plan.handle, out[GUARD:].data_ptr(), 0, 1)
        st = pin.pin_sync(plan.handle, -1)
        body = out[GUARD:-GUARD]
        assert (out[:GUARD] == -7).all() and (out[-GUARD:] == -7).all()
        assert ((body >= 0) & (body < n ** 3) | (body == -7)).all()
        if st == pin.PIN_OK:  # every count had arrived
            assert torch.equal(body, ref)
        else:
            assert st == pin.PIN_ECUDA, pin.pin_strerror(st)
            assert pin.pin_sync(plan.handle, -1) == pin.PIN_OK  # reported once
            gave_up += 1
    if n == 128:
        assert gave_up > 0
    pin.pin_set_wait_budget(plan.handle, 0)
    o, _ = plan.fragment_order()
    assert torch.equal(o, ref)
    assert np.array_equal(F.cpu().numpy().ravel()[o.cpu().numpy()], np.sort(F.cpu().numpy().ravel())[::-1])
    plan.close()


def test_the_failure_names_the_call_that_gave_up():
    import torch
    from paper_1305_1505_gb300 import pin
    n = 128
    plan = pin.Plan(n, 2.0 * n, [8.0, 2.0], stream=torch.cuda.Stream())
    plan.set_ic(torch.from_numpy(parity.inputs(n, 2.0 * n, 5)[0]).cuda())
    plan.collapse_times()
    order = torch.empty(n ** 3, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    pin.pin_set_wait_budget(plan.handle, 1)
    for _ in range(8):
        pin.pin_fragment_order(plan.handle, order.data_ptr(), 0, 1)
        if pin.pin_sync(plan.handle, -1) == pin.PIN_ECUDA:
            break
    else:
        pytest.fail("no wait ran out")
    msg = pin.pin_last_error(plan.handle)
    assert "order" in msg and "transfer" not in msg, msg
    # a failed radius loop before the order: the loop's failure is the one reported
    plan.collapse_times(sync=False)
    pin.pin_fragment_order(plan.handle, order.data_ptr(), 0, 1)
    assert pin.pin_sync(plan.handle, -1) == pin.PIN_ECUDA
    assert "transfer" in pin.pin_last_error(plan.handle)
    plan.close()
