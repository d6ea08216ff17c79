"""Memory budgets and groups of radii: what a plan takes within a number of
bytes, and that a server's budget still admits the requests, and as many of
them at once, as it does with one radius at a time."""
import threading
import time

import pytest

from paper_1305_1505_gb300 import pin, serve

SINGLE = {64: 20e6, 96: 50e6, 128: 110e6}  # one radius at a time, rounded up


def _desc(n, **kw):
    return pin.make_desc(n, 2.0 * n, [8.0, 4.0], **kw)


@pytest.mark.parametrize("n", [8, 64, 96, 128, 192, (64, 32, 128)])
def test_footprint_within(n):
    d = _desc(n) if not isinstance(n, tuple) else pin.make_desc(n, 128.0, [8.0])
    full, least = pin.pin_footprint_bytes(d), pin.pin_footprint_within(d, 0)
    assert 0 < least <= full
    assert (least < full) == (max(n if isinstance(n, tuple) else (n,)) <= 128)
    if n in SINGLE:
        assert least < SINGLE[n] < full
    last = least
    for k in range(41):
        limit = least + (full - least) * k // 40
        got = pin.pin_footprint_within(d, limit)
        assert last <= got <= limit
        last = got
    assert last == full == pin.pin_footprint_within(d, 1 << 62)
    assert pin.pin_footprint_within(d, least - 1) == least
    d.nscales = 0
    assert pin.pin_footprint_within(d, 1 << 62) == 0


class Engine(serve.PinEngine):
    """PinEngine's accounting without a device."""

    def __init__(self):
        self.lock, self.active, self.peak = threading.Lock(), 0, 0

    def run(self, req, timeout_s=None):
        with self.lock:
            self.active += 1
            self.peak = max(self.peak, self.active)
        time.sleep(0.05)
        with self.lock:
            self.active -= 1
        return req.footprint


@pytest.mark.parametrize("n,budget,at_once", [(64, 100 << 20, 4), (64, 20 << 20, 1), (96, 200 << 20, 4),
                                              (128, 330 << 20, 3)])
def test_a_budget_admits_what_it_did(n, budget, at_once):
    least = pin.pin_footprint_within(_desc(n), 0)
    assert min(4, budget // least) == at_once  # by one radius at a time
    eng = Engine()
    srv = serve.Server(eng, budget, max_slots=4)
    reqs = [srv.submit(serve.Request(i, n, 2.0 * n, i, [8.0, 4.0])) for i in range(3 * at_once)]
    assert srv.drain(timeout=30)
    srv.close()
    assert all(r.status == "done" for r in reqs), [r.error for r in reqs]
    assert eng.peak == at_once and srv.peak_in_use <= budget


def test_a_large_budget_keeps_the_groups():
    eng = Engine()
    srv = serve.Server(eng, 8 << 30, max_slots=4)
    r = srv.submit(serve.Request(0, 64, 128.0, 1, [8.0, 4.0]))
    assert srv.drain(timeout=10)
    srv.close()
    assert r.result == pin.pin_footprint_bytes(_desc(64))


@pytest.mark.gpu
def test_plans_within_a_budget_give_the_same_bits():
    import torch

    from paper_1305_1505_gb300 import ic
    from tests import parity
    n, radii = 64, ic.log_radii(2.0, 24.0, 20)
    dk = torch.from_numpy(parity.inputs(n, 2.0 * n, 3)[0]).cuda()
    least, full = pin.pin_footprint_within(_desc(n), 0), pin.pin_footprint_bytes(_desc(n))
    out, launches = [], []
    for limit in (None, (least + full) // 2, least, 0):
        plan = pin.Plan(n, 2.0 * n, radii, max_bytes=limit)
        plan.set_ic(dk)
        out.append(plan.collapse_times())
        launches.append(pin.pin_kernels_per_call(plan.handle))
        plan.close()
    assert launches == sorted(launches) and launches[0] < launches[1] < launches[2] == launches[3] == 4 * 20
    assert all(torch.equal(F, out[0][0]) and torch.equal(I, out[0][1]) for F, I in out)
