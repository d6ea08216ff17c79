"""The particle order at the edges of the sort: one tile and several, part
tiles, key ranges from one value to all of FP32 (one to four passes), heavy
ties, never-collapsed particles, an unaligned count output, host outputs."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_noncubic import _field

pytestmark = pytest.mark.gpu


def _order(shape, delta, radii, **kw):
    import torch
    from paper_1305_1505_gb300 import pin
    plan = pin.Plan(shape, 2.0 * shape[0], radii, **kw)
    plan.set_ic(torch.from_numpy(delta).cuda())
    F, _ = plan.collapse_times()
    o, c = plan.fragment_order()
    again = plan.fragment_order()
    assert torch.equal(again[0], o) and torch.equal(again[1], c)
    # host outputs, the counts at an odd address
    n3 = int(np.prod(shape))
    ho, hc = np.empty(n3, np.int32), np.empty(n3 + 1, np.uint8)
    pin.pin_fragment_order(plan.handle, ho.ctypes.data, hc.ctypes.data + 1, 0)
    dc = torch.empty(n3 + 1, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    pin.pin_fragment_order(plan.handle, 0, dc.data_ptr() + 1, 1)
    plan.sync()
    assert np.array_equal(ho, o.cpu().numpy()) and np.array_equal(hc[1:], c.cpu().numpy().ravel())
    assert torch.equal(dc[1:], c.reshape(-1))
    plan.close()
    return F.cpu().numpy(), o.cpu().numpy(), c.cpu().numpy()


@pytest.mark.parametrize("shape,vel", [((8, 8, 8), False), ((8, 8, 8), True), ((16, 32, 16), False),
                                       ((32, 16, 24 * 2), False), ((64, 48, 96), True), ((192, 16, 128), False)])
def test_order_matches_lexsort(shape, vel):
    d, _ = _field(shape, 2.0 * shape[0], 33)
    for radii in ([2.0], [1.0, 0.5 * min(shape)]):
        F, o, c = _order(shape, d, radii, velocities=vel)
        oref, cref = oracle.fragment_order(F)
        assert np.array_equal(o, oref) and np.array_equal(c.astype(np.int64), cref)


@pytest.mark.parametrize("scale", [0.0, 1e-12, 1.0, 1e12])
def test_key_ranges(scale):
    """Fields whose F_max spans nothing, a few octaves, or (one plane wave
    times a steep envelope) very many."""
    shape = (32, 32, 32)
    d, _ = _field(shape, 64.0, 34)
    d = (d * scale).astype(np.complex64)
    F, o, c = _order(shape, d, [2.0, 6.0])
    oref, cref = oracle.fragment_order(F)
    assert np.array_equal(o, oref) and np.array_equal(c.astype(np.int64), cref)


def test_wide_range_of_values():
    """One mode along z: F falls through every octave towards the nodes."""
    shape = (16, 16, 768)
    d = np.zeros((16, 16, 385), np.complex64)
    d[0, 0, 1] = 16 * 16 * 768
    d[1, 0, 0] = d[-1, 0, 0] = 1e-9
    F, o, c = _order(shape, d, [1.0])
    assert F.max() > 0 and (F[F > 0].min() < 1e-3 * F.max() or (F == 0).any())
    oref, cref = oracle.fragment_order(F)
    assert np.array_equal(o, oref) and np.array_equal(c.astype(np.int64), cref)
