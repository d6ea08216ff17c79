"""The z pass at every line family it runs (one, two and three levels, odd
factors, the longest two-level line) computes the collapse times of its lines
itself: against the oracle, and with the velocity fields against without."""
import numpy as np
import pytest

import oracle
from paper_1305_1505_gb300 import ic
from tests import parity
from tests.test_gpu_noncubic import _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [8, 48, 96, 192, 512])
def test_z_pass_line_sizes(nz):
    import torch
    from paper_1305_1505_gb300 import pin
    shape, box = (16, 32, nz), 32.0
    radii = ic.log_radii(1.0, 2.0 * min(shape) / 4, 5)
    d32, d64 = _field(shape, box, 90 + nz)
    out = []
    for vel in (False, True):
        plan = pin.Plan(shape, box, radii, velocities=vel)
        plan.set_ic(torch.from_numpy(d32).cuda())
        out.append([t.clone() for t in plan.collapse_times()])
        plan.close()
    (F, I), (Fv, Iv) = out
    assert torch.equal(F, Fv) and torch.equal(I, Iv)
    assert (I >= 0).float().mean() > 0.5
    orc = oracle.collapse_times(d64, box, radii, keep_all=True)
    parity.assert_parity(F.cpu().numpy(), I.cpu().numpy(), orc, d64, box, radii, label="nz %d" % nz)
