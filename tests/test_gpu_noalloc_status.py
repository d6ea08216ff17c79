"""pin_noalloc_status reads what the last call to have run recorded, also when a
call on another grid size has been captured into a graph since."""
import pytest

from paper_1305_1505_gb300 import ic, pin
from tests import parity

pytestmark = pytest.mark.gpu


def _buffers(n, seed):
    import torch
    dk = torch.from_numpy(parity.inputs(n, 2.0 * n, seed)[0]).cuda()
    return dk, torch.empty((n, n, n), dtype=torch.float32, device="cuda"), \
        torch.empty((n, n, n), dtype=torch.int32, device="cuda")


def _call(n, dk, F, I, stream):
    pin.pin_collapse_times_noalloc(dk.data_ptr(), pin.PIN_C64, n, 2.0 * n, ic.log_radii(2.0, 0.4 * n, 8), 1,
                                   F.data_ptr(), I.data_ptr(), stream.cuda_stream)


@pytest.mark.parametrize("n,other", [(64, 16), (16, 48), (32, 8)])
def test_status_of_the_last_call_that_ran(n, other):
    import torch
    stream = torch.cuda.Stream()
    a, b = _buffers(n, 21), _buffers(other, 22)
    torch.cuda.synchronize()
    _call(n, *a, stream)
    stream.synchronize()
    st, failed, counters = pin.pin_noalloc_status()
    assert (st, failed) == (pin.PIN_OK, 0) and counters[0] < n ** 3 and counters[2] == 0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        _call(other, *b, stream)
    # nothing has run since
    assert pin.pin_noalloc_status() == (st, failed, counters)
    graph.replay()
    torch.cuda.synchronize()
    F, I = b[1].clone(), b[2].clone()
    st2, failed2, counters2 = pin.pin_noalloc_status()
    assert (st2, failed2) == (pin.PIN_OK, 0) and counters2[2] == 0
    _call(other, *b, stream)
    stream.synchronize()
    assert torch.equal(F, b[1]) and torch.equal(I, b[2])
