"""The particle order over every number of passes: F_max whose bits span one
value up to nearly all of FP32, at both sides of each width of key that takes
another pass, on one tile, whole tiles and part tiles, with ties and
never-collapsed particles, against numpy's lexsort."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
OUT = os.path.join(ROOT, "paper_1305_1505_gb300", "_build", "libsort_device.so")

# the largest key: (widest bits of F) - (narrowest) + 1
TOPS = {1: (1, 2, 2 ** 9 - 1), 2: (2 ** 9, 2 ** 17, 2 ** 18 - 1), 3: (2 ** 18, 2 ** 26 + 5, 2 ** 27 - 1),
        4: (2 ** 27, 2 ** 28 + 3, 0x7f000000)}


@pytest.fixture(scope="module")
def lib():
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1305_1505_gb300", "csrc"),
                           "-o", OUT, os.path.join(HERE, "sort_device.cu")])
    L = ctypes.CDLL(OUT)
    p, i = ctypes.c_void_p, ctypes.c_int
    L.dev_order.argtypes = [p, i, i, i, p, p, p]
    return L


def _field(rng, n, top, zeros, ties):
    """n values of F whose non-zero bits run over top - 1 steps down from a
    value, both ends present."""
    umax = 0x7f7fffff if top > 2 ** 29 else 0x40000000 + rng.integers(1000)
    key = rng.integers(0, top, size=n)
    if ties:
        key = key[rng.integers(0, max(1, n // 50), size=n)]
    key[rng.integers(n)] = 0
    key[(np.flatnonzero(key == 0)[0] + 1) % n] = top - 1
    u = (umax - key).astype(np.uint32)
    if zeros:
        z = rng.random(n) < 0.3
        z[np.flatnonzero(key == 0)[0]] = z[np.flatnonzero(key == top - 1)[0]] = False
        u[z] = 0
    return u.view(np.float32)


@pytest.mark.parametrize("passes", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [(8, 8, 8), (32, 32, 8), (32, 32, 12), (48, 64, 96)])
def test_every_number_of_passes(lib, passes, shape):
    n = int(np.prod(shape))
    for t, top in enumerate(TOPS[passes]):
        for zeros in (False, True):
            rng = np.random.default_rng([passes, n, t, zeros])
            F = _field(rng, n, top, zeros, ties=t == 1).reshape(shape)
            nz = F[F > 0].view(np.uint32)
            span = int(nz.max() - nz.min()) + 1
            assert span == top and -(-span.bit_length() // 9) == passes
            order, nb, width = np.empty(n, np.int32), np.empty(n, np.uint8), ctypes.c_int(0)
            got = lib.dev_order(F.ctypes.data, *shape, order.ctypes.data, nb.ctypes.data, ctypes.byref(width))
            assert got == passes and width.value == -(-span.bit_length() // passes)
            oref, cref = oracle.fragment_order(F)
            assert np.array_equal(order, oref)
            assert np.array_equal(nb.astype(np.int64).reshape(shape), cref)


def test_all_zero(lib):
    n = 32 * 32 * 12
    F = np.zeros((32, 32, 12), np.float32)
    order, nb, width = np.empty(n, np.int32), np.empty(n, np.uint8), ctypes.c_int(0)
    assert lib.dev_order(F.ctypes.data, 32, 32, 12, order.ctypes.data, nb.ctypes.data, ctypes.byref(width)) == 1
    assert np.array_equal(order, np.arange(n))
