"""A seeded request takes nothing over from the request before it: each
pin_set_ic_seed call evaluates the amplitude of its spectrum, also when the
plan has just used the same one."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# counts the calls of libpin to its amplitude function, which it reaches by name
COUNTER = """
#include "pin_ic.h"
static int calls;
int amplitude_calls(void) { return calls; }
double pin_ic_amplitude(const pin_spectrum* ps) { ++calls; return 1e4 * ps->sigma8; }
"""

CHILD = """
import ctypes, sys
counter = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
import torch
from paper_1305_1505_gb300 import pin
plan = pin.Plan(16, 32.0, [4.0, 2.0])
out = []
for sigma8 in (0.8, 0.8, 0.8, 0.9, 0.8):
    plan.set_ic_seed(7, sigma8=sigma8)
    out.append(counter.amplitude_calls())
plan.close()
print("calls", *out)
"""


def test_each_call_evaluates_its_amplitude(tmp_path):
    src, lib = tmp_path / "counter.c", tmp_path / "counter.so"
    src.write_text(COUNTER)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-o", str(lib), str(src)])
    p = subprocess.run([sys.executable, "-c", CHILD, str(lib)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    assert "calls 1 2 3 4 5" in p.stdout, p.stdout
