"""Host check of the rule that gives a transform's launch its block shape."""

import json
import os
import subprocess
import sys

import pytest

from paper_2204_12201_gb300 import build

LARGE = 1 << 30
LIMBS = (1, 76, 77, 152, 153, LARGE)
# in a process of its own, where nothing has overridden a shape
CHILD = """
import ctypes, json, sys
fn = ctypes.CDLL(sys.argv[1])._Z10ntt_configiibmPiS_   # ntt_config(int, int, bool, size_t, int*, int*)
fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_bool, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p]
def shape(*a):
    m, e = ctypes.c_int(), ctypes.c_int()
    assert fn(*a, ctypes.byref(m), ctypes.byref(e)) == 0
    return m.value, e.value
print(json.dumps([[a, shape(*a)] for a in json.loads(sys.argv[2])]))
"""


@pytest.fixture(scope="module")
def shape():
    """The library's own rule (not part of its ABI): (logN, inverse, pm, limbs) -> (log_m, log_e)."""
    if not os.path.exists(build.lib_path()):
        build.build()
    args = [(logN, inv, pm, n) for logN in range(10, 16) for inv in (0, 1) for pm in (False, True) for n in LIMBS]
    env = {k: v for k, v in os.environ.items() if not k.startswith("BFHE_")}
    out = subprocess.run([sys.executable, "-c", CHILD, build.lib_path(), json.dumps(args)], env=env, check=True,
                         capture_output=True, text=True).stdout
    table = {tuple(a): tuple(s) for a, s in json.loads(out)}
    return lambda *a: table[a]


@pytest.mark.parametrize("inverse", [0, 1])
@pytest.mark.parametrize("logN", [10, 11, 12, 13, 14, 15])
def test_large_launches(shape, logN, inverse):
    """One shape per ring degree and direction; the forward at N = 16384 alone differs between the products."""
    want = {10: (10, 4), 11: (11, 4), 12: (12, 4), 13: (13, 5), 14: (14, 5), 15: (14, 5)}[logN]
    assert shape(logN, inverse, True, LARGE) == want
    assert shape(logN, inverse, False, LARGE) == ((13, 5) if logN == 14 and not inverse else want)


@pytest.mark.parametrize("pm", [True, False])
def test_small_launches(shape, pm):
    """Launches whose halves fit the SMs at one block each take halves of 16 words."""
    assert shape(14, 0, pm, 76) == shape(14, 1, pm, 76) == (13, 4)
    assert shape(14, 0, pm, 77) == shape(14, 0, pm, LARGE) and shape(14, 1, pm, 77) == (14, 5)
    assert shape(13, 0, pm, 76) == (12, 4) and shape(13, 0, pm, 77) == (13, 5)
    assert shape(13, 1, pm, 152) == (13, 4) and shape(13, 1, pm, 153) == (13, 5)
