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
def table():
    return [[a, shape(*a)] for a in json.loads(sys.argv[2])]
first = table()
lib = ctypes.CDLL(sys.argv[1])
cfg = lib.bfhe_ntt_config
cfg.argtypes = [ctypes.c_uint32, ctypes.c_int, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_void_p, ctypes.c_void_p]
def config(logN, inv, log_m=0, log_e=0):
    m, e = ctypes.c_uint32(), ctypes.c_uint32()
    assert cfg(logN, inv, log_m, log_e, ctypes.byref(m), ctypes.byref(e)) == 0
    return m.value, e.value
same = []
for logN in range(10, 16):
    for inv in (0, 1):
        read = config(logN, inv)
        assert config(logN, inv, *read) == read
        same.append(table() == first)
        other = (logN - 1 if 10 < logN else logN, 4 if read != (logN - 1, 4) else 5)
        if other != read:   # an override holds for every launch until what was read is set again
            assert config(logN, inv, *other) == config(logN, inv) == other
            assert all(tuple(s) == other for a, s in table() if a[:2] == [logN, inv])
            assert config(logN, inv, *read) == read
            same.append(table() == first)
print(json.dumps([first, same]))
"""


@pytest.fixture(scope="module")
def child():
    """The library's own rule (not part of its ABI) as (logN, inverse, pm, limbs) -> (log_m, log_e), and whether it was the
    same after each time that a shape had been read and written back."""
    if not os.path.exists(build.lib_path()):
        build.build()
    args = [(logN, inv, pm, n) for logN in range(10, 16) for inv in (0, 1) for pm in (False, True) for n in LIMBS]
    env = {k: v for k, v in os.environ.items() if not k.startswith("BFHE_")}
    out = subprocess.run([sys.executable, "-c", CHILD, build.lib_path(), json.dumps(args)], env=env, check=True,
                         capture_output=True, text=True).stdout
    first, same = json.loads(out)
    return {tuple(a): tuple(s) for a, s in first}, same


@pytest.fixture(scope="module")
def shape(child):
    return lambda *a: child[0][a]


def test_writing_back_a_shape_keeps_the_rule(child):
    assert len(child[1]) >= 12 and all(child[1])


def test_the_tuner_leaves_the_rule_alone_on_a_near_tie():
    from paper_2204_12201_gb300.autotune import _pick
    t = {"13,5/13,5": 1.0, "14,5/14,5": 1.009, "13,4/14,5": 1.2}
    assert _pick(t, "14,5/14,5") == "14,5/14,5"
    assert _pick(t, "13,4/14,5") == "13,5/13,5"
    assert _pick(t, "15,5/15,5") == "13,5/13,5"


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
