"""Host check of what the kernels may read through the non-coherent path.

A kernel of the library is resident while the one before it on the stream still runs (programmatic dependent launch), and
only the wait at its start orders the two.  `const ... __restrict__` and `__ldg` promise that a buffer does not change
for as long as the kernel is resident, and let the compiler load it ahead of that wait.  That holds for the tables made
with the context, for no buffer that a kernel writes: ciphertexts, scratch, keys.
"""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_12201_gb300", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
# twiddles, twists, mod-down constants, moduli, scaled plaintext units: uploaded when the context is made
TABLES = {"tw", "twc", "twl", "itw", "twist", "xtw", "mtw", "mpc", "qtab", "delta"}
# pointers into those tables, local to their kernels
INTO_TABLES = {"f": {"twist_at", "xtw", "mtw", "tw2"}}


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _base(expr):
    """The pointer an address expression starts from."""
    return re.match(r"(?:reinterpret_cast<[^>]*>\()?\(?\s*(\w+)", expr.strip()).group(1)


@pytest.mark.parametrize("name", SOURCES)
def test_only_tables_are_read_through_the_non_coherent_path(name):
    src = _source(name)
    for m in re.finditer(r"__restrict__\s+(\w+)", src):
        assert m.group(1) in TABLES, "%s: __restrict__ %s" % (name, m.group(1))
    for m in re.finditer(r"__ldg\(([^;]*)", src):
        base = _base(m.group(1))
        if base in INTO_TABLES:   # every definition of the local pointer starts at a table
            starts = set(re.findall(r"ulonglong2\s*\*\s*%s\s*=\s*(\w+)" % base, src))
            starts |= set(re.findall(r"ulonglong2\s+%s\s*=\s*(\w+)" % base, src))
            assert starts <= INTO_TABLES[base], (name, base, starts)
            continue
        assert base in TABLES, "%s: __ldg(%s" % (name, m.group(1)[:60])


@pytest.mark.parametrize("name", SOURCES)
def test_every_kernel_waits_before_it_reads(name):
    """Each __global__ body begins the wait itself, before any statement that loads through a pointer."""
    src = _source(name)
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", src):
        body = src[src.index("{", m.end()):]
        wait = re.search(r"\bpdl_(begin|wait)\(\)", body)
        assert wait, (name, m.group(1))
        head = body[:wait.start()]
        for read in re.findall(r"(\w[\w.]*)\[", head):   # declarations of arrays, and moduli
            assert read in {"x", "sm", "a.tab.q", "a.tab.mu", "tab.q"}, (name, m.group(1), read)
        assert "*reinterpret_cast" not in head and "__ldg" not in head, (name, m.group(1))
