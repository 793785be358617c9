"""Kernels started by programmatic dependent launch are resident while their
predecessor still writes, so their read-only loads (`const ... __restrict__`
parameters, __ldg) may only name the plan's constant tables."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2106_12487_gb300", "csrc")
FILES = ["passes.cuh", "fpasses.cuh", "vec.cuh", "cg.cuh"]
CONSTANT = {"twz", "twa", "twx", "tw", "ids", "tab", "Cg", "Cpk"}   # twiddles, grain ids, material tables


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def closing(s, i, pair):
    """Index of the bracket that closes s[i]."""
    depth = 0
    for j in range(i, len(s)):
        depth += (s[j] == pair[0]) - (s[j] == pair[1])
        if depth == 0:
            return j
    raise AssertionError("unbalanced source")


def functions(s):
    """(name, parameter list, body) of every kernel and device function."""
    for m in re.finditer(r"__(?:global|device)__[^;{}=]*?\b(\w+)(?=\([^()]*(?:\([^()]*\)[^()]*)*\)\s*\{)", s):
        a = m.end()
        b = closing(s, a, "()")
        c = s.index("{", b)
        yield m.group(1), s[a + 1:b], s[c:closing(s, c, "{}") + 1]


def read_only(params):
    return set(re.findall(r"const\s+[\w:<>]+\s*\*\s*__restrict__\s+(\w+)", params))


@pytest.mark.parametrize("name", FILES)
def test_dependent_kernels_promise_read_only_for_constants_only(name):
    found = list(functions(source(name)))
    kernels = [f for f in found if "pdl_wait()" in f[2]]
    if name in ("passes.cuh", "fpasses.cuh", "vec.cuh"):
        assert len(kernels) >= 3        # the parser sees them
    for kernel, params, _ in kernels:
        assert read_only(params) <= CONSTANT, kernel
    # what they call
    if name != "vec.cuh":
        for func, params, body in found:
            assert read_only(params) <= CONSTANT, func
            for arg in re.findall(r"\b(?:__ldg|ldg_t|ldg_pair)\((?:reinterpret_cast<[^>]*>\()?\s*(\w+)", body):
                assert arg in CONSTANT, (func, arg)


def test_every_dependent_launch_waits():
    """Each kernel that is started as a dependent waits for its predecessor."""
    text = {f: source(f) for f in FILES}
    waits = {k for s in text.values() for k, _, body in functions(s) if "pdl_wait()" in body}
    started = set()
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            started |= set(re.findall(r"launch_pdl\(\s*(k_\w+)", source(f)))
    assert started and started <= waits
