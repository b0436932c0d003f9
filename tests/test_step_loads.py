"""Loads in kernels that come up while their predecessor still writes.

A kernel that calls ``step_begin`` may be resident before the kernel in front of
it has ended. Read-only loads are defined only for data that nothing writes
while the reading kernel runs, and the compiler may move them over the wait, so
such a kernel reads what a step produces (fields, forces, populations, clocks)
with ordinary loads: ``__ldg`` is left to the slit tables, and no argument is a
``const __restrict__`` pointer, from which the compiler makes read-only loads
by itself.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0712_2247_gb300", "csrc")
TABLES = ("P.zslit", "P.done")  # written by the host between steps only


def source(name):
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", s)


def closing(s, i, pair="{}"):
    """Index past the bracket that closes the one at s[i]."""
    depth = 0
    for k in range(i, len(s)):
        depth += (s[k] == pair[0]) - (s[k] == pair[1])
        if depth == 0:
            return k + 1
    raise ValueError("unbalanced")


def kernels(s):
    """(name, arguments, body) of every kernel defined in s."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*(?=\())?", s):
        i = m.end()
        if s[i] == "(":
            i = closing(s, i, "()")
        name = re.match(r"\s*(\w+)\s*", s[i:])
        a = i + name.end()
        e = closing(s, a, "()")
        b = s.index("{", e)
        yield name.group(1), s[a:e], s[b:closing(s, b)]


FILES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
OVERLAPPING = [(f, k) for f in FILES for k in kernels(source(f)) if "step_begin(" in k[2]]


def test_the_kernels_of_a_step_are_found():
    names = {k[0] for _, k in OVERLAPPING}
    assert {"k_tick", "k_ball", "k_ball_tma", "k_ball_direct", "k_force", "k_force4", "k_pull_pair",
            "k_pull_block"} <= names


@pytest.mark.parametrize("kernel", [k for _, k in OVERLAPPING], ids=[k[0] for _, k in OVERLAPPING])
def test_waits_first_and_takes_no_read_only_argument(kernel):
    name, args, body = kernel
    first = next(t for t in (x.strip() for x in body[1:].split(";")) if t and not t.startswith("constexpr"))
    assert first.startswith("step_begin("), name
    for a in args[1:-1].split(","):
        assert not ("const" in a and "__restrict__" in a), (name, a.strip())
    for m in re.finditer(r"__ldg\s*\(\s*([^,)]*)", body):
        assert m.group(1).startswith(TABLES), (name, m.group(0))


@pytest.mark.parametrize("name", ["lbif_device.cuh", "lbif_force.cu", "lbif_pull.cu"])
def test_helpers_read_step_data_with_ordinary_loads(name):
    """The files whose device functions the step's kernels are made of."""
    s = source(name)
    for m in re.finditer(r"__ldg\s*\(\s*([^,)]*)", s):
        assert m.group(1).startswith(TABLES), m.group(0)
    assert "ld.global.nc" not in s
    for m in re.finditer(r"\([^(){};]*\)\s*\{", s):
        for a in m.group(0).split(","):
            assert not ("const" in a and "__restrict__" in a and "*" in a), a.strip()
