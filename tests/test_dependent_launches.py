"""Kernels launched with programmatic serialisation start while the kernel
before them in the stream may still be writing what they read.  A read-only load
(``__ldg``) asks for data that nothing writes for as long as the kernel runs, and
an ordinary load intrinsic may be moved over the wait; so in the sources of these
kernels every ``__ldg`` reads one of the plan's tables, and the caller's data
(transform, weights, scale) goes through ``ld_data``, which stays behind
``grid_wait``."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_06449_gb300", "csrc")
TABLES = {"a.tau", "a.lo", "a.hi", "args.frag", "args.lo", "args.hi", "a.twL", "args.twL"}


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _waiting():
    return sorted(n for n in os.listdir(CSRC)
                  if n.endswith((".cu", ".cuh")) and re.search(r"grid_wait\(\)|griddepcontrol\.wait", _source(n)))


def test_the_dependent_kernels_are_found():
    assert {"paco_fold.cuh", "paco_power.cuh", "paco_tcpass.cuh", "paco_cluster.cu"} <= set(_waiting())


@pytest.mark.parametrize("name", _waiting())
def test_read_only_loads_read_tables(name):
    src = _source(name)
    assert "__ldcg(" not in src and "__ldca(" not in src
    names = dict(re.findall(r"const \w+ \*(\w+) = reinterpret_cast<const \w+ \*>\(([\w.]+)\)", src))
    loads = re.findall(r"__ldg\(&?(?:reinterpret_cast<const \w+ \*>\()?([\w.]+)", src)
    assert loads
    for arg in loads:
        assert names.get(arg, arg) in TABLES, arg
