"""The kernels' sources hold no wait without a time limit, and no loop that goes on for as long as memory says so.

A wait that never ends cannot be tested by running it, so this is read off the sources: grid-wide barriers of cooperative groups
have no limit and are not used, and every loop that polls a shared-memory barrier or a word in global memory looks at
the clock.  The same goes for loops: after a sweep that gave up the kernels behind it run on whatever the workspace held, so each loop has a
limit in its head or uses up something that the thread holds.
"""
import os
import re

import numpy as np
import pytest

from paper_2601_17818_b200.build import CSRC

SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
POLL = re.compile(r"\bwhile \(.*(?:mbar_try_wait|ld_acquire_u32|load)\(|\bfor \([^;]*;\s*; \+\+it\)")


def _code(name):
    with open(os.path.join(CSRC, name)) as fh:
        return [re.sub(r"//.*", "", line) for line in fh]


@pytest.mark.parametrize("name", SOURCES)
def test_no_barrier_without_a_limit(name):
    code = "".join(_code(name))
    assert "cooperative_groups" not in code and not re.search(r"\bbarrier_wait\(|\bgrid\.sync\(", code)


def test_every_poll_looks_at_the_clock():
    polls = 0
    for name in SOURCES:
        code = _code(name)
        for i, line in enumerate(code):
            if POLL.search(line):
                polls += 1
                assert re.search(r"global_ns\(\)|%globaltimer", "".join(code[i:i + 7])), f"{name}:{i + 1}"
    assert polls == 4                                      # mbar_wait, mbar_drain, a factor, the grid's barrier


ENDLESS = re.compile(r"\bfor \([^;]*;\s*;|\bwhile \((?:true|1)\)")
# the blocks of a warp's lanes; the bits of a key and then of an index
USES_UP = {"nearest.cu": 1, "select.cu": 1, "vic_labels.cuh": 1}


def test_no_loop_without_a_limit():
    found = {}
    for name in SOURCES:
        loops = sum(1 for line in _code(name) if ENDLESS.search(line) and not POLL.search(line))
        if loops:
            found[name] = loops
    assert found == USES_UP


def test_rounds_of_the_chase_reach_every_root():
    """A host model of the chase of vic_labels.cuh on the longest possible chain (token i's parent is i - 1): what a token reads depends
    on its depth alone, so no forest needs more rounds."""
    source = "".join(_code("vic_labels.cuh"))
    steps, limit = (int(re.search(rf"\b{name} = (\d+)", source).group(1)) for name in ("kChase", "kChaseRounds"))
    n = 16384
    table = np.maximum(np.arange(n) - 1, 0)
    at, is_open, rounds = np.arange(n), np.ones(n, bool), 0
    while is_open.any():
        for _ in range(1, steps):
            at = np.where(is_open, table[at], at)
        is_open &= table[at] != at
        table = np.where(is_open, at, table)
        rounds += 1
    assert not at.any() and rounds <= limit
