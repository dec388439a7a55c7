"""The kernels' sources hold no wait without a time limit.

A wait that never ends cannot be tested by running it, so this is read off the sources: grid-wide barriers of cooperative groups
have no limit and are not used, and every loop that polls a shared-memory barrier or a word in global memory looks at
the clock.
"""
import os
import re

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
