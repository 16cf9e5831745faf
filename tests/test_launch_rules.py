"""The arithmetic that kernels and launchers share (csrc/launch_rules.h), compiled by itself for the host."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1412_7580_b200", "csrc")
EXPORTS = """
#include "launch_rules.h"
extern "C" int ring_uses(long long requested, int slot, int slots) { return fc::ring_uses(requested, slot, slots); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch_rules")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text(EXPORTS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("slots", [1, 2, 3, 6])
def test_ring_drain_waits_for_the_last_request_of_every_slot(rules, slots):
    """A barrier whose phase k completes when its k-th request has landed: for every number of requests, the parity
    that the drain waits for is passed exactly when nothing is in flight into the slot any more."""
    for requested in range(0, 5 * slots + 2):
        per_slot = [0] * slots
        for r in range(requested):
            per_slot[r % slots] += 1
        for s in range(slots):
            uses = rules.ring_uses(ctypes.c_longlong(requested), s, slots)
            assert uses == per_slot[s]
            if uses:
                parity = (uses - 1) & 1
                for landed in (uses - 1, uses):     # earlier ones were consumed before the slot was asked for again
                    passed = (landed & 1) != parity         # a wait on `parity` returns once that phase is over
                    assert passed == (landed == uses)
