"""The arithmetic that kernels and launchers share (csrc/launch_rules.h), compiled by itself for the host."""
import ctypes
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1412_7580_b200", "csrc")
EXPORTS = """
#include "launch_rules.h"
extern "C" void tc_share(int rows_a, int rows_b, int N, int k_blocks, long long tiles, int sms, long long* out) {
    const fc::TcShare s = fc::tc_share(rows_a, rows_b, N, k_blocks, tiles, sms);
    const long long v[6] = {s.per_sm, s.stages, s.ring_bytes, s.epi_bytes, s.smem, s.acc_cols};
    for (int i = 0; i < 6; ++i) out[i] = v[i];
}
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


def test_contraction_ctas_per_sm(rules):
    """Every CTA that shared memory admits to an SM also finds tensor memory; a stage's reads stay inside the CTA."""
    SM, RESERVED, SMS, TMEM, KB = 228 * 1024, 1024, 148, 512, 1024
    out = (ctypes.c_longlong * 6)()
    seen = set()
    for rows_a in range(8, 129, 8):
        for rows_b, N in ((r, n) for r in range(16, 129, 16) for n in (r - 15, r)):
            for k_blocks, tiles in itertools.product((1, 2), (1, SMS, SMS + 1, 2 * SMS, 2 * SMS + 1, 3 * SMS + 1, 10 ** 6)):
                rules.tc_share(rows_a, rows_b, N, k_blocks, ctypes.c_longlong(tiles), SMS, out)
                per_sm, stages, ring, epi, smem, acc = out
                a, b = 128 * rows_a, 128 * rows_b
                assert per_sm * (smem + RESERVED) <= SM and smem <= 227 * KB
                fit = SM // (smem + RESERVED)
                assert fit * 4 * acc <= TMEM and N <= acc           # not one that would wait for tensor memory
                assert per_sm == 1 or (fit == per_sm and (per_sm - 1) * SMS < tiles)
                assert stages == 4 or (per_sm > 1 and stages >= (3 if N > 32 and k_blocks > 1 else 2)) or (stages == 3 and 5 * 2 * (a + b) > smem)
                assert stages * 2 * (a + b) <= ring and ring + epi + 1536 <= smem
                # an MMA reads 128 rows of A_im of the last stage, and N rounded up to 16 rows of B_im
                assert (stages - 1) * 2 * (a + b) + a + 16 * KB <= ring + epi
                assert epi >= 2 * 4 * KB * -(-rows_a // 32)
                if N > 64:
                    assert (per_sm, ring, epi, acc) == (1, 3 * 64 * KB, 32 * KB, 128)
                seen.add(per_sm)
    assert seen == {1, 2, 3, 4}
