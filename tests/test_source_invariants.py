"""Invariants of the CUDA sources that no run on a single shape would catch.

A kernel launched with the stream-serialization attribute may start before its predecessor has
finished; it is only ordered after it by its own `dep_wait()`.  A kernel that is launched through
`dep_launch` and never waits would silently race with the previous kernel of the stream, and so
would every later kernel that relies on it for transitive ordering.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1412_7580_b200", "csrc")


def kernels_of(text):
    """(name, body) of every __global__ kernel: the body runs to the next kernel or launcher."""
    parts = re.split(r"\n__global__ ", text)
    out = []
    for chunk in parts[1:]:
        m = re.search(r"([A-Za-z_0-9]*_kernel)\s*\(", chunk)
        end = chunk.find("\nstatic ")
        out.append((m.group(1), chunk if end < 0 else chunk[:end]))
    return out


def test_every_kernel_launched_as_a_dependent_waits_for_its_predecessor():
    checked = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")) or name == "dep_launch.cuh":
            continue
        text = open(os.path.join(CSRC, name)).read()
        if "dep_launch(" not in text:
            assert "dep_wait()" not in text
            continue
        for kern, body in kernels_of(text):
            assert "dep_wait();" in body, f"{name}: {kern} is launched through dep_launch but never waits"
            assert "dep_trigger();" in body, f"{name}: {kern} never lets its dependents start"
            first_wait = body.index("dep_wait();")
            # no global-memory traffic before the wait: none of the access helpers may appear above it
            head = body[:first_wait]
            for token in ("__ldg(", "tma_load", "tma_store", "fk_tma_", "fk_cp16(", "cp.async", "atomic"):
                if token in head:
                    # lambdas defined above the wait may name these; they must not be *called* there:
                    # a call outside a lambda body sits at brace depth 1 of the kernel
                    depth, i, offending = 0, 0, False
                    while i < len(head):
                        c = head[i]
                        if c == "{":
                            depth += 1
                        elif c == "}":
                            depth -= 1
                        elif head.startswith(token, i) and depth <= 1:
                            offending = True
                            break
                        i += 1
                    assert not offending, f"{name}: {kern} touches global memory ({token}) before dep_wait()"
            checked += 1
    assert checked >= 6      # forward and inverse transforms, three contractions


def test_plain_launch_syntax_is_not_mixed_into_files_with_dependent_launches():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if "dep_launch(" in text and name != "dep_launch.cuh":
            assert "<<<" not in text, f"{name}: a kernel here bypasses dep_launch"


def test_no_wait_runs_out_in_silence():
    """A bounded wait on an asynchronous copy that gives up without raising the status word leaves outputs unwritten
    behind a call that returned OK.  So the kernels wait through fk_wait_or_report (or, after it has reported, drain
    with the result ignored), and the 1-D transforms, which have no status word, have no wait that can run out."""
    bare = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if name == "fft_kernels.cuh":
            a = text.index("__device__ __forceinline__ bool fk_mbar_wait(")
            b = text.index("__device__ __forceinline__ void fk_bulk_g2s(")
            assert text[a:b].count("fk_mbar_wait(") == 3       # its definition, and twice in fk_wait_or_report
            text = text[:a] + text[b:]
        for m in re.finditer(r"(\(void\))?\bfk_mbar_wait\(", text):
            assert m.group(1), f"{name}: a wait that can run out without a report"
        if "struct Fft1dParams" in text:
            bare += 1
            code = re.sub(r"//[^\n]*", "", text)
            assert "status" not in code and "mbar" not in code
    assert bare == 1


def test_outputs_written_before_the_last_input_is_read_are_early_clobbers():
    """A predicated load that zeroes its destination first (mov, then @p ld from an address operand) may only have an
    output that shares no register with the address: "=&"."""
    checked = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r'asm volatile\("([^;]|;(?!\s*$))*?;\s*$', text, re.M):
            stmt = m.group(0)
            first = re.search(r"mov\.b(?:32|64) %0, 0;", stmt)
            if first and re.search(r"ld\.[a-z.]+b?\d+ %0, \[%[1-9]", stmt[first.end():]):
                assert re.search(r':\s*"=&[a-z]"', stmt), f"{name}: {stmt}"
                checked += 1
    assert checked >= 4


def lambdas_of(text):
    """(name, body) of every named lambda."""
    for m in re.finditer(r"\bauto\s+(\w+)\s*=\s*\[&\][^{;]*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


def test_no_block_barrier_under_a_condition_that_differs_between_warps():
    """__syncthreads() is defined only where the whole block takes the same path to it; a step that some warps run in
    another form than the others has to meet at a barrier outside the branch (or at a numbered one)."""
    branches = 0
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        bodies = {}
        for lam, body in lambdas_of(text):
            bodies.setdefault(lam, []).append(body)
        for m in re.finditer(r"if \(\(?(?:warp|lane|tid|team|q4?)\b[^)]*\)?[^)]*\)\s*(\w+)\(", text):
            for body in bodies.get(m.group(1), []):
                branches += 1
                assert "__syncthreads" not in body, f"{name}: {m.group(0)}...) reaches a block barrier"
    assert branches >= 6


def test_kernels_with_a_ring_of_boxes_drain_it_when_they_give_up():
    """A kernel that stops waiting after a load that never landed may have further boxes in flight; it must wait for
    them before its shared memory is released, ask for no more, and store nothing formed without the data."""
    def kernel(name, kern):
        body = dict(kernels_of(open(os.path.join(CSRC, name)).read()))[kern]
        return re.sub(r"//[^\n]*", "", body)
    for name, kern in (("fft_inv64.cuh", "c2r_inv64_kernel"), ("fft_big.cuh", "c2r_big_kernel")):
        body = kernel(name, kern)
        tail = body[body.rindex("if ("):]
        assert "dead" in tail.split("{")[0] and tail.count("fk_ring_drain(") == 2, kern
        assert body.count("|| dead) return;") == 2, f"{kern}: a request after the give-up"
        gone = body.index("gone = dead;")
        assert re.search(r"if \((gone\) break|!gone &&)", body[gone:]), f"{kern}: results without data are stored"
    body = kernel("fft_small.cuh", "c2r_small_kernel")
    assert "if (ok && j + NST < items) issue();" in body
    for leave in re.finditer(r"return;", body):
        assert "fk_ring_drain(" in body[max(0, leave.start() - 160):leave.start()]
