"""Kernels that are set up while their predecessor runs (those that begin with
block_after()) read what it wrote.  Nothing in their source may let the compiler
move such a read ahead of the wait: no __restrict__ parameter and no read-only
load, whose values it may take for invariant, and no inline assembly that loads
global memory without being volatile."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_08119_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def _braces(s, start):
    depth = 0
    for i in range(start, len(s)):
        depth += {"{": 1, "}": -1}.get(s[i], 0)
        if depth == 0:
            return s[start:i + 1]
    raise AssertionError("unbalanced braces")


def _kernels():
    for name in sorted(os.listdir(CSRC)):
        s = _source(name)
        for m in re.finditer(r"__global__", s):
            end = min(i for i in (s.find("{", m.start()), s.find(";", m.start())) if i >= 0)
            if s[end] == ";":
                continue
            head, body = s[m.start():end], _braces(s, end)
            if "block_after()" in body:
                yield re.findall(r"\b(k_\w+)\s*\(", head)[0], head, body


KERNELS = {k: (head, body) for k, head, body in _kernels()}


def test_the_kernels_are_found():
    assert {"k_site", "k_assemble", "k_list_direct", "k_kick_drift", "k_contract_bulk", "k_loss"} <= set(KERNELS)


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_reads_stay_behind_the_wait(kernel):
    head, body = KERNELS[kernel]
    assert "__restrict__" not in head
    before = body[:body.index("block_after()")]
    for line in before.splitlines():  # only declarations ahead of the wait
        assert "__shared__" in line or "[" not in line or "if constexpr" in line, line
    # recv_load reads these two through __ldcg, which is not volatile
    if re.search(r"\brecv_load\(|\bbulk_receive_chunk<", body):
        for p in ("fown", "w6in"):
            assert f"{p} = reread({p});" in body


def test_no_movable_loads():
    for name in sorted(os.listdir(CSRC)):
        s = _source(name)
        assert "__ldg(" not in s and ".nc." not in s, name
        for m in re.finditer(r"\basm\s*\((.*?)\);", s, flags=re.S):  # asm without volatile
            assert "ld.global" not in m.group(1), (name, m.group(1))
