"""The unpack warps of the packed-operand GEMM (gemm_direct.cu) as a model on the CPU: two groups take K blocks in turn, every
wait is a parity wait, and copies of different slots may land in any order."""
import re
from pathlib import Path

import pytest

SOURCE = Path(__file__).resolve().parent.parent / "paper_2504_18547_b200" / "csrc" / "gemm_direct.cu"


def kernel_wait_order():
    """The barriers an unpack group waits for in front of a block, in the order of the source."""
    loop = SOURCE.read_text().split("direct_unpack(P.ca,")[0].rsplit("while (ok", 1)[1]
    return re.findall(r"mbar_wait\(ptx::smem_addr\(&bars\.(\w+)\[", loop)


def stale_block(order, ns, ns_p, blocks=10):
    """Walks every interleaving of copies, unpack groups and contraction; the first block that a group would expand before its
    packed bytes have landed, or None.  ns, ns_p: slots of the operand and of the packed ring."""
    start = (frozenset(), (0, 1), (0, 0), frozenset(), 0)     # landed; per group: its block, waits passed; expanded; contracted
    seen, todo = {start}, [start]
    while todo:
        landed, block, passed, expanded, contracted = todo.pop()
        nxt = []
        for it in range(blocks):                               # a copy lands once its slot's last block has been expanded
            if it not in landed and (it < ns_p or it - ns_p in expanded):
                nxt.append((landed | {it}, block, passed, expanded, contracted))
        for g in range(2):
            it = block[g]
            if it >= blocks:
                continue
            if passed[g] == 2:
                if it not in landed:
                    return it
                nxt.append((landed, tuple(it + 2 if k == g else b for k, b in enumerate(block)),
                            tuple(0 if k == g else p for k, p in enumerate(passed)), expanded | {it}, contracted))
                continue
            if order[passed[g]] == "p_full":                   # phases completed so far; the wait asks for the one with this parity
                done, want = sum(1 for j in landed if j % ns_p == it % ns_p), (it // ns_p) & 1
            else:
                done, want = len(range(it % ns, contracted, ns)), (it // ns + 1) & 1
            if (done & 1) != want:
                nxt.append((landed, block, tuple(p + 1 if k == g else p for k, p in enumerate(passed)), expanded, contracted))
        if contracted in expanded:
            nxt.append((landed, block, passed, expanded, contracted + 1))
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


@pytest.mark.parametrize("ns", [2, 3])
@pytest.mark.parametrize("ns_p", [2, 3, 4, 5, 6])
def test_no_block_is_expanded_before_it_has_landed(ns, ns_p):
    order = kernel_wait_order()
    assert sorted(order) == ["empty", "p_full"]
    assert stale_block(order, ns, ns_p) is None


def test_the_model_tells_the_unsafe_order():
    assert stale_block(["p_full", "empty"], 3, 3) is not None
