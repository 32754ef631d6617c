"""Kernels that start while their predecessor still runs (they call pdl_wait)
read memory that it writes.  A __restrict__ parameter tells the compiler that
nothing else touches that memory, so that its loads may move above the wait,
whose memory clobber does not bind them: no such kernel, and no device function
of a file that has one, takes a __restrict__ pointer."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2609_24456_gb300", "csrc")


def _functions(src):
    """(head, body) of every function defined with __global__ or __device__."""
    for m in re.finditer(r"__(?:global|device)__", src):
        brace, semi = src.find("{", m.start()), src.find(";", m.start())
        if brace < 0 or (0 <= semi < brace):
            continue
        depth, end = 0, brace
        while True:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
            if not depth:
                break
        yield src[m.start():brace], src[brace:end]


def _code(path):
    with open(path) as f:
        src = f.read()
    return re.sub(r"//[^\n]*", "", src)


def test_the_parser_finds_the_kernels():
    heads = [h for f in glob.glob(os.path.join(CSRC, "*.cu")) for h, b in _functions(_code(f))
             if "__global__" in h and "pdl_wait" in b]
    names = " ".join(heads)
    for k in ("k_update_small", "k_pack_gather_short", "k_gae_norm", "k_perm_rank",
              "k_sample_prio", "k_deliver_stack_flat", "k_tree_total"):
        assert re.search(r"\b%s\(" % k, names), k


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu"))),
                         ids=os.path.basename)
def test_no_restrict_above_a_wait(path):
    functions = list(_functions(_code(path)))
    if not any("pdl_wait" in body for _, body in functions):
        return
    for head, body in functions:
        if "__global__" in head and "pdl_wait" not in body:
            continue  # launched plainly
        assert "__restrict__" not in head, " ".join(head.split())
