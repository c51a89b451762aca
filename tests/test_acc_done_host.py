"""The barriers on which the slice's and the slot pass's warpgroups wait before they flush an
accumulator (acc_done), by their index and phase as the kernels' source gives them.

A parity wait passes wrongly on a barrier that is two phases behind, and never on one that has
moved on.  At tile i a warpgroup waits for the products of tile i - 2, and knows only those
commits to have arrived that were issued before the products of tile i - 4: tile i - 6's and
earlier ones'.  No tile after i is committed into its accumulator before it hands tile i over.
"""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32525_gb300", "csrc")


def _function(name):
    text = open(os.path.join(SRC, "fs_tc_common.cuh")).read()
    body = re.search(r"\b%s\(int i\) \{ return (.*?); \}" % name, text).group(1)
    return eval("lambda i: " + body.replace("(uint32_t)", "").replace("1u", "1"))


def test_flush_waits_cannot_pass_early():
    of, phase = _function("acc_done_of"), _function("acc_done_phase")
    for i in range(2, 200):
        b = of(i - 2)
        tiles = [t for t in range(i + 8) if of(t) == b]  # in the order of their commits
        k = tiles.index(i - 2)
        assert phase(i - 2) == k & 1
        assert k == 0 or tiles[k - 1] <= i - 6
        assert tiles[k + 1] > i and all((t ^ i) & 1 == 0 for t in tiles)


def test_kernels_use_them():
    for f in ("fs_tc_fwd.cu", "fs_tc_bwd.cu"):
        uses = re.findall(r"&acc_done\[([^\]]*)\]", open(os.path.join(SRC, f)).read())
        assert sorted(re.sub(r"\b[iu]\b", "n", u) for u in uses) == ["acc_done_of(n - 2)", "acc_done_of(n)", "n"]
