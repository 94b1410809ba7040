"""Hand-overs between the two CTAs of a cluster in the tile kernel, read from its source: a missing wait or
a scope that is too narrow shows in no result until it does, so these are not left to runs on a GPU."""
import os
import re

from conftest import ROOT

SRC = open(os.path.join(ROOT, "paper_2607_21927_gb300", "csrc", "attn_tile.cu")).read()
KERNEL = SRC[SRC.index("k_attn_tile(const AttnArgs"):SRC.index("// ---------------------------------------------------------------- host side")]
SOFTMAX = KERNEL[KERNEL.index("=== softmax"):KERNEL.index("atomicOr(&g_ris_tile_error")]
CLOSING = KERNEL[KERNEL.index("atomicOr(&g_ris_tile_error"):]


def test_commits_are_waited_for_in_each_cta():
    """A commit arrives in both CTAs, asynchronously: the closing cluster barrier does not order it. So it
    goes only to barriers that softmax warps, which both CTAs have, wait on for every tile, and that
    the closing part waits on again where a wait gave up."""
    targets = re.findall(r"tc_commit<CG>\((.*)\);", KERNEL)
    assert len(targets) == 2
    for target in targets:
        bar = re.fullmatch(r"sbase \+ BAR\(L::(B_\w+) \+ ST\)", target)
        assert bar, f"commit to a barrier of its own: {target}"
        assert f"mbar_wait(sbase + BAR(L::{bar[1]} + " in SOFTMAX, bar[1]
        assert f"mbar_wait_own(sbase + BAR(L::{bar[1]} + " in CLOSING, bar[1]
    # the second wait of the closing part ends before either CTA leaves
    assert CLOSING.index("mbar_wait_own") < CLOSING.rindex("cluster_sync()") < CLOSING.index("tmem_dealloc<CG>(tmem)")
