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
        # (softmax warps arrive on barriers only through arrive_lead: an address taken here is waited on)
        assert re.search(rf"(mbar_(wait|test)<CG[^>]*>\(|uint32_t bar = )sbase \+ BAR\(L::{bar[1]} \+ ", SOFTMAX), bar[1]
        assert f"mbar_wait_own<CG>(sbase + BAR(L::{bar[1]} + " in CLOSING, bar[1]
    # the second wait of the closing part ends before either CTA leaves
    assert CLOSING.index("mbar_wait_own") < CLOSING.rindex("cluster_sync()") < CLOSING.index("tmem_dealloc<CG>(tmem)")


def _asm(head):
    """Inline PTX statements (their string literals joined) in which `head` occurs."""
    joined = ("".join(re.findall(r'"((?:[^"\\]|\\.)*)"', m)) for m in re.findall(r"asm(?: volatile)?\((.*?)\);", SRC, re.S))
    return [s for s in joined if head in s]


def test_hand_overs_between_ctas_name_the_cluster_scope():
    """Without a scope an arrival and a wait order within a CTA only, and what the other CTA of the pair
    copied or wrote need not be there when its products start."""
    remote = [s for s in _asm("mbarrier.arrive") if "shared::cluster" in s and "tcgen05.commit" not in s]
    assert remote
    for s in remote:
        assert re.search(r"mbarrier\.arrive(\.expect_tx)?\.(relaxed|release)\.cluster\.shared::cluster", s), s
    for wait in ("try_wait", "test_wait"):
        scopes = sorted(re.search(rf"mbarrier\.{wait}\.parity\.((?:\w+\.\w+\.)?)shared::cta\.", s)[1] for s in _asm(f"mbarrier.{wait}"))
        assert scopes == ["", "acquire.cluster.", "relaxed.cluster."], wait  # of one CTA, and of two
    # every wait of the kernel says for how many CTAs it is, and only the softmax warps, which take nothing but
    # tensor memory from the other CTA's products, do without the acquire (not at the end, where shared
    # memory that the products read is written)
    assert not re.search(r"mbar_(wait|test|wait_own|try_wait)\(", KERNEL)
    assert KERNEL.count("<CG, true>") == SOFTMAX.count("<CG, true>") == 3
    assert "<CG, true>" not in SOFTMAX[SOFTMAX.index("the row's maximum and sum from both threads"):]


def test_copies_complete_on_the_issuing_ctas_barriers():
    """Both CTAs' copies signal the CTA that issues the products, whose relay sees them at cluster scope:
    no arrival of a thread of the other CTA stands for a copy that it saw."""
    loads = _asm("cp.async.bulk.tensor")
    assert any("cta_group::2" in s for s in loads)
    assert not re.search(r"tma_load_3d\(", KERNEL)  # the form is chosen by the number of CTAs
    for bar in ("bq", "bk", "bv"):
        assert re.findall(rf"\b{bar} = (\w+)", KERNEL).count("lead") == len(re.findall(rf"\b{bar} = ", KERNEL)) > 0, bar
    relay = KERNEL[KERNEL.index("=== relay"):KERNEL.index("=== product issuers")]
    assert "arrive_lead" not in relay and relay.count("mbar_arrive(sbase + BAR(") == 2
