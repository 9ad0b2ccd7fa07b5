"""Properties of the kernels' sources that no run shows reliably.

Kernels that start while the kernel before them runs must not promise the compiler that what that kernel writes is constant: no
__restrict__ and no __ldg on the buffers that the calls hand from one kernel to the next."""
import os
import re

from paper_2410_13276_b200 import build

HANDED_ON = r"(?:scores|stats|row_ptr\w*|col_idx\w*|gq|gk|lse|src)"


def test_buffers_between_kernels_are_not_promised_constant():
    for name in ("gate_scores.cu", "mask.cu", "attn_tc.cu", "attn_tc_common.cuh"):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())
        assert not re.findall(r"__restrict__\s+" + HANDED_ON + r"\b", text), name
        assert not re.findall(r"__ldg\([^;]*\b" + HANDED_ON + r"\b", text), name


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())


def test_a_product_of_another_shape_waits_for_the_ones_before_it():
    """The pair kernel's product for the second block alone goes to an accumulator that products of another form and shape write: MMAs of one
    accumulator keep their order by themselves only within a shape, so a wait for the commit of the tile before stands between them."""
    text = code("attn_pair.cu")
    lone = [m.start() for m in re.finditer(r"\btc_mma_ws_ts\(", text)]
    assert len(lone) == 1
    before = text[:lone[0]]
    wait = before.rfind("mbar_wait(sh, PV_DONE")
    assert wait > max(before.rfind("tc_mma_ts("), before.rfind("tc_mma_ss(")), "no wait between the two forms"
    assert "tc_fence_after()" in before[wait:]


def test_lanes_agree_before_an_aligned_barrier():
    """named_bar_or is an aligned barrier: all lanes of a warp come to it together.  A bounded wait returns lane by lane, so where a softmax or maxima
    warp keeps its outcome, the warp votes before it goes on to a barrier."""
    for name in ("attn_tc.cu", "attn_pair.cu"):
        text = code(name)
        assert "bar.red.or.pred" in code("attn_tc_common.cuh")
        kept = list(re.finditer(r"\bfail = (?:[^;]*\|\| )?!mbar_wait\(", text))
        assert kept, name
        for m in kept:
            after = text[m.end():]
            vote, bar = after.find("__any_sync("), after.find("named_bar_or(")
            assert 0 <= vote < (bar if bar >= 0 else len(after)), (name, text[m.start():m.start() + 90])


def test_warps_of_the_maxima_go_into_an_item_together():
    """The two warps of a block meet inside an item, at a barrier without a limit: a warp that lost its wait for the item must not be the one its
    neighbour waits for.  So behind that wait every warp comes to a vote, whatever its own outcome, before it looks at the item."""
    for name, start, meeting in (("attn_tc.cu", "!mbar_wait(sh, item_full(s, n), (n >> 2) & 1u, status);\n      Slot it{}", "named_bar_or(5 + 2 * s + half"),
                                 ("block_max_pair.cuh", "!mbar_wait_warp(sh, M_ITEM_FULL", "named_bar_or(bar_block")):
        text = code(name)
        between = text[text.index(start):text.index(meeting)]
        assert re.search(r"\n *if \(named_bar_or\(bar_vote, \w+, fail\) \|\| [\w.]+ < 0\) break;", between), name
