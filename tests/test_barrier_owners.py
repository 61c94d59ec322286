"""Warps 0 and 3 of the tensor-core kernel do not wait for the others once the barriers are set up, so each of them may only use barriers that it has set
up itself.  Read from the source: a missing order between two warps shows in no run that goes well."""
import re
from pathlib import Path

SOURCE = (Path(__file__).resolve().parent.parent / "paper_2605_10380_b200" / "csrc" / "agx_attn_tile.cu").read_text()


def part(begin, end):
    at = SOURCE.index(begin)
    return SOURCE[at:SOURCE.index(end, at)]


def bars(text):
    return set(re.findall(r"\bBAR_(?!COUNT)\w+", re.sub(r"//.*", "", text)))


def test_warps_that_do_not_wait_use_their_own_barriers():
    every = {n.strip().split(" ")[0] for n in part("BAR_K_FULL = 0", "BAR_COUNT").split(",") if n.strip()}
    others = set(re.findall(r"i != (BAR_\w+)", part("if (tid == 0) {", "*abort_flag = 0;")))   # not thread 0's
    by_warp_3 = set(re.findall(r"mbar_init\(bar\((BAR_\w+)\)", part("if (warp == 3 && elect_one()) {", "One Q tile")))
    assert others == by_warp_3 and by_warp_3 < every
    assert "warp == 0 || warp == 3" in SOURCE and "bar.arrive 2" in SOURCE   # (else this test can go)
    used_3 = bars(part("} else {   // warp 3", 'asm volatile("setmaxnreg.inc'))
    used_0 = bars(part("= TMA producer =", "= MMA issuers:"))
    assert used_3 and used_3 <= by_warp_3, used_3 - by_warp_3
    assert used_0 and not used_0 & by_warp_3
