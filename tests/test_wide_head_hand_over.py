"""The pass over a very wide output layer: a parity wait cannot tell a barrier's phase from the one after the next.  The warp
that stores updated tiles may be held up while the updates of the next low-half tiles complete, so each of those
tiles needs a barrier of its own.  Such a wait need not show in a run, so the source is what is checked."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_02120_b200", "csrc")


def test_updated_tiles_have_a_barrier_each():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "wide_head.cu")).read())
    assert re.search(r"\bupd_done\[kLo\]", text)
    assert re.search(r"mbar_wait\(&upd_done\[j % kLo\], \(j / kLo\) & 1", text)
    assert re.findall(r"mbar_arrive\(&upd_done\[([^\]]*)\]\)", text) == ["i % kLo"]
    # the store that frees a low-half tile comes before the load that fills it again
    body = text[text.index("auto store ="):]
    assert body.index("if (i >= kLo) ok = store(i - kLo)") < body.index("&maps.lo, &lo_full[i % kLo]")
