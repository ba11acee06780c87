"""CTA pairs of the fp32 products: what one CTA writes to its shared memory is read by MMAs that the other issues.
The arrival that hands it over must release, and be acquired, at cluster scope; an arrival at CTA scope
orders nothing for another CTA.  A race of this kind need not show in results, so the source is what is checked."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_02120_b200", "csrc")


def test_pairs_hand_over_operands_at_cluster_scope():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "gemm_f32.cu")).read())
    assert "mbar_arrive_cluster<false>" not in text
    remote = re.findall(r"(mbar_arrive\w*(?:<\w+>)?)\(map_to_cta\(&(\w+)\[", text)
    assert sorted(remote) == [("mbar_arrive_cluster<true>", "peer"), ("mbar_arrive_relaxed_cluster", "taken")]
    # the same two are waited for at cluster scope
    assert re.search(r"mbar_wait<true>\(rank \? &full\[sl\] : &peer\[sl\]", text)
    assert "mbar_wait<PAIR == 2>(&taken" in text
