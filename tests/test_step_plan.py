"""The iteration in one launch (prb_step.cu), what can be said of it without a GPU."""
import os
import re

from conftest import ROOT

STEP = os.path.join(ROOT, "paper_2311_09445_b200", "csrc", "prb_step.cu")


def test_both_builds_synchronise_alike():
    # the checked build is what the race-prone paths are tested with: it may check more, but not order more, than the other
    text = re.sub(r"//[^\n]*", "", open(STEP).read())
    assert "PEARL_CHECKED" not in text
    # a CTA's staged levels are read by its peers from the barrier of level U on: an arrival there releases them
    release = text.index("fence.release.sync_restrict::shared::cta.cluster")
    arrive = text.index("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];\" ::\"r\"(at_rank(bar_up, lane))")
    assert release < arrive < text.index("RowOfPeer{")


def test_no_wait_is_taken_for_granted():
    # a wait that ran out is an answer: nothing may be summed, drawn or moved on from what has not come
    text = re.sub(r"//[^\n]*", "", open(STEP).read())
    waits = [m.end() for m in re.finditer(r"prb_wait_first_phase<true>\(plan\.state, bar_\w+\)", text)]
    assert len(waits) == 4
    for at in waits:
        assert re.match(r" == kPrb(InTime|Never)", text[at:]), text[at - 80:at + 40]
    # level U's wait decides about the sums that CTA 0 stores, and with the visibility's about cursor, walk and indices
    assert text.count("rank == 0u && sound, l, from, i)") == 4 and text.count("sound = tree_sync_all(sound);") == 2
    assert "if (sound) move_cursor();" in text and "&& sound) move_cursor();" in text
    assert "if (walks && sound)" in text and "if (holds && sound) plan.out_idx[k]" in text
