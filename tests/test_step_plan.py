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
