"""The iteration in one launch (prb_step.cu), what can be said of it without a GPU."""
import os
import random
import re
import struct
from fractions import Fraction

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


def test_quotient_of_total_and_batch_size():
    # prb_quotient (prb_descend.cuh) in exact arithmetic, each operation rounded once: the correctly rounded total / B for every batch size
    # that a cluster takes, totals from the smallest subnormal binary32 to the largest
    text = open(os.path.join(ROOT, "paper_2311_09445_b200", "csrc", "prb_descend.cuh")).read()
    assert "const double q = __dmul_rn(a, y);\n    return __fma_rn(__fma_rn(-q, b, a), y, q);" in text
    assert "kPrbClusterStrata = 1536;" in open(os.path.join(ROOT, "paper_2311_09445_b200", "csrc", "prb_internal.cuh")).read()
    rng = random.Random(3)

    def binary32(bits):
        return struct.unpack("<f", struct.pack("<I", bits))[0]
    ends = [binary32(x) for x in (0x1, 0x2, 0x3, 0x7FFFFF, 0x800000, 0x800001, 0x3F800000, 0x3F7FFFFF, 0x3FFFFFFF, 0x7F7FFFFF, 0x7F000001)]
    for b in range(1, 1537):
        y = float(Fraction(1, b))
        for a in ends + [binary32(rng.randrange(1, 0x7F800000)) for _ in range(12)]:
            q = float(Fraction(a) * Fraction(y))
            r = float(Fraction(a) - Fraction(q) * b)
            assert float(Fraction(r) * Fraction(y) + Fraction(q)) == float(Fraction(a) / b), (a, b)
