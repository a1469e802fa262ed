// A bounded wait for transfers that this CTA's memory is the target of.
#pragma once
#include "prb_arith.cuh"

enum PrbWaited { kPrbInTime = 0, kPrbLate = 1, kPrbNever = 2 };

template <typename Poll>
PRB_HD bool prb_poll(Poll poll, uint32_t limit)
{
    bool there = false;
    for (uint32_t spins = 0; spins < limit && !there; ++spins) there = poll();
    return there;
}

// Polls up to `limit` times.  If that was not enough ran_out() reports it and answers with what came of as many polls again:
// a CTA that leaves hands its shared memory back under whatever is still on its way.
template <typename Poll, typename RanOut>
PRB_HD PrbWaited prb_wait_bounded(Poll poll, uint32_t limit, RanOut ran_out)
{
    return prb_poll(poll, limit) ? kPrbInTime : ran_out();
}
