// Evaluates the index arithmetic of the tree work (csrc/prb_arith.cuh) and the bounded wait (csrc/prb_wait.cuh) on the
// host.  stdin, per line: "nodes CAPACITY SHIFT", "place INDEX SHIFT", "wait READY LIMIT" (something that is there from poll READY on);
// stdout: the result, one per line (wait: outcome and polls made).
#include "prb_arith.cuh"
#include "prb_wait.cuh"

#include <cinttypes>
#include <cstdio>
#include <cstring>

int main()
{
    char what[16];
    unsigned a, b;
    while (std::scanf("%15s %u %u", what, &a, &b) == 3) {
        if (!std::strcmp(what, "nodes")) std::printf("%" PRIu32 "\n", prb_nodes_covering(a, b));
        if (!std::strcmp(what, "place")) std::printf("%" PRIu32 "\n", prb_hash_place(a, b));
        if (!std::strcmp(what, "wait")) {
            unsigned polls = 0;
            auto poll = [&]() { return ++polls >= a; };
            const PrbWaited w = prb_wait_bounded(poll, b, [&]() { return prb_poll(poll, b) ? kPrbLate : kPrbNever; });
            std::printf("%d:%u\n", (int)w, polls);
        }
    }
    return 0;
}
