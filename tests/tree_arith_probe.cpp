// Evaluates the index arithmetic of the tree work (csrc/prb_arith.cuh) on the host.
// stdin: "nodes CAPACITY SHIFT" per line; stdout: the result, one per line.
#include "prb_arith.cuh"

#include <cinttypes>
#include <cstdio>
#include <cstring>

int main()
{
    char what[16];
    unsigned a, b;
    while (std::scanf("%15s %u %u", what, &a, &b) == 3) {
        if (!std::strcmp(what, "nodes")) std::printf("%" PRIu32 "\n", prb_nodes_covering(a, b));
    }
    return 0;
}
