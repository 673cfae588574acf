// Host-only check of the cost line of the unit lists (csrc/vpm_far.cuh): entries with the
// costs of a unit's groups, summed in the lists' own type up to the largest number of units,
// fall into every range in order, and each entry's range is the one that the lists' consumers
// compute for it.  Prints "OK" or the failure.
#include <stdio.h>

#include "vpm_far.cuh"

using namespace vpm;

// `cost` of entry q; most is the largest.
template <class Cost>
static int check(const char* name, long long entries, int most, int B, Cost cost)
{
    decltype(uint2::y) sum = 0;  // as the scan and the lists hold it
    long long exact = 0;
    for (long long q = 0; q < entries; ++q) sum += cost(q), exact += cost(q);
    const CostLine cl{sum, B, most};
    const int nb = cl.blocks();
    if ((long long)cl.tot != exact || nb < 1 || nb > B || (exact >= (long long)B * most && nb != B)) {
        printf("%s: total %lld held as %lld, %d ranges of %d\n", name, exact, (long long)cl.tot, nb, B);
        return 1;
    }
    decltype(uint2::y) before = 0;
    int range = -1;
    for (long long q = 0; q < entries; before += cost(q), ++q) {
        while (range + 1 < nb && (long long)before >= cl.begin(range + 1)) {
            ++range;
            if ((long long)before - cl.begin(range) >= most) {
                printf("%s: range %d holds no entry\n", name, range);
                return 1;
            }
        }
        // the entries at either end of a range, and some others
        if (((q & 1023) == 0 || (long long)before - cl.begin(range) < most || cl.begin(range + 1) - (long long)before <= most) &&
            cl.block_of(before) != range) {
            printf("%s: entry %lld (cost %lld) in range %d, computed %d\n", name, q, (long long)before, range,
                   cl.block_of(before));
            return 1;
        }
    }
    if (range != nb - 1 || cl.begin(nb) != exact) {
        printf("%s: %d of %d ranges, end %lld of %lld\n", name, range + 1, nb, cl.begin(nb), exact);
        return 1;
    }
    return 0;
}

int main()
{
    constexpr int WARPS = SWEEP_CW / FAR_GROUPS, NEAR = WARPS * NEAR_COST, FAR = FAR_COST_FIRST + FAR_GROUPS - 1;
    auto mixed = [](long long q) { return WARPS + 2 * (int)((unsigned long long)q * 2654435761u >> 13 & 3u) * (NEAR_COST - 1) / 2; };
    int bad = 0;
    // pair sweep: every group of every unit within 7 sigma, up to the most units there can be
    for (long long units : {1LL, 37LL, 152LL, 5000LL, 44739242LL, 44739243LL, 51600000LL, FAR_MAX_UNITS})
        bad |= check("near", units * FAR_GROUPS, NEAR, 608, [](long long) { return NEAR; });
    for (long long units : {41LL, 3000LL, FAR_MAX_UNITS}) bad |= check("mixed", units * FAR_GROUPS, NEAR, 608, mixed);
    // tensor-core sweep: all groups of every unit
    for (long long units : {1LL, 151LL, 2049LL, FAR_MAX_UNITS})
        bad |= check("far", units, FAR, 152, [](long long) { return FAR; });
    // a ragged group's unit costs what a whole group's costs when its warps are alike, and no
    // more than the dearest
    for (int left = -3; left <= FAR_GROUP + 70; ++left) {
        const int w = group_warps(left);
        if (w != (left <= 0 ? 0 : left > 192 ? 4 : left > 128 ? 3 : left > 64 ? 2 : 1)) bad = 1, printf("warps of %d targets: %d\n", left, w);
        for (int near = 0; w > 0 && near <= w; ++near) {
            const int c = ragged_cost(near * NEAR_COST + (w - near), w);
            if (c < WARPS || c > NEAR || (near == 0 && c != WARPS) || (near == w && c != NEAR))
                bad = 1, printf("ragged cost of %d warps, %d near: %d\n", w, near, c);
        }
    }
    if (!bad) printf("OK\n");
    return bad;
}
