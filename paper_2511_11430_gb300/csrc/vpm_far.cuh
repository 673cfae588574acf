// Far-field part of the particle sweep on the 5th-generation tensor cores.
//
// A source tile (128 consecutive particles) seen from far away is a contraction: with
// c the tile's centre, a its scale, d_j = (x_j - c)/a, and for a target y = x - c,
// n = y/|y|, e = a/|y|, the separation is r = |y| (n - e d_j) and every pair's kernels are
//   r^-5 = |y|^-5 t^(-5/2),  r^-3 = |y|^-5 t^(-5/2) r^2,   t = 1 - 2 e n.d_j + e^2 |d_j|^2.
// u and grad u are then fixed combinations (polynomials in n and e) of the sums
//   m_f = sum_j t_j^(-5/2) F_f(j)
// over 29 source features F (Gamma, Gamma x d, their products with d, |d|^2): a matrix
// product [targets x sources] [sources x features].  Every pair's t^(-5/2) is evaluated
// (7 FP32 operations and one rsqrt against 32 and one in the pair loop); the product runs
// on tcgen05 with the targets in the rows of a TMEM operand.
//
// Precision.  m_f is split as sum_j F_f(j) + sum_j (t_j^(-5/2) - 1) F_f(j): the first sum
// is formed once per tile in FP32, so only the small second one passes through the tensor
// core, as FP16 pairs (hi + lo, 22 bits) of both factors with FP32 accumulation.  The
// result of a tile is folded into the running sums as in the pair sweep.
//
// Bound and layout.  Per pair: 7 packed FP32 lanes' worth of FMA-pipe work and one rsqrt for
// the weight, two conversions and a subtraction for its FP16 pair, one word of TMEM written;
// the products (3 x 29 columns per pair) keep the tensor core a fifth busy.  The loop is
// bound by issue slots and the FMA pipe (65% and 62% busy; the XU pipe 50%).  A thread owns two targets, one
// row in each of two 128-row accumulators, and takes sources in pairs, so that a packed
// register pair is one operand word and the source data is not duplicated; four warpgroups
// per block work at their own pace on a shared ring of source tiles.  A chunk is 32 sources
// (32 TMEM columns, the accumulators take the other 32 of a tile's 64); the last warp of a
// group to store its rows issues the chunk's twelve MMAs while the others go on.
// 400,000 particles onto themselves, compensated: 161 ms by the pair sweep alone, 70 ms so
// (2.3e12 pairs/s); 100,000: 10.2 and 5.0 ms.
//
// A (target group, tile) pair takes this path when the tile's radius is at most FAR_TAU of
// its centre's distance to the group's boxes and every pair is at least 7 sigma apart (the
// point-vortex form); all others go to the pair sweep.  far_mask_kernel decides once, and
// both launches walk the unit lists that it leaves.
#pragma once

#include "vpm_common.cuh"
#include "vpm_internal.h"

namespace vpm {

constexpr int FAR_GROUP = 256;                   // targets per far group (a warpgroup, two per thread)
constexpr int FAR_GROUPS = TGT_TILE / FAR_GROUP; // groups of a target tile
constexpr unsigned FAR_ALL = (1u << FAR_GROUPS) - 1u;
// Cost in the pair sweep of a warp's tile within 7 sigma, against one of a tile beyond.
constexpr int NEAR_COST = 3;
constexpr int FAR_COST_FIRST = 3;                // cost of a far unit's first group, against one of each further
// Acceptance ratio.  The error hardly depends on it, since every pair is evaluated at any ratio
// (right-hand side of the 100,000-particle hover wake at 0.33, 0.4 and 0.5: dx/dt 1.08e-7, 1.09e-7 and
// 1.13e-7, nu_t 9.96e-7, 9.96e-7 and 9.97e-7, with the near tiles' sums folded once a tile); beyond 0.5
// the weights (up to 31 there) and the cancellation in t grow and little time is gained (the same
// call 7.05, 6.94 and 6.82 ms; u and grad u alone 5.88 ms at 0.5 and 5.63 at 0.6 in an earlier form).
constexpr float FAR_TAU = 0.5f;
// (1,024-target, 128-source) units from which the far sweep is used: below, packing and
// listing (about 40 us) cost more than it saves.  Velocity only, 1,280 control points:
// 100,000 sources (1,564 units) 146 us without it and 171 us with it, 160,000 (2,500 units)
// 205 and 212, 200,000 (3,126 units) 245 and 241, 300,000 337 and 310 us.  With the gradient, the
// adjoint of 1,280 control points at 60,000 particles (590 units) 199 and 230 us, at 100,000
// (980 units) 267 and 210 us.  As many targets as sources, in tensors of their own, depend on the
// order that they come in (20,000, u and grad u: hover wake 559 and 613 us, BVI wake 597 and 430).
constexpr long long FAR_MIN_UNITS_VEL = 2048, FAR_MIN_UNITS_GRAD = 900;
constexpr long long FAR_MAX_UNITS = 1LL << 26;   // ... and to which (the unit lists take up to 44 bytes each)
// Particles onto themselves: smallest count put in curve order and swept this way (right-hand
// side, without and with it: BVI wake 12,000 particles 617 and 628 us, 16,000 822 and 743 us, 20,000
// 1,050 and 876 us; hover wake 571 and 586, 724 and 727, 945 and 864 us).
constexpr int FAR_SORT_MIN = 16384;
// Coordinates up to which |x - y|^2 stays finite in FP32.  Beyond, a pair contributes nothing
// in the pair sweep (1/r of an infinite r^2), which takes the groups and tiles concerned.
constexpr float FAR_XMAX = 4e18f;
constexpr int FAR_KCH = 2048;                    // source tiles per block of the mask and list kernels
constexpr int FAR_FEXP = 8;                      // features are scaled to at most 2^8 before their FP16 split

// Packed far tile: FP16 features hi then lo in the tensor core's K-major core-matrix
// order, the scaled offsets in source pairs, the header.
template <bool GRAD>
struct FarTile {
    static constexpr int N = GRAD ? 32 : 16;              // feature columns (29 / 6 used)
    static constexpr int NF = GRAD ? 29 : 6;
    static constexpr int FEAT = SRC_TILE * N * 2;         // bytes of one FP16 half
    static constexpr int OFF_D = 2 * FEAT;                // float4 per source pair: (dx,dx,dy,dy) (dz,dz,q,q)
    static constexpr int OFF_H = OFF_D + SRC_TILE * 16;   // header: N feature sums, then cx, cy, cz, a, gamma
    static constexpr int BYTES = OFF_H + 256;
};
constexpr size_t far_tile_bytes(bool grad) { return grad ? FarTile<true>::BYTES : FarTile<false>::BYTES; }

// Warps of a group that hold targets, when `left` targets remain from its first on.
__host__ __device__ __forceinline__ int group_warps(int left)
{
    return left <= 0 ? 0 : (left >= FAR_GROUP ? FAR_GROUP / 64 : (left + 63) / 64);
}
// Cost of a ragged group's unit from that of its `warps` warps: as if the others were like them.
// A unit takes as long as its slowest warp, not the sum; counted by the sum, the last group's units
// went to one team that took twice as long as the others (39,999 targets, 63 in the last group,
// particles in no order: 3.23 and 2.3 ms).
__host__ __device__ __forceinline__ int ragged_cost(int cost, int warps)
{
    return (cost * (FAR_GROUP / 64) + warps - 1) / warps;
}

// The cost line of a unit list, cut into equal ranges: at most B, each at least a whole unit
// long, so that every range holds the start of one.  Costs are unsigned: a dense cloud in no
// order at FAR_MAX_UNITS units costs 3.2e9.
struct CostLine {
    unsigned tot;
    int B;
    int max_cost;  // of one unit

    __host__ __device__ __forceinline__ int blocks() const
    {
        const int whole = (int)(tot / (unsigned)max_cost);
        return whole < 1 ? 1 : (whole < B ? whole : B);
    }
    // First cost of range b.
    __host__ __device__ __forceinline__ long long begin(int b) const { return (long long)b * tot / blocks(); }
    // Range owning the unit whose cost starts at c.
    __host__ __device__ __forceinline__ int block_of(unsigned c) const
    {
        return (int)((((long long)c + 1) * blocks() - 1) / tot);
    }
};
static_assert(FAR_MAX_UNITS * SWEEP_CW * NEAR_COST < (1LL << 32), "the pair sweep's costs fit 32 bits");
static_assert(FAR_MAX_UNITS * (FAR_COST_FIRST + FAR_GROUPS - 1) < (1LL << 32), "the tensor-core sweep's costs fit 32 bits");
static_assert(FAR_MAX_UNITS * FAR_GROUPS < (1LL << 31), "entry numbers fit 31 bits");

// A list of units ordered by target tile: (source tile << 4 | group mask, cost of the
// units before it); the pair sweep's is ordered by group and holds the source tile alone.
// A unit's cost in the tensor-core list is far_cost of its groups, in the pair sweep's the
// number of the group's warps, those within 7 sigma counted NEAR_COST times.  One block or
// team runs the units whose cost starts in its range of the cost line and writes one partial
// sum per target tile into slot b + t.
struct UnitList {
    const uint2* list;
    const uint2* off;  // (entries, cost) before each (target tile, chunk); [TT * KY + 1]
    int TT, KY, B;
    int max_cost;      // of one unit

    __device__ __forceinline__ int end(int t) const { return (int)off[(t + 1) * KY].x; }
    __device__ __forceinline__ CostLine line() const { return CostLine{off[TT * KY].y, B, max_cost}; }
    // First index in [0, n) with key(index) >= v (n if none), key nondecreasing, by a whole warp:
    // 32 probes a round instead of one, since each round waits for memory.
    template <class Key>
    static __device__ __forceinline__ int warp_lower_bound(int n, long long v, Key key)
    {
        const int lane = threadIdx.x & 31;
        int a = 0, z = n;  // the answer lies in [a, z]
        while (a < z) {
            const int step = (z - a + 31) / 32, q = a + lane * step;
            const bool below = q < z && (long long)key(q) < v;
            const int k = __popc(__ballot_sync(0xffffffffu, below));  // probes 0 .. k-1 are below
            if (k == 0) return a;
            const int last = a + (k - 1) * step;
            z = min(z, a + k * step);
            a = last + 1;
        }
        return a;
    }
    // The entries [lo, hi) of block b and the target tile of the first; by a whole warp.
    __device__ __forceinline__ void range(int b, int& lo, int& hi, int& t) const
    {
        const int entries = (int)off[TT * KY].x;
        const CostLine cl = line();
        lo = hi = t = 0;
        if (b >= cl.blocks()) return;
        const uint2* l = list;
        auto cost = [l](int q) { return l[q].y; };
        lo = warp_lower_bound(entries, cl.begin(b), cost);
        hi = warp_lower_bound(entries, cl.begin(b + 1), cost);
        const uint2* o = off;
        const int ky = KY;
        t = warp_lower_bound(TT, (long long)lo + 1, [o, ky](int q) { return o[(q + 1) * ky].x; });
    }
};

struct FarArgs {
    const float4* tgt;
    int n_tgt;
    const unsigned char* tiles;
    UnitList ul;
    float* part;
    int* dev_err;
};

cudaError_t run_far_pack(const float4* pos, const float4* str, int n, const float4* box, int SP, bool grad,
                         unsigned char* tiles, cudaStream_t st);
cudaError_t run_far_lists(const float4* tgt, int n_tgt, const unsigned char* tiles, int SP, int TT, bool grad,
                          const float4* pbox, float far2, unsigned* mask, uint2* cnt, uint2* near_list,
                          uint2* near_off, uint2* far_list, uint2* far_off, cudaStream_t st);
cudaError_t run_far_sweep(const FarArgs& A, bool grad, bool comp, cudaStream_t st);

}  // namespace vpm
