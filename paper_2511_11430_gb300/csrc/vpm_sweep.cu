// Pair sweeps of the vortex-particle hot path on sm_103a.
//
//  * Gaussian-particle velocity and gradient (Eq. 2-4): u = sum_j K (Gamma_j x r),
//    J = [S x]/(4 pi) + sum_j H (Gamma_j x r) (x) r with S = sum_j K Gamma_j.
//  * Vatistas-cored straight segments (Sec. II.A), their velocity and exact gradient.
//  * Optionally the transposed stretching J^T Gamma_i of Eq. 5 per target.
//  * The stream-K reduction of per-warp partial sums and the per-target epilogue:
//    the velocity/gradient outputs, or the right-hand side of Eq. 4-5 (Vreman eddy
//    viscosity, stretching) formed in FP64 from the reduced sums.
//  * Particle strength exchange (the nu lap(Gamma) term of Eq. 5).
//
// Kernel organisation.  A thread owns two targets, kept in the two lanes of packed
// float2 registers so that each FFMA2/FADD2/FMUL2 advances two pair interactions.
// Sources are packed once per call into 128-source tiles (duplicated into both
// lanes, negated copies included so that every subtraction is an add).  The sweep
// block streams the tiles through a ring of shared-memory stages with the bulk-copy
// engine (cp.async.bulk completing on a per-stage "full" mbarrier); each of its 16
// warps waits on "full", reads every source by broadcast and counts itself out of
// the stage, and the last warp to leave a stage refills it with the tile six units
// ahead.  Warps drift freely within the ring and no block-wide barrier sits in the
// loop.  Work is split stream-K over
// (target tile, source tile) cost units so every SM gets the same cost however few
// targets there are.  Far from a warp's 64 targets (the tile's bounding box more
// than 7 sigma from both of the warp's two target boxes) the blob kernel equals
// the point-vortex kernel to FP32 precision, so far tiles run the 1/r^3 form with
// one rsqrt; near tiles evaluate the regularised kernel for the sources within 7 sigma (of
// the warp's boxes with stretching, of a thread's targets without).  In larger problems the tiles that are far and compact run on the
// tensor cores instead (vpm_far.cuh), over particles in curve order.  Each tile's sums start from zero and are folded into a
// per-thread running sum kept in shared memory: a compensated (hi, lo) pair with
// Knuth's two-sum, or a plain sum, so long source lists keep a tile-sized error.
#include <float.h>
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "vpm_common.cuh"
#include "vpm_far.cuh"
#include "vpm_internal.h"
#include "vpm_kernel.cuh"

namespace vpm {

// The sources of a particle tile.  The velocity-only loop is unrolled twice; the
// gradient loop, whose body already holds enough independent work, is not (measured:
// unrolling it costs 3.5%, unrolling the velocity loop gains 7%).
template <bool GRAD, bool STRETCH, bool NEAR>
__device__ __forceinline__ void particle_tile(Acc<GRAD, STRETCH>& a, const float4* __restrict__ s, int cnt, f2 X,
                                              f2 Y, f2 Z, const NearConst& nc, const Own& o)
{
    if constexpr (GRAD) {
#pragma unroll 1
        for (int j = 0; j < cnt; ++j) particle_source<GRAD, STRETCH, NEAR>(a, s + j * P_F4, X, Y, Z, nc, o);
    } else {
#pragma unroll 2
        for (int j = 0; j < cnt; ++j) particle_source<GRAD, STRETCH, NEAR>(a, s + j * P_F4, X, Y, Z, nc, o);
    }
}

// The sources of a particle tile selected by `keep` (bit j of keep[h]: source 32 h + j), words
// h0 to h1.
template <bool GRAD, bool STRETCH, bool NEAR>
__device__ __forceinline__ void particle_subset(Acc<GRAD, STRETCH>& a, const float4* __restrict__ s,
                                                const unsigned (&keep)[SRC_TILE / 32], int h0, int h1, bool invert,
                                                int cnt, f2 X, f2 Y, f2 Z, const NearConst& nc, const Own& o)
{
#pragma unroll 1
    for (int h = h0; h < h1 && 32 * h < cnt; ++h) {
        unsigned m = h == 0 ? keep[0] : h == 1 ? keep[1] : h == 2 ? keep[2] : keep[3];
        const int left = cnt - 32 * h;
        if (invert) m = ~m & (left >= 32 ? 0xffffffffu : (1u << left) - 1u);
        for (const float4* sh = s + 32 * h * P_F4; m; m &= m - 1)
            particle_source<GRAD, STRETCH, NEAR>(a, sh + (__ffs(m) - 1) * P_F4, X, Y, Z, nc, o);
    }
}

// The tile's sums without stretching (a far particle tile or a segment tile) into the
// fold rows of the stretching sweep: rows 0..13 copied, rows 14..16 set to the tile's
// transposed stretching J_tile^T Gamma_i (times 4 pi), formed from its partial S and
// G' -- for these tiles the two terms do not cancel.  The target's own strength is
// read here, after the tile's loop, so that it is not held in registers through it.
template <bool GRAD, bool STRETCH>
__device__ __forceinline__ void finish_tile(Acc<GRAD, STRETCH>& a, const Acc<GRAD, false>& t, const float4* tstr,
                                            int i0, int i1, int n_tgt)
{
    static_assert(GRAD || !STRETCH, "stretching needs the gradient sums");
#pragma unroll
    for (int q = 0; q < Acc<GRAD, false>::N; ++q) a.v[q] = t.v[q];
    if constexpr (STRETCH) {
    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;
    if (i0 < n_tgt) g0 = tstr[i0];
    if (i1 < n_tgt) g1 = tstr[i1];
    const f2 ogx = make_float2(g0.x, g1.x), ogy = make_float2(g0.y, g1.y), ogz = make_float2(g0.z, g1.z);
    const f2 Sx = t.v[3], Sy = t.v[4], Sz = t.v[5];
    const f2 Gxx = t.v[6], Gxy = t.v[7], Gxz = t.v[8], Gyx = t.v[9], Gyy = t.v[10], Gyz = t.v[11], Gzx = t.v[12],
             Gzy = t.v[13];
    const f2 Gzz = mul2(add2(Gxx, Gyy), splat(-1.f));
    const f2 m3 = splat(-3.f);
    // Gamma_i x S - 3 G'^T Gamma_i
    const f2 tx = sub2(mul2(ogy, Sz), mul2(ogz, Sy));
    const f2 ty = sub2(mul2(ogz, Sx), mul2(ogx, Sz));
    const f2 tz = sub2(mul2(ogx, Sy), mul2(ogy, Sx));
    const f2 gx = fma2(Gzx, ogz, fma2(Gyx, ogy, mul2(Gxx, ogx)));
    const f2 gy = fma2(Gzy, ogz, fma2(Gyy, ogy, mul2(Gxy, ogx)));
    const f2 gz = fma2(Gzz, ogz, fma2(Gyz, ogy, mul2(Gxz, ogx)));
    a.v[14] = fma2(m3, gx, tx);
    a.v[15] = fma2(m3, gy, ty);
    a.v[16] = fma2(m3, gz, tz);
    }
}

// ---------------------------------------------------------------------------
// Packing kernels (one thread per source slot, 128 per block = one tile).
// ---------------------------------------------------------------------------
// perm (may be null): the order in which to take the particles, which are then also written
// out in that order.
__global__ void __launch_bounds__(SRC_TILE) pack_particles_kernel(const float4* __restrict__ pos,
                                                                  const float4* __restrict__ str, int n,
                                                                  const int* __restrict__ perm,
                                                                  float4* __restrict__ spos, float4* __restrict__ sstr,
                                                                  float4* __restrict__ out, float4* __restrict__ box)
{
    const int j = blockIdx.x * SRC_TILE + threadIdx.x;
    const bool valid = j < n;
    float x = 0.f, y = 0.f, z = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
    if (valid) {
        const int i = perm ? perm[j] : j;
        const float4 p = pos[i], g = str[i];
        x = p.x, y = p.y, z = p.z;
        gx = g.x, gy = g.y, gz = g.z;
        if (perm) spos[j] = p, sstr[j] = g;
    }
    float4* o = out + (size_t)j * P_F4;
    o[0] = make_float4(-x, -x, -y, -y);
    o[1] = make_float4(-z, -z, gx, gx);
    o[2] = make_float4(gy, gy, gz, gz);
    o[3] = make_float4(-gx, -gx, -gy, -gy);
    o[4] = make_float4(-gz, -gz, 0.f, 0.f);
    float lo[3] = {valid ? x : INFINITY, valid ? y : INFINITY, valid ? z : INFINITY};
    float hi[3] = {valid ? x : -INFINITY, valid ? y : -INFINITY, valid ? z : -INFINITY};
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o2));
            hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o2));
        }
    __shared__ float sb[SRC_TILE / 32][6];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int c = 0; c < 3; ++c) sb[w][c] = lo[c], sb[w][3 + c] = hi[c];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int ww = 1; ww < SRC_TILE / 32; ++ww)
            for (int c = 0; c < 3; ++c) lo[c] = fminf(lo[c], sb[ww][c]), hi[c] = fmaxf(hi[c], sb[ww][3 + c]);
        box[2 * blockIdx.x] = make_float4(lo[0], lo[1], lo[2], 0.f);
        box[2 * blockIdx.x + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    }
}

__global__ void __launch_bounds__(SRC_TILE) pack_segments_kernel(const float4* __restrict__ sa,
                                                                 const float4* __restrict__ sb, int m, float core,
                                                                 int vn, int rings, float4* __restrict__ out,
                                                                 float4* __restrict__ box)
{
    const int j = blockIdx.x * SRC_TILE + threadIdx.x;
    const bool valid = j < m;
    float ax = 0.f, ay = 0.f, az = 0.f, rx = 1.f, ry = 0.f, rz = 0.f, g = 0.f;
    float4 bb = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) {
        const float4 a = sa[j];
        bb = sb[j];
        ax = a.x, ay = a.y, az = a.z;
        rx = bb.x - a.x, ry = bb.y - a.y, rz = bb.z - a.z;
        g = a.w;
    }
    const float L2 = rx * rx + ry * ry + rz * rz;
    const float cl2 = core * core * L2;
    float e = vn == 2 ? cl2 * cl2 : cl2;
    if (!(L2 > 0.f)) g = 0.f, e = 1.f;  // a zero-length segment induces nothing; keeps D > 0
    // Closed four-sided rings: in every group of four segments of the tile, each one's
    // end point is the next one's start point (k -> k + 1 mod 4), bit for bit; groups
    // wholly past the end do not count.  Such a tile is packed by ring.
    const int lane = threadIdx.x & 31, nxt = (lane & ~3) | ((lane + 1) & 3);
    const float nax = __shfl_sync(0xffffffffu, ax, nxt), nay = __shfl_sync(0xffffffffu, ay, nxt),
                naz = __shfl_sync(0xffffffffu, az, nxt);
    const bool joins = valid && __float_as_uint(bb.x) == __float_as_uint(nax) &&
                       __float_as_uint(bb.y) == __float_as_uint(nay) && __float_as_uint(bb.z) == __float_as_uint(naz);
    const unsigned vmask = __ballot_sync(0xffffffffu, valid), jmask = __ballot_sync(0xffffffffu, joins);
    const int g4 = lane & ~3;
    const bool ring_ok = ((vmask >> g4) & 0xFu) == 0u || ((jmask >> g4) & 0xFu) == 0xFu;
    const bool closed = __syncthreads_and(ring_ok && rings) != 0;
    if (closed) {
        float2* o2 = reinterpret_cast<float2*>(out + (size_t)blockIdx.x * SRC_TILE * S_F4) + (threadIdx.x >> 2) * 48;
        const int k = threadIdx.x & 3;
        o2[3 * k] = make_float2(-ax, -ax);
        o2[3 * k + 1] = make_float2(-ay, -ay);
        o2[3 * k + 2] = make_float2(-az, -az);
        o2[12 + 3 * k] = make_float2(rx, rx);
        o2[13 + 3 * k] = make_float2(ry, ry);
        o2[14 + 3 * k] = make_float2(rz, rz);
        o2[24 + 3 * k] = make_float2(-rx, -rx);
        o2[25 + 3 * k] = make_float2(-ry, -ry);
        o2[26 + 3 * k] = make_float2(-rz, -rz);
        o2[36 + 2 * k] = make_float2(L2, L2);
        o2[37 + 2 * k] = make_float2(e, e);
        o2[44 + k] = make_float2(g, g);
    } else {
        float4* o = out + (size_t)j * S_F4;
        o[0] = make_float4(-ax, -ax, -ay, -ay);
        o[1] = make_float4(-az, -az, rx, rx);
        o[2] = make_float4(ry, ry, rz, rz);
        o[3] = make_float4(-rx, -rx, -ry, -ry);
        o[4] = make_float4(-rz, -rz, -L2, -L2);
        o[5] = make_float4(g, g, e, e);
    }
    // tile box of both end points, and the longest segment (in lo.w)
    const float bx = ax + rx, by = ay + ry, bz = az + rz;
    float lo[4] = {valid ? fminf(ax, bx) : INFINITY, valid ? fminf(ay, by) : INFINITY,
                   valid ? fminf(az, bz) : INFINITY, valid ? -sqrtf(L2) : 0.f};
    float hi[3] = {valid ? fmaxf(ax, bx) : -INFINITY, valid ? fmaxf(ay, by) : -INFINITY,
                   valid ? fmaxf(az, bz) : -INFINITY};
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) {
#pragma unroll
        for (int c = 0; c < 4; ++c) lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o2));
#pragma unroll
        for (int c = 0; c < 3; ++c) hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o2));
    }
    __shared__ float sbx[SRC_TILE / 32][7];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        for (int c = 0; c < 4; ++c) sbx[w][c] = lo[c];
        for (int c = 0; c < 3; ++c) sbx[w][4 + c] = hi[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int ww = 1; ww < SRC_TILE / 32; ++ww) {
            for (int c = 0; c < 4; ++c) lo[c] = fminf(lo[c], sbx[ww][c]);
            for (int c = 0; c < 3; ++c) hi[c] = fmaxf(hi[c], sbx[ww][4 + c]);
        }
        box[2 * blockIdx.x] = make_float4(lo[0], lo[1], lo[2], -lo[3]);
        box[2 * blockIdx.x + 1] = make_float4(hi[0], hi[1], hi[2], closed ? 1.f : 0.f);
    }
}

// ---------------------------------------------------------------------------
// The stream-K sweep: SWEEP_CW warps per block sharing a ring of source stages.
// ---------------------------------------------------------------------------
struct SweepArgs {
    const float4* tgt;
    const float4* tstr;  // target strengths (stretching), may be null
    int n_tgt;
    const float4* psrc;
    const float4* pbox;
    int n_src;
    const float4* ssrc;
    const float4* sbox;
    int m_seg;
    int vn;
    int core_pos;  // the segment core is > 0
    StreamK sk;
    UnitList ul;  // SWEEP_NEAR: the listed units
    NearConst nc;
    float* part;
    int* dev_err;
};

constexpr uint64_t WAIT_LIMIT = 2000000000ull;  // 2 s of wall time

template <bool GRAD, bool STRETCH>
__host__ __device__ constexpr int n_rows()
{
    return Acc<GRAD, STRETCH>::N;
}


// KIND: the source tiles a launch sweeps.  SWEEP_SMALL (teams, below) takes particle tiles
// and, where the segments are few, segment tiles one segment at a time; SWEEP_PARTICLES
// takes the particle tiles of larger problems that have no tensor-core part (those without
// a caller workspace, or beyond its unit limit).  SWEEP_SEGMENTS and SWEEP_SEG_SMALL take
// only segment tiles, including those packed as closed rings.
// The ring loop needs more registers than the particle loop; in a launch of its own
// it costs the particle tiles nothing.  SWEEP_NEAR takes the particle tiles of a unit
// list: those the tensor-core sweep (vpm_far.cuh) leaves.  They cluster (a source tile is
// near a few neighbouring target groups), so each warpgroup takes its own range of
// (256-target group, source tile) units: with blocks of 1,024 targets three quarters of
// the warps had nothing to do.  (Measured: the particle launch compiled
// without its segment loop is allocated fewer registers and runs 4% slower.)
constexpr int SWEEP_PARTICLES = 0, SWEEP_SEGMENTS = 1, SWEEP_NEAR = 2, SWEEP_SMALL = 3, SWEEP_SEG_SMALL = 4;
constexpr int SWEEP_KINDS = 5;

// A ring of source stages serves a team of warps: the whole block, or each warpgroup its
// own.  Teams of four warps make finer work units (256 targets instead of 1,024, and with
// half tiles 64 sources): a small problem then reaches every SM, and a few targets or a few
// waves of units leave less idle.  (2,000 particles and 640 segments: 42 units of
// 1,024 x 128, 73 us.)
// Units (1,024 targets x 128 sources) below which teams sweep the particle tiles; above, whole
// blocks, which share a source tile among 16 warps, unless the targets fill few tiles, whose last
// is mostly empty (u and grad u of a wake's particles by vpm_induce_noalloc, teams and whole
// blocks: 16,000 of the hover wake 363 and 357 us, 30,000 1,111 and 1,036 us; of the BVI wake 382
// and 412, 1,182 and 1,235 us.  Teams alone took up to 9% longer than the whole blocks that they
// had replaced on the hover wake).  Likewise for the
// segment tiles (whose loop pays more for the folds after half tiles: 5,120 segments onto
// 100,000 particles 1.25 ms with whole blocks and tiles, 1.43 ms with teams; onto 20,000, 5.3
// units a block, 317 and 324 us).
constexpr long long SMALL_MAX_UNITS = 4096, SEG_SMALL_MAX_UNITS = 512;
constexpr int SMALL_FEW_TILES = 8;
// Segment tiles up to which a small problem sweeps them, one segment at a time, with its
// particle tiles.
constexpr int MIXED_MAX_TILES = 8;

template <int KIND>
struct Ring {
    static constexpr bool LIST = KIND == SWEEP_NEAR;
    static constexpr int TEAMS = KIND == SWEEP_PARTICLES || KIND == SWEEP_SEGMENTS ? 1 : SWEEP_CW / 4;
    static constexpr int WARPS = SWEEP_CW / TEAMS;
    static constexpr bool SEG = KIND == SWEEP_SEGMENTS || KIND == SWEEP_SEG_SMALL;
    static constexpr int UNIT = KIND == SWEEP_SMALL || KIND == SWEEP_SEG_SMALL ? SRC_TILE / 2 : SRC_TILE;  // sources
    static constexpr int PER_TILE = SRC_TILE / UNIT;
    static constexpr int STAGES = TEAMS > 1 ? 2 : SWEEP_STAGES;  // per team
    static constexpr int BOX = UNIT * (LIST ? P_F4 : S_F4);      // the tile's bounding box, float4s into a stage
    static constexpr int F4 = BOX + 2;
    static constexpr int TGT = WARPS * 64;                       // targets of a team
};

// Dynamic shared memory: the source stages, then the running sums of the consumer
// threads, [row][hi|lo][thread] as float2 (the two targets).
template <bool GRAD, bool COMP, bool STRETCH, int KIND>
__host__ __device__ constexpr size_t sweep_smem_bytes()
{
    return (size_t)Ring<KIND>::TEAMS * Ring<KIND>::STAGES * Ring<KIND>::F4 * 16 +
           (size_t)n_rows<GRAD, STRETCH>() * (COMP ? 2 : 1) * SWEEP_CW * 32 * 8;
}

template <bool GRAD, bool COMP, bool STRETCH, int KIND>
__global__ void __launch_bounds__(SWEEP_TPB, 1) sweep_kernel(const SweepArgs A)
{
    using R = Ring<KIND>;
    constexpr bool LIST = R::LIST;
    constexpr int NST = R::TEAMS * R::STAGES;
    extern __shared__ __align__(128) float4 dsm[];
    __shared__ __align__(8) uint64_t full[NST];
    __shared__ int released[NST];
    __shared__ int issued_round[NST];  // round of the latest copy into each stage
    __shared__ float wbox[SWEEP_CW][12];
    constexpr int NR = n_rows<GRAD, STRETCH>();
    constexpr int NT = SWEEP_CW * 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int team = warp / R::WARPS, s0 = team * R::STAGES;  // this team's first stage
    float4* stage = dsm;
    f2* run = reinterpret_cast<f2*>(dsm + NST * R::F4);  // [NR][COMP?2:1][NT]

    const StreamK& sk = A.sk;
    const UnitList& ul = A.ul;
    // teams of different blocks first, so that few teams spread over the SMs
    const int b = team * gridDim.x + blockIdx.x;
    bool mine = true;      // the team has a unit
    long long lo_b, hi_b;  // this team's range: of the cost line, or of the list's entries
    int t0, k0;
    if constexpr (LIST) {
        __shared__ int range_s[R::TEAMS][3];
        if (warp % R::WARPS == 0) {
            int l, h, t;
            ul.range(b, l, h, t);
            if (lane == 0) range_s[team][0] = l, range_s[team][1] = h, range_s[team][2] = t;
        }
        __syncthreads();
        lo_b = range_s[team][0], hi_b = range_s[team][1], t0 = range_s[team][2];
        k0 = 0;
        mine = lo_b < hi_b;
    } else {
        lo_b = sk.lo(min(b, sk.B)), hi_b = sk.lo(min(b + 1, sk.B));
        sk.first_at_or_after(lo_b, t0, k0);
        mine = t0 < sk.TT && sk.unit_start(t0, k0) < hi_b;
    }
    const int nunits = sk.np + sk.ns;

    // Copies source unit kk (and its bounding box) into stage s, completing on full[s].
    auto issue = [&](int kk, int s, int round) {
        issued_round[s] = round;
        fence_proxy_async_smem();
        if (LIST || kk < sk.np) {
            const uint32_t bytes = R::UNIT * P_F4 * 16;
            mbar_expect_tx(&full[s], bytes + 32);
            bulk_g2s(stage + (size_t)s * R::F4, A.psrc + (size_t)kk * R::UNIT * P_F4, bytes, &full[s]);
            bulk_g2s(stage + (size_t)s * R::F4 + R::BOX, A.pbox + 2 * (kk / R::PER_TILE), 32, &full[s]);
        } else {
            const uint32_t bytes = R::UNIT * S_F4 * 16;
            mbar_expect_tx(&full[s], bytes + 32);
            bulk_g2s(stage + (size_t)s * R::F4, A.ssrc + (size_t)(kk - sk.np) * R::UNIT * S_F4, bytes, &full[s]);
            bulk_g2s(stage + (size_t)s * R::F4 + R::BOX, A.sbox + 2 * ((kk - sk.np) / R::PER_TILE), 32, &full[s]);
        }
    };
    // The unit `ahead` places after the i-th, (t, k), in this team's run, if the team owns it.
    auto unit_ahead = [&](int i, int t, int k, int ahead, int& kk) {
        if constexpr (LIST) {
            const long long q = lo_b + i + ahead;
            if (q >= hi_b) return false;
            kk = (int)ul.list[q].x;
            return true;
        }
        for (int q = 0; q < ahead; ++q)
            if (++k == nunits) k = 0, ++t;
        kk = k;
        return t < sk.TT && sk.unit_start(t, k) < hi_b;
    };

    if (warp % R::WARPS == 0 && lane == 0) {
        for (int s = 0; s < R::STAGES; ++s) {
            mbar_init(&full[s0 + s], 1);
            released[s0 + s] = 0;
            issued_round[s0 + s] = -1;
        }
        mbar_fence_init();
        for (int s = 0; mine && s < R::STAGES; ++s) {  // first fill of the ring
            int kk;
            if (!unit_ahead(0, t0, k0, s, kk)) break;
            issue(kk, s0 + s, 0);
        }
    }
    __syncthreads();
    if (!mine) return;  // the team owns no unit

    // ---------------- consumers ----------------
    const int ct = warp * 32 + lane;  // consumer thread index
    Acc<GRAD, STRETCH> acc;
    f2 X = zero2(), Y = zero2(), Z = zero2();
    int t = t0, k = k0, cur_t = -1;
    int t_end = 0;  // LIST: end of target group t's entries
    if constexpr (LIST) {
        t_end = ul.end(t);
        k = (int)ul.list[lo_b].x;
    }
    auto zero_run = [&]() {
#pragma unroll
        for (int q = 0; q < NR * (COMP ? 2 : 1); ++q) run[q * NT + ct] = zero2();
    };
    zero_run();
    auto fold_acc = [&]() {  // the sums of a tile (or half of one) into the running sums
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            if (COMP) {
                f2 hi = run[(2 * q) * NT + ct], lo = run[(2 * q + 1) * NT + ct];
                fold2(hi, lo, acc.v[q]);
                run[(2 * q) * NT + ct] = hi;
                run[(2 * q + 1) * NT + ct] = lo;
            } else {
                run[q * NT + ct] = add2(run[q * NT + ct], acc.v[q]);
            }
        }
    };
    for (int i = 0;; ++i) {
        const int s = s0 + i % R::STAGES, r = i / R::STAGES;
        int nt = t, nk = k + 1;
        bool has_next;
        if constexpr (LIST) {
            has_next = lo_b + i + 1 < hi_b;
            if (has_next) {
                nk = (int)ul.list[lo_b + i + 1].x;
                while (lo_b + i + 1 >= t_end) t_end = ul.end(++nt);
            }
        } else {
            if (nk == nunits) {
                nk = 0;
                ++nt;
            }
            has_next = nt < sk.TT && sk.unit_start(nt, nk) < hi_b;
        }
        if (t != cur_t) {  // new target tile: this warp's 64 targets, their box and strengths
            cur_t = t;
            const int i0 = t * R::TGT + (warp % R::WARPS) * 64 + lane, i1 = i0 + 32;
            float4 p0 = make_float4(0.f, 0.f, 0.f, 0.f), p1 = p0;
            const bool v0 = i0 < A.n_tgt, v1 = i1 < A.n_tgt;
            if (v0) p0 = A.tgt[i0];
            if (v1) p1 = A.tgt[i1];
            X = make_float2(p0.x, p1.x);
            Y = make_float2(p0.y, p1.y);
            Z = make_float2(p0.z, p1.z);
            warp_two_boxes(make_float3(p0.x, p0.y, p0.z), v0, make_float3(p1.x, p1.y, p1.z), v1, wbox[warp]);
        }
        if (!mbar_wait_bounded(&full[s], r & 1, A.dev_err, WAIT_LIMIT)) {
            // latched; the results are invalid.  Let this team's copies in flight land
            // (bounded) before its shared memory is released, then leave.
            if (lane == 0)
                for (int q = s0; q < s0 + R::STAGES; ++q)
                    if (issued_round[q] >= 0) mbar_wait_bounded(&full[q], issued_round[q] & 1, A.dev_err, WAIT_LIMIT);
            break;
        }

        const float4* src = stage + (size_t)s * R::F4;
        // Far particle tiles and segment tiles accumulate without the stretching rows and
        // the target strengths (fewer live registers in their loops); finish_tile adds the
        // stretching from the tile's sums afterwards.  Near particle tiles accumulate the
        // stretching pair by pair (it cancels there) with the strengths loaded for them.
        const int ti0 = t * R::TGT + (warp % R::WARPS) * 64 + lane, ti1 = ti0 + 32;
        // Near sources summed in a row before the fold.  In curve order a target's neighbours fill whole
        // tiles, and the rounding of their sums grows with the run, where in the caller's order they were
        // spread over many tiles; in halves it is below what it was there (20,011-particle hover wake,
        // error of nu_t: 8.9e-7 in the caller's order, 9.8e-7 in curve order and whole tiles, 7.1e-7 in
        // halves; 886 and 884 us a right-hand side; plain sums 9.6e-7, 1.13e-6, 7.8e-7).  Without
        // stretching near and far sources come mixed and there are fewer rows to fold: 32 (velocity at
        // 1,280 points of the BVI wake, 250,007 particles: 8.4e-8 with whole tiles, 4.7e-8; its adjoint
        // dL/dx 2.0e-7 with halves, 1.6e-7; the times within 1%).  Teams' half tiles are short enough.
        constexpr int NEAR_RUN = KIND == SWEEP_PARTICLES ? R::UNIT
                                 : !GRAD                 ? 32
                                 : !LIST                 ? R::UNIT
                                 : !STRETCH && COMP      ? 32
                                                         : SRC_TILE / 2;
        if (LIST || (!R::SEG && k < sk.np)) {
            const int cnt = min(R::UNIT, A.n_src - k * R::UNIT);  // (the last half tile may be empty)
            const float4 tlo = src[R::BOX], thi = src[R::BOX + 1];
            if (boxes_near(wbox[warp], tlo, thi, A.nc.far2)) {
                if constexpr (!STRETCH) {
                    for (int j = 0;; j += NEAR_RUN) {
                        acc.zero();
                        particle_tile<GRAD, false, true>(acc, src + j * P_F4, min(NEAR_RUN, cnt - j), X, Y, Z, A.nc, Own{});
                        if (j + NEAR_RUN >= cnt) break;
                        fold_acc();
                    }
                } else {
                    Own own;
                    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;
                    if (ti0 < A.n_tgt) g0 = A.tstr[ti0];
                    if (ti1 < A.n_tgt) g1 = A.tstr[ti1];
                    own.gx = make_float2(g0.x, g1.x);
                    own.gy = make_float2(g0.y, g1.y);
                    own.gz = make_float2(g0.z, g1.z);
                    // Sources at least 7 sigma from both of the warp's boxes take the point-vortex
                    // form and give their stretching from their sums, as a far tile does.  (Without
                    // stretching the two forms cost alike, and one loop over the tile is cheaper:
                    // 60,000 particles, u and grad u by vpm_induce_noalloc, 4.12 and 3.79 ms.)
                    unsigned keep[SRC_TILE / 32] = {};
#pragma unroll
                    for (int h = 0; h < R::UNIT / 32; ++h) {
                        const int j = 32 * h + lane;
                        const float4 q0 = src[j * P_F4], q1 = src[j * P_F4 + 1];
                        const float4 pt = make_float4(-q0.x, -q0.z, -q1.x, 0.f);
                        keep[h] = __ballot_sync(0xffffffffu, j < cnt && boxes_near(wbox[warp], pt, pt, A.nc.far2 * 1.00001f));
                    }
                    {
                        Acc<GRAD, false> tf;
                        tf.zero();
                        particle_subset<GRAD, false, false>(tf, src, keep, 0, SRC_TILE / 32, true, cnt, X, Y, Z, A.nc, Own{});
                        finish_tile<GRAD, STRETCH>(acc, tf, A.tstr, ti0, ti1, A.n_tgt);
                    }
                    particle_subset<GRAD, true, true>(acc, src, keep, 0, NEAR_RUN / 32, false, cnt, X, Y, Z, A.nc, own);
                    if (LIST && (keep[2] | keep[3])) {
                        fold_acc();
                        acc.zero();
                        particle_subset<GRAD, true, true>(acc, src, keep, NEAR_RUN / 32, SRC_TILE / 32, false, cnt, X, Y, Z, A.nc,
                                                          own);
                    }
                }
            } else {
                Acc<GRAD, false> tf;
                tf.zero();
                particle_tile<GRAD, false, false>(tf, src, cnt, X, Y, Z, A.nc, Own{});
                finish_tile<GRAD, STRETCH>(acc, tf, A.tstr, ti0, ti1, A.n_tgt);
            }
        } else {
            const int cnt = min(R::UNIT, A.m_seg - (k - sk.np) * R::UNIT);
            const float4 tlo = src[R::BOX], thi = src[R::BOX + 1];
            const float margin = 1e-3f * tlo.w;
            const bool safe = A.core_pos && margin > 0.f && !boxes_near(wbox[warp], tlo, thi, margin * margin);
            Acc<GRAD, false> tf;
            tf.zero();
            if (R::SEG && thi.w != 0.f) {  // closed four-sided rings, packed by corner
                if (safe)
                    ring_tile<GRAD, true>(tf, src, cnt >> 2, X, Y, Z, A.vn);
                else
                    ring_tile<GRAD, false>(tf, src, cnt >> 2, X, Y, Z, A.vn);
            } else if (safe) {
                segment_tile<GRAD, false, true>(tf, src, cnt, X, Y, Z, A.vn);
            } else {
                segment_tile<GRAD, false, false>(tf, src, cnt, X, Y, Z, A.vn);
            }
            finish_tile<GRAD, STRETCH>(acc, tf, A.tstr, ti0, ti1, A.n_tgt);
        }
        __syncwarp();
        if (lane == 0) {  // the last warp to finish with stage s refills it with unit i + STAGES
            __threadfence_block();
            if (atomicAdd(&released[s], 1) == R::WARPS - 1) {
                released[s] = 0;
                __threadfence_block();
                int kk;
                if (unit_ahead(i, t, k, R::STAGES, kk)) issue(kk, s, r + 1);
            }
        }
        fold_acc();
        if (!has_next || nt != t) {  // this warp's partial of target tile (LIST: group) t
            float* P = A.part + ((size_t)(b + t) * (COMP ? 2 * NR : NR)) * R::TGT + (warp % R::WARPS) * 64 + lane;
#pragma unroll
            for (int q = 0; q < NR * (COMP ? 2 : 1); ++q) {
                const f2 v = run[q * NT + ct];
                // rows: hi of every accumulator first, then lo
                const int row = COMP ? ((q & 1) ? NR + (q >> 1) : (q >> 1)) : q;
                P[(size_t)row * R::TGT] = v.x;
                P[(size_t)row * R::TGT + 32] = v.y;
            }
            zero_run();
        }
        if (!has_next) break;
        t = nt;
        k = nk;
    }
}

// ---------------------------------------------------------------------------
// Reduction of the stream-K partial sums (fixed order) and epilogue.
// ---------------------------------------------------------------------------
struct EpiArgs {
    StreamK sk, sks;  // the particle and the segment launch
    const float* part;
    const float* part_s;
    int tgt, tgt_s;     // targets per partial sum of the two launches
    int far;            // the particle units are split between two lists
    UnitList uln, ulf;  // ... those of the particle launch and of the tensor-core launch
    const float* part_f;
    int ncomp_f;        // rows of the tensor-core launch (no stretching rows)
    int n, ncomp, comp;
    EpilogueOut o;
    const int* perm;  // where target i's outputs go (null: i)
    int* dev_err;
};

__device__ __forceinline__ void check_finite(int* dev_err, double v)
{
    if (!isfinite(v)) atomicOr(dev_err, DEV_ERR_NONFINITE);
}

// PARTS threads of a block share a target's partial sums (a few targets have many, one
// per block of a sweep), each folding every PARTS-th; 256 / PARTS targets per block.
// Latency bound: a target's partial sums are read one after the other (1,280 control
// points, 152 partial sums each: 231 us with one thread per target, 31 us with eight).
template <int PARTS>
__global__ void __launch_bounds__(256) epilogue_kernel(const EpiArgs E)
{
    constexpr int TB = 256 / PARTS;
    const int part_i = threadIdx.x / TB;
    const int i = blockIdx.x * TB + threadIdx.x % TB;
    if (PARTS == 1 && i >= E.n) return;
    // The partial sums are folded in FP32 double-float arithmetic (hi by Knuth's
    // two-sum, the low words added apart: about 48 bits) and converted to FP64 once
    // per row; the FP64 pipe, a small fraction of the FP32 rate here, keeps only the
    // per-target algebra below.
    float H[17], Lw[17];
#pragma unroll
    for (int c = 0; c < 17; ++c) H[c] = 0.f, Lw[c] = 0.f;
    // ld: targets per partial sum, a constant
    using Whole = std::integral_constant<int, TGT_TILE>;
    using Team = std::integral_constant<int, FAR_GROUP>;
    static_assert(FAR_GROUP == Ring<SWEEP_SMALL>::TGT, "targets of a team");
    auto add = [&](const float* P, int ncomp, auto ldc) {
        constexpr int ld = decltype(ldc)::value;
#pragma unroll
        for (int c = 0; c < 17; ++c) {  // a constant bound keeps the sums in registers
            if (c < ncomp) {
                float sum, err;
                two_sum(H[c], P[(size_t)c * ld], sum, err);
                H[c] = sum;
                Lw[c] = __fadd_rn(Lw[c], err);
                if (E.comp) Lw[c] = __fadd_rn(Lw[c], P[(size_t)(ncomp + c) * ld]);
            }
        }
    };
    auto add_list = [&](const UnitList& ul, const float* part, int ncomp, auto ldc) {
        constexpr int ld = decltype(ldc)::value;
        const int t = min(i, E.n - 1) / ld, l = i % ld;
        const uint2 s = ul.off[t * ul.KY], e = ul.off[(t + 1) * ul.KY];
        if (s.x >= e.x) return;
        const CostLine cl = ul.line();
        const int b0 = cl.block_of(s.y), b1 = cl.block_of(ul.list[e.x - 1].y), rows = E.comp ? 2 * ncomp : ncomp;
        for (int b = b0 + part_i; b <= b1; b += PARTS) add(part + (size_t)(b + t) * rows * ld + l, ncomp, ldc);
    };
    if (E.far) {
        add_list(E.ulf, E.part_f, E.ncomp_f, Whole{});
        if (E.ncomp == 17) {
            // the far units' transposed stretching (times 4 pi) from their sums, Gamma_i x S - 3 G'^T Gamma_i
            const float4 g = reinterpret_cast<const float4*>(E.o.str)[min(i, E.n - 1)];
            double v[14];
#pragma unroll
            for (int c = 3; c < 14; ++c) v[c] = (double)H[c] + (double)Lw[c];
            const double gzz = -(v[6] + v[10]);
            const double s[3] = {
                (g.y * v[5] - g.z * v[4]) - 3.0 * (v[6] * g.x + v[9] * g.y + v[12] * g.z),
                (g.z * v[3] - g.x * v[5]) - 3.0 * (v[7] * g.x + v[10] * g.y + v[13] * g.z),
                (g.x * v[4] - g.y * v[3]) - 3.0 * (v[8] * g.x + v[11] * g.y + gzz * g.z)};
#pragma unroll
            for (int c = 0; c < 3; ++c) H[14 + c] = (float)s[c], Lw[14 + c] = (float)(s[c] - (double)H[14 + c]);
        }
        add_list(E.uln, E.part, E.ncomp, Team{});
    }
    auto add_stream = [&](const StreamK& sk, const float* part, auto ldc) {
        constexpr int ld = decltype(ldc)::value;
        const int nunits = sk.np + sk.ns;
        if (nunits == 0) return;
        const int t = min(i, E.n - 1) / ld, l = i % ld, rows = E.comp ? 2 * E.ncomp : E.ncomp;
        const int b0 = sk.block_of(sk.unit_start(t, 0));
        const int b1 = sk.block_of(sk.unit_start(t, nunits - 1));
        for (int b = b0 + part_i; b <= b1; b += PARTS) {
            const long long lo_b = sk.lo(b), hi_b = sk.lo(b + 1);
            long long c0 = lo_b > (long long)t * sk.C ? lo_b : (long long)t * sk.C;
            int tt, kk;
            sk.first_at_or_after(c0, tt, kk);
            if (tt != t || sk.unit_start(tt, kk) >= hi_b) continue;  // block b ran no unit of tile t
            add(part + (size_t)(b + t) * rows * ld + l, E.ncomp, ldc);
        }
    };
    // the partial sums of the particle launch, then those of the segment launch
    for (int launch = E.far ? 1 : 0; launch < 2; ++launch) {
        const StreamK& sk = launch ? E.sks : E.sk;
        const float* part = launch ? E.part_s : E.part;
        if ((launch ? E.tgt_s : E.tgt) == TGT_TILE)
            add_stream(sk, part, Whole{});
        else
            add_stream(sk, part, Team{});
    }
    if constexpr (PARTS > 1) {  // fold the parts, in order
        __shared__ float sh[17][2][256];
#pragma unroll
        for (int c = 0; c < 17; ++c)
            if (c < E.ncomp) sh[c][0][threadIdx.x] = H[c], sh[c][1][threadIdx.x] = Lw[c];
        __syncthreads();
        if (part_i > 0 || i >= E.n) return;
        for (int p = 1; p < PARTS; ++p)
#pragma unroll
            for (int c = 0; c < 17; ++c)
                if (c < E.ncomp) {
                    float sum, err;
                    two_sum(H[c], sh[c][0][threadIdx.x + p * TB], sum, err);
                    H[c] = sum;
                    Lw[c] = __fadd_rn(__fadd_rn(Lw[c], err), sh[c][1][threadIdx.x + p * TB]);
                }
    }
    double acc[17];
#pragma unroll
    for (int c = 0; c < 17; ++c) acc[c] = (double)H[c] + (double)Lw[c];
    const double f4pi = 0.079577471545947667884;  // 1/(4 pi)
    const EpilogueOut& o = E.o;
    const double u0 = acc[0] * f4pi, u1 = acc[1] * f4pi, u2 = acc[2] * f4pi;
    double J[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (E.ncomp >= 14) {
        const double Sx = acc[3], Sy = acc[4], Sz = acc[5];
        const double Gzz = -(acc[6] + acc[10]);
        // J = ([S x] - 3 G') / (4 pi)
        J[0] = (-3.0 * acc[6]) * f4pi;
        J[1] = (-Sz - 3.0 * acc[7]) * f4pi;
        J[2] = (Sy - 3.0 * acc[8]) * f4pi;
        J[3] = (Sz - 3.0 * acc[9]) * f4pi;
        J[4] = (-3.0 * acc[10]) * f4pi;
        J[5] = (-Sx - 3.0 * acc[11]) * f4pi;
        J[6] = (-Sy - 3.0 * acc[12]) * f4pi;
        J[7] = (Sx - 3.0 * acc[13]) * f4pi;
        J[8] = (-3.0 * Gzz) * f4pi;
    }
    const int d = E.perm ? E.perm[i] : i;
    if (o.mode == 0) {
        o.u[d] = (float)u0;
        o.u[E.n + d] = (float)u1;
        o.u[2 * E.n + d] = (float)u2;
        if (o.grad_u)
            for (int c = 0; c < 9; ++c) o.grad_u[(size_t)c * E.n + d] = (float)J[c];
        if (o.check_finite) {
            check_finite(E.dev_err, u0 + u1 + u2);
            if (o.grad_u) check_finite(E.dev_err, J[0] + J[1] + J[2] + J[3] + J[4] + J[5] + J[6] + J[7] + J[8]);
        }
        return;
    }
    if (o.mode == 2) {  // the adjoint at particle i: u and J^T Gamma_i, the strength the target's own
        const float4 G = reinterpret_cast<const float4*>(o.str)[d];  // in the caller's order
        o.dGdt[d] = (float)u0;
        o.dGdt[E.n + d] = (float)u1;
        o.dGdt[2 * E.n + d] = (float)u2;
        for (int a = 0; a < 3; ++a) o.dxdt[(size_t)a * E.n + d] = (float)(J[a] * G.x + J[3 + a] * G.y + J[6 + a] * G.z);
        return;
    }
    // Right-hand side of Eq. 4-5 for particle i.
    const float4 G4 = reinterpret_cast<const float4*>(o.str)[i];
    const double Gm[3] = {G4.x, G4.y, G4.z};
    // Vreman: alpha = J^T, beta = Delta^2 g with g = J J^T (symmetric), Delta = sigma, so
    // B_beta = Delta^4 B_g and alpha:alpha = trace g: nu_t = c_V Delta^2 sqrt(B_g / trace g).
    auto dot3 = [&](int p, int q) { return J[3 * p] * J[3 * q] + J[3 * p + 1] * J[3 * q + 1] + J[3 * p + 2] * J[3 * q + 2]; };
    const double g00 = dot3(0, 0), g11 = dot3(1, 1), g22 = dot3(2, 2);
    const double g01 = dot3(0, 1), g02 = dot3(0, 2), g12 = dot3(1, 2);
    const double aa = g00 + g11 + g22;
    const double B = g00 * g11 - g01 * g01 + g00 * g22 - g02 * g02 + g11 * g22 - g12 * g12;
    const double nut =
        (aa > 0.0 && B > 0.0) ? (double)o.c_v * ((double)o.sigma * (double)o.sigma) * sqrt(B / aa) : 0.0;
    double s[3];
    if (E.ncomp == 17) {  // transposed stretching accumulated per target
        s[0] = acc[14] * f4pi;
        s[1] = acc[15] * f4pi;
        s[2] = acc[16] * f4pi;
    } else {
        for (int a = 0; a < 3; ++a) {
            double v = 0.0;
            for (int c = 0; c < 3; ++c) v += o.classic ? J[3 * a + c] * Gm[c] : J[3 * c + a] * Gm[c];
            s[a] = v;
        }
    }
    o.dxdt[d] = (float)(u0 + o.uinf[0]);
    o.dxdt[E.n + d] = (float)(u1 + o.uinf[1]);
    o.dxdt[2 * E.n + d] = (float)(u2 + o.uinf[2]);
    o.dGdt[d] = (float)s[0];
    o.dGdt[E.n + d] = (float)s[1];
    o.dGdt[2 * E.n + d] = (float)s[2];
    o.nu_t[d] = (float)nut;

    if (o.check_finite) check_finite(E.dev_err, u0 + u1 + u2 + s[0] + s[1] + s[2] + nut);
}

// ---------------------------------------------------------------------------
// Particle strength exchange (Eq. 5's diffusion term):
//   p_i = (2/sigma^2) sum_j nu_ij (v_i Gamma_j - v_j Gamma_i) zeta_sigma(r_ij),
//   nu_ij = nu + (nu_t,i + nu_t,j)/2, zeta of Eq. 3.
// Each block owns 64 consecutive particles (two per lane of every warp) with two bounding
// boxes (split at the largest index-order jump).  Its warps walk the source tiles 32 at a
// time, one box test per lane, and share the tiles within 7 sigma of either box among
// them, 32 sources at a time: a warp stages its sources (positions, strengths, nu_t) in its
// own slice of shared memory with coalesced loads, then every lane sums over them; the
// warps' sums are added in a fixed order.  (One warp per 64 particles left most SMs idle
// below 50,000 particles: 71 us for 2,000 and 86 us for 20,000; sixteen warps 21 and 34 us.)
// v_i Gamma_j - v_j Gamma_i is formed from two
// rounded products so that the i == j term is exactly zero; pairs beyond 7 sigma
// get exp(-r^2/2s^2) < 3e-11 and are skipped.
// ---------------------------------------------------------------------------
constexpr int PSE_T = 512;
constexpr int PSE_W = PSE_T / 32;
// FAN: particles in curve order, where 32 consecutive tiles are compact too: their common box is
// tested first, and the tiles of the few in reach.  Every block looks at every box, which with the
// tiles' alone is quadratic in the count (treecode right-hand side, 4,000,000 of the BVI wake
// 104.1 and 97.8 ms, 8,000,000 of the two-rotor wake 493 and 469 ms).
constexpr int PSE_FAN = 32;

__device__ __forceinline__ void pse_pair(float4 pi, float4 gi, float base, float4 pj, float4 gj, float ntj,
                                         float inv2s2, float cut2, float& ax, float& ay, float& az)
{
    const float rx = pi.x - pj.x, ry = pi.y - pj.y, rz = pi.z - pj.z;
    const float r2 = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
    if (r2 < cut2) {
        const float w = fmaf(0.5f, ntj, base) * expf(-r2 * inv2s2);
        const float vi = pi.w, vj = pj.w;
        ax = fmaf(w, __fsub_rn(__fmul_rn(vi, gj.x), __fmul_rn(vj, gi.x)), ax);
        ay = fmaf(w, __fsub_rn(__fmul_rn(vi, gj.y), __fmul_rn(vj, gi.y)), ay);
        az = fmaf(w, __fsub_rn(__fmul_rn(vi, gj.z), __fmul_rn(vj, gi.z)), az);
    }
}

template <bool FAN>
__global__ void __launch_bounds__(PSE_T) pse_kernel(const float4* __restrict__ pos, const float4* __restrict__ str,
                                                    const float* __restrict__ nu_t, int n,
                                                    const float4* __restrict__ box, int ntiles, float inv2s2,
                                                    float cut2, float nu, float pref, const int* __restrict__ perm,
                                                    float* __restrict__ dGdt)
{
    __shared__ float4 stage[2][PSE_W][32];  // positions and strengths; the warps' sums at the end
    __shared__ float snt[PSE_W][32];
    __shared__ float wbox[PSE_W][12];
    __shared__ unsigned found[2][PSE_W];  // tiles in reach, 32 per warp: this round's and the last one's
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 64 + lane, i1 = i0 + 32;
    const bool v0 = i0 < n, v1 = i1 < n;
    float4 p0 = make_float4(0.f, 0.f, 0.f, 0.f), p1 = p0, g0 = p0, g1 = p0;
    float nt0 = 0.f, nt1 = 0.f;
    if (v0) p0 = pos[i0], g0 = str[i0], nt0 = nu_t ? nu_t[i0] : 0.f;
    if (v1) p1 = pos[i1], g1 = str[i1], nt1 = nu_t ? nu_t[i1] : 0.f;
    warp_two_boxes(make_float3(p0.x, p0.y, p0.z), v0, make_float3(p1.x, p1.y, p1.z), v1, wbox[warp]);
    const float base0 = nu + 0.5f * nt0, base1 = nu + 0.5f * nt1;
    float a0x = 0.f, a0y = 0.f, a0z = 0.f, a1x = 0.f, a1y = 0.f, a1z = 0.f;
    float4* sp = stage[0][warp];
    float4* sg = stage[1][warp];
    // warp w takes the 32 sources w mod 4 of the tiles in reach whose number is w / 4 (mod PSE_W / 4)
    const int word = warp & 3, slot = warp >> 2;
    int met = 0;  // tiles in reach so far
    auto visit = [&](int tile) {
        if ((met++ & (PSE_W / 4 - 1)) != slot) return;
        const int j = tile * SRC_TILE + 32 * word + lane;
        // stage the sources; one at least 7 sigma from both of the warp's target boxes
        // reaches none of its targets and is left out (warp-uniformly, by ballot)
        __syncwarp();
        bool kp = false;
        if (j < n) {
            const float4 pq = pos[j];
            sp[lane] = pq;
            sg[lane] = str[j];
            snt[warp][lane] = nu_t ? nu_t[j] : 0.f;
            const float4 pt = make_float4(pq.x, pq.y, pq.z, 0.f);
            kp = boxes_near(wbox[warp], pt, pt, cut2);
        }
        unsigned m = __ballot_sync(0xffffffffu, kp);
        __syncwarp();
        for (; m; m &= m - 1) {
            const int q = __ffs(m) - 1;
            const float4 pj = sp[q], gj = sg[q];
            const float ntj = snt[warp][q];
            pse_pair(p0, g0, base0, pj, gj, ntj, inv2s2, cut2, a0x, a0y, a0z);
            pse_pair(p1, g1, base1, pj, gj, ntj, inv2s2, cut2, a1x, a1y, a1z);
        }
    };
    // one box a thread and round: of the tiles, or of PSE_FAN tiles each, which follow the tiles' boxes
    const int nboxes = FAN ? (ntiles + PSE_FAN - 1) / PSE_FAN : ntiles;
    const float4* outer = FAN ? box + 2 * (size_t)ntiles : box;
    for (int tb = 0, r = 0; tb < nboxes; tb += PSE_T, r ^= 1) {
        const int tt = tb + 32 * warp + lane;
        const bool near = tt < nboxes && boxes_near(wbox[warp], outer[2 * tt], outer[2 * tt + 1], cut2);
        const unsigned mine = __ballot_sync(0xffffffffu, near);
        if (lane == 0) found[r][warp] = mine;
        if (!__syncthreads_or((int)mine)) continue;
#pragma unroll 1
        for (int w = 0; w < PSE_W; ++w)
            for (unsigned mask = found[r][w]; mask; mask &= mask - 1) {
                const int k = tb + 32 * w + __ffs(mask) - 1;
                if constexpr (FAN) {
                    const int t = k * PSE_FAN + lane;
                    unsigned in = __ballot_sync(
                        0xffffffffu, t < ntiles && boxes_near(wbox[warp], box[2 * (size_t)t], box[2 * (size_t)t + 1], cut2));
#pragma unroll 1
                    for (; in; in &= in - 1) visit(k * PSE_FAN + __ffs(in) - 1);
                } else {
                    visit(k);
                }
            }
    }
    // the warps' sums in a fixed order, one thread per target
    __syncthreads();
    float4* sums = &stage[0][0][0];  // [PSE_W][64]
    sums[warp * 64 + lane] = make_float4(a0x, a0y, a0z, 0.f);
    sums[warp * 64 + 32 + lane] = make_float4(a1x, a1y, a1z, 0.f);
    __syncthreads();
    const int i = blockIdx.x * 64 + threadIdx.x;
    if (threadIdx.x < 64 && i < n) {
        float4 v = sums[threadIdx.x];
        for (int w = 1; w < PSE_W; ++w) {
            const float4 x = sums[w * 64 + threadIdx.x];
            v.x += x.x, v.y += x.y, v.z += x.z;
        }
        const int d = perm ? perm[i] : i;
        dGdt[d] += pref * v.x;
        dGdt[n + d] += pref * v.y;
        dGdt[2 * n + d] += pref * v.z;
    }
}

// Bounding boxes of the particle tiles in the caller's order.
__global__ void __launch_bounds__(SRC_TILE) tile_box_kernel(const float4* __restrict__ pos, int n,
                                                            float4* __restrict__ box)
{
    const int j = blockIdx.x * SRC_TILE + threadIdx.x;
    float v[6] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};  // least of x and of -x
    if (j < n) {
        const float4 p = pos[j];
        v[0] = p.x, v[1] = p.y, v[2] = p.z, v[3] = -p.x, v[4] = -p.y, v[5] = -p.z;
    }
    __shared__ float sb[SRC_TILE / 32][6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        for (int o = 16; o > 0; o >>= 1) v[c] = fminf(v[c], __shfl_xor_sync(0xffffffffu, v[c], o));
        if ((threadIdx.x & 31) == 0) sb[threadIdx.x >> 5][c] = v[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < SRC_TILE / 32; ++w)
            for (int c = 0; c < 6; ++c) v[c] = fminf(v[c], sb[w][c]);
        box[2 * blockIdx.x] = make_float4(v[0], v[1], v[2], 0.f);
        box[2 * blockIdx.x + 1] = make_float4(-v[3], -v[4], -v[5], 0.f);
    }
}

// Boxes of PSE_FAN tiles each, behind the ntiles tile boxes; a warp per box.
__global__ void __launch_bounds__(256) fan_box_kernel(float4* __restrict__ box, int ntiles)
{
    const int k = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31, t = k * PSE_FAN + lane;
    static_assert(PSE_FAN == 32, "a tile per lane");
    if (k * PSE_FAN >= ntiles) return;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (t < ntiles) {
        const float4 a = box[2 * (size_t)t], b = box[2 * (size_t)t + 1];
        lo[0] = a.x, lo[1] = a.y, lo[2] = a.z, hi[0] = b.x, hi[1] = b.y, hi[2] = b.z;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
    if (lane == 0) {
        float4* out = box + 2 * ((size_t)ntiles + k);
        out[0] = make_float4(lo[0], lo[1], lo[2], 0.f);
        out[1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    }
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
__device__ int g_dev_err;  // device error word (one instance per device)

namespace {
std::mutex g_mu;
int g_sm[64];
int g_blocks[64][8 * SWEEP_KINDS];
bool g_attr[64][8 * SWEEP_KINDS];
}  // namespace

static int cur_dev()
{
    int d = 0;
    cudaGetDevice(&d);
    return d;
}

int sm_count()
{
    const int d = cur_dev();
    std::lock_guard<std::mutex> lk(g_mu);
    if (d < 0 || d >= 64) return 0;
    if (!g_sm[d]) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d) != cudaSuccess) v = 0;
        g_sm[d] = v;
    }
    return g_sm[d];
}

// The device error word of the current device, looked up on every call (a cheap
// query once the module is loaded) so that the address is never stale.
int* dev_err_ptr()
{
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_dev_err) != cudaSuccess) return nullptr;
    return static_cast<int*>(p);
}

static int variant(bool G, bool C, bool S, int K) { return 8 * K + (G ? 4 : 0) + (C ? 2 : 0) + (S ? 1 : 0); }

// Opts the kernel into its dynamic shared memory (once per device) and returns the resident blocks per SM.
template <bool G, bool C, bool S, int K>
static int prepare_kernel(int d)
{
    const int v = variant(G, C, S, K);
    const size_t smem = sweep_smem_bytes<G, C, S, K>();
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (d >= 0 && d < 64 && g_attr[d][v]) return g_blocks[d][v];
    }
    cudaFuncSetAttribute(sweep_kernel<G, C, S, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, sweep_kernel<G, C, S, K>, SWEEP_TPB, smem) != cudaSuccess)
        nb = 1;
    if (nb < 1) nb = 1;
    std::lock_guard<std::mutex> lk(g_mu);
    if (d >= 0 && d < 64) {
        g_blocks[d][v] = nb;
        g_attr[d][v] = true;
    }
    return nb;
}

template <int K>
static int blocks_per_sm_kind(bool g, bool c, bool s)
{
    const int d = cur_dev();
    if (g && s) return c ? prepare_kernel<true, true, true, K>(d) : prepare_kernel<true, false, true, K>(d);
    if (g) return c ? prepare_kernel<true, true, false, K>(d) : prepare_kernel<true, false, false, K>(d);
    return c ? prepare_kernel<false, true, false, K>(d) : prepare_kernel<false, false, false, K>(d);
}

static int blocks_per_sm(bool g, bool c, bool s, int kind)
{
    return kind == SWEEP_SEGMENTS ? blocks_per_sm_kind<SWEEP_SEGMENTS>(g, c, s)
           : kind == SWEEP_SEG_SMALL ? blocks_per_sm_kind<SWEEP_SEG_SMALL>(g, c, s)
           : kind == SWEEP_NEAR   ? blocks_per_sm_kind<SWEEP_NEAR>(g, c, s)
           : kind == SWEEP_SMALL  ? blocks_per_sm_kind<SWEEP_SMALL>(g, c, s)
                                  : blocks_per_sm_kind<SWEEP_PARTICLES>(g, c, s);
}

int sweep_blocks(bool grad, bool comp, bool stretch, int kind)
{
    const int sms = sm_count();
    return blocks_per_sm(grad, comp, stretch && grad, kind) * (sms > 0 ? sms : 1);
}

SweepPlan plan_sweep(int64_t n_tgt, int64_t n_src, int64_t m_seg, bool grad, bool comp, Carve& cv, bool stretch,
                     bool allow_far)
{
    SweepPlan p;
    p.n_tgt = (int)n_tgt;
    p.n_src = (int)n_src;
    p.m_seg = (int)m_seg;
    p.grad = grad;
    p.comp = comp;
    p.stretch = stretch && grad;
    p.ncomp = grad ? (p.stretch ? 17 : 14) : 3;
    p.TT = (int)((n_tgt + TGT_TILE - 1) / TGT_TILE);
    p.SP = (int)((n_src + SRC_TILE - 1) / SRC_TILE);
    p.SS = (int)((m_seg + SRC_TILE - 1) / SRC_TILE);
    const long long units_p = (long long)p.TT * p.SP;
    // The workspace must not shrink as a count grows (a caller may hold one for the largest counts it
    // will have), so what the far sweep needs is reserved by the units alone, also where it is not used:
    // particles onto themselves below FAR_SORT_MIN, and beyond FAR_MAX_UNITS.
    const bool reserve = allow_far && units_p >= (grad ? FAR_MIN_UNITS_GRAD : FAR_MIN_UNITS_VEL);
    p.far = reserve && units_p <= FAR_MAX_UNITS && !(n_tgt == n_src && grad && n_src < FAR_SORT_MIN);
    // particle tiles and segment tiles: one stream-K plan (and launch) each
    auto plan = [&](StreamK& sk, int kind, int np, int ns) {
        const bool teams = kind == SWEEP_SMALL || kind == SWEEP_SEG_SMALL;
        const int per_tile = teams ? Ring<SWEEP_SMALL>::PER_TILE : 1;
        const int tgt = teams ? Ring<SWEEP_SMALL>::TGT : TGT_TILE;
        sk.TT = (int)((n_tgt + tgt - 1) / tgt);
        sk.np = np * per_tile;
        sk.ns = ns * per_tile;
        sk.wp = UNIT_W_P;
        sk.ws = grad ? UNIT_W_S_GRAD : UNIT_W_S_VEL;
        sk.C = (long long)sk.np * sk.wp + (long long)sk.ns * sk.ws;
        sk.tot = (long long)sk.TT * sk.C;
        const long long units = (long long)sk.TT * (sk.np + sk.ns);
        long long B = (long long)sweep_blocks(grad, comp, p.stretch, kind) * (teams ? Ring<SWEEP_SMALL>::TEAMS : 1);
        if (B > units) B = units;
        if (B < 1) B = 1;
        sk.B = (int)B;
    };
    // A small problem with few segments sweeps both kinds of tile in one launch; otherwise the
    // segment tiles have a launch of their own, where closed rings are packed by corner.
    const long long units_s = (long long)p.TT * p.SS;
    p.kind = units_p < SMALL_MAX_UNITS || p.TT < SMALL_FEW_TILES ? SWEEP_SMALL : SWEEP_PARTICLES;
    p.mixed = p.SP > 0 && p.SS > 0 && p.SS <= MIXED_MAX_TILES && !p.far && p.kind == SWEEP_SMALL;
    p.kind_s = units_s < SEG_SMALL_MAX_UNITS ? SWEEP_SEG_SMALL : SWEEP_SEGMENTS;
    plan(p.sk, p.kind, p.SP, p.mixed ? p.SS : 0);
    plan(p.sks, p.kind_s, 0, p.mixed ? 0 : p.SS);
    const size_t tgt_k = p.kind == SWEEP_SMALL ? Ring<SWEEP_SMALL>::TGT : TGT_TILE,
                 tgt_s = p.kind_s == SWEEP_SEG_SMALL ? Ring<SWEEP_SEG_SMALL>::TGT : TGT_TILE;
    p.off_psrc = cv.take((size_t)p.SP * SRC_TILE * P_F4 * 16);
    p.off_pbox = cv.take((size_t)p.SP * 2 * 16);
    p.off_ssrc = cv.take((size_t)p.SS * SRC_TILE * S_F4 * 16);
    p.off_sbox = cv.take((size_t)p.SS * 2 * 16);
    const size_t rows = (size_t)(comp ? 2 : 1) * p.ncomp;
    size_t part = p.sk.np + p.sk.ns > 0 ? (size_t)(p.sk.TT + p.sk.B) * rows * tgt_k * sizeof(float) : 0;
    if (reserve) {  // one buffer for the particle launch's sums in either form
        p.B_near = sweep_blocks(grad, comp, p.stretch, SWEEP_NEAR);
        part = std::max(part, (size_t)(p.TT * FAR_GROUPS + p.B_near * Ring<SWEEP_NEAR>::TEAMS) * rows * FAR_GROUP * sizeof(float));
    }
    if (part > 0) p.off_part = cv.take(part);
    if (p.sks.ns > 0) p.off_part_s = cv.take((size_t)(p.sks.TT + p.sks.B) * rows * tgt_s * sizeof(float));
    // Units on the tensor cores
    if (reserve) {
        p.KY = (p.SP + FAR_KCH - 1) / FAR_KCH;
        const long long units = std::min(units_p, FAR_MAX_UNITS);
        p.B_far = (int)std::min<long long>(std::max(sm_count(), 1), units);
        const size_t rows_f = (size_t)(comp ? 2 : 1) * (grad ? 14 : 3);
        p.off_ftile = cv.take((size_t)p.SP * far_tile_bytes(grad));
        p.off_fmask = cv.take((size_t)units * sizeof(unsigned));
        p.off_fcnt = cv.take((size_t)p.TT * p.KY * (1 + FAR_GROUPS) * sizeof(uint2));
        p.off_nlist = cv.take((size_t)units * FAR_GROUPS * sizeof(uint2));
        p.off_noff = cv.take(((size_t)p.TT * p.KY * FAR_GROUPS + 1) * sizeof(uint2));
        p.off_flist = cv.take((size_t)units * sizeof(uint2));
        p.off_foff = cv.take(((size_t)p.TT * p.KY + 1) * sizeof(uint2));
        p.off_part_f = cv.take((size_t)(p.TT + p.B_far) * rows_f * TGT_TILE * sizeof(float));
        if (grad) {  // particles onto themselves, which fewer targets or sources may be
            const size_t n = (size_t)std::min(n_src, n_tgt);
            const bool sortable = curve_layout((int64_t)n, cv, p.curve);
            // With the gradient only: the velocity alone costs so little that the sort does not pay on a
            // wake in its own order (17,000 of the BVI wake 294 us without and 329 us with it, 60,000
            // 1,582 and 1,679; of the hover wake 296 and 314, 1,771 and 1,716 us).
            p.sort = p.far && n_tgt == n_src && sortable;
            p.off_spos = cv.take(n * 16);
            p.off_sstr = cv.take(n * 16);
            p.off_obox = cv.take((n + SRC_TILE - 1) / SRC_TILE * 2 * 16);
        }
    }
    p.bytes = cv.off;
    return p;
}

// (7 sigma)^2, above zero for any core: a pair at zero distance is near, and contributes nothing.
static float far2_of(float sigma)
{
    return std::max((float)((double)RHO_FAR * RHO_FAR * (double)sigma * (double)sigma), FLT_MIN);
}

template <bool G, bool C, bool S>
static void launch_sweep(const SweepArgs& A, int B, int kind, cudaStream_t st)
{
    if (kind == SWEEP_SEG_SMALL)
        sweep_kernel<G, C, S, SWEEP_SEG_SMALL><<<B, SWEEP_TPB, sweep_smem_bytes<G, C, S, SWEEP_SEG_SMALL>(), st>>>(A);
    else if (kind == SWEEP_NEAR)
        sweep_kernel<G, C, S, SWEEP_NEAR><<<B, SWEEP_TPB, sweep_smem_bytes<G, C, S, SWEEP_NEAR>(), st>>>(A);
    else if (kind == SWEEP_SMALL)
        sweep_kernel<G, C, S, SWEEP_SMALL><<<B, SWEEP_TPB, sweep_smem_bytes<G, C, S, SWEEP_SMALL>(), st>>>(A);
    else if (kind == SWEEP_SEGMENTS)
        sweep_kernel<G, C, S, SWEEP_SEGMENTS><<<B, SWEEP_TPB, sweep_smem_bytes<G, C, S, SWEEP_SEGMENTS>(), st>>>(A);
    else
        sweep_kernel<G, C, S, SWEEP_PARTICLES><<<B, SWEEP_TPB, sweep_smem_bytes<G, C, S, SWEEP_PARTICLES>(), st>>>(A);
}

cudaError_t run_sweep(const SweepPlan& p, char* ws, const float* tgt, const float* src_pos, const float* src_str,
                      const float* seg_a, const float* seg_b, float sigma, float seg_core, int vatistas_n,
                      const EpilogueOut& out, cudaStream_t st)
{
    if (p.n_tgt == 0) return cudaSuccess;
    float4* psrc = reinterpret_cast<float4*>(ws + p.off_psrc);
    float4* pbox = reinterpret_cast<float4*>(ws + p.off_pbox);
    float4* ssrc = reinterpret_cast<float4*>(ws + p.off_ssrc);
    float4* sbox = reinterpret_cast<float4*>(ws + p.off_sbox);
    float* part = reinterpret_cast<float*>(ws + p.off_part);
    float* part_s = reinterpret_cast<float*>(ws + p.off_part_s);
    // Particles onto themselves are swept in curve order
    const bool sorted = p.sort && tgt == src_pos;
    const int* perm = nullptr;
    float4* spos = reinterpret_cast<float4*>(ws + p.off_spos);
    float4* sstr = reinterpret_cast<float4*>(ws + p.off_sstr);
    if (sorted) {
        const cudaError_t e = run_curve_sort(p.curve, ws, reinterpret_cast<const float4*>(src_pos), p.n_src, st);
        if (e != cudaSuccess) return e;
        perm = reinterpret_cast<const int*>(ws + p.curve.perm);
    }
    if (p.SP > 0) {
        trace_launch();
        pack_particles_kernel<<<p.SP, SRC_TILE, 0, st>>>(reinterpret_cast<const float4*>(src_pos),
                                                         reinterpret_cast<const float4*>(src_str), p.n_src, perm, spos,
                                                         sstr, psrc, pbox);
    }
    const float* own = out.str;  // the targets' own strengths, in the targets' order
    if (sorted) {
        tgt = src_pos = reinterpret_cast<const float*>(spos);
        src_str = reinterpret_cast<const float*>(sstr);
        own = src_str;
    }
    if (p.SS > 0) {
        trace_launch();
        pack_segments_kernel<<<p.SS, SRC_TILE, 0, st>>>(reinterpret_cast<const float4*>(seg_a),
                                                        reinterpret_cast<const float4*>(seg_b), p.m_seg, seg_core,
                                                        vatistas_n, p.mixed ? 0 : 1, ssrc, sbox);
    }
    int* err = dev_err_ptr();
    UnitList uln{}, ulf{};
    const unsigned char* ftile = reinterpret_cast<const unsigned char*>(ws + p.off_ftile);
    if (p.far) {
        auto list = [&](size_t l, size_t o, int T, int B, int max_cost) {
            UnitList u;
            u.list = reinterpret_cast<const uint2*>(ws + l);
            u.off = reinterpret_cast<const uint2*>(ws + o);
            u.TT = T;
            u.KY = p.KY;
            u.B = B;
            u.max_cost = max_cost;
            return u;
        };
        uln = list(p.off_nlist, p.off_noff, p.TT * FAR_GROUPS, p.B_near * Ring<SWEEP_NEAR>::TEAMS,
                   Ring<SWEEP_NEAR>::WARPS * NEAR_COST);
        ulf = list(p.off_flist, p.off_foff, p.TT, p.B_far, FAR_COST_FIRST + FAR_GROUPS - 1);
        cudaError_t e = run_far_pack(reinterpret_cast<const float4*>(src_pos), reinterpret_cast<const float4*>(src_str),
                                     p.n_src, pbox, p.SP, p.grad, reinterpret_cast<unsigned char*>(ws + p.off_ftile), st);
        if (e == cudaSuccess)
            e = run_far_lists(reinterpret_cast<const float4*>(tgt), p.n_tgt, ftile, p.SP, p.TT, p.grad, pbox,
                              far2_of(sigma),
                              reinterpret_cast<unsigned*>(ws + p.off_fmask),
                              reinterpret_cast<uint2*>(ws + p.off_fcnt), reinterpret_cast<uint2*>(ws + p.off_nlist),
                              reinterpret_cast<uint2*>(ws + p.off_noff), reinterpret_cast<uint2*>(ws + p.off_flist),
                              reinterpret_cast<uint2*>(ws + p.off_foff), st);
        if (e != cudaSuccess) return e;
    }
    if (p.SP + p.SS > 0) {
        // shared-memory opt-in
        if (p.sk.np + p.sk.ns > 0) blocks_per_sm(p.grad, p.comp, p.stretch, p.far ? SWEEP_NEAR : p.kind);
        if (p.sks.ns > 0) blocks_per_sm(p.grad, p.comp, p.stretch, p.kind_s);
        SweepArgs A;
        A.tgt = reinterpret_cast<const float4*>(tgt);
        A.tstr = p.stretch ? reinterpret_cast<const float4*>(own) : nullptr;
        A.n_tgt = p.n_tgt;
        A.psrc = psrc;
        A.pbox = pbox;
        A.n_src = p.n_src;
        A.ssrc = ssrc;
        A.sbox = sbox;
        A.core_pos = seg_core > 0.f ? 1 : 0;
        A.m_seg = p.m_seg;
        A.vn = vatistas_n;
        A.sk = p.sk;
        const double s = sigma;
        A.nc.inv_s2 = (float)(1.0 / (s * s));
        A.nc.inv_s3 = (float)(1.0 / (s * s * s));
        A.nc.inv_s5 = (float)(1.0 / (s * s * s * s * s));
        A.nc.far2 = far2_of(sigma);
        A.dev_err = err;
        for (int kind = 0; kind < 2; ++kind) {
            const bool seg = kind == 1;
            if ((seg ? p.sks.ns : p.sk.np + p.sk.ns) == 0) continue;
            TraceScope ts(seg ? VPM_TRACE_SEGMENTS : out.mode == 2 ? VPM_TRACE_ADJOINT : p.grad ? VPM_TRACE_SWEEP : VPM_TRACE_SWEEP_VEL, st);
            A.sk = seg ? p.sks : p.sk;
            A.part = seg ? part_s : part;
            const int k = seg ? p.kind_s : p.far ? SWEEP_NEAR : p.kind;
            // with teams: a block for each of the first teams, up to the resident number
            const int B = k == SWEEP_NEAR    ? p.B_near
                          : k == SWEEP_PARTICLES || k == SWEEP_SEGMENTS ? A.sk.B
                                             : std::min(A.sk.B, sweep_blocks(p.grad, p.comp, p.stretch, k));
            if (k == SWEEP_NEAR) {
                A.ul = uln;
                FarArgs F;
                F.tgt = A.tgt;
                F.n_tgt = p.n_tgt;
                F.tiles = ftile;
                F.ul = ulf;
                F.part = reinterpret_cast<float*>(ws + p.off_part_f);
                F.dev_err = err;
                trace_launch();
                const cudaError_t e = run_far_sweep(F, p.grad, p.comp, st);
                if (e != cudaSuccess) return e;
            }
            if (p.grad && p.stretch) {
                if (p.comp)
                    launch_sweep<true, true, true>(A, B, k, st);
                else
                    launch_sweep<true, false, true>(A, B, k, st);
            } else if (p.grad) {
                if (p.comp)
                    launch_sweep<true, true, false>(A, B, k, st);
                else
                    launch_sweep<true, false, false>(A, B, k, st);
            } else {
                if (p.comp)
                    launch_sweep<false, true, false>(A, B, k, st);
                else
                    launch_sweep<false, false, false>(A, B, k, st);
            }
        }
    }
    EpiArgs E;
    E.sk = p.sk;
    E.part = part;
    E.sks = p.sks;
    E.part_s = part_s;
    E.tgt = p.kind == SWEEP_SMALL ? Ring<SWEEP_SMALL>::TGT : TGT_TILE;
    E.tgt_s = p.kind_s == SWEEP_SEG_SMALL ? Ring<SWEEP_SEG_SMALL>::TGT : TGT_TILE;
    E.far = p.far ? 1 : 0;
    E.uln = uln;
    E.ulf = ulf;
    E.part_f = reinterpret_cast<const float*>(ws + p.off_part_f);
    E.ncomp_f = p.grad ? 14 : 3;
    E.n = p.n_tgt;
    E.ncomp = p.ncomp;
    E.comp = p.comp ? 1 : 0;
    E.o = out;
    if (out.mode != 2) E.o.str = own;  // (in the adjoint the sources' strengths are not the targets')
    E.perm = perm;
    E.dev_err = err;
    trace_launch();
    // Threads per target: enough to give every SM a few blocks
    const long long want = 4LL * 256 * std::max(sm_count(), 1);
    if (16LL * p.n_tgt <= want)
        epilogue_kernel<16><<<(p.n_tgt + 15) / 16, 256, 0, st>>>(E);
    else if (2LL * p.n_tgt <= want)
        epilogue_kernel<8><<<(p.n_tgt + 31) / 32, 256, 0, st>>>(E);
    else
        epilogue_kernel<1><<<(p.n_tgt + 255) / 256, 256, 0, st>>>(E);
    return cudaGetLastError();
}

static cudaError_t launch_pse(const float4* pos, const float4* str, const float* nu_t, const int* perm,
                              const float4* box, bool fan, int n, float sigma, float nu, float* dGdt, cudaStream_t st)
{
    const double s = sigma;
    const float inv2s2 = (float)(0.5 / (s * s));
    const float cut2 = (float)((double)RHO_FAR * RHO_FAR * s * s);
    // (2/sigma^2) (2 pi sigma^2)^(-3/2)
    const float pref = (float)(2.0 / (s * s) * pow(2.0 * 3.14159265358979323846 * s * s, -1.5));
    TraceScope ts(VPM_TRACE_PSE, st);
    (fan ? pse_kernel<true> : pse_kernel<false>)<<<(n + 63) / 64, PSE_T, 0, st>>>(
        pos, str, nu_t, n, box, (n + SRC_TILE - 1) / SRC_TILE, inv2s2, cut2, nu, pref, perm, dGdt);
    return cudaGetLastError();
}

size_t pse_box_bytes(int64_t n)
{
    const size_t tiles = (size_t)((n + SRC_TILE - 1) / SRC_TILE);
    return (tiles + (tiles + PSE_FAN - 1) / PSE_FAN) * 32;
}

cudaError_t run_pse_sorted(const float4* pos, const float4* str, const float* nu_t, const int* perm, float4* box, int n,
                           float sigma, float nu, float* dGdt, cudaStream_t st)
{
    const int tiles = (n + SRC_TILE - 1) / SRC_TILE;
    trace_launch(2);
    tile_box_kernel<<<tiles, SRC_TILE, 0, st>>>(pos, n, box);
    fan_box_kernel<<<((tiles + PSE_FAN - 1) / PSE_FAN + 7) / 8, 256, 0, st>>>(box, tiles);
    return launch_pse(pos, str, nu_t, perm, box, true, n, sigma, nu, dGdt, st);
}

cudaError_t run_pse(const SweepPlan& p, char* ws, const float* pos, const float* str, const float* nu_t, int n,
                    float sigma, float nu, float* dGdt, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    const float4* pos4 = reinterpret_cast<const float4*>(pos);
    const float4* str4 = reinterpret_cast<const float4*>(str);
    // the exchange takes the particles in the caller's order, which needs no sorted copy of nu_t
    // (100,000 particles of the hover wake: 164 us, in curve order 158; 20,000: 34 and 44)
    float4* box = reinterpret_cast<float4*>(ws + (p.sort ? p.off_obox : p.off_pbox));
    if (p.sort) {
        trace_launch();
        tile_box_kernel<<<(n + SRC_TILE - 1) / SRC_TILE, SRC_TILE, 0, st>>>(pos4, n, box);
    }
    return launch_pse(pos4, str4, nu_t, nullptr, box, false, n, sigma, nu, dGdt, st);
}

}  // namespace vpm
