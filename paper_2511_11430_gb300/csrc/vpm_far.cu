// The tensor-core far sweep and the unit lists (vpm_far.cuh).
#include <cuda_fp16.h>

#include <algorithm>
#include <cub/device/device_radix_sort.cuh>
#include <mutex>
#include <type_traits>

#include "vpm_far.cuh"
#include "vpm_kernel.cuh"

namespace vpm {

// ---------------------------------------------------------------------------
// tcgen05 wrappers (cta_group::1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tm_alloc(uint32_t* dst, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(cols)
                 : "memory");
}
__device__ __forceinline__ void tm_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tm_dealloc(uint32_t addr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}
__device__ __forceinline__ void tm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tm_st8(uint32_t addr, const uint32_t* r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
__device__ __forceinline__ void tm_st4(uint32_t addr, const uint32_t* r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
}
__device__ __forceinline__ void tm_ld8(uint32_t addr, float* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(addr));
}
// True in one lane of the warp.  The instruction stream guarded by it is known to run in a
// single thread: MMAs issue every 16 cycles there (N = 32), against 45 behind `lane == 0`.
__device__ __forceinline__ bool elect_one()
{
    uint32_t e;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 r;\n\t"
        "elect.sync r|p, 0xffffffff;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(e));
    return e != 0;
}
// Arrives on `bar` when every MMA this thread has issued is complete.
__device__ __forceinline__ void tm_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// D[128 x N] (+)= A[128 x 16] (TMEM, FP16) B[16 x N] (shared memory, FP16).
__device__ __forceinline__ void tm_mma_f16(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(bdesc), "r"(idesc), "r"(acc)
        : "memory");
}
// K-major shared-memory operand without swizzle: 8 x 16-byte core matrices of 128
// contiguous bytes; `lead` bytes between the two along K, `stride` between those along N.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lead, uint32_t stride)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lead >> 4) << 16) | ((uint64_t)(stride >> 4) << 32) |
           (1ull << 46);
}
// Instruction descriptor of kind::f16: FP32 accumulator, FP16 operands, both K-major.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N)
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

constexpr uint32_t IDESC_NEG_A = 1u << 13;

__device__ __forceinline__ uint32_t pack_h2(f2 v)
{
    const __half2 h = __float22half2_rn(v);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// The weights w = t^(-5/2) - 1 (velocity only: t^(-3/2) - 1) of two sources as FP16 pairs:
// hi = fp16(w) and neg = fp16(hi - w), the second multiplied with the operand's sign flipped.
template <bool GRAD>
__device__ __forceinline__ void far_weight(f2 t, uint32_t& hi, uint32_t& neg)
{
    const f2 rs = rsqrt2_approx(t);
    const f2 i2 = mul2(rs, rs);
    const f2 w = GRAD ? fma2(mul2(i2, i2), rs, splat(-1.f)) : fma2(i2, rs, splat(-1.f));
    hi = pack_h2(w);
    f2 d;
    asm("{\n\t.reg .b16 a, b;\n\t"
        "mov.b32 {a, b}, %2;\n\t"
        "sub.rn.f32.f16 %0, a, %3;\n\t"
        "sub.rn.f32.f16 %1, b, %4;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "r"(hi), "f"(w.x), "f"(w.y));
    neg = pack_h2(d);
}

// ---------------------------------------------------------------------------
// Curve order.  Particles come in the caller's order (filament after filament, or row
// after row of a converted wake), in which 128 consecutive ones can span the wake; along
// a Hilbert curve they are compact, and so are the target groups.  (Morton order leaves
// jumps: on the 20,000-particle hover wake 74% of the pairs pass the acceptance test in
// Morton order, 80% in Hilbert order and 1% in the generator's filament order.)
// 8 bits per axis: three radix passes, and cells far smaller than a tile.  Where the cost of a
// poor order grows with the square of the count (the treecode's exchange), 21 bits: a stray
// particle a thousand wake lengths away leaves the rest in a few of the coarse cells, in the
// caller's order (1,000,000 particles in no order, right-hand side: 531 ms, with the fine cells 31).
// ---------------------------------------------------------------------------
template <bool FINE>
struct Curve {
    using Key = typename std::conditional<FINE, unsigned long long, unsigned>::type;
    static constexpr int BITS = FINE ? 21 : 8;
};
constexpr int CURVE_BND_BLOCKS = 128;  // partial boxes of the curve's bounding cube

__global__ void __launch_bounds__(256) curve_bounds_kernel(const float4* __restrict__ pos, int n, float* __restrict__ bnd)
{
    float v[6] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};  // least of x and of -x
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const float4 p = pos[i];
        v[0] = fminf(v[0], p.x), v[1] = fminf(v[1], p.y), v[2] = fminf(v[2], p.z);
        v[3] = fminf(v[3], -p.x), v[4] = fminf(v[4], -p.y), v[5] = fminf(v[5], -p.z);
    }
    __shared__ float sh[8][6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        for (int o = 16; o > 0; o >>= 1) v[c] = fminf(v[c], __shfl_xor_sync(0xffffffffu, v[c], o));
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][c] = v[c];
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        float m = sh[0][threadIdx.x];
        for (int w = 1; w < 8; ++w) m = fminf(m, sh[w][threadIdx.x]);
        bnd[blockIdx.x * 6 + threadIdx.x] = m;
    }
}

// Position along the Hilbert curve of a cell (Skilling, "Programming the Hilbert curve",
// AIP Conf. Proc. 707, 2004: the transpose form).
template <bool FINE>
__device__ __forceinline__ typename Curve<FINE>::Key hilbert_key(unsigned x, unsigned y, unsigned z)
{
    constexpr int BITS = Curve<FINE>::BITS;
    unsigned X[3] = {x, y, z};
#pragma unroll
    for (unsigned Q = 1u << (BITS - 1); Q > 1; Q >>= 1) {
        const unsigned P = Q - 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (X[i] & Q) {
                X[0] ^= P;
            } else {
                const unsigned t = (X[0] ^ X[i]) & P;
                X[0] ^= t;
                X[i] ^= t;
            }
        }
    }
    X[1] ^= X[0];
    X[2] ^= X[1];
    unsigned t = 0;
#pragma unroll
    for (unsigned Q = 1u << (BITS - 1); Q > 1; Q >>= 1)
        if (X[2] & Q) t ^= Q - 1;
    typename Curve<FINE>::Key k = 0;
#pragma unroll
    for (int b = BITS - 1; b >= 0; --b)
#pragma unroll
        for (int i = 0; i < 3; ++i) k = (k << 1) | (((X[i] ^ t) >> b) & 1u);
    return k;
}

template <bool FINE>
__global__ void __launch_bounds__(256) curve_keys_kernel(const float4* __restrict__ pos, int n,
                                                       const float* __restrict__ bnd, int nb,
                                                       typename Curve<FINE>::Key* __restrict__ key,
                                                       int* __restrict__ idx)
{
    constexpr int BITS = Curve<FINE>::BITS;
    __shared__ float box[6];
    if (threadIdx.x < 192) {  // six warps, one component each
        const int c = threadIdx.x >> 5;
        float m = INFINITY;
        for (int i = threadIdx.x & 31; i < nb; i += 32) m = fminf(m, bnd[6 * i + c]);
        for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0) box[c] = m;
    }
    __syncthreads();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float4 p = pos[i];
    const float ext = fmaxf(-box[3] - box[0], fmaxf(-box[4] - box[1], -box[5] - box[2]));
    const float s = ext > 0.f && isfinite(ext) ? (float)(1 << BITS) / ext : 0.f;
    auto cell = [&](float x, float lo) {
        const float f = (x - lo) * s;  // a non-finite coordinate goes to cell 0
        return f > 0.f ? min((unsigned)fminf(f, 4e6f), (1u << BITS) - 1u) : 0u;
    };
    key[i] = hilbert_key<FINE>(cell(p.x, box[0]), cell(p.y, box[1]), cell(p.z, box[2]));
    idx[i] = i;
}

template <bool FINE>
static cudaError_t curve_sort(void* ws, size_t& bytes, const void* key, void* key2, const int* idx, int* perm, int n,
                              cudaStream_t st)
{
    using Key = typename Curve<FINE>::Key;
    return cub::DeviceRadixSort::SortPairs(ws, bytes, static_cast<const Key*>(key), static_cast<Key*>(key2), idx, perm,
                                           n, 0, 3 * Curve<FINE>::BITS, st);
}

bool curve_layout(int64_t n, Carve& cv, CurveWs& w, bool fine)
{
    const bool ok = (fine ? curve_sort<true> : curve_sort<false>)(nullptr, w.cub_bytes, nullptr, nullptr, nullptr,
                                                                  nullptr, (int)n, nullptr) == cudaSuccess;
    const size_t key_bytes = fine ? sizeof(Curve<true>::Key) : sizeof(Curve<false>::Key);
    w.fine = fine;
    w.bnd = cv.take(CURVE_BND_BLOCKS * 6 * sizeof(float));
    w.key = cv.take((size_t)n * key_bytes);
    w.key2 = cv.take((size_t)n * key_bytes);
    w.idx = cv.take((size_t)n * 4);
    w.perm = cv.take((size_t)n * 4);
    w.cub = cv.take(w.cub_bytes);
    return ok;
}

cudaError_t run_curve_sort(const CurveWs& w, char* ws, const float4* pos, int n, cudaStream_t st)
{
    float* bnd = reinterpret_cast<float*>(ws + w.bnd);
    int* idx = reinterpret_cast<int*>(ws + w.idx);
    int* perm = reinterpret_cast<int*>(ws + w.perm);
    const int nb = std::min(CURVE_BND_BLOCKS, (n + 255) / 256);
    trace_launch(2);
    curve_bounds_kernel<<<nb, 256, 0, st>>>(pos, n, bnd);
    if (w.fine)
        curve_keys_kernel<true><<<(n + 255) / 256, 256, 0, st>>>(
            pos, n, bnd, nb, reinterpret_cast<Curve<true>::Key*>(ws + w.key), idx);
    else
        curve_keys_kernel<false><<<(n + 255) / 256, 256, 0, st>>>(
            pos, n, bnd, nb, reinterpret_cast<Curve<false>::Key*>(ws + w.key), idx);
    size_t bytes = w.cub_bytes;
    const cudaError_t e = (w.fine ? curve_sort<true> : curve_sort<false>)(ws + w.cub, bytes, ws + w.key, ws + w.key2,
                                                                         idx, perm, n, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Far tiles: one block per source tile, one thread per source.
// ---------------------------------------------------------------------------
template <bool GRAD>
__global__ void __launch_bounds__(SRC_TILE) far_pack_kernel(const float4* __restrict__ pos,
                                                            const float4* __restrict__ str, int n,
                                                            const float4* __restrict__ box,
                                                            unsigned char* __restrict__ tiles)
{
    using T = FarTile<GRAD>;
    __shared__ __align__(16) unsigned char img[T::BYTES];
    __shared__ float feat[T::NF][SRC_TILE + 1];
    __shared__ float red[2][SRC_TILE / 32];
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, j = k * SRC_TILE + tid;
    const bool valid = j < n;
    const float4 blo = box[2 * k], bhi = box[2 * k + 1];
    const float c[3] = {0.5f * (blo.x + bhi.x), 0.5f * (blo.y + bhi.y), 0.5f * (blo.z + bhi.z)};
    float d[3] = {0.f, 0.f, 0.f}, G[3] = {0.f, 0.f, 0.f};
    if (valid) {
        const float4 p = pos[j], s = str[j];
        d[0] = p.x - c[0], d[1] = p.y - c[1], d[2] = p.z - c[2];
        G[0] = s.x, G[1] = s.y, G[2] = s.z;
    }
    float r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], gm = fmaxf(fabsf(G[0]), fmaxf(fabsf(G[1]), fabsf(G[2])));
    const bool bad = !isfinite(r2) || !isfinite(G[0]) || !isfinite(G[1]) || !isfinite(G[2]) ||
                     !(fmaxf(fabsf(c[0]), fmaxf(fabsf(c[1]), fabsf(c[2]))) < FAR_XMAX);
    const bool any_bad = __syncthreads_or(bad) != 0;
    for (int o = 16; o > 0; o >>= 1) {
        r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
        gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    }
    if (lane == 0) red[0][tid >> 5] = r2, red[1][tid >> 5] = gm;
    __syncthreads();
    for (int w = 0; w < SRC_TILE / 32; ++w) r2 = fmaxf(r2, red[0][w]), gm = fmaxf(gm, red[1][w]);
    const float rad = sqrtf(r2) * 1.000001f;
    // scales: powers of two above the radius and the largest strength component, so that the
    // scaled values are exact (strengths at most 2^FAR_FEXP; eg is kept where both its
    // scale and the inverse are normal numbers)
    int ea = 0, eg = 0;
    frexpf(rad, &ea);
    frexpf(gm, &eg);
    eg = max(eg, FAR_FEXP - 126);
    const bool tiny = !(rad > 1e-30f);
    const float a = tiny || any_bad ? 1.f : ldexpf(1.f, ea);
    const float gam = any_bad ? 1.f : ldexpf(1.f, eg - FAR_FEXP), ig = any_bad ? 1.f : ldexpf(1.f, FAR_FEXP - eg);
    const float ia = 1.f / a;
    const float x = d[0] * ia, y = d[1] * ia, z = d[2] * ia, q = x * x + y * y + z * z;
    const float gx = G[0] * ig, gy = G[1] * ig, gz = G[2] * ig;
    const float mx = gy * z - gz * y, my = gz * x - gx * z, mz = gx * y - gy * x;  // Gamma x d
    float f[T::N];
#pragma unroll
    for (int i = 0; i < T::N; ++i) f[i] = 0.f;
    f[0] = gx, f[1] = gy, f[2] = gz, f[3] = mx, f[4] = my, f[5] = mz;
    if constexpr (GRAD) {
        f[6] = q * gx, f[7] = q * gy, f[8] = q * gz;
        f[9] = q * mx, f[10] = q * my, f[11] = q * mz;
        f[12] = gx * x, f[13] = gx * y, f[14] = gx * z;
        f[15] = gy * x, f[16] = gy * y, f[17] = gy * z;
        f[18] = gz * x, f[19] = gz * y, f[20] = gz * z;
        f[21] = mx * x, f[22] = mx * y, f[23] = mx * z;
        f[24] = my * x, f[25] = my * y, f[26] = my * z;
        f[27] = mz * x, f[28] = mz * y;
    }
#pragma unroll
    for (int i = 0; i < T::N; ++i) {
        const __half h = __float2half_rn(f[i]);
        const __half l = __float2half_rn(f[i] - __half2float(h));
        const int at = ((tid >> 3) * (T::N / 8) + (i >> 3)) * 128 + (i & 7) * 16 + (tid & 7) * 2;
        *reinterpret_cast<__half*>(img + at) = h;
        *reinterpret_cast<__half*>(img + T::FEAT + at) = l;
        if (i < T::NF) feat[i][tid] = f[i];
    }
    float* sd = reinterpret_cast<float*>(img + T::OFF_D) + (tid >> 1) * 8 + (tid & 1);
    sd[0] = x, sd[2] = y, sd[4] = z, sd[6] = q;
    __syncthreads();
    float* hdr = reinterpret_cast<float*>(img + T::OFF_H);
    {  // feature sums (they carry almost all of the result) in double-float, four threads each
        const int i = tid >> 2, s = tid & 3;
        float v = 0.f, w = 0.f;
        if (i < T::NF)
            for (int p = s; p < SRC_TILE; p += 4) {
                float e;
                two_sum(v, feat[i][p], v, e);
                w += e;
            }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const float v2 = __shfl_xor_sync(0xffffffffu, v, o), w2 = __shfl_xor_sync(0xffffffffu, w, o);
            float e;
            two_sum(fminf(v, v2), fmaxf(v, v2), v, e);  // the same order in both threads
            w = (w + w2) + e;
        }
        if (s == 0 && i < T::N) hdr[i] = v + w;
    }
    if (tid < 8) {
        const float v[8] = {c[0], c[1], c[2], a, gam, any_bad ? INFINITY : rad, 0.f, 0.f};
        hdr[T::N + tid] = v[tid];
    }
    for (int i = T::N + 8 + tid; i < 64; i += SRC_TILE) hdr[i] = 0.f;
    __syncthreads();
    uint4* o = reinterpret_cast<uint4*>(tiles + (size_t)k * T::BYTES);
    for (int i = tid; i < T::BYTES / 16; i += SRC_TILE) o[i] = reinterpret_cast<const uint4*>(img)[i];
}

cudaError_t run_far_pack(const float4* pos, const float4* str, int n, const float4* box, int SP, bool grad,
                         unsigned char* tiles, cudaStream_t st)
{
    trace_launch();
    if (grad)
        far_pack_kernel<true><<<SP, SRC_TILE, 0, st>>>(pos, str, n, box, tiles);
    else
        far_pack_kernel<false><<<SP, SRC_TILE, 0, st>>>(pos, str, n, box, tiles);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Unit lists.  far_mask_kernel: for each (target tile, source tile) the groups that are
// far, and the counts of listed units per chunk; far_scan_kernel: their exclusive scans;
// far_emit_kernel: the lists, in order.
// ---------------------------------------------------------------------------
constexpr int LIST_TPB = SWEEP_TPB;

// A unit's mask word: bit g set where group g is far; from bit 8, six bits for each
// group's cost in the pair sweep.
__device__ __forceinline__ int near_cost(unsigned m, int g) { return (m >> (8 + 6 * g)) & 63u; }

// A unit's cost in the tensor-core sweep: a lone warpgroup runs at less than half the rate
// of four, so the first group costs as much as the other three.
__device__ __forceinline__ int far_cost(unsigned m)
{
    const int c = __popc(m & FAR_ALL);
    return c ? FAR_COST_FIRST + c - 1 : 0;
}

// cnt[0 .. TT KY): (units, cost) of the tensor-core list by (target tile, chunk); then the
// pair sweep's by (target tile, group, chunk).
template <bool GRAD>
__global__ void __launch_bounds__(LIST_TPB) far_mask_kernel(const float4* __restrict__ tgt, int n_tgt,
                                                            const unsigned char* __restrict__ tiles, int SP,
                                                            float far2, const float4* __restrict__ pbox,
                                                            unsigned* __restrict__ mask, uint2* __restrict__ cnt)
{
    constexpr int GW = SWEEP_CW / FAR_GROUPS;  // warps per group
    __shared__ float wbox[SWEEP_CW][12];
    __shared__ int tot[1 + FAR_GROUPS][2];
    __shared__ int beyond[SWEEP_CW];  // a target of the warp lies beyond FAR_XMAX (or is not finite)
    const int t = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < 2 * (1 + FAR_GROUPS)) (&tot[0][0])[threadIdx.x] = 0;
    const int i0 = t * TGT_TILE + warp * 64 + lane, i1 = i0 + 32;
    float4 p0 = make_float4(0.f, 0.f, 0.f, 0.f), p1 = p0;
    const bool v0 = i0 < n_tgt, v1 = i1 < n_tgt;
    if (v0) p0 = tgt[i0];
    if (v1) p1 = tgt[i1];
    warp_two_boxes(make_float3(p0.x, p0.y, p0.z), v0, make_float3(p1.x, p1.y, p1.z), v1, wbox[warp]);
    auto inside = [](float4 p) { return fabsf(p.x) < FAR_XMAX && fabsf(p.y) < FAR_XMAX && fabsf(p.z) < FAR_XMAX; };
    const bool all_in = __all_sync(0xffffffffu, inside(p0) && inside(p1));  // (a lane without a target holds zeros)
    if (lane == 0) beyond[warp] = !all_in;
    __syncthreads();
    const int k0 = blockIdx.y * FAR_KCH, k1 = min(SP, k0 + FAR_KCH);
    int v[1 + FAR_GROUPS][2] = {};
    for (int k = k0 + threadIdx.x; k < k1; k += LIST_TPB) {
        const float4* h = reinterpret_cast<const float4*>(tiles + (size_t)k * FarTile<GRAD>::BYTES +
                                                          FarTile<GRAD>::OFF_H + FarTile<GRAD>::N * 4);
        const float4 c = h[0];  // centre, scale
        const float rad = h[1].y;  // radius; +inf for a tile with a non-finite source or beyond FAR_XMAX
        const float sep = rad + sqrtf(far2) * 1.0001f;
        const float need = fmaxf(rad * (1.f / FAR_TAU), sep), need2 = need * need;
        const float4 tlo = pbox[2 * k], thi = pbox[2 * k + 1];
        unsigned m = 0;
#pragma unroll
        for (int g = 0; g < FAR_GROUPS; ++g) {
            bool far = true;
#pragma unroll
            for (int w = g * GW; w < (g + 1) * GW; ++w) far = far && !beyond[w];
#pragma unroll 1
            for (int w = g * GW; w < (g + 1) * GW; ++w)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const float* lo = &wbox[w][6 * q];
                    const float dx = fmaxf(0.f, fmaxf(c.x - lo[3], lo[0] - c.x));
                    const float dy = fmaxf(0.f, fmaxf(c.y - lo[4], lo[1] - c.y));
                    const float dz = fmaxf(0.f, fmaxf(c.z - lo[5], lo[2] - c.z));
                    far = far && dx * dx + dy * dy + dz * dz > need2;
                }
            int cn = 0;
            const int warps = group_warps(n_tgt - (t * TGT_TILE + g * FAR_GROUP));
            if (warps == 0)
                ;  // no target: in neither list
            else if (far)
                m |= 1u << g;
            else {
#pragma unroll 1
                for (int w = g * GW; w < g * GW + warps; ++w) cn += boxes_near(wbox[w], tlo, thi, far2) ? NEAR_COST : 1;
                cn = ragged_cost(cn, warps);
            }
            m |= (unsigned)cn << (8 + 6 * g);
            v[1 + g][0] += cn != 0, v[1 + g][1] += cn;
        }
        mask[(size_t)t * SP + k] = m;
        const int c1 = far_cost(m);
        v[0][0] += c1 != 0, v[0][1] += c1;
    }
#pragma unroll
    for (int q = 0; q < 1 + FAR_GROUPS; ++q)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int x = __reduce_add_sync(0xffffffffu, v[q][e]);
            if (lane == 0) atomicAdd(&tot[q][e], x);
        }
    __syncthreads();
    const int KY = gridDim.y;
    if (threadIdx.x == 0) cnt[(size_t)t * KY + blockIdx.y] = make_uint2(tot[0][0], tot[0][1]);
    if (threadIdx.x < FAR_GROUPS)
        cnt[(size_t)gridDim.x * KY + ((size_t)t * FAR_GROUPS + threadIdx.x) * KY + blockIdx.y] =
            make_uint2(tot[1 + threadIdx.x][0], tot[1 + threadIdx.x][1]);
}

// Exclusive scans of the two count arrays, one per block.
__global__ void __launch_bounds__(1024) far_scan_kernel(const uint2* __restrict__ cnt, int m, uint2* __restrict__ off_f,
                                                        uint2* __restrict__ off_n)
{
    __shared__ uint2 ws[32];
    const bool second = blockIdx.x != 0;
    const uint2* c = second ? cnt + m : cnt;
    uint2* off = second ? off_n : off_f;
    const int len = second ? m * FAR_GROUPS : m;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto scan = [lane](uint2 x) {
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y0 = __shfl_up_sync(0xffffffffu, x.x, o), y1 = __shfl_up_sync(0xffffffffu, x.y, o);
            if (lane >= o) x.x += y0, x.y += y1;
        }
        return x;
    };
    uint2 base = make_uint2(0, 0);
    for (int s = 0; s < len; s += 1024) {
        const int i = s + threadIdx.x;
        const uint2 own = i < len ? c[i] : make_uint2(0, 0);
        const uint2 x = scan(own);
        if (lane == 31) ws[warp] = x;
        __syncthreads();
        if (warp == 0) ws[lane] = scan(ws[lane]);
        __syncthreads();
        const uint2 before = warp ? ws[warp - 1] : make_uint2(0, 0);
        if (i < len) off[i] = make_uint2(base.x + before.x + x.x - own.x, base.y + before.y + x.y - own.y);
        base.x += ws[31].x, base.y += ws[31].y;
        __syncthreads();
    }
    if (threadIdx.x == 0) off[len] = base;
}

// blockIdx.z = 0: the tensor-core list of a (target tile, chunk); 1 + g: the pair sweep's of group g.
__global__ void __launch_bounds__(LIST_TPB) far_emit_kernel(const unsigned* __restrict__ mask, int SP,
                                                            const uint2* __restrict__ off_f,
                                                            const uint2* __restrict__ off_n,
                                                            uint2* __restrict__ list_f, uint2* __restrict__ list_n)
{
    constexpr int NW = LIST_TPB / 32;
    __shared__ uint2 ws[NW];
    const int t = blockIdx.x, g = (int)blockIdx.z - 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k0 = blockIdx.y * FAR_KCH, k1 = min(SP, k0 + FAR_KCH);
    uint2 base = g < 0 ? off_f[t * gridDim.y + blockIdx.y] : off_n[(t * FAR_GROUPS + g) * gridDim.y + blockIdx.y];
    uint2* list = g < 0 ? list_f : list_n;
    const unsigned lt = (1u << lane) - 1u;
    for (int ks = k0; ks < k1; ks += LIST_TPB) {
        const int k = ks + threadIdx.x;
        const unsigned m = k < k1 ? mask[(size_t)t * SP + k] : 0u;
        const int c = g < 0 ? far_cost(m) : near_cost(m, g);
        const bool in = c != 0;
        const unsigned q = __ballot_sync(0xffffffffu, in);
        int s = c;  // costs up to this lane
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane == 31) ws[warp] = make_uint2(__popc(q), s);
        __syncthreads();
        uint2 p = base;
        for (int w = 0; w < NW; ++w) {
            const uint2 x = ws[w];
            if (w < warp) p.x += x.x, p.y += x.y;
            base.x += x.x, base.y += x.y;
        }
        if (in)
            list[p.x + __popc(q & lt)] =
                make_uint2(g < 0 ? ((unsigned)k << 4) | (m & FAR_ALL) : (unsigned)k, (unsigned)(p.y + s - c));
        __syncthreads();
    }
}

cudaError_t run_far_lists(const float4* tgt, int n_tgt, const unsigned char* tiles, int SP, int TT, bool grad,
                          const float4* pbox, float far2, unsigned* mask, uint2* cnt, uint2* near_list,
                          uint2* near_off, uint2* far_list, uint2* far_off, cudaStream_t st)
{
    const int KY = (SP + FAR_KCH - 1) / FAR_KCH;
    const dim3 grid(TT, KY), grid_emit(TT, KY, 1 + FAR_GROUPS);
    trace_launch(3);
    if (grad)
        far_mask_kernel<true><<<grid, LIST_TPB, 0, st>>>(tgt, n_tgt, tiles, SP, far2, pbox, mask, cnt);
    else
        far_mask_kernel<false><<<grid, LIST_TPB, 0, st>>>(tgt, n_tgt, tiles, SP, far2, pbox, mask, cnt);
    far_scan_kernel<<<2, 1024, 0, st>>>(cnt, TT * KY, far_off, near_off);
    far_emit_kernel<<<grid_emit, LIST_TPB, 0, st>>>(mask, SP, far_off, near_off, far_list, near_list);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The far sweep: four warpgroups per block, each holding 256 targets (two per thread, in
// the rows of two 128-row accumulators) of a 1,024-target tile.
// ---------------------------------------------------------------------------
constexpr int FAR_STAGES = 5;
constexpr uint64_t FAR_WAIT = 2000000000ull;
constexpr int FAR_CH = 32;        // sources per chunk: two K steps of the FP16 MMA
constexpr int FAR_COLS = 64;      // TMEM columns of a 128-row tile: 32 accumulators, 32 operand columns
constexpr int FAR_TMEM = 512;

template <bool GRAD, bool COMP>
__host__ __device__ constexpr size_t far_smem_bytes()
{
    return (size_t)FAR_STAGES * FarTile<GRAD>::BYTES + (size_t)(GRAD ? 14 : 3) * (COMP ? 2 : 1) * SWEEP_TPB * 8;
}

// Counts a warp in; true for the last of a group's four.  Orders the group's earlier
// operand stores before what the last one does next.
__device__ __forceinline__ bool arrive_last(unsigned* c)
{
    unsigned v;
    asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(v) : "r"(smem_u32(c)) : "memory");
    return (v & 3u) == 3u;
}

template <bool GRAD, bool COMP>
__global__ void __launch_bounds__(SWEEP_TPB, 1) far_sweep_kernel(const FarArgs A)
{
    using T = FarTile<GRAD>;
    extern __shared__ __align__(1024) unsigned char fsm[];
    __shared__ __align__(8) uint64_t full[FAR_STAGES];
    __shared__ __align__(8) uint64_t mdone[FAR_GROUPS];
    __shared__ unsigned ready[FAR_GROUPS];  // warps that have stored their rows of a chunk
    __shared__ int released[FAR_STAGES];
    __shared__ int issued_round[FAR_STAGES];
    __shared__ uint32_t tm_base_s;
    constexpr int NR = GRAD ? 14 : 3;
    constexpr int NT = SWEEP_TPB;
    // running sums [row][thread]: (hi, lo) of the two targets, or their plain sums
    using Run = typename std::conditional<COMP, float4, float2>::type;
    Run* run = reinterpret_cast<Run*>(fsm + (size_t)FAR_STAGES * T::BYTES);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = warp >> 2, quad = warp & 3;
    const UnitList& ul = A.ul;
    const int b = blockIdx.x;
    __shared__ int range_s[3];
    if (warp == 0) {
        int l, h, t;
        ul.range(b, l, h, t);
        if (lane == 0) range_s[0] = l, range_s[1] = h, range_s[2] = t;
    }
    __syncthreads();
    const int lo = range_s[0], hi = range_s[1];
    if (lo >= hi) return;  // uniform

    auto issue = [&](int i, int s, int round) {
        issued_round[s] = round;
        fence_proxy_async_smem();
        mbar_expect_tx(&full[s], T::BYTES);
        bulk_g2s(fsm + (size_t)s * T::BYTES, A.tiles + (size_t)(ul.list[i].x >> 4) * T::BYTES, T::BYTES, &full[s]);
    };
    if (warp == 0) {
        tm_alloc(&tm_base_s, FAR_TMEM);
        tm_relinquish();
    }
    if (tid == 0) {
        for (int s = 0; s < FAR_STAGES; ++s) {
            mbar_init(&full[s], 1);
            released[s] = 0;
            issued_round[s] = -1;
        }
        for (int q = 0; q < FAR_GROUPS; ++q) {
            mbar_init(&mdone[q], 1);
            ready[q] = 0;
        }
        mbar_fence_init();
        for (int s = 0; s < FAR_STAGES && lo + s < hi; ++s) issue(lo + s, s, 0);
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tm = __shfl_sync(0xffffffffu, tm_base_s, 0);
    const uint32_t tm_row = tm + ((uint32_t)(quad * 32) << 16);
    const uint32_t col0 = (uint32_t)g * 2 * FAR_COLS, col1 = col0 + FAR_COLS;
    constexpr uint32_t IDESC = idesc_f16(128, T::N);

    auto zero_run = [&]() {
#pragma unroll
        for (int q = 0; q < NR; ++q) run[q * NT + tid] = Run{};
    };
    zero_run();

    f2 X = zero2(), Y = zero2(), Z = zero2();
    int t = range_s[2], t_end = ul.end(t), cur_t = -1;
    unsigned entry = ul.list[lo].x;
    unsigned uses = 0;  // chunks this group has handed to the tensor core so far
    const f2 one = splat(1.f), none = splat(-1.f);
    bool ok = true;
    for (int i = lo;; ++i) {
        const int s = (i - lo) % FAR_STAGES, r = (i - lo) / FAR_STAGES;
        const bool has_next = i + 1 < hi;
        const unsigned next = has_next ? ul.list[i + 1].x : 0u;
        if (t != cur_t) {
            cur_t = t;
            const int i0 = t * TGT_TILE + g * FAR_GROUP + quad * 32 + lane, i1 = i0 + 128;
            const float4 p0 = A.tgt[min(i0, A.n_tgt - 1)], p1 = A.tgt[min(i1, A.n_tgt - 1)];
            X = make_float2(p0.x, p1.x);
            Y = make_float2(p0.y, p1.y);
            Z = make_float2(p0.z, p1.z);
        }
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[s], r & 1, A.dev_err, FAR_WAIT))) {
            ok = false;
            break;
        }
        if ((entry >> g) & 1u) {
            const unsigned char* st = fsm + (size_t)s * T::BYTES;
            const float* hdr = reinterpret_cast<const float*>(st + T::OFF_H);
            const float4* sd = reinterpret_cast<const float4*>(st + T::OFF_D);
            // y = x - c, s = 1/|y|, e = a s; the weights' coefficients -2 e n, e^2 of the two rows
            f2 sv;
            f2 kx0, ky0, kz0, e20, kx1, ky1, kz1, e21;
            {
                const f2 yx = add2(X, splat(-hdr[T::N])), yy = add2(Y, splat(-hdr[T::N + 1])),
                         yz = add2(Z, splat(-hdr[T::N + 2]));
                const f2 w2 = fma2(yz, yz, fma2(yy, yy, mul2(yx, yx)));
                sv = rsqrt2_approx(w2);
                // one Newton step: the scale is shared by the tile's 128 pairs
                sv = fma2(mul2(fma2(mul2(w2, none), mul2(sv, sv), one), splat(0.5f)), sv, sv);
                const f2 ev = mul2(sv, splat(hdr[T::N + 3])), e2 = mul2(ev, ev);
                const f2 m2 = mul2(mul2(ev, sv), splat(-2.f));
                const f2 kx = mul2(yx, m2), ky = mul2(yy, m2), kz = mul2(yz, m2);
                kx0 = splat(kx.x), ky0 = splat(ky.x), kz0 = splat(kz.x), e20 = splat(e2.x);
                kx1 = splat(kx.y), ky1 = splat(ky.y), kz1 = splat(kz.y), e21 = splat(e2.y);
            }
            const uint64_t dh0 = smem_desc(smem_u32(st), T::N * 16, 128);
#pragma unroll 1
            for (int c = 0; c < SRC_TILE / FAR_CH; ++c) {
#pragma unroll 4
                for (int e = 0; e < 4; ++e) {  // 8 sources
                    const float4* sq = sd + (4 * c + e) * 8;
                    uint32_t h0[4], l0[4], h1[4], l1[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 a = sq[2 * q], d = sq[2 * q + 1];
                        const f2 dx = make_float2(a.x, a.y), dy = make_float2(a.z, a.w), dz = make_float2(d.x, d.y),
                                 qq = make_float2(d.z, d.w);
                        far_weight<GRAD>(fma2(kx0, dx, fma2(ky0, dy, fma2(kz0, dz, fma2(e20, qq, one)))), h0[q], l0[q]);
                        far_weight<GRAD>(fma2(kx1, dx, fma2(ky1, dy, fma2(kz1, dz, fma2(e21, qq, one)))), h1[q], l1[q]);
                    }
                    if (e == 0) {  // the operand buffer is free once the previous chunk is multiplied
                        if (uses > 0)
                            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&mdone[g], (uses - 1) & 1, A.dev_err, FAR_WAIT)) && ok;
                    }
                    const uint32_t buf = 32 + 16 * (e >> 1) + 4 * (e & 1);
                    tm_st4(tm_row + col0 + buf, h0);
                    tm_st4(tm_row + col0 + buf + 8, l0);
                    tm_st4(tm_row + col1 + buf, h1);
                    tm_st4(tm_row + col1 + buf + 8, l1);
                }
                tm_wait_st();
                tm_fence_before();
                // the last of the group's warps to have stored its rows issues the products;
                // the others go on at once
                int last = 0;
                if (lane == 0) last = arrive_last(&ready[g]);
                if (__shfl_sync(0xffffffffu, last, 0)) {
                    __syncwarp();
                    tm_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            // K step: two core-matrix columns of N/8 core matrices each
                            const uint64_t dh = dh0 + (uint64_t)((2 * c + hf) * (2 * T::N * 16 >> 4));
                            const uint64_t dl = dh + (uint64_t)(T::FEAT >> 4);
#pragma unroll
                            for (int row = 0; row < 2; ++row) {
                                const uint32_t cd = tm + (row ? col1 : col0), ca = cd + 32 + 16 * hf;
                                tm_mma_f16(cd, ca, dh, IDESC, c + hf > 0);
                                tm_mma_f16(cd, ca, dl, IDESC, 1);
                                tm_mma_f16(cd, ca + 8, dh, IDESC | IDESC_NEG_A, 1);
                            }
                        }
                        tm_commit(&mdone[g]);
                    }
                    __syncwarp();
                }
                ++uses;
            }
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(&mdone[g], (uses - 1) & 1, A.dev_err, FAR_WAIT)) && ok;
            if (!ok) break;
            tm_fence_after();
            // the tile's sums of the group's targets
            f2 o[NR];
            // n, e again rather than held in registers through the loop
            const volatile float* vh = hdr + T::N;
            const f2 nx = mul2(add2(X, splat(-vh[0])), sv), ny = mul2(add2(Y, splat(-vh[1])), sv),
                     nz = mul2(add2(Z, splat(-vh[2])), sv);
            const f2 ev = mul2(sv, splat(vh[3]));
            if constexpr (GRAD) {
                const f2 kx = make_float2(kx0.x, kx1.x), ky = make_float2(ky0.x, ky1.x), kz = make_float2(kz0.x, kz1.x),
                         e2 = make_float2(e20.x, e21.x);
                // columns: 0-2 V, 3-5 M, 6-8 V2, 9-11 M2, 12-20 W (12 + 3 c + b), 21-28 Q
                f2 m[32];
                float d0[32], d1[32];
#pragma unroll
                for (int q = 0; q < 32; q += 8) {
                    tm_ld8(tm_row + col0 + q, d0 + q);
                    tm_ld8(tm_row + col1 + q, d1 + q);
                }
                tm_wait_ld();
#pragma unroll
                for (int q = 0; q < 32; q += 4) {
                    const float4 h = *reinterpret_cast<const float4*>(hdr + q);
                    m[q] = make_float2(d0[q] + h.x, d1[q] + h.x);
                    m[q + 1] = make_float2(d0[q + 1] + h.y, d1[q + 1] + h.y);
                    m[q + 2] = make_float2(d0[q + 2] + h.z, d1[q + 2] + h.z);
                    m[q + 3] = make_float2(d0[q + 3] + h.w, d1[q + 3] + h.w);
                }
                const f2 ne = mul2(ev, none);
                // S = V - 2e W n + e^2 V2
                f2 S[3], P[3], Bv[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    S[c] = fma2(e2, m[6 + c], m[c]);
                    S[c] = fma2(kx, m[12 + 3 * c], fma2(ky, m[13 + 3 * c], fma2(kz, m[14 + 3 * c], S[c])));
                }
                const f2 Qzz = mul2(add2(m[21], m[25]), none);
                const f2 Q[9] = {m[21], m[22], m[23], m[24], m[25], m[26], m[27], m[28], Qzz};
                // P = e (M - 2e Q n + e^2 M2)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    P[c] = fma2(e2, m[9 + c], m[3 + c]);
                    P[c] = fma2(kx, Q[3 * c], fma2(ky, Q[3 * c + 1], fma2(kz, Q[3 * c + 2], P[c])));
                }
                const f2 mnx = mul2(nx, none), mny = mul2(ny, none), mnz = mul2(nz, none);
                // u = S x n - P,  B = V x n - e M
                o[0] = fma2(ne, P[0], fma2(S[1], nz, mul2(S[2], mny)));
                o[1] = fma2(ne, P[1], fma2(S[2], nx, mul2(S[0], mnz)));
                o[2] = fma2(ne, P[2], fma2(S[0], ny, mul2(S[1], mnx)));
                Bv[0] = fma2(ne, m[3], fma2(m[1], nz, mul2(m[2], mny)));
                Bv[1] = fma2(ne, m[4], fma2(m[2], nx, mul2(m[0], mnz)));
                Bv[2] = fma2(ne, m[5], fma2(m[0], ny, mul2(m[1], mnx)));
                o[3] = S[0], o[4] = S[1], o[5] = S[2];
                // G_ab = B_a n_b - (W_.b x e n)_a + e^2 Q_ab
                const f2 ex = mul2(nx, ev), ey = mul2(ny, ev), ez = mul2(nz, ev);
                const f2 mex = mul2(ex, none), mey = mul2(ey, none), mez = mul2(ez, none);
#pragma unroll
                for (int bb = 0; bb < 3; ++bb) {
                    const f2 nb = bb == 0 ? nx : (bb == 1 ? ny : nz);
                    const f2 W0 = m[12 + bb], W1 = m[15 + bb], W2 = m[18 + bb];
                    o[6 + bb] = fma2(Bv[0], nb, fma2(W1, mez, fma2(W2, ey, mul2(e2, Q[bb]))));
                    o[9 + bb] = fma2(Bv[1], nb, fma2(W2, mex, fma2(W0, ez, mul2(e2, Q[3 + bb]))));
                    if (bb < 2) o[12 + bb] = fma2(Bv[2], nb, fma2(W0, mey, fma2(W1, ex, mul2(e2, Q[6 + bb]))));
                }
                const f2 fu = mul2(mul2(sv, sv), splat(hdr[T::N + 4])), fg = mul2(fu, sv);
#pragma unroll
                for (int q = 0; q < 3; ++q) o[q] = mul2(o[q], fu);
#pragma unroll
                for (int q = 3; q < NR; ++q) o[q] = mul2(o[q], fg);
            } else {
                // columns: 0-2 V, 3-5 M (weights t^(-3/2));  u = V x n - e M
                float d0[8], d1[8];
                tm_ld8(tm_row + col0, d0);
                tm_ld8(tm_row + col1, d1);
                tm_wait_ld();
                f2 m[6];
#pragma unroll
                for (int p = 0; p < 6; ++p) m[p] = make_float2(d0[p] + hdr[p], d1[p] + hdr[p]);
                const f2 ne = mul2(ev, none);
                const f2 mnx = mul2(nx, none), mny = mul2(ny, none), mnz = mul2(nz, none);
                const f2 fu = mul2(mul2(sv, sv), splat(hdr[T::N + 4]));
                o[0] = mul2(fu, fma2(ne, m[3], fma2(m[1], nz, mul2(m[2], mny))));
                o[1] = mul2(fu, fma2(ne, m[4], fma2(m[2], nx, mul2(m[0], mnz))));
                o[2] = mul2(fu, fma2(ne, m[5], fma2(m[0], ny, mul2(m[1], mnx))));
            }
            tm_fence_before();  // the next tile's MMAs overwrite the accumulators after the next barrier
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                if constexpr (COMP) {
                    const float4 v = run[q * NT + tid];
                    f2 h = make_float2(v.x, v.y), l = make_float2(v.z, v.w);
                    fold2(h, l, o[q]);
                    run[q * NT + tid] = make_float4(h.x, h.y, l.x, l.y);
                } else {
                    run[q * NT + tid] = add2(run[q * NT + tid], o[q]);
                }
            }
        }
        __syncwarp();
        if (lane == 0) {  // the last warp to leave stage s refills it
            __threadfence_block();
            if (atomicAdd(&released[s], 1) == SWEEP_CW - 1) {
                released[s] = 0;
                __threadfence_block();
                if (i + FAR_STAGES < hi) issue(i + FAR_STAGES, s, r + 1);
            }
        }
        if (!has_next || i + 1 >= t_end) {
            float* P = A.part + ((size_t)(b + t) * (COMP ? 2 * NR : NR)) * TGT_TILE + g * FAR_GROUP + quad * 32 + lane;
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const Run v = run[q * NT + tid];
                P[(size_t)q * TGT_TILE] = v.x;
                P[(size_t)q * TGT_TILE + 128] = v.y;
                if constexpr (COMP) {
                    P[(size_t)(NR + q) * TGT_TILE] = v.z;
                    P[(size_t)(NR + q) * TGT_TILE + 128] = v.w;
                }
            }
            zero_run();
        }
        if (!has_next) break;
        while (i + 1 >= t_end) t_end = ul.end(++t);
        entry = next;
    }
    if (!ok && lane == 0)  // let the copies in flight land before the shared memory is released
        for (int q = 0; q < FAR_STAGES; ++q)
            if (issued_round[q] >= 0) mbar_wait_bounded(&full[q], issued_round[q] & 1, A.dev_err, FAR_WAIT);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (warp == 0) tm_dealloc(tm, FAR_TMEM);
}

namespace {
std::mutex g_far_mu;
bool g_far_ready[64][4];
}  // namespace

template <bool G, bool C>
static cudaError_t launch_far(const FarArgs& A, cudaStream_t st)
{
    int d = 0;
    cudaGetDevice(&d);
    constexpr int v = (G ? 2 : 0) + (C ? 1 : 0);
    {
        std::lock_guard<std::mutex> lk(g_far_mu);
        if (d < 0 || d >= 64 || !g_far_ready[d][v]) {
            const cudaError_t e = cudaFuncSetAttribute(far_sweep_kernel<G, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)far_smem_bytes<G, C>());
            if (e != cudaSuccess) return e;
            if (d >= 0 && d < 64) g_far_ready[d][v] = true;
        }
    }
    far_sweep_kernel<G, C><<<A.ul.B, SWEEP_TPB, far_smem_bytes<G, C>(), st>>>(A);
    return cudaGetLastError();
}

cudaError_t run_far_sweep(const FarArgs& A, bool grad, bool comp, cudaStream_t st)
{
    if (grad) return comp ? launch_far<true, true>(A, st) : launch_far<true, false>(A, st);
    return comp ? launch_far<false, true>(A, st) : launch_far<false, false>(A, st);
}

}  // namespace vpm
