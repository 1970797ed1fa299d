// twk_prep.cu -- O(N d) preparation for the audit (TwinKV, arXiv 2608.27128), one pass over
// the keys, bound by memory:
//   * float32 keys -> bf16 (round to nearest even),
//   * per key k . k and 1/||k|| (the l2 normalisation of Sec. 3.2 Eq. 1, applied later
//     as a scale; a zero key gets 0, so it has similarity 0 with every key),
//   * the retained-first column layout used by the repair audit: retained keys in
//     position order, padded to a 256-column tile, then evicted keys in position order,
//     with per-column 1/||k|| (NaN on padding columns, which the audit then ignores)
//     and per-column original position.
#include <algorithm>

#include <cuda_bf16.h>

#include "twk_df.cuh"
#include "twk_internal.h"
#include "twk_ptx.cuh"

namespace twk {
namespace {

__device__ __forceinline__ float nan_f() { return __uint_as_float(0x7FFFFFFFu); }

constexpr int kPrepThreads = 256;
constexpr int kKeysPerStep = kPrepThreads / kParts;
// Keys per lane group: 64 bytes of loads per thread are in flight, and the block's reduction
// and atomic serve them all (twice as many keys, or blocks of 128 threads, measured within
// 3 % either way).
template <int D>
constexpr int kKeys = 128 / D;
template <int D>
constexpr int kKeysPerBlock = kKeysPerStep * kKeys<D>;   // NP is a multiple of this
// prep_unit_kernel: CTAs per unit, threads, a CTA's slots (one per lane group), and the
// largest N whose column stride they cover.
constexpr int kUnitCtas = 8;
constexpr int kUnitThreads = 1024;
constexpr int kUnitSlots = kUnitThreads / kParts;
constexpr int kUnitMaxN = kUnitCtas * kUnitSlots - kBN;

// A lane's 16-byte chunks part, part + kParts, ... of a key's bf16 row, from bf16 keys or
// from float32 ones rounded to nearest even (8 floats per chunk).
template <int D>
__device__ __forceinline__ void load_key(const uint16_t* __restrict__ keys, int64_t row, int part,
                                         uint4 (&v)[D / 8 / kParts])
{
    const uint4* src = reinterpret_cast<const uint4*>(keys + row * D) + part;
#pragma unroll
    for (int q = 0; q < D / 8 / kParts; ++q) v[q] = __ldg(src + q * kParts);
}

__device__ __forceinline__ uint32_t round2(float a, float b)
{
    return static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(a))) |
           static_cast<uint32_t>(__bfloat16_as_ushort(__float2bfloat16_rn(b))) << 16;
}

template <int D>
__device__ __forceinline__ void load_key(const float* __restrict__ keys, int64_t row, int part,
                                         uint4 (&v)[D / 8 / kParts])
{
    const float4* src = reinterpret_cast<const float4*>(keys + row * D) + 2 * part;
#pragma unroll
    for (int q = 0; q < D / 8 / kParts; ++q) {
        const float4 f = __ldg(src + 2 * q * kParts), g = __ldg(src + 2 * q * kParts + 1);
        v[q] = make_uint4(round2(f.x, f.y), round2(f.z, f.w), round2(g.x, g.y), round2(g.z, g.w));
    }
}

template <int D>
__device__ __forceinline__ void store_key(uint16_t* out, int64_t row, int part,
                                          const uint4 (&v)[D / 8 / kParts])
{
    uint4* dst = reinterpret_cast<uint4*>(out + row * D) + part;
#pragma unroll
    for (int q = 0; q < D / 8 / kParts; ++q) dst[q * kParts] = v[q];
}

// The norm record of one key, computed by its kParts-lane group: k.k and 1/||k|| as
// double-floats (for the exact similarity values) and 1/||k|| in fp32 (for the audit).
template <int Q>
__device__ __forceinline__ float4 key_norms(const uint4 (&v)[Q], float& rinv32)
{
    const DF sq = group_square_df(v);
    const DF rn = sq.h > 0.f ? df_rsqrt(sq) : DF{0.f, 0.f};
    rinv32 = rn.h;
    return make_float4(sq.h, sq.l, rn.h, rn.l);
}

// The largest k.k of unit u so far, as float bits (k.k >= 0, so the unsigned order of
// the bits is the float order): one atomic per block (hundreds of blocks share a unit's
// word, so per-warp atomics queue up).  Every thread of the block calls it; lanes pass
// 0 for nothing.
__device__ __forceinline__ void unit_max_kk(unsigned* unit_kk, int64_t u, float kk)
{
    __shared__ unsigned wmax[kPrepThreads / 32];
    const unsigned m = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(kk));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t = 0u;
#pragma unroll
        for (int w = 0; w < kPrepThreads / 32; ++w) t = max(t, wmax[w]);
        if (t != 0u) atomicMax(unit_kk + u, t);
    }
}

// Mode 0 (keys as given): per column p of unit blockIdx.y, colrinv = rscale/||k_p||
// (rscale a power of two, so the scaling is exact) and colpos = p, NaN / -1 on the
// padding columns [N, NP); norms[u][p] = the norm record; unit_kk[u] (if given) =
// the unit's largest k.k.  float32 keys also leave their rounded rows in keys16: one pass
// over them, where a separate rounding pass wrote the bf16 keys for this one to read back
// (16 units of 5003 x 128: 50 -> 18 us with the launches).  Grid (NP / kKeysPerBlock<D>, U),
// kParts lanes per column.
template <int D, typename Key>
__global__ void __launch_bounds__(kPrepThreads)
    norms_identity_kernel(const Key* __restrict__ keys, int N, int64_t NP,
                          float* __restrict__ colrinv, int* __restrict__ colpos,
                          float4* __restrict__ norms, float rscale, unsigned* unit_kk,
                          uint16_t* __restrict__ keys16)
{
    wait_for_previous();
    constexpr int Q = D / 8 / kParts, K = kKeys<D>;
    const int part = threadIdx.x % kParts;
    const int p0 = blockIdx.x * kKeysPerBlock<D> + threadIdx.x / kParts;
    const int64_t u = blockIdx.y;
    uint4 v[K][Q];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        // every lane takes part in the shuffles of the norms: padding columns use key 0
        const int p = p0 + k * kKeysPerStep;
        load_key<D>(keys, u * N + (p < N ? p : 0), part, v[k]);
    }
    float top = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = p0 + k * kKeysPerStep;
        if constexpr (sizeof(Key) == 4)
            if (p < N) store_key<D>(keys16, u * N + p, part, v[k]);
        float r32;
        const float4 nr = key_norms(v[k], r32);
        if (part == 0) {
            colrinv[u * NP + p] = p < N ? r32 * rscale : nan_f();
            colpos[u * NP + p] = p < N ? p : -1;
            if (p < N) {
                norms[u * N + p] = nr;
                top = fmaxf(top, nr.x);
            }
        }
    }
    if (unit_kk) unit_max_kk(unit_kk, u, top);
}

constexpr int kScanBytes = 16;   // mask bytes per thread and step

// Bit j: position p0 + j of a unit's mask m is retained (a non-zero byte).  vec: N and m are
// multiples of 16.
__device__ __forceinline__ uint32_t keep_bits(const uint8_t* m, int p0, int N, bool vec)
{
    uint32_t keep = 0;
    if (vec) {
        if (p0 < N) {
            const uint4 v = *reinterpret_cast<const uint4*>(m + p0);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < kScanBytes; ++j)
                keep |= ((w[j / 4] >> (8 * (j % 4))) & 255u) != 0u ? 1u << j : 0u;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kScanBytes; ++j)
            if (p0 + j < N && m[p0 + j] != 0) keep |= 1u << j;
    }
    return keep;
}

// c[p0 + j] = run + the bits of `keep` below j, for the positions below N.
__device__ __forceinline__ void store_counts(int* c, int p0, int N, bool vec, uint32_t keep, int run)
{
    if (vec) {   // N, and so every row of cnt, is a multiple of 16 entries
        if (p0 < N) {
#pragma unroll
            for (int j = 0; j < kScanBytes; j += 4) {
                int4 o;
                o.x = run;
                o.y = o.x + ((keep >> j) & 1u);
                o.z = o.y + ((keep >> (j + 1)) & 1u);
                o.w = o.z + ((keep >> (j + 2)) & 1u);
                run = o.w + ((keep >> (j + 3)) & 1u);
                *reinterpret_cast<int4*>(c + p0 + j) = o;
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < kScanBytes; ++j) {
            if (p0 + j < N) c[p0 + j] = run;
            run += (keep >> j) & 1u;
        }
    }
}

// The inclusive sum of x over the warp's lanes up to this one.
__device__ __forceinline__ int warp_prefix(int x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Mode 1, step 1: cnt[u][p] = number of retained positions before p; kb[u] = |S0|;
// unit_kk[u] = 0.  One block per unit; a mask byte counts as retained when non-zero.  A
// thread takes 16 consecutive positions, so that a block covers 16384 per step of one
// barrier (with one position per thread and four barriers per step of 1024, the prep of 8
// units of 131072 x 128 took 189 us, now 118; 128 units of 8192 x 64 69 -> 62).
__global__ void scan_kernel(const uint8_t* __restrict__ mask, int N, int* __restrict__ cnt,
                            int* __restrict__ kb, unsigned* __restrict__ unit_kk)
{
    wait_for_previous();
    __shared__ int warp_tot[2][32];
    const int u = blockIdx.x;
    const uint8_t* m = mask + static_cast<int64_t>(u) * N;
    int* c = cnt + static_cast<int64_t>(u) * N;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const bool vec = N % kScanBytes == 0 && (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
    int carry = 0, step = 0;
    for (int base = 0; base < N; base += blockDim.x * kScanBytes, step ^= 1) {
        const int p0 = base + threadIdx.x * kScanBytes;
        const uint32_t keep = keep_bits(m, p0, N, vec);
        const int f = __popc(keep), x = warp_prefix(f, lane);
        if (lane == 31) warp_tot[step][wid] = x;
        __syncthreads();
        const int t = lane < nw ? warp_tot[step][lane] : 0;
        const int all = __reduce_add_sync(0xFFFFFFFFu, t);
        const int mine = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? t : 0);
        store_counts(c, p0, N, vec, keep, carry + mine + x - f);
        carry += all;
        // the next step writes the other half of warp_tot; the one after it follows the
        // next step's barrier
    }
    if (threadIdx.x == 0) {
        kb[u] = carry;
        unit_kk[u] = 0u;
    }
}

// Mode 1, step 2: slot p < N of unit blockIdx.y is key p: its kParts-lane group copies
// it to its column of the retained-first layout (retained keys in position order, then
// from the next tile boundary the evicted ones), with 1/||k_p|| (fp32) and p as column
// metadata, and writes its norm record (and, for float32 keys, its rounded row).  Slots
// p >= N are the padding columns [K, Kpad) and [Kpad + N - K, NP): zero keys, NaN, -1.
// Without `evicted` (b_i(all) is not wanted) the audit reads the columns [0, Kpad) only, and
// only those are written: half of the copy at a ratio of 0.5 (128 units of 8192 x 64:
// prep 61 -> 58 us; 144 of 8192 x 128, 30 % kept: 110 -> 91).
// unit_kk[u] = the unit's largest k.k.  Grid (NP / kKeysPerBlock<D>, U).
template <int D, typename Key>
__global__ void __launch_bounds__(kPrepThreads)
    gather_kernel(const Key* __restrict__ keys, const uint8_t* __restrict__ mask,
                  const int* __restrict__ cnt, const int* __restrict__ kb, int N, int64_t NP,
                  uint16_t* __restrict__ kp, float* __restrict__ colrinv,
                  int* __restrict__ colpos, float4* __restrict__ norms, unsigned* unit_kk,
                  uint16_t* __restrict__ keys16, bool evicted)
{
    wait_for_previous();
    constexpr int Q = D / 8 / kParts, K = kKeys<D>;
    const int part = threadIdx.x % kParts;
    const int p0 = blockIdx.x * kKeysPerBlock<D> + threadIdx.x / kParts;
    const int64_t u = blockIdx.y;
    const int kept = kb[u];
    const int kpad = ((kept + kBN - 1) / kBN) * kBN;
    uint4 v[K][Q];
    int before[K], in[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = p0 + k * kKeysPerStep;
        const int64_t row = u * N + (p < N ? p : 0);   // every lane takes part in the shuffles
        load_key<D>(keys, row, part, v[k]);
        before[k] = cnt[row];
        in[k] = mask[row];
    }
    float top = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = p0 + k * kKeysPerStep;
        int col;
        if (p < N) {
            col = in[k] ? before[k] : kpad + (p - before[k]);
        } else {
            const int r = p - N;
            col = r < kpad - kept ? kept + r : kpad + (N - kept) + (r - (kpad - kept));
        }
        if constexpr (sizeof(Key) == 4)
            if (p < N) store_key<D>(keys16, u * N + p, part, v[k]);
        float r32;
        const float4 nr = key_norms(v[k], r32);
        if (p >= N) {
#pragma unroll
            for (int q = 0; q < Q; ++q) v[k][q] = make_uint4(0u, 0u, 0u, 0u);
        }
        const bool read = evicted || col < kpad;
        if (read) store_key<D>(kp, u * NP + col, part, v[k]);
        if (part == 0) {
            if (read) {
                colrinv[u * NP + col] = p < N ? r32 : nan_f();
                colpos[u * NP + col] = p < N ? p : -1;
            }
            if (p < N) {
                norms[u * N + p] = nr;
                top = fmaxf(top, nr.x);
            }
        }
    }
    unit_max_kk(unit_kk, u, top);
}

// ceil(E / 2) for kk < 2^E: the largest ||k|| of a unit is below 2 to this.
__device__ __forceinline__ int unit_exponent(float kk)
{
    int E;
    (void)frexpf(kk, &E);
    return (E + 1) >> 1;   // also for E <= 0
}

// colrinv[u][c] *= 2^-e_u, the power of two with 2^e_u >= the largest ||k|| of unit u
// (from unit_kk), so that every scaled similarity x_ij * colrinv_j = sim(i,j) ||k_i||
// 2^-e_u lies in [-1, 1].  Exact (a power of two); NaN padding stays NaN.  A unit of
// zero keys keeps its scale.  Given kb, only the retained columns, padded to a tile, are
// scaled.  Four columns per thread: the prep of 144 units of 8192 x 128 79.8 -> 76.6 us, of 128 of
// 8192 x 64 54.6 -> 52.8, of 128 of 16384 x 128 184 -> 179.
// Grid (NP / (4 kPrepThreads) rounded up, U).
__global__ void __launch_bounds__(kPrepThreads)
    scale_columns_kernel(float* __restrict__ colrinv, int64_t NP,
                         const unsigned* __restrict__ unit_kk, const int* __restrict__ kb)
{
    wait_for_previous();
    const int64_t u = blockIdx.y;
    const int64_t c = (static_cast<int64_t>(blockIdx.x) * kPrepThreads + threadIdx.x) * 4;
    const float kk = __uint_as_float(unit_kk[u]);
    const int64_t cols = kb ? (static_cast<int64_t>(kb[u]) + kBN - 1) / kBN * kBN : NP;
    if (c >= cols || !(kk > 0.f)) return;   // cols and NP are multiples of a tile
    const int e = unit_exponent(kk);
    float4* p = reinterpret_cast<float4*>(colrinv + u * NP + c);
    float4 v = *p;
    v.x = ldexpf(v.x, -e);
    v.y = ldexpf(v.y, -e);
    v.z = ldexpf(v.z, -e);
    v.w = ldexpf(v.w, -e);
    *p = v;
}

// Mode 1 in one launch, for the smallest calls, where three launches and the waits between
// them take longer than their work: a cluster of kUnitCtas CTAs does a unit's scan, gather
// and scaling.  Every CTA scans the whole mask (16 bytes per thread) for the retained
// positions before its slots [r NP / 8, (r + 1) NP / 8), so that only the largest k.k
// crosses the cluster; each lane group keeps its slot's 1/||k|| until the scale is known.
// Same values as the three kernels above.  Grid 8 U.
template <int D, typename Key>
__global__ void __cluster_dims__(kUnitCtas, 1, 1) __launch_bounds__(kUnitThreads)
    prep_unit_kernel(const Key* __restrict__ keys, const uint8_t* __restrict__ mask, int N,
                     int64_t NP, int* __restrict__ cnt, int* __restrict__ kb,
                     uint16_t* __restrict__ kp, float* __restrict__ colrinv,
                     int* __restrict__ colpos, float4* __restrict__ norms,
                     uint16_t* __restrict__ keys16, bool evicted)
{
    wait_for_previous();
    constexpr int Q = D / 8 / kParts, kWarps = kUnitThreads / 32;
    static_assert(kWarps == 32, "one warp's total per lane");
    __shared__ int warp_tot[kWarps];
    __shared__ unsigned warp_top[kWarps];
    __shared__ unsigned peer_top[kUnitCtas];
    __shared__ int slot[kUnitSlots];         // retained positions before it; bit 31: retained
    const int rank = static_cast<int>(cluster_rank());
    const int64_t u = blockIdx.x / kUnitCtas;
    const int per = static_cast<int>(NP) / kUnitCtas;   // at most kUnitSlots, a multiple of 32
    const int lo = rank * per;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int part = threadIdx.x % kParts, j = threadIdx.x / kParts, p = lo + j;
    uint4 v[Q];                              // in flight over the scan
    load_key<D>(keys, u * N + (j < per && p < N ? p : 0), part, v);
    const bool vec = N % kScanBytes == 0 && (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
    const int s0 = threadIdx.x * kScanBytes;
    const uint32_t keep = keep_bits(mask + u * N, s0, N, vec);
    const int f = __popc(keep), x = warp_prefix(f, lane);
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    const int t = warp_tot[lane];
    const int kept = __reduce_add_sync(0xFFFFFFFFu, t);
    const int first = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? t : 0) + x - f;
    const int kpad = ((kept + kBN - 1) / kBN) * kBN;
    if (s0 >= lo && s0 < lo + per) {         // 16 slots lie in one CTA's share
        store_counts(cnt + u * N, s0, N, vec, keep, first);
#pragma unroll
        for (int k = 0; k < kScanBytes; ++k)
            slot[s0 - lo + k] = (first + __popc(keep & ((1u << k) - 1u))) |
                                static_cast<int>(((keep >> k) & 1u) << 31);
    }
    if (rank == 0 && threadIdx.x == 0) kb[u] = kept;
    float r32;
    const float4 nr = key_norms(v, r32);     // every lane takes part in its shuffles
    const bool key = j < per && p < N;
    const unsigned wt = __reduce_max_sync(0xFFFFFFFFu, key ? __float_as_uint(fmaxf(nr.x, 0.f)) : 0u);
    if (lane == 0) warp_top[wid] = wt;
    __syncwarp();
    cluster_barrier();                       // slot and warp_top; the other CTAs have started
    if (wid == 0) {
        const unsigned bt = __reduce_max_sync(0xFFFFFFFFu, warp_top[lane]);
        if (lane < kUnitCtas)
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(peer_top + rank, lane)),
                         "r"(bt)
                         : "memory");
    }
    int col = 0;
    bool read = false;
    if (j < per) {
        const int r = p - N, before = slot[j] & 0x7FFFFFFF;
        col = p >= N       ? (r < kpad - kept ? kept + r : kpad + (N - kept) + (r - (kpad - kept)))
              : slot[j] < 0 ? before
                            : kpad + (p - before);
        read = evicted || col < kpad;
        if constexpr (sizeof(Key) == 4)
            if (p < N) store_key<D>(keys16, u * N + p, part, v);
        if (p >= N) {
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] = make_uint4(0u, 0u, 0u, 0u);
        }
        if (read) store_key<D>(kp, u * NP + col, part, v);
        if (part == 0 && p < N) norms[u * N + p] = nr;
    }
    __syncwarp();
    cluster_barrier();
    if (part != 0 || !read) return;
    unsigned kk = 0u;
#pragma unroll
    for (int r = 0; r < kUnitCtas; ++r) kk = max(kk, peer_top[r]);
    const int e = kk != 0u ? unit_exponent(__uint_as_float(kk)) : 0;
    colrinv[u * NP + col] = p < N ? ldexpf(r32, -e) : nan_f();
    colpos[u * NP + col] = p < N ? p : -1;
}

}  // namespace

cudaError_t launch_norms_identity(const void* keys, bool f32, uint16_t* keys16, int U, int N,
                                  int d, int64_t NP, float* colrinv, int* colpos,
                                  float4* norms, cudaStream_t st, float rscale,
                                  unsigned* unit_kk)
{
    const int per = d == 128 ? kKeysPerBlock<128> : kKeysPerBlock<64>;
    const dim3 grid(static_cast<unsigned>(NP / per), U);
    auto go = [&](auto kernel, auto* k) {
        kernel<<<grid, kPrepThreads, 0, st>>>(k, N, NP, colrinv, colpos, norms, rscale, unit_kk,
                                              keys16);
    };
    const float* kf = static_cast<const float*>(keys);
    const uint16_t* kh = static_cast<const uint16_t*>(keys);
    if (f32 && d == 128) go(norms_identity_kernel<128, float>, kf);
    else if (f32) go(norms_identity_kernel<64, float>, kf);
    else if (d == 128) go(norms_identity_kernel<128, uint16_t>, kh);
    else go(norms_identity_kernel<64, uint16_t>, kh);
    return cudaGetLastError();
}

cudaError_t launch_scale_columns(float* colrinv, int U, int64_t NP, const unsigned* unit_kk,
                                 const int* kb, cudaStream_t st)
{
    constexpr int per = 4 * kPrepThreads;
    const dim3 grid(static_cast<unsigned>((NP + per - 1) / per), U);
    return launch_dependent(scale_columns_kernel, grid, kPrepThreads, 0, st, colrinv, NP, unit_kk,
                            kb);
}

cudaError_t launch_scan(const uint8_t* mask, int U, int N, int* cnt, int* kb, unsigned* unit_kk,
                        cudaStream_t st)
{
    // one step where 1024 threads cover the unit, in no more warps than it needs
    const int threads = std::min(1024, (N + 32 * kScanBytes - 1) / (32 * kScanBytes) * 32);
    scan_kernel<<<U, threads, 0, st>>>(mask, N, cnt, kb, unit_kk);
    return cudaGetLastError();
}

cudaError_t launch_prep_unit(const void* keys, bool f32, uint16_t* keys16, const uint8_t* mask,
                             int* cnt, int* kb, int U, int N, int d, int64_t NP, uint16_t* kp,
                             float* colrinv, int* colpos, float4* norms, bool evicted, int sms,
                             cudaStream_t st, bool* launched)
{
    *launched = false;
    // One slot per lane group, half of the SMs at most, and 64 KB of keys per CTA.  us per
    // call, three kernels / one: 1 unit of 512 x 64 (fp32) 31.7 / 27.0, 8 of 1024 x 128
    // 30.0 / 26.2, of 1792 29.5 / 26.8.  Beyond: two slots per group, 8 units of 3072 36.4 /
    // 37.5; 16 units of 1792, whose clusters do not all fit at once, 32.2 / 35.8; 8 fp32 ones of
    // 1792 x 128 with both audits 32.8 / 34.6.
    const int64_t bytes = static_cast<int64_t>(N) * d * (f32 ? 4 : 2);
    if (N > kUnitMaxN || static_cast<int64_t>(U) * kUnitCtas * 2 > sms ||
        bytes > kUnitCtas * (64 << 10))
        return cudaSuccess;
    auto go = [&](auto kernel, auto* k) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(static_cast<unsigned>(U) * kUnitCtas);
        cfg.blockDim = dim3(kUnitThreads);
        cfg.stream = st;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess || clusters < 1) {
            cudaGetLastError();   // no room for a cluster: the caller's other kernels need none
            return cudaSuccess;
        }
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, k, mask, N, NP, cnt, kb, kp, colrinv,
                                                 colpos, norms, keys16, evicted);
        *launched = e == cudaSuccess;
        return e;
    };
    const float* kf = static_cast<const float*>(keys);
    const uint16_t* kh = static_cast<const uint16_t*>(keys);
    if (f32 && d == 128) return go(prep_unit_kernel<128, float>, kf);
    if (f32) return go(prep_unit_kernel<64, float>, kf);
    if (d == 128) return go(prep_unit_kernel<128, uint16_t>, kh);
    return go(prep_unit_kernel<64, uint16_t>, kh);
}

cudaError_t launch_gather(const void* keys, bool f32, uint16_t* keys16, const uint8_t* mask,
                          const int* cnt, const int* kb, int U, int N, int d, int64_t NP,
                          uint16_t* kp, float* colrinv, int* colpos, float4* norms,
                          unsigned* unit_kk, bool evicted, cudaStream_t st)
{
    const int per = d == 128 ? kKeysPerBlock<128> : kKeysPerBlock<64>;
    const dim3 grid(static_cast<unsigned>(NP / per), U);
    auto go = [&](auto kernel, auto* k) {
        return launch_dependent(kernel, grid, kPrepThreads, 0, st, k, mask, cnt, kb, N, NP, kp,
                                colrinv, colpos, norms, unit_kk, keys16, evicted);
    };
    const float* kf = static_cast<const float*>(keys);
    const uint16_t* kh = static_cast<const uint16_t*>(keys);
    if (f32 && d == 128) return go(gather_kernel<128, float>, kf);
    if (f32) return go(gather_kernel<64, float>, kf);
    if (d == 128) return go(gather_kernel<128, uint16_t>, kh);
    return go(gather_kernel<64, uint16_t>, kh);
}

}  // namespace twk
