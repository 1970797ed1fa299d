// twk_policy.cu -- selection of the standalone TwinKV policy (arXiv 2608.27128, Sec. 3.2,
// Eq. 3).
//
// The score of position i is s_i = -r_i / n (Eq. 3) with r_i the redundancy count of
// Eq. 2; the sink and recent regions get the maximum score; the budget's worth of
// highest scores is kept.  Ranking by s descending is ranking by r ascending, so each
// position gets the 32-bit key
//     key_i = 0 for a protected position, r_i + 1 otherwise,
// and the K smallest keys are kept, equal keys in position order (lower first).
//
// One 1024-thread block per unit:
//   1. a radix select over the keys finds the cut: the key value c and how many items equal
//      to c are still to be kept (stopping early when every item sharing the selected
//      prefix is kept).  A key is at most N, so the digits start at N's top bit; 12 bits
//      at a time make one pass below 4096 positions and two up to 16 million;
//   2. one ordered pass keeps every key below the cut and the first `need` keys equal
//      to it, in position order, writing the mask.
// A thread takes eight consecutive positions, so a step covers 8192 and the counts of
// shorter units are read once and stay in registers.  Bound by latency: the steps' barriers
// and the shared-memory atomics.  With byte digits from the top of the word, one position per
// thread and step and one thread walking the 256 counts it took 11.7 us for 128 units of
// 3001 positions and 35.8 for 288 of 8192, now 9.4 and 16.8 (two blocks per SM at 32 registers:
// 10.3 and 16.4; blocks of 512 threads with 16 positions each: 10.2 and 15.7, but the policy
// call of the first shape then takes 190 us instead of 187).
// Counts are read from global memory (once, or once per pass above 8192 positions).
#include "twk_internal.h"
#include "twk_ptx.cuh"

namespace twk {
namespace {

constexpr int kPT = 1024;
constexpr int kPW = kPT / 32;
constexpr int kPV = 8;        // consecutive positions per thread and step
constexpr int kDigit = 12;    // key bits per pass
constexpr int kBins = 1 << kDigit;

struct PolicyShared {
    int hist[kBins];
    int wsum[kPW];
    int sel_digit, sel_before, sel_count;
};

// The keys of positions [p0, p0 + kPV) (p0 below N rounded up); wide: the counts can be
// read 16 bytes at a time.
__device__ __forceinline__ void policy_keys(const int* count, int p0, int N, int n_sink,
                                            int n_recent, bool wide, uint32_t (&key)[kPV])
{
    int c[kPV];
    if (wide) {
#pragma unroll
        for (int j = 0; j < kPV; j += 4) {
            const int4 v = p0 < N ? *reinterpret_cast<const int4*>(count + p0 + j) : int4{};
            c[j] = v.x;
            c[j + 1] = v.y;
            c[j + 2] = v.z;
            c[j + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kPV; ++j) c[j] = p0 + j < N ? count[p0 + j] : 0;
    }
#pragma unroll
    for (int j = 0; j < kPV; ++j) {
        const bool prot = p0 + j < n_sink || p0 + j >= N - n_recent;
        key[j] = prot ? 0u : static_cast<uint32_t>(c[j]) + 1u;
    }
}

// Exclusive block prefix of v; every thread also gets the total.
__device__ __forceinline__ int block_scan(PolicyShared& s, int v, int& total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s.wsum[wid] = x;
    __syncthreads();
    const int t = s.wsum[lane];   // kPW == 32
    total = __reduce_add_sync(0xFFFFFFFFu, t);
    const int before = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? t : 0);
    __syncthreads();
    return before + x - v;
}

__global__ void __launch_bounds__(kPT, 1)
    policy_select_kernel(const int* __restrict__ count_all, int N, const int* __restrict__ budget,
                         int n_sink, int n_recent, uint8_t* __restrict__ mask_all,
                         int* __restrict__ status)
{
    static_assert(kPW == 32, "one warp holds the per-warp totals");
    wait_for_previous();
    __shared__ PolicyShared s;
    const int u = blockIdx.x;
    const int* count = count_all + static_cast<int64_t>(u) * N;
    uint8_t* mask = mask_all + static_cast<int64_t>(u) * N;
    const int K = budget[u];

    if (K < 0 || K > N) {
        for (int i = threadIdx.x; i < N; i += kPT) mask[i] = 0;
        if (status && threadIdx.x == 0) status[u] = 1;   // TWINKV_ERR_INVALID_ARG
        return;
    }
    if (status && threadIdx.x == 0) status[u] = 0;
    if (K == 0 || K == N) {
        for (int i = threadIdx.x; i < N; i += kPT) mask[i] = K == N ? 1 : 0;
        return;
    }
    const bool wide = N % kPV == 0 && (reinterpret_cast<uintptr_t>(count) & 15) == 0;
    const bool wide_mask = N % kPV == 0 && (reinterpret_cast<uintptr_t>(mask) & 3) == 0;
    constexpr int kStep = kPT * kPV;
    const bool once = N <= kStep;   // one step: the keys stay in registers
    const int mine = threadIdx.x * kPV;
    uint32_t key[kPV];
    if (once) policy_keys(count, mine, N, n_sink, n_recent, wide, key);

    // 1. radix select of the cut from the top: `prefix` is the cut's key >> top
    uint32_t prefix = 0;
    int top = 32 - __clz(N);
    int need = K;
    bool whole = false;
    while (top > 0 && !whole) {
        const int shift = max(top - kDigit, 0), bins = 1 << (top - shift);
        for (int d = threadIdx.x; d < bins; d += kPT) s.hist[d] = 0;
        __syncthreads();
        for (int c0 = 0; c0 < N; c0 += kStep) {
            if (!once) policy_keys(count, c0 + mine, N, n_sink, n_recent, wide, key);
#pragma unroll
            for (int j = 0; j < kPV; ++j)
                if (c0 + mine + j < N && (key[j] >> top) == prefix)
                    atomicAdd(&s.hist[(key[j] >> shift) & (bins - 1)], 1);
        }
        __syncthreads();
        // the bin that holds the need-th key: a thread adds up kBins / kPT of them
        constexpr int kPer = kBins / kPT;
        int h[kPer], sum = 0, all;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int d = threadIdx.x * kPer + j;
            h[j] = d < bins ? s.hist[d] : 0;
            sum += h[j];
        }
        int run = block_scan(s, sum, all);
        if (run < need && need <= run + sum) {
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
                if (run < need && need <= run + h[j]) {
                    s.sel_digit = threadIdx.x * kPer + j;
                    s.sel_before = run;
                    s.sel_count = h[j];
                }
                run += h[j];
            }
        }
        __syncthreads();
        need -= s.sel_before;
        prefix = prefix << (top - shift) | static_cast<uint32_t>(s.sel_digit);
        whole = s.sel_count == need;
        top = shift;   // the barriers of the next pass come before sel_* is written again
    }

    // 2. keep the keys below the cut and the first `need` equal to it
    int seen_eq = 0;
    for (int c0 = 0; c0 < N; c0 += kStep) {
        if (!once) policy_keys(count, c0 + mine, N, n_sink, n_recent, wide, key);
        int eq = 0;
#pragma unroll
        for (int j = 0; j < kPV; ++j)
            eq += c0 + mine + j < N && !whole && (key[j] >> top) == prefix ? 1 : 0;
        int total = 0, at = 0;
        if (!whole) at = seen_eq + block_scan(s, eq, total);   // alike in the whole block
        seen_eq += total;
        uint32_t keep[kPV / 4] = {};   // a mask byte per position
#pragma unroll
        for (int j = 0; j < kPV; ++j) {
            const uint32_t km = key[j] >> top;
            const bool same = km == prefix;
            if (km < prefix || (same && (whole || at < need))) keep[j / 4] |= 1u << (8 * (j % 4));
            at += same ? 1 : 0;
        }
        if (wide_mask) {
#pragma unroll
            for (int j = 0; j < kPV; j += 4)
                if (c0 + mine < N) *reinterpret_cast<uint32_t*>(mask + c0 + mine + j) = keep[j / 4];
        } else {
#pragma unroll
            for (int j = 0; j < kPV; ++j)
                if (c0 + mine + j < N)
                    mask[c0 + mine + j] = (keep[j / 4] >> (8 * (j % 4))) & 1u;
        }
    }
}

}  // namespace

cudaError_t launch_policy_select(const int* count, int U, int N, const int* budget, int n_sink,
                                 int n_recent, uint8_t* out_mask, int* out_status,
                                 cudaStream_t st)
{
    return launch_dependent(policy_select_kernel, dim3(U), kPT, 0, st, count, N, budget, n_sink,
                            n_recent, out_mask, out_status);
}

}  // namespace twk
