// twk_repair.cu -- budget-exact repair swap of TwinKV (arXiv 2608.27128, Sec. 3.4).
//
// Per unit (layer, KV head):
//   classify  orphan = i not in S0 and b_i < tau,
//             donor  = j in S0, outside [0, n_sink) and [N - n_recent, N), b_j >= tau,
//   each entry a (severity key, position) pair: orphans keyed by b ascending, donors by
//   b descending, through an order-preserving fp64 -> u64 map (-0 folded into +0);
//   m = min(|O|, |D|); the m most severe orphans and donors, ordered by (key, position)
//   so that equal severities keep position order (lower position first);
//   S1 = S0 with the m donors cleared and the m orphans set; swaps[k] = (donor k,
//   orphan k); a unit whose mask has a byte > 1 or whose popcount differs from its
//   budget gets status, nswaps = -1 and S1 = S0.
//
// The literal rule (select_kernel<C>) runs each unit on a cluster of C CTAs (C = 1 to 16 by
// select_cluster_size): by buckets in shared memory (see "bucket path" below) up to 2^18
// positions, a unit with an overfull bucket of several values and longer ones by a radix
// select and sorts over the workspace ("cluster selection").  Its scratch is caller workspace
// ([U][N] keys and positions, twice) and 72 KB of dynamic shared memory per CTA.
//
// Dedup variant (dedup_kernel, given the twin of every position; one 512-thread block
// per unit): evicting a donor keeps its twin, so a twin pair never loses both members.
// Where all donors fit, by buckets too, with the walk in rounds (dedup_swap); else:
// All donors are sorted; each gets the donor rank of its twin (through a position ->
// rank table in the workspace); one thread then walks the ranks in severity order with
// two bits of state per rank in shared memory (evicted, pinned): a donor is skipped
// when it is pinned (the twin of an evicted donor) or its twin is evicted, and the
// walk stops after |O| evictions.  The ranks it needs are staged in shared memory
// chunk by chunk, so the walk itself touches shared memory only.  m = the evictions;
// the m most severe orphans are then selected with a radix select (byte histograms
// from the top) and sorted: up to 4096 items by a bitonic network in shared memory,
// more by a stable LSD radix sort (8-bit digits, warp match + per-warp digit counts; a
// digit position shared by every key is skipped).
#include <algorithm>

#include <cooperative_groups.h>

#include "twk_internal.h"
#include "twk_ptx.cuh"

namespace twk {
namespace {

constexpr int kT = 512;   // two blocks per SM: every unit of a prefill in one wave
constexpr int kW = kT / 32;

// Order-preserving map of an fp64 value to a u64 key (-0 folded into +0), in integer
// operations only: fp64 comparisons run on this GPU's narrow FP64 pipe.
__device__ __forceinline__ uint64_t ordered(double b)
{
    uint64_t u = static_cast<uint64_t>(__double_as_longlong(b));
    if (u == 0x8000000000000000ull) u = 0ull;
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

__device__ __forceinline__ bool is_nan_bits(double b)
{
    return (static_cast<uint64_t>(__double_as_longlong(b)) & 0x7FFFFFFFFFFFFFFFull) >
           0x7FF0000000000000ull;
}

struct Shared {
    int warp_cnt[kW][256];   // per-warp digit counts, then their prefix over warps
    int base[256];           // running output offset of each digit
    int chunk_tot[256];
    int wsum[2][kW];         // block-scan scratch for the two lists
    int red[4];
    int flag;
    int sel_digit, sel_before, sel_count;
};

// Block-wide exclusive scan of two 0/1 flags; returns the prefixes and the chunk totals.
__device__ __forceinline__ void scan2(Shared& s, int fo, int fd, int& po, int& pd, int& to,
                                      int& td)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t bo = __ballot_sync(0xFFFFFFFFu, fo);
    const uint32_t bd = __ballot_sync(0xFFFFFFFFu, fd);
    const uint32_t lt = (1u << lane) - 1u;
    if (lane == 0) {
        s.wsum[0][wid] = __popc(bo);
        s.wsum[1][wid] = __popc(bd);
    }
    __syncthreads();
    if (wid == 0) {
        int a = lane < kW ? s.wsum[0][lane] : 0, b = lane < kW ? s.wsum[1][lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ya = __shfl_up_sync(0xFFFFFFFFu, a, o);
            const int yb = __shfl_up_sync(0xFFFFFFFFu, b, o);
            if (lane >= o) {
                a += ya;
                b += yb;
            }
        }
        if (lane < kW) {
            s.wsum[0][lane] = a;   // inclusive
            s.wsum[1][lane] = b;
        }
    }
    __syncthreads();
    po = (wid ? s.wsum[0][wid - 1] : 0) + __popc(bo & lt);
    pd = (wid ? s.wsum[1][wid - 1] : 0) + __popc(bd & lt);
    to = s.wsum[0][kW - 1];
    td = s.wsum[1][kW - 1];
    __syncthreads();
}

// Called by warp 0 only: the 256 digit counts in cnt become their exclusive prefix
// (eight digits per lane and a shuffle scan); returns whether one digit holds all n.
__device__ __forceinline__ bool digit_prefix(int* cnt, int n)
{
    const int lane = threadIdx.x & 31;
    int c[8], t = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        c[j] = cnt[lane * 8 + j];
        t += c[j];
    }
    int incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    int run = incl - t;
    bool one = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        one |= c[j] == n;
        cnt[lane * 8 + j] = run;
        run += c[j];
    }
    return __any_sync(0xFFFFFFFFu, one);
}

// Called by warp 0 only: the smallest digit d whose counts up to and including d reach
// `need` (255 at most), the count before it and its own count, into s.
__device__ __forceinline__ void digit_cut(const int* cnt, int need, int& sel_digit,
                                          int& sel_before, int& sel_count)
{
    const int lane = threadIdx.x & 31;
    int c[8], t = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        c[j] = cnt[lane * 8 + j];
        t += c[j];
    }
    int incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t reach = __ballot_sync(0xFFFFFFFFu, incl >= need);
    const int L = reach ? __ffs(reach) - 1 : 31;
    if (lane == L) {
        // the first of the lane's digits whose running count reaches need (its last
        // digit otherwise: digit 255 for lane 31); constant indices keep c in registers
        int run = incl - t, sel = 7, before = 0, count = c[7];
        bool found = false;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (!found && (j == 7 || run + c[j] >= need)) {
                sel = j;
                before = run;
                count = c[j];
                found = true;
            }
            if (!found) run += c[j];
        }
        sel_digit = L * 8 + sel;
        sel_before = before;
        sel_count = count;
    }
}

// Block-wide exclusive scan of two per-thread counts; returns each thread's prefixes
// and the totals.
__device__ __forceinline__ void scan2n(Shared& s, int co, int cd, int& po, int& pd, int& to,
                                       int& td)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int io = co, id = cd;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int yo = __shfl_up_sync(0xFFFFFFFFu, io, o);
        const int yd = __shfl_up_sync(0xFFFFFFFFu, id, o);
        if (lane >= o) {
            io += yo;
            id += yd;
        }
    }
    if (lane == 31) {
        s.wsum[0][wid] = io;
        s.wsum[1][wid] = id;
    }
    __syncthreads();
    if (wid == 0) {
        int x = lane < kW ? s.wsum[0][lane] : 0, y = lane < kW ? s.wsum[1][lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int xo = __shfl_up_sync(0xFFFFFFFFu, x, o);
            const int yo = __shfl_up_sync(0xFFFFFFFFu, y, o);
            if (lane >= o) {
                x += xo;
                y += yo;
            }
        }
        if (lane < kW) {
            s.wsum[0][lane] = x;   // inclusive
            s.wsum[1][lane] = y;
        }
    }
    __syncthreads();
    po = (wid ? s.wsum[0][wid - 1] : 0) + io - co;
    pd = (wid ? s.wsum[1][wid - 1] : 0) + id - cd;
    to = s.wsum[0][kW - 1];
    td = s.wsum[1][kW - 1];
    __syncthreads();
}

constexpr int kE = 4;   // consecutive positions per thread in the streaming passes
constexpr int kH = 4;   // items per thread per round of a digit histogram

// One stable counting pass on digit (key >> shift) & 255 of n items; returns false
// (and moves nothing) when every item has the same digit.
__device__ bool radix_pass(Shared& s, const uint64_t* kin, const int* iin, uint64_t* kout,
                           int* iout, int n, int shift)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kW * 256; i += kT) (&s.warp_cnt[0][0])[i] = 0;
    if (threadIdx.x < 256) s.base[threadIdx.x] = 0;
    __syncthreads();
    for (int c0 = 0; c0 < n; c0 += kT * kH) {
        int dg[kH];
#pragma unroll
        for (int e = 0; e < kH; ++e) {   // the loads first: kH in flight per thread
            const int i = c0 + e * kT + threadIdx.x;
            dg[e] = i < n ? static_cast<int>((kin[i] >> shift) & 255) : 256;
        }
#pragma unroll
        for (int e = 0; e < kH; ++e) {
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, dg[e]);
            if (dg[e] < 256 && lane == __ffs(peers) - 1) atomicAdd(&s.base[dg[e]], __popc(peers));
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const bool single = digit_prefix(s.base, n);
        if (threadIdx.x == 0) s.flag = single;
    }
    __syncthreads();
    if (s.flag) return false;
    for (int c0 = 0; c0 < n; c0 += kT) {
        const int i = c0 + threadIdx.x;
        const bool valid = i < n;
        const uint64_t key = valid ? kin[i] : 0ull;
        const int dg = valid ? static_cast<int>((key >> shift) & 255) : 256;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, dg);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (valid && rank == 0) s.warp_cnt[wid][dg] = __popc(peers);
        __syncthreads();
        if (threadIdx.x < 256) {
            int run = 0;
            for (int w = 0; w < kW; ++w) {
                const int t = s.warp_cnt[w][threadIdx.x];
                s.warp_cnt[w][threadIdx.x] = run;
                run += t;
            }
            s.chunk_tot[threadIdx.x] = run;
        }
        __syncthreads();
        if (valid) {
            const int dst = s.base[dg] + s.warp_cnt[wid][dg] + rank;
            kout[dst] = key;
            iout[dst] = iin[i];
        }
        __syncthreads();
        if (threadIdx.x < 256) {
            s.base[threadIdx.x] += s.chunk_tot[threadIdx.x];
            for (int w = 0; w < kW; ++w) s.warp_cnt[w][threadIdx.x] = 0;
        }
        __syncthreads();
    }
    return true;
}

// Sorts n (key, position) items held at offset `off` of buffer 0; returns the buffer
// (0 or 1) that holds the sorted result.
__device__ int radix_sort(Shared& s, uint64_t* k0, int* i0, uint64_t* k1, int* i1, int n)
{
    int cur = 0;
    for (int shift = 0; shift < 64; shift += 8) {
        const bool moved = cur == 0 ? radix_pass(s, k0, i0, k1, i1, n, shift)
                                    : radix_pass(s, k1, i1, k0, i0, n, shift);
        if (moved) cur ^= 1;
        __syncthreads();
    }
    return cur;
}

// Moves the m smallest of the n (key, position) items in (kin, iin) to (kout, iout),
// keeping their order (position order), so that ties at the cut go to the lower
// positions.  The cut is found byte by byte from the top (a radix select: one
// histogram per byte over the items that still share the selected prefix), stopping
// early once the whole boundary bucket is selected.  Requires 0 < m <= n.
__device__ void select_smallest(Shared& s, const uint64_t* kin, const int* iin, uint64_t* kout,
                                int* iout, int n, int m)
{
    const int lane = threadIdx.x & 31;
    uint64_t prefix = 0, pmask = 0;
    int need = m;                 // items still to take among those matching the prefix
    bool whole = false;           // every item matching the prefix is taken
    for (int shift = 56; shift >= 0 && !whole; shift -= 8) {
        if (threadIdx.x < 256) s.base[threadIdx.x] = 0;
        __syncthreads();
        for (int c0 = 0; c0 < n; c0 += kT * kH) {
            int dg[kH];
#pragma unroll
            for (int e = 0; e < kH; ++e) {   // the loads first: kH in flight per thread
                const int i = c0 + e * kT + threadIdx.x;
                dg[e] = 256;
                if (i < n) {
                    const uint64_t key = kin[i];
                    if ((key & pmask) == prefix) dg[e] = static_cast<int>((key >> shift) & 255);
                }
            }
#pragma unroll
            for (int e = 0; e < kH; ++e) {
                const uint32_t peers = __match_any_sync(0xFFFFFFFFu, dg[e]);
                if (dg[e] < 256 && lane == __ffs(peers) - 1)
                    atomicAdd(&s.base[dg[e]], __popc(peers));
            }
        }
        __syncthreads();
        if (threadIdx.x < 32) digit_cut(s.base, need, s.sel_digit, s.sel_before, s.sel_count);
        __syncthreads();
        need -= s.sel_before;
        prefix |= static_cast<uint64_t>(s.sel_digit) << shift;
        pmask |= 255ull << shift;
        whole = s.sel_count == need;
        __syncthreads();
    }
    // Ordered compaction: items below the prefix, then those equal to it (all of them
    // when `whole`, else the first `need` in position order).
    int base = 0, seen_eq = 0;
    for (int c0 = 0; c0 < n; c0 += kT) {
        const int i = c0 + threadIdx.x;
        int fl = 0, fe = 0;
        uint64_t key = 0;
        if (i < n) {
            key = kin[i];
            const uint64_t km = key & pmask;
            fl = km < prefix || (whole && km == prefix);
            fe = !whole && km == prefix;
        }
        int pl, pe, tl, te;
        scan2(s, fl, fe, pl, pe, tl, te);
        const int k_eq = max(0, min(te, need - seen_eq));   // eq items taken in this chunk
        if (fl || (fe && pe < k_eq)) {
            const int dst = base + pl + min(pe, k_eq);
            kout[dst] = key;
            iout[dst] = iin[i];
        }
        base += tl + k_eq;
        seen_eq += te;
    }
    __syncthreads();
}

// Lists of at most kSortMax items are sorted in shared memory (kSortMax * 12 bytes of
// dynamic shared memory), longer ones by the radix passes over the workspace.
constexpr int kSortMax = 4096;

// Sorts the n <= kSortMax items (kin, iin) ascending by (key, position) into (kout,
// iout), with a bitonic network in shared memory (sk, si) padded to a power of two by
// items that sort last.  Positions are distinct, so the order equals that of a stable
// sort by key of a list in position order.
__device__ void smem_sort(uint64_t* sk, int* si, const uint64_t* kin, const int* iin, int n,
                          uint64_t* kout, int* iout)
{
    int P = 1;
    while (P < n) P <<= 1;
    for (int t = threadIdx.x; t < P; t += kT) {
        sk[t] = t < n ? kin[t] : ~0ull;
        si[t] = t < n ? iin[t] : 0x7FFFFFFF;
    }
    __syncthreads();
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < P / 2; t += kT) {
                const int lo = 2 * t - (t & (stride - 1));
                const int hi = lo + stride;
                const uint64_t ka = sk[lo], kb = sk[hi];
                const int pa = si[lo], pb = si[hi];
                const bool gt = ka > kb || (ka == kb && pa > pb);
                if (gt == ((lo & size) == 0)) {   // ascending blocks swap a greater first
                    sk[lo] = kb;
                    sk[hi] = ka;
                    si[lo] = pb;
                    si[hi] = pa;
                }
            }
            __syncthreads();
        }
    }
    for (int t = threadIdx.x; t < n; t += kT) {
        kout[t] = sk[t];
        iout[t] = si[t];
    }
    __syncthreads();
}

// The m most severe items of one list, in severity order: (key, position) pairs at
// (k, i) with scratch (kx, ix) of the same extent; returns the position array holding
// them.  (sk, si): kSortMax items of shared memory.
__device__ const int* most_severe(Shared& s, uint64_t* k, int* i, uint64_t* kx, int* ix, int n,
                                  int m, uint64_t* sk, int* si)
{
    if (n > m) {
        select_smallest(s, k, i, kx, ix, n, m);
        if (m <= kSortMax) {
            smem_sort(sk, si, kx, ix, m, k, i);
            return i;
        }
        return radix_sort(s, kx, ix, k, i, m) ? i : ix;
    }
    if (n <= kSortMax) {
        smem_sort(sk, si, k, i, n, kx, ix);
        return ix;
    }
    return radix_sort(s, k, i, kx, ix, n) ? ix : i;
}

constexpr int kWalkChunk = 4096;   // twin ranks staged per step of the dedup walk

// Dynamic shared memory of the dedup variant: 2 state bits per donor rank (n_d <= N),
// then one chunk of staged twin ranks (the sort buffers follow, 16-byte aligned).
__host__ __device__ inline size_t dedup_smem_bytes(int N)
{
    return static_cast<size_t>((N + 15) / 16) * 4 + kWalkChunk * 4;
}

// Offset of the shared-memory sort buffers (kSortMax keys, then kSortMax positions) in
// the dynamic shared memory, and the total dynamic bytes.
__host__ __device__ inline size_t sort_smem_offset(int N)
{
    return (dedup_smem_bytes(N) + 15) / 16 * 16;
}

__host__ __device__ inline size_t dedup_kernel_smem_bytes(int N)
{
    return sort_smem_offset(N) + static_cast<size_t>(kSortMax) * 12;
}

// ---------------------------------------------------------------- cluster selection
//
// The literal repair (Sec. 3.4) of one unit on a cluster of C CTAs (C = 1: one CTA).
// CTA r of the cluster owns the slice [r S, (r + 1) S) of the unit's positions.
//   A. One pass over the slice: S1 = S0, validation counts, and the slice's orphans
//      (forward from the slice start) and donors (backward from the slice end) as
//      (severity key, position) pairs in keys0/idx0.  n_o + n_d never exceeds the
//      slice length, so the two lists never meet.
//   B. Counts through distributed shared memory: totals, this CTA's offsets, status,
//      m = min(|O|, |D|).  The side with more than m items is cut by a radix select
//      whose digit histograms are summed over the cluster (each CTA histograms its own
//      items; the sums, and so every decision, are identical in every CTA); the other
//      side is taken whole; each CTA's own counts below and at the cut come from its
//      own histograms.  An ordered compaction writes the m items of each side, in
//      position order, to keys1/idx1 (orphans at [0, m), donors at [N/2, N/2 + m)).
//   C. Each CTA sorts its share of both lists by (key, position) with a bitonic
//      network held in registers (eight slots per thread; warp shuffles for strides up
//      to 128, shared memory beyond): both sides at once for shares of up to kChunk
//      items, one side after the other for shares of up to 2 kChunk.  An item's place
//      in the swap list is its rank in its own share plus, for every other share, the
//      number of that share's items ordered before it (binary search in the other
//      CTA's shared memory).  Larger shares are sorted by one CTA per side with the
//      stable radix passes over the workspace.
// Every CTA of a cluster runs the same sequence of cluster barriers: each branch and
// loop bound that leads to one depends only on values that are identical in every CTA.
namespace cg = cooperative_groups;

constexpr int kChunk = 2048;   // items per side a CTA sorts at once (both sides)

template <int C>
__device__ __forceinline__ void cluster_sync()
{
    if constexpr (C == 1) __syncthreads();
    else cg::this_cluster().sync();
}

// The value of the same shared-memory object in CTA `rank` of the cluster, by a 32-bit
// shared::cluster address (generic pointers made the kernel spill).
__device__ __forceinline__ int load_at(uint32_t at, int)
{
    int v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ uint64_t load_at(uint32_t at, uint64_t)
{
    uint64_t v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(at) : "memory");
    return v;
}
template <int C, typename T>
__device__ __forceinline__ T peer(const T* p, int rank)
{
    if constexpr (C == 1) return *p;
    else return load_at(cluster_addr(p, static_cast<uint32_t>(rank)), T());
}

constexpr int kMaxHeavy = 32;   // buckets ranked by position in a unit's selection

struct ClusterShared {
    int cnt[8];          // this CTA's orphans, donors, retained count, invalid-byte flag;
                         // bucket path: smallest and largest orphan, then donor, as_int order
    int all[8];          // bucket path: the same over the cluster
    // the bucket path's overfull buckets (see rank_heavy): how many; which, how many items,
    // the first one's rank, the least and largest key and the count in this slice, the rank
    // of the slice's next item
    int n_heavy;
    int hk[kMaxHeavy], hc[kMaxHeavy], hrank[kMaxHeavy], hcnt[kMaxHeavy], hnext[kMaxHeavy];
    uint64_t hmin[kMaxHeavy], hmax[kMaxHeavy];
    int lcnt[2];         // compaction: this CTA's items below the cut and at it
    int hist[2][256];    // this CTA's digit histogram, alternating between passes
    int tot[8];          // cluster-wide values derived by thread 0
};

__device__ __forceinline__ bool before(uint64_t ka, int pa, uint64_t kb, int pb)
{
    return ka < kb || (ka == kb && pa < pb);
}

// Number of entries of the sorted (key, position) array of P = 2^k entries in CTA `rank`'s
// shared memory that order before (k, p).
__device__ __forceinline__ int count_before(const uint64_t* sk, const int* si, int rank, int P,
                                            uint64_t k, int p)
{
    const uint32_t ak = cluster_addr(sk, static_cast<uint32_t>(rank));
    const uint32_t ai = cluster_addr(si, static_cast<uint32_t>(rank));
    auto first = [&](int at) {
        return before(load_at(ak + 8u * at, uint64_t()), load_at(ai + 4u * at, 0), k, p);
    };
    int pos = 0;
    for (int half = P >> 1; half > 0; half >>= 1)
        if (first(pos + half - 1)) pos += half;
    if (first(pos)) ++pos;
    return pos;
}

constexpr int kR = 8;   // items per thread in the share sort's registers

// Compare-exchange of two items: afterwards a orders before b when `up`, after it
// otherwise.
__device__ __forceinline__ void cx(uint64_t& ka, int& pa, uint64_t& kb, int& pb, bool up)
{
    const bool sw = before(kb, pb, ka, pa) == up;
    const uint64_t k0 = sw ? kb : ka, k1 = sw ? ka : kb;
    const int p0 = sw ? pb : pa, p1 = sw ? pa : pb;
    ka = k0;
    kb = k1;
    pa = p0;
    pb = p1;
}

// kR items between registers and the shared-memory slots [at, at + kR) (16-byte
// aligned: at is a multiple of kR).
__device__ __forceinline__ void store_run(uint64_t* sk, int* si, int at, const uint64_t* kx,
                                          const int* px)
{
#pragma unroll
    for (int e = 0; e < kR; e += 2)
        *reinterpret_cast<ulonglong2*>(sk + at + e) = make_ulonglong2(kx[e], kx[e + 1]);
#pragma unroll
    for (int e = 0; e < kR; e += 4)
        *reinterpret_cast<int4*>(si + at + e) = make_int4(px[e], px[e + 1], px[e + 2], px[e + 3]);
}

__device__ __forceinline__ void load_run(const uint64_t* sk, const int* si, int at, uint64_t* kx,
                                         int* px)
{
#pragma unroll
    for (int e = 0; e < kR; e += 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(sk + at + e);
        kx[e] = v.x;
        kx[e + 1] = v.y;
    }
#pragma unroll
    for (int e = 0; e < kR; e += 4) {
        const int4 v = *reinterpret_cast<const int4*>(si + at + e);
        px[e] = v.x;
        px[e + 1] = v.y;
        px[e + 2] = v.z;
        px[e + 3] = v.w;
    }
}

// x, as a value that the compiler knows nothing about.
__device__ __forceinline__ void forget(int& x) { asm volatile("" : "+r"(x)); }

constexpr int kEA = 8;   // consecutive positions per thread in the classification pass

// Slice length: ceil(N / C) rounded up to a multiple of kEA.
__host__ __device__ inline int slice_len(int N, int C)
{
    const int q = (N + C - 1) / C;
    return (q + kEA - 1) / kEA * kEA;
}

// ---- bucket path -------------------------------------------------------------------
//
// The usual case of the selection: no list is written to memory and nothing is sorted by
// comparisons across the CTA.  Three passes read the slice's b and mask (coalesced, in any
// order):
//   1. S1 = S0, the counts, and the smallest and largest b of each side;
//   2. a histogram of each side over kBk intervals of its range, summed over the cluster;
//      its prefix sums give every bucket's first rank.  Buckets whose first rank is below m
//      hold the m most severe items (and the rest of the bucket at the cut);
//   3. their items go to the bucket's place in the shared memory of the CTA that owns the
//      bucket (buckets are dealt out by first rank, so that each CTA gets about 1/C).
// An item's rank is its bucket's first rank plus the number of items of its bucket ordered
// before it, counted one by one.  The intervals are taken on b rounded toward zero to fp32,
// which keeps the order, so the ranks are those of the (key, position) order whatever the
// values.  A unit that does not fit so goes on in rank_many: lists beyond the shared memory
// window by window, overfull buckets of one value (exact duplicate keys, coarse scores) by
// position (rank_heavy).  Only an overfull bucket of several values is left to the general
// path.
// Why: the selection is bound by latency, the round trips of its passes and barriers.  The
// general path's radix select takes up to eight passes over lists in memory with several
// block barriers each, and its bitonic sort was 58 of 182 thousand cycles per unit at 16384
// positions.  General -> buckets, half of the positions kept, 20 % of b near 1: 288 units of
// 16384 positions 119 -> 59 us, 128 of 8192 62 -> 23, 8 of 4096 55 -> 14, 8 of 8192 67 -> 19,
// 8 of 131072 289 -> 89; 50 % near 1 (lists beyond one window) 288 of 16384 394 -> 109, 8 of
// 131072 629 -> 203; 30 % equal to 1 288 of 16384 182 -> 125, 288 of 4096 58 -> 39, 8 of
// 131072 363 -> 174.  What is left to the general path has paid for the attempt: with 60 % of
// b within 1e-6 of 0.5, 288 of 16384 197 -> 231, 288 of 4096 62 -> 76 (8 of 8192 88 -> 64, by
// fewer CTAs).
constexpr int kBk = 1024;      // buckets per side
constexpr int kCap = 3072;     // items per side a CTA holds (36 KB): two CTAs per SM fit
// The number of items of a bucket above which counting one by one costs too much.  Buckets
// are as full as the unit is long: at 131072 positions with normally distributed b up to 330
// items (8 units 89 us counted through, 267 by the general path).
__host__ __device__ inline int max_bucket(int N) { return min(1024, max(256, N / 256)); }

// Beyond this a unit's buckets are too full whatever its values: the general path only.
constexpr int kBucketMaxN = 1 << 18;

// Where a unit has an overfull bucket, its buckets of one value and more than this many items
// are ranked by position as well.
constexpr int kFew = 48;

// How far the bucket path got: all done; counts and ranges are in cs.all (and S1 = S0); or
// also the buckets' first ranks are in s.warp_cnt and the ends of what is in play in cs.tot.
enum Attempt { kNone, kDone, kCounted, kRanked };

// A float's bits as an int with the float's order.
__device__ __forceinline__ int as_int(float f)
{
    const int i = __float_as_int(f);
    return i ^ ((i >> 31) & 0x7FFFFFFF);
}
__device__ __forceinline__ float from_int(int i)
{
    return __int_as_float(i ^ ((i >> 31) & 0x7FFFFFFF));
}

// A double's bits (not a NaN's) as an fp32 value, rounded toward zero: monotone, in integer
// operations.  Beyond fp32's range it is 0 or the largest fp32 value.
__device__ __forceinline__ float narrow(uint64_t u)
{
    const uint32_t hi = static_cast<uint32_t>(u >> 32), lo = static_cast<uint32_t>(u);
    const int e = static_cast<int>((hi >> 20) & 0x7FFu) - 896;
    const uint32_t mant = ((hi & 0xFFFFFu) << 3) | (lo >> 29);
    const uint32_t mag = e <= 0 ? 0u : e >= 255 ? 0x7F7FFFFFu : (static_cast<uint32_t>(e) << 23) | mant;
    return __uint_as_float((hi & 0x80000000u) | mag);
}

// How a side's values map to buckets.  d is a value's distance from the side's most severe
// end, w the whole range: half of the buckets divide w evenly, the other half divide the
// 16 octaves below w, and a value's bucket is the sum of its two shares.  Evenly spread
// values keep a bucket each per 1/512 of the range, and the twins that crowd within 1e-5 to
// 1e-3 of the largest b spread over the octaves (with 1024 even intervals they filled one
// bucket, and the Llama-3.2-1B cache's units went to the general path, 60 us).
// Non-decreasing in d (each operation is).
struct Buckets {
    float end;     // the most severe value, as fp32
    float inv;     // (kBk / 2 - 1) / w, or 0: every value in bucket 0
    int floor;     // bits of w 2^-16, as an int
};

__device__ __forceinline__ Buckets make_buckets(float severe, float mild)
{
    const float w = fabsf(mild - severe);
    Buckets k{severe, (kBk / 2 - 1) / w, __float_as_int(w) - (16 << 23)};
    if (!(w > 0.f && w <= 3.4e38f && k.inv <= 3.4e38f)) {
        k.inv = 0.f;
        k.floor = 0x7FFFFFFF;
    }
    return k;
}

__device__ __forceinline__ int bucket_of(float f, const Buckets& k)
{
    const float d = fabsf(f - k.end);
    const int over = max(0, __float_as_int(d) - max(k.floor, 0));   // 2^23 per octave
    const float v = __fmaf_rn(d, k.inv, static_cast<float>(k.inv == 0.f ? 0 : over) * 0x1p-18f);
    return min(kBk - 1, static_cast<int>(v));
}

// The b whose severity key (side 0: orphans, 1: donors) is k, as the double's bits.
__device__ __forceinline__ uint64_t bits_of_key(uint64_t k, int side)
{
    const uint64_t o = side ? ~k : k;
    return (o >> 63) ? (o & 0x7FFFFFFFFFFFFFFFull) : ~o;
}

// What a position is: 0 an orphan, 1 a donor, 2 neither.
__device__ __forceinline__ int side_of(uint32_t m, double bi, uint64_t ki, int i,
                                       const RepairArgs& a, uint64_t ktau)
{
    if (is_nan_bits(bi)) return 2;
    if (m == 0u) return ki < ktau ? 0 : 2;
    const bool prot = i < a.n_sink || i >= a.N - a.n_recent;
    return !prot && ki >= ktau ? 1 : 2;
}

// Accesses to the same shared-memory object in CTA `rank` of the cluster, by 32-bit
// shared::cluster addresses (generic pointers made the kernel spill).
__device__ __forceinline__ int peer_add(int* p, int rank, int v)
{
    int old;
    asm volatile("atom.relaxed.cluster.shared::cluster.add.s32 %0, [%1], %2;"
                 : "=r"(old)
                 : "r"(cluster_addr(p, static_cast<uint32_t>(rank))), "r"(v)
                 : "memory");
    return old;
}
__device__ __forceinline__ void peer_store(uint64_t* p, int rank, uint64_t v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(
                     cluster_addr(p, static_cast<uint32_t>(rank))),
                 "l"(v)
                 : "memory");
}
__device__ __forceinline__ void peer_store(int* p, int rank, int v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(
                     cluster_addr(p, static_cast<uint32_t>(rank))),
                 "r"(v)
                 : "memory");
}

__device__ void dedup_swap(Shared& s, uint64_t* sk, int* si, const Buckets& bd,
                           const RepairArgs& a, int u, const int* end, int n_o, uint64_t ktau,
                           const int (&rank)[2][kCap / kT]);

// The thread's kP positions of the step at c0: c0 + tid, + kT, ...
template <int kP>
__device__ __forceinline__ void load_step(const uint8_t* S0, const double* b, int c0, int hi,
                                          uint32_t (&mv)[kP], double (&bv)[kP])
{
#pragma unroll
    for (int j = 0; j < kP; ++j) {
        const int i = c0 + j * kT + static_cast<int>(threadIdx.x);
        mv[j] = i < hi ? S0[i] : 255u;
        bv[j] = i < hi ? b[i] : 0.0;
    }
}

// For a unit with an overfull bucket (more than max_bucket items in play): the buckets of one
// value and more than kFew items are ranked by position, which takes no counting and no place
// in shared memory.  They leave the buckets' places (base, cur): base is marked with the top
// bit and cur holds the bucket's number.  A first pass finds which candidates hold one value
// and counts this slice's items; a second one goes through the slice in position order (warp
// votes, then a prefix over the rows of a step, as in a radix pass) and writes their swaps.
// cs.tot is then the fullest of the other buckets and the ends of the places in play.  False,
// with nothing written, where an overfull bucket holds several values or there are too many.
template <int C>
__device__ bool rank_heavy(Shared& s, ClusterShared& cs, int* rows, const RepairArgs& a, int u,
                           int r, int m)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t off = static_cast<int64_t>(u) * a.N;
    const uint8_t* S0 = a.mask + off;
    const double* b = a.b + off;
    const int slice = slice_len(a.N, C);
    const int lo = min(a.N, r * slice), hi = min(a.N, lo + slice);
    const uint64_t ktau = ordered(a.tau);
    int* base = &s.warp_cnt[0][0];
    int* cur = base + 2 * kBk;
    constexpr int kPer = 2 * kBk / kT;
    const int b0 = tid * kPer, side = b0 / kBk, limit = max_bucket(a.N);

    // 1. the candidates
    int first[kPer + 1];
#pragma unroll
    for (int k = 0; k < kPer; ++k) first[k] = base[b0 + k];
    first[kPer] = (b0 + kPer) % kBk ? base[b0 + kPer] : cs.all[side];
    int least = kFew, id, unused, n_all;
    for (;;) {
        int n = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) n += first[k] < m && first[k + 1] - first[k] > least;
        scan2n(s, n, 0, id, unused, n_all, unused);   // (every thread has read base and tot)
        if (n_all <= kMaxHeavy) break;
        if (least == limit) return false;             // alike in every CTA
        least = limit;
    }
    if (tid == 0) cs.n_heavy = n_all;
    if (tid < kMaxHeavy) {
        cs.hmin[tid] = ~0ull;
        cs.hmax[tid] = 0ull;
        cs.hcnt[tid] = 0;
    }
#pragma unroll
    for (int k = 0, h = id; k < kPer; ++k) {
        const int c = first[k + 1] - first[k];
        if (first[k] >= m || c <= least) continue;
        cs.hc[h] = c;
        cs.hk[h] = b0 + k;
        cs.hrank[h] = first[k];
        base[b0 + k] |= static_cast<int>(0x80000000u);
        cur[b0 + k] = h++;
    }
    __syncthreads();

    const Buckets bo = make_buckets(from_int(cs.all[4]), from_int(cs.all[5]));
    const Buckets bd = make_buckets(from_int(cs.all[7]), from_int(cs.all[6]));
    constexpr int kStep = 4, kRows = kStep * kW;   // rows of 512 positions at a time
    static_assert(kRows == 64, "two rows per lane");
    // the overfull bucket of position i, or -1; its side and severity key
    auto heavy_at = [&](int i, uint32_t mi, double bi, int& x, uint64_t& key) {
        const uint64_t ki = ordered(bi);
        x = i < hi ? side_of(mi, bi, ki, i, a, ktau) : 2;
        if (x == 2) return -1;
        key = x ? ~ki : ki;
        const int k = x * kBk + bucket_of(narrow(static_cast<uint64_t>(__double_as_longlong(bi))),
                                          x ? bd : bo);
        return base[k] < 0 ? cur[k] : -1;
    };

    // 2. one value each?  And how many this slice holds
#pragma unroll 1
    for (int c0 = lo; c0 < hi; c0 += kT * kStep) {
        uint32_t mv[kStep];
        double bv[kStep];
        load_step<kStep>(S0, b, c0, hi, mv, bv);
        int mixed = 0;
#pragma unroll
        for (int j = 0; j < kStep; ++j) {
            int x;
            uint64_t key = 0;
            const int h = heavy_at(c0 + j * kT + tid, mv[j], bv[j], x, key);
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, h);
            if (h < 0) continue;
            volatile uint64_t* mn = &cs.hmin[h];
            volatile uint64_t* mx = &cs.hmax[h];
            if (lane == __ffs(peers) - 1) atomicAdd(&cs.hcnt[h], __popc(peers));
            if (key < *mn) atomicMin(reinterpret_cast<unsigned long long*>(&cs.hmin[h]), key);
            if (key > *mx) atomicMax(reinterpret_cast<unsigned long long*>(&cs.hmax[h]), key);
            mixed |= *mn != *mx && cs.hc[h] > limit;
        }
        if (__syncthreads_or(mixed)) break;   // the verdict below sees it in every CTA
    }
    cluster_sync<C>();
    int mixed = 0;
    if (tid < n_all) {
        uint64_t mn = ~0ull, mx = 0ull;
        int before_me = cs.hrank[tid];
        for (int q = 0; q < C; ++q) {
            mn = min(mn, peer<C>(cs.hmin + tid, q));
            mx = max(mx, peer<C>(cs.hmax + tid, q));
            if (q < r) before_me += peer<C>(cs.hcnt + tid, q);
        }
        mixed = mn != mx && cs.hc[tid] > limit;
        if (mn != mx) cs.hc[tid] = 0;                 // counted through after all
        cs.hnext[tid] = before_me;
    }
    if (__syncthreads_or(mixed)) return false;        // alike in every CTA

    // the ones of one value leave the places
    int items = 0, top = 0, last = 0, before_me, all;
#pragma unroll
    for (int k = 0, h = id; k < kPer; ++k) {
        const int c = first[k + 1] - first[k];
        if (first[k] >= m) continue;
        if (c > least && cs.hc[h++] > 0) items += c;
        else top = max(top, c);
    }
    scan2n(s, items, 0, before_me, unused, all, unused);
    if (tid == kT / 2) s.flag = before_me;            // what the orphans' side holds
    if (tid < 3) cs.tot[tid] = 0;
    __syncthreads();
    if (side) before_me -= s.flag;
#pragma unroll
    for (int k = 0, h = id; k < kPer; ++k) {
        const int c = first[k + 1] - first[k], place = first[k] - before_me;
        const bool candidate = first[k] < m && c > least;
        if (candidate && cs.hc[h] > 0) {
            base[b0 + k] = place | static_cast<int>(0x80000000u);
            before_me += c;
        } else {
            base[b0 + k] = cur[b0 + k] = place;
            if (first[k] < m) last = max(last, place + c);
        }
        h += candidate;
    }
    atomicMax(&cs.tot[0], top);
    atomicMax(&cs.tot[1 + side], last);
    __syncthreads();

    // 3. their ranks in position order
    int* swaps = a.out_swaps + static_cast<int64_t>(u) * 2 * (a.N / 2);
    uint8_t* S1 = a.out_mask + off;
#pragma unroll 1
    for (int c0 = lo; c0 < hi; c0 += kT * kStep) {
        for (int i = tid; i < n_all * kRows; i += kT) rows[i] = 0;
        __syncthreads();
        int code[kStep];   // bucket, rank within the warp's row, side; or -1
        uint32_t mv[kStep];
        double bv[kStep];
        load_step<kStep>(S0, b, c0, hi, mv, bv);
#pragma unroll
        for (int j = 0; j < kStep; ++j) {
            int x;
            uint64_t key;
            const int h = heavy_at(c0 + j * kT + tid, mv[j], bv[j], x, key);
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, h);
            const int rk = __popc(peers & ((1u << lane) - 1u));
            if (h >= 0 && rk == 0) rows[h * kRows + j * kW + wid] = __popc(peers);
            code[j] = h < 0 ? -1 : h << 6 | rk << 1 | x;
        }
        __syncthreads();
        for (int h = wid; h < n_all; h += kW) {
            const int at = h * kRows + 2 * lane;
            const int r0 = rows[at], r1 = rows[at + 1], next = cs.hnext[h];
            int incl = r0 + r1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += y;
            }
            rows[at] = next + incl - r0 - r1;
            rows[at + 1] = next + incl - r1;
            if (lane == 31) cs.hnext[h] = next + incl;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kStep; ++j) {
            if (code[j] < 0) continue;
            const int h = code[j] >> 6, x = code[j] & 1, i = c0 + j * kT + tid;
            const int rank = rows[h * kRows + j * kW + wid] + ((code[j] >> 1) & 31);
            if (rank < m) {
                swaps[2 * rank + (x ? 0 : 1)] = i;
                S1[i] = x ? 0 : 1;
            }
        }
        __syncthreads();
    }
    cluster_sync<C>();   // the rows are free for the peers' items
    return true;
}

// The end of the bucket path: the items in play go to their buckets' owners, and every owner
// writes the swaps of its own.  kMany: window by window of C * share places, beside overfull
// buckets that have none.
template <int C, bool kDedup, bool kMany>
__device__ __forceinline__ void place_and_rank(Shared& s, ClusterShared& cs, uint64_t* sk, int* si,
                                               const RepairArgs& a, int u, int r, int m, int share,
                                               const int (&end)[2], const Buckets& bo,
                                               const Buckets& bd, const uint8_t* S0,
                                               const double* b, uint8_t* S1, int lo, int hi,
                                               uint64_t ktau)
{
    constexpr int kP = C == 1 && !kMany ? 8 : 4;   // positions per thread and step
    const int tid = threadIdx.x;
    int* base = &s.warp_cnt[0][0];
    int* cur = base + 2 * kBk;
    constexpr int kPlace = kMany ? 0x7FFFFFFF : -1;   // overfull buckets have the top bit
    constexpr bool kWrap = C > 1 || kMany;            // a CTA's places need not start at 0
    auto slot = [](int g) { return kWrap ? g % kCap : g; };
    auto bucket = [&](int x, uint64_t bits) { return bucket_of(narrow(bits), x ? bd : bo); };
    // the place of a bucket in the window, or beyond its end (an overfull one always)
    auto in_window = [&](int x, int place, int w0) {
        if constexpr (!kMany) return place < (kDedup && x ? cs.all[1] : m);
        return static_cast<unsigned>(place) - static_cast<unsigned>(w0) <
               static_cast<unsigned>(max(0, min(end[x] - w0, C * share)));
    };

    for (int w0 = 0;; w0 += C * share) {
        // the window's items to their buckets' owners
        for (int c0 = lo; c0 < hi; c0 += kT * kP) {
            uint32_t mv[kP];
            double bv[kP];
            load_step<kP>(S0, b, c0, hi, mv, bv);
#pragma unroll
            for (int j = 0; j < kP; ++j) {
                const int i = c0 + j * kT + tid;
                const uint64_t ki = ordered(bv[j]);
                const int x = i < hi ? side_of(mv[j], bv[j], ki, i, a, ktau) : 2;
                if (x == 2) continue;
                const int k = x * kBk + bucket(x, static_cast<uint64_t>(__double_as_longlong(bv[j])));
                if (!in_window(x, base[k], w0)) continue;
                if constexpr (C == 1) {
                    const int at = x * kCap + slot(atomicAdd(&cur[k], 1));
                    sk[at] = x ? ~ki : ki;
                    si[at] = i;
                } else {
                    const int t = (base[k] - w0) / share;
                    const int at = x * kCap + slot(peer_add(cur + k, t, 1));
                    peer_store(sk + at, t, x ? ~ki : ki);
                    peer_store(si + at, t, i);
                }
            }
        }
        // this CTA's own items: the places from its first bucket's to its last one's end
        int g0[2] = {0, 0}, g1[2] = {end[0], end[1]};
        if constexpr (C > 1 || kMany) {
#pragma unroll 1
            for (int k = threadIdx.x; k < 2 * kBk; k += kT) {
                const int x = k / kBk, bk = base[k];
                const int ek = (k + 1) % kBk ? base[k + 1] & kPlace : kMany ? end[x] : cs.all[x];
                if (in_window(x, bk, w0) && ek > bk && (C == 1 || (bk - w0) / share == r)) {
                    atomicMin(&cs.tot[4 + x], bk);
                    atomicMax(x ? &s.sel_before : &s.sel_digit, ek);
                }
            }
        }
        cluster_sync<C>();
        if constexpr (C > 1 || kMany) {
            g0[0] = cs.tot[4];
            g0[1] = cs.tot[5];
            g1[0] = s.sel_digit;
            g1[1] = s.sel_before;
        }
        // the rank of the item at place g of side x
        auto rank_of = [&](int x, int g) {
            const uint64_t key = sk[x * kCap + slot(g)];
            const int pos = si[x * kCap + slot(g)];
            const int k = bucket(x, bits_of_key(key, x));
            const int from_g = base[x * kBk + k];
            const int to_g =
                k + 1 < kBk ? base[x * kBk + k + 1] & kPlace : kMany ? end[x] : cs.all[x];
            int rank = from_g;
            if constexpr (kMany)   // the overfull buckets before it have ranks but no places
                for (int h = 0; h < cs.n_heavy; ++h)
                    rank += cs.hk[h] / kBk == x && cs.hk[h] < x * kBk + k ? cs.hc[h] : 0;
            int at = x * kCap + slot(from_g);
#pragma unroll 4
            for (int n = to_g - from_g; n > 0; --n) {
                rank += before(sk[at], si[at], key, pos) ? 1 : 0;
                ++at;
                if (kWrap && at == (x + 1) * kCap) at = x * kCap;
            }
            return rank;
        };
        if constexpr (kDedup) {
            int rank[2][kCap / kT];
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int j = 0; j < kCap / kT; ++j) {
                    const int g = tid + j * kT;
                    rank[x][j] = g < end[x] ? rank_of(x, g) : -1;
                }
            dedup_swap(s, sk, si, bd, a, u, end, cs.all[0], ktau, rank);
            return;
        }
        int* swaps = a.out_swaps + static_cast<int64_t>(u) * 2 * (a.N / 2);
#pragma unroll
        for (int x = 0; x < 2; ++x)
            for (int g = g0[x] + tid; g < g1[x]; g += kT) {
                const int rank = rank_of(x, g), pos = si[x * kCap + slot(g)];
                if (rank < m) {
                    swaps[2 * rank + (x ? 0 : 1)] = pos;
                    S1[pos] = x ? 0 : 1;
                }
            }
        if (!kMany || w0 + C * share >= max(end[0], end[1])) break;
        cluster_sync<C>();   // the window's items and its ends have been read
        if (tid < 2) cs.tot[4 + tid] = 1 << 30;
        if (tid == 0) s.sel_digit = s.sel_before = 0;
        __syncthreads();
    }
    if (r == 0 && tid == 0) {
        a.out_nswaps[u] = m;
        if (a.out_status) a.out_status[u] = 0;
    }
}

// The rest of the bucket path for a unit with overfull buckets or with lists too long for one
// window.  A function by itself, so that the usual path keeps its registers.
template <int C>
__device__ __noinline__ bool rank_many(Shared& s, ClusterShared& cs, const RepairArgs& a, int u,
                                       int r)
{
    extern __shared__ __align__(16) uint32_t dyn[];
    uint64_t* sk = reinterpret_cast<uint64_t*>(dyn);
    int* si = reinterpret_cast<int*>(sk + 2 * kCap);
    const int m = min(cs.all[0], cs.all[1]);
    if (cs.tot[0] > max_bucket(a.N) && !rank_heavy<C>(s, cs, reinterpret_cast<int*>(sk), a, u, r, m))
        return false;
    // as few windows as hold all places, and these dealt out evenly
    const int end[2] = {cs.tot[1], cs.tot[2]}, places = max(end[0], end[1]);
    const int most = C * (kCap - cs.tot[0]), wins = max(1, (places + most - 1) / most);
    const int share = max(1, (places + C * wins - 1) / (C * wins));
    const Buckets bo = make_buckets(from_int(cs.all[4]), from_int(cs.all[5]));
    const Buckets bd = make_buckets(from_int(cs.all[7]), from_int(cs.all[6]));
    const int64_t off = static_cast<int64_t>(u) * a.N;
    const int slice = slice_len(a.N, C);
    const int lo = min(a.N, r * slice), hi = min(a.N, lo + slice);
    place_and_rank<C, false, true>(s, cs, sk, si, a, u, r, m, share, end, bo, bd, a.mask + off,
                                   a.b + off, a.out_mask + off, lo, hi, ordered(a.tau));
    return true;
}

// Runs the unit by buckets; every thread of the cluster calls it.  Not kDone (and, apart from
// S1 = S0, nothing written) where the unit is left to the general path.  kDedup (C = 1): every
// donor is in play, not only the m most severe, and dedup_swap ends the unit.
template <int C, bool kDedup = false>
__device__ Attempt select_by_buckets(Shared& s, ClusterShared& cs, uint64_t* sk, int* si,
                                  const RepairArgs& a, int u, int r)
{
    const int64_t off = static_cast<int64_t>(u) * a.N;
    const uint8_t* S0 = a.mask + off;
    const double* b = a.b + off;
    uint8_t* S1 = a.out_mask + off;
    const int slice = slice_len(a.N, C);
    const int lo = min(a.N, r * slice), hi = min(a.N, lo + slice);
    const uint64_t ktau = ordered(a.tau);
    constexpr int kP = C == 1 ? 8 : 4;   // positions per thread and step
    const int tid = threadIdx.x, lane = tid & 31;
    int* base = &s.warp_cnt[0][0];   // [2][kBk] first rank of each bucket
    int* cur = base + 2 * kBk;       // [2][kBk] counts, then the next free place
    static_assert(sizeof(s.warp_cnt) == 4 * kBk * sizeof(int), "bucket arrays fill warp_cnt");

    // 1. counts and ranges
    int bad = 0, cnt = 0, n[2] = {0, 0};
    int mn[2] = {0x7FFFFFFF, 0x7FFFFFFF}, mx[2] = {-0x7FFFFFFF - 1, -0x7FFFFFFF - 1};
    for (int c0 = lo; c0 < hi; c0 += kT * kP) {
        uint32_t mv[kP];
        double bv[kP];
        load_step<kP>(S0, b, c0, hi, mv, bv);
#pragma unroll
        for (int j = 0; j < kP; ++j) {
            const int i = c0 + j * kT + tid;
            if (i >= hi) continue;
            S1[i] = static_cast<uint8_t>(mv[j]);
            bad |= mv[j] > 1u;
            cnt += mv[j] != 0u;
            const int x = side_of(mv[j], bv[j], ordered(bv[j]), i, a, ktau);
            const int f = as_int(narrow(static_cast<uint64_t>(__double_as_longlong(bv[j]))));
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                n[y] += x == y;
                mn[y] = x == y ? min(mn[y], f) : mn[y];
                mx[y] = x == y ? max(mx[y], f) : mx[y];
            }
        }
    }
    if (tid < 8) cs.cnt[tid] = tid < 4 ? 0 : (tid & 1) ? -0x7FFFFFFF - 1 : 0x7FFFFFFF;
    for (int i = tid; i < 2 * kBk; i += kT) cur[i] = 0;
    __syncthreads();
    bad = __reduce_or_sync(0xFFFFFFFFu, bad);
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
#pragma unroll
    for (int y = 0; y < 2; ++y) {
        n[y] = __reduce_add_sync(0xFFFFFFFFu, n[y]);
        mn[y] = __reduce_min_sync(0xFFFFFFFFu, mn[y]);
        mx[y] = __reduce_max_sync(0xFFFFFFFFu, mx[y]);
    }
    if (lane == 0) {
        atomicAdd(&cs.cnt[0], n[0]);
        atomicAdd(&cs.cnt[1], n[1]);
        atomicAdd(&cs.cnt[2], cnt);
        atomicOr(&cs.cnt[3], bad);
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            atomicMin(&cs.cnt[4 + 2 * y], mn[y]);
            atomicMax(&cs.cnt[5 + 2 * y], mx[y]);
        }
    }
    cluster_sync<C>();
    if (tid < 8) {   // totals and ranges over the cluster, identical in every CTA
        const bool mini = tid == 4 || tid == 6, maxi = tid == 5 || tid == 7;
        int v = mini ? 0x7FFFFFFF : maxi ? -0x7FFFFFFF - 1 : 0;
        for (int q = 0; q < C; ++q) {
            const int x = peer<C>(cs.cnt + tid, q);   // cnt[4], then ends[4]
            v = mini ? min(v, x) : maxi ? max(v, x) : tid == 3 ? v | x : v + x;
        }
        cs.all[tid] = v;
    }
    __syncthreads();
    const int* tot = cs.all;
    const int* ends = cs.all + 4;
    int status = 0;
    if (tot[3]) status = 1;                                  // TWINKV_ERR_INVALID_ARG
    else if (a.budget && a.budget[u] != tot[2]) status = 3;  // TWINKV_ERR_BUDGET
    const int m = status ? 0 : min(tot[0], tot[1]);
    if (m == 0) {
        cluster_sync<C>();   // every CTA has read the counts before any CTA exits
        if (r == 0 && tid == 0) {
            a.out_nswaps[u] = status ? -1 : 0;
            if (a.out_status) a.out_status[u] = status;
        }
        return kDone;
    }
    // ranks in play per side; the dedup variant needs all of them at once
    const int lim_o = m, lim_d = kDedup ? tot[1] : m;
    if (kDedup && max(lim_o, lim_d) > kCap) return kCounted;
    // side x's bucket: orphans from the smallest b up, donors from the largest down
    const Buckets bo = make_buckets(from_int(ends[0]), from_int(ends[1]));
    const Buckets bd = make_buckets(from_int(ends[3]), from_int(ends[2]));
    auto bucket = [&](int x, uint64_t bits) {
        return bucket_of(narrow(bits), x ? bd : bo);
    };

    // 2. histogram, summed over the cluster, and its prefix sums
    for (int c0 = lo; c0 < hi; c0 += kT * kP) {
        uint32_t mv[kP];
        double bv[kP];
        load_step<kP>(S0, b, c0, hi, mv, bv);
#pragma unroll
        for (int j = 0; j < kP; ++j) {
            const int i = c0 + j * kT + tid;
            const int x = i < hi ? side_of(mv[j], bv[j], ordered(bv[j]), i, a, ktau) : 2;
            if (x < 2)
                atomicAdd(&cur[x * kBk + bucket(x, static_cast<uint64_t>(
                                                       __double_as_longlong(bv[j])))],
                          1);
        }
    }
    // maxima, then minima (beyond every place, yet far from overflow for a CTA without items)
    if (tid < 8) cs.tot[tid] = (tid & 4) ? 1 << 30 : 0;
    if (tid == 0) s.sel_digit = s.sel_before = cs.n_heavy = 0;
    cluster_sync<C>();
    constexpr int kPer = 2 * kBk / kT;   // buckets per thread; side 0: the lower half of the block
    static_assert(kPer * kT == 2 * kBk && kW % 2 == 0, "whole warps per side");
    const int b0 = tid * kPer, side = b0 / kBk;
    int c[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        c[k] = 0;
#pragma unroll 1
        for (int q = 0; q < C; ++q) c[k] += peer<C>(cur + b0 + k, q);
        sum += c[k];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s.wsum[0][tid >> 5] = incl;
    cluster_sync<C>();   // (every CTA has read this one's counts)
    int run = incl - sum;
    for (int w = side * (kW / 2); w < (tid >> 5); ++w) run += s.wsum[0][w];
    int full = 0, last = 0;   // the fullest bucket in play, and the end of the last one
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        base[b0 + k] = run;
        cur[b0 + k] = run;
        if (run < (side ? lim_d : lim_o)) {
            full = max(full, c[k]);
            last = max(last, run + c[k]);
        }
        run += c[k];
    }
    atomicMax(&cs.tot[0], full);
    atomicMax(&cs.tot[1 + side], last);
    cluster_sync<C>();
    full = cs.tot[0];
    const int end[2] = {cs.tot[1], cs.tot[2]};   // items in play per side
    const int share = (max(end[0], end[1]) + C - 1) / C;
    if (full > max_bucket(a.N) || share + full > kCap) return kRanked;   // alike in every CTA
    // 3. (one window)
    place_and_rank<C, kDedup, false>(s, cs, sk, si, a, u, r, m, share, end, bo, bd, S0, b, S1, lo,
                                     hi, ktau);
    return kDone;
}

// The end of the dedup variant's bucket path: the walk over the donors in severity order as
// rounds over all of them.  A donor conflicts with its twin, and with the donors whose twin
// it is; it is evicted unless a more severe one that it conflicts with is.  In each round an
// edge (donor, its twin) whose more severe end is evicted rejects the other end, one whose
// more severe end is undecided holds the other end back, and every undecided donor that
// nothing holds back is evicted: the same set as the walk's.  Twins are mostly mutual, so a
// few rounds decide all; a chain longer than kRounds is finished by one thread in rank
// order.  (The walk by one thread took about half of the kernel's 78 us at 144 units of 8192.)
// rank: the ranks of the thread's items, places tid + j kT.  The keys at sk are no longer
// needed: their memory takes the lists by rank.
constexpr int kRounds = 64;

__device__ void dedup_swap(Shared& s, uint64_t* sk, int* si, const Buckets& bd,
                           const RepairArgs& a, int u, const int* end, int n_o, uint64_t ktau,
                           const int (&rank)[2][kCap / kT])
{
    const int tid = threadIdx.x, N = a.N, n_d = end[1];
    const int64_t off = static_cast<int64_t>(u) * N;
    const int* base = &s.warp_cnt[0][0] + kBk;   // the donors' buckets
    uint8_t* state = reinterpret_cast<uint8_t*>(&s.warp_cnt[0][0] + 2 * kBk);   // by rank
    uint8_t* held = state + kCap;
    static_assert(2 * kCap <= 2 * kBk * 4, "state and held take the place of the cursors");
    int* orph = reinterpret_cast<int*>(sk);   // [kCap] orphans by rank
    int* don = orph + kCap;                   // [kCap] donors by rank
    int* rank_at = don + kCap;                // [kCap] rank of the donor at each place
    int* twin = rank_at + kCap;               // [kCap] by rank: the rank of the donor's twin
    __syncthreads();                          // every rank has been counted
#pragma unroll
    for (int j = 0; j < kCap / kT; ++j) {
        const int g = tid + j * kT;
        if (rank[0][j] >= 0) orph[rank[0][j]] = si[g];
        if (rank[1][j] >= 0) {
            don[rank[1][j]] = si[kCap + g];
            rank_at[g] = rank[1][j];
        }
    }
    for (int k = tid; k < n_d; k += kT) state[k] = 0;   // 1: evicted, 2: rejected
    __syncthreads();
    for (int k = tid; k < n_d; k += kT) {
        const int t = a.twin[off + don[k]];
        int r = -1;
        if (t >= 0 && t < N) {
            const double bt = a.b[off + t];
            if (side_of(a.mask[off + t], bt, ordered(bt), t, a, ktau) == 1) {
                const int bk = bucket_of(narrow(static_cast<uint64_t>(__double_as_longlong(bt))), bd);
                const int to = bk + 1 < kBk ? base[bk + 1] : n_d;
                for (int g = base[bk]; g < to; ++g)
                    if (si[kCap + g] == t) r = rank_at[g];
            }
        }
        twin[k] = r == k ? -1 : r;
    }
    __syncthreads();
    int undecided = 1;
    for (int round = 0; round < kRounds && undecided; ++round) {
        for (int k = tid; k < n_d; k += kT) held[k] = 0;
        __syncthreads();
        for (int k = tid; k < n_d; k += kT) {
            const int t = twin[k];
            if (t < 0) continue;
            const int first = state[min(k, t)];
            if (first == 1) state[max(k, t)] = 2;
            else if (first == 0) held[max(k, t)] = 1;
        }
        __syncthreads();
        int left = 0;
        for (int k = tid; k < n_d; k += kT)
            if (state[k] == 0) {
                if (held[k]) left = 1;
                else state[k] = 1;
            }
        undecided = __syncthreads_or(left);
    }
    if (undecided) {
        if (tid == 0)
            for (int k = 0; k < n_d; ++k) {
                const int t = twin[k];
                if (state[k] == 0) state[k] = t >= 0 && t < k && state[t] == 1 ? 2 : 1;
                if (state[k] == 1 && t > k) state[t] = 2;
            }
        __syncthreads();
    }
    // the first n_o evictions in rank order
    int* out = rank_at;
    int total = 0;
    for (int c0 = 0; c0 < n_d; c0 += kT) {
        const int k = c0 + tid;
        const int f = k < n_d && state[k] == 1;
        int p, q, to, tq;
        scan2(s, f, 0, p, q, to, tq);
        if (f) out[total + p] = don[k];
        total += to;
    }
    __syncthreads();
    const int m = min(total, n_o);
    uint8_t* S1 = a.out_mask + off;
    int* swaps = a.out_swaps + static_cast<int64_t>(u) * 2 * (N / 2);
    for (int k = tid; k < m; k += kT) {
        swaps[2 * k] = out[k];
        swaps[2 * k + 1] = orph[k];
        S1[out[k]] = 0;
        S1[orph[k]] = 1;
    }
    if (tid == 0) {
        a.out_nswaps[u] = m;
        if (a.out_status) a.out_status[u] = 0;
    }
}

template <int C>
__global__ void __launch_bounds__(kT, 2) select_kernel(const RepairArgs a)
{
    __shared__ Shared s;
    __shared__ ClusterShared cs;
    extern __shared__ __align__(16) uint32_t dyn[];
    uint64_t* sk_o = reinterpret_cast<uint64_t*>(dyn);   // [kChunk] orphans' keys
    uint64_t* sk_d = sk_o + kChunk;                      // [kChunk] donors' keys
    int* si_o = reinterpret_cast<int*>(sk_d + kChunk);   // [kChunk] positions
    int* si_d = si_o + kChunk;

    int tid = threadIdx.x;
    int r = 0;
    if constexpr (C > 1) r = static_cast<int>(cg::this_cluster().block_rank());
    int u = static_cast<int>(blockIdx.x / C);
    wait_for_previous();
    if (a.N <= kBucketMaxN) {
        int* si = reinterpret_cast<int*>(sk_o + 2 * kCap);
        if (select_by_buckets<C>(s, cs, sk_o, si, a, u, r) == kDone) return;
        forget(u);   // nothing computed from them stays in registers over what follows
        forget(r);
        if (rank_many<C>(s, cs, a, u, r)) return;
        forget(u);
        forget(r);
        forget(tid);
    }
    const int lane = tid & 31;
    cluster_sync<C>();   // what the attempt left in shared memory is free

    const int N = a.N;
    const int64_t off = static_cast<int64_t>(u) * N;
    const uint8_t* S0 = a.mask + off;
    const double* b = a.b + off;
    uint8_t* S1 = a.out_mask + off;
    int* swaps = a.out_swaps + static_cast<int64_t>(u) * 2 * (N / 2);
    uint64_t* K0 = a.keys0 + off;
    int* I0 = a.idx0 + off;
    uint64_t* K1 = a.keys1 + off;
    int* I1 = a.idx1 + off;
    const int S = slice_len(N, C);
    const int lo = min(N, r * S), hi = min(N, lo + S);
    const uint64_t ktau = ordered(a.tau);

    // A. S1 = S0, counts, and the slice's lists (orphans forward from lo, donors
    // backward from hi: donor k in position order sits at hi - 1 - k).  A thread takes
    // kEA consecutive positions: one 8-byte mask load and four 16-byte b loads when
    // every unit's rows are aligned for them (N a multiple of 8, aligned base
    // pointers), else one at a time.
    int bad = 0, cnt = 0, my_o = 0, my_d = 0;
    const bool vec = (N % kEA) == 0 && (reinterpret_cast<uintptr_t>(a.mask) & 7) == 0 &&
                     (reinterpret_cast<uintptr_t>(a.out_mask) & 7) == 0 &&
                     (reinterpret_cast<uintptr_t>(a.b) & 15) == 0;
    for (int c0 = lo; c0 < hi; c0 += kT * kEA) {
        const int i0 = c0 + tid * kEA;
        uint32_t mv[kEA];
        double bv[kEA];
        if (vec && i0 + kEA <= hi) {
            const uint2 m8 = *reinterpret_cast<const uint2*>(S0 + i0);
            *reinterpret_cast<uint2*>(S1 + i0) = m8;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mv[j] = (m8.x >> (8 * j)) & 255u;
                mv[4 + j] = (m8.y >> (8 * j)) & 255u;
            }
            const double2* b2 = reinterpret_cast<const double2*>(b + i0);
#pragma unroll
            for (int j = 0; j < kEA / 2; ++j) {
                const double2 t = b2[j];
                bv[2 * j] = t.x;
                bv[2 * j + 1] = t.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < kEA; ++j) {
                const int i = i0 + j;
                mv[j] = 0u;
                bv[j] = 0.0;
                if (i < hi) {
                    mv[j] = S0[i];
                    bv[j] = b[i];
                    S1[i] = static_cast<uint8_t>(mv[j]);
                }
            }
        }
        // b < tau and b >= tau decided on the order-preserving keys (a NaN b is
        // neither an orphan nor a donor, as in fp64 comparisons)
        int fo[kEA], fd[kEA], co = 0, cd = 0;
        uint64_t kv[kEA];
#pragma unroll
        for (int j = 0; j < kEA; ++j) {
            const int i = i0 + j;
            const bool in = i < hi && !is_nan_bits(bv[j]);
            kv[j] = ordered(bv[j]);
            bad |= mv[j] > 1u;
            cnt += mv[j] != 0u;
            const bool prot = i < a.n_sink || i >= N - a.n_recent;
            fo[j] = in && mv[j] == 0u && kv[j] < ktau;
            fd[j] = in && mv[j] != 0u && !prot && kv[j] >= ktau;
            co += fo[j];
            cd += fd[j];
        }
        int po, pd, to, td;
        scan2n(s, co, cd, po, pd, to, td);
#pragma unroll
        for (int j = 0; j < kEA; ++j) {
            const int i = i0 + j;
            if (fo[j]) {
                K0[lo + my_o + po] = kv[j];
                I0[lo + my_o + po] = i;
                ++po;
            }
            if (fd[j]) {
                K0[hi - 1 - (my_d + pd)] = ~kv[j];
                I0[hi - 1 - (my_d + pd)] = i;
                ++pd;
            }
        }
        my_o += to;
        my_d += td;
    }
    if (tid < 4) s.red[tid] = 0;
    __syncthreads();
    bad = __reduce_or_sync(0xFFFFFFFFu, bad);
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    if (lane == 0) {
        atomicOr(&s.red[0], bad);
        atomicAdd(&s.red[1], cnt);
    }
    __syncthreads();
    if (tid == 0) {
        cs.cnt[0] = my_o;
        cs.cnt[1] = my_d;
        cs.cnt[2] = s.red[1];
        cs.cnt[3] = s.red[0];
    }
    cluster_sync<C>();

    // B. totals, offsets, status and m (identical in every CTA of the cluster)
    if (tid == 0) {
        int n_o = 0, n_d = 0, tc = 0, tb = 0, bo = 0, bd = 0;
        for (int q = 0; q < C; ++q) {
            if (q == r) {
                bo = n_o;
                bd = n_d;
            }
            n_o += peer<C>(cs.cnt, q);
            n_d += peer<C>(cs.cnt + 1, q);
            tc += peer<C>(cs.cnt + 2, q);
            tb |= peer<C>(cs.cnt + 3, q);
        }
        int status = 0;
        if (tb) status = 1;                                  // TWINKV_ERR_INVALID_ARG
        else if (a.budget && a.budget[u] != tc) status = 3;  // TWINKV_ERR_BUDGET
        cs.tot[0] = n_o;
        cs.tot[1] = n_d;
        cs.tot[2] = bo;
        cs.tot[3] = bd;
        cs.tot[4] = status;
        cs.tot[5] = status ? 0 : min(n_o, n_d);
    }
    __syncthreads();
    const int n_o = cs.tot[0], n_d = cs.tot[1], bo = cs.tot[2], bd = cs.tot[3];
    const int status = cs.tot[4], m = cs.tot[5];
    if (status != 0 || m == 0) {
        cluster_sync<C>();   // every CTA has read the counts before any CTA exits
        if (r == 0 && tid == 0) {
            a.out_nswaps[u] = status ? -1 : 0;
            if (a.out_status) a.out_status[u] = status;
        }
        return;
    }

    // The side with more than m items is cut (at most one: m = min(n_o, n_d)); the
    // other is taken whole.  Item k (position order) of this CTA's list on side x:
    auto item_key = [&](int x, int k) { return x == 0 ? K0[lo + k] : K0[hi - 1 - k]; };
    auto item_pos = [&](int x, int k) { return x == 0 ? I0[lo + k] : I0[hi - 1 - k]; };
    const int half = N / 2;
    for (int x = 0; x < 2; ++x) {
        const int mine = x == 0 ? my_o : my_d;
        const int my_before = x == 0 ? bo : bd;
        const int dst0 = x == 0 ? 0 : half;
        if ((x == 0 ? n_o : n_d) == m) {
            for (int k = tid; k < mine; k += kT) {
                K1[dst0 + my_before + k] = item_key(x, k);
                I1[dst0 + my_before + k] = item_pos(x, k);
            }
            continue;
        }
        // radix select of the m smallest keys over the cluster, a byte at a time from
        // the top, stopping once the boundary bucket is taken whole
        uint64_t prefix = 0, pmask = 0;
        int need = m;
        bool whole = false;
        int pass = 0;
        int below = 0, at_cut = 0;   // this CTA's items below the cut and at it, per digit
        for (int shift = 56; shift >= 0 && !whole; shift -= 8, ++pass) {
            int* h = cs.hist[pass & 1];
            if (tid < 256) h[tid] = 0;
            __syncthreads();
            for (int c0 = 0; c0 < mine; c0 += kT * kH) {
                int dg[kH];
#pragma unroll
                for (int e = 0; e < kH; ++e) {
                    const int k = c0 + e * kT + tid;
                    dg[e] = 256;
                    if (k < mine) {
                        const uint64_t key = item_key(x, k);
                        if ((key & pmask) == prefix) dg[e] = static_cast<int>((key >> shift) & 255);
                    }
                }
#pragma unroll
                for (int e = 0; e < kH; ++e) {
                    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, dg[e]);
                    if (dg[e] < 256 && lane == __ffs(peers) - 1) atomicAdd(&h[dg[e]], __popc(peers));
                }
            }
            cluster_sync<C>();   // every CTA's histogram of this pass is complete
            int own = 0;
            if (tid < 256) {
                int t = 0;
                for (int q = 0; q < C; ++q) t += peer<C>(h + tid, q);
                s.base[tid] = t;
                own = h[tid];
            }
            __syncthreads();
            if (tid < 32) digit_cut(s.base, need, s.sel_digit, s.sel_before, s.sel_count);
            __syncthreads();
            need -= s.sel_before;
            prefix |= static_cast<uint64_t>(s.sel_digit) << shift;
            pmask |= 255ull << shift;
            whole = s.sel_count == need;
            // digit tid of this CTA's own histogram: below the selected digit, or at it
            below += tid < s.sel_digit ? own : 0;
            at_cut = tid == s.sel_digit ? own : 0;
            __syncthreads();
        }
        // ordered compaction: every item below the cut (and at it when `whole`), then
        // the first `need` items at the cut in position order over the cluster
        int nl = below + (whole ? at_cut : 0), ne = whole ? 0 : at_cut;
        if (tid < 2) s.red[tid] = 0;
        __syncthreads();
        nl = __reduce_add_sync(0xFFFFFFFFu, nl);
        ne = __reduce_add_sync(0xFFFFFFFFu, ne);
        if (lane == 0) {
            atomicAdd(&s.red[0], nl);
            atomicAdd(&s.red[1], ne);
        }
        __syncthreads();
        if (tid == 0) {
            cs.lcnt[0] = s.red[0];
            cs.lcnt[1] = s.red[1];
        }
        cluster_sync<C>();
        if (tid == 0) {
            int sel_before = 0, eq_before = 0;
            for (int q = 0; q < r; ++q) {
                const int at_cut_q = peer<C>(cs.lcnt + 1, q);
                sel_before += peer<C>(cs.lcnt, q) + max(0, min(at_cut_q, need - eq_before));
                eq_before += at_cut_q;
            }
            cs.tot[6] = sel_before;
            cs.tot[7] = eq_before;
        }
        __syncthreads();
        constexpr int kEB = kEA / 2;   // (kEA would spill beside rank_many's call)
        int base = cs.tot[6], seen_eq = cs.tot[7];
        for (int c0 = 0; c0 < mine; c0 += kT * kEB) {
            // a thread takes kEB consecutive items; fl: below the cut (or at it when
            // `whole`), fe: at the cut
            const int k0 = c0 + tid * kEB;
            uint64_t kk[kEB];
            int pp[kEB];
            uint32_t fl = 0, fe = 0;
#pragma unroll
            for (int j = 0; j < kEB; ++j) {
                kk[j] = 0;
                pp[j] = 0;
                if (k0 + j < mine) {
                    kk[j] = item_key(x, k0 + j);
                    pp[j] = item_pos(x, k0 + j);
                    const uint64_t km = kk[j] & pmask;
                    fl |= static_cast<uint32_t>(km < prefix || (whole && km == prefix)) << j;
                    fe |= static_cast<uint32_t>(!whole && km == prefix) << j;
                }
            }
            int pl, pe, tl, te;
            scan2n(s, __popc(fl), __popc(fe), pl, pe, tl, te);
            const int k_eq = max(0, min(te, need - seen_eq));   // taken at the cut here
#pragma unroll
            for (int j = 0; j < kEB; ++j) {
                const int l = (fl >> j) & 1, e = (fe >> j) & 1;
                if (l || (e && pe < k_eq)) {
                    const int dst = base + pl + min(pe, k_eq);
                    K1[dst0 + dst] = kk[j];
                    I1[dst0 + dst] = pp[j];
                }
                pl += l;
                pe += e;
            }
            base += tl + k_eq;
            seen_eq += te;
        }
    }
    cluster_sync<C>();   // both lists of m items are in keys1/idx1, in position order

    // C. the swap list: m items per side in severity order
    const int q = (m + C - 1) / C;
    if (q <= 2 * kChunk) {
        // Each CTA sorts its share of both lists by (key, position) with a bitonic
        // network over P = 2^k >= max(q, kR) slots per side; padding sorts last.  Thread
        // tt of a side holds the slots [kR*tt, kR*tt + kR) in registers: strides below
        // kR are exchanged inside the thread, strides up to 16*kR between the lanes of
        // a warp by shuffles, and longer ones through shared memory.  Shares of up to
        // kChunk items sort both sides at once (half of the threads and of the buffer
        // each); longer ones (up to 2*kChunk) sort one side after the other, each over
        // all threads and the whole buffer (sk_o..sk_d and si_o..si_d are contiguous).
        const bool both = q <= kChunk;
        const int nside = both ? 2 : 1;
        int P = kR;
        while (P < q) P <<= 1;
        const int TP = P / kR;   // threads per side; threads from nside*TP on hold padding
        const int c_lo = min(m, r * q), c_n = min(m, c_lo + q) - c_lo;
        for (int pass = 0; pass < 3 - nside; ++pass) {
            const int sd = both && tid >= TP;     // the thread's side among those sorted
            const int side = both ? sd : pass;    // 0: orphans, 1: donors
            const int tt = tid - sd * TP;
            const bool live = tid < nside * TP;
            uint64_t* sk = sd ? sk_d : sk_o;
            int* si = sd ? si_d : si_o;
            uint64_t kx[kR];
            int px[kR];
#pragma unroll
            for (int e = 0; e < kR; ++e) {
                const int t = tt * kR + e;
                const bool in = live && t < c_n;
                kx[e] = in ? K1[side * half + c_lo + t] : ~0ull;
                px[e] = in ? I1[side * half + c_lo + t] : 0x7FFFFFFF;
            }
            for (int size = 2; size <= P; size <<= 1) {
                const bool up_t = ((tt * kR) & size) == 0;   // the direction once size >= kR
                if (size >= 64 * kR) {
                    if (live) store_run(sk, si, tt * kR, kx, px);
                    __syncthreads();
                    for (int stride = size >> 1; stride >= 32 * kR; stride >>= 1) {
                        for (int t = tid; t < nside * (P / 2); t += kT) {
                            const int s2 = t >= P / 2;   // pairs of the second side (both)
                            const int ts = s2 ? t - P / 2 : t;
                            uint64_t* k2 = s2 ? sk_d : sk_o;
                            int* i2 = s2 ? si_d : si_o;
                            const int lo2 = 2 * ts - (ts & (stride - 1));
                            const int hi2 = lo2 + stride;
                            uint64_t ka = k2[lo2], kb = k2[hi2];
                            int pa = i2[lo2], pb = i2[hi2];
                            cx(ka, pa, kb, pb, (lo2 & size) == 0);
                            k2[lo2] = ka;
                            k2[hi2] = kb;
                            i2[lo2] = pa;
                            i2[hi2] = pb;
                        }
                        __syncthreads();
                    }
                    if (live) load_run(sk, si, tt * kR, kx, px);
                }
                for (int stride = min(size >> 1, 16 * kR); stride >= kR; stride >>= 1) {
                    const int lm = stride / kR;
                    const bool keep_first = ((tt & lm) == 0) == up_t;
#pragma unroll
                    for (int e = 0; e < kR; ++e) {
                        const uint64_t ok = __shfl_xor_sync(0xFFFFFFFFu, kx[e], lm);
                        const int op = __shfl_xor_sync(0xFFFFFFFFu, px[e], lm);
                        if (before(ok, op, kx[e], px[e]) == keep_first) {
                            kx[e] = ok;
                            px[e] = op;
                        }
                    }
                }
#pragma unroll
                for (int stride = kR / 2; stride > 0; stride >>= 1) {
                    if (stride >= size) continue;
#pragma unroll
                    for (int e = 0; e < kR; ++e)
                        if ((e & stride) == 0)
                            cx(kx[e], px[e], kx[e + stride], px[e + stride],
                               (((tt * kR) | e) & size) == 0);
                }
            }
            if (live) store_run(sk, si, tt * kR, kx, px);
            cluster_sync<C>();   // every share of the sides sorted in this pass is sorted
            for (int t = tid; t < nside * c_n; t += kT) {
                const int s2 = t >= c_n;
                const int ts = s2 ? t - c_n : t;
                const int sdx = both ? s2 : pass;   // 0: orphans, 1: donors
                const uint64_t* k2 = s2 ? sk_d : sk_o;
                const int* i2 = s2 ? si_d : si_o;
                const uint64_t key = k2[ts];
                const int pos = i2[ts];
                // its rank: its place in its own share plus, in every other share, the
                // number of items ordered before it
                int rank = ts;
                for (int qq = 0; qq < C; ++qq)
                    if (qq != r)
                        rank += count_before(k2, i2, qq, P, key, pos);
                swaps[2 * rank + (sdx ? 0 : 1)] = pos;
                S1[pos] = sdx ? 0 : 1;
            }
            cluster_sync<C>();   // every lookup into this CTA's shares is done
        }
    } else {
        // long lists: one CTA per side sorts its m items with the stable radix passes
        // (keys0/idx0, free by now, as the second buffer)
        for (int x = 0; x < 2; ++x) {
            if (r != (C > 1 ? x : 0)) continue;
            const int o = x == 0 ? 0 : half;
            const int cur = radix_sort(s, K1 + o, I1 + o, K0 + o, I0 + o, m);
            const int* ip = (cur == 0 ? I1 : I0) + o;
            for (int k = tid; k < m; k += kT) {
                const int pos = ip[k];
                swaps[2 * k + (x == 0 ? 1 : 0)] = pos;
                S1[pos] = x == 0 ? 1 : 0;
            }
            __syncthreads();
        }
    }
    if (r == 0 && tid == 0) {
        a.out_nswaps[u] = m;
        if (a.out_status) a.out_status[u] = 0;
    }
}

// The dedup variant's counts where no attempt by buckets has left them: cs.all[0..3] (orphans,
// donors, retained positions, whether a mask byte is invalid), and S1 = S0.
__device__ void count_unit(ClusterShared& cs, const RepairArgs& a, int64_t off, uint64_t ktau)
{
    const uint8_t* S0 = a.mask + off;
    const double* b = a.b + off;
    uint8_t* S1 = a.out_mask + off;
    int bad = 0, cnt = 0, no = 0, nd = 0;
    for (int c0 = 0; c0 < a.N; c0 += kT * kE) {
#pragma unroll
        for (int j = 0; j < kE; ++j) {
            const int i = c0 + threadIdx.x * kE + j;
            if (i >= a.N) continue;
            const uint32_t v = S0[i];
            const double bi = b[i];
            S1[i] = static_cast<uint8_t>(v);
            bad |= v > 1u;
            cnt += v != 0u;
            const int x = side_of(v, bi, ordered(bi), i, a, ktau);
            no += x == 0;
            nd += x == 1;
        }
    }
    if (threadIdx.x < 4) cs.all[threadIdx.x] = 0;
    __syncthreads();
    bad = __reduce_or_sync(0xFFFFFFFFu, bad);
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    no = __reduce_add_sync(0xFFFFFFFFu, no);
    nd = __reduce_add_sync(0xFFFFFFFFu, nd);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&cs.all[0], no);
        atomicAdd(&cs.all[1], nd);
        atomicAdd(&cs.all[2], cnt);
        atomicOr(&cs.all[3], bad);
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kT, 2) dedup_kernel(const RepairArgs a)   // 2 blocks/SM
{
    __shared__ Shared s;
    __shared__ ClusterShared cs;
    extern __shared__ __align__(16) uint32_t dyn[];
    wait_for_previous();
    const int u = blockIdx.x;
    Attempt by_buckets = kNone;
    if (a.N <= kBucketMaxN) {
        uint64_t* keys = reinterpret_cast<uint64_t*>(dyn);
        by_buckets = select_by_buckets<1, true>(s, cs, keys, reinterpret_cast<int*>(keys + 2 * kCap),
                                                a, u, 0);
        if (by_buckets == kDone) return;
    }
    __syncthreads();   // what the attempt left in shared memory can be written
    const int N = a.N;
    const int64_t off = static_cast<int64_t>(u) * N;
    const uint8_t* S0 = a.mask + off;
    const double* b = a.b + off;
    uint8_t* S1 = a.out_mask + off;
    int* swaps = a.out_swaps + static_cast<int64_t>(u) * 2 * (N / 2);

    // 1. counts and S1 = S0 (also the answer for a failed unit or m = 0), unless the attempt has
    // done them
    const uint64_t ktau = ordered(a.tau);
    if (by_buckets == kNone) count_unit(cs, a, off, ktau);
    int status = 0;
    if (cs.all[3]) status = 1;                                   // TWINKV_ERR_INVALID_ARG
    else if (a.budget && a.budget[u] != cs.all[2]) status = 3;   // TWINKV_ERR_BUDGET
    const int m = status ? 0 : min(cs.all[0], cs.all[1]);

    if (status != 0 || m == 0) {
        if (threadIdx.x == 0) {
            a.out_nswaps[u] = status ? -1 : 0;
            if (a.out_status) a.out_status[u] = status;
        }
        return;
    }

    // 2-3. classify and compact: orphans at [0, n_o), donors at [n_o, n_o + n_d).  Where the
    // attempt has filled the buckets, of the orphans only those of the buckets that hold the m
    // most severe ones, as no other can be admitted.
    const bool ranked = by_buckets == kRanked;
    const int n_o = ranked ? cs.tot[1] : cs.all[0], n_d = cs.all[1];
    const Buckets bo = make_buckets(from_int(cs.all[4]), from_int(cs.all[5]));
    const int* first_rank = &s.warp_cnt[0][0];
    uint64_t* k0 = a.keys0 + off;
    int* i0 = a.idx0 + off;
    uint64_t* k1 = a.keys1 + off;
    int* i1 = a.idx1 + off;
    int base_o = 0, base_d = n_o;
    for (int c0 = 0; c0 < N; c0 += kT * kE) {
        int fo[kE], fd[kE], co = 0, cd = 0;
        double bv[kE];
#pragma unroll
        for (int j = 0; j < kE; ++j) {
            const int i = c0 + threadIdx.x * kE + j;
            fo[j] = fd[j] = 0;
            bv[j] = 0.0;
            if (i < N) {
                const uint8_t v = S0[i];
                bv[j] = b[i];
                const bool prot = i < a.n_sink || i >= N - a.n_recent;
                const uint64_t kj = ordered(bv[j]);
                const bool num = !is_nan_bits(bv[j]);
                fo[j] = (v == 0 && num && kj < ktau);
                fd[j] = (v != 0 && !prot && num && kj >= ktau);
                if (fo[j] && ranked)
                    fo[j] = first_rank[bucket_of(
                                narrow(static_cast<uint64_t>(__double_as_longlong(bv[j]))), bo)] < m;
            }
            co += fo[j];
            cd += fd[j];
        }
        int po, pd, to, td;
        scan2n(s, co, cd, po, pd, to, td);
#pragma unroll
        for (int j = 0; j < kE; ++j) {
            const int i = c0 + threadIdx.x * kE + j;
            if (fo[j]) {
                k0[base_o + po] = ordered(bv[j]);
                i0[base_o + po] = i;
                ++po;
            }
            if (fd[j]) {
                k0[base_d + pd] = ~ordered(bv[j]);
                i0[base_d + pd] = i;
                ++pd;
            }
        }
        base_o += to;
        base_d += td;
    }
    __syncthreads();

    // 4. the m most severe orphans and donors, in severity order
    uint64_t* sk = reinterpret_cast<uint64_t*>(
        reinterpret_cast<unsigned char*>(dyn) + sort_smem_offset(N));
    int* si = reinterpret_cast<int*>(sk + kSortMax);
    const int* orph;
    const int* don;
    int m_eff = m;
    {
        uint32_t* state = dyn;                                   // 2 bits per rank
        int* trs = reinterpret_cast<int*>(dyn + (N + 15) / 16);  // staged twin ranks
        // every donor in severity order; the other position buffer and the key
        // buffers' donor regions are free afterwards
        const int* spos =
            most_severe(s, k0 + n_o, i0 + n_o, k1 + n_o, i1 + n_o, n_d, n_d, sk, si);
        int* tr = spos == i0 + n_o ? i1 + n_o : i0 + n_o;
        int* dlist = reinterpret_cast<int*>(k0 + n_o);
        int* R = a.rank_of + off;
        for (int i = threadIdx.x; i < N; i += kT) R[i] = -1;
        for (int w = threadIdx.x; w < (n_d + 15) / 16; w += kT) state[w] = 0;
        __syncthreads();
        for (int k = threadIdx.x; k < n_d; k += kT) R[spos[k]] = k;
        __syncthreads();
        const int* tw = a.twin + off;
        for (int k = threadIdx.x; k < n_d; k += kT) {
            const int t = tw[spos[k]];
            tr[k] = (t >= 0 && t < N) ? R[t] : -1;
        }
        __syncthreads();
        int acc = 0;
        for (int c0 = 0; c0 < n_d && acc < n_o; c0 += kWalkChunk) {
            const int len = min(kWalkChunk, n_d - c0);
            for (int j = threadIdx.x; j < len; j += kT) trs[j] = tr[c0 + j];
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int j = 0; j < len && acc < n_o; ++j) {
                    const int k = c0 + j;
                    if ((state[k >> 4] >> ((k & 15) * 2)) & 2u) continue;          // pinned
                    const int t = trs[j];
                    if (t >= 0 && ((state[t >> 4] >> ((t & 15) * 2)) & 1u)) continue;  // twin out
                    state[k >> 4] |= 1u << ((k & 15) * 2);
                    if (t >= 0) state[t >> 4] |= 2u << ((t & 15) * 2);
                    dlist[acc++] = k;
                }
                s.flag = acc;
            }
            __syncthreads();
            acc = s.flag;
            __syncthreads();
        }
        m_eff = acc;
        for (int j = threadIdx.x; j < m_eff; j += kT) dlist[j] = spos[dlist[j]];
        __syncthreads();
        orph = most_severe(s, k0, i0, k1, i1, n_o, m_eff, sk, si);
        don = dlist;
    }
    __syncthreads();

    // 5. swap
    for (int k = threadIdx.x; k < m_eff; k += kT) {
        const int out_ = don[k], in_ = orph[k];
        S1[out_] = 0;
        S1[in_] = 1;
        swaps[2 * k] = out_;
        swaps[2 * k + 1] = in_;
    }
    if (threadIdx.x == 0) {
        a.out_nswaps[u] = m_eff;
        if (a.out_status) a.out_status[u] = 0;
    }
}

}  // namespace

namespace {

template <int C>
cudaError_t config_select(const RepairArgs& a, cudaStream_t st, cudaLaunchConfig_t& cfg,
                          cudaLaunchAttribute* at)
{
    const size_t bytes = 2 * static_cast<size_t>(kCap) * 12;   // the two sides' items
    static_assert(kCap >= kChunk, "the general path's shares fit too");
    cudaError_t e = cudaFuncSetAttribute(select_kernel<C>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(bytes));
    if (e != cudaSuccess) return e;
    if (C > 8) {
        e = cudaFuncSetAttribute(select_kernel<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(static_cast<unsigned>(a.U) * C);
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = st;
    cfg.attrs = at;
    if (a.dependent) {   // as launch_dependent
        cudaLaunchAttribute& p = at[cfg.numAttrs++];
        p.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        p.val.programmaticStreamSerializationAllowed = 1;
    }
    if (C > 1) {         // one CTA per unit: no cluster
        cudaLaunchAttribute& p = at[cfg.numAttrs++];
        p.id = cudaLaunchAttributeClusterDimension;
        p.val.clusterDim.x = C;
        p.val.clusterDim.y = 1;
        p.val.clusterDim.z = 1;
    }
    return cudaSuccess;
}

// Launches select_kernel<C> if a cluster of C CTAs can be resident; *launched says
// whether it was.
template <int C>
cudaError_t try_select(const RepairArgs& a, cudaStream_t st, bool* launched)
{
    *launched = false;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    cudaError_t e = config_select<C>(a, st, cfg, at);
    if (e != cudaSuccess) return e;
    if (C > 1) {
        int clusters = 0;
        e = cudaOccupancyMaxActiveClusters(&clusters, select_kernel<C>, &cfg);
        if (e != cudaSuccess || clusters < 1) {
            cudaGetLastError();   // not resident: the caller tries a smaller cluster
            return cudaSuccess;
        }
    }
    e = cudaLaunchKernelEx(&cfg, select_kernel<C>, a);
    *launched = e == cudaSuccess;
    return e;
}

}  // namespace

int select_cluster_size(int U, int N, int sms)
{
    // More CTAs per unit while each has an SM to itself and 4096 positions or more: below
    // that the cluster's barriers cost more than the shorter passes save, and a second CTA
    // on an SM halves both (us per selection with C = 1 / 2 / 4 / 8, half kept and 20 % of b
    // near 1: 8 units of 4096 positions 14 / 15 / 15 / 19, 8 of 32768 117 / 55 / 35 / 29, 72 of
    // 8192 23 / 19 / 25 / 70, 288 of 16384 59 / 80 / 111 / 284; 30 % of b equal to 1: 28 / 25 / 23
    // / 27, 215 / 117 / 72 / 51, 48 / 37 / 37 / 108, 125 / 152 / 195 / 404).  Slices above 24576
    // positions are split whatever the number of units, since their swap lists seldom fit one
    // CTA's buckets at once (16 units of 65536 312 / 174 / 69 / 64; 8 of 131072 919 / 461 / 217 /
    // 89, and 103 at 16).
    // Beyond the buckets' reach (kBucketMaxN): as many CTAs as two per SM allow, up to 16 (one
    // unit of 2^20 by the general path 3.80 ms at C = 4, 3.46 at 8, 3.31 at 16).
    int C = 1;
    if (N > kBucketMaxN) {
        while (C < 16 && static_cast<int64_t>(U) * (2 * C) <= 2LL * sms) C <<= 1;
        return C;
    }
    while (C < 8 && ((static_cast<int64_t>(U) * (2 * C) <= sms && N / (2 * C) >= 4096) ||
                     N / C > 24576))
        C <<= 1;
    return C;
}

cudaError_t launch_repair(const RepairArgs& a, cudaStream_t st)
{
    if (!a.twin) {
        int C = a.cluster;
        cudaError_t e = cudaSuccess;
        bool done = false;
        while (!done) {
            switch (C) {
            case 16: e = try_select<16>(a, st, &done); break;
            case 8: e = try_select<8>(a, st, &done); break;
            case 4: e = try_select<4>(a, st, &done); break;
            case 2: e = try_select<2>(a, st, &done); break;
            default: e = try_select<1>(a, st, &done); C = 1; break;
            }
            if (e != cudaSuccess) return e;
            if (!done && C == 1) return cudaErrorLaunchFailure;
            C >>= 1;
        }
        return cudaSuccess;
    }
    if (a.N > kDedupMaxN) return cudaErrorInvalidValue;
    const size_t bytes = std::max(dedup_kernel_smem_bytes(a.N), 2 * static_cast<size_t>(kCap) * 12);
    const cudaError_t e = cudaFuncSetAttribute(
        dedup_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (e != cudaSuccess) return e;
    if (a.dependent) return launch_dependent(dedup_kernel, dim3(a.U), kT, bytes, st, a);
    dedup_kernel<<<a.U, kT, bytes, st>>>(a);
    return cudaGetLastError();
}

}  // namespace twk
