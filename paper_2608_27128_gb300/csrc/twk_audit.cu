// twk_audit.cu -- fused redundancy audit for sm_103a (TwinKV, arXiv 2608.27128).
//
// For every key i of every unit it computes, without materialising the N x N matrix,
//   Sec. 3.2 Eq. 1   sim(i,j) = k_i . k_j / (||k_i|| ||k_j||)
//   Sec. 3.2         only j with |i - j| > w count (this also drops j = i)
//   Sec. 3.4 Eq. 4   b_i(S0) = max over retained j, -1 if none; and its argmax
//   (b_i(all))       the same over every j
//
// Design (persistent pairs of CTAs, one CTA per SM, 384 threads each, warp-specialised).  A
// pair shares each 256-row work item: CTA r holds rows [128 r, 128 r + 128) of A and of
// each B tile, and the accumulators of its own rows.
//   warp 0      TMA producer: its CTA's 128 rows of the keys i (once per work item), then
//               per 256-column tile its half of the keys j (in 64-wide K chunks) and the
//               whole tile's column metadata (1/||k_j|| and original positions).  Key
//               copies of both CTAs complete on the even CTA's barriers.
//   warp 1      owns TMEM (512 columns = two 128x256 fp32 accumulators); in the even CTA
//               one thread issues tcgen05.mma.cta_group::2 (M=256, N=256, K=16,
//               bf16 -> fp32) for both and commits to both CTAs' barriers.
//   warps 2, 3  merge the column groups of every finished row and write the results.
//   warps 4..   epilogue: four warps per column group (128 columns of each tile; in the count
//               mode at d = 128 every second tile); a thread owns one row (TMEM lane) and
//               keeps its running maximum.
// Why pairs: with one CTA per 128 rows, each tile moves 64 KB of B into shared memory
// and 96 KB of operands out of it (d = 128), beside the epilogue's broadcast loads; a
// pair moves 32 KB in and 64 KB out per SM.  Whole calls, one CTA -> pair: Qwen3-4B
// repair 36x8x16384x128 17.29 -> 16.71 ms, Llama-3.2-1B repair 16x8x8192x64
// 1032 -> 1010 us, policy 36x8x8192x128 3965 -> 3838 us; the same outputs bit for bit.
// The release of an accumulator to the even CTA is a remote arrival without a
// cluster-scope release (only TMEM reads precede it): with one, each cost the epilogue
// warp several hundred ns per tile (24.3 ms for the first of these calls).
// Keys enter the tensor cores un-normalised (bf16 products are exact in fp32);
// 1/||k_j|| (times a power of two per unit) is applied per element in fp32.
// 1/||k_i|| > 0 does not change the argmax over j, so it is never applied: this kernel
// outputs the twin positions, and the exact similarity of each chosen twin is computed
// afterwards (twk_refine.cu).
//
// Max and argmax: each 32-column chunk is scaled (the column scales carry a power of two
// per unit that brings every value into [-1, 1]), offset to be positive and reduced with
// 3-input maxima.  The column of a maximum is the lowest of its chunk among the values
// equal at 2^-18 relative (near-equal candidates only; exact ties go to the lowest column
// whatever their sign, as the values are never negative).  Columns to ignore carry NaN
// (max skips NaN): padding columns have 1/||k_j|| = NaN, and window columns
// (|i - j| <= w) are set to NaN on the few tiles that intersect the window band of the
// row block.
//
// What bounds it, from copies with parts left out (TFLOP/s of redundancy 16x8x16384x128,
// repair 16x8x8192x64, policy 36x8x8192x128 and 16x8x3001x64):
//   every part                        1579   745  1662   848
//   no reduction                      1968  1502  1937  1378
//   no MMAs                           1934   816  2169   910
//   no MMAs, no accumulator loads     2125   878  2406  1000
//   no loads of the column scales     1632   782  1670   923
//   no column codes (d = 64)             -   963     -     -
// At d = 64 it is the reduction: per thread and tile 64 paired multiply-adds, 128 column
// codes and 64 three-input maxima, the last two on an ALU that issues one instruction every
// two cycles.  At d = 128 MMAs and reduction overlap to within a fifth of the MMAs alone, at a
// rate that a seconds-long run holds under the power limit only just.  Two warps per
// scheduler hide little latency, so:
//   * the warpgroups trade registers (setmaxnreg): with 200 and more the four chunks of
//     a warp are scaled and reduced side by side (at 168 the compiler kept them apart);
//   * at d = 128 a row that improves only copies its chunk's values to its slot in shared
//     memory, and the column is looked up once per row block and segment;
//   * at d = 64 a row sees few columns and some row improves in most chunks, so the copies
//     (512 bytes of store path each) cost more than they save: there every value takes its
//     column code along in its low 5 bits;
//   * the next tile's barriers are tested while the current one is reduced (a wait on a
//     completed barrier took 150 cycles), the next item's counts are loaded one item
//     ahead, and two spare warps merge and write what the last item found.
// Audit alone, one CTA per 128 rows and 320 threads -> as built: Qwen3-4B 16x8x16384x128
// 1279 -> 1570 TFLOP/s, Llama-3.2-1B 16x8x8192x64 672 -> 746, policy 36x8x8192x128
// 1629 -> 1680, policy 16x8x3001x64 728 -> 853.  Sixteen epilogue warps of 64 columns (104
// registers): 1322, 674, 1522, 811.
//
// Count mode (Sec. 3.2 Eq. 2, the standalone scorer): instead of the maximum, each row i
// counts the columns j outside the window with sim(i,j) > tau.  With x_ij the raw dot
// product, that is x_ij * (1/||k_j||) > tau * ||k_i||.  The column scales arrive
// multiplied by S = 2^32 (exact), so one fused multiply-add with saturation,
// sat(x_ij * S/||k_j|| - S tau ||k_i||), is 1 when the pair counts and 0 when it does
// not (NaN, for masked and padding columns, saturates to 0); only a pair within
// 2^-32 of the threshold could give a fraction.  The product is never rounded before
// the comparison, the count accumulates in fp32 (exact below 2^24), and all of it
// runs on the FMA pipe.
//
// Column layout: in repair mode the columns of a unit are stored retained-first
// (retained keys in position order, padded to a tile, then evicted keys in position
// order), so every tile belongs to exactly one of the two maxima.  The kernel writes
// both winners; the maximum over all columns is the larger of the two, taken on the
// exact similarities computed afterwards.
#include <atomic>
#include <cfloat>

#include "twk_bound.cuh"
#include "twk_internal.h"
#include "twk_ptx.cuh"

namespace twk {
namespace {

constexpr int kHelperWarps = 4;                    // TMA, MMA, two that merge: a whole warpgroup
constexpr int kEpiWarps = 8;                       // epilogue warps: 2 per SM sub-partition
constexpr int kGroups = kEpiWarps / 4;             // column groups per tile
constexpr int kGW = kBN / kGroups;                 // columns per group
constexpr int kCh = kGW / 32;                      // 32-column chunks per group
constexpr int kThreads = 32 * (kHelperWarps + kEpiWarps);
constexpr int kLaunchRegs = 168;                   // registers per thread at launch
constexpr uint32_t kTmemCols = 512;
// a row's slot for the values of its best chunk: 32 floats and 16 bytes of padding, which
// spreads the lanes of a 16-byte access over the banks
constexpr int kSlot = 144;

template <int D, bool kCount = false, bool kSym = false>
struct AuditCfg {
    // Registers per thread after the warpgroups have traded theirs.  The epilogue's number
    // decides how far the compiler interleaves its chunks: d = 128 ran at 1571 TFLOP/s
    // with 200, 1520 with 216, 1465 with 232; d = 64 at 721 with 192, 718 with 200, 749
    // with 216.
    static constexpr int HELPER_REGS = D == 128 ? 104 : 72;
    static constexpr int EPI_REGS = D == 128 ? 200 : 216;
    static_assert(kHelperWarps * HELPER_REGS + kEpiWarps * EPI_REGS <=
                      (kHelperWarps + kEpiWarps) * kLaunchRegs,
                  "the split draws on the registers of the launch");
    static constexpr int KC = D / 64;                 // 128-byte K chunks per key row
    static constexpr int A_CHUNK = kBM * 128;         // 16 KB
    static constexpr int A_BYTES = KC * A_CHUNK;
    static constexpr int B_STAGE = kBN / 2 * 128;     // 16 KB: this CTA's half of a K chunk
    static constexpr int STAGES = 6;
    static constexpr int MSLOTS = 4;
    // Count mode at d = 128: a column group takes every second tile whole, in two passes,
    // instead of its half of every tile, so that one group's accumulator loads run beside the
    // other's counting (policy 36x8x8192x128: 2977 -> 2940 us of audit).  At d = 64 it changes
    // nothing (172.5 -> 173.4), and the argmax loses 3 to 4 %.
    static constexpr bool WHOLE = kCount && D == 128;
    static constexpr int TILE_WARPS = WHOLE ? kEpiWarps / kGroups : kEpiWarps;   // of a CTA
    static constexpr int META = kBN * 8;              // rinv[256] + pos[256]
    static constexpr int OFF_A = 0;
    static constexpr int OFF_B = OFF_A + 2 * A_BYTES;
    static constexpr int OFF_META = OFF_B + STAGES * B_STAGE;
    static constexpr int OFF_X = OFF_META + MSLOTS * META;   // 2 x groups x 128 x 16 B
    // symmetric mode: each group's four warps exchange their per-column maxima here
    // (two tile parities x groups x 4 lane quarters x 128 columns)
    static constexpr int OFF_CB = OFF_X + 2 * kGroups * kBM * 16;
    static constexpr int CB_BYTES = kSym ? 2 * kGroups * 4 * kBM * 4 : 0;
    // argmax mode: the 32 values of each thread's best chunk so far
    static constexpr int OFF_BEST = OFF_CB + CB_BYTES;
    static constexpr int BEST_BYTES =
        kCount || kSym || D == 64 ? 0 : kGroups * kBM * kSlot;
    // and the best value each group has published for each row, with its segment's stamp
    static constexpr int OFF_PUB = OFF_BEST + BEST_BYTES;
    static constexpr int PUB_BYTES = BEST_BYTES ? kGroups * kBM * 4 : 0;
    static constexpr int OFF_BAR = OFF_PUB + PUB_BYTES;
    static constexpr int NBAR = 2 + 2 + 2 * STAGES + 2 * MSLOTS + 2 + 2 + 2 + 2 + 1 +
                                (kSym ? 2 * kGroups : 0);
    static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
    static constexpr int BYTES = OFF_MISC + 16 + 1024;       // + 1024 for alignment
    static_assert(BYTES <= 232448, "shared memory per CTA");
    static_assert(kGroups == 2, "a group reads the other one's published bests");
};

__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// (v with its lowest mantissa bits replaced by idx); mask (0xFFFFFFE0) is a kernel
// argument, held in a register, so that idx can be the instruction's immediate.
__device__ __forceinline__ float pack(float v, uint32_t idx, uint32_t mask)
{
    return __uint_as_float((__float_as_uint(v) & mask) | idx);
}

__device__ __forceinline__ float nan_f() { return __uint_as_float(0x7FFFFFFFu); }

// Orders every later use of x after the preceding tcgen05.wait::ld: the registers
// written by tcgen05.ld are only valid after the wait, which the compiler cannot see.
__device__ __forceinline__ void reg_fence(uint32_t (&x)[32])
{
    asm volatile(""
                 : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4]), "+r"(x[5]),
                   "+r"(x[6]), "+r"(x[7]), "+r"(x[8]), "+r"(x[9]), "+r"(x[10]), "+r"(x[11]),
                   "+r"(x[12]), "+r"(x[13]), "+r"(x[14]), "+r"(x[15]), "+r"(x[16]),
                   "+r"(x[17]), "+r"(x[18]), "+r"(x[19]), "+r"(x[20]), "+r"(x[21]),
                   "+r"(x[22]), "+r"(x[23]), "+r"(x[24]), "+r"(x[25]), "+r"(x[26]),
                   "+r"(x[27]), "+r"(x[28]), "+r"(x[29]), "+r"(x[30]), "+r"(x[31]));
}

// Maximum of 32 values as a tree of 3-input maxima (depth 4); NaN entries are skipped.
__device__ __forceinline__ float tree32(const float (&p)[32])
{
    float q[11];
#pragma unroll
    for (int j = 0; j < 10; ++j) q[j] = fmax3(p[3 * j], p[3 * j + 1], p[3 * j + 2]);
    q[10] = fmaxf(p[30], p[31]);
    const float r0 = fmax3(q[0], q[1], q[2]);
    const float r1 = fmax3(q[3], q[4], q[5]);
    const float r2 = fmax3(q[6], q[7], q[8]);
    const float r3 = fmaxf(q[9], q[10]);
    return fmax3(r0, r1, fmaxf(r2, r3));
}

// Running best of one row over one segment: the largest scaled similarity so far and the
// first column of its 32-column chunk (the column itself once resolved, see keep_chunk).
struct Best {
    float v;
    int col;
};

// The offset added to every scaled similarity.  The column scales of a unit are
// 2^-e_u / ||k_j||, 2^e_u above every key norm of the unit, so x_ij times the scale is
// sim(i,j) ||k_i|| 2^-e_u, in [-1, 1]; with the offset (a little above 1, for the fp32
// error of x_ij) every value is positive.  A compile-time constant: the fused
// multiply-add then needs no register for it.
constexpr float kOffset = 1.0f + 0x1p-10f;

// Where `up`, the thread's 32 values go to its slot.
__device__ __forceinline__ void keep_chunk(uint32_t slot, const float (&v)[32], bool up)
{
#pragma unroll
    for (int q = 0; q < 8; ++q)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.u32 p, %0, 0;\n\t"
            "@p st.shared.v4.f32 [%1], {%2, %3, %4, %5};\n\t}" ::"r"(up ? 1u : 0u),
            "r"(slot + 16u * q), "f"(v[4 * q]), "f"(v[4 * q + 1]), "f"(v[4 * q + 2]),
            "f"(v[4 * q + 3]));
}

// The column of a running best: the lowest of its chunk whose value agrees with the
// maximum to 2^-18 relative (the 5 lowest mantissa bits cleared; the values are positive,
// so "at least the cleared maximum" is that comparison).
__device__ __forceinline__ void resolve_best(uint32_t slot, uint32_t mask, Best& b)
{
    if (b.col < 0) return;
    const float floor_v = __uint_as_float(__float_as_uint(b.v) & mask);
    int c = 31;
#pragma unroll
    for (int q = 7; q >= 0; --q) {
        float v[4];
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                     : "r"(slot + 16u * q));
#pragma unroll
        for (int e = 3; e >= 0; --e) c = v[e] >= floor_v ? 4 * q + e : c;
    }
    b.col += c;
}

// Each accumulator value scaled and offset, v = x_ij 2^-e_u/||k_j|| + kOffset > 0, in one
// fused multiply-add (NaN where the window drops the column, or where the column scale is
// NaN on padding).
template <bool kMasked>
__device__ __forceinline__ void scale32(const uint32_t (&x)[32], const float* rinv,
                                        const int* pos, int rw, uint32_t w2, float (&v)[32])
{
    const float2 ofs = make_float2(kOffset, kOffset);
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
        const float4 r = *reinterpret_cast<const float4*>(rinv + k);
        const float2 p01 = __ffma2_rn(make_float2(__uint_as_float(x[k]), __uint_as_float(x[k + 1])),
                                      make_float2(r.x, r.y), ofs);
        const float2 p23 = __ffma2_rn(
            make_float2(__uint_as_float(x[k + 2]), __uint_as_float(x[k + 3])),
            make_float2(r.z, r.w), ofs);
        v[k] = p01.x;
        v[k + 1] = p01.y;
        v[k + 2] = p23.x;
        v[k + 3] = p23.y;
        if (kMasked) {
            // column j is dropped when |pos_j - row| <= w, i.e. (unsigned)(pos_j - (row - w)) <= 2w
            const int4 q = *reinterpret_cast<const int4*>(pos + k);
            v[k] = (static_cast<uint32_t>(q.x - rw) > w2) ? v[k] : nan_f();
            v[k + 1] = (static_cast<uint32_t>(q.y - rw) > w2) ? v[k + 1] : nan_f();
            v[k + 2] = (static_cast<uint32_t>(q.z - rw) > w2) ? v[k + 2] : nan_f();
            v[k + 3] = (static_cast<uint32_t>(q.w - rw) > w2) ? v[k + 3] : nan_f();
        }
    }
}

// The symmetric mode's row direction: each value's 5 lowest mantissa bits are replaced by
// (31 - column) and one tree gives the lowest column among the values equal to the maximum
// at 2^-18 relative; the running best moves at that resolution.
template <bool kMasked>
__device__ __forceinline__ void fold32_packed(const uint32_t (&x)[32], const float* rinv,
                                              const int* pos, int rw, uint32_t w2, uint32_t mask,
                                              int col0, Best& b)
{
    float v[32];
    scale32<kMasked>(x, rinv, pos, rw, w2, v);
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = pack(v[k], 31u - static_cast<uint32_t>(k), mask);
    const uint32_t mp = __float_as_uint(tree32(v));
    const float m = __uint_as_float(mp & mask);
    if (m > b.v) {
        b.v = m;
        b.col = col0 + 31 - static_cast<int>(mp & 31u);
    }
}

// The thread's accumulator columns of one tile, loaded into registers (after this, the
// accumulator may be released: the MMA can overwrite it while x is reduced).
__device__ __forceinline__ void load_group(uint32_t taddr, uint32_t (&x)[kCh][32])
{
#pragma unroll
    for (int k = 0; k < kCh; ++k) tmem_ld_32x32b_x32(taddr + 32 * k, x[k]);
    tmem_wait_ld();
#pragma unroll
    for (int k = 0; k < kCh; ++k) reg_fence(x[k]);
}

// The loaded group scaled, and the maximum of each of its chunks, with nothing between the
// chunks that would keep their instructions apart.
template <bool kMasked>
__device__ __forceinline__ void scale_group(const uint32_t (&x)[kCh][32], const float* rinv,
                                            const int* pos, int rw, uint32_t w2,
                                            float (&v)[kCh][32], float (&m)[kCh])
{
#pragma unroll
    for (int k = 0; k < kCh; ++k) scale32<kMasked>(x[k], rinv + 32 * k, pos + 32 * k, rw, w2, v[k]);
#pragma unroll
    for (int k = 0; k < kCh; ++k) m[k] = tree32(v[k]);
}

// A best value published to the thread of the row's other column group, which reads it with
// nothing ordering the two: one 32-bit word (twk_bound.cuh) that is written and read whole by
// relaxed accesses, whatever mixture of segments the two threads are at.  (As a (value, stamp)
// pair in one vector access it could be seen half written, since a vector access is several
// scalar ones in no given order, and an old segment's value would then drop a row's maximum.)
__device__ __forceinline__ void publish(uint32_t at, uint32_t word)
{
    asm volatile("st.relaxed.cta.shared::cta.u32 [%0], %1;" ::"r"(at), "r"(word));
}

// What the word at `at` bounds from below in segment `stamp` (-inf: nothing).
__device__ __forceinline__ float published(uint32_t at, uint32_t stamp)
{
    uint32_t word;
    asm volatile("ld.relaxed.cta.shared::cta.u32 %0, [%1];" : "=r"(word) : "r"(at));
    return __uint_as_float(bound_bits(word, stamp));
}

// Where a row of the warp improves on its best (strictly, so an earlier chunk keeps a
// tie), its first chunk with the group's largest maximum is kept: the 32 values go to the
// row's slot, and which column it was is looked up once, when the segment ends.
// `other` is the best that the row's other column group has published for this segment
// (-inf if none): what stays below it cannot be the row's maximum and is not kept.  The
// improved best is published at `mine` with the segment's stamp.  The two groups of a row
// then improve 4.1 instead of 6.8 times over 32 tiles.  Calls without the exchange -> with it:
// dedup 18x8x8192x128 (10 tiles per row block) 831 -> 820 us, redundancy 2x8x5003x128 118 ->
// 116, repair 1x8x131072x128 11625 -> 11300, Qwen3-4B 0.3 %.
__device__ __forceinline__ void keep_best(const float (&v)[kCh][32], const float (&m)[kCh],
                                          int col0, uint32_t slot, uint32_t mine,
                                          uint32_t stamp, float other, Best& b)
{
    float top = m[0];
#pragma unroll
    for (int k = 1; k < kCh; ++k) top = fmaxf(top, m[k]);
    const bool up = top > b.v && top >= other;   // an equal value may be the lower column
    bool here[kCh];
    unsigned any[kCh];
    bool left = up;
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
        here[k] = left && m[k] == top;
        left = left && !here[k];
        any[k] = __ballot_sync(0xFFFFFFFFu, here[k]);   // the votes overlap each other
    }
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
        if (any[k]) keep_chunk(slot, v[k], here[k]);
        b.col = here[k] ? col0 + 32 * k : b.col;
    }
    b.v = up ? top : b.v;
    // a value that is not positive (keys whose norms overflow) has no word that rounds down
    if (up && top > 0.f) publish(mine, bound_word(__float_as_uint(top), stamp));
}

// The same without a slot: the low 5 mantissa bits of each value give way to (31 - column),
// so that one more maximum returns the lowest column among the values equal at 2^-18
// relative, and the running best moves at that resolution.
template <bool kMasked>
__device__ __forceinline__ void fold_packed(const uint32_t (&x)[kCh][32], const float* rinv,
                                            const int* pos, int rw, uint32_t w2, uint32_t mask,
                                            int col0, Best& b)
{
    float v[kCh][32];
    uint32_t mp[kCh];
#pragma unroll
    for (int k = 0; k < kCh; ++k) scale32<kMasked>(x[k], rinv + 32 * k, pos + 32 * k, rw, w2, v[k]);
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
#pragma unroll
        for (int c = 0; c < 32; ++c) v[k][c] = pack(v[k][c], 31u - static_cast<uint32_t>(c), mask);
        mp[k] = __float_as_uint(tree32(v[k]));
    }
#pragma unroll
    for (int k = 0; k < kCh; ++k) {
        const float m = __uint_as_float(mp[k] & mask);
        if (m > b.v) {
            b.v = m;
            b.col = col0 + 32 * k + 31 - static_cast<int>(mp[k] & 31u);
        }
    }
}

// sat(a * b + c): fp32 fused multiply-add clamped to [0, 1], NaN to 0.
__device__ __forceinline__ float fma_sat(float a, float b, float c)
{
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Eq. 2 over 32 columns: how many x_j * S/||k_j|| exceed ts = S tau ||k_i||, as two
// partial sums.
template <bool kMasked>
__device__ __forceinline__ float2 count32(const uint32_t (&x)[32], const float* rinv,
                                          const int* pos, int rw, uint32_t w2, float ts)
{
    float2 ca = make_float2(0.f, 0.f), cb = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
        const float4 r = *reinterpret_cast<const float4*>(rinv + k);
        float v0 = __uint_as_float(x[k]), v1 = __uint_as_float(x[k + 1]);
        float v2 = __uint_as_float(x[k + 2]), v3 = __uint_as_float(x[k + 3]);
        if (kMasked) {
            const int4 q = *reinterpret_cast<const int4*>(pos + k);
            v0 = (static_cast<uint32_t>(q.x - rw) > w2) ? v0 : nan_f();
            v1 = (static_cast<uint32_t>(q.y - rw) > w2) ? v1 : nan_f();
            v2 = (static_cast<uint32_t>(q.z - rw) > w2) ? v2 : nan_f();
            v3 = (static_cast<uint32_t>(q.w - rw) > w2) ? v3 : nan_f();
        }
        ca = __fadd2_rn(ca, make_float2(fma_sat(v0, r.x, -ts), fma_sat(v1, r.y, -ts)));
        cb = __fadd2_rn(cb, make_float2(fma_sat(v2, r.z, -ts), fma_sat(v3, r.w, -ts)));
    }
    return __fadd2_rn(ca, cb);
}

template <bool kMasked>
__device__ __forceinline__ float count_group(const uint32_t (&x)[kCh][32], const float* rinv,
                                             const int* pos, int rw, uint32_t w2, float ts)
{
    float2 c = count32<kMasked>(x[0], rinv, pos, rw, w2, ts);
#pragma unroll
    for (int k = 1; k < kCh; ++k)
        c = __fadd2_rn(c, count32<kMasked>(x[k], rinv + 32 * k, pos + 32 * k, rw, w2, ts));
    return c.x + c.y;
}

__device__ __forceinline__ uint32_t redux_max(uint32_t v)
{
    uint32_t r;
    asm volatile("redux.sync.max.u32 %0, %1, 0xffffffff;" : "=r"(r) : "r"(v));
    return r;
}

// Symmetric mode, the column direction of one 32-column chunk: for every column j of
// the chunk the largest x_ij s_i + kOffset over the warp's 32 rows i (s_i = the row's
// own column scale, so the value is that of row j's candidate i), its low 5 bits
// replaced by (31 - lane) so that a tie goes to the lowest row.  Masked: window pairs
// and rows past the end give 0, below every candidate.  Lane l returns column l's.
template <bool kMasked>
__device__ __forceinline__ uint32_t colpass32(const uint32_t (&x)[32], const int* pos, int rw,
                                              uint32_t w2, float si, bool row_ok)
{
    const int lane = threadIdx.x & 31;
    const uint32_t code = 31u - static_cast<uint32_t>(lane);
    uint32_t keep = 0u;
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
        int4 q = make_int4(0, 0, 0, 0);
        if (kMasked) q = *reinterpret_cast<const int4*>(pos + k);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float v = fmaf(__uint_as_float(x[k + e]), si, kOffset);
            if (kMasked) {
                const int pj = e == 0 ? q.x : e == 1 ? q.y : e == 2 ? q.z : q.w;
                v = (row_ok && static_cast<uint32_t>(pj - rw) > w2) ? v : 0.f;
            }
            const uint32_t r = redux_max((__float_as_uint(v) & 0xFFFFFFE0u) | code);
            keep = lane == k + e ? r : keep;
        }
    }
    return keep;
}

struct Tiles {
    int tr;   // tiles of segment 0 (retained, or every column in mode 0)
    int te;   // tiles of segment 1 (evicted; 0 unless b_all is wanted)
    int t0;   // the first tile (symmetric mode: the tile holding the row block's columns)
};

// The work items of one CTA pair in order.  The next item's retained count is loaded while
// the current item is worked on, so that no role waits for it between items.
template <bool kSym>
struct Items {
    int item, u, rb;        // the item at hand: its unit and row block
    int kb = 0;             // |S0| of its unit (repair mode)
    int nu = 0, nrb = 0, nkb = 0;   // the next one's

    __device__ __forceinline__ Items(const AuditArgs& a, int first) : item(first)
    {
        u = item / a.RB;
        rb = item - u * a.RB;
        if (a.repair_mode && item < a.U * a.RB) kb = a.kb[u];
    }
    __device__ __forceinline__ void prefetch(const AuditArgs& a, int step)
    {
        const int n = item + step;
        nu = n / a.RB;
        nrb = n - nu * a.RB;
        if (a.repair_mode && n < a.U * a.RB) nkb = a.kb[nu];
    }
    __device__ __forceinline__ void advance(int step)
    {
        item += step;
        u = nu;
        rb = nrb;
        kb = nkb;
    }
    // Symmetric mode: row block rb takes the tiles from the one holding its own columns, rb,
    // to the last; the pairs left of them reach rb's rows through the column maxima of
    // the row blocks before it.
    __device__ __forceinline__ Tiles tiles(const AuditArgs& a) const
    {
        if (kSym) return {(a.N + kBN - 1) / kBN - rb, 0, rb};
        if (!a.repair_mode) return {(a.N + kBN - 1) / kBN, 0, 0};
        return {(kb + kBN - 1) / kBN, a.need_all ? (a.N - kb + kBN - 1) / kBN : 0, 0};
    }
};

// Every lane waits (each needs the acquire), the warp agrees on the verdict.
__device__ __forceinline__ bool all_wait(uint64_t* bar, uint32_t parity, const WaitCtl& w,
                                         int where)
{
    const bool ok = mbar_wait(bar, parity, w, where);
    return __all_sync(0xFFFFFFFFu, ok);
}

// Bounded wait that ignores the abort flag (used to drain in-flight copies and MMAs
// after a give-up), never shorter than kDrainFloorNs whatever the caller's limit.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns)
{
    const uint64_t limit = limit_ns > kDrainFloorNs ? limit_ns : kDrainFloorNs;
    const uint32_t a = smem_u32(bar);
    const uint64_t t0 = globaltimer_ns();
    while (!mbar_try_wait_sleep(a, parity, 1000000u))
        if (globaltimer_ns() - t0 > limit) return;
}

// Lets `ns` nanoseconds pass.
__device__ __forceinline__ void hold_ns(uint64_t ns)
{
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < ns) __nanosleep(1000000u);
}

// Position in a ring of kN slots: the slot in use and the parity of its current phase.
template <int kN>
struct Ring {
    uint32_t slot = 0, phase = 0;

    __device__ __forceinline__ void next()
    {
        if (++slot == kN) {
            slot = 0;
            phase ^= 1u;
            wrapped = true;
        }
    }
    // Parity of the last use of slot s, or -1 if it was never used.
    __device__ __forceinline__ int last_parity(uint32_t s) const
    {
        if (s < slot) return static_cast<int>(phase);
        return wrapped ? static_cast<int>(phase ^ 1u) : -1;
    }

private:
    bool wrapped = false;
};

template <int D, bool kCount, bool kSym>
__global__ void __cluster_dims__(2, 1, 1)
    __launch_bounds__(kThreads, 1)
    audit_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ AuditArgs a)
{
    using C = AuditCfg<D, kCount, kSym>;
    // Chunks are compared with each other exactly at d = 128, and at 2^-18 relative (the
    // earlier chunk on a tie) at d = 64.
    constexpr bool kPacked = D == 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* sA = smem + C::OFF_A;
    uint8_t* sB = smem + C::OFF_B;
    uint8_t* sMeta = smem + C::OFF_META;
    float4* sX = reinterpret_cast<float4*>(smem + C::OFF_X);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
    uint64_t* a_full = bars;
    uint64_t* a_empty = a_full + 2;
    uint64_t* b_full = a_empty + 2;
    uint64_t* b_empty = b_full + C::STAGES;
    uint64_t* m_full = b_empty + C::STAGES;
    uint64_t* m_empty = m_full + C::MSLOTS;
    uint64_t* t_full = m_empty + C::MSLOTS;
    uint64_t* t_empty = t_full + 2;
    uint64_t* x_full = t_empty + 2;
    uint64_t* x_empty = x_full + 2;
    uint64_t* drain = x_empty + 2;
    uint64_t* cbar = drain + 1;   // symmetric mode: [tile parity][group], 128 arrivals
    uint32_t* sCB = reinterpret_cast<uint32_t*>(smem + C::OFF_CB);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);

    // From a shuffle the compiler knows that the warp's number is the same in every lane
    // (d = 128: 1559 TFLOP/s against 1482 without; at d = 64 it then spills, for 1 %).
    const int warp = D == 64 && !kCount
                         ? static_cast<int>(threadIdx.x >> 5)
                         : __shfl_sync(0xFFFFFFFFu, static_cast<int>(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&a_full[i], 1);
            mbar_init(&a_empty[i], 1);
            mbar_init(&t_full[i], 1);
            mbar_init(&t_empty[i], 2 * C::TILE_WARPS);   // both CTAs' epilogues
            mbar_init(&x_full[i], kGroups * kBM);
            mbar_init(&x_empty[i], 64);
        }
        for (int i = 0; i < C::STAGES; ++i) {
            mbar_init(&b_full[i], 1);
            mbar_init(&b_empty[i], 1);
        }
        for (int i = 0; i < C::MSLOTS; ++i) {
            mbar_init(&m_full[i], 1);
            mbar_init(&m_empty[i], C::TILE_WARPS);
        }
        mbar_init(drain, 1);
        if (kSym)
            for (int i = 0; i < 2 * kGroups; ++i) mbar_init(&cbar[i], 4 * 32);
        *abort_flag = 0;
        fence_mbarrier_init();
    }
    for (int i = threadIdx.x; i < C::PUB_BYTES / 4; i += kThreads)
        publish(smem_u32(smem + C::OFF_PUB) + 4 * i, bound_word(kNoBound, 0u));
    if (warp == 0 && lane == 0) {
        prefetch_tensormap(&tmA);
        prefetch_tensormap(&tmB);
    }
    if (warp == 1) tmem_alloc<2>(tmem_slot, kTmemCols);
    tc_fence_before();
    cluster_barrier();   // barriers of both CTAs initialised, tensor memory allocated
    tc_fence_after();
    wait_for_previous();
    const uint32_t tmem = *tmem_slot;

    WaitCtl wc;
    wc.limit_ns = a.timeout_ns;
    wc.abort_flag = abort_flag;
    wc.err = a.err;
    wc.where = 0;
    const int n_items = a.U * a.RB;
    const int pair = static_cast<int>(blockIdx.x >> 1);
    const int n_pairs = static_cast<int>(gridDim.x >> 1);
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;

    if (warp < kHelperWarps) {
        setmaxnreg_dec<C::HELPER_REGS>();
        if (warp == 0) {
            // ------------------------------------------------------------ TMA producer
            // One thread runs the whole role: its waits are the shortest path from a released
            // stage to the copy that fills it.
            if (lane == 0) {
                Ring<2> ra;
                Ring<C::STAGES> rb_;
                Ring<C::MSLOTS> rm;
                bool ok = true;
                for (Items<kSym> it(a, pair); it.item < n_items && ok; it.advance(n_pairs)) {
                    const int u = it.u, rb = it.rb;
                    const Tiles ut = it.tiles(a);
                    it.prefetch(a, n_pairs);
                    ok = mbar_wait(&a_empty[ra.slot], ra.phase ^ 1u, wc, 1);
                    if (!ok) break;
                    if (leader) mbar_arrive_expect_tx(&a_full[ra.slot], 2 * C::A_BYTES);
                    const uint32_t full = cluster_addr(&a_full[ra.slot], 0);
                    const int y = u * a.N + rb * kPM + static_cast<int>(rank) * kBM;
#pragma unroll
                    for (int kc = 0; kc < C::KC; ++kc)
                        tma_load_2d_pair(sA + ra.slot * C::A_BYTES + kc * C::A_CHUNK, &tmA, full,
                                         kc * 64, y);
                    ra.next();
                    const int nt = ut.tr + ut.te;
                    int64_t off = static_cast<int64_t>(u) * a.NP + ut.t0 * kBN;
                    int yb = static_cast<int>(u * a.b_rows_per_unit + ut.t0 * kBN) +
                             static_cast<int>(rank) * (kBN / 2);
                    for (int t = 0; t < nt; ++t, off += kBN, yb += kBN) {
                        ok = mbar_wait(&m_empty[rm.slot], rm.phase ^ 1u, wc, 2);
                        if (!ok) break;
                        uint8_t* meta = sMeta + rm.slot * C::META;
                        mbar_arrive_expect_tx(&m_full[rm.slot], C::META);
                        bulk_load(meta, a.colrinv + off, kBN * 4, &m_full[rm.slot]);
                        bulk_load(meta + kBN * 4, a.colpos + off, kBN * 4, &m_full[rm.slot]);
                        rm.next();
#pragma unroll
                        for (int kc = 0; kc < C::KC; ++kc) {
                            ok = mbar_wait(&b_empty[rb_.slot], rb_.phase ^ 1u, wc, 3);
                            if (!ok) break;
                            if (leader) mbar_arrive_expect_tx(&b_full[rb_.slot], 2 * C::B_STAGE);
                            tma_load_2d_pair(sB + rb_.slot * C::B_STAGE, &tmB,
                                             cluster_addr(&b_full[rb_.slot], 0), kc * 64, yb);
                            rb_.next();
                        }
                        if (!ok) break;
                    }
                }
                // The even CTA's commits release the rings in both CTAs: each CTA stays until
                // the last release of every slot has reached it.
                for (int s = 0; ok && s < 2; ++s) {
                    const int p = ra.last_parity(s);
                    if (p >= 0) ok = mbar_wait(&a_empty[s], static_cast<uint32_t>(p), wc, 12);
                }
                for (int s = 0; ok && s < C::STAGES; ++s) {
                    const int p = rb_.last_parity(s);
                    if (p >= 0) ok = mbar_wait(&b_empty[s], static_cast<uint32_t>(p), wc, 13);
                }
                if (!ok) {
                    // Let every copy this warp started land before the block exits.  A and B
                    // copies of both CTAs complete on the even CTA's barriers, which waits for
                    // the slots that it has armed itself.  The odd CTA can be a ring ahead of
                    // that and cannot wait on those barriers: it stays for as long as a drain
                    // lasts at least (a copy takes microseconds).
                    if (!leader) hold_ns(kDrainFloorNs);
                    for (int s = 0; leader && s < 2; ++s) {
                        const int p = ra.last_parity(s);
                        if (p >= 0) drain_wait(&a_full[s], p, a.timeout_ns);
                    }
                    for (int s = 0; leader && s < C::STAGES; ++s) {
                        const int p = rb_.last_parity(s);
                        if (p >= 0) drain_wait(&b_full[s], p, a.timeout_ns);
                    }
                    for (int s = 0; s < C::MSLOTS; ++s) {
                        const int p = rm.last_parity(s);
                        if (p >= 0) drain_wait(&m_full[s], p, a.timeout_ns);
                    }
                }
            }
            __syncwarp();
        } else if (warp == 1) {
            // ------------------------------------------------------------ MMA issuer
            // One thread of the even CTA issues for both.
            if (leader && lane == 0) {
                constexpr uint32_t idesc = umma_idesc_bf16_f32(kPM, kBN);
                Ring<2> ra, rt;
                Ring<C::STAGES> rb_;
                bool ok = true;
                for (Items<kSym> it(a, pair); it.item < n_items && ok; it.advance(n_pairs)) {
                    const Tiles ut = it.tiles(a);
                    it.prefetch(a, n_pairs);
                    ok = mbar_wait(&a_full[ra.slot], ra.phase, wc, 4);
                    if (!ok) break;
                    const uint64_t ad = umma_desc_sw128(smem_u32(sA + ra.slot * C::A_BYTES));
                    const int nt = ut.tr + ut.te;
                    for (int t = 0; t < nt; ++t) {
                        ok = mbar_wait(&t_empty[rt.slot], rt.phase ^ 1u, wc, 5);
                        if (!ok) break;
                        const uint32_t d_tmem = tmem + rt.slot * kBN;
#pragma unroll
                        for (int kc = 0; kc < C::KC; ++kc) {
                            ok = mbar_wait(&b_full[rb_.slot], rb_.phase, wc, 6);
                            if (!ok) break;
                            tc_fence_after();
                            const uint64_t bd =
                                umma_desc_sw128(smem_u32(sB + rb_.slot * C::B_STAGE));
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                umma_bf16_pair(d_tmem, ad + (kc * C::A_CHUNK >> 4) + 2u * k,
                                               bd + 2u * k, idesc, (kc | k) != 0 ? 1u : 0u);
                            umma_commit_pair(&b_empty[rb_.slot]);
                            rb_.next();
                        }
                        if (!ok) break;
                        umma_commit_pair(&t_full[rt.slot]);
                        rt.next();
                    }
                    if (!ok) break;
                    umma_commit_pair(&a_empty[ra.slot]);
                    ra.next();
                }
                // Every MMA this thread issued completes before TMEM is released.
                umma_commit_own(drain);
                drain_wait(drain, 0, a.timeout_ns);
            }
            __syncwarp();
        } else {
            // ------------------------------------------------------------ merge
            // Two warps combine the column groups of every row and write the result, while the
            // epilogue is already at the next item.
            uint32_t n_x = 0;
            bool ok = true;
            for (Items<kSym> it(a, pair); it.item < n_items && ok; it.advance(n_pairs), ++n_x) {
                it.prefetch(a, n_pairs);
                const int xb = static_cast<int>(n_x & 1);
                ok = all_wait(&x_full[xb], (n_x >> 1) & 1, wc, 10);
                if (!ok) break;
                const int64_t rbase = static_cast<int64_t>(it.u) * a.N;
                const int64_t cbase = static_cast<int64_t>(it.u) * a.NP;
#pragma unroll
                for (int k = 0; k < kBM / 64; ++k) {
                    const int rl = k * 64 + (warp - 2) * 32 + lane;
                    const int row = it.rb * kPM + static_cast<int>(rank) * kBM + rl;
                    const float4* X = sX + xb * kGroups * kBM + rl;
                    float4 o = X[0];
                    int c0 = __float_as_int(o.y), c1 = __float_as_int(o.w);
#pragma unroll
                    for (int g = 1; g < kGroups; ++g) {
                        const float4 n = X[g * kBM];
                        if (kCount) {
                            o.x += n.x;
                            continue;
                        }
                        const int nc0 = __float_as_int(n.y), nc1 = __float_as_int(n.w);
                        if (nc0 >= 0 && (c0 < 0 || n.x > o.x || (n.x == o.x && nc0 < c0))) {
                            o.x = n.x;
                            c0 = nc0;
                        }
                        if (nc1 >= 0 && (c1 < 0 || n.z > o.z || (n.z == o.z && nc1 < c1))) {
                            o.z = n.z;
                            c1 = nc1;
                        }
                    }
                    if (row >= a.N) continue;
                    if (kCount) {
                        a.out_count[rbase + row] = __float2int_rn(o.x);
                    } else if (kSym) {
                        // the row direction's best joins the column maxima of earlier row
                        // blocks in the row's slot: value (low 5 bits cleared) then lowest
                        // position
                        if (c0 >= 0)
                            atomicMax(a.slots + rbase + row,
                                      (static_cast<unsigned long long>(__float_as_uint(o.x) &
                                                                       0xFFFFFFE0u) << 32) |
                                          (0xFFFFFFFFull - static_cast<uint32_t>(c0)));
                    } else {
                        a.out_t0[rbase + row] =
                            c0 < 0 ? -1 : (a.repair_mode ? a.colpos[cbase + c0] : c0);
                        if (a.repair_mode && a.need_all)
                            a.out_t1[rbase + row] = c1 < 0 ? -1 : a.colpos[cbase + c1];
                    }
                }
                mbar_arrive(&x_empty[xb]);
            }
            __syncwarp();
        }
        // Neither CTA frees its tensor memory or exits while the pair's MMAs, commits or
        // arrivals can still reach it.  (The epilogue ends with its own copy of the barrier:
        // with a common end, the compiler spills what lives across its tile loop.)
        tc_fence_before();
        cluster_barrier();
        tc_fence_after();
        if (warp == 1) tmem_dealloc<2>(*tmem_slot, kTmemCols);
    } else {
        // ------------------------------------------------------------ epilogue
        setmaxnreg_inc<C::EPI_REGS>();
        const int ew = warp - kHelperWarps;
        const int h = ew >> 2;            // column group of the tile
        const int q = warp & 3;           // TMEM lane quarter this warp may read
        const int row_local = q * 32 + lane;
        const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
        const int w = a.window;
        const uint32_t w2 = 2u * static_cast<uint32_t>(w);
        const uint32_t mask = a.mant_mask;
        const uint32_t slot = smem_u32(smem + C::OFF_BEST) +
                              static_cast<uint32_t>((h * kBM + row_local) * kSlot);
        const uint32_t release0 = cluster_addr(&t_empty[0], 0);
        const uint32_t release1 = cluster_addr(&t_empty[1], 0);
        const uint32_t m_full0 = smem_u32(m_full), t_full0 = smem_u32(t_full);
        uint32_t n_t = 0;   // tiles seen: metadata slot n_t mod MSLOTS, accumulator n_t mod 2
        // the row's published bests, one per group; stamps count this CTA's segments, and a
        // thread clears its word when it enters one (see twk_bound.cuh)
        const uint32_t pub = smem_u32(smem + C::OFF_PUB) + static_cast<uint32_t>(row_local * 4);
        uint32_t n_x = 0;
        uint32_t n_c = 0;   // symmetric mode: tiles whose column maxima were merged
        bool ok = true;
        // the coming tile's metadata and accumulator were seen complete (tested while the
        // tile before it was reduced, so that the test's latency is hidden)
        uint32_t ready = 0;
        // Column counts at the ends of the window band [r0 - w, r0 + 128 + w) of a row block
        // (repair mode), loaded one item ahead like its retained count.
        auto band_counts = [&](int bu, int brb, int bkb, int& clo, int& chi) {
            const int b0r = brb * kPM + static_cast<int>(rank) * kBM;
            const int lo = max(b0r - w, 0), hi = min(b0r + kBM + w, a.N);
            const int* cnt = a.cnt + static_cast<int64_t>(bu) * a.N;
            clo = lo < a.N ? cnt[lo] : bkb;
            chi = hi < a.N ? cnt[hi] : bkb;
        };
        Items<kSym> it(a, pair);
        int clo = 0, chi = 0, nclo = 0, nchi = 0;
        if (a.repair_mode && it.item < n_items) band_counts(it.u, it.rb, it.kb, clo, chi);
        for (; it.item < n_items && ok; it.advance(n_pairs), clo = nclo, chi = nchi) {
            const int u = it.u, rb = it.rb;
            const Tiles ut = it.tiles(a);
            const int nt = ut.tr + ut.te;
            const int r0 = rb * kPM + static_cast<int>(rank) * kBM;
            const int row = r0 + row_local;
            it.prefetch(a, n_pairs);
            // symmetric mode: the row's own column scale (the value of row j's candidate
            // i is x_ij s_i), and whether this row block runs past the end of the unit
            const bool row_ok = row < a.N;
            const float si = (kSym && row_ok) ? a.colrinv[static_cast<int64_t>(u) * a.NP + row] : 0.f;
            const bool pad_item = r0 + kBM > a.N;

            // Column ranges that meet the window band of this row block: only tiles meeting
            // them need the per-element window test.  A group's columns [c_lo, c_lo + GW)
            // meet [s, e) when c_lo - (s - GW + 1), as unsigned, is below e - s + GW - 1.
            const int lo = max(r0 - w, 0);
            const int hi = min(r0 + kBM + w, a.N);
            int s0a, s1a = 0;
            uint32_t s0n, s1n = 0;
            if (!a.repair_mode) {
                s0a = lo - (kGW - 1);
                s0n = hi > lo ? hi - lo + kGW - 1 : 0;
            } else {
                const int nlo = lo - clo, nhi = hi - chi;   // evicted before each end
                s0a = clo - (kGW - 1);
                s0n = chi > clo ? chi - clo + kGW - 1 : 0;
                s1a = ut.tr * kBN + nlo - (kGW - 1);
                s1n = nhi > nlo ? nhi - nlo + kGW - 1 : 0;
                if (it.item + n_pairs < n_items) band_counts(it.nu, it.nrb, it.nkb, nclo, nchi);
            }

            Best b0{-INFINITY, -1}, b1{-INFINITY, -1};   // retained (or all) / evicted
            Best best = b0;                              // of the segment at hand
            const int rw = row - w;
            if constexpr (C::PUB_BYTES != 0)
                publish(pub + h * kBM * 4, bound_word(kNoBound, 2u * n_x));

            float cnt = 0.f;                               // count mode: r_i so far
            float thr = 0.f;                               // count mode: S tau ||k_i||
            if (kCount)
                thr = (a.count_tau /
                       (a.colrinv[static_cast<int64_t>(u) * a.NP + row] * (1.0f / kCountScale))) *
                      kCountScale;
            constexpr int kStep = C::WHOLE ? kGroups : 1;
            const uint32_t n_item = n_t;   // the item's first tile
            // whole tiles: group h takes those whose accumulator is h
            const int t_first =
                C::WHOLE ? static_cast<int>((n_t ^ static_cast<uint32_t>(h)) & 1u) : 0;
            if (C::WHOLE) n_t += static_cast<uint32_t>(t_first);
            for (int t = t_first; t < nt; t += kStep) {
                const uint32_t ms = n_t % C::MSLOTS, acc = n_t & 1u;
                if (!__all_sync(0xFFFFFFFFu, ready != 0u)) {
                    ok = all_wait(&m_full[ms], (n_t / C::MSLOTS) & 1u, wc, 7);
                    if (ok) ok = all_wait(&t_full[acc], (n_t >> 1) & 1u, wc, 8);
                    if (!ok) break;
                }
                n_t += kStep;
                tc_fence_after();
                auto test_next = [&]() {
                    ready = mbar_test2(m_full0 + 8u * (n_t % C::MSLOTS), (n_t / C::MSLOTS) & 1u,
                                       t_full0 + 8u * (n_t & 1u), (n_t >> 1) & 1u);
                };
                int g = C::WHOLE ? 0 : h;   // the half of the tile
                do {
                    const float* rinv = reinterpret_cast<const float*>(sMeta + ms * C::META) + g * kGW;
                    const int* pos =
                        reinterpret_cast<const int*>(sMeta + ms * C::META + kBN * 4) + g * kGW;
                    const int c_lo = (ut.t0 + t) * kBN + g * kGW;
                    const bool band = static_cast<uint32_t>(c_lo - s0a) < s0n ||
                                      static_cast<uint32_t>(c_lo - s1a) < s1n;
                    const uint32_t taddr = tmem + lane_base + acc * kBN + static_cast<uint32_t>(g * kGW);
                    uint32_t x[kCh][32];
                    load_group(taddr, x);
                    // The tile is in registers: hand the accumulator back to the MMA warp now,
                    // so it can compute the next-but-one tile while this one is reduced.
                    tc_fence_before();
                    if (lane == 0 && (!C::WHOLE || g == kGroups - 1))
                        mbar_arrive_cluster(acc ? release1 : release0);
                    if constexpr (kSym) {
                        ready = 0;
                        // row maxima (the eager fold: the column pass already costs more than
                        // the vote saves) and each chunk's column maxima over this warp's 32
                        // rows right after it (while its registers are live)
                        uint32_t cr[4];
                        if (band) {
                            fold32_packed<true>(x[0], rinv, pos, rw, w2, mask, c_lo, b0);
                            cr[0] = colpass32<true>(x[0], pos, rw, w2, si, row_ok);
                            fold32_packed<true>(x[1], rinv + 32, pos + 32, rw, w2, mask, c_lo + 32, b0);
                            cr[1] = colpass32<true>(x[1], pos + 32, rw, w2, si, row_ok);
                            fold32_packed<true>(x[2], rinv + 64, pos + 64, rw, w2, mask, c_lo + 64, b0);
                            cr[2] = colpass32<true>(x[2], pos + 64, rw, w2, si, row_ok);
                            fold32_packed<true>(x[3], rinv + 96, pos + 96, rw, w2, mask, c_lo + 96, b0);
                            cr[3] = colpass32<true>(x[3], pos + 96, rw, w2, si, row_ok);
                        } else if (pad_item) {
                            fold32_packed<false>(x[0], rinv, pos, rw, w2, mask, c_lo, b0);
                            cr[0] = colpass32<true>(x[0], pos, rw, w2, si, row_ok);
                            fold32_packed<false>(x[1], rinv + 32, pos + 32, rw, w2, mask, c_lo + 32, b0);
                            cr[1] = colpass32<true>(x[1], pos + 32, rw, w2, si, row_ok);
                            fold32_packed<false>(x[2], rinv + 64, pos + 64, rw, w2, mask, c_lo + 64, b0);
                            cr[2] = colpass32<true>(x[2], pos + 64, rw, w2, si, row_ok);
                            fold32_packed<false>(x[3], rinv + 96, pos + 96, rw, w2, mask, c_lo + 96, b0);
                            cr[3] = colpass32<true>(x[3], pos + 96, rw, w2, si, row_ok);
                        } else {
                            fold32_packed<false>(x[0], rinv, pos, rw, w2, mask, c_lo, b0);
                            cr[0] = colpass32<false>(x[0], pos, rw, w2, si, row_ok);
                            fold32_packed<false>(x[1], rinv + 32, pos + 32, rw, w2, mask, c_lo + 32, b0);
                            cr[1] = colpass32<false>(x[1], pos + 32, rw, w2, si, row_ok);
                            fold32_packed<false>(x[2], rinv + 64, pos + 64, rw, w2, mask, c_lo + 64, b0);
                            cr[2] = colpass32<false>(x[2], pos + 64, rw, w2, si, row_ok);
                            fold32_packed<false>(x[3], rinv + 96, pos + 96, rw, w2, mask, c_lo + 96, b0);
                            cr[3] = colpass32<false>(x[3], pos + 96, rw, w2, si, row_ok);
                        }
                        // merge the four lane quarters of this group: the warps exchange their
                        // 128 column maxima, then warp q takes columns 32q .. 32q + 31
                        const int par = static_cast<int>(n_c & 1);
                        uint32_t* cb = sCB + (par * kGroups + h) * 4 * kBM;
#pragma unroll
                        for (int k = 0; k < 4; ++k) cb[q * kBM + 32 * k + lane] = cr[k];
                        mbar_arrive(&cbar[par * kGroups + h]);
                        ok = all_wait(&cbar[par * kGroups + h], (n_c >> 1) & 1, wc, 11);
                        ++n_c;
                        if (!ok) break;
                        const int c = q * 32 + lane;
                        uint32_t best = cb[c];
                        int bq = 0;
#pragma unroll
                        for (int qq = 1; qq < 4; ++qq) {
                            const uint32_t vq = cb[qq * kBM + c];
                            if ((vq & 0xFFFFFFE0u) > (best & 0xFFFFFFE0u)) {
                                best = vq;
                                bq = qq;
                            }
                        }
                        const int gcol = c_lo + c;
                        if (gcol < a.N && (best & 0xFFFFFFE0u) != 0u) {
                            const uint32_t win = static_cast<uint32_t>(r0 + 32 * bq + 31) - (best & 31u);
                            atomicMax(a.slots + static_cast<int64_t>(u) * a.N + gcol,
                                      (static_cast<unsigned long long>(best & 0xFFFFFFE0u) << 32) |
                                          (0xFFFFFFFFull - win));
                        }
                    } else if constexpr (kCount) {
                        cnt += band ? count_group<true>(x, rinv, pos, rw, w2, thr)
                                    : count_group<false>(x, rinv, pos, rw, w2, thr);
                        test_next();
                    } else {
                        if (t == ut.tr) {
                            // The evicted segment matters only where it reaches the retained
                            // one: start its running best just below this group's retained
                            // best (exact similarities decide between the two later; the
                            // FLT_MIN keeps an exact tie at 0 in play).
                            if constexpr (!kPacked) resolve_best(slot, mask, best);
                            b0 = best;
                            best = Best{b0.v - (fabsf(b0.v) * 0x1p-13f + FLT_MIN), -1};
                            if constexpr (C::PUB_BYTES != 0)
                                publish(pub + h * kBM * 4, bound_word(kNoBound, 2u * n_x + 1u));
                        }
                        if constexpr (kPacked) {
                            if (band) fold_packed<true>(x, rinv, pos, rw, w2, mask, c_lo, best);
                            else fold_packed<false>(x, rinv, pos, rw, w2, mask, c_lo, best);
                            test_next();
                        } else {
                            float v[kCh][32], m[kCh];
                            if (band) scale_group<true>(x, rinv, pos, rw, w2, v, m);
                            else scale_group<false>(x, rinv, pos, rw, w2, v, m);
                            const uint32_t stamp = 2u * n_x + (t < ut.tr ? 0u : 1u);
                            const float other = published(pub + (1 - h) * kBM * 4, stamp);
                            test_next();
                            keep_best(v, m, c_lo, slot, pub + h * kBM * 4, stamp, other, best);
                        }
                    }
                } while (C::WHOLE && ++g < kGroups);
                if (kSym && !ok) break;
                __syncwarp();
                if (lane == 0) mbar_arrive(&m_empty[ms]);
            }
            if (!ok) break;
            if (C::WHOLE) n_t = n_item + static_cast<uint32_t>(nt);
            if constexpr (!kCount && !kSym) {
                if constexpr (!kPacked) resolve_best(slot, mask, best);
                if (nt > ut.tr) b1 = best;
                else b0 = best;
            }
            // Every row's (value, column) pairs go to the merging warps.
            const int xb = static_cast<int>(n_x & 1);
            ok = all_wait(&x_empty[xb], ((n_x >> 1) & 1) ^ 1, wc, 9);
            if (!ok) break;
            sX[(xb * kGroups + h) * kBM + row_local] =
                kCount ? make_float4(cnt, 0.f, 0.f, 0.f)
                       : make_float4(b0.v, __int_as_float(b0.col), b1.v, __int_as_float(b1.col));
            mbar_arrive(&x_full[xb]);
            ++n_x;
        }
        tc_fence_before();
        cluster_barrier();
    }
}

}  // namespace

size_t audit_smem_bytes(int d)
{
    return d == 128 ? AuditCfg<128>::BYTES : AuditCfg<64>::BYTES;
}

template <int D, bool kCount, bool kSym>
cudaError_t launch_audit_t(const CUtensorMap& tmA, const CUtensorMap& tmB, const AuditArgs& a,
                           int grid, cudaStream_t st)
{
    const int bytes = AuditCfg<D, kCount, kSym>::BYTES;
    // The warpgroups' shares after setmaxnreg add up to the launch's registers: with fewer
    // than kLaunchRegs per thread the second share would never be granted.
    static std::atomic<int> regs{0};   // a property of the build; 0: not asked yet
    if (regs.load(std::memory_order_relaxed) == 0) {
        cudaFuncAttributes f;
        const cudaError_t q = cudaFuncGetAttributes(&f, audit_kernel<D, kCount, kSym>);
        if (q != cudaSuccess) return q;
        regs.store(f.numRegs, std::memory_order_relaxed);
    }
    if (regs.load(std::memory_order_relaxed) < kLaunchRegs) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(audit_kernel<D, kCount, kSym>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    return launch_dependent(audit_kernel<D, kCount, kSym>, dim3(grid), kThreads, bytes, st, tmA,
                            tmB, a);
}

cudaError_t launch_audit(int d, AuditMode mode, const CUtensorMap& tmA, const CUtensorMap& tmB,
                         const AuditArgs& a, int grid, cudaStream_t st)
{
    if (d == 128) {
        if (mode == AuditMode::kCount) return launch_audit_t<128, true, false>(tmA, tmB, a, grid, st);
        if (mode == AuditMode::kSymmetric)
            return launch_audit_t<128, false, true>(tmA, tmB, a, grid, st);
        return launch_audit_t<128, false, false>(tmA, tmB, a, grid, st);
    }
    if (mode == AuditMode::kCount) return launch_audit_t<64, true, false>(tmA, tmB, a, grid, st);
    if (mode == AuditMode::kSymmetric) return launch_audit_t<64, false, true>(tmA, tmB, a, grid, st);
    return launch_audit_t<64, false, false>(tmA, tmB, a, grid, st);
}

namespace {
// twin of every row from its slot: the low word holds 0xFFFFFFFF - position; an empty
// slot (no candidate beyond the window) gives -1
__global__ void slots_to_twins_kernel(const unsigned long long* __restrict__ slots, int64_t n,
                                      int* __restrict__ twin)
{
    wait_for_previous();
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned long long sv = slots[i];
    twin[i] = sv == 0ull ? -1 : static_cast<int>(0xFFFFFFFFull - (sv & 0xFFFFFFFFull));
}
}  // namespace

cudaError_t launch_slots_to_twins(const unsigned long long* slots, int64_t n, int* twin,
                                  cudaStream_t st)
{
    const int64_t blocks = (n + 255) / 256;
    return launch_dependent(slots_to_twins_kernel, dim3(static_cast<unsigned>(blocks)), 256, 0, st,
                            slots, n, twin);
}

// ---------------------------------------------------------------- wait probe

namespace {
__global__ void wait_probe_kernel(int* err, unsigned long long timeout_ns)
{
    __shared__ uint64_t bar;
    __shared__ uint32_t slot;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        fence_mbarrier_init();
    }
    if (threadIdx.x < 32) tmem_alloc<1>(&slot, 32);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    WaitCtl wc;
    wc.limit_ns = timeout_ns;
    wc.abort_flag = &abort_flag;
    wc.err = err;
    wc.where = 0;
    // Nothing ever arrives on `bar`: its phase 0 never completes.
    (void)mbar_wait(&bar, 0, wc, 99);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (threadIdx.x < 32) tmem_dealloc<1>(slot, 32);
}
}  // namespace

cudaError_t launch_wait_probe(int* err, unsigned long long timeout_ns, cudaStream_t st)
{
    wait_probe_kernel<<<1, 64, 0, st>>>(err, timeout_ns);
    return cudaGetLastError();
}

}  // namespace twk
