// twk_internal.h -- kernel argument blocks and launchers shared by the translation
// units of libtwinkv (host-side declarations only).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

namespace twk {

constexpr int kBM = 128;       // rows (keys i) per CTA of a pair
constexpr int kPM = 2 * kBM;   // rows per work item, a CTA pair's: the UMMA M
constexpr int kBN = 256;       // columns (keys j) per tile: the UMMA N

// Bounded waits.  A wait on work that another role of the block has to do gives up
// after the caller's limit (twinkv_set_wait_timeout_ns, never below kMinWaitLimitNs).
// After a give-up, the copies and MMAs a CTA already started are drained before it
// frees its tensor memory and exits; those drain waits use at least kDrainFloorNs,
// whatever the caller's limit, since in-flight copies and MMAs complete in
// microseconds unless the device itself is failing.
constexpr unsigned long long kMinWaitLimitNs = 10000000ull;    // 10 ms
constexpr unsigned long long kDrainFloorNs = 200000000ull;     // 200 ms

// Column stride of the per-unit column arrays (a multiple of kBN with room for the
// padding of both the retained and the evicted segment).
inline int64_t column_stride(int N) { return ((int64_t)(N + kBN - 1) / kBN) * kBN + kBN; }

struct AuditArgs {
    int U, N, NP, RB;           // units, keys per unit, column stride, kPM-row blocks per unit
    int window;                 // w, clamped to [0, N]
    int repair_mode;            // 0: one segment over the keys as given; 1: retained-first
    int need_all;               // repair mode: also scan the evicted segment
    int64_t b_rows_per_unit;    // row stride of a unit in the B tensor map
    const float* colrinv;       // [U][NP]  1/||k|| per column, NaN on padding columns
    const int* colpos;          // [U][NP]  original position of each column
    const int* cnt;             // [U][N]   retained positions before p (repair mode)
    const int* kb;              // [U]      |S0| (repair mode)
    int* out_t0;                // [U][N]   argmax of segment 0 (retained, or all in mode 0)
    int* out_t1;                // [U][N]   argmax of segment 1, the evicted columns
                                //          (repair mode with need_all), -1 if none
    int* err;
    unsigned long long timeout_ns;
    uint32_t mant_mask;         // 0xFFFFFFE0: clears the 5 mantissa bits that carry the
                                // column; a runtime value, so the compiler keeps it in a
                                // register and the pack is a single 3-input logic op
    // count mode (Eq. 2): mode 0 columns only, colrinv scaled by kCountScale;
    // out_t0/out_t1 unused
    float count_tau;            // tau, compared strictly
    int* out_count;             // [U][N] r_i
    // symmetric mode (mode 0 columns, upper-triangle tiles): per row, the best
    // candidate as (value bits with the 5 low bits cleared) << 32 | (0xFFFFFFFF - pos),
    // combined with atomicMax from both directions; zero-initialised by the caller
    unsigned long long* slots;  // [U][N]
};

enum class AuditMode { kArgmax, kCount, kSymmetric };

struct RepairArgs {
    int U, N;
    const double* b;            // [U][N] b_i(S0)
    const uint8_t* mask;        // [U][N]
    const int* budget;          // [U] or null
    double tau;                 // threshold rounded to float, widened
    int n_sink, n_recent;
    uint8_t* out_mask;          // [U][N]
    int* out_swaps;             // [U][N/2][2]
    int* out_nswaps;            // [U]
    int* out_status;            // [U] or null
    uint64_t* keys0;            // [U][N] sort buffers (ping-pong)
    int* idx0;
    uint64_t* keys1;
    int* idx1;
    // dedup variant (twin != null): a donor is not evicted together with its twin
    const int* twin;            // [U][N] argmax position of b_i(S0), or null
    int* rank_of;               // [U][N] scratch: donor rank of each position
    int cluster;                // literal variant: CTAs per unit (1, 2, 4, 8 or 16)
    bool dependent;             // launched as the programmatic dependent of the kernel before it
};

// CTAs per unit of the literal repair's selection: a power of two up to 16 (see the
// definition for where the lines lie).
int select_cluster_size(int U, int N, int sms);

// The count mode's column scales are 1/||k|| times this power of two: one saturated
// fused multiply-add per pair then gives exactly 1 or 0 (see twk_audit.cu).
constexpr float kCountScale = 0x1p32f;

// Largest N the dedup variant accepts: its walk keeps 2 bits per donor in shared memory.
constexpr int kDedupMaxN = 1 << 19;

// Every kernel that follows another one of the library on a stream is launched as its
// programmatic dependent: its blocks are set up while the last ones before it still run, and
// wait (wait_for_previous in twk_ptx.cuh) before they touch memory.  Each kernel waits at its
// start, in every thread, so that a kernel's end implies the end of all before it.  A caller's
// kernel need not do that (itself launched so, it may end while what it depends on still
// writes), so the first kernel of a call is a plain launch, ordered after everything.  A call is
// five or six kernels of 4 to 10 us on a small cache, where the gaps between them count:
// one layer 1x8x4096x128 59 -> 49 us per call, policy 16x8x3001x64 198 -> 192, redundancy
// 2x8x5003x128 125 -> 119, host repair 9x8x8192x128 1003 -> 981.
template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem,
                             cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// prep kernels
// keys: bf16 patterns, or (f32) float32, whose rounded rows also go to keys16 [U][N][d].
// NP must be a multiple of 256 (as column_stride gives).
// rscale: a power of two that multiplies every colrinv (1 except for the count mode)
// unit_kk (zeroed by the caller, or null): receives each unit's largest k.k, as float bits.
cudaError_t launch_norms_identity(const void* keys, bool f32, uint16_t* keys16, int U, int N,
                                  int d, int64_t NP, float* colrinv, int* colpos,
                                  float4* norms, cudaStream_t st, float rscale = 1.0f,
                                  unsigned* unit_kk = nullptr);
// launch_scan, launch_gather and launch_scale_columns in one kernel; *launched = false where
// the sizes are not its own.
cudaError_t launch_prep_unit(const void* keys, bool f32, uint16_t* keys16, const uint8_t* mask,
                             int* cnt, int* kb, int U, int N, int d, int64_t NP, uint16_t* kp,
                             float* colrinv, int* colpos, float4* norms, bool evicted, int sms,
                             cudaStream_t st, bool* launched);
// Also zeroes unit_kk for launch_gather.  `evicted`: the evicted segment is wanted too.
cudaError_t launch_scan(const uint8_t* mask, int U, int N, int* cnt, int* kb, unsigned* unit_kk,
                        cudaStream_t st);
cudaError_t launch_gather(const void* keys, bool f32, uint16_t* keys16, const uint8_t* mask,
                          const int* cnt, const int* kb, int U, int N, int d, int64_t NP,
                          uint16_t* kp, float* colrinv, int* colpos, float4* norms,
                          unsigned* unit_kk, bool evicted, cudaStream_t st);
// colrinv of every unit times 2^-e_u, 2^e_u the smallest power of two >= the unit's
// largest ||k|| (unit_kk as written by the kernels above), so that the audit's scaled
// similarities lie in [-1, 1] (argmax mode; not for the count mode's scales).
// kb (or null): only the retained segments.
cudaError_t launch_scale_columns(float* colrinv, int U, int64_t NP, const unsigned* unit_kk,
                                 const int* kb, cudaStream_t st);

// exact similarity of the chosen twins
// norms[r] = {k.k hi, k.k lo, 1/||k|| hi, 1/||k|| lo} (double-float pairs) per key, as
// written by the prep kernels.
// b0 = sim(i, twin0); with twin1 given (the evicted-segment winner), twin1 is
// overwritten with the overall winner and b1 (nullable) receives its similarity.
cudaError_t launch_refine(const uint16_t* keys, int U, int N, int d, const float4* norms,
                          const int* twin0, int* twin1, double* b0, double* b1,
                          cudaStream_t st,
                          bool between_audits = false);

// audit kernel (tensor maps built by the caller)
size_t audit_smem_bytes(int d);
// kArgmax: max/argmax (Eq. 1, Eq. 4); kCount: redundancy counts (Eq. 2); kSymmetric:
// max/argmax from the upper-triangle tiles only, into a.slots
cudaError_t launch_audit(int d, AuditMode mode, const CUtensorMap& tmA, const CUtensorMap& tmB,
                         const AuditArgs& a, int grid, cudaStream_t st);
// slots [n] (as the symmetric audit leaves them) -> twin positions, -1 for an empty slot
cudaError_t launch_slots_to_twins(const unsigned long long* slots, int64_t n, int* twin,
                                  cudaStream_t st);

// standalone policy selection (Sec. 3.2, Eq. 3): per unit, keep budget[u] positions
// ordered by (protected first, count ascending, position ascending)
cudaError_t launch_policy_select(const int* count, int U, int N, const int* budget, int n_sink,
                                 int n_recent, uint8_t* out_mask, int* out_status,
                                 cudaStream_t st);

// repair kernel
cudaError_t launch_repair(const RepairArgs& a, cudaStream_t st);

// wait probe (exercises the bounded-wait give-up path)
cudaError_t launch_wait_probe(int* err, unsigned long long timeout_ns, cudaStream_t st);

}  // namespace twk
