// Launchers shared between the translation units of libxfp.  Every launcher queues work on
// `stream` and returns the cudaError_t of the launch.
#pragma once
#include <cstdlib>
#include <cuda_runtime.h>

#include <atomic>

#include "xfp_common.cuh"

namespace xfp {

// Function attributes (the opt-in shared-memory size) belong to a device: every kernel instantiation remembers
// on which devices it has set them, so a process that drives several GPUs sets them on each.
// Host threads may race to the first launch: the bits are atomic (setting an attribute twice is harmless, losing
// another thread's bit is not).
struct DeviceOnce {
    std::atomic<unsigned long long> mask[4] = {};   // devices 0..255
    static int current() {
        int d = 0;
        cudaGetDevice(&d);
        return d & 255;
    }
    bool is_set(int d) const { return (mask[d >> 6].load(std::memory_order_acquire) >> (d & 63)) & 1ull; }
    void set(int d) { mask[d >> 6].fetch_or(1ull << (d & 63), std::memory_order_release); }
};

// Streaming multiprocessors of the current device, asked once per device.  Schedules (CTA slots per round, K
// splits) are built from it; workspace SIZES are a function of the descriptor alone and never depend on it.
int sm_count();
// The SM count the workspace sizes of the split-K kernels allow for: a launch never plans for more SMs than this,
// so its partial sums fit the size xfp_packed_size reported without asking a device (a B200 has 148).
constexpr int kSizingSMs = 148;
inline int sched_sms() {
    const int n = sm_count();
    return n < kSizingSMs ? n : kSizingSMs;
}

struct PackInputs {
    const uint8_t* idx;
    const uint16_t* codebook;
    const uint8_t* gid;
    const uint16_t* gscale;
    const uint16_t* gmid;
    const int32_t* rowptr;
    const void* ocol;
    int col_bits;
    const uint16_t* oval;
};

// counted: the kernel leaves the blob as it is when the last row pointer is not l.nnz
cudaError_t launch_pack(const Layout& l, const PackInputs& in, void* packed, int* err_word, cudaStream_t s, bool counted = false);
cudaError_t launch_dequant(const Layout& l, const void* packed, uint16_t* W, cudaStream_t s);
void dequant_plan_report(const Layout& l, int32_t* out);                            // for tests

// One GEMV problem set: either a single blob (packed/x/y) or n blobs through device pointer lists.
struct GemvCall {
    const void* packed;
    const uint16_t* x;
    void* y;
    const void* const* packed_list;
    const uint16_t* const* x_list;
    void* const* y_list;
    int n;          // number of problems (1 for the single form)
    int batch;      // rows of x (1..16)
    int y_is_fp16;  // type of y: 0 fp32, 1 fp16, 2 bf16
    void* workspace;
    size_t workspace_bytes;  // per problem
    int epilogue = 0;                      // XFP_EPI_* (grouped V2a launches only)
    const float* epi_weights = nullptr;    // XFP_EPI_COMBINE: [n] routing weights on the device
    int x_bf16 = 0;                        // x holds bf16 instead of fp16
};

// Split-K factor the generic kernel uses for this shape and batch tile on `sms` SMs (host-side policy).
int generic_ksplit(const Layout& l, int batch_tile, int sms);
size_t generic_workspace_bytes(const Layout& l);
cudaError_t launch_gemv_generic(const Layout& l, const GemvCall& c, cudaStream_t s);

// Fast V2 path (pair tables + mma.sync fragments); see xfp_gemv_pair.cu.
bool pair_supported(const Layout& l, int batch, int n_problems);
size_t pair_workspace_bytes(const Layout& l);
cudaError_t launch_gemv_pair(const Layout& l, const GemvCall& c, cudaStream_t s);

// Batch 1, one channel per lane, V2 and V2a; see xfp_gemv_lane.cu.
bool lane_supported(const Layout& l, const GemvCall& c);
cudaError_t launch_gemv_lane(const Layout& l, const GemvCall& c, cudaStream_t s);
// The same decode for 2..16 rows of x (tiles of 2, 4, 8 rows); see xfp_gemv_lane_batch.cu.
bool lane_batch_supported(const Layout& l, const GemvCall& c);
cudaError_t launch_gemv_lane_batch(const Layout& l, const GemvCall& c, cudaStream_t s);

// 1..16 rows of x, V2 and V2a, in the mma's own operand layout; see xfp_gemv_frag.cu.
bool frag_supported(const Layout& l, const GemvCall& c);
cudaError_t launch_gemv_frag(const Layout& l, const GemvCall& c, cudaStream_t s);

// Fast V2a path (per-bank library + mma.sync fragments, one or several blobs); see xfp_gemv_v2a.cu.
bool v2a_supported(const Layout& l, int batch);
size_t v2a_workspace_bytes(const Layout& l);
cudaError_t launch_gemv_v2a(const Layout& l, const GemvCall& c, cudaStream_t s);
// Of these the fused stores of a routed expert block at N <= 4; see xfp_gemv_expert.cu.
bool expert_supported(const Layout& l, const GemvCall& c);
cudaError_t launch_gemv_expert(const Layout& l, const GemvCall& c, cudaStream_t s);

// Batched path (3..16 rows of x), V2 and V2a; see xfp_gemv_batch.cu.
bool batch_supported(const Layout& l, int batch);
cudaError_t launch_gemv_batch(const Layout& l, const GemvCall& c, cudaStream_t s);

// Prefill form on the tcgen05 tensor cores (V2 and V2a, up to 64 rows of x); see xfp_gemm_tc.cu.
struct GemmCall {
    const void* packed;
    const uint16_t* x;   // [M][cols] fp16
    void* y;             // [M][rows]
    int M;
    int y_kind;          // 0 fp32, 1 fp16, 2 bf16
    void* workspace;
    size_t workspace_bytes;
    int short_cta = -1;  // tests of the pair kernel's failure path: the CTA whose bounded waits give up at once
};
bool gemm_tc_supported(const Layout& l, int M);
// The counters of both prefill kernels: one region at the start of the workspace whose size does not depend on the rows of x, so
// that calls of different rows may share a workspace (what one call keeps as a sum must not lie where another counts).  An error
// word, then the larger of two words per dealt tile of the pair kernel (fewer tiles than pairs of SMs) and one per tile of 128
// channels of the 64-row kernel; and the counters of the GEMV kernels, whose workspace a batch brings along.
inline size_t prefill_ctrl_bytes(const Layout& l) {
    const int tiles = (l.RB + 3) / 4;
    const size_t own = align256(4 * (size_t)(1 + (tiles > kSizingSMs ? tiles : kSizingSMs))), tickets = align256((size_t)l.RB * 4);
    return own > tickets ? own : tickets;
}
size_t gemm_core_bytes(const Layout& l, int M);        // counters and the partial sums of K slices
size_t gemm_xt_bytes(const Layout& l, int M);          // the transposed copy of x of the sparse outlier product (0: not used)
size_t gemm_xt_offset(const Layout& l, int M);         // where that copy starts in the workspace
size_t gemm_workspace_bytes(const Layout& l, int M);   // all of it
cudaError_t launch_gemm_tc(const Layout& l, const GemmCall& c, cudaStream_t s);
// bf16 activations: converted to fp16 into a scratch area behind the GEMM's own workspace, then the same kernel
size_t gemm_x_scratch_bytes(const Layout& l, int M);
cudaError_t launch_x_to_f16(const void* x_bf16, void* x_f16, size_t elems, cudaStream_t s);

// The prefill form for many rows of x on pairs of SMs; see xfp_gemm_fused.cu.
bool fused_preferred(const Layout& l, int M);          // which of the two kernels xfp_gemm takes
size_t fused_workspace_bytes(const Layout& l, int M);
cudaError_t launch_gemm_fused(const Layout& l, const GemmCall& c, void* x_f16, cudaStream_t s);
void fused_plan_report(const Layout& l, int M, int64_t* out);                       // for tests
int fused_piece_report(const Layout& l, int M, int g, int i, int32_t* out);         // for tests
// what a call of M rows uses
inline size_t prefill_workspace_bytes(const Layout& l, int M) {
    return fused_preferred(l, M) ? fused_workspace_bytes(l, M) : gemm_workspace_bytes(l, M);
}
// what the caller is asked for: enough for a call of any number of rows up to M (what a call uses neither grows nor falls with M)
size_t prefill_workspace_for_up_to(const Layout& l, int M);

// Batches of 9..16 rows of fp16 x run on the tensor-core kernel (xfp_gemm_tc.cu) when the matrix is large and the blob
// sparse in outliers: the tcgen05 kernel decodes once for all rows (measurements at batch_prefers_gemm).
// Layout of a GEMV workspace, shared by every kernel that may be given it: counters (split-K tickets, one int per
// row-block and blob at most) in [0, align256(4 * RB * n)), zero-filled before first use and left zero-filled by every
// call; partial sums behind it, written before they are read.
// matrices with more tiles of 128 channels than SMs: batches of 9..16 rows of x may go to the tensor-core kernel
inline bool gemm_batch_shape(const Layout& l) { return (l.RB + 3) / 4 > kSizingSMs && gemm_tc_supported(l, 16); }

inline size_t workspace_bytes_for(const Layout& l) {
    size_t w = generic_workspace_bytes(l);
    const size_t p = l.mode ? v2a_workspace_bytes(l) : pair_workspace_bytes(l);
    if (p > w) w = p;
    // room for that kernel's partial sums and its transposed copy of x at 16 rows
    const size_t g = gemm_batch_shape(l) ? gemm_workspace_bytes(l, 16) : 0;
    return w > g ? w : g;
}

inline bool batch_prefers_gemm(const Layout& l, int batch) {
    // 28672 x 8192, us per call, tensor-core kernel against xfp_gemv_frag.cu (0.3 % outliers):
    //   9..16 rows: V2 N = 4 78 against 107
    //   5..8 rows:  where xfp_gemv_frag.cu (68..77) does not take the blob (V2a in groups of 64 weights): V2a 102 against 123,
    //               V2 N = 6 98 against 115
    int least = ((l.mode || l.bits >= 5) && l.nnz * 100 <= (long long)l.rows * l.cols) ? 5 : 9;
#ifdef LANE_TUNE
    if (const char* e = getenv("XFP_GEMM_MIN")) least = atoi(e);
#endif
    if (batch < least || batch > 16 || !gemm_batch_shape(l)) return false;
    // at most 2.5 % outliers: the kernel adds them as a sparse product whose cost grows with their count
    return l.nnz * 40 <= (long long)l.rows * l.cols;
}

}  // namespace xfp
