// Prefill form in two steps: W^ = fp16(D16 + S) decoded once into GEMM tiles (xfp_dequant.cu) in the call's workspace, then a
// dense tcgen05 GEMM  y[t][i] = sum_k W^[i][k] x[t][k]  on them, both operands from shared memory.
//
// The kernel of xfp_gemm_tc.cu decodes inside the GEMM and so decodes the weights once per 256 rows of x, with the outliers
// walked or multiplied per tile; it is bound by that decode (28672 x 8192, 1024 rows, 0.3 %: 614 us, of which the products
// need 300).  Decoding once costs a pass over 2 bytes per weight instead, which stays in L2 when the matrix is cut into
// chunks of row tiles: two chunk buffers take turns, and the decode of the next chunk runs on the SMs' CUDA cores beside
// the products of the current one (programmatic dependent launches).
//
//   pair      two CTAs (a cluster, tcgen05 cta_group::2) share a tile of 256 channels x T rows of x (T <= 256): each stages
//             its own 128 channels of W^ (16 KB per 64 k, one bulk copy: a tile is contiguous, in core-matrix order) and
//             half of the rows of x (one tensor copy, 128-byte swizzle); the first CTA issues the products of both.  A tile of
//             128 x 256 per CTA would read half as much again from L2 (96 bytes per clock and SM at full product rate).
//   CTA       a thread that issues the copies, a thread that issues the products (in the second CTA: that passes on to the
//             first that a stage has landed), four warps for the epilogue.
//   schedule  many tiles: resident pairs walk them, two accumulators in tensor memory take turns so that a tile's epilogue
//             runs under the next one's products.  Few tiles: a cluster of 2 or 4 pairs cuts the tile along K; the partial
//             sums meet through distributed shared memory, added in slice order.
// Waits on barriers have an iteration limit; when one runs out the CTA records it in the first word of the workspace.
#include <cuda.h>

#include "xfp_internal.h"

namespace xfp {

namespace {

constexpr int kRows = 128;                     // channels of a tile
constexpr int kStageK = 64;
constexpr int kABytes = kRows * kStageK * 2;   // one A stage
constexpr int kMaxStages = 10;
constexpr int kDenseThreads = 192;             // copy warp, product warp, four epilogue warps
constexpr uint32_t kSpins = 1u << 20, kPollHint = 1000;
constexpr size_t kDenseSmem = 225 * 1024;      // dynamic shared memory of a CTA

struct DenseArgs {
    const unsigned char* tiles;   // [row tile][k / 64][16 KB]
    void* y;
    int* ctrl;                    // [0] error word
    int M, rows, KT;              // KT: stages along K
    int row0;                     // first channel of this launch
    int pair_tiles, tok_tiles, T; // tiles of 256 channels, tiles of T rows of x
    int stages, b_bytes;          // bytes of one x stage
    int ks, kt_slice;             // pairs of a cluster along K, stages of each
    int y_kind, tmem_cols;
};

__device__ __forceinline__ uint32_t sa(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity) {
    for (uint32_t i = 0; i < kSpins; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity), "r"(kPollHint) : "memory");
        if (ok) return true;
    }
    return false;
}
// one lane of a converged warp: instructions that take uniform registers are then issued by one thread as the compiler
// sees it (behind a plain lane == 0 it serialises over the lanes it cannot rule out)
__device__ __forceinline__ bool elected() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// the same barrier (or address) in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(bar) : "memory");
}
// K-major operand descriptors (version 1).  A: core matrices of 8 rows x 16 bytes, the next 8 k 2048 bytes on, the next 8
// rows 128 bytes on, no swizzle.  B: rows of 128 bytes in the 128-byte swizzle, 8 rows 1024 bytes.
__device__ __forceinline__ uint64_t desc_a(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)(2048 >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ uint64_t desc_b(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void mma_ss(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :: "r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
// the products issued so far arrive on the barrier of both CTAs of the pair
__device__ __forceinline__ void commit(uint32_t bar, uint32_t mask) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(bar), "h"((uint16_t)mask) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// SPLIT: a cluster of a.ks pairs per tile, one tile per cluster; else resident pairs walk the tiles.
template <bool SPLIT>
__global__ void __launch_bounds__(kDenseThreads, 1) gemm_dense_kernel(const DenseArgs a, const __grid_constant__ CUtensorMap tmap) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (sa(smem_raw) & 1023u)) & 1023u);    // the same offset in every CTA
    __shared__ __align__(8) uint64_t full[kMaxStages], both[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t crank = cluster_rank(), h = crank & 1u, lead = crank & ~1u;        // half of the pair, its first CTA
    const int slice = (int)(crank >> 1);
    const int first = SPLIT ? (int)blockIdx.x / (2 * a.ks) : (int)blockIdx.x >> 1, step = SPLIT ? 1 << 30 : (int)gridDim.x >> 1;
    const int tiles = a.pair_tiles * a.tok_tiles;
    const int k0 = slice * a.kt_slice, k1 = min(a.KT, k0 + a.kt_slice);
    const uint32_t pair_mask = 3u << lead;
    unsigned char* sA = smem;
    unsigned char* sB = smem + (size_t)a.stages * kABytes;

    if (tid == 0) {
        for (int i = 0; i < a.stages; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sa(&full[i])));      // this CTA's stage has landed
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sa(&both[i])));      // the other CTA's too (in the first CTA)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sa(&empty[i])));     // its products are done
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(sa(&acc_full[i])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" :: "r"(sa(&acc_empty[i]))); // four epilogue warps of each CTA
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(sa(&s_tmem)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();                                          // every CTA's barriers exist
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t half = (uint32_t)a.tmem_cols >> 1;        // columns of one accumulator (when two take turns)

    // Each role is a whole warp in uniform control flow; one elected lane issues.
    bool ok = true;
    if (warp == 0) {
        // The tiles come from the previous kernel of the stream.  Dependents are released only now: a decode of the next
        // chunk then starts when the GEMM before this one, which reads the buffer it writes, is known to be over.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;");
        int s = 0;
        uint32_t ph = 1;                                     // "empty" passes at once in the first round
        for (int t = first; t < tiles && ok; t += step) {
            const int tx = t / a.tok_tiles, ty = t % a.tok_tiles, t0 = ty * a.T, Tn = min(a.T, (a.M - t0 + 15) & ~15);
            const unsigned char* src = a.tiles + ((size_t)(2 * tx + (int)h) * a.KT + k0) * kABytes;
            const int xrow = t0 + (int)h * (Tn >> 1);
            for (int k = k0; k < k1; ++k, src += kABytes) {
                if (!(ok = wait_bar(sa(&empty[s]), ph))) break;
                if (elected()) {
                    const uint32_t bar = sa(&full[s]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"((uint32_t)(kABytes + a.b_bytes)) : "memory");
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 :: "r"(sa(sA) + (uint32_t)(s * kABytes)), "l"(src), "r"(kABytes), "r"(bar) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 :: "r"(sa(sB) + (uint32_t)(s * a.b_bytes)), "l"(&tmap), "r"(k * kStageK), "r"(xrow), "r"(bar) : "memory");
                }
                __syncwarp();
                if (++s == a.stages) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 1 && h == 1) {                        // the second CTA: tell the first that this stage has landed
        int s = 0;
        uint32_t ph = 0;
        for (int t = first; t < tiles && ok; t += step) {
            for (int k = k0; k < k1; ++k) {
                if (!(ok = wait_bar(sa(&full[s]), ph))) break;
                if (elected()) arrive_cluster(peer(sa(&both[s]), lead));
                __syncwarp();
                if (++s == a.stages) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 1) {
        int s = 0, n = 0;
        uint32_t ph = 0;
        const uint64_t da0 = desc_a(sa(sA)), db0 = desc_b(sa(sB));     // a stage on: the start address field moves
        for (int t = first; t < tiles && ok; t += step, ++n) {
            const int ty = t % a.tok_tiles, Tn = min(a.T, (a.M - ty * a.T + 15) & ~15);
            const uint32_t idesc = (1u << 4) | ((uint32_t)(Tn >> 3) << 17) | ((uint32_t)(2 * kRows >> 4) << 24);
            const int buf = SPLIT ? 0 : n & 1;
            const uint32_t d = tmem + (uint32_t)buf * half;
            if (!SPLIT && !(ok = wait_bar(sa(&acc_empty[buf]), (uint32_t)((n >> 1) & 1) ^ 1u))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int k = k0; k < k1; ++k) {
                if (!(ok = wait_bar(sa(&full[s]), ph) && wait_bar(sa(&both[s]), ph))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (elected()) {
                    const uint64_t da = da0 + (uint64_t)((uint32_t)(s * kABytes) >> 4), db = db0 + (uint64_t)((uint32_t)(s * a.b_bytes) >> 4);
#pragma unroll
                    for (int i = 0; i < kStageK / 16; ++i) mma_ss(d, da + i * 256, db + i * 2, idesc, (k > k0 || i > 0) ? 1u : 0u);
                    commit(sa(&empty[s]), pair_mask);
                    if (k + 1 == k1) commit(sa(&acc_full[buf]), pair_mask);
                }
                __syncwarp();
                if (++s == a.stages) { s = 0; ph ^= 1u; }
            }
        }
    } else {
        const int q = warp & 3;                              // the warp's quarter of the tensor-memory lanes
        const int r = q * 32 + lane;
        int n = 0;
        for (int t = first; t < tiles && ok; t += step, ++n) {
            const int tx = t / a.tok_tiles, ty = t % a.tok_tiles, t0 = ty * a.T, Tn = min(a.T, (a.M - t0 + 15) & ~15);
            const int buf = SPLIT ? 0 : n & 1;
            ok = wait_bar(sa(&acc_full[buf]), (uint32_t)(n >> 1) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int row = a.row0 + (2 * tx + (int)h) * kRows + r;
            for (int c = 0; c * 16 < Tn; ++c) {
                uint32_t v[16];
                tmem_ld16(tmem + (uint32_t)buf * half + ((uint32_t)(q * 32) << 16) + (uint32_t)(c * 16), v);
                if (SPLIT) {
                    // every product of the pair is complete, its stages are free: the partial sums go there, [t][channel]
                    float* p = (float*)smem + (size_t)c * 16 * kRows + r;
#pragma unroll
                    for (int j = 0; j < 16; ++j) p[(size_t)j * kRows] = __uint_as_float(v[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (t0 + c * 16 + j < a.M && row < a.rows)
                            put_y(a.y, (size_t)(t0 + c * 16 + j) * a.rows + row, __uint_as_float(v[j]), a.y_kind);
                }
            }
            if (!SPLIT) {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive_cluster(peer(sa(&acc_empty[buf]), lead));
            }
        }
    }
    if (!ok) { s_fail = 1; atomicExch(a.ctrl, 1); }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (s_fail && tid == 0)      // copies in flight land before the CTA goes
        for (int i = 0; i < a.stages; ++i) wait_bar(sa(&full[i]), 0);
    __syncwarp();
    cluster_sync();
    if (SPLIT) {
        // this CTA's share of the rows of x of its 128 channels: the slices' sums added in slice order
        if (first < tiles) {
            const int tx = first / a.tok_tiles, ty = first % a.tok_tiles, t0 = ty * a.T, Tn = min(a.T, a.M - t0);
            const int share = (Tn + a.ks - 1) / a.ks, b0 = slice * share, b1 = min(Tn, b0 + share);
            const uint32_t own = sa(smem);
            for (int i = b0 * (kRows / 4) + tid; i < b1 * (kRows / 4); i += kDenseThreads) {
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int z = 0; z < a.ks; ++z) {
                    float4 v;
                    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(peer(own + (uint32_t)i * 16u, 2u * z + h)));
                    sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
                }
                const int tt = t0 + i / (kRows / 4), row = a.row0 + (2 * tx + (int)h) * kRows + (i % (kRows / 4)) * 4;
                const size_t o = (size_t)tt * a.rows + row;
                if (row < a.rows) put_y(a.y, o, sum.x, a.y_kind);
                if (row + 1 < a.rows) put_y(a.y, o + 1, sum.y, a.y_kind);
                if (row + 2 < a.rows) put_y(a.y, o + 2, sum.z, a.y_kind);
                if (row + 3 < a.rows) put_y(a.y, o + 3, sum.w, a.y_kind);
            }
        }
        __syncwarp();
        cluster_sync();          // no CTA leaves while another reads its shared memory
    }
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(a.tmem_cols) : "memory");
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn() {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
        return nullptr;
    return (EncodeTiledFn)fn;
}

// ------------------------------------------------------------------ plan

struct DensePlan {
    int T, tok_tiles;          // rows of x per tile
    int pairs, chunk, chunks;  // tiles of 256 channels: of the matrix, of a chunk; number of chunks
    int ks, kt_slice;          // pairs per tile along K
    int stages;
    size_t smem, buffer;       // bytes of a CTA's shared memory, of one chunk's tiles
    double us;                 // what the model expects
};

constexpr double kDecodeWeightsPerUs = 4.0e6;   // decode into tiles, alone on the GPU
constexpr size_t kScratchMax = size_t(160) << 20;   // chunk buffers in all: they should stay in L2

// us of one chunk's products: pairs x tok_tiles tiles of `stages` 64-k steps.  A step takes the products' clocks (2 T), or
// the time its operands take to arrive from L2 (16 KB of W^ and T / 2 rows of x per CTA at about 50 bytes per clock).
double gemm_us(int tiles, int T, int KT, int ks) {
    const double feed = (16384.0 + 64.0 * T) / 50.0, step = feed > 2.0 * T ? feed : 2.0 * T;
    const int slots = ks == 1 ? 74 : ks == 2 ? 34 : 16;     // clusters of 2, 4, 8 CTAs that run at once
    const int waves = (tiles + slots - 1) / slots;
    const double clocks = waves * (double)((KT + ks - 1) / ks) * step + (ks > 1 ? waves * (1500.0 + 12.0 * T) : 1500.0 + 8.0 * T);
    return clocks / 1800.0 + 3.0;
}

DensePlan plan_dense(const Layout& l, int M) {
    DensePlan best = {};
    const int KT = l.cols / kStageK, pairs = (l.RB + 7) / 8;
    const size_t pair_bytes = (size_t)2 * KT * kABytes;
    const double decode_us = (double)l.rows * l.cols / kDecodeWeightsPerUs;
    int last_T = 0;
    for (int n = (M + 255) / 256; n <= (M + 15) / 16; ++n) {           // tiles along the rows of x
        const int T = ((M + n - 1) / n + 15) & ~15;
        if (T == last_T) continue;
        last_T = T;
        if (T < 64 && n > (M + 255) / 256) break;
        const int tok = (M + T - 1) / T;
        for (int chunks = 1; chunks <= 16 && chunks <= pairs; ++chunks) {
            const int chunk = (pairs + chunks - 1) / chunks, nch = (pairs + chunk - 1) / chunk;
            if (nch != chunks) continue;
            if ((size_t)chunk * pair_bytes * (nch > 1 ? 2 : 1) > kScratchMax && chunks < 16 && chunk > 1) continue;
            for (int ks = 1; ks <= 4; ks *= 2) {
                if (ks > 1 && ((KT + ks - 1) / ks < 4 || (ks - 1) * ((KT + ks - 1) / ks) >= KT)) break;
                const double d = decode_us * chunk / pairs, g = gemm_us(chunk * tok, T, KT, ks);
                const int rest = pairs - chunk * (nch - 1);
                const double last = gemm_us(rest * tok, T, KT, ks);
                const double us = d + 2.5 + (nch - 1) * ((g > d ? g : d) * (nch > 1 ? 1.08 : 1.0)) + last;
                if (best.us == 0.0 || us < best.us) {
                    best.T = T; best.tok_tiles = tok; best.pairs = pairs; best.chunk = chunk; best.chunks = nch;
                    best.ks = ks; best.kt_slice = (KT + ks - 1) / ks; best.us = us; best.buffer = (size_t)chunk * pair_bytes;
                }
            }
        }
    }
    const int stage = kABytes + best.T * 64;
    // the partial sums of a cut tile take the stages' place; beside the CTA two blocks of the decode fit on the SM
    int stages = (int)((196 * 1024) / stage);
    if (stages > kMaxStages) stages = kMaxStages;
    best.stages = stages;
    best.smem = (size_t)stages * stage + 1024;
    if (best.ks > 1 && best.smem < (size_t)best.T * kRows * 4 + 1024) best.smem = (size_t)best.T * kRows * 4 + 1024;
    return best;
}

size_t dense_ctrl_bytes(const Layout& l, int M) { return gemm_ctrl_bytes(l, M); }

}  // namespace

bool dense_preferred(const Layout& l, int M) {
    if (!gemm_tc_supported(l, M)) return false;
#ifdef LANE_TUNE
    if (const char* e = getenv("XFP_DENSE")) return atoi(e) != 0;
#endif
    return M > 64;
}

size_t dense_workspace_bytes(const Layout& l, int M) {
    const DensePlan p = plan_dense(l, M);
    return dense_ctrl_bytes(l, M) + p.buffer * (p.chunks > 1 ? 2 : 1);
}

// c.x: the activations (bf16 when x_f16 is given: converted there on the way)
cudaError_t launch_gemm_dense(const Layout& l, const GemmCall& c, void* x_f16, cudaStream_t s) {
    const DensePlan p = plan_dense(l, c.M);
    static const EncodeTiledFn encode = encode_fn();
    if (!encode) return cudaErrorNotSupported;
    const void* x = x_f16 ? x_f16 : (const void*)c.x;
    CUtensorMap tmap;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)l.cols, (cuuint64_t)c.M};
        const cuuint64_t strides[1] = {(cuuint64_t)l.cols * 2};
        const cuuint32_t box[2] = {64, (cuuint32_t)(p.T / 2)};
        const cuuint32_t estr[2] = {1, 1};
        if (encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(x), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        cudaError_t e = cudaFuncSetAttribute(gemm_dense_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDenseSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_dense_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDenseSmem);
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    unsigned char* buf0 = (unsigned char*)c.workspace + dense_ctrl_bytes(l, c.M);
    DenseArgs a = {};
    a.y = c.y; a.ctrl = (int*)c.workspace; a.M = c.M; a.rows = l.rows; a.KT = l.cols / kStageK;
    a.tok_tiles = p.tok_tiles; a.T = p.T; a.stages = p.stages; a.b_bytes = p.T * 64;
    a.ks = p.ks; a.kt_slice = p.kt_slice; a.y_kind = c.y_kind;
    a.tmem_cols = p.ks > 1 ? (p.T <= 32 ? 32 : p.T <= 64 ? 64 : p.T <= 128 ? 128 : 256) : (p.T <= 128 ? 256 : 512);
    const int pair_slots = sm_count() / 2;
    for (int i = 0; i < p.chunks; ++i) {
        const int pair0 = i * p.chunk, n = p.pairs - pair0 < p.chunk ? p.pairs - pair0 : p.chunk;
        const int rb0 = pair0 * 8, n_rb = l.RB - rb0 < n * 8 ? l.RB - rb0 : n * 8;
        unsigned char* buf = buf0 + (size_t)(i & 1) * p.buffer;
        cudaError_t e = launch_decode_tiles(l, c.packed, rb0, n_rb, (uint16_t*)buf, i == 0 && x_f16 ? c.x : nullptr, x_f16,
                                            (size_t)c.M * l.cols / 8, i > 0, s);
        if (e != cudaSuccess) return e;
        a.tiles = buf; a.row0 = pair0 * 256; a.pair_tiles = n;
        const int tiles = n * p.tok_tiles, ctas = p.ks > 1 ? tiles * 2 * p.ks : 2 * (tiles < pair_slots ? tiles : pair_slots);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ctas, 1, 1);
        cfg.blockDim = dim3(kDenseThreads, 1, 1);
        cfg.dynamicSmemBytes = p.smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)(2 * p.ks); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        e = p.ks > 1 ? cudaLaunchKernelEx(&cfg, gemm_dense_kernel<true>, a, tmap) : cudaLaunchKernelEx(&cfg, gemm_dense_kernel<false>, a, tmap);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace xfp
