// The routed expert block's two grouped launches with fused stores (V2a, N <= 4, one row of x):
//   XFP_EPI_SWIGLU    h_j = SiLU(gate) * up for every expert j of a token
//   XFP_EPI_COMBINE   y = sum_j w_j W_j h_j
//
// The decode is that of the lane kernel (xfp_gemv_lane.cu): one channel per lane, the codebook of the lane's group in registers as
// byte planes, the decoded words as the A fragment of mma.sync.m16n8k16 with x on the diagonal lanes of the B fragment, groups
// folded with their scale and mid-point.  What is dealt differs:
//   SWIGLU    a CTA of 8 warps owns a block of 64 channels of one expert (32 gates and the 32 matching up channels); warps of even
//             number take the gates' row-block, the others the up channels'.  Three CTAs per SM (80 registers): the 384 blocks of 8
//             experts of 3072 x 4096 are resident at once, where 296 resident CTAs with two channels per lane left most SMs waiting
//             for those with a second block.
//   COMBINE   a CTA of 16 or 8 warps (combine_plan) owns one row-block of 32 channels of ALL experts (or of a run of them): (expert, super-chunk) units
//             are dealt to the warps in one sequence, so that short rows (12 super-chunks) leave no warp idle and the experts cost
//             one staging of x, one reduction and no barrier between them.  A lane's sum of one expert is scaled by its weight when
//             the expert ends.  Runs of a row-block meet through the workspace in run order; one run per row-block needs none.
// Eight experts, us for both launches (two channels per lane with tables -> this): 4096 x 1536 N = 3 45.0 -> 34.7, N = 2 42.3 -> 30.8,
// N = 4 60.5 -> 44.9; 7168 x 2048 N = 3 93.7 -> 75.  A few weighted sums of two to five short experts are still 3 - 12 % behind the
// tables (3 of 5120 x 1536 N = 4 13.0 -> 14.6, 5 of 3200 x 2048 N = 4 14.6 -> 15.2).
// Bound by the ALU pipe in the K loop (PRMT and the selectors), around it by the chain pointer list - blob - first indices and the
// staging of x behind the dependency wait.
#include <algorithm>

#include "xfp_internal.h"
#include "xfp_pair_common.cuh"
#include "xfp_reg_decode.cuh"

namespace xfp {

namespace {

constexpr int kExpertBlobs = 32;                        // blobs of a CTA at most
constexpr size_t kExpertSmemOne = 200 * 1024, kExpertSmemTwo = 80 * 1024, kExpertSmemThree = 72 * 1024;

struct ExpertArgs {
    Offsets off;
    const void* const* packed_list;
    const uint16_t* const* x_list;
    void* const* y_list;
    const float* epi_w;      // COMBINE: [n] weights
    float* partial;          // COMBINE: [run][rows_ws]
    int* tickets;            // COMBINE: [row-block]
    int rows, RB, SC, L, n, rows_ws;
    int y_kind, x_bf16;
    int blocks;              // SWIGLU: blocks of 64 channels of one blob
    int G, ng;               // COMBINE: runs per row-block, blobs per run
    int tab_bytes;           // byte planes of one library
};

// 16 bytes of staged x for the diagonal lanes of the B fragment; the other lanes keep their zeros (see xfp_gemv_lane.cuh).
__device__ __forceinline__ void ld_x16(uint4& v, uint32_t addr, uint32_t take) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t@p ld.shared.v4.u32 {%0,%1,%2,%3}, [%5];\n\t}"
        : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w)
        : "r"(take), "r"(addr));
}

// R row-blocks of a CTA (2: SWIGLU, 1: COMBINE); W warps, W / R of them per row-block
template <int N, int W, int R, int MINB>
__global__ void __launch_bounds__(W * 32, MINB) gemv_expert_kernel(const ExpertArgs a) {
    constexpr bool kCombine = R == 1;
    constexpr int KW = W / R, E = 1 << N, kThreads = W * 32;
    constexpr bool kEvenOdd = N == 2;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ const char* s_blob[kExpertBlobs];
    __shared__ const uint32_t* s_ell[kExpertBlobs];
    __shared__ const uint16_t* s_x[kExpertBlobs];
    __shared__ int s_slots[kExpertBlobs], s_width[kExpertBlobs][R];
    __shared__ float s_w[kExpertBlobs];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, kw = warp / R, rl = warp % R;
    asm volatile("griddepcontrol.launch_dependents;");
    const int K = a.SC * kSuper;
    // ---- what this CTA owns: blobs [j0, j0 + nb), row-block rb of this warp
    int j0, nb, blk, run = 0;
    if (kCombine) {
        blk = (int)blockIdx.x / a.G; run = (int)blockIdx.x % a.G;
        j0 = run * a.ng; nb = min(a.ng, a.n - j0);
    } else {
        j0 = (int)blockIdx.x / a.blocks; blk = (int)blockIdx.x % a.blocks; nb = 1;
    }
    const int rb = blk * R + rl;
    const int most = kCombine ? a.ng : 1;                 // blobs that the shared-memory regions are laid out for
    unsigned char* planes = smem;                                        // [most][tab_bytes]
    unsigned char* xs = smem + (size_t)most * a.tab_bytes;               // [most][K] fp16, permuted
    float* xg = (float*)(xs + (size_t)most * K * 2);                     // [most][SC][2] sums of x over half super-chunks
    float* red = xg + (size_t)most * a.SC * 2;                           // [W][32]

    // ---- loads that do not depend on earlier kernels: this warp's first indices, the blobs' geometry, libraries
    // the warp's units: (blob jb, super-chunk s), KW apart in the sequence of all (blob, super-chunk)
    int jb = 0, s = kw;
    while (s >= a.SC) { s -= a.SC; ++jb; }
    uint32_t w[4 * N + 1];
    w[4 * N] = 0u;
    uint32_t id = 0u, sm = 0u;
    if (jb < nb) {
        const char* p = (const char*)a.packed_list[j0 + jb];
        const size_t unit = (size_t)rb * a.SC + s;
        const uint4* ip = (const uint4*)(p + a.off.idx) + unit * N * 32 + lane;
#pragma unroll
        for (int v = 0; v < N; ++v) {
            const uint4 t = ld_stream(ip + v * 32);
            w[4 * v] = t.x; w[4 * v + 1] = t.y; w[4 * v + 2] = t.z; w[4 * v + 3] = t.w;
        }
        id = ((const uint8_t*)(p + a.off.gid))[unit * 32 + lane];
        sm = ((const uint32_t*)(p + a.off.gsm))[unit * 32 + lane];
    }
    if (tid < nb) {
        const char* p = (const char*)a.packed_list[j0 + tid];
        const int* hdr = (const int*)(p + a.off.hdr);
        s_blob[tid] = p;
        s_x[tid] = a.x_list[j0 + tid];
        s_slots[tid] = __ldg(hdr);
        s_ell[tid] = (const uint32_t*)(p + *(const long long*)(hdr + 2));
    }
    for (int i = tid; i < nb * a.L; i += kThreads) {
        const int j = i / a.L, l = i - j * a.L;
        store_book<N>(planes + (size_t)j * a.tab_bytes, a.L, l, make_book<N>((const uint16_t*)((const char*)a.packed_list[j0 + j] + a.off.cb) + (size_t)l * E));
    }
    __syncthreads();                                   // the blobs' geometry
    // the widest channel of every blob's row-block (outlier slots to walk): loaded here, looked at behind the staging of x
    auto slots_used = [&](int j) {
        const int q = j / R, slots = s_slots[q];
        return slots ? __ldg(s_ell[q] + (size_t)(blk * R + j % R) * (slots + 1) * 32 + lane) : 0u;
    };
    uint32_t len = warp < nb * R ? slots_used(warp) : 0u;

    // ---- x and the weights may come from the previous kernel of the stream
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (kCombine && tid < nb) s_w[tid] = __ldg(a.epi_w + j0 + tid);
    {
        const int vec = K / 8, all = nb * vec;
        for (int t = tid; t < ((all + 31) & ~31); t += kThreads) {         // whole warps: the sums below shuffle
            const bool in = t < all;
            const int j = in ? t / vec : 0, k8 = t - j * vec;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (in) v = x8_as_f16(__ldg((const uint4*)s_x[j] + k8), a.x_bf16);
            if (in) {
                unsigned char* xd = xs + (size_t)j * K * 2;
                const uint2 p = kEvenOdd ? make_uint2(prmt(v.x, v.y, 0x5410u), prmt(v.z, v.w, 0x5410u)) : make_uint2(v.x, v.y);
                const uint2 q = kEvenOdd ? make_uint2(prmt(v.x, v.y, 0x7632u), prmt(v.z, v.w, 0x7632u)) : make_uint2(v.z, v.w);
                *(uint2*)(xd + xpos_of<kEvenOdd>(8u * k8) * 2) = p;
                *(uint2*)(xd + xpos_of<kEvenOdd>(8u * k8 + (kEvenOdd ? 1u : 4u)) * 2) = q;
            }
            // 8 consecutive threads hold 64 consecutive k (a blob's K is a multiple of 128)
            const float2 p0 = __half22float2(*(const __half2*)&v.x), p1 = __half22float2(*(const __half2*)&v.y);
            const float2 p2 = __half22float2(*(const __half2*)&v.z), p3 = __half22float2(*(const __half2*)&v.w);
            float sx = ((p0.x + p0.y) + (p1.x + p1.y)) + ((p2.x + p2.y) + (p3.x + p3.y));
            sx += __shfl_xor_sync(0xffffffffu, sx, 1);
            sx += __shfl_xor_sync(0xffffffffu, sx, 2);
            sx += __shfl_xor_sync(0xffffffffu, sx, 4);
            if (in && (t & 7) == 0) xg[t >> 3] = sx;
        }
    }
    for (int j = warp; j < nb * R; j += W) {
        if (j != warp) len = slots_used(j);
        const int m = __reduce_max_sync(0xffffffffu, (int)len);
        if (lane == 0) s_width[j / R][j % R] = m;
    }
    __syncthreads();

    // ---- K loop: 16 mma steps per unit; an index vector is reloaded with the warp's next unit when its last step is decoded
    const int g = lane >> 2, t4 = lane & 3;
    const uint32_t dq = (g == t4) || (g == t4 + 4);
    const uint32_t xlane = (uint32_t)__cvta_generic_to_shared(xs) + ((g == t4 + 4) ? 16u : 0u);
    const int src_a = (lane & ~3) | (t4 >> 1);
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    float acc = 0.f, total = 0.f;       // of the current blob; weighted over the blobs
    while (jb < nb) {
        int jn = jb, sn = s + KW;
        while (sn >= a.SC) { sn -= a.SC; ++jn; }
        const bool has_next = jn < nb;
        const char* pn = s_blob[has_next ? jn : jb];
        const size_t unit_n = (size_t)rb * a.SC + sn;
        const uint4* nx = (const uint4*)(pn + a.off.idx) + unit_n * N * 32 + lane;
        const RegBook<N> book = load_book<N>(planes + (size_t)jb * a.tab_bytes, a.L, id);
        uint32_t id_n = 0u, sm_n = 0u;
        if (has_next) {
            id_n = ((const uint8_t*)(pn + a.off.gid))[unit_n * 32 + lane];
            sm_n = ((const uint32_t*)(pn + a.off.gsm))[unit_n * 32 + lane];
        }
        const uint32_t xp = xlane + (uint32_t)(jb * K + s * kSuper) * 2u;
        uint32_t fa[4], fb[4];
        uint4 xr = make_uint4(0u, 0u, 0u, 0u);
        reg_decode8<N>(fa, w, 0, book);
#pragma unroll
        for (int j = 0; j < kSuper / 8; j += 2) {
            ld_x16(xr, xp + j * 16, dq);
            reg_decode8<N>(fb, w, j + 1, book);
#pragma unroll
            for (int v = 0; v < N; ++v) {
                const int last = (128 * (v + 1) - 1) / (8 * N);       // last step that reads vector v
                if ((last == j || last == j + 1) && has_next) {
                    const uint4 t = ld_stream(nx + v * 32);
                    w[4 * v] = t.x; w[4 * v + 1] = t.y; w[4 * v + 2] = t.z; w[4 * v + 3] = t.w;
                }
            }
            mma16816(c, fa[0], fa[1], fa[2], fa[3], xr.x, xr.y);
            if (j + 2 < kSuper / 8) reg_decode8<N>(fa, w, j + 2, book);
            mma16816(c, fb[0], fb[1], fb[2], fb[3], xr.z, xr.w);
        }
        // the group's sum to the lane that owns the channel, folded with scale and mid-point
        {
            const float a0 = __shfl_sync(0xffffffffu, c[0], src_a), a1 = __shfl_sync(0xffffffffu, c[1], src_a);
            const float b2 = __shfl_sync(0xffffffffu, c[2], src_a + 2), b3 = __shfl_sync(0xffffffffu, c[3], src_a + 2);
            const float Gs = (t4 & 1) ? a1 + b3 : a0 + b2;
            const float2 X = *(const float2*)(xg + ((size_t)jb * a.SC + s) * 2);
            acc = fmaf(h2f((uint16_t)(sm & 0xffffu)), Gs, fmaf(h2f((uint16_t)(sm >> 16)), X.x + X.y, acc));
            c[0] = c[1] = c[2] = c[3] = 0.f;
        }
        if (kCombine && jn != jb) { total = fmaf(s_w[jb], acc, total); acc = 0.f; }
        jb = jn; s = sn; id = id_n; sm = sm_n;
    }
    if (!kCombine) total = acc;

    // ---- outliers: the slots of every blob's slab are dealt to the warps of the row-block, four loads in flight
    const int row = rb * kRowsPerBlock + lane;
    for (int b0 = 0; b0 < nb; ++b0) {
        const int slots = s_slots[b0], width = min(s_width[b0][rl], slots);
        const uint32_t* slab = s_ell[b0] + (size_t)rb * (slots + 1) * 32 + lane;
        const unsigned char* xb = xs + (size_t)b0 * K * 2;
        float o = 0.f;
        // the warps that begin rotate with the blob
        for (int j = (kw + KW - (b0 * 4) % KW) % KW; j < width; j += 4 * KW) {
            uint32_t e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = j + i * KW < width ? __ldg(slab + (size_t)(1 + j + i * KW) * 32) : 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) o = fmaf(h2f((uint16_t)(e[i] >> 16)), h2f(*(const uint16_t*)(xb + xpos_of<kEvenOdd>(e[i] & 0xffffu) * 2)), o);
        }
        if (kw == 0 && slots && s_width[b0][rl] >= slots) {          // channels that fill their slab continue in the CSR arrays
            if ((int)__ldg(slab) >= slots) {
                const int* rowptr = (const int*)(s_blob[b0] + a.off.rowptr);
                const uint32_t* oent = (const uint32_t*)(s_blob[b0] + a.off.oent);
                const int p1 = __ldg(rowptr + row + 1);
                for (int p = __ldg(rowptr + row) + slots; p < p1; ++p) {
                    const uint32_t e = __ldg(oent + p);
                    o = fmaf(h2f((uint16_t)(e >> 16)), h2f(*(const uint16_t*)(xb + xpos_of<kEvenOdd>(e & 0xffffu) * 2)), o);
                }
            }
        }
        total = kCombine ? fmaf(s_w[b0], o, total) : total + o;
    }

    // ---- fixed-order sum over the warps, then the fused store
    red[warp * 32 + lane] = total;
    __syncthreads();
    float sum = 0.f;
    if (tid < 32 * R) {
#pragma unroll
        for (int k = 0; k < KW; ++k) sum += red[(k * R + tid / 32) * 32 + lane];
    }
    if (!kCombine) {
        __syncthreads();
        if (tid < 64) red[tid] = sum;
        __syncthreads();
        if (tid < 32) {
            const float gate = red[tid], up = red[tid + 32];
            put_y(a.y_list[j0], (size_t)blk * 32 + tid, gate / (1.f + expf(-gate)) * up, a.y_kind);
        }
        return;
    }
    const int ch = blk * 32 + lane;
    if (a.G == 1) {
        if (tid < 32 && ch < a.rows) put_y(a.y_list[0], ch, sum, a.y_kind);
        return;
    }
    // the runs of this row-block leave their sums in the workspace, the last one to arrive adds them in run order
    if (tid < 32) a.partial[(size_t)run * a.rows_ws + ch] = sum;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(a.tickets + blk, 1) == a.G - 1);
    __syncthreads();
    if (s_last) {
        __threadfence();
        if (tid < 32 && ch < a.rows) {
            float y = 0.f;
            for (int r = 0; r < a.G; ++r) y += __ldcg(a.partial + (size_t)r * a.rows_ws + ch);
            put_y(a.y_list[0], ch, y, a.y_kind);
        }
        if (tid == 0) a.tickets[blk] = 0;
    }
}

int plane_bytes(const Layout& l) { return (l.L * l.E * 2 + 15) & ~15; }
size_t expert_smem(const Layout& l, int blobs, int warps) {
    return (size_t)blobs * (plane_bytes(l) + (size_t)l.cols * 2 + (size_t)l.SC * 8) + (size_t)warps * 128;
}

template <int N, int W, int R, int MINB>
cudaError_t launch(const ExpertArgs& a, int grid, size_t smem, cudaStream_t s) {
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        cudaError_t e = cudaFuncSetAttribute(gemv_expert_kernel<N, W, R, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(MINB == 1 ? kExpertSmemOne : kExpertSmemTwo));
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(W * 32, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemv_expert_kernel<N, W, R, MINB>, a);
}

// The weighted sum: CTAs of 16 warps, one per SM, or of 8 warps, three per SM, and runs per row-block (G; ng blobs each).
struct CombinePlan { int warps, G, ng; };

// Up to one row-block per SM: 16 warps.  Rounds of CTAs times an item's time -- 150 clocks per unit of 32 channels and 128 weights,
// 5000 around them, 2500 more where runs meet through the workspace -- over the runs that fit shared memory and the scratch of one
// GEMV call.  Beyond, a second round of 16-warp CTAs leaves most SMs idle: 8 warps, three CTAs per SM, and more runs (us for 16 warps
// -> this, N = 3: 6 experts 5120 x 1536 23.9 -> 17.5, 2 of 7168 x 3072 16.7 -> 16.1, 8 of 6144 x 2048 36.4 -> 26.4; 8 of 4096 x 1536 take
// 15.3 in 16 warps, 17.5 in 8).  A CTA's time is its units, three to an SM in full rounds; of a last round of one CTA per SM a unit
// takes 1.8 of the time it would take alone at full occupancy, and a further round costs 18 units of x and first loads.
CombinePlan combine_plan(const Layout& l, int n) {
    const int sms = sched_sms(), slots = 3 * sms;
    CombinePlan best{16, 0, 0};
    double least = 0.0;
    for (int warps = l.RB > sms ? 8 : 16; warps <= 16 && !best.G; warps += 8)
        for (int G = 1; G <= n && G <= 64; ++G) {
            const int ng = (n + G - 1) / G, runs = (n + ng - 1) / ng;
            if (runs != G || ng > kExpertBlobs || expert_smem(l, ng, warps) > (warps == 8 ? kExpertSmemThree : kExpertSmemOne)) continue;
            const long long ctas = (long long)l.RB * G;
            const double run = (double)ng * l.SC;
            double t;
            if (warps == 16) {
                t = (double)((ctas + sms - 1) / sms) * (run * 150.0 + 5000.0) + (G > 1 ? 2500.0 : 0.0);
            } else {
                const long long full = ctas / slots, rest = ctas % slots;
                t = (double)full * 3.0 * run + (double)(full + (rest > 0) - 1) * 18.0 + (rest == 0 ? 0.0 : rest <= sms ? 1.8 : 3.0) * run;
            }
            if (!best.G || t < least) { best = CombinePlan{warps, G, ng}; least = t; }
        }
    return best;
}

}  // namespace

// fused stores of V2a blobs at N <= 4, groups of 128 or 256 weights, where x and the libraries fit shared memory
bool expert_supported(const Layout& l, const GemvCall& c) {
    if (l.mode != 1 || l.bits > 4 || l.GH != 1 || c.batch != 1 || !c.packed_list) return false;
    if (c.epilogue == 1) return expert_smem(l, 1, 8) <= kExpertSmemThree;
    return c.epilogue == 2 && combine_plan(l, c.n).G > 0;
}

cudaError_t launch_gemv_expert(const Layout& l, const GemvCall& c, cudaStream_t s) {
    ExpertArgs a{};
    a.off = offsets_of(l);
    a.packed_list = c.packed_list; a.x_list = c.x_list; a.y_list = c.y_list; a.epi_w = c.epi_weights;
    a.rows = l.rows; a.RB = l.RB; a.SC = l.SC; a.L = l.L; a.n = c.n; a.rows_ws = l.RB * kRowsPerBlock;
    a.y_kind = c.y_is_fp16; a.x_bf16 = c.x_bf16;
    a.tab_bytes = plane_bytes(l);
    a.tickets = (int*)c.workspace;
    a.partial = (float*)((char*)c.workspace + align256((size_t)l.RB * 4 * c.n));   // behind the common counter region
    if (c.epilogue == 1) {
        a.blocks = l.RB / 2;
        const int grid = a.blocks * c.n;
        // CTAs are packed on SMs that have room for more: no more of them to an SM than it takes to hold all, by asking for as much
        // shared memory; one to an SM with 16 warps
        size_t smem = expert_smem(l, 1, 8);
        if (grid <= sched_sms()) {
            smem = expert_smem(l, 1, 16);
            switch (l.bits) {
                case 2: return launch<2, 16, 2, 1>(a, grid, smem, s);
                case 3: return launch<3, 16, 2, 1>(a, grid, smem, s);
                default: return launch<4, 16, 2, 1>(a, grid, smem, s);
            }
        }
        if (grid <= 2 * sched_sms()) smem = std::max(smem, kExpertSmemTwo);
        switch (l.bits) {
            case 2: return launch<2, 8, 2, 3>(a, grid, smem, s);
            case 3: return launch<3, 8, 2, 3>(a, grid, smem, s);
            default: return launch<4, 8, 2, 3>(a, grid, smem, s);
        }
    }
    const CombinePlan p = combine_plan(l, c.n);
    a.G = p.G; a.ng = p.ng;
    const int grid = l.RB * p.G;
    const size_t smem = expert_smem(l, p.ng, p.warps);
    switch (l.bits) {
        case 2: return p.warps == 8 ? launch<2, 8, 1, 3>(a, grid, smem, s) : launch<2, 16, 1, 1>(a, grid, smem, s);
        case 3: return p.warps == 8 ? launch<3, 8, 1, 3>(a, grid, smem, s) : launch<3, 16, 1, 1>(a, grid, smem, s);
        default: return p.warps == 8 ? launch<4, 8, 1, 3>(a, grid, smem, s) : launch<4, 16, 1, 1>(a, grid, smem, s);
    }
}

}  // namespace xfp
