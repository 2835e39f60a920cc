// The one-channel-per-lane decode kernel (xfp_gemv_lane.cuh) with codebooks in registers: V2a at N = 2, 3, one row of x or 2, 4, 8.
//
// Mapping, x on the diagonal lanes, outlier slabs, K slices and their finish, resident CTAs of several rows: those of the lane
// kernel.  What differs: no tables.  The library sits in shared memory once, as byte planes (at most 4 KB); a lane loads the
// codebook of its channel's group into registers and decodes with PRMTs (xfp_reg_decode.cuh).  x is staged in the order that decode
// gives (N = 2: even k first).  The fragment accumulates sum lib * x of ONE group, and after the group's steps the sum moves to the
// lane that owns the channel:  acc += scale * G + mid * X_g,  X_g = sum of x over the group.
//
// One row, us per call (graph replay, 1 % outliers), tables of the lane kernel -> this:
//   N = 2  4096 x 4096 5.5 -> 4.6, 12288 x 4096 13.7 -> 10.8, 8192 x 8192 13.7 -> 13.7, 28672 x 8192 45.5 -> 38.3
//   N = 3  4096 x 4096 6.0 -> 5.1, 12288 x 4096 16.4 -> 12.0, 8192 x 8192 18.2 -> 15.3, 28672 x 8192 55.0 -> 42.4
// N = 4 takes 21 ALU instructions for eight weights and was even (4096 x 4096 6.18 against 6.12 us, 4096 x 12288 14.5 against 13.5,
// 28672 x 8192 56.4 both); V2 at N = 2, 3 loses to its quad and pair tables (28672 x 8192 32.8 and 37.6 against 29.7 and 31.7).
// Bound by the ALU pipe: 17.4 of 29.8 instructions per 256 weights, 69 % busy while an SM is active (28672 x 8192, N = 3).
#include "xfp_gemv_lane.cuh"
#include "xfp_reg_decode.cuh"

namespace xfp {

namespace {

// NB rows of x (1, 2, 4 or 8); TIO (one row or two): bf16 x, bf16 y, several blobs through pointer lists (see xfp_gemv_lane.cuh)
template <int N, int W, int MINB, bool TIO, int NB>
__global__ void __launch_bounds__(W * 32, MINB) gemv_reg_kernel(const LaneArgs a) {
    constexpr int E = 1 << N;
    constexpr bool kEvenOdd = N == 2;        // order of the staged x
    constexpr int kThreads = W * 32;
    constexpr bool kMulti = NB > 1;          // resident CTA over several row-blocks
    constexpr int RH = NB < 4 ? NB : 4;      // rows of x whose B registers are live at a time
    static_assert(NB * 32 <= kThreads, "one thread per channel and row of x in the final sum");
    extern __shared__ __align__(16) unsigned char smem[];
    // [byte planes of the library | x fp16 [NB][K] permuted | red [NB][W][32] | sums of x]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;");
    const int K = a.SC * kSuper;
    const size_t xrow = (size_t)K * 2;             // bytes of one staged row of x
    unsigned char* tab = smem;
    unsigned char* xs = smem + a.tab_bytes;
    float* red = (float*)(xs + NB * xrow);         // [NB][W][32]
    float* xg = red + NB * W * 32;                 // [NB][SC][2] sums of x over the halves of every super-chunk
    const int g = lane >> 2, t4 = lane & 3;
    const bool dq = (g == t4) || (g == t4 + 4);
    // where the two halves of this lane's group sum land in the fragment (see the end of the kernel)
    const int src_a = (lane & ~3) | (t4 >> 1);
#pragma unroll 1
    for (int it = 0;; ++it) {
    // ---- this CTA's block and K slice
    int blk, slice, nslices, sc0, nsc;
    if (kMulti) {
        const int v = it * (int)gridDim.x + (int)blockIdx.x;
        if (v < a.tier_blk[0]) {
            blk = v; slice = 0; nslices = 1; sc0 = 0; nsc = a.SC;
        } else {
            const int c = v - a.tier_blk[0];   // the K slices of the remaining blocks are dealt the same way
            if (c >= a.tier_cta[1]) break;
            nslices = a.tier_kst[0];
            blk = a.tier_blk[0] + c / nslices;
            slice = c - (c / nslices) * nslices;
            sc0 = slice * a.tier_spp[0];
            nsc = max(0, min(a.SC, sc0 + a.tier_spp[0]) - sc0);
        }
        if (it > 0) __syncthreads();   // the previous block's sums are no longer read
    } else {
        int tier = 0;
#pragma unroll
        for (int i = 1; i < 4; ++i)
            if ((int)blockIdx.x >= a.tier_cta[i]) tier = i;
        const int c = blockIdx.x - a.tier_cta[tier];
        nslices = a.tier_kst[tier];
        blk = a.tier_blk[tier] + c / nslices;
        slice = c - (c / nslices) * nslices;
        sc0 = slice * a.tier_spp[tier];
        nsc = max(0, min(a.SC, sc0 + a.tier_spp[tier]) - sc0);
    }
    const int gw = slice * W + warp, ostride = nslices * W;
    // the blob of this block: `gblk` numbers the row-blocks of the whole launch, `blk` those of its blob
    const int gblk = blk;
    const void* packed = a.packed;
    const uint16_t* xsrc = a.x;
    void* ydst = a.y;
    int ell_slots = a.ell_slots;
    if (TIO && a.packed_list) {
        const int prob = blk / a.RB;
        blk -= prob * a.RB;
        packed = a.packed_list[prob];
        xsrc = a.x_list[prob];
        ydst = a.y_list[prob];
        ell_slots = __ldg((const int*)((const char*)packed + a.off.hdr));   // the blobs' outlier counts differ
    }
    const Blob b = blob_at(packed, a.off);

    // ---- loads that do not depend on earlier kernels: first index vectors, outlier slab, the library
    uint32_t w[4 * N + 1];
    w[4 * N] = 0u;
    const uint4* ip = b.idx + ((size_t)(blk * a.SC + sc0) * N) * 32 + lane;
    if (warp < nsc) {
#pragma unroll
        for (int v = 0; v < N; ++v) {
            const uint4 t = ld_stream(ip + ((size_t)warp * N + v) * 32);
            w[4 * v] = t.x; w[4 * v + 1] = t.y; w[4 * v + 2] = t.z; w[4 * v + 3] = t.w;
        }
    }
    // library id and (scale, mid) of the lane's channel for the two halves of the super-chunk ([1] repeats [0]
    // unless the groups hold 64 weights), current and next
    const int GH = a.GH;
    const size_t m0 = ((size_t)(blk * a.SC + sc0) * GH) * 32 + lane;
    uint32_t gid_c[2] = {0u, 0u}, gsm_c[2] = {0u, 0u}, gid_n[2] = {0u, 0u}, gsm_n[2] = {0u, 0u};
    if (warp < nsc) {
        gid_c[0] = b.gid[m0 + (size_t)warp * GH * 32]; gsm_c[0] = b.gsm[m0 + (size_t)warp * GH * 32];
        gid_c[1] = b.gid[m0 + ((size_t)warp * GH + GH - 1) * 32]; gsm_c[1] = b.gsm[m0 + ((size_t)warp * GH + GH - 1) * 32];
    }
    const uint32_t* ell = (TIO && a.packed_list)
        ? (const uint32_t*)((const char*)packed + *(const long long*)((const char*)packed + a.off.hdr + 8)) : b.ell;
    const uint32_t* slab = ell + (size_t)blk * (ell_slots + 1) * 32 + lane;
    uint32_t olen = ell_slots ? __ldg(slab) : 0u;
    uint32_t oe[kLaneSlots];
#pragma unroll
    for (int q = 0; q < kLaneSlots; ++q) {
        const int j = gw + q * ostride;
        oe[q] = j < ell_slots ? __ldg(slab + (size_t)(1 + j) * 32) : 0u;   // every slot below the capacity is readable
    }
    if (!kMulti || it == 0)   // one library per blob: a resident CTA fills it once
        for (int id = threadIdx.x; id < a.L; id += kThreads) store_book<N>(tab, a.L, id, make_book<N>(b.cb + (size_t)id * E));

    // ---- x may come from the previous kernel of the stream
    if (!kMulti || it == 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll 1
    for (int r = 0; r < NB; ++r) {
        const bool have = r < a.batch;   // rows beyond the batch are staged as zeros
        const uint4* xrsrc = (const uint4*)(xsrc + (size_t)r * a.cols);
        unsigned char* xd = xs + r * xrow;
        for (int t = threadIdx.x; t < ((K / 8 + 31) & ~31); t += kThreads) {   // whole warps: the sums below shuffle
            const bool in = t < K / 8;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (in && have) {
                v = __ldg(xrsrc + t);
                if (TIO) v = x8_as_f16(v, a.x_bf16);
            }
            if (in) {
                if constexpr (kEvenOdd) {   // k = 8t .. 8t+7: the even and the odd k
                    *(uint2*)(xd + xpos_of<true>(8u * t) * 2) = make_uint2(prmt(v.x, v.y, 0x5410u), prmt(v.z, v.w, 0x5410u));
                    *(uint2*)(xd + xpos_of<true>(8u * t + 1u) * 2) = make_uint2(prmt(v.x, v.y, 0x7632u), prmt(v.z, v.w, 0x7632u));
                } else {
                    // k = 8t .. 8t+7: its two blocks of four go to positions xpos(8t) and xpos(8t + 4)
                    *(uint2*)(xd + xpos_of<false>(8u * t) * 2) = make_uint2(v.x, v.y);
                    *(uint2*)(xd + xpos_of<false>(8u * t + 4u) * 2) = make_uint2(v.z, v.w);
                }
            }
            // 8 consecutive threads hold 64 consecutive k: sums of x over the halves of the super-chunks, in a fixed order
            const float2 p0 = __half22float2(*(const __half2*)&v.x), p1 = __half22float2(*(const __half2*)&v.y);
            const float2 p2 = __half22float2(*(const __half2*)&v.z), p3 = __half22float2(*(const __half2*)&v.w);
            float sx = ((p0.x + p0.y) + (p1.x + p1.y)) + ((p2.x + p2.y) + (p3.x + p3.y));
            sx += __shfl_xor_sync(0xffffffffu, sx, 1);
            sx += __shfl_xor_sync(0xffffffffu, sx, 2);
            sx += __shfl_xor_sync(0xffffffffu, sx, 4);
            if (in && (t & 7) == 0) xg[r * a.SC * 2 + (t >> 3)] = sx;
        }
    }
    }
    __syncthreads();   // the library and x visible

    // a diagonal lane reads 16 bytes per two mma steps: bytes [0,16) of every 32 for g == t, [16,32) for g == t + 4
    const unsigned char* xq = xs + (size_t)sc0 * (kSuper * 2) + ((g == t4 + 4) ? 16 : 0);

    float c[NB][4];
    float oacc[NB];   // the channel's folded group sums and its outliers
#pragma unroll
    for (int r = 0; r < NB; ++r) { c[r][0] = c[r][1] = c[r][2] = c[r][3] = 0.f; oacc[r] = 0.f; }
    // the rows' slot counts have arrived: outlier rounds of this warp
    int width = (int)olen;
#pragma unroll
    for (int o = 16; o; o >>= 1) width = max(width, __shfl_xor_sync(0xffffffffu, width, o));
    width = min(width, ell_slots);
    const int mine = width > gw ? (width - gw + ostride - 1) / ostride : 0;
    const int nrounds = (mine + kLaneSlots - 1) / kLaneSlots;
    int oround = 0;
    auto consume_slots = [&]() {
#pragma unroll
        for (int q = 0; q < kLaneSlots; ++q) {
            const float v = h2f((uint16_t)(oe[q] >> 16));
            const unsigned char* xo = xs + xpos_of<kEvenOdd>(oe[q] & 0xffffu) * 2;
#pragma unroll
            for (int r = 0; r < NB; ++r) oacc[r] = fmaf(v, h2f(*(const uint16_t*)(xo + r * xrow)), oacc[r]);
        }
    };
    auto fetch_slots = [&](int round) {
#pragma unroll
        for (int q = 0; q < kLaneSlots; ++q) {
            const int j = gw + (round * kLaneSlots + q) * ostride;
            oe[q] = j < width ? __ldg(slab + (size_t)(1 + j) * 32) : 0u;
        }
    };

    // ---- K loop: 16 mma steps per super-chunk, look-ups one step ahead of the tensor pipe; an index vector is
    //      reloaded with the same vector of this warp's next super-chunk as soon as its last step has been looked up
#pragma unroll 1
    for (int s = warp; s < nsc; s += W) {
        if (oround < nrounds) {
            consume_slots();
            if (++oround < nrounds) fetch_slots(oround);
        }
        const bool has_next = s + W < nsc;
        const uint4* nx = ip + (size_t)(s + W) * N * 32;
        const unsigned char* xp = xq + (size_t)s * (kSuper * 2);
        uint32_t fa[4], fb[4];
        uint4 xr[RH];
#pragma unroll
        for (int r = 0; r < RH; ++r) xr[r] = make_uint4(0u, 0u, 0u, 0u);
        RegBook<N> book = load_book<N>(tab, a.L, gid_c[0]);
        if (has_next) {   // metadata of the next super-chunk travels during this one
            const size_t mn = m0 + (size_t)(s + W) * GH * 32;
            gid_n[0] = b.gid[mn]; gsm_n[0] = b.gsm[mn];
            gid_n[1] = b.gid[mn + (size_t)(GH - 1) * 32]; gsm_n[1] = b.gsm[mn + (size_t)(GH - 1) * 32];
        }
        // the group's sum leaves the fragment (two halves of the channel's sum sit in two other lanes of the
        // quad) and is folded with the group's scale and mid-point
        auto fold = [&](int h) {
            const float scale = h2f((uint16_t)(gsm_c[h] & 0xffffu)), mid = h2f((uint16_t)(gsm_c[h] >> 16));
#pragma unroll
            for (int r = 0; r < NB; ++r) {
                const float a0 = __shfl_sync(0xffffffffu, c[r][0], src_a), a1 = __shfl_sync(0xffffffffu, c[r][1], src_a);
                const float b2 = __shfl_sync(0xffffffffu, c[r][2], src_a + 2), b3 = __shfl_sync(0xffffffffu, c[r][3], src_a + 2);
                const float G = (t4 & 1) ? a1 + b3 : a0 + b2;
                const float* xgr = xg + (r * a.SC + sc0 + s) * 2;
                const float X = GH == 2 ? xgr[h] : xgr[0] + xgr[1];
                oacc[r] = fmaf(scale, G, fmaf(mid, X, oacc[r]));
                c[r][0] = c[r][1] = c[r][2] = c[r][3] = 0.f;
            }
        };
        reg_decode8<N>(fa, w, 0, book);
#pragma unroll
        for (int j = 0; j < kSuper / 8; j += 2) {
            if (NB <= RH) {
#pragma unroll
                for (int r = 0; r < NB; ++r) ld_x16_if(xr[r], xp + r * xrow + j * 16, dq);   // steps j and j + 1
            }
            reg_decode8<N>(fb, w, j + 1, book);
#pragma unroll
            for (int v = 0; v < N; ++v)
                if ((last_step_of_vector<N>(v) == j || last_step_of_vector<N>(v) == j + 1) && has_next) {
                    const uint4 t = ld_stream(nx + v * 32);
                    w[4 * v] = t.x; w[4 * v + 1] = t.y; w[4 * v + 2] = t.z; w[4 * v + 3] = t.w;
                }
            if (NB <= RH) {
#pragma unroll
                for (int r = 0; r < NB; ++r) mma16816(c[r], fa[0], fa[1], fa[2], fa[3], xr[r].x, xr[r].y);
                if (GH == 2 && j + 2 == kSuper / 16) book = load_book<N>(tab, a.L, gid_c[1]);   // the second half's group
                if (j + 2 < kSuper / 8) reg_decode8<N>(fa, w, j + 2, book);
#pragma unroll
                for (int r = 0; r < NB; ++r) mma16816(c[r], fb[0], fb[1], fb[2], fb[3], xr[r].z, xr[r].w);
            } else {
                // more rows than B registers kept live: RH rows at a time through both steps
                uint32_t fn[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int h = 0; h < NB / RH; ++h) {
#pragma unroll
                    for (int r = 0; r < RH; ++r) ld_x16_if(xr[r], xp + (h * RH + r) * xrow + j * 16, dq);
                    if (h == NB / RH - 1) {
                        if (GH == 2 && j + 2 == kSuper / 16) book = load_book<N>(tab, a.L, gid_c[1]);   // the second half's group
                        if (j + 2 < kSuper / 8) reg_decode8<N>(fn, w, j + 2, book);
                    }
#pragma unroll
                    for (int r = 0; r < RH; ++r) mma16816(c[h * RH + r], fa[0], fa[1], fa[2], fa[3], xr[r].x, xr[r].y);
#pragma unroll
                    for (int r = 0; r < RH; ++r) mma16816(c[h * RH + r], fb[0], fb[1], fb[2], fb[3], xr[r].z, xr[r].w);
                }
                fa[0] = fn[0]; fa[1] = fn[1]; fa[2] = fn[2]; fa[3] = fn[3];
            }
            if (j + 2 == kSuper / 16 && GH == 2) fold(0);   // the first group of 64 weights is complete
        }
        fold(1);
        gid_c[0] = gid_n[0]; gid_c[1] = gid_n[1]; gsm_c[0] = gsm_n[0]; gsm_c[1] = gsm_n[1];
    }
    while (oround < nrounds) {   // more outlier rounds than super-chunks
        consume_slots();
        if (++oround < nrounds) fetch_slots(oround);
    }
    // rows that fill their slab continue in the CSR arrays (pathological skew only): warp 0 of the first slice
    if (warp == 0 && slice == 0 && ell_slots && (int)olen >= ell_slots) {
        const int row = blk * kRowsPerBlock + lane;
        const int p1 = __ldg(b.rowptr + row + 1);
        for (int p = __ldg(b.rowptr + row) + ell_slots; p < p1; ++p) {
            const uint32_t e = __ldg(b.oent + p);
            const float v = h2f((uint16_t)(e >> 16));
            const unsigned char* xo = xs + xpos_of<kEvenOdd>(e & 0xffffu) * 2;
#pragma unroll
            for (int r = 0; r < NB; ++r) oacc[r] = fmaf(v, h2f(*(const uint16_t*)(xo + r * xrow)), oacc[r]);
        }
    }

    // ---- every lane owns its channel's sum
#pragma unroll
    for (int r = 0; r < NB; ++r) red[(size_t)(r * W + warp) * 32 + lane] = oacc[r];
    __syncthreads();

    // ---- fixed-order sum over the warps, then store or combine the block's slices
    const int t = threadIdx.x;
    const int er = t >> 5, ech = t & 31;   // row of x and channel of this thread in the final sum
    const bool active = er < NB;
    const int row = blk * 32 + ech;       // channel inside its blob (y index)
    const int wrow = gblk * 32 + ech;     // channel inside the launch (workspace index)
    float total = 0.f;
    if (active) {
#pragma unroll
        for (int ww = 0; ww < W; ++ww) total += red[(er * W + ww) * 32 + ech];
    }
    bool writer = true;
    if (nslices > 1) {
        __shared__ int s_last;
        if (active) a.partial[((size_t)slice * NB + er) * a.rows_ws + wrow] = total;
        __threadfence();
        __syncthreads();
        if (t == 0) s_last = (atomicAdd(a.tickets + gblk, 1) == nslices - 1);
        __syncthreads();
        writer = s_last != 0;
        if (writer) {
            __threadfence();
            if (active) {
                total = 0.f;
                for (int k2 = 0; k2 < nslices; ++k2) total += __ldcg(a.partial + ((size_t)k2 * NB + er) * a.rows_ws + wrow);
            }
            if (t == 0) a.tickets[gblk] = 0;
        }
    }
    if (writer && active && er < a.batch && row < a.rows) store_y<TIO>(ydst, (size_t)er * a.rows + row, total, a.y_is_fp16);
    if (!kMulti) break;
    }
}

template <int N, int W, int MINB, bool TIO, int NB>
cudaError_t launch_io(const LaneArgs& a, int grid, size_t smem, cudaStream_t s) {
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        cudaError_t e = cudaFuncSetAttribute(gemv_reg_kernel<N, W, MINB, TIO, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             MINB == 1 ? 224 * 1024 : MINB == 2 ? 110 * 1024 : 73 * 1024);
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
    return cudaLaunchKernelEx(&cfg, gemv_reg_kernel<N, W, MINB, TIO, NB>, a);
}

template <int N, int W, int MINB>
cudaError_t launch_rows(const LaneArgs& a, int nb, int grid, size_t smem, cudaStream_t s) {
    if (nb == 1) {
        if (a.x_bf16 || a.y_is_fp16 == 2 || a.packed_list) return launch_io<N, W, MINB, true, 1>(a, grid, smem, s);
        return launch_io<N, W, MINB, false, 1>(a, grid, smem, s);
    }
    if constexpr (MINB < 3) {
        if (nb == 2 && (a.x_bf16 || a.y_is_fp16 == 2)) return launch_io<N, W, MINB, true, 2>(a, grid, smem, s);
        if (nb == 2) return launch_io<N, W, MINB, false, 2>(a, grid, smem, s);
        if (nb == 4) return launch_io<N, W, MINB, false, 4>(a, grid, smem, s);
        return launch_io<N, W, MINB, false, 8>(a, grid, smem, s);
    }
    return cudaErrorInvalidValue;
}

template <int N>
cudaError_t launch_cfg(const LaneArgs& a, int per_sm, int nb, int grid, size_t smem, cudaStream_t s) {
    if (per_sm == 1) return launch_rows<N, 16, 1>(a, nb, grid, smem, s);
    if (per_sm == 2) return launch_rows<N, 8, 2>(a, nb, grid, smem, s);
    return launch_rows<N, 8, 3>(a, nb, grid, smem, s);
}

}  // namespace

cudaError_t launch_reg(const LaneArgs& a, int bits, int per_sm, int nb, int grid, size_t smem, cudaStream_t s) {
    return bits == 2 ? launch_cfg<2>(a, per_sm, nb, grid, smem, s) : launch_cfg<3>(a, per_sm, nb, grid, smem, s);
}

}  // namespace xfp
