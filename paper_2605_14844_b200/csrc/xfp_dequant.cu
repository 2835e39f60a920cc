// xfp_dequant: device layout -> fp16 matrix W^ = fp16(D16 + S), bit-exact ("Reconstruct" in Algorithm 1).
//
// A block of eight warps takes one row-block (32 channels, a lane each) and a range of super-chunks; a warp decodes one
// super-chunk at a time from index vectors fetched one super-chunk ahead.
//   V2   the channels' codebooks in shared memory, one word per lane and entry (no bank conflicts); up to N = 3 indexed by
//        a PAIR of indices.
//   V2a  a lane decodes the 2^N entries its channel's group can take once -- D16 = fp16(fp32(scale * lib[id] + mid)) --
//        into a column of a table of its warp, and the weights of the group are look-ups as in V2: 2^N conversions per
//        group instead of one per weight (N = 2: pairs; at N = 6 64 entries serve 128 weights).
//   out  a tile of shared memory turns a lane's 64 weights into whole 128-byte lines of the channels' rows.
//   S    when the block has stored its range, its outliers are added in place, one correctly rounded fp16 addition each:
//        the slots of the transposed slab are dealt to the warps eight at a time, so that the loads of a batch overlap.
#include "xfp_internal.h"
#include "xfp_pair_common.cuh"

namespace xfp {

namespace {

constexpr int kDqWarps = 8;
constexpr int kDqRange = 32;        // super-chunks of a block at most: the tail of outliers stays short
constexpr int kTileRow = 144;       // bytes of a row of 64 weights in the staging tile: eight lanes' rows in distinct banks
constexpr int kLibEntries = 8192;   // library entries (L * 2^N) that are staged in shared memory

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory"); }

// The decode tables: PAIR: entry t = (first index | second index << N) holds both fp16 values; else entry q holds one.
// N = 4 entries lie 256 bytes apart (two tables interleaved), so that an index isolated in its own byte becomes the second
// byte of the address with one PRMT.
template <int N, int MODE>
struct DqTab {
    static constexpr int E = 1 << N;
    static constexpr bool kPair = MODE == 0 ? N <= 3 : N == 2;
    static constexpr int kEntries = kPair ? E * E : E;
    static constexpr int kBytes = N == 4 ? 4096 : kEntries * 128;            // of one table (N = 4: of an interleaved pair)
    static constexpr int kTables = MODE == 0 ? 1 : (N == 4 ? kDqWarps / 2 : kDqWarps);
    static constexpr int kStride = N == 4 ? 256 : 128;                      // bytes between entries
};

struct DqArgs {
    Blob b;
    uint16_t* out;
    int rows, cols, RB, SC, GH, L, ell_slots;
    int range;                // super-chunks of a block
};

template <int N, int MODE>
__global__ void __launch_bounds__(kDqWarps * 32) dequant_kernel(const DqArgs a) {
    using T = DqTab<N, MODE>;
    constexpr int E = T::E;
    extern __shared__ unsigned char dq_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int parts = (a.SC + a.range - 1) / a.range;
    const int rb = (int)blockIdx.x / parts, part = (int)blockIdx.x % parts;
    const int s0 = part * a.range, s1 = min(a.SC, s0 + a.range);
    // tables aligned to their size in the shared window (at least 1 KB), so that an entry's offset is merged, not added
    constexpr uint32_t kAlign = T::kBytes < 1024 ? 1024 : T::kBytes;
    const uint32_t raw = smem_addr(dq_smem), tab0 = (raw + kAlign - 1) & ~(kAlign - 1);
    unsigned char* base = dq_smem + (tab0 - raw);
    unsigned char* tiles = base + T::kTables * kAlign;                        // [warps][32 * kTileRow]
    uint16_t* slib = (uint16_t*)(tiles + kDqWarps * 32 * kTileRow);   // [L][lib_stride]
    constexpr int kLibStride = E + 8;                                        // 16 bytes of padding spread the ids over the banks
    const bool staged = MODE == 1 && a.L * E <= kLibEntries;
    if (MODE == 0) {
        const uint16_t* cb = a.b.cb + (size_t)(rb * kRowsPerBlock + lane) * E;    // padding rows exist in the blob
        for (int t = warp; t < T::kEntries; t += kDqWarps) {
            uint32_t v;
            if (T::kPair) v = (uint32_t)__ldg(cb + (t & (E - 1))) | ((uint32_t)__ldg(cb + (t >> N)) << 16);
            else v = (uint32_t)__ldg(cb + t);
            sts_u32(tab0 + (uint32_t)(t * T::kStride + lane * 4), v);
        }
        __syncthreads();
    } else if (staged) {
        for (int i = tid; i < a.L * E; i += kDqWarps * 32) slib[(i / E) * kLibStride + i % E] = __ldg(a.b.cb + i);
        __syncthreads();
    }
    // this lane's column of its table
    const uint32_t tab = MODE == 0 ? tab0 + (uint32_t)lane * 4u
                       : N == 4    ? tab0 + (uint32_t)(warp >> 1) * kAlign + (uint32_t)(warp & 1) * 128u + (uint32_t)lane * 4u
                                   : tab0 + (uint32_t)warp * kAlign + (uint32_t)lane * 4u;
    const uint32_t nib = ((tab >> 12) & 0xfu) * 0x10101010u;
    const int row = rb * kRowsPerBlock + lane;
    unsigned char* tile = tiles + warp * 32 * kTileRow;

    uint4 nx[N];
    uint32_t id_n[2] = {0, 0}, sm_n[2] = {0, 0};
    auto fetch = [&](int sc) {
        const uint4* src = a.b.idx + (((size_t)rb * a.SC + sc) * N) * 32 + lane;
#pragma unroll
        for (int v = 0; v < N; ++v) nx[v] = ld_stream(src + (size_t)v * 32);
        if (MODE == 1) {
            const size_t m0 = ((size_t)rb * a.SC + sc) * a.GH * 32 + lane, m1 = m0 + (size_t)(a.GH - 1) * 32;
            id_n[0] = __ldg(a.b.gid + m0); sm_n[0] = __ldg(a.b.gsm + m0);
            id_n[1] = __ldg(a.b.gid + m1); sm_n[1] = __ldg(a.b.gsm + m1);
        }
    };
    if (s0 + warp < s1) fetch(s0 + warp);
    for (int sc = s0 + warp; sc < s1; sc += kDqWarps) {
        uint32_t w[4 * N + 1];
#pragma unroll
        for (int v = 0; v < N; ++v) { w[4 * v] = nx[v].x; w[4 * v + 1] = nx[v].y; w[4 * v + 2] = nx[v].z; w[4 * v + 3] = nx[v].w; }
        w[4 * N] = 0u;
        const uint32_t id[2] = {id_n[0], id_n[1]}, sm[2] = {sm_n[0], sm_n[1]};
        if (sc + kDqWarps < s1) fetch(sc + kDqWarps);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (MODE == 1 && (h == 0 || a.GH == 2)) {
                const float scale = h2f((uint16_t)(sm[h] & 0xffffu)), mid = h2f((uint16_t)(sm[h] >> 16));
                auto decoded = [&](uint16_t l) { return (uint32_t)f2h(__fmaf_rn(scale, h2f(l), mid)); };
                if (N == 2) {
                    uint32_t d[4];
                    uint2 l4;
                    if (staged) l4 = *(const uint2*)(slib + id[h] * kLibStride);
                    else l4 = __ldg((const uint2*)(a.b.cb + (size_t)id[h] * E));
                    d[0] = decoded((uint16_t)l4.x); d[1] = decoded((uint16_t)(l4.x >> 16));
                    d[2] = decoded((uint16_t)l4.y); d[3] = decoded((uint16_t)(l4.y >> 16));
#pragma unroll
                    for (int t = 0; t < 16; ++t) sts_u32(tab + t * 128, join16(d[t & 3], d[t >> 2]));
                } else {
#pragma unroll
                    for (int e = 0; e < E; e += 8) {
                        uint4 l8;
                        if (staged) l8 = *(const uint4*)(slib + id[h] * kLibStride + e);
                        else l8 = __ldg((const uint4*)(a.b.cb + (size_t)id[h] * E + e));
                        const uint32_t lw[4] = {l8.x, l8.y, l8.z, l8.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            sts_u32(tab + (e + 2 * i) * T::kStride, decoded((uint16_t)lw[i]));
                            sts_u32(tab + (e + 2 * i + 1) * T::kStride, decoded((uint16_t)(lw[i] >> 16)));
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {                 // 8 weights = 16 bytes
                uint32_t d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int p = h * 32 + c * 4 + i;
                    if (T::kPair) {
                        d[i] = lds_u32(pair_addr<N, 1>(w, p, tab));
                    } else if (N == 4) {
                        const uint32_t wlo = (w[p >> 2] & 0x0f0f0f0fu) | nib, whi = ((w[p >> 2] >> 4) & 0x0f0f0f0fu) | nib;
                        const uint32_t sel = 0x7604u | ((uint32_t)(p & 3) << 4);   // [tab.b3, tab.b2, index byte, tab.b0]
                        d[i] = join16(lds_u32(__byte_perm(wlo, tab, sel)), lds_u32(__byte_perm(whi, tab, sel)));
                    } else {
                        d[i] = join16(lds_u32(single_addr<N, 1>(w, 2 * p, tab)), lds_u32(single_addr<N, 1>(w, 2 * p + 1, tab)));
                    }
                }
                const uint4 v = make_uint4(d[0], d[1], d[2], d[3]);
                *(uint4*)(tile + lane * kTileRow + c * 16) = v;
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {                 // four channels' 128 bytes per step
                const int r = 4 * i + (lane >> 3), orow = rb * kRowsPerBlock + r;
                if (orow < a.rows)
                    *(uint4*)(a.out + (size_t)orow * a.cols + (size_t)sc * kSuper + h * 64 + (lane & 7) * 8) =
                        *(const uint4*)(tile + r * kTileRow + (lane & 7) * 16);
            }
            __syncwarp();
        }
    }
    // ---- W^ += S on the values this block has just stored ----
    if (a.ell_slots) {
        __syncthreads();
        const uint32_t* slab = a.b.ell + (size_t)rb * (a.ell_slots + 1) * 32 + lane;
        const int len = row < a.rows ? (int)__ldg(slab) : 0, in_slab = min(len, a.ell_slots);
        const uint32_t k0 = (uint32_t)s0 * kSuper, k1 = (uint32_t)s1 * kSuper;
        uint16_t* out = a.out + (size_t)row * a.cols;
        constexpr int kBatch = 8;
        auto batch = [&](const uint32_t* src, int stride, int first, int end) {       // entries first, first + kDqWarps, ...
            uint32_t e[kBatch];
            uint16_t old[kBatch];
            bool ok[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; ++i) e[i] = first + i * kDqWarps < end ? __ldg(src + (size_t)(first + i * kDqWarps) * stride) : 0u;
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const uint32_t col = e[i] & 0xffffu;
                ok[i] = first + i * kDqWarps < end && col >= k0 && col < k1;
                if (ok[i]) old[i] = out[col];
            }
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (ok[i]) out[e[i] & 0xffffu] = __half_as_ushort(__hadd(__ushort_as_half(old[i]), __ushort_as_half((uint16_t)(e[i] >> 16))));
        };
        const int most = __reduce_max_sync(0xffffffffu, in_slab);
        for (int j = warp; j < most; j += kBatch * kDqWarps) batch(slab + 32, 32, j, in_slab);
        if (len >= a.ell_slots && row < a.rows) {        // the channel overflows its slab: the rest is in the CSR arrays
            const int p0 = __ldg(a.b.rowptr + row), n = __ldg(a.b.rowptr + row + 1) - p0;
            for (int j = a.ell_slots + warp; j < n; j += kBatch * kDqWarps) batch(a.b.oent + p0, 1, j, n);
        }
    }
}

template <int N, int MODE>
cudaError_t launch_decode(const Layout& l, const void* packed, uint16_t* W, cudaStream_t s) {
    using T = DqTab<N, MODE>;
    constexpr size_t kAlign = T::kBytes < 1024 ? 1024 : T::kBytes;
    DqArgs a = {};
    a.b = blob_at(packed, offsets_of(l));
    a.out = W;
    a.rows = l.rows; a.cols = l.cols; a.RB = l.RB; a.SC = l.SC; a.GH = l.GH; a.L = l.L; a.ell_slots = l.ell_slots;
    const size_t lib = MODE == 1 && a.L * T::E <= kLibEntries ? (size_t)a.L * (T::E + 8) * 2 : 0;
    const size_t smem = kAlign + T::kTables * kAlign + kDqWarps * 32 * kTileRow + lib;
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(dequant_kernel<N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    // few row-blocks: shorter ranges, at least one super-chunk per warp, until the blocks fill the GPU twice
    int range = a.SC < kDqRange ? a.SC : kDqRange;
    while (range > kDqWarps && (long long)l.RB * ((a.SC + range - 1) / range) < 4ll * sm_count()) range = (range + 1) / 2;
    a.range = range;
    dequant_kernel<N, MODE><<<(unsigned)(l.RB * ((a.SC + range - 1) / range)), kDqWarps * 32, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dequant(const Layout& l, const void* packed, uint16_t* W, cudaStream_t s) {
    if (l.mode == 0) {
        switch (l.bits) {
            case 2: return launch_decode<2, 0>(l, packed, W, s);
            case 3: return launch_decode<3, 0>(l, packed, W, s);
            case 4: return launch_decode<4, 0>(l, packed, W, s);
            case 5: return launch_decode<5, 0>(l, packed, W, s);
            default: return launch_decode<6, 0>(l, packed, W, s);
        }
    }
    switch (l.bits) {
        case 2: return launch_decode<2, 1>(l, packed, W, s);
        case 3: return launch_decode<3, 1>(l, packed, W, s);
        case 4: return launch_decode<4, 1>(l, packed, W, s);
        case 5: return launch_decode<5, 1>(l, packed, W, s);
        default: return launch_decode<6, 1>(l, packed, W, s);
    }
}

}  // namespace xfp
