// xfp_dequant: device layout -> fp16 matrix W^ = fp16(D16 + S), bit-exact ("Reconstruct" in Algorithm 1).
//
// A block of eight warps takes one row-block (32 channels, a lane each) and a range of super-chunks; a warp decodes one
// super-chunk at a time from index vectors fetched one super-chunk ahead.
//   V2   N <= 4: the channel's codebook in registers (xfp_reg_decode.cuh); above, codebooks in shared memory, one word per lane
//        and entry (no bank conflicts).
//   V2a  a lane decodes the 2^N entries its channel's group can take once -- D16 = fp16(fp32(scale * lib[id] + mid)) -- into
//        registers (N <= 4) or a column of a table of its warp, and the weights of the group are look-ups as in V2: 2^N
//        conversions per group instead of one per weight.
//   S    up to N = 4, where outliers are many (plan_of), the block notes where every super-chunk's outliers begin in its channels'
//        slabs and a lane adds those of its channel to the staged row, one correctly rounded fp16 addition each.  What a slab
//        cannot say (channels longer than their slab, columns that do not ascend), and all of them elsewhere, is added in place
//        behind the block's stores (above N = 4, where tables leave one or two blocks to an SM, the list in front of the decode
//        cost more: 12288 x 4096 V2a N = 6 38.2 -> 46.1 us with pack, half of both).
//   out  a tile of shared memory turns a lane's 64 weights into whole 128-byte lines of the channels' rows.
// Tables in shared memory and outliers in place behind the stores -> this, cold: 12289 x 4096 V2a N = 4, 1 % outliers 35.2 -> 32.0 us,
// 3072 x 4096 V2a N = 2 14.2 -> 10.8, 12288 x 4096 V2 N = 4 33.3 -> 29.1; warm, 28672 x 8192 V2 N = 4, 0.3 % 123.5 -> 99.7, where DRAM
// is at 67 % of its peak.  At 12289 x 4096 100 MB of stores and 29 MB of loads are 20 us at the copy rate; what is left is the chain
// of a block's first loads and the outliers' way back from L2.
#include "xfp_internal.h"
#include "xfp_pair_common.cuh"
#include "xfp_reg_decode.cuh"

namespace xfp {

namespace {

constexpr int kDqWarps = 8;
constexpr int kDqRange = 32;        // super-chunks of a block at most: the tail of outliers stays short
constexpr int kTileRow = 144;       // bytes of a row of 64 weights in the staging tile: eight lanes' rows in distinct banks
constexpr int kLibEntries = 8192;   // library entries (L * 2^N) that are staged in shared memory
constexpr int kDqSlots = 64;        // outliers of a channel in the block's range that are staged in shared memory; where there are more,
                                    // the channel's are read from the blob
constexpr int kDqStarts = (kDqRange + 1) * 32 * 2, kDqEntries = kDqSlots * 32 * 4;   // bytes of the starts and of the staged slots

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory"); }

// The decode tables of N = 5, 6: entry q holds one value per lane.
template <int N, int MODE>
struct DqTab {
    static constexpr int E = 1 << N;
    static constexpr bool kReg = N <= 4;
    static constexpr int kBytes = kReg ? 0 : E * 128;                        // of one table
    static constexpr int kTables = kReg ? 0 : MODE == 0 ? 1 : kDqWarps;
    static constexpr size_t kAlign = kReg ? 16 : kBytes;                     // aligned to its size: an entry's offset is merged, not added
};

struct DqArgs {
    Blob b;
    uint16_t* out;
    int rows, cols, RB, SC, GH, L, ell_slots;
    int range;                // super-chunks of a block
    bool lists;               // outliers are added to the staged rows
};

template <int N, int MODE>
__global__ void __launch_bounds__(kDqWarps * 32, N <= 4 ? 3 : 0) dequant_kernel(const DqArgs a) {
    using T = DqTab<N, MODE>;
    constexpr int E = T::E;
    extern __shared__ unsigned char dq_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int parts = (a.SC + a.range - 1) / a.range;
    const int rb = (int)blockIdx.x / parts, part = (int)blockIdx.x % parts;
    const int s0 = part * a.range, s1 = min(a.SC, s0 + a.range);
    constexpr uint32_t kAlign = (uint32_t)T::kAlign;
    const uint32_t raw = smem_addr(dq_smem), tab0 = (raw + kAlign - 1) & ~(kAlign - 1);
    unsigned char* base = dq_smem + (tab0 - raw);
    unsigned char* tiles = base + T::kTables * kAlign;                        // [warps][32 * kTileRow]
    uint32_t* ents = (uint32_t*)(tiles + kDqWarps * 32 * kTileRow);          // [kDqSlots][32]
    uint16_t* starts = (uint16_t*)((unsigned char*)ents + kDqEntries);       // [range + 1][32]
    uint16_t* slib = (uint16_t*)(T::kReg ? (unsigned char*)starts + kDqStarts : (unsigned char*)ents);     // [L][lib_stride]
    constexpr int kLibStride = E + 8;                                        // 16 bytes of padding spread the ids over the banks
    const bool staged = MODE == 1 && a.L * E <= kLibEntries;
    RegBook<T::kReg ? N : 2> book;
    const uint16_t* cb = a.b.cb + (size_t)(rb * kRowsPerBlock + lane) * E;   // V2: padding rows exist in the blob
    if constexpr (MODE == 0 && T::kReg) {
        book = make_book<N>(cb);
    } else if constexpr (MODE == 0) {
        for (int t = warp; t < E; t += kDqWarps) sts_u32(tab0 + (uint32_t)(t * 128 + lane * 4), (uint32_t)__ldg(cb + t));
    } else if (staged) {
        for (int i = tid; i < a.L * E; i += kDqWarps * 32) slib[(i / E) * kLibStride + i % E] = __ldg(a.b.cb + i);
    }
    // this lane's column of its table
    const uint32_t tab = tab0 + (MODE == 0 ? 0u : (uint32_t)warp * kAlign) + (uint32_t)lane * 4u;
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
    // where the outliers of every super-chunk begin: slot j is the first of the super-chunks behind that of slot j - 1
    const int nsc = s1 - s0;
    const uint32_t* slab = a.b.ell + (size_t)rb * (a.ell_slots + 1) * 32 + lane;
    const int len = a.ell_slots && row < a.rows ? (int)__ldg(slab) : 0, in_slab = min(len, a.ell_slots);
    bool in_place = a.ell_slots != 0 && !(T::kReg && a.lists);
    if (T::kReg && a.lists) {
        bool descends = false;
        auto rel = [&](uint32_t e) { return max(-1, min(nsc, (int)((e & 0xffffu) >> 7) - s0)); };
        // a run of slots to every warp, slot `in_slab` closes a channel's list; the loads do not wait for the channels' lengths
        const int chunk = (a.ell_slots + kDqWarps) / kDqWarps, j1 = min((warp + 1) * chunk, a.ell_slots + 1);
        for (int jb = warp * chunk; jb < j1; jb += 8) {
            uint32_t v[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i] = jb + i > 0 && jb + i <= a.ell_slots ? __ldg(slab + (size_t)(jb + i) * 32) : 0u;   // slot jb + i - 1
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                const int j = jb + i - 1;
                if (j >= j1 || j > in_slab) continue;
                const bool have = j < in_slab;
                descends |= j > 0 && have && (v[i] & 0xffffu) <= (v[i - 1] & 0xffffu);
                const int b0 = j > 0 ? rel(v[i - 1]) : -1, b1 = have ? rel(v[i]) : nsc;
                if (have && b1 >= 0 && b1 < nsc) ents[(j % kDqSlots) * 32 + lane] = v[i];
                for (int t = b0 + 1; t <= b1; ++t) starts[t * 32 + lane] = (uint16_t)j;
            }
        }
        in_place = __syncthreads_or(descends) != 0;
    } else {
        __syncthreads();
    }
    const bool in_tile = T::kReg && a.ell_slots != 0 && !in_place;
    const bool ents_whole = in_tile && starts[nsc * 32 + lane] - starts[lane] <= kDqSlots;
    for (int sc = s0 + warp; sc < s1; sc += kDqWarps) {
        int j = 0, jend = 0;
        if (in_tile) { j = starts[(sc - s0) * 32 + lane]; jend = starts[(sc - s0 + 1) * 32 + lane]; }
        auto entry = [&](int i) { return ents_whole ? ents[(i % kDqSlots) * 32 + lane] : __ldg(slab + (size_t)(1 + i) * 32); };
        uint32_t e = j < jend ? entry(j) : 0u;
        uint32_t w[4 * N + 1];
#pragma unroll
        for (int v = 0; v < N; ++v) { w[4 * v] = nx[v].x; w[4 * v + 1] = nx[v].y; w[4 * v + 2] = nx[v].z; w[4 * v + 3] = nx[v].w; }
        w[4 * N] = 0u;
        const uint32_t id[2] = {id_n[0], id_n[1]}, sm[2] = {sm_n[0], sm_n[1]};
        if (sc + kDqWarps < s1) fetch(sc + kDqWarps);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (MODE == 1 && (h == 0 || a.GH == 2)) {
                if constexpr (T::kReg) {
                    uint32_t d[E / 2];
                    if (staged) load_entries<N>(d, slib + id[h] * kLibStride, [](auto* p) { return *p; });
                    else load_entries<N>(d, a.b.cb + (size_t)id[h] * E, [](auto* p) { return __ldg(p); });
                    affine_entries<N>(d, sm[h]);
                    book = book_of<N>(d);
                } else {
                    const float scale = h2f((uint16_t)(sm[h] & 0xffffu)), mid = h2f((uint16_t)(sm[h] >> 16));
                    auto decoded = [&](uint32_t v) { return (uint32_t)f2h(__fmaf_rn(scale, h2f((uint16_t)v), mid)); };
#pragma unroll
                    for (int q = 0; q < E; q += 8) {
                        uint4 l8;
                        if (staged) l8 = *(const uint4*)(slib + id[h] * kLibStride + q);
                        else l8 = __ldg((const uint4*)(a.b.cb + (size_t)id[h] * E + q));
                        const uint32_t lw[4] = {l8.x, l8.y, l8.z, l8.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            sts_u32(tab + (q + 2 * i) * 128, decoded(lw[i] & 0xffffu));
                            sts_u32(tab + (q + 2 * i + 1) * 128, decoded(lw[i] >> 16));
                        }
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {                 // 8 weights = 16 bytes
                uint4 v;
                if constexpr (T::kReg) {
                    v = reg_decode8_ordered<N>(w, h * 8 + c, book);
                } else {
                    uint32_t d[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int p = h * 32 + c * 4 + i;
                        d[i] = join16(lds_u32(single_addr<N, 1>(w, 2 * p, tab)), lds_u32(single_addr<N, 1>(w, 2 * p + 1, tab)));
                    }
                    v = make_uint4(d[0], d[1], d[2], d[3]);
                }
                *(uint4*)(tile + lane * kTileRow + c * 16) = v;
            }
            const uint32_t k0 = (uint32_t)sc * kSuper + h * 64;
            while (T::kReg && j < jend && (e & 0xffffu) < k0 + 64) {
                __half* t = (__half*)(tile + lane * kTileRow) + ((e & 0xffffu) - k0);
                *t = __hadd(*t, __ushort_as_half((uint16_t)(e >> 16)));
                if (++j < jend) e = entry(j);
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
    // ---- what is left of S, on the values this block has just stored ----
    const bool spills = a.ell_slots && len >= a.ell_slots && row < a.rows;
    if (__syncthreads_or(in_place || spills)) {
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
        if (in_place) {
            const int most = __reduce_max_sync(0xffffffffu, in_slab);
            for (int j = warp; j < most; j += kBatch * kDqWarps) batch(slab + 32, 32, j, in_slab);
        }
        if (spills) {                                   // the rest of the channel is in the CSR arrays
            const int p0 = __ldg(a.b.rowptr + row), n = __ldg(a.b.rowptr + row + 1) - p0;
            for (int j = a.ell_slots + warp; j < n; j += kBatch * kDqWarps) batch(a.b.oent + p0, 1, j, n);
        }
    }
}

// Super-chunks of a block, blocks of a row-block, whether outliers are added to the staged rows.
struct DqPlan { int range, parts; bool lists; };

DqPlan plan_of(const Layout& l) {
    const int sms = sm_count();
    const long long slots = 3ll * sms;
    int range = l.SC < kDqRange ? l.SC : kDqRange;
    auto parts = [&](int r) { return (l.SC + r - 1) / r; };
    if (l.bits > 4) {       // few row-blocks: shorter ranges, at least one super-chunk per warp, until the blocks fill the GPU twice
        while (range > kDqWarps && (long long)l.RB * parts(range) < 4ll * sms) range = (range + 1) / 2;
        return DqPlan{range, parts(range), false};
    }
    // Rounds of three blocks per SM times (turns of a warp and one for the block's first loads), in the fewest parts that reach
    // the least: 3072 x 4096 V2 N = 4 6.5 us with ranges of 8, 4096 x 4096 8.2 with 16, 10.9 with 24.
    long long best = -1;
    for (int n = parts(kDqRange); n <= parts(kDqWarps); ++n) {
        const int r = (l.SC + n - 1) / n;
        const long long cost = (l.RB * (long long)parts(r) + slots - 1) / slots * ((r + kDqWarps - 1) / kDqWarps + 1);
        if (best < 0 || cost < best) { best = cost; range = r; }
    }
    // Lists of the outliers in front of the decode, or in place behind the stores.  Every block walks all slots of its row-block
    // for either; the lists' walk stands in front of everything else.  They win where outliers are many and the matrix is not
    // cut into many parts: from 3 % on, and at N <= 3, whose decode is the shorter, from 1/128 on beyond four row-blocks per SM
    // and from 1/64 on for one part of up to 16 super-chunks (us, lists | in place: 28672 x 2048 N = 2, 2 % 36.8 | 41.5, 28672 x 8192
    // N = 2, 2 % 136 | 148, 1 % 115 | 121, 8192 x 2048 N = 3, 2 % 11.1 | 11.9; 12288 x 4096 N = 4, 5 % 49.9 | 74.9, 2 % 35.9 | 34.3,
    // 0.3 % 27.8 | 24.5; 512 x 2048 N = 4, 2 % 6.8 | 4.8).
    const long long weights = (long long)l.rows * l.cols;
    const bool many = l.nnz * 100 >= 3 * weights || (l.bits <= 3 && ((l.RB > 4 * sms && l.nnz * 128 >= weights) ||
                                                                     (l.SC <= 16 && l.nnz * 64 >= weights)));
    const bool lists = l.ell_slots != 0 && many && l.RB > sms && parts(range) <= 4;
    // More than a round of blocks without lists: short ranges, whose blocks the SMs take as they become free -- 16 super-chunks,
    // so that the slots are not walked too often, or 8 where there are none (28672 x 8192 V2 N = 4, 2 % 144 us with 16, 162
    // with 8, 196 with 32; without outliers 96.8, 92.7, 107; N = 2 without outliers 91.0, 85.2, 100).
    const int s = l.SC < 16 ? l.SC : l.ell_slots ? 16 : 8;
    if (!lists && (long long)l.RB * parts(16) > slots) range = (l.SC + parts(s) - 1) / parts(s);
    return DqPlan{range, parts(range), lists};
}

template <int N, int MODE>
cudaError_t launch_decode(const Layout& l, const void* packed, uint16_t* W, cudaStream_t s) {
    using T = DqTab<N, MODE>;
    DqArgs a = {};
    a.b = blob_at(packed, offsets_of(l));
    a.out = W;
    a.rows = l.rows; a.cols = l.cols; a.RB = l.RB; a.SC = l.SC; a.GH = l.GH; a.L = l.L; a.ell_slots = l.ell_slots;
    const size_t lib = MODE == 1 && a.L * T::E <= kLibEntries ? (size_t)a.L * (T::E + 8) * 2 : 0;
    const size_t smem = (1 + T::kTables) * T::kAlign + kDqWarps * 32 * kTileRow + (T::kReg ? kDqEntries + kDqStarts : 0) + lib;
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(dequant_kernel<N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    const DqPlan p = plan_of(l);
    a.range = p.range;
    a.lists = p.lists;
    dequant_kernel<N, MODE><<<(unsigned)(l.RB * p.parts), kDqWarps * 32, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

void dequant_plan_report(const Layout& l, int32_t* out) {
    const DqPlan p = plan_of(l);
    out[0] = p.range; out[1] = p.parts; out[2] = p.lists;
}

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
