// xfp_pack: unpacked tensors -> device layout (with range validation and clamping).
#include <cstdlib>

#include "xfp_internal.h"
#include "xfp_pair_common.cuh"

namespace xfp {

// ------------------------------------------------------------------------------------ pack
//
// One launch: the blocks of the grid are dealt to the six parts of the blob (index stream, codebooks, group
// metadata, row pointers, outlier entries, transposed slabs) by block index.  Every part reads the caller's tensors
// only -- the slabs apply the same clamping and neutralisation as the row pointers and entries they mirror -- so no
// part waits for another.  (As seven launches the small parts cost 28 of 94 us at 28672 x 8192 and set a floor of
// ~32 us on small matrices.)

constexpr int kPackThreads = 256;
constexpr int kPackWarps = kPackThreads / 32;

struct PackArgs {
    PackInputs in;
    char* base;             // the blob
    Layout l;
    int* err_word;
    bool counted;           // nothing is written when the last row pointer is not l.nnz
    // first block of every part, in this order: slabs, entries, rowptr, group, codebook, idx; [6] = grid.  (Spreading
    // the blocks of the small parts evenly among those of the index part measured the same: 110.6 against 106.5 us at
    // 28672 x 8192 with 2 % outliers.)
    unsigned first[7];
};

__device__ __forceinline__ int clampi(long long v, long long lo, long long hi) {
    return (int)(v < lo ? lo : (v > hi ? hi : v));
}

__device__ __forceinline__ long long col_at(const void* ocol, int col_bits, long long p) {
    return col_bits == 16 ? (long long)((const uint16_t*)ocol)[p] : (long long)((const int32_t*)ocol)[p];
}

// outlier p as the blob stores it: column | fp16 value << 16; a column outside the matrix becomes column 0, value +0
__device__ __forceinline__ uint32_t entry_at(const PackInputs& in, long long p, int cols, bool* bad) {
    long long c = col_at(in.ocol, in.col_bits, p);
    uint32_t v = in.oval[p];
    if (c < 0 || c >= cols) { *bad = true; c = 0; v = 0; }
    return (uint32_t)c | (v << 16);
}

// One warp per (row-block, super-chunk): 128 byte-indices of every channel -> N uint4 per lane.  The warp fetches its
// 32 x 128-byte tile of indices with whole 128-byte lines per quarter-warp and hands every lane its channel's row through
// shared memory (a lane reading its own row from global memory made every 16-byte load a line of its own: 16.3 M
// wavefronts on the L1 data pipe at 28672 x 8192 against 7.6 M this way).
template <int N>
__device__ __forceinline__ void pack_idx_block(const PackArgs& a, unsigned vblk, unsigned char* tiles) {
    constexpr uint32_t E = 1u << N;
    constexpr int kRowB = 144;   // bytes per tile row: 16-byte aligned, the lanes of a quarter-warp in distinct banks
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long unit = (long long)vblk * kPackWarps + warp;
    if (unit >= (long long)a.l.RB * a.l.SC) return;
    const int rb = (int)(unit / a.l.SC), sc = (int)(unit % a.l.SC);
    unsigned char* tile = tiles + warp * 32 * kRowB;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 4 * i + (lane >> 3), c = lane & 7;   // rows 4i .. 4i+3 of the tile, 16-byte chunk c
        const int row_g = rb * kRowsPerBlock + r;
        uint4 t = make_uint4(0u, 0u, 0u, 0u);
        if (row_g < a.l.rows) t = __ldg((const uint4*)(a.in.idx + (size_t)row_g * a.l.cols + (size_t)sc * kSuper) + c);
        *(uint4*)(tile + r * kRowB + c * 16) = t;
    }
    __syncwarp();
    uint32_t w[4 * N + 1];
#pragma unroll
    for (int i = 0; i < 4 * N + 1; ++i) w[i] = 0u;
    bool bad = false;
    if constexpr (N == 5) {         // index by index: 28672 x 8192 78 us against 87
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint4 t = *(const uint4*)(tile + lane * kRowB + i * 16);
            const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int b = 0; b < 16; ++b) {
                uint32_t q = (tw[b >> 2] >> ((b & 3) * 8)) & 0xffu;
                bad |= (q >= E);
                q &= E - 1u;
                const int j = i * 16 + b;
                const int bit = j * N, wi = bit >> 5, off = bit & 31;
                w[wi] |= q << off;
                if (off + N > 32) w[wi + 1] |= q >> (32 - off);
            }
        }
    } else {                        // four indices of a byte each to 4 N adjacent bits: 28672 x 8192 V2 N = 4 80 -> 70 us, N = 6 97 both ways
        uint32_t over = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint4 t = *(const uint4*)(tile + lane * kRowB + i * 16);
            const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                over |= tw[b];
                uint32_t q = tw[b] & ((E - 1u) * 0x01010101u);
                q = (q & 0x00ff00ffu) | ((q & 0xff00ff00u) >> (8 - N));
                q = (q & 0x0000ffffu) | ((q & 0xffff0000u) >> (16 - 2 * N));
                const int bit = (i * 4 + b) * 4 * N, wi = bit >> 5, off = bit & 31;
                w[wi] |= q << off;
                if (off + 4 * N > 32) w[wi + 1] |= q >> (32 - off);
            }
        }
        bad = (over & ~((E - 1u) * 0x01010101u)) != 0;
    }
    if (bad && a.err_word) atomicOr(a.err_word, 1);
    uint4* dst = (uint4*)(a.base + a.l.off_idx) + ((size_t)unit * N) * 32 + lane;
#pragma unroll
    for (int v = 0; v < N; ++v) dst[(size_t)v * 32] = make_uint4(w[4 * v], w[4 * v + 1], w[4 * v + 2], w[4 * v + 3]);
}

__device__ __forceinline__ void pack_codebook_block(const PackArgs& a, unsigned vblk) {
    const long long n_src = (long long)(a.l.mode ? a.l.L : a.l.rows) * a.l.E;
    const long long n_dst = (long long)(a.l.mode ? a.l.L : a.l.rows_pad) * a.l.E;
    const long long t = (long long)vblk * kPackThreads + threadIdx.x;
    uint16_t* out = (uint16_t*)(a.base + a.l.off_cb);
    if (t < n_dst) out[t] = t < n_src ? a.in.codebook[t] : (uint16_t)0;
}

__device__ __forceinline__ void pack_group_block(const PackArgs& a, unsigned vblk) {
    // one thread per (row-block, super-chunk, part of the super-chunk, lane); the group that holds the part's first
    // weight supplies its metadata (a group of 256 weights is stored with both of its super-chunks)
    const Layout& l = a.l;
    const long long t = (long long)vblk * kPackThreads + threadIdx.x;
    if (t >= (long long)l.RB * l.SC * l.GH * 32) return;
    const int lane = (int)(t & 31);
    const long long part = t >> 5;
    const long long unit = part / l.GH;
    const int h = (int)(part % l.GH);
    const int rb = (int)(unit / l.SC), sc = (int)(unit % l.SC);
    const int row = rb * kRowsPerBlock + lane;
    const int groups = l.SC * kSuper / l.G;                        // groups per channel
    const int grp = (sc * kSuper + h * (kSuper / l.GH)) / l.G;
    uint32_t id = 0, sm = 0;
    if (row < l.rows) {
        id = a.in.gid[(size_t)row * groups + grp];
        if ((int)id >= l.L) {
            if (a.err_word) atomicOr(a.err_word, 2);
            id = (uint32_t)(l.L - 1);
        }
        sm = (uint32_t)a.in.gscale[(size_t)row * groups + grp] | ((uint32_t)a.in.gmid[(size_t)row * groups + grp] << 16);
    }
    ((uint8_t*)(a.base + l.off_gid))[t] = (uint8_t)id;
    ((uint32_t*)(a.base + l.off_gsm))[t] = sm;
}

// rowptr -> clamped copy (padding rows empty); checks monotonicity and the end points (that the columns of a row
// ascend strictly is checked where the entries are read in order, in ell_fill_block).  The first thread writes the
// header words.
__device__ __forceinline__ void pack_rowptr_block(const PackArgs& a, unsigned vblk) {
    const Layout& l = a.l;
    const int t = (int)(vblk * kPackThreads + threadIdx.x);
    if (t == 0) {
        int* hdr = (int*)(a.base + l.off_hdr);
        hdr[0] = l.ell_slots;
        hdr[1] = 0;
        *(long long*)(hdr + 2) = (long long)l.off_ell;
    }
    if (t > l.rows_pad) return;
    int* out = (int*)(a.base + l.off_rowptr);
    if (l.nnz == 0) {
        out[t] = 0;
        return;
    }
    const long long nnz = l.nnz;
    int bad = 0;
    long long v = t <= l.rows ? (long long)a.in.rowptr[t] : nnz;
    if (t == 0 && v != 0) bad |= 4;
    if (t == l.rows && v != nnz) bad |= 4;
    if (v < 0 || v > nnz) bad |= 4;
    if (t < l.rows) {
        long long nx = a.in.rowptr[t + 1];
        if (nx < v) bad |= 4;
    }
    out[t] = clampi(v, 0, nnz);
    if (bad && a.err_word) atomicOr(a.err_word, bad);
}

__device__ __forceinline__ void pack_entries_block(const PackArgs& a, unsigned vblk) {
    const long long p = (long long)vblk * kPackThreads + threadIdx.x;
    if (p >= a.l.nnz) return;
    bool bad = false;
    ((uint32_t*)(a.base + a.l.off_oent))[p] = entry_at(a.in, p, a.l.cols, &bad);
    if (bad && a.err_word) atomicOr(a.err_word, 8);
}

// Transposed outlier slab of row-block b: word [0][lane] = slots used by channel b*32+lane, word [1+j][lane] = its
// j-th outlier or the neutral entry (column 0, value +0).  Reads the caller's row pointers and entries with the
// clamping of pack_rowptr_block and pack_entries_block.  The block's entries are one contiguous range of the CSR
// arrays: a warp takes a channel and reads its entries in order (coalesced), each entry goes to its slot of a copy of
// the slab in shared memory (windows of 256 slots), which is then written out in whole lines.  (Every lane walking its
// own row -- 32 scattered sectors per load --, scattered 4-byte stores into the slab, and a binary search of every
// entry for its channel each made this part 50-60 us at 2 % outliers on 28672 x 8192.)  The same pass checks that the
// columns of a row ascend strictly.  Row pointers that do not ascend (reported by pack_rowptr_block) leave slots
// neutral, never an access outside the arrays.
constexpr int kEllWindow = 256;   // slots of the slab held in shared memory at a time
__device__ __forceinline__ void ell_fill_block(const PackArgs& a, unsigned b, unsigned char* smem) {
    const Layout& l = a.l;
    uint32_t* sl = (uint32_t*)smem;                       // [kEllWindow][33]: consecutive slots of one channel in consecutive banks
    int* rp = (int*)(smem + kEllWindow * 33 * 4);         // [33]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = l.ell_slots;
    const long long nnz = l.nnz;
    if (threadIdx.x < 33) {
        const int row = (int)b * 32 + (int)threadIdx.x;
        rp[threadIdx.x] = row <= l.rows ? clampi(a.in.rowptr[row], 0, nnz) : (int)nnz;
    }
    __syncthreads();
    uint32_t* slab = (uint32_t*)(a.base + l.off_ell) + (size_t)b * (C + 1) * 32;
    if (warp == 0) {
        const int p0 = rp[lane], p1 = rp[lane + 1];
        slab[lane] = (uint32_t)(p1 > p0 ? min(p1 - p0, C) : 0);
    }
    int bad = 0;   // a column outside the matrix is reported by pack_entries_block
    for (int j0 = 0; j0 < C; j0 += kEllWindow) {
        const int nj = min(kEllWindow, C - j0);
        for (int i = threadIdx.x; i < nj * 33; i += kPackThreads) sl[i] = 0u;
        __syncthreads();
        for (int r = warp; r < 32; r += kPackWarps) {   // a warp per channel, its lanes along the channel's entries
            const int p0 = rp[r], n = rp[r + 1] - p0;   // n <= 0: an empty channel, or row pointers that descend
            for (int jj = lane; jj < n; jj += 32) {
                const int p = p0 + jj;
                if (j0 == 0 && jj > 0 && col_at(a.in.ocol, a.in.col_bits, p) <= col_at(a.in.ocol, a.in.col_bits, p - 1)) bad = 16;
                bool outside = false;
                if (jj >= j0 && jj < j0 + nj) sl[(jj - j0) * 33 + r] = entry_at(a.in, p, l.cols, &outside);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nj * 32; i += kPackThreads) slab[(size_t)(1 + j0) * 32 + i] = sl[(i >> 5) * 33 + (i & 31)];
        __syncthreads();
    }
    if (bad && a.err_word) atomicOr(a.err_word, bad);
}

template <int N>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(const PackArgs a) {
    __shared__ __align__(16) unsigned char tiles[kPackWarps * 32 * 144];   // 36864 bytes; the slab part uses 33792 + 132
    static_assert(kPackWarps * 32 * 144 >= kEllWindow * 33 * 4 + 33 * 4, "slab window and row pointers fit the tile area");
    const unsigned b = blockIdx.x;
    if (a.counted && __ldg(a.in.rowptr + a.l.rows) != a.l.nnz) return;
    if (b < a.first[1]) ell_fill_block(a, b, tiles);
    else if (b < a.first[2]) pack_entries_block(a, b - a.first[1]);
    else if (b < a.first[3]) pack_rowptr_block(a, b - a.first[2]);
    else if (b < a.first[4]) pack_group_block(a, b - a.first[3]);
    else if (b < a.first[5]) pack_codebook_block(a, b - a.first[4]);
    else pack_idx_block<N>(a, b - a.first[5], tiles);
}

cudaError_t launch_pack(const Layout& l, const PackInputs& in, void* packed, int* err_word, cudaStream_t s, bool counted) {
    PackArgs a;
    a.in = in; a.base = (char*)packed; a.l = l; a.err_word = err_word; a.counted = counted;
    auto blocks = [](long long n, int per) { return (unsigned)((n + per - 1) / per); };
    const long long n_cb = (long long)(l.mode ? l.L : l.rows_pad) * l.E;
    unsigned n[6];
    n[0] = l.nnz ? (unsigned)l.RB : 0u;
    n[1] = l.nnz ? blocks(l.nnz, kPackThreads) : 0u;
    n[2] = blocks((long long)l.rows_pad + 1, kPackThreads);
    n[3] = l.mode ? blocks((long long)l.RB * l.SC * l.GH * 32, kPackThreads) : 0u;
    n[4] = blocks(n_cb, kPackThreads);
    n[5] = blocks((long long)l.RB * l.SC, kPackWarps);
#ifdef LANE_TUNE
    if (const char* e = getenv("XFP_PACK_SKIP"))   // tuning build: leave parts out (bit i = part i) to time the others
        for (int i = 0; i < 6; ++i)
            if ((atoi(e) >> i) & 1) n[i] = 0;
#endif
    a.first[0] = 0;
    for (int i = 0; i < 6; ++i) a.first[i + 1] = a.first[i] + n[i];
    switch (l.bits) {
        case 2: pack_kernel<2><<<a.first[6], kPackThreads, 0, s>>>(a); break;
        case 3: pack_kernel<3><<<a.first[6], kPackThreads, 0, s>>>(a); break;
        case 4: pack_kernel<4><<<a.first[6], kPackThreads, 0, s>>>(a); break;
        case 5: pack_kernel<5><<<a.first[6], kPackThreads, 0, s>>>(a); break;
        default: pack_kernel<6><<<a.first[6], kPackThreads, 0, s>>>(a); break;
    }
    return cudaGetLastError();
}

}  // namespace xfp
