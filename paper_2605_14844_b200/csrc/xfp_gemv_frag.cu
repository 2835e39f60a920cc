// Fused decode for 1..16 rows of x, V2 and V2a, in the tensor cores' own operand layout:  y[b] = (D + S) x[b].
//
// The lane kernels (xfp_gemv_lane.cuh, xfp_gemv_pair.cu, xfp_gemv_batch.cu) keep a channel's decoded weights in one lane, so x
// has to sit on the diagonal lanes of the B operand and every row of x costs an mma and two shared-memory wavefronts per 8
// weights of a lane.  Here lane (g, t) of a warp, g = lane / 4, t = lane mod 4, takes the t-th 32 of a super-chunk's 128
// weights of the four channels g, g + 8, g + 16, g + 24 of a row-block.  That is the A operand of mma.m16n8k16 as it stands --
// the order of k inside a super-chunk is free, and step s multiplies the k 32 t + 4 s .. + 3 of every t -- so one mma serves
// eight rows of x, none of the staged x that is read is wasted, and an accumulator holds four channels' sums: V2a's scale and
// mid-point are applied in place, without a shuffle.
//
//   look-ups  four lanes share a channel, so a table is kept in four copies, one per t: entry (..)*128 + lane*4 lies in the
//             lane's own bank.  V2: pair tables up to N = 4 (128 KB of four channels' tables at N = 4), one entry per index
//             above.  V2a: the library once per bank, two library ids to a word.  At N = 4 entries lie 256 bytes apart, two
//             tables interleaved, so that one PRMT turns an index (V2: a byte of two) into the address.
//   x         staged once per CTA (fp16; bf16 is converted on the way), 16 bytes = eight rows per k, for ldmatrix.trans.  CTAs
//             are resident and walk the row-blocks, so that x is staged once; a K too long for shared memory is cut into
//             slices, a CTA staying in its slice.
//   outliers  a lane per channel, slots of the transposed slab dealt to the warps; eight products per load of x.
//             (The same walk over x as rows of k cost eight loads of two bytes per entry, 5 way conflicts each: 12288 x 4096, 8
//             rows, 5 % outliers 32.1 -> 24.0 us.)
//   sums      fragments -> shared memory -> fixed order over the warps; K slices meet in the workspace, the last to come adds
//             them in order (a ticket, no waiting).
#include "xfp_internal.h"
#include "xfp_pair_common.cuh"

namespace xfp {

namespace {

constexpr int kFW = 16;              // warps
constexpr int kFThreads = kFW * 32;
constexpr size_t kFSmem = 224 * 1024;

struct FragArgs {
    Blob b;
    const uint16_t* x;
    void* y;
    float* partial;   // [row-block][slice][NB][32]
    int* tickets;     // [row-block]
    int rows, cols, RB, SC, ell_slots, L;
    int nb, y_kind, x_bf16;
    int S, sc_slice;  // K slices, super-chunks of each
    int x_off, red_off;   // bytes behind the tables: staged x, per-warp sums
};

// Tables.  V2: one per channel group j, [entries][32 lanes] words (entry = pair of indices with PAIR, N <= 4).  V2a: one per two
// library ids, [2^N][32] words of two fp16.  kStride bytes from entry to entry: 128, at N = 4 256 with tables 2 i and 2 i + 1
// interleaved.
template <int N, int MODE, bool PAIR>
struct FTab {
    static constexpr int E = 1 << N;
    static constexpr bool kPair = PAIR;
    static constexpr int kEntries = kPair ? E * E : E;
    static constexpr int kStride = N == 4 ? 256 : 128;
    // byte offset of table i
    __host__ __device__ static constexpr uint32_t at(uint32_t i) {
        return N == 4 ? (i >> 1) * (uint32_t)(kEntries * 256) + (i & 1u) * 128u : i * (uint32_t)(kEntries * 128);
    }
};

// The lane's words [t N, (t + 1) N) of the index streams of its four channels of super-chunk sc.
template <int N>
__device__ __forceinline__ void load_words(uint32_t (&w)[4][N], const uint4* idx, int g, int t) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int ch = g + 8 * j;
        if (N == 4) {
            const uint4 v = ld_stream(idx + t * 32 + ch);
            w[j][0] = v.x; w[j][1] = v.y; w[j][2 % N] = v.z; w[j][3 % N] = v.w;
        } else if (N % 2 == 0) {
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                const int wd = t * N + 2 * i;
                const uint2 v = __ldg((const uint2*)(idx + (wd >> 2) * 32 + ch) + ((wd >> 1) & 1));
                w[j][(2 * i) % N] = v.x; w[j][(2 * i + 1) % N] = v.y;
            }
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int wd = t * N + i;
                w[j][i] = __ldg((const uint32_t*)(idx + (wd >> 2) * 32 + ch) + (wd & 3));
            }
        }
    }
}

// A load that stays where it is written: the compiler sank the plain form of these early loads to their uses, behind the K loop,
// where a row-block then waited 2000 - 3800 clocks for them.
__device__ __forceinline__ uint32_t ld_early(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld_early2(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_early4(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_early16(const uint16_t* p) {
    uint16_t v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// Staged x: [tile of eight rows][k][8 rows], 16 bytes per k, which ldmatrix.trans turns into B fragments and which gives an outlier
// its eight values in one load.  The byte offset of k in a tile: the place of k among the eight of its chunk is exclusive-or'ed so that the eight k of a fragment (32 t + 0, 1) and eight staging threads (consecutive chunks) each
// meet eight bank groups.
__device__ __forceinline__ uint32_t x_at(int k) {
    const int c = k >> 3;
    return (uint32_t)(k ^ (c & 7) ^ (((c >> 2) & 3) << 1)) << 4;
}

__device__ __forceinline__ uint32_t word(const uint4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

__device__ __forceinline__ uint4 ldmatrix_x4_trans(uint32_t addr) {
    uint4 v;
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

template <int N, int MODE, int NB, bool PAIR>
__global__ void __launch_bounds__(kFThreads, 1) gemv_frag_kernel(const FragArgs a) {
    using T = FTab<N, MODE, PAIR>;
    constexpr int E = T::E;
    constexpr int NT = NB > 8 ? 2 : 1;                 // tiles of eight rows of x
    constexpr int kAhead = N <= 4 ? 2 : 1;             // super-chunks of indices in flight per warp
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sX = smem + a.x_off;
    float* red = (float*)(smem + a.red_off);           // [warp][NB][33]
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int slice = (int)blockIdx.x % a.S;
    const int sc0 = slice * a.sc_slice, sc1 = min(a.SC, sc0 + a.sc_slice), nsc = sc1 - sc0;
    float* sXg = (float*)(sX + (size_t)nsc * kSuper * NB * 2);      // V2a: sums of x over a group, [super-chunk][NB]
    const int step = (int)gridDim.x / a.S;
    const uint32_t tile = (uint32_t)nsc * kSuper * 16;              // bytes of a tile of eight rows
    // the lane's row of the four 8 x 8 matrices of two mma steps: k = 32 (r / 2) + 2 m + r mod 2, r = lane mod 8, m = lane / 8
    const uint32_t xrow = (uint32_t)__cvta_generic_to_shared(sX) + x_at(32 * ((lane & 7) >> 1) + 2 * (lane >> 3) + (lane & 1));

    // a thread's share of a row-block's codebooks (V2), on its way while the previous row-block is finished: the whole codebook
    // of its channel where pairs are built, else the entries its warp stores
    constexpr int kCb = MODE ? 1 : T::kPair ? E / 2 : (E + kFW - 1) / kFW;
    uint32_t cbn[kCb];
    auto book = [&](int rb) {
        const uint16_t* cb = a.b.cb + (size_t)(rb * kRowsPerBlock + lane) * E;
        if (T::kPair) {
            if (E == 4) {
                const uint2 p = ld_early2((const uint2*)cb);
                cbn[0] = p.x; cbn[1 % kCb] = p.y;
            } else {
#pragma unroll
                for (int e = 0; e < E / 8; ++e) {
                    const uint4 p = ld_early4((const uint4*)cb + e);
                    cbn[(4 * e) % kCb] = p.x; cbn[(4 * e + 1) % kCb] = p.y; cbn[(4 * e + 2) % kCb] = p.z; cbn[(4 * e + 3) % kCb] = p.w;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < kCb; ++i) cbn[i] = ld_early16(cb + warp + i * kFW);
        }
    };
    auto fill = [&]() {
        const int ch = lane, j = ch >> 3;
        unsigned char* dst = smem + T::at(j) + (ch & 7) * 16;
        if (T::kPair) {
            // a thread takes a channel and every sixteenth entry; one 16-byte store writes the four copies
#pragma unroll
            for (int hi = 0; hi < E; ++hi) {
                if (hi != warp % (E < kFW ? E : kFW)) continue;
#pragma unroll
                for (int lo = 0; lo < E; ++lo) {
                    if (E < kFW && (lo % (kFW / E)) != warp / E) continue;
                    const uint32_t p = __byte_perm(cbn[(lo / 2) % kCb], cbn[(hi / 2) % kCb], ((lo & 1) ? 0x32 : 0x10) | ((hi & 1) ? 0x7600 : 0x5400));
                    *(uint4*)(dst + (size_t)(lo | (hi << N)) * T::kStride) = make_uint4(p, p, p, p);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < kCb; ++i) {
                const uint32_t p = cbn[i];
                *(uint4*)(dst + (size_t)(warp + i * kFW) * T::kStride) = make_uint4(p, p, p, p);
            }
        }
    };
    // indices (and V2a metadata) of the warp's next super-chunks
    uint32_t nx[kAhead][4][N];
    uint32_t id_n[kAhead][4], sm_n[kAhead][4];
    auto fetch = [&](int rb, int sc, int slot) {
        load_words<N>(nx[slot], a.b.idx + ((size_t)rb * a.SC + sc) * N * 32, g, t);
        if (MODE == 1) {
            const size_t m = ((size_t)rb * a.SC + sc) * 32 + g;
#pragma unroll
            for (int j = 0; j < 4; ++j) { id_n[slot][j] = __ldg(a.b.gid + m + 8 * j); sm_n[slot][j] = __ldg(a.b.gsm + m + 8 * j); }
        }
    };

    // ---- what does not depend on the previous kernel: indices, tables ----
    asm volatile("griddepcontrol.launch_dependents;");
    int rb = (int)blockIdx.x / a.S;
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
        if (rb < a.RB && sc0 + warp + i * kFW < sc1) fetch(rb, sc0 + warp + i * kFW, i);
    if (MODE == 1) {
        const int words = (a.L + 1) / 2 * E;
        for (int i0 = warp * 32; i0 < words; i0 += kFW * 32) {      // a lane fetches a word, the warp stores 32 of them
            const int i = i0 + lane, id = i / E * 2, q = i % E;
            uint32_t v = 0;
            if (i < words) v = (uint32_t)__ldg(a.b.cb + id * E + q) | (id + 1 < a.L ? (uint32_t)__ldg(a.b.cb + (id + 1) * E + q) << 16 : 0u);
#pragma unroll 8
            for (int k = 0; k < 32; ++k) {
                const uint32_t o = __shfl_sync(0xffffffffu, v, k);
                if (i0 + k < words) *(uint32_t*)(smem + T::at((uint32_t)((i0 + k) / E)) + (size_t)((i0 + k) % E) * T::kStride + lane * 4) = o;
            }
        }
    } else if (rb < a.RB) {
        book(rb);
        fill();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ---- x: chunks of a row by consecutive threads ----
    {
        constexpr int kRows = 8;                       // loads in flight per thread
        const int chunks = nsc * (kSuper / 8);
        const uint4* xs = (const uint4*)(a.x + (size_t)sc0 * kSuper);
        const int row16 = a.cols / 8;
#pragma unroll
        for (int b0 = 0; b0 < NB; b0 += kRows) {
            for (int c = tid; c < chunks; c += kFThreads) {
                uint4 v[kRows];
#pragma unroll
                for (int b = 0; b < kRows; ++b) v[b] = b0 + b < a.nb ? __ldg(xs + (size_t)(b0 + b) * row16 + c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int b = 0; b < kRows; ++b) v[b] = x8_as_f16(v[b], a.x_bf16);
                unsigned char* dst = sX + (size_t)(b0 / 8) * tile;
#pragma unroll
                for (int i = 0; i < 8; ++i) {          // k = 8 c + i of the eight rows
                    auto two = [&](int b) { return __byte_perm(word(v[b], i >> 1), word(v[b + 1], i >> 1), (i & 1) ? 0x7632 : 0x5410); };
                    *(uint4*)(dst + x_at(8 * c + i)) = make_uint4(two(0), two(2), two(4), two(6));
                }
                if constexpr (MODE == 1) {
                    // sums of a super-chunk: over the thread's eight k, then over the sixteen threads that hold its chunks
                    float f[kRows];
#pragma unroll
                    for (int b = 0; b < kRows; ++b) {
                        const float2 p0 = __half22float2(*(const __half2*)&v[b].x), p1 = __half22float2(*(const __half2*)&v[b].y),
                                     p2 = __half22float2(*(const __half2*)&v[b].z), p3 = __half22float2(*(const __half2*)&v[b].w);
                        f[b] = ((p0.x + p0.y) + (p1.x + p1.y)) + ((p2.x + p2.y) + (p3.x + p3.y));
                    }
                    const uint32_t half = 0xffffu << (lane & 16);
                    int row = 0;
#pragma unroll
                    for (int w = kRows / 2, d = 1; w >= 1; w /= 2, d *= 2) {   // halve the rows a lane keeps
                        const bool up = lane & d;
#pragma unroll
                        for (int b = 0; b < w; ++b) {
                            const float give = up ? f[b] : f[b + w], keep = up ? f[b + w] : f[b];
                            f[b] = keep + __shfl_xor_sync(half, give, d);
                        }
                        if (up) row += w;
                    }
                    f[0] += __shfl_xor_sync(half, f[0], 8);
                    if ((lane & 15) < kRows) sXg[(c >> 4) * NB + b0 + row] = f[0];
                }
            }
        }
    }
    __syncthreads();

    const uint32_t lbase = (uint32_t)lane * 4u;
    for (bool later = false; rb < a.RB; rb += step, later = true) {
        if (later) {
            __syncthreads();                           // tables and sums of the previous row-block are done with
            if (MODE == 0) { fill(); __syncthreads(); }
        }
        float acc[NT][2][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[n][i >> 2][i & 3] = 0.f;
        // the row-block's first outliers travel under the loop
        const int row = rb * kRowsPerBlock + lane;
        const uint32_t* slab = a.b.ell + (size_t)rb * (a.ell_slots + 1) * 32 + lane;
        constexpr int kEnt = 3;
        uint32_t len = 0, ent[kEnt] = {};
        if (a.ell_slots) {
            len = ld_early(slab);
#pragma unroll
            for (int i = 0; i < kEnt; ++i)
                if (warp + i * kFW < a.ell_slots) ent[i] = ld_early(slab + (size_t)(1 + warp + i * kFW) * 32);
        }
        for (int scu = sc0 + warp; scu < sc1; scu += kAhead * kFW) {
#pragma unroll
          for (int u = 0; u < kAhead; ++u) {
            const int sc = scu + u * kFW;
            if (sc >= sc1) break;
            uint32_t base[4];
            float scale[4], mid[4];
            if (MODE == 1) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const __half2 sm = *(const __half2*)&sm_n[u][j];
                    scale[j] = __low2float(sm); mid[j] = __high2float(sm);
                    base[j] = T::at(id_n[u][j] >> 1) + lbase + (id_n[u][j] & 1u) * 2u;
                }
            }
            const int lsc = sc - sc0;
            float c[NT][2][4];
            if (MODE == 1) {
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int i = 0; i < 8; ++i) c[n][i >> 2][i & 3] = 0.f;
            }
            float(&d)[NT][2][4] = MODE == 1 ? c : acc;
#pragma unroll
            for (int s2 = 0; s2 < 4; ++s2) {           // two mma steps: 8 k of every t
                uint4 xb[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    // chunk s2 of each t: the exclusive-or of x_at has s2 as its two low bits
                    xb[n] = ldmatrix_x4_trans((xrow ^ (uint32_t)(s2 << 4)) + (uint32_t)(lsc * kSuper * 16 + s2 * 128) + n * tile);
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int p0 = 4 * s2 + 2 * s;     // pairs p0, p0 + 1 of the lane's 16
                    uint32_t av[4][2];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int v = 0; v < 2; ++v) {
                            const uint32_t* w = nx[u][j];
                            const int p = p0 + v;
                            if (T::kPair) {
                                // the second of two interleaved tables: its 128 bytes ride in the base
                                const uint32_t off = N == 4 ? pair_addr<N, 2>(w, p, lbase | ((j & 1) * 128u)) : pair_addr<N, 1>(w, p, lbase);
                                av[j][v] = *(const uint32_t*)(smem + (N == 4 ? T::at(j & ~1) : T::at(j)) + off);
                            } else if (MODE == 0 && N == 4) {
                                const uint32_t lb = lbase | ((j & 1) * 128u), sel = 0x7604u | ((uint32_t)(p & 3) << 4);
                                const uint32_t lo = *(const uint32_t*)(smem + T::at(j & ~1) + __byte_perm(w[p >> 2] & 0x0f0f0f0fu, lb, sel));
                                const uint32_t hi = *(const uint32_t*)(smem + T::at(j & ~1) + __byte_perm((w[p >> 2] >> 4) & 0x0f0f0f0fu, lb, sel));
                                av[j][v] = join16(lo, hi);
                            } else if (MODE == 0) {
                                const uint32_t lo = *(const uint32_t*)(smem + T::at(j) + single_addr<N, 1>(w, 2 * p, lbase));
                                const uint32_t hi = *(const uint32_t*)(smem + T::at(j) + single_addr<N, 1>(w, 2 * p + 1, lbase));
                                av[j][v] = join16(lo, hi);
                            } else if (N == 4) {
                                // byte 1 of the address: index and the low four bits of id / 4
                                const uint32_t nib = ((base[j] >> 12) & 0xfu) * 0x10101010u, sel = 0x7604u | ((uint32_t)(p & 3) << 4);
                                const uint32_t wlo = (w[p >> 2] & 0x0f0f0f0fu) | nib, whi = ((w[p >> 2] >> 4) & 0x0f0f0f0fu) | nib;
                                const uint32_t lo = *(const uint16_t*)(smem + __byte_perm(wlo, base[j], sel));
                                const uint32_t hi = *(const uint16_t*)(smem + __byte_perm(whi, base[j], sel));
                                av[j][v] = join16(lo, hi);
                            } else {
                                const uint32_t lo = *(const uint16_t*)(smem + single_addr<N, 1>(w, 2 * p, base[j]));
                                const uint32_t hi = *(const uint16_t*)(smem + single_addr<N, 1>(w, 2 * p + 1, base[j]));
                                av[j][v] = join16(lo, hi);
                            }
                        }
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        const uint32_t b0 = s ? xb[n].z : xb[n].x, b1 = s ? xb[n].w : xb[n].y;
                        mma16816(d[n][0], av[0][0], av[1][0], av[0][1], av[1][1], b0, b1);
                        mma16816(d[n][1], av[2][0], av[3][0], av[2][1], av[3][1], b0, b1);
                    }
                }
            }
            if (MODE == 1) {
                // accumulator element e of tile i: channel g + 8 (e / 2) + 16 i, row of x 2 t + e mod 2
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const int b = 2 * t + 8 * n;
                    const float2 xs = *(const float2*)(sXg + lsc * NB + b);
                    const float x0 = xs.x, x1 = xs.y;
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int j = 2 * i + (e >> 1);
                            acc[n][i][e] = fmaf(scale[j], c[n][i][e], fmaf(mid[j], (e & 1) ? x1 : x0, acc[n][i][e]));
                        }
                }
            }
            // the slot's next super-chunk, or the one that it holds first of the CTA's next row-block
            if (sc + kAhead * kFW < sc1) fetch(rb, sc + kAhead * kFW, u);
            else if (rb + step < a.RB) fetch(rb + step, sc0 + warp + u * kFW, u);
          }
        }
        if (MODE == 0 && rb + step < a.RB) book(rb + step);
        // ---- outliers: lane = channel ----
        float ao[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) ao[b] = 0.f;
        if (a.ell_slots) {
            const int nslab = min((int)len, a.ell_slots);
            const uint32_t k0 = (uint32_t)sc0 * kSuper, kn = (uint32_t)nsc * kSuper;
            auto add = [&](uint32_t e) {
                const uint32_t k = (e & 0xffffu) - k0;
                if (k < kn) {
                    const float v = h2f((uint16_t)(e >> 16));
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        const uint4 x8 = *(const uint4*)(sX + n * tile + x_at((int)k));
                        const uint32_t u[4] = {x8.x, x8.y, x8.z, x8.w};
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const float2 f = __half22float2(*(const __half2*)&u[b]);
                            ao[8 * n + 2 * b] = fmaf(v, f.x, ao[8 * n + 2 * b]);
                            ao[8 * n + 2 * b + 1] = fmaf(v, f.y, ao[8 * n + 2 * b + 1]);
                        }
                    }
                }
            };
            const int most = __reduce_max_sync(0xffffffffu, nslab);
#pragma unroll
            for (int i = 0; i < kEnt; ++i)
                if (warp + i * kFW < nslab) add(ent[i]);
            for (int j0 = warp + kEnt * kFW; j0 < most; j0 += 4 * kFW) {
                uint32_t e[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) e[i] = j0 + i * kFW < nslab ? __ldg(slab + (size_t)(1 + j0 + i * kFW) * 32) : 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i) if (j0 + i * kFW < nslab) add(e[i]);
            }
            if ((int)len >= a.ell_slots && row < a.rows) {  // the channel overflows its slab: the rest is in the CSR arrays
                const int p1 = __ldg(a.b.rowptr + row + 1);
                for (int p = __ldg(a.b.rowptr + row) + a.ell_slots + warp; p < p1; p += kFW) add(__ldg(a.b.oent + p));
            }
        }
        // ---- sums over the warps ----
        float* mine = red + (size_t)warp * NB * 33;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int b = 2 * t + 8 * n + (e & 1);
                    mine[b * 33 + g + 8 * (2 * i + (e >> 1))] = acc[n][i][e];
                }
        __syncwarp();
        if (a.ell_slots) {
#pragma unroll
            for (int b = 0; b < NB; ++b) mine[b * 33 + lane] += ao[b];
        }
        __syncthreads();
        float sum = 0.f;
        const int b = tid >> 5;
        if (b < a.nb) {
#pragma unroll
            for (int w = 0; w < kFW; ++w) sum += red[(w * NB + b) * 33 + lane];
        }
        if (a.S == 1) {
            if (b < a.nb && row < a.rows) put_y(a.y, (size_t)b * a.rows + row, sum, a.y_kind);
        } else {
            float* part = a.partial + ((size_t)rb * a.S * NB + b) * 32 + lane;
            if (b < a.nb) __stcg(part + (size_t)slice * NB * 32, sum);
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                s_last = atomicAdd(a.tickets + rb, 1) == a.S - 1;
                if (s_last) a.tickets[rb] = 0;
                __threadfence();
            }
            __syncthreads();
            if (s_last && b < a.nb && row < a.rows) {
                sum = 0.f;
                for (int s = 0; s < a.S; ++s) sum += __ldcg(part + (size_t)s * NB * 32);
                put_y(a.y, (size_t)b * a.rows + row, sum, a.y_kind);
            }
        }
    }
}

struct FragPlan { int S, sc_slice, grid, pair, room; size_t x_off, red_off, smem; };

size_t table_bytes(const Layout& l, bool pair) {
    if (l.mode) { const int n = (l.L + 1) / 2; return (size_t)(l.bits == 4 ? (n + 1) & ~1 : n) * l.E * 128; }
    return (size_t)4 * (pair ? l.E * l.E : l.E) * 128;
}

bool plan_frag(const Layout& l, int batch, int sms, FragPlan& p) {
    const int NB = batch <= 8 ? 8 : 16;
    const size_t red = (size_t)kFW * NB * 33 * 4 + 16;
    const size_t per_sc = (size_t)kSuper * NB * 2 + (l.mode ? NB * 4 : 0);
    auto slices = [&](bool pair) {                                    // K slices that x needs beside the tables
        const size_t used = table_bytes(l, pair) + red;
        const int fit = used + per_sc > kFSmem ? 0 : (int)((kFSmem - used) / per_sc);
        return fit ? (l.SC + fit - 1) / fit : 0;
    };
    // N = 4: pair tables take 128 of 224 KB, and a slice more means that the tables are built once more and the outliers walked
    // once more; where single entries (8 KB) need fewer slices they are the faster ones
    p.pair = l.mode == 0 && l.bits <= 4;
    int S = slices(p.pair);
    if (p.pair && l.bits == 4) {
        const int s1 = slices(false);
        if (!S || s1 < S) { p.pair = 0; S = s1; }
    }
    if (!S) return false;
    p.room = S;
    // few row-blocks: K slices until the SMs are busy, at least one super-chunk per warp, and no more than the workspace that
    // every GEMV kernel shares holds partial sums of, behind the counters
    const size_t ws = workspace_bytes_for(l), ctrl = align256((size_t)l.RB * 4), per_slice = (size_t)l.RB * NB * 32 * 4;
    const long long held = ws > ctrl ? (long long)((ws - ctrl) / per_slice) : 0;
    while (l.RB * (S + 1) <= sms && l.SC / (S + 1) >= kFW && S < held) ++S;
    p.sc_slice = (l.SC + S - 1) / S;
    p.S = (l.SC + p.sc_slice - 1) / p.sc_slice;
    if (p.S > 1 && p.S > held) return false;
    const int ctas = sms / p.S * p.S;
    if (ctas < 1) return false;
    p.grid = l.RB * p.S < ctas ? l.RB * p.S : ctas;
    p.x_off = table_bytes(l, p.pair);
    p.red_off = (p.x_off + (size_t)p.sc_slice * per_sc + 15) & ~size_t(15);
    p.smem = p.red_off + red;
    return true;
}

template <int N, int MODE, int NB, bool PAIR>
cudaError_t launch_one(const FragArgs& a, const FragPlan& p, cudaStream_t s) {
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(gemv_frag_kernel<N, MODE, NB, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFSmem);
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.grid, 1, 1);
    cfg.blockDim = dim3(kFThreads, 1, 1);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemv_frag_kernel<N, MODE, NB, PAIR>, a);
}

template <int N, int MODE, bool PAIR = MODE == 0 && N <= 4>
cudaError_t launch_rows(int NB, const FragArgs& a, const FragPlan& p, cudaStream_t s) {
    return NB == 8 ? launch_one<N, MODE, 8, PAIR>(a, p, s) : launch_one<N, MODE, 16, PAIR>(a, p, s);
}

// Where this kernel is the faster one.  us per call on a B200, the kernel that otherwise takes the call -> this one, 0.3 %
// outliers:
//   * 5 rows and more: everywhere.  4096 x 4096 V2 N = 4, 8 rows 11.0 -> 6.5, 16 rows 21.4 -> 8.5; bf16 x 11.9 -> 7.3; V2a
//     15.7 -> 8.2.  28672 x 8192, 8 rows: V2 N = 4 74.9 -> 68.7, V2a 103 -> 75.  Only 9 rows and more of fp16 x on a matrix
//     that fills the chip with tiles of 128 channels stay on the tcgen05 kernel (16 rows, V2 N = 4: 77 against 107).
//   * A tile has eight rows, whether they are used or not.  3 or 4 rows: V2 N <= 4 up to 2^24 weights (4096 x 4096 N = 4
//     7.2 -> 6.4; 12288 x 4096 even, 28672 x 8192 53 -> 70) and N = 2 up to 2^26, V2 N >= 5 up to 2^23 (1536 x 4096 N = 5
//     7.2 -> 6.5; 4096 x 4096 7.5 -> 8.2), V2a up to 2^26 where x needs no K slices (12288 x 4096 26 -> 19; 4096 x 12288 N = 3
//     22 -> 23) or N = 6; with bf16 x also every V2a matrix (28672 x 8192 N = 4 91 -> 76) and those V2 ones that only the
//     general kernel takes (12288 x 4096 N = 6 56 -> 24)
//   * 2 rows: V2a up to 2^23 weights, with bf16 x up to 2^24 and every one of N = 6 (4096 x 4096 N = 4, bf16: 12.2 -> 9.0; fp16
//     7.7 -> 8.1)
//   * 1 row: up to 2^19 weights, where a call is launch and latency (256 x 1024 V2 N = 4 4.0 -> 3.1 us)
bool frag_preferred(const Layout& l, const GemvCall& c, const FragPlan& p) {
    const long long w = (long long)l.rows * l.cols;
    if (c.batch > 8) return c.x_bf16 || !batch_prefers_gemm(l, c.batch);
    if (c.batch > 4) return true;
    if (c.batch > 2) {
        if (c.x_bf16 && (l.mode || !batch_supported(l, c.batch))) return true;
        if (l.mode) return w <= 1 << 26 && (p.room == 1 || l.bits == 6);
        return w <= 1 << (l.bits == 2 ? 26 : l.bits <= 4 ? 24 : 23);
    }
    if (c.batch == 2) return l.mode && (w <= 1 << (c.x_bf16 ? 24 : 23) || (c.x_bf16 && l.bits == 6));
    return w <= 1 << 19;
}

}  // namespace

bool frag_supported(const Layout& l, const GemvCall& c) {
    if (c.n != 1 || c.packed_list || c.epilogue != 0 || l.GH != 1) return false;
    FragPlan p;
    return plan_frag(l, c.batch, sched_sms(), p) && frag_preferred(l, c, p);
}

cudaError_t launch_gemv_frag(const Layout& l, const GemvCall& c, cudaStream_t s) {
    FragPlan p;
    if (!plan_frag(l, c.batch, sched_sms(), p)) return cudaErrorInvalidValue;
    FragArgs a = {};
    a.b = blob_at(c.packed, offsets_of(l));
    a.x = c.x; a.y = c.y;
    a.tickets = (int*)c.workspace;
    a.partial = (float*)((char*)c.workspace + align256((size_t)l.RB * 4));
    a.rows = l.rows; a.cols = l.cols; a.RB = l.RB; a.SC = l.SC; a.ell_slots = l.ell_slots; a.L = l.L;
    a.nb = c.batch; a.y_kind = c.y_is_fp16; a.x_bf16 = c.x_bf16;
    a.S = p.S; a.sc_slice = p.sc_slice; a.x_off = (int)p.x_off; a.red_off = (int)p.red_off;
    const int NB = c.batch <= 8 ? 8 : 16;
    if (l.mode) {
        switch (l.bits) {
            case 2: return launch_rows<2, 1>(NB, a, p, s);
            case 3: return launch_rows<3, 1>(NB, a, p, s);
            case 4: return launch_rows<4, 1>(NB, a, p, s);
            case 5: return launch_rows<5, 1>(NB, a, p, s);
            default: return launch_rows<6, 1>(NB, a, p, s);
        }
    }
    switch (l.bits) {
        case 2: return launch_rows<2, 0>(NB, a, p, s);
        case 3: return launch_rows<3, 0>(NB, a, p, s);
        case 4: return p.pair ? launch_rows<4, 0>(NB, a, p, s) : launch_rows<4, 0, false>(NB, a, p, s);
        case 5: return launch_rows<5, 0>(NB, a, p, s);
        default: return launch_rows<6, 0>(NB, a, p, s);
    }
}

}  // namespace xfp
