// Prefill form of the fused decode kernel, Y = X (D + S)^T for many rows of x ("Fused Decode Kernel", steps (1)-(4): depack,
// codebook gather, outlier scatter-add into the dequantised tile, GEMM on the tensor cores), on pairs of SMs.
//
//   pair     two CTAs (tcgen05 cta_group::2) share a tile of 256 channels x T rows of x, T up to 512: each decodes its own
//            128 channels and stages half of the rows of x, the first CTA issues the products of both.  What bounds a GEMM
//            on this layout is the path from L2 (about 9 TB/s, 32 bytes per clock and SM): decoded in place the weights cost
//            N / 16 of an fp16 operand there, and sharing x in a pair halves the rest.  (Decoding into global tiles first
//            and multiplying from there ran at those 9 TB/s: 4096 x 4096, 100 rows 26 us, 28672 x 8192, 1024 rows 640 us.)
//   stage    64 k: A = W^ [128 channels][64 k] fp16 in core-matrix order (k / 8, channel, 8), 16 KB; B = the CTA's half of
//            the rows of x in the 128-byte swizzle, by tensor copies.  4 .. 12 stages in a ring: a stage is in decode for
//            about 1900 clocks (four of them at once), then 300 for its outliers, then in the products.
//   warps    1 products, 2 copies, 4 outliers, 16 decode.  A stage is decoded by four warps, one per row-block: 64 look-ups per
//            lane, stored as eight 16-byte vectors.  Outliers: a lane per channel with the next entries of its list in
//            registers adds those that fall into two stages to the stored values, one correctly rounded fp16 addition each, by
//            address.  (In the decode warps, in registers, where the register has to be found by nested tests, the same
//            addition cost as much as the decode; in the decode warps by address it lengthened a stage's decode from 1900 to
//            3000 clocks, the SM's issue slots being full.)  Roles meet at mbarriers only: a stage is "ready" on the first
//            CTA's barrier when all row-blocks of both CTAs are stored and the x of both has landed (the copies of both count
//            their bytes there).
//   schedule resident pairs.  Whole rounds of tiles run whole tiles; what remains is one stream of super-chunks that is dealt
//            evenly over the pairs, so a pair ends one tile and begins the next (28672 x 8192, 1024 rows: 4.5 rounds instead of
//            5; 10007 x 4992, 301 rows: 40 tiles on 74 pairs).  A CTA that had part of a tile leaves fp32 sums in the
//            workspace; the last to come of a tile adds the parts in order of K.  Nobody waits for another pair.
//            Where clusters of 2 or 3 pairs on one tile each fit the GPU at once (few tiles), they cut K instead and the sums
//            meet through distributed shared memory: writing and reading them through L2 takes 9 us at 4096 x 4096, 100 rows
//            in four parts, the exchange in a cluster of three pairs 3 us.
//   look-ups up to N = 4: the codebook in registers, PRMT look-ups (xfp_reg_decode.cuh); a stage's operands,
//            their copies and 64 look-ups per lane share the data pipe of shared memory, and the PRMTs stay off it (look-ups in
//            tables -> registers: 10007 x 4992 V2a, 301 rows 57.5 -> 49.1 us; 28672 x 8192 V2a, 512 rows 282 -> 268, V2, 1024 rows
//            421 -> 406; 4096 x 4096 V2, 100 rows 21.3 -> 20.9).  V2 at N <= 3
//            in a cluster: pair tables; above N = 4 one entry per index.
//   V2a      a lane decodes the 2^N entries its channel's group can take once per 64 weights (D16 = fp16(fp32(scale * lib + mid)));
//            the look-ups are then those of V2.
// Waits on barriers have an iteration limit; when one runs out the CTA records it in the first word of the workspace and stops
// issuing; its cluster then stores no sums that lack a part, waits for what is in flight and leaves through the exit that frees
// its tensor memory.
#include <cuda.h>

#include "xfp_internal.h"
#include "xfp_pair_common.cuh"
#include "xfp_reg_decode.cuh"

namespace xfp {

namespace {

constexpr int kCh = 128;                       // channels of a CTA
constexpr int kStageK = 64;
constexpr int kABytes = kCh * kStageK * 2;     // A of one stage
constexpr int kMaxSlots = 12;
// A decode warp takes every fourth stage.  At stage j it waits, by parity, for the products of stage j - slots; that is only
// unambiguous once stage j - 2 slots is known to be done, and what the warp knows from its own stage j - 4 is that stage
// j - 4 - slots is.  With three stages in the ring a warp ahead of the others could pass early and arrive in another stage's
// phase (which faulted: V2a, N = 2, 7959 x 1920, 1991 rows, no outliers).
constexpr int kMinSlots = 4;
// Warp roles, the short ones first: the scheduler serves older warps first, and behind the decode warps, which can issue in
// every clock, the others' few instructions waited.
constexpr int kMmaWarp = 0, kCopyWarp = 1, kCopyWarps = 2, kOutWarp = 4, kOutWarps = 4, kDecodeWarp = 8, kDecodeWarps = 16;
constexpr int kThreads = (kDecodeWarp + kDecodeWarps) * 32;
constexpr uint32_t kSpins = 1u << 20, kPollHint = 1000;
constexpr size_t kSmemMax = 226 * 1024;
constexpr int kMaxCut = 4;                     // pairs of a cluster
constexpr int kClusters[kMaxCut + 1] = {0, 74, 33, 22, 15};   // clusters of k pairs that a B200 runs at once (cudaOccupancyMaxActiveClusters:
                                                              // a cluster stays inside a GPC); more of them run in turn
constexpr int kPairs = kSizingSMs / 2;         // pairs that the schedule deals to; a device with fewer runs them in turn

struct FusedArgs {
    Blob b;
    void* y;
    int* ctrl;                  // [0] error word, [1 + 2 * tile + half] arrivals of the parts of a dealt tile (see prefill_ctrl_bytes)
    float* part;                // [2 * pair + which][half][T][128] sums of a part
    int rows, RB, SC, M, ell_slots, GH, L, y_kind;
    int tok_tiles;              // tiles along x; a tile has 256 channels and T rows of x
    int T, Tp, parts;           // one product instruction covers Tp <= 256 rows, the second T - Tp; both multiples of 32
    int slots, x_bytes;         // stages in the ring; bytes of x per stage and CTA
    int tab_bytes;
    int ks, sc_slice;           // ks > 1: pairs of a cluster and the super-chunks of each; the schedule below is not used
    int whole;                  // whole tiles per pair; the rest (`stream` super-chunks from tile whole * kPairs on) is dealt
    int stream, dealt;          // evenly to pairs 0 .. dealt - 1
    int tmem_cols;
    int converted;              // the kernel in front is the library's conversion of bf16 rows
    int short_cta;              // tests: the CTA whose waits give up at once (-1: none)
};

__device__ __forceinline__ uint32_t sa(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool test_bar(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// By a whole warp, which leaves it together (a lane that gave up alone would keep the others from the warp's next instruction).
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, uint32_t spins) {
    for (uint32_t i = 0; i < spins; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity), "r"(kPollHint) : "memory");
        if (__all_sync(0xffffffffu, ok)) return true;
    }
    return false;
}
// One lane of a converged warp.  Instructions that take uniform registers are then issued by one thread as the compiler
// sees it; behind a plain lane == 0 it serialises over the lanes it cannot rule out (a copy or a product took 70 - 250 clocks).
__device__ __forceinline__ bool elected() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// the same address in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void arrive_local(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory"); }
__device__ __forceinline__ void arrive_cluster(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(bar) : "memory"); }
__device__ __forceinline__ void init_bar(const uint64_t* bar, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(sa(bar)), "r"(n)); }
__device__ __forceinline__ uint32_t lds32(uint32_t a) { uint32_t v; asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a)); return v; }
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" :: "r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// K-major operand descriptors (version 1).  A: core matrices of 8 rows x 16 bytes, the next 8 k 2048 bytes on, the next 8
// rows 128 bytes on, no swizzle.  B: rows of 128 bytes in the 128-byte swizzle, 8 rows 1024 bytes.
__device__ __forceinline__ uint64_t desc_a(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)(2048 >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}
__device__ __forceinline__ uint64_t desc_b(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void mma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        :: "r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
// the products issued so far arrive on the barrier of both CTAs of the pair
__device__ __forceinline__ void commit_pair(uint32_t bar, uint32_t mask) {
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
// the other half of the kernel's first arrival at the cluster barrier: the other CTA's barriers exist
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void decode_sync() { asm volatile("bar.sync 1, %0;" :: "n"(kDecodeWarps * 32) : "memory"); }

// Position in the ring after a number of stages: slot and the parity of its current use.
struct Ring {
    int slot;
    uint32_t phase;
    __device__ __forceinline__ void step(int n, int slots) {
        slot += n;
        while (slot >= slots) { slot -= slots; phase ^= 1u; }
    }
    __device__ __forceinline__ void jump(int n, int slots) {
        const int q = (slot + n) / slots;
        slot += n - q * slots;
        phase ^= (uint32_t)q & 1u;
    }
};

// The i-th piece of work of pair g: super-chunks [sc0, sc1) of a tile.  Pair g has [g S / D, (g + 1) S / D) of the S dealt
// super-chunks, at most a tile's worth, so at most two pieces.
struct Piece { int tile, sc0, sc1; };
template <bool SPLIT>
__host__ __device__ __forceinline__ bool piece_of(const FusedArgs& a, int g, int i, Piece& p) {
    if (SPLIT) {
        const int s = g % a.ks;
        p.tile = g / a.ks; p.sc0 = s * a.sc_slice; p.sc1 = a.SC < p.sc0 + a.sc_slice ? a.SC : p.sc0 + a.sc_slice;
        return i == 0;
    }
    if (i < a.whole) { p.tile = g + i * kPairs; p.sc0 = 0; p.sc1 = a.SC; return true; }
    i -= a.whole;
    if (g >= a.dealt || i > 1) return false;
    const int u0 = g * a.stream / a.dealt, u1 = (g + 1) * a.stream / a.dealt;      // below 74 * 74 * 512
    const int t = u0 / a.SC + i, b = t * a.SC;
    if (u1 <= b) return false;
    p.tile = a.whole * kPairs + t; p.sc0 = u0 > b ? u0 - b : 0; p.sc1 = a.SC < u1 - b ? a.SC : u1 - b;
    return true;
}
// rows of x of the p-th product of a stage, which begins at row p0: those that exist, rounded up to 32
__device__ __forceinline__ int product_rows(const FusedArgs& a, int p0, int p) {
    return min(p ? a.T - a.Tp : a.Tp, max((a.M - p0 + 31) & ~31, 32));
}
// the pair that has dealt super-chunk u: the largest g with g S / D <= u
__device__ __forceinline__ int dealt_to(const FusedArgs& a, int u) { return ((u + 1) * a.dealt - 1) / a.stream; }

// Decode tables, where codebooks do not sit in registers (kReg).  kPair (V2, N <= 3): entry t = first index | second index << N holds
// two fp16 values; else entry q one.  V2: a table per row-block.  V2a: a table per warp.
template <int N, int MODE>
struct Tab {
    static constexpr int E = 1 << N;
    static constexpr bool kPair = MODE == 0 && N <= 3;
    static constexpr int kEntries = kPair ? E * E : E;
    static constexpr int kOne = kEntries * 128;      // of one table
    // address of table u's entry 0 for this lane
    __device__ static __forceinline__ uint32_t at(uint32_t base, int u, int lane) { return base + (uint32_t)u * kOne + (uint32_t)lane * 4u; }
};

// W^ = fp16(D16 + S) in place
__device__ __forceinline__ void add_outlier(uint32_t addr, uint16_t val) {
    uint16_t w;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(w) : "r"(addr));
    w = __half_as_ushort(__hadd(__ushort_as_half(w), __ushort_as_half(val)));
    asm volatile("st.shared.u16 [%0], %1;" :: "r"(addr), "h"(w) : "memory");
}

// The 16-byte vectors that hold words [PART * 2N, PART * 2N + 2N) of a lane's 128 * N-bit stream.
template <int N, int PART>
struct Half {
    static constexpr int V0 = PART * 2 * N / 4, V1 = (PART * 2 * N + 2 * N + 3) / 4, NV = V1 - V0;
};

// V2: the codebooks of the CTA's four row-blocks into their tables (all decode warps).
template <int N>
__device__ __forceinline__ void fill_tables(const FusedArgs& a, uint32_t tab0, int rb0, int warp, int lane) {
    using T = Tab<N, 0>;
    constexpr int E = T::E;
    const int q = warp & 3, sub = warp >> 2, rb = rb0 + q;
    if (rb >= a.RB) return;
    const uint16_t* cb = a.b.cb + (size_t)(rb * kRowsPerBlock + lane) * E;      // padding rows exist in the blob
    const uint32_t t = T::at(tab0, q, lane);
    if (T::kPair) {
        uint32_t v[E];
#pragma unroll
        for (int e = 0; e < E; e += 4) {
            const uint2 p = __ldg((const uint2*)(cb + e));
            v[e] = p.x & 0xffffu; v[e + 1] = p.x >> 16; v[e + 2] = p.y & 0xffffu; v[e + 3] = p.y >> 16;
        }
#pragma unroll
        for (int hi = 0; hi < E; ++hi)
            if ((hi & 3) == sub) {
#pragma unroll
                for (int lo = 0; lo < E; ++lo) sts32(t + (uint32_t)((lo | (hi << N)) * 128), __byte_perm(v[lo], v[hi], 0x5410));
            }
    } else {
#pragma unroll
        for (int e = 0; e < E / 4; e += 4) {
            const int e0 = sub * (E / 4) + e;
            const uint2 p = __ldg((const uint2*)(cb + e0));
            sts32(t + (uint32_t)(e0 * 128), p.x & 0xffffu); sts32(t + (uint32_t)((e0 + 1) * 128), p.x >> 16);
            sts32(t + (uint32_t)((e0 + 2) * 128), p.y & 0xffffu); sts32(t + (uint32_t)((e0 + 3) * 128), p.y >> 16);
        }
    }
}

// A channel's outliers in ascending column order: transposed slab first, the CSR arrays behind it.
struct Outliers {
    const uint32_t* slab;
    const uint32_t* spill;
    int nslab, total;
    __device__ __forceinline__ const uint32_t* addr(int j) const { return j < nslab ? slab + (size_t)(1 + j) * 32 : spill + j; }
    __device__ __forceinline__ uint32_t at(int j) const { return __ldg(addr(j)); }
    __device__ __forceinline__ void open(const FusedArgs& a, int rb, int row, int lane) {
        slab = a.b.ell + (size_t)rb * (a.ell_slots + 1) * 32 + lane;
        spill = a.b.oent;
        nslab = total = 0;
        if (rb < a.RB && row < a.rows) {
            const int len = (int)__ldg(slab);
            nslab = total = min(len, a.ell_slots);
            if (len >= a.ell_slots) {
                const int p0 = __ldg(a.b.rowptr + row);
                total = __ldg(a.b.rowptr + row + 1) - p0;
                spill = a.b.oent + p0;
            }
        }
    }
    // first entry at or behind column k0: sixteen independent loads at a time (every 16th entry, then the 15 in front of the hit)
    __device__ __forceinline__ int find(uint32_t k0) const {
        if (!k0 || !total) return 0;
        int coarse = 0, fine = 0;
        for (int j = 15; j < total; j += 16) coarse += (at(j) & 0xffffu) < k0;
#pragma unroll
        for (int j = 0; j < 15; ++j) fine += coarse * 16 + j < total && (at(min(coarse * 16 + j, total - 1)) & 0xffffu) < k0;
        return coarse * 16 + fine;
    }
};

struct Bars {
    uint32_t decoded, freed;      // address of slot 0's; slot s is 8 s further
    uint32_t ready;               // of the first CTA of the pair
    uint32_t spins;               // polls of a wait
};

// The decode warps' share of one tile: half PART of super-chunks grp, grp + 2, ... of [sc0, sc1): every fourth stage.
// REG: from a codebook in registers.
template <int N, int MODE, int PART, bool REG>
__device__ __forceinline__ bool decode_tile(const FusedArgs& a, int rb, bool rb_ok, int q, int grp, int lane, int sc0, int sc1,
                                            uint32_t tab, RegBook<REG ? N : 2>& book, const uint16_t* slib, uint32_t sA,
                                            const Bars& bars, Ring ring, bool& met) {
    using T = Tab<N, MODE>;
    using H = Half<N, PART>;
    constexpr int E = T::E;
    const uint4* idx = a.b.idx + ((size_t)rb * a.SC + sc0 + grp) * N * 32 + lane;
    const size_t meta0 = (((size_t)rb * a.SC + sc0 + grp) * a.GH + (a.GH - 1) * PART) * 32 + lane;
    uint4 nx[H::NV];
    uint32_t id_n = 0, sm_n = 0;
    auto fetch = [&](int it) {                    // the vectors of this warp's super-chunk `it` steps of two ahead
#pragma unroll
        for (int v = 0; v < H::NV; ++v) nx[v] = ld_stream(idx + (size_t)it * 2 * N * 32 + (size_t)(H::V0 + v) * 32);
        if (MODE == 1) {
            const size_t m = meta0 + (size_t)it * 2 * a.GH * 32;
            id_n = __ldg(a.b.gid + m); sm_n = __ldg(a.b.gsm + m);
        }
    };
    if (rb_ok && sc0 + grp < sc1) fetch(0);
    ring.step(2 * grp + PART, a.slots);
    int it = 0;
    for (int sc = sc0 + grp; sc < sc1; sc += 2, ++it) {
        uint32_t w[4 * N + 1];
        if (rb_ok) {
#pragma unroll
            for (int i = 0; i <= 4 * N; ++i) w[i] = 0u;
#pragma unroll
            for (int v = 0; v < H::NV; ++v) {
                w[4 * (H::V0 + v)] = nx[v].x; w[4 * (H::V0 + v) + 1] = nx[v].y;
                w[4 * (H::V0 + v) + 2] = nx[v].z; w[4 * (H::V0 + v) + 3] = nx[v].w;
            }
            const uint32_t id = id_n, sm = sm_n;
            if (sc + 2 < sc1) fetch(it + 1);
            if (MODE == 1) {
                if constexpr (REG) {
                    uint32_t d[E / 2];
                    load_entries<N>(d, slib + id * (E + 8), [](auto* p) { return *p; });
                    affine_entries<N>(d, sm);
                    book = book_of<N>(d);
                } else {
                    const float scale = h2f((uint16_t)(sm & 0xffffu)), mid = h2f((uint16_t)(sm >> 16));
                    auto decoded = [&](uint32_t l) { return (uint32_t)f2h(__fmaf_rn(scale, h2f((uint16_t)l), mid)); };
#pragma unroll
                    for (int e = 0; e < E; e += 8) {
                        const uint4 l8 = *(const uint4*)(slib + id * (E + 8) + e);
                        const uint32_t lw[4] = {l8.x, l8.y, l8.z, l8.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            sts32(tab + (e + 2 * i) * 128, decoded(lw[i] & 0xffffu));
                            sts32(tab + (e + 2 * i + 1) * 128, decoded(lw[i] >> 16));
                        }
                    }
                }
            }
        }
        // the slot's previous use: its products are done
        if (!wait_bar(bars.freed + 8u * ring.slot, ring.phase ^ 1u, bars.spins)) return false;
        if (rb_ok) {
            const uint32_t dst = sA + (uint32_t)ring.slot * kABytes + (uint32_t)(q * 32 + lane) * 16u;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                uint4 v;
                if constexpr (REG) {
                    v = reg_decode8_ordered<N>(w, PART * 8 + c, book);
                } else {
                    uint32_t d[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int p = PART * 32 + c * 4 + i;
                        if (T::kPair) d[i] = lds32(pair_addr<N, 1>(w, p, tab));
                        else d[i] = join16(lds32(single_addr<N, 1>(w, 2 * p, tab)), lds32(single_addr<N, 1>(w, 2 * p + 1, tab)));
                    }
                    v = make_uint4(d[0], d[1], d[2], d[3]);
                }
                sts128(dst + (uint32_t)c * 2048u, v.x, v.y, v.z, v.w);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the products read through the async proxy
        __syncwarp();
        if (!a.ell_slots && !met) { cluster_wait(); met = true; }             // the first arrival at the other CTA
        if (elected()) {
            if (a.ell_slots) arrive_local(bars.decoded + 8u * ring.slot);      // the outlier warps come next
            else arrive_cluster(bars.ready + 8u * ring.slot);
        }
        ring.step(4, a.slots);
    }
    return true;
}

// The outlier warps' share of one tile (matrices with outliers): warp q adds those of row-block q, two stages at a time.
__device__ __forceinline__ bool outlier_tile(const FusedArgs& a, int rb, int q, int lane, int sc0, int sc1, uint32_t sA,
                                             const Bars& bars, Ring ring) {
    constexpr int kAhead = 6;
    Outliers o;
    o.open(a, rb, rb * kRowsPerBlock + lane, lane);
    int cur = o.find((uint32_t)sc0 * kSuper);
    const bool spills = __any_sync(0xffffffffu, o.total > o.nslab);
    const uint32_t mine = sA + (uint32_t)(q * 32 + lane) * 16u;
    uint32_t e[kAhead];
    auto look = [&]() {                     // behind the list's end: an entry that adds +0 to the last weight a row can have
        if (!spills) {
            const uint32_t* p = o.slab + (size_t)(1 + cur) * 32;
#pragma unroll
            for (int i = 0; i < kAhead; ++i) e[i] = cur + i < o.total ? __ldg(p + i * 32) : 0xffffu;
        } else {
#pragma unroll
            for (int i = 0; i < kAhead; ++i) e[i] = cur + i < o.total ? o.at(cur + i) : 0xffffu;
        }
    };
    look();
    for (int sc = sc0; sc < sc1; ++sc) {
        Ring on = ring;
        on.step(1, a.slots);
        const uint32_t k0 = (uint32_t)sc * kSuper, first = mine + (uint32_t)ring.slot * kABytes, second = mine + (uint32_t)on.slot * kABytes;
        if (!wait_bar(bars.decoded + 8u * ring.slot, ring.phase, bars.spins) || !wait_bar(bars.decoded + 8u * on.slot, on.phase, bars.spins)) return false;
        for (;;) {
            int n = 0;
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                const uint32_t k = (e[i] & 0xffffu) - k0;           // ascending: never below
                if (k < (uint32_t)kSuper) {
                    ++n;
                    add_outlier((k < (uint32_t)kStageK ? first : second) + ((k >> 3) & 7u) * 2048u + (k & 7u) * 2u, (uint16_t)(e[i] >> 16));
                }
            }
            cur += n;
            const bool more = __any_sync(0xffffffffu, n == kAhead && cur < o.total);
            if (!more) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (elected()) {
                    arrive_cluster(bars.ready + 8u * ring.slot);
                    arrive_cluster(bars.ready + 8u * on.slot);
                }
            }
            if (n) look();                  // they travel while the next stages are decoded
            if (!more) break;
        }
        ring = on;
        ring.step(1, a.slots);
    }
    return true;
}

// 16 sums of one channel, rows of x t0 .. t0 + n - 1
__device__ __forceinline__ void store_rows(const FusedArgs& a, int t0, int n, int row, const uint32_t (&v)[16]) {
    const size_t o = (size_t)t0 * a.rows + row;
    if (a.y_kind == 1) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < n) ((uint16_t*)a.y)[o + (size_t)j * a.rows] = f2h(__uint_as_float(v[j]));
    } else if (a.y_kind == 2) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < n) ((uint16_t*)a.y)[o + (size_t)j * a.rows] = __bfloat16_as_ushort(__float2bfloat16_rn(__uint_as_float(v[j])));
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < n) ((float*)a.y)[o + (size_t)j * a.rows] = __uint_as_float(v[j]);
    }
}

// sums of four consecutive channels (from `row` on) of row t of x
__device__ __forceinline__ void store_quad(const FusedArgs& a, int t, int row, const float4& v) {
    const size_t o = (size_t)t * a.rows + row;
    if ((a.rows & 3) == 0 && row < a.rows) {
        if (a.y_kind == 0) *(float4*)((float*)a.y + o) = v;
        else if (a.y_kind == 1) {
            const __half2 lo = __floats2half2_rn(v.x, v.y), hi = __floats2half2_rn(v.z, v.w);
            *(uint2*)((uint16_t*)a.y + o) = make_uint2(*(const uint32_t*)&lo, *(const uint32_t*)&hi);
        } else {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
            *(uint2*)((uint16_t*)a.y + o) = make_uint2(*(const uint32_t*)&lo, *(const uint32_t*)&hi);
        }
        return;
    }
    if (row < a.rows) put_y(a.y, o, v.x, a.y_kind);
    if (row + 1 < a.rows) put_y(a.y, o + 1, v.y, a.y_kind);
    if (row + 2 < a.rows) put_y(a.y, o + 2, v.z, a.y_kind);
    if (row + 3 < a.rows) put_y(a.y, o + 3, v.w, a.y_kind);
}

// After a wait has run out and every warp of the pair has stopped: returns when the copies into ring slot `slot` of both CTAs have
// landed.  They count their bytes on the first CTA's "ready" barrier (`bar`), whose phase ends when its arrivals are complete and no
// bytes are outstanding: what one CTA copied and the other did not any more is balanced, the missing arrivals are made up.
__device__ __noinline__ void drain_copies(int slot, int slots, int x_bytes, const int* copied, uint32_t bar, uint32_t crank) {
    int last[2];                 // the last stage that each CTA copied into the slot: warp w took the stages of parity w below `end`
    for (int c = 0; c < 2; ++c) {
        int end[kCopyWarps], top = 0;
        for (int w = 0; w < kCopyWarps; ++w) {
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(end[w]) : "r"(peer(sa(copied + w), crank + c)));
            top = max(top, end[w]);
        }
        int j = top - 1 - (top - 1 - slot + slots) % slots;     // the largest below `top` that falls into the slot
        while (j >= 0 && j >= end[j & 1]) j -= slots;
        last[c] = max(j, -1);
    }
    if (last[0] < 0 && last[1] < 0) return;
    if (last[0] > last[1]) asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(x_bytes) : "memory");
    if (last[1] > last[0]) asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(x_bytes) : "memory");
    uint64_t state;
    uint32_t pending, ok = 0;
    do {
        asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(state) : "r"(bar) : "memory");
        asm volatile("mbarrier.pending_count.b64 %0, %1;" : "=r"(pending) : "l"(state));
    } while (pending > 1);
    for (uint32_t i = 0; i < kSpins && !ok; ++i)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "l"(state) : "memory");
}

// SPLIT: a cluster of a.ks pairs on one tile, cut along K.
template <int N, int MODE, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1) gemm_fused_kernel(const FusedArgs a, const __grid_constant__ CUtensorMap tmap) {
    using T = Tab<N, MODE>;
    // Codebooks in registers: V2a up to N = 4 and V2 at N = 4, which would take a look-up per weight; V2 at N = 2, 3 instead of pair
    // tables where a pair walks its tiles (10007 x 4992 N = 3, 301 rows 42.5 -> 40.3 us, 28672 x 8192, 512 rows 237 -> 233; 192 rows
    // at N = 2 29.3 -> 30.0 at 12288 x 4096), not where a cluster cuts one tile (4096 x 4096, 100 rows 21.3 against 21.5)
    constexpr bool kReg = MODE == 0 ? N == 4 || (N <= 3 && !SPLIT) : N <= 4;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // tables aligned to 8 KB of the shared window, so that an entry's offset is merged with the address, not added
    unsigned char* smem = smem_raw + ((8192u - (sa(smem_raw) & 8191u)) & 8191u);      // the same offset in every CTA
    __shared__ __align__(8) uint64_t b_decoded[kMaxSlots], b_ready[kMaxSlots], b_freed[kMaxSlots], acc_full, acc_empty, b_drain;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail, s_last, s_copied[kCopyWarps];
    __shared__ const float* s_part[kPairs];
    // the warp index through a shuffle: uniform as the compiler sees it, so that the roles run on uniform registers
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t crank = cluster_rank(), h = crank & 1u, lead = crank & ~1u;        // half of the pair; CTA 0 of it issues the products
    const int g = (int)blockIdx.x >> 1;
    unsigned char* pA = smem + a.tab_bytes;
    unsigned char* pB = pA + (size_t)a.slots * kABytes;
    uint16_t* lib = (uint16_t*)(pB + (size_t)a.slots * a.x_bytes);
    const Bars bars{sa(b_decoded), sa(b_freed), peer(sa(b_ready), lead), (int)blockIdx.x == a.short_cta ? 0u : kSpins};
    asm volatile("griddepcontrol.launch_dependents;");

    if (tid < a.slots) {
        init_bar(&b_decoded[tid], 4);                         // a warp per row-block
        init_bar(&b_ready[tid], 2 * 4 + 1);                   // four row-blocks of both CTAs, and the bytes of x
        init_bar(&b_freed[tid], 1);
    }
    if (tid == 32) {
        init_bar(&acc_full, 1);
        init_bar(&acc_empty, 2 * kDecodeWarps);
        init_bar(&b_drain, 1);
        s_fail = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // The blob may come from the kernel in front of the call, and that one may have released its dependents early: nothing of it
    // is read, and no bounded wait begins, before it is complete.  Behind the conversion of bf16 rows this kernel starts only when
    // the conversion has found everything in front of it complete; the decode then overlaps the conversion.  (Starting beside the
    // previous call's tail, as before, read weights that an early-releasing producer had not written yet; behind itself a call of
    // 4096 x 4096, 100 rows bf16 was 1.4 us faster for it, 19.8 us.)
    if (!a.converted) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (MODE == 1)               // at most 1024 entries (gemm_tc_supported)
        for (int i = tid; i < a.L * T::E; i += kThreads) lib[(i / T::E) * (T::E + 8) + i % T::E] = __ldg(a.b.cb + i);
    __syncthreads();
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(sa(&s_tmem)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    // Nothing remote happens before the wait that belongs to this arrival: the decode warps begin at once and wait in front of
    // their first arrival at the other CTA, the others before they start.
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

    bool ok = true;
    Ring ring{0, 0u};
    uint32_t acc_ph = 0;
    Piece pc;
    if (warp >= kDecodeWarp) {
        const int dw = warp - kDecodeWarp, q = dw & 3, part = (dw >> 2) & 1, grp = dw >> 3;
        const uint32_t tab = T::at(sa(smem), MODE == 0 ? q : dw, lane);
        bool met = false;                                     // has waited for the other CTA's barriers
        int have = -1;                                        // tile of channels whose codebooks are in place
        RegBook<kReg ? N : 2> book;
        for (int i = 0; piece_of<SPLIT>(a, g, i, pc); ++i) {         // a warp whose wait ran out still meets the others at their barrier
            const int tx = pc.tile / a.tok_tiles, ty = pc.tile % a.tok_tiles, t0 = ty * a.T;
            const int rb = (2 * tx + (int)h) * 4 + q;
            if (MODE == 0 && tx != have) {
                if constexpr (kReg) {
                    if (rb < a.RB) book = make_book<N>(a.b.cb + (size_t)(rb * kRowsPerBlock + lane) * T::E);
                } else {
                    decode_sync();                            // every warp is done with the previous tables
                    fill_tables<N>(a, sa(smem), rb - q, dw, lane);
                    decode_sync();
                }
                have = tx;
            }
            ok = ok && (part == 0 ? decode_tile<N, MODE, 0, kReg>(a, rb, rb < a.RB, q, grp, lane, pc.sc0, pc.sc1, tab, book, lib, sa(pA), bars, ring, met)
                                  : decode_tile<N, MODE, 1, kReg>(a, rb, rb < a.RB, q, grp, lane, pc.sc0, pc.sc1, tab, book, lib, sa(pA), bars, ring, met));
            ring.jump(2 * (pc.sc1 - pc.sc0), a.slots);
            ok = ok && wait_bar(sa(&acc_full), acc_ph, bars.spins);
            acc_ph ^= 1u;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc = s_tmem + ((uint32_t)(q * 32) << 16);
            const int r = q * 32 + lane, row = (2 * tx + (int)h) * kCh + r;
            const int tend = min(a.T, a.M - t0);
            const bool whole = !SPLIT && pc.sc0 == 0 && pc.sc1 == a.SC;
            // a CTA that has part of a tile: its sums as [t][channel] -- into its idle stages, every product being complete, or
            // into the workspace
            float* sums = (float*)pA + r;
            int g0 = 0, g1 = 0;
            const size_t psize = (size_t)a.T * kCh;
            // part of pair z: its second piece unless its first begins in this tile
            auto part_at = [&](int z) {
                const int first = z * a.stream / a.dealt / a.SC;
                return a.part + ((size_t)(2 * z + (first == pc.tile - a.whole * kPairs ? 0 : 1)) * 2 + h) * psize;
            };
            if (!SPLIT && !whole) {
                const int u0 = (pc.tile - a.whole * kPairs) * a.SC;
                g0 = dealt_to(a, u0); g1 = dealt_to(a, u0 + a.SC - 1);
                sums = part_at(g) + r;
            }
            if (ok)
                for (int c = dw >> 2; c * 16 < tend; c += kDecodeWarps / 4) {
                    uint32_t v[16];
                    tmem_ld16(acc + (uint32_t)(c * 16), v);             // the whole warp
                    if (whole) {
                        if (row < a.rows) store_rows(a, t0 + c * 16, min(16, tend - c * 16), row, v);
                    } else {
                        float* p = sums + (size_t)c * 16 * kCh;
#pragma unroll
                        for (int j = 0; j < 16; ++j) p[(size_t)j * kCh] = __uint_as_float(v[j]);
                    }
                }
            if (!SPLIT && !whole) {
                __threadfence();
                if (!ok) s_fail = 1;                          // a part that is not there is not counted: nobody adds up this tile
                if (dw < 4 && dw * 32 + lane <= g1 - g0) s_part[dw * 32 + lane] = part_at(g0 + dw * 32 + lane);
                decode_sync();
                if (dw == 0 && lane == 0) {
                    int* count = a.ctrl + 1 + 2 * (pc.tile - a.whole * kPairs) + h;
                    const int last = !s_fail && atomicAdd(count, 1) == g1 - g0;
                    if (last) *count = 0;
                    s_last = last;
                    __threadfence();
                }
                decode_sync();
                if (s_last) {
                    // four channels of a row of x per thread and step, four rows and two parts in flight
                    constexpr int kRowsIn = 4;
                    const int ch = lane * 4, orow = (2 * tx + (int)h) * kCh + ch;
                    for (int t = dw; t < tend; t += kDecodeWarps * kRowsIn) {
                        float4 sum[kRowsIn];
#pragma unroll
                        for (int u = 0; u < kRowsIn; ++u) sum[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
                        for (int z = 0; z <= g1 - g0; ++z) {
                            const float* p = s_part[z] + (size_t)t * kCh + ch;
                            float4 v[kRowsIn];
#pragma unroll
                            for (int u = 0; u < kRowsIn; ++u)      // rows behind the last one exist in the part as well
                                v[u] = __ldcg((const float4*)(p + (size_t)(t + u * kDecodeWarps < tend ? u * kDecodeWarps : 0) * kCh));
#pragma unroll
                            for (int u = 0; u < kRowsIn; ++u) { sum[u].x += v[u].x; sum[u].y += v[u].y; sum[u].z += v[u].z; sum[u].w += v[u].w; }
                        }
#pragma unroll
                        for (int u = 0; u < kRowsIn; ++u)
                            if (t + u * kDecodeWarps < tend) store_quad(a, t0 + t + u * kDecodeWarps, orow, sum[u]);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            if (!met) { cluster_wait(); met = true; }
            __syncwarp();
            if (elected()) arrive_cluster(peer(sa(&acc_empty), lead));
        }
    } else if (warp >= kOutWarp) {
        const int q = warp - kOutWarp;
        cluster_wait();
        if (a.ell_slots)
            for (int i = 0; ok && piece_of<SPLIT>(a, g, i, pc); ++i) {
                ok = outlier_tile(a, (2 * (pc.tile / a.tok_tiles) + (int)h) * 4 + q, q, lane, pc.sc0, pc.sc1, sa(pA), bars, ring);
                ring.jump(2 * (pc.sc1 - pc.sc0), a.slots);
            }
    } else if (warp >= kCopyWarp && warp < kCopyWarp + kCopyWarps) {
        cluster_wait();
        asm volatile("griddepcontrol.wait;" ::: "memory");    // x may come from the previous kernel of the stream
        int n = warp - kCopyWarp, done = 0;                   // the two warps take the stages in turn; those copied so far end at `done`
        for (int i = 0; ok && piece_of<SPLIT>(a, g, i, pc); ++i) {
            const int t0 = (pc.tile % a.tok_tiles) * a.T;
            for (int st = 2 * pc.sc0; st < 2 * pc.sc1; ++st, ring.step(1, a.slots)) {
                if (n++ & 1) continue;
                if (!(ok = wait_bar(bars.freed + 8u * ring.slot, ring.phase ^ 1u, bars.spins))) break;
                if (elected()) {
                    const uint32_t bar = bars.ready + 8u * ring.slot;
                    uint32_t dst = sa(pB) + (uint32_t)(ring.slot * a.x_bytes);
                    if (h == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(sa(b_ready) + 8u * ring.slot), "r"((uint32_t)(2 * a.x_bytes)) : "memory");
                    for (int p = 0; p < a.parts; ++p, dst += (uint32_t)a.Tp * 64u) {
                        // this CTA's half of the rows that the product takes (more may be copied along)
                        const int p0 = t0 + p * a.Tp, xrow = p0 + (int)h * (product_rows(a, p0, p) >> 1);
                        asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                     :: "r"(dst), "l"(&tmap), "r"(st * kStageK), "r"(xrow), "r"(bar) : "memory");
                    }
                }
                __syncwarp();
                done = n - (warp - kCopyWarp);
            }
        }
        if (lane == 0) s_copied[warp - kCopyWarp] = done;
    } else if (h == 1 || warp != kMmaWarp) {
        cluster_wait();                                       // the first CTA issues the pair's products
    } else {
        const uint64_t da0 = desc_a(sa(pA)), db0 = desc_b(sa(pB));
        const uint32_t mask = 3u << lead;
        cluster_wait();
        const uint32_t tmem = s_tmem;
        for (int i = 0; ok && piece_of<SPLIT>(a, g, i, pc); ++i) {
            const int t0 = (pc.tile % a.tok_tiles) * a.T, st1 = 2 * pc.sc1;
            const uint32_t id = (1u << 4) | ((uint32_t)(2 * kCh >> 4) << 24);
            const uint32_t id0 = id | ((uint32_t)(product_rows(a, t0, 0) >> 3) << 17);
            const uint32_t id1 = a.parts > 1 && t0 + a.Tp < a.M ? id | ((uint32_t)(product_rows(a, t0 + a.Tp, 1) >> 3) << 17) : 0u;
            if (i) {
                ok = wait_bar(sa(&acc_empty), acc_ph, bars.spins);        // the previous piece's sums have been read
                acc_ph ^= 1u;
                if (!ok) break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t acc = 0;
            bool there = test_bar(bars.ready + 8u * ring.slot, ring.phase);
            for (int st = 2 * pc.sc0; st < st1; ++st) {
                if (!__all_sync(0xffffffffu, there) && !(ok = wait_bar(bars.ready + 8u * ring.slot, ring.phase, bars.spins))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                Ring on = ring;
                if (++on.slot == a.slots) { on.slot = 0; on.phase ^= 1u; }
                there = st + 1 < st1 && test_bar(bars.ready + 8u * on.slot, on.phase);     // the answer comes under the products
                if (elected()) {
                    const uint64_t da = da0 + (uint64_t)((uint32_t)ring.slot * (kABytes >> 4)), db = db0 + (uint64_t)((uint32_t)(ring.slot * a.x_bytes) >> 4);
#pragma unroll
                    for (int k = 0; k < kStageK / 16; ++k) mma_pair(tmem, da + k * 256, db + k * 2, id0, k ? 1u : acc);
                    if (id1) {
                        const uint64_t db1 = db + (uint64_t)(a.Tp * 4);
#pragma unroll
                        for (int k = 0; k < kStageK / 16; ++k) mma_pair(tmem + (uint32_t)a.Tp, da + k * 256, db1 + k * 2, id1, k ? 1u : acc);
                    }
                    commit_pair(bars.freed + 8u * ring.slot, mask);
                    if (st + 1 == st1) commit_pair(sa(&acc_full), mask);
                }
                acc = 1;
                __syncwarp();
                ring = on;
            }
        }
    }
    if (!ok) {                   // every CTA of the cluster learns of it behind the barrier below
        atomicExch(a.ctrl, 1);
        for (uint32_t r = 0; r < (SPLIT ? 2u * a.ks : 2u); ++r) asm volatile("st.shared::cluster.u32 [%0], 1;" :: "r"(peer(sa(&s_fail), r)) : "memory");
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    cluster_sync();
    const bool failed = *(volatile int*)&s_fail != 0;             // the same answer in the whole cluster
    if (failed) {                // nobody leaves before the pair's products and copies in flight are done
        if (h == 0 && warp == kMmaWarp) {
            if (elected()) commit_pair(sa(&b_drain), 3u << lead);
            __syncwarp();
            wait_bar(sa(&b_drain), 0u, kSpins);
        }
        if (h == 0 && tid >= 32 && tid < 32 + a.slots) drain_copies(tid - 32, a.slots, a.x_bytes, s_copied, sa(b_ready) + 8u * (uint32_t)(tid - 32), crank);
        __syncwarp();
        cluster_sync();
    }
    if (SPLIT && !failed) {
        // this CTA's share of the rows of x of its 128 channels: the slices' sums added in slice order
        const int tile = g / a.ks, slice = g % a.ks, t0 = (tile % a.tok_tiles) * a.T, Tn = min(a.T, a.M - t0);
        const int share = (Tn + a.ks - 1) / a.ks, b0 = slice * share * (kCh / 4), b1 = min(Tn, (slice + 1) * share) * (kCh / 4);
        const uint32_t own = sa(pA);
        for (int i0 = b0 + tid; i0 < b1; i0 += 2 * kThreads) {
            float4 v[2][kMaxCut];                             // two places, every slice's share in flight
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int z = 0; z < kMaxCut; ++z)
                    if (z < a.ks && i0 + u * kThreads < b1)
                        asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[u][z].x), "=f"(v[u][z].y), "=f"(v[u][z].z), "=f"(v[u][z].w)
                                     : "r"(peer(own + (uint32_t)(i0 + u * kThreads) * 16u, 2u * (uint32_t)z + h)));
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int i = i0 + u * kThreads;
                if (i >= b1) break;
                float4 sum = v[u][0];
#pragma unroll
                for (int z = 1; z < kMaxCut; ++z)
                    if (z < a.ks) { sum.x += v[u][z].x; sum.y += v[u][z].y; sum.z += v[u][z].z; sum.w += v[u][z].w; }
                store_quad(a, t0 + i / (kCh / 4), (2 * (tile / a.tok_tiles) + (int)h) * kCh + (i % (kCh / 4)) * 4, sum);
            }
        }
        __syncwarp();
        cluster_sync();          // no CTA leaves while another reads its shared memory
    }
    if (warp == kMmaWarp)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(s_tmem), "r"(a.tmem_cols) : "memory");
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

struct FusedPlan {
    int T, Tp, parts, tok_tiles, pairs, slots, whole, stream, dealt, ks, sc_slice;
    size_t tab, lib, smem;
    double clocks;             // what the model expects
};

// Clocks of a tile's super-chunk: the products (4 T), or shared memory, which every byte crosses at 128 per clock -- per 64 k
// the look-ups of 4 warps (one wavefront each, half with pair tables), V2a's tables, 128 for storing A, 128 for the products'
// reading it, T / 2 for x coming in and T / 2 for its being read --, or the operands' way from L2.  Fitted to look-ups in tables at
// every width: where codebooks sit in registers now (kReg) a stage leaves shared memory more time than this.
double slot_clocks(const Layout& l, int T) {
    const bool pair = l.mode ? l.bits == 2 : l.bits <= 3;
    const double smem = 2.0 * ((pair ? 128 : 256) + (l.mode ? (l.bits == 2 ? 64 : 4 * l.E) : 0) + 256 + T) * 1.08;
    const double products = 4.0 * T, feed = (l.bits * 2048.0 + 128.0 * T) / 40.0, issue = 1250.0;
    double m = products > smem ? products : smem;
    if (m < issue) m = issue;
    return m > feed ? m : feed;
}

// The room of the tables in the plans, that of widths whose codebooks sit in registers included: the costs above were fitted with it,
// and without it (a stage more at 10007 x 4992 V2a N = 4, 301 rows, and at 4096 x 4096 V2 N = 4, 100 rows) they have not been yet.
size_t table_bytes(const Layout& l) {
    const size_t one = l.mode == 0 ? (l.bits <= 3 ? l.E * l.E : l.E) : (l.bits == 2 ? 16 : l.E);
    const size_t units = l.mode == 0 ? 4 : kDecodeWarps;
    if (l.bits == 4) return 4096 * units / 2;
    return (one * 128 < 1024 ? 1024 : one * 128) * units;
}

FusedPlan plan_fused(const Layout& l, int M) {
    FusedPlan best = {};
    const size_t tab = (table_bytes(l) + 1023) & ~size_t(1023);
    const size_t lib = l.mode ? ((size_t)l.L * (l.E + 8) * 2 + 15) & ~size_t(15) : 0;
    const int pairs = (l.RB + 7) / 8;
    int last_T = 0;
    for (int n = (M + 511) / 512; n <= (M + 15) / 16; ++n) {          // tiles along the rows of x
        const int t = (M + n - 1) / n, parts = t > 256 ? 2 : 1, T = (t + 31) & ~31, Tp = parts == 1 ? T : (T / 2 + 31) & ~31;
        if (T == last_T) continue;
        last_T = T;
        if (T < 64 && best.clocks > 0.0) break;
        const int tok = (M + T - 1) / T;
        int slots = (int)((kSmemMax - 8192 - tab - lib) / (kABytes + (size_t)parts * Tp * 64));
        if (slots > kMaxSlots) slots = kMaxSlots;
        if (slots < kMinSlots) continue;
        // a stage's way through decode, outliers and products takes about 2900 clocks and its share of the products
        const double chain = (2900.0 + 2.0 * T) / slots * 2.0, busy = slot_clocks(l, T), step = busy > chain ? busy : chain;
        // a CTA's sums to or from the workspace at 40 bytes a clock, and all of them through DRAM at 2 KB a clock (10007 x 4992,
        // 301 rows, dealt over 74 pairs: 83 us, 23 MB of sums; 40 whole tiles 60 us)
        const double move = T * 512.0 / 40.0, dram = T * 1024.0 / 2000.0;
        const int tiles = pairs * tok, whole = tiles / kPairs, rest = tiles - whole * kPairs;
        const double rounds = whole * (l.SC * step + 1500.0 + 10.0 * T);
        for (int k = 1; k <= 9; ++k) {     // every remaining tile in k parts; or an even deal
            const int dealt = rest == 0 ? 0 : k > 8 ? kPairs : rest * k, stream = rest * l.SC;
            if (k > 1 && (dealt > kPairs || dealt > stream / 2)) continue;  // a part has at least two super-chunks
            const int most = rest ? (stream + dealt - 1) / dealt : 0, cuts = k == 1 ? 1 : k > 8 ? (l.SC - 1) / most + 2 : k;
            const double clocks = rounds + (rest ? most * step + 1500.0 + 10.0 * T + (k > 8 ? 2000.0 : 0.0) : 0.0) + (cuts > 1 ? 6000.0 + cuts * move + 2.0 * dealt * dram : 0.0);
            if (best.clocks == 0.0 || clocks < best.clocks) {
                best.T = T; best.Tp = Tp; best.parts = parts; best.tok_tiles = tok; best.pairs = pairs; best.slots = slots;
                best.whole = whole; best.stream = stream; best.dealt = dealt; best.ks = 1; best.sc_slice = 0; best.clocks = clocks;
            }
            if (!rest) break;
        }
        for (int ks = 2; ks <= kMaxCut; ++ks) {
            const int spp = (l.SC + ks - 1) / ks;
            if ((ks - 1) * spp >= l.SC || spp < 2 || (size_t)T * kCh * 4 > slots * (kABytes + (size_t)parts * Tp * 64) || tiles > kClusters[ks]) continue;
            const double clocks = spp * step + 1500.0 + 4500.0 + 20.0 * T;
            if (clocks < best.clocks) {
                best = FusedPlan{};
                best.T = T; best.Tp = Tp; best.parts = parts; best.tok_tiles = tok; best.pairs = pairs; best.slots = slots;
                best.ks = ks; best.sc_slice = spp; best.clocks = clocks;
            }
        }
    }
    best.tab = tab; best.lib = lib;
    best.smem = 8192 + tab + lib + (size_t)best.slots * (kABytes + (size_t)best.parts * best.Tp * 64);
    return best;
}

// what the kernel is told of a plan
FusedArgs args_of(const Layout& l, int M, const FusedPlan& p) {
    FusedArgs a = {};
    a.rows = l.rows; a.RB = l.RB; a.SC = l.SC; a.M = M; a.ell_slots = l.ell_slots; a.GH = l.GH; a.L = l.L;
    a.tok_tiles = p.tok_tiles; a.T = p.T; a.Tp = p.Tp; a.parts = p.parts;
    a.slots = p.slots; a.x_bytes = p.parts * p.Tp * 64; a.tab_bytes = (int)p.tab;
    a.ks = p.ks; a.sc_slice = p.sc_slice; a.whole = p.whole; a.stream = p.stream; a.dealt = p.dealt;
    a.tmem_cols = p.T <= 32 ? 32 : p.T <= 64 ? 64 : p.T <= 128 ? 128 : p.T <= 256 ? 256 : 512;
    return a;
}
int pairs_of(const FusedPlan& p) { return p.ks > 1 ? p.pairs * p.tok_tiles * p.ks : p.whole ? kPairs : p.dealt; }

template <int N, int MODE>
cudaError_t launch_n(const Layout& l, const GemmCall& c, bool converted, cudaStream_t s) {
    const FusedPlan p = plan_fused(l, c.M);
    static const EncodeTiledFn encode = encode_fn();
    if (!encode || !p.slots) return cudaErrorNotSupported;
    CUtensorMap tmap;
    {
        const cuuint64_t dims[2] = {(cuuint64_t)l.cols, (cuuint64_t)c.M};
        const cuuint64_t strides[1] = {(cuuint64_t)l.cols * 2};
        const cuuint32_t box[2] = {64, (cuuint32_t)(p.Tp / 2)};
        const cuuint32_t estr[2] = {1, 1};
        if (encode(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t*>(c.x), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    static DeviceOnce attr_done;
    const int dev = DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        cudaError_t e = cudaFuncSetAttribute(gemm_fused_kernel<N, MODE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_fused_kernel<N, MODE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    FusedArgs a = args_of(l, c.M, p);
    a.b = blob_at(c.packed, offsets_of(l));
    a.y = c.y; a.ctrl = (int*)c.workspace; a.part = (float*)((char*)c.workspace + prefill_ctrl_bytes(l));
    a.y_kind = c.y_kind; a.converted = converted; a.short_cta = c.short_cta;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs_of(p)), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)(2 * p.ks); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return p.ks > 1 ? cudaLaunchKernelEx(&cfg, gemm_fused_kernel<N, MODE, true>, a, tmap)
                    : cudaLaunchKernelEx(&cfg, gemm_fused_kernel<N, MODE, false>, a, tmap);
}

}  // namespace

bool fused_preferred(const Layout& l, int M) {
    static_assert(2 * kPairs <= kSizingSMs, "two counters for each of fewer than kPairs dealt tiles (prefill_ctrl_bytes)");
    return M > 64 && gemm_tc_supported(l, M);
}
size_t fused_workspace_bytes(const Layout& l, int M) {
    const FusedPlan p = plan_fused(l, M);
    const bool cut = p.dealt && p.dealt * l.SC != p.stream;
    return prefill_ctrl_bytes(l) + (cut ? (size_t)p.dealt * 4 * p.T * kCh * 4 : 0);
}

size_t prefill_workspace_for_up_to(const Layout& l, int M) {
    size_t most = 0;
    // the 64-row kernel: a function of the rows in sixteens; behind its range also with the transposed x that outliers take, so that
    // the size of a longer prompt does not depend on their count
    Layout any = l;
    if (M > 64 && any.nnz == 0) any.nnz = 1;
    for (int m = 16; m < M + 16 && m <= 64; m += 16) {
        const size_t w = gemm_workspace_bytes(any, m < M ? m : M);
        if (w > most) most = w;
    }
    // the pair kernel: its plan is a function of the rows in 32s.  Every plan up to 8192 rows (a few microseconds each); beyond, the
    // most that any plan writes: a part of 512 rows at both ends of every pair's share.
    constexpr int kExact = 8192;
    for (int m = 96; m < M + 32 && m <= kExact; m += 32) {
        if (!fused_preferred(l, m < M ? m : M)) continue;
        const size_t w = fused_workspace_bytes(l, m < M ? m : M);
        if (w > most) most = w;
    }
    if (M > kExact && fused_preferred(l, M)) {
        const size_t w = prefill_ctrl_bytes(l) + (size_t)kPairs * 4 * 512 * kCh * 4;
        if (w > most) most = w;
    }
    return most;
}

void fused_plan_report(const Layout& l, int M, int64_t* out) {
    const FusedPlan p = plan_fused(l, M);
    const int64_t v[] = {p.T, p.Tp, p.parts, p.tok_tiles, p.pairs, p.slots, p.whole, p.stream, p.dealt, p.ks, p.sc_slice, (int64_t)p.smem,
                         (int64_t)kSmemMax, kMinSlots, kPairs, pairs_of(p), (int64_t)prefill_ctrl_bytes(l),
                         (int64_t)fused_workspace_bytes(l, M), l.SC};
    for (size_t i = 0; i < sizeof v / sizeof v[0]; ++i) out[i] = v[i];
}
int fused_piece_report(const Layout& l, int M, int g, int i, int32_t* out) {
    const FusedPlan p = plan_fused(l, M);
    const FusedArgs a = args_of(l, M, p);
    Piece pc = {};
    const bool is = p.ks > 1 ? piece_of<true>(a, g, i, pc) : piece_of<false>(a, g, i, pc);
    out[0] = pc.tile; out[1] = pc.sc0; out[2] = pc.sc1;
    return is;
}

// c.x: the activations as fp16; or bf16, converted first into x_f16
cudaError_t launch_gemm_fused(const Layout& l, const GemmCall& call, void* x_f16, cudaStream_t s) {
    GemmCall c = call;
    if (x_f16) {
        const cudaError_t e = launch_x_to_f16(c.x, x_f16, (size_t)c.M * l.cols, s);
        if (e != cudaSuccess) return e;
        c.x = (const uint16_t*)x_f16;
    }
    if (l.mode == 1) {
        switch (l.bits) {
            case 2: return launch_n<2, 1>(l, c, x_f16 != nullptr, s);
            case 3: return launch_n<3, 1>(l, c, x_f16 != nullptr, s);
            case 4: return launch_n<4, 1>(l, c, x_f16 != nullptr, s);
            case 5: return launch_n<5, 1>(l, c, x_f16 != nullptr, s);
            default: return launch_n<6, 1>(l, c, x_f16 != nullptr, s);
        }
    }
    switch (l.bits) {
        case 2: return launch_n<2, 0>(l, c, x_f16 != nullptr, s);
        case 3: return launch_n<3, 0>(l, c, x_f16 != nullptr, s);
        case 4: return launch_n<4, 0>(l, c, x_f16 != nullptr, s);
        case 5: return launch_n<5, 0>(l, c, x_f16 != nullptr, s);
        default: return launch_n<6, 0>(l, c, x_f16 != nullptr, s);
    }
}

}  // namespace xfp
