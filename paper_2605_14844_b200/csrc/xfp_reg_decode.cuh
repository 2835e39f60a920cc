// Codebooks in registers: N <= 4 bits, no look-up table in shared memory.
//
// A PRMT picks four bytes of eight by four 4-bit selectors, so it looks four indices up in a codebook of eight entries held as byte
// planes (the low bytes of the entries in two registers, the high bytes in two more); two further PRMTs interleave the planes into
// the half2 words of an A fragment.  At N = 4 both halves of the codebook are looked up and a third PRMT takes each byte from the
// half that its index names.  Per eight weights, on the ALU pipe (half a warp instruction per clock and scheduler):
//   N = 2  10.5   (2 selector words of eight indices each per 32 stream bits, 4 shifts and masks, 16 PRMT per 16 weights)
//   N = 3  13.5   (24 bits spread to eight nibbles: three masks here and three multiply-adds on the FMA pipe, 8 PRMT)
//   N = 4  21     (indices are nibbles as they stand: 5 shifts and masks, 16 PRMT)
// against 8 look-ups of one weight or 4 of two on the data pipe of shared memory, a wavefront each where no banks conflict.
#pragma once
#include "xfp_common.cuh"

namespace xfp {

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
__device__ __forceinline__ uint32_t mad_u32(uint32_t a, uint32_t b, uint32_t c) {   // FMA pipe
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// Byte planes of a codebook: low bytes of its entries in ascending order, then the high bytes; 2^N / 4 registers each.
template <int N>
struct RegBook {
    static constexpr int P = (1 << N) / 4;   // registers per plane
    uint32_t lo[P], hi[P];
};

// planes from the 2^N fp16 entries at `cb` (8-byte aligned)
template <int N>
__device__ __forceinline__ RegBook<N> make_book(const uint16_t* __restrict__ cb) {
    RegBook<N> b;
#pragma unroll
    for (int p = 0; p < RegBook<N>::P; ++p) {
        const uint2 e = __ldg((const uint2*)cb + p);   // entries 4p .. 4p+3
        b.lo[p] = prmt(e.x, e.y, 0x6420u);
        b.hi[p] = prmt(e.x, e.y, 0x7531u);
    }
    return b;
}
// planes from entries (2i, 2i + 1) in e[i]
template <int N>
__device__ __forceinline__ RegBook<N> book_of(const uint32_t (&e)[(1 << N) / 2]) {
    RegBook<N> b;
#pragma unroll
    for (int p = 0; p < RegBook<N>::P; ++p) {
        b.lo[p] = prmt(e[2 * p], e[2 * p + 1], 0x6420u);
        b.hi[p] = prmt(e[2 * p], e[2 * p + 1], 0x7531u);
    }
    return b;
}
// V2a: the values D16 = fp16(fp32(scale * lib + mid)) that a group can take, `e` the library's entries
template <int N>
__device__ __forceinline__ void affine_entries(uint32_t (&e)[(1 << N) / 2], uint32_t scale_mid) {
    const float2 sm = __half22float2(*(const __half2*)&scale_mid);
#pragma unroll
    for (int i = 0; i < (1 << N) / 2; ++i) {
        const float2 f = __half22float2(*(const __half2*)&e[i]);
        const __half2 d = __floats2half2_rn(__fmaf_rn(sm.x, f.x, sm.y), __fmaf_rn(sm.x, f.y, sm.y));
        e[i] = *(const uint32_t*)&d;
    }
}
// entries [8 v, 8 v + 8) of a codebook (all four at N = 2) as 32-bit words
template <int N, class Load>
__device__ __forceinline__ void load_entries(uint32_t (&e)[(1 << N) / 2], const uint16_t* cb, Load load) {
    if constexpr (N == 2) {
        const uint2 t = load((const uint2*)cb);
        e[0] = t.x; e[1] = t.y;
    } else {
#pragma unroll
        for (int v = 0; v < (1 << N) / 8; ++v) {
            const uint4 t = load((const uint4*)cb + v);
            e[4 * v] = t.x; e[4 * v + 1] = t.y; e[4 * v + 2] = t.z; e[4 * v + 3] = t.w;
        }
    }
}

// The library as byte planes in shared memory: 16-byte vectors [2^N / 8][L] (8-byte ones [L] at N = 2), so that lanes with
// different ids spread over the bank groups.
template <int N>
__device__ __forceinline__ void store_book(unsigned char* tab, int L, int id, const RegBook<N>& b) {
    if constexpr (N == 2) {
        ((uint2*)tab)[id] = make_uint2(b.lo[0], b.hi[0]);
    } else if constexpr (N == 3) {
        ((uint4*)tab)[id] = make_uint4(b.lo[0], b.lo[1], b.hi[0], b.hi[1]);
    } else {
        ((uint4*)tab)[id] = make_uint4(b.lo[0], b.lo[1], b.hi[0], b.hi[1]);
        ((uint4*)tab)[L + id] = make_uint4(b.lo[2], b.lo[3], b.hi[2], b.hi[3]);
    }
}
template <int N>
__device__ __forceinline__ RegBook<N> load_book(const unsigned char* tab, int L, uint32_t id) {
    RegBook<N> b;
    if constexpr (N == 2) {
        const uint2 t = ((const uint2*)tab)[id];
        b.lo[0] = t.x; b.hi[0] = t.y;
    } else {
        const uint4 t = ((const uint4*)tab)[id];
        b.lo[0] = t.x; b.lo[1] = t.y; b.hi[0] = t.z; b.hi[1] = t.w;
        if constexpr (N == 4) {
            const uint4 u = ((const uint4*)tab)[L + id];
            b.lo[2] = u.x; b.lo[3] = u.y; b.hi[2] = u.z; b.hi[3] = u.w;
        }
    }
    return b;
}

// Weights 8j .. 8j+7 (j compile time) of a 128-weight stream w[4N], as four half2 in the order of the A fragment.
//   N = 3, 4:  f[0] = (0, 1)  f[2] = (2, 3)  f[1] = (4, 5)  f[3] = (6, 7)
//   N = 2:     f[0] = (0, 2)  f[2] = (4, 6)  f[1] = (1, 3)  f[3] = (5, 7)   (nibbles hold every second index)
template <int N>
__device__ __forceinline__ void reg_decode8(uint32_t (&f)[4], const uint32_t* w, int j, const RegBook<N>& b) {
    if constexpr (N == 2) {
        const uint32_t v = w[j >> 1];
        uint32_t e = v & 0x33333333u, o = (v >> 2) & 0x33333333u;
        if (j & 1) { e >>= 16; o >>= 16; }
        const uint32_t el = prmt(b.lo[0], 0u, e), eh = prmt(b.hi[0], 0u, e);
        const uint32_t ol = prmt(b.lo[0], 0u, o), oh = prmt(b.hi[0], 0u, o);
        f[0] = prmt(el, eh, 0x5140u); f[2] = prmt(el, eh, 0x7362u);
        f[1] = prmt(ol, oh, 0x5140u); f[3] = prmt(ol, oh, 0x7362u);
    } else if constexpr (N == 3) {
        const int q = (j >> 2) * 3;
        uint32_t t;      // bits 24j .. 24j+23
        switch (j & 3) {
            case 0: t = w[q] & 0xffffffu; break;
            case 1: t = __funnelshift_r(w[q], w[q + 1], 24) & 0xffffffu; break;
            case 2: t = __funnelshift_r(w[q + 1], w[q + 2], 16) & 0xffffffu; break;
            default: t = w[q + 2] >> 8; break;
        }
        t = mad_u32(t & 0xfff000u, 15u, t);         // two fields of 12 bits, 16 apart
        t = mad_u32(t & 0x0fc00fc0u, 3u, t);        // four of 6, 8 apart
        t = mad_u32(t & 0x38383838u, 1u, t);        // eight of 3, 4 apart
        const uint32_t u = t >> 16;
        const uint32_t l0 = prmt(b.lo[0], b.lo[1], t), h0 = prmt(b.hi[0], b.hi[1], t);
        const uint32_t l1 = prmt(b.lo[0], b.lo[1], u), h1 = prmt(b.hi[0], b.hi[1], u);
        f[0] = prmt(l0, h0, 0x5140u); f[2] = prmt(l0, h0, 0x7362u);
        f[1] = prmt(l1, h1, 0x5140u); f[3] = prmt(l1, h1, 0x7362u);
    } else {
        const uint32_t v = w[j];
        const uint32_t s = v & 0x77777777u, m = ((v >> 1) & 0x44444444u) | 0x32103210u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t sh = h ? s >> 16 : s, mh = h ? m >> 16 : m;
            const uint32_t l = prmt(prmt(b.lo[0], b.lo[1], sh), prmt(b.lo[2], b.lo[3], sh), mh);
            const uint32_t g = prmt(prmt(b.hi[0], b.hi[1], sh), prmt(b.hi[2], b.hi[3], sh), mh);
            f[h] = prmt(l, g, 0x5140u); f[2 + h] = prmt(l, g, 0x7362u);
        }
    }
}

// The same eight weights in ascending order, two to a word.
template <int N>
__device__ __forceinline__ uint4 reg_decode8_ordered(const uint32_t* w, int j, const RegBook<N>& b) {
    uint32_t f[4];
    reg_decode8<N>(f, w, j, b);
    if constexpr (N == 2) return make_uint4(prmt(f[0], f[1], 0x5410u), prmt(f[0], f[1], 0x7632u), prmt(f[2], f[3], 0x5410u), prmt(f[2], f[3], 0x7632u));
    return make_uint4(f[0], f[2], f[1], f[3]);
}

// Position of activation k in the staged copy of x that matches: a diagonal lane of the B fragment fetches the values of two steps
// with one 16-byte load, lanes (g == t) the first half of every 16 positions and lanes (g == t + 4) the second.
//   N = 2: the even k of every 16, then the odd ones;  else the middle blocks of four of every 16 trade places
template <bool EVEN_ODD>
__device__ __forceinline__ uint32_t xpos_of(uint32_t k) {
    if (EVEN_ODD) return (k & ~15u) | ((k & 1u) << 3) | ((k & 15u) >> 1);
    return (k & ~12u) | ((k & 4u) << 1) | ((k & 8u) >> 1);
}

}  // namespace xfp
