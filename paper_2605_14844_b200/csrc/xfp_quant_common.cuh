// Device helpers shared by the encoder's translation units (xfp_quant.cu, xfp_quant_lloyd.cu, xfp_quant_libfit.cu).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

namespace xq {

__device__ __forceinline__ double h2d(uint16_t h) { return (double)__half2float(__ushort_as_half(h)); }
__device__ __forceinline__ uint16_t d2h(double d) { return __half_as_ushort(__double2half(d)); }

// D16 of a V2a weight: one fp32 rounding of scale*lib + mid (the product of two fp16 is exact in fp32),
// then one fp16 rounding ("V2a: Shared Codebook Library").
__device__ __forceinline__ uint16_t v2a_value16(uint16_t scale, uint16_t lib, uint16_t mid) {
    const float r = __fmaf_rn(__half2float(__ushort_as_half(scale)), __half2float(__ushort_as_half(lib)),
                              __half2float(__ushort_as_half(mid)));
    return __half_as_ushort(__float2half_rn(r));
}

// Index of the entry nearest to x among e[0..E), ties to the lower index: the answer of a linear scan that keeps an
// entry only when it is strictly nearer.  When the entries ascend (codebooks and decoded library entries do) x is
// bracketed by bisection and only its two neighbours are measured; the scan's answer is the nearer of the two
// (the lower on an exact tie: fp64 rounding is monotone and distinct fp16 values are too far apart to round to
// the same distance), moved down over duplicates of its value.
__device__ __forceinline__ int nearest_entry(const double* e, int E, double x, bool ascending) {
    if (!ascending) {
        int best = 0;
        double bd = fabs(__dsub_rn(x, e[0]));
        for (int j = 1; j < E; ++j) {
            const double d = fabs(__dsub_rn(x, e[j]));
            if (d < bd) { bd = d; best = j; }
        }
        return best;
    }
    int lo = 0, hi = E;   // first index whose entry is >= x
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (e[mid] < x) lo = mid + 1; else hi = mid;
    }
    int best;
    if (lo == 0) best = 0;
    else if (lo == E) best = E - 1;
    else best = fabs(__dsub_rn(x, e[lo - 1])) <= fabs(__dsub_rn(x, e[lo])) ? lo - 1 : lo;
    while (best > 0 && e[best - 1] == e[best]) --best;
    return best;
}

// Sum over the block in a fixed tree order; every thread gets the result.
__device__ __forceinline__ double block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = blockDim.x >> 1; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] = __dadd_rn(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

// Exclusive scan of one int per thread over the block (blockDim.x <= 1024, a multiple of 32); returns
// the thread's offset and leaves the block total in *total.
__device__ __forceinline__ int block_excl_scan(int v, int* sh_warp, int* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += t;
    }
    if (lane == 31) sh_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        int x = lane < nw ? sh_warp[lane] : 0;
        int xi = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, xi, d);
            if (lane >= d) xi += t;
        }
        if (lane < nw) sh_warp[lane] = xi - x;
        if (lane == 31) *total = xi;
    }
    __syncthreads();
    const int r = sh_warp[w] + inc - v;
    __syncthreads();
    return r;
}

// The value Lloyd and LibFit see at weight t: mu at an extracted position.
__device__ __forceinline__ double bulk_value(const float* __restrict__ W, const uint8_t* __restrict__ mask,
                                             int64_t t, double mu) {
    return (mask != nullptr && mask[t]) ? mu : (double)W[t];
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// floats in the order of their values as integers
__device__ __forceinline__ int ordered(float f) { const int i = __float_as_int(f); return i < 0 ? (int)(0x80000000u - (uint32_t)i) : i; }
__device__ __forceinline__ float unordered(int o) { return __int_as_float(o < 0 ? (int)(0x80000000u - (uint32_t)o) : o); }

// Largest float x in [a, b) that the nearest-entry rule gives to entry a: |x - a| <= |x - b| in fp64.  The rule is
// monotone in x; the float below the midpoint keeps it, and the next one nearly always breaks it.
__device__ __forceinline__ float last_of_lower(double a, double b) {
    const double mid = __dmul_rn(0.5, __dadd_rn(a, b));       // exact: a and b are fp16 values
    const float c = __double2float_rd(mid);
    int lo = ordered(c), hi = ordered(__double2float_rn(b));   // the rule holds at lo, breaks at hi
    if (lo + 1 < hi) {
        const double x = (double)unordered(lo + 1);
        if (fabs(__dsub_rn(x, a)) <= fabs(__dsub_rn(x, b))) {
            while (lo + 1 < hi) {
                const int m = lo + ((hi - lo) >> 1);
                const double y = (double)unordered(m);
                if (fabs(__dsub_rn(y, a)) <= fabs(__dsub_rn(y, b))) lo = m; else hi = m;
            }
        }
    }
    return unordered(lo);
}

}  // namespace xq
