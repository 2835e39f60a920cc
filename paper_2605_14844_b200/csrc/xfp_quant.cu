// The XFP encoder on the GPU ("Quantization": Outlier Extraction, Learned Codebook via Lloyd Iteration,
// V2a LibFit, the residual of Eq. 1, Algorithm 1's cosine gate and auto-select).
//
// Every decision that yields an integer or an fp16 value is taken in IEEE fp64 with explicit
// round-to-nearest intrinsics (no fused multiply-add), in the order the method states: a Lloyd cell
// boundary is the midpoint of two entries, a cell mean is a difference of two SERIAL prefix sums over
// the sorted channel divided by the count, a nearest entry is found by a linear scan with a strict
// "less than", a group's squared error is summed value by value.  The serial parts are short (one
// channel, one group) and the parallelism is across channels, groups and library entries.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "../../include/xfp_quant.h"
#include "xfp_internal.h"   // sm_count()
#include "xfp_quant_common.cuh"
#include "xfp_quant_internal.h"

namespace xq {

constexpr int kRedBlocks = 1024;   // partial sums of a whole-matrix reduction
constexpr int kRedThreads = 256;
constexpr int kTieChunk = 4096;    // elements per block in the ordered tie pass (256 threads x 16)
constexpr int kTiePer = 16;

// ------------------------------------------------------------------ statistics

// One pass for both moments: a block sums d and d^2 of its chunk, d = w - p with p the mean of the chunk's first values,
// and leaves (sum of w, sum of squared deviations from the chunk's own mean); stats_final combines the chunks around the
// matrix mean.  The shift keeps the cancellation of sum d^2 - (sum d)^2 / n at a factor near one, so sigma is as good as
// that of a second pass over the matrix (which took another 37 us of 12288 x 4096 weights).
__global__ void __launch_bounds__(kRedThreads) stats_partial(const float* __restrict__ W, int64_t n, double2* part) {
    __shared__ double sh[kRedThreads];
    const int64_t n4 = n >> 2, per = (n4 + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = b0 + per < n4 ? b0 + per : n4;
    const float4* W4 = (const float4*)W;
    const int tail = blockIdx.x == 0 ? (int)(n & 3) : 0;      // the last n mod 4 weights belong to block 0
    int64_t cnt = (b1 > b0 ? b1 - b0 : 0) * 4 + tail;
    double s = 0.0;
    int64_t t = b0 + threadIdx.x;
    int have = 0;
    if (t < b1) { const float4 w = __ldg(W4 + t); s = ((double)w.x + (double)w.y) + ((double)w.z + (double)w.w); have = 4; }
    else if ((int)threadIdx.x < tail && b1 <= b0) { s = (double)W[(n & ~(int64_t)3) + threadIdx.x]; have = 1; }
    const double ps = block_sum(s, sh), pn = block_sum((double)have, sh);
    double p = pn > 0.0 ? ps / pn : 0.0;
    if (!(fabs(p) < INFINITY)) p = 0.0;        // an infinite weight makes the mean infinite, not the differences from an infinite shift NaN
    double a[4] = {0.0, 0.0, 0.0, 0.0}, q[4] = {0.0, 0.0, 0.0, 0.0};
    for (; t < b1; t += 4 * kRedThreads) {
        float4 w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (t + u * kRedThreads < b1) w[u] = __ldg(W4 + t + u * kRedThreads);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (t + u * kRedThreads < b1) {
                const float f[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) { const double d = (double)f[i] - p; a[i] += d; q[i] = fma(d, d, q[i]); }
            }
        }
    }
    if ((int)threadIdx.x < tail) { const double d = (double)W[(n & ~(int64_t)3) + threadIdx.x] - p; a[0] += d; q[0] = fma(d, d, q[0]); }
    const double sa = block_sum((a[0] + a[1]) + (a[2] + a[3]), sh), sq = block_sum((q[0] + q[1]) + (q[2] + q[3]), sh);
    if (threadIdx.x == 0)
        part[blockIdx.x] = cnt ? make_double2(p * (double)cnt + sa, sq - sa * (sa / (double)cnt)) : make_double2(0.0, 0.0);
}

__global__ void __launch_bounds__(kRedThreads) stats_final(const double2* part, int64_t n, double* ms) {
    __shared__ double sh[kRedThreads];
    const int64_t n4 = n >> 2, per = (n4 + kRedBlocks - 1) / kRedBlocks;
    double2 v[kRedBlocks / kRedThreads];
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < kRedBlocks / kRedThreads; ++i) { v[i] = part[threadIdx.x + i * kRedThreads]; acc += v[i].x; }
    const double mu = block_sum(acc, sh) / (double)n;
    acc = 0.0;
#pragma unroll
    for (int i = 0; i < kRedBlocks / kRedThreads; ++i) {
        const int b = threadIdx.x + i * kRedThreads;
        const int64_t b0 = (int64_t)b * per, b1 = b0 + per < n4 ? b0 + per : n4;
        const int64_t cnt = (b1 > b0 ? b1 - b0 : 0) * 4 + (b == 0 ? (n & 3) : 0);
        if (cnt) { const double d = v[i].x / (double)cnt - mu; acc += v[i].y + (double)cnt * d * d; }
    }
    const double ss = block_sum(acc, sh);
    if (threadIdx.x == 0) { ms[0] = mu; ms[1] = sqrt((ss < 0.0 ? 0.0 : ss) / (double)n); }   // NaN stays NaN
}

// ------------------------------------------------------------------ exact selection by radix descent

// State of one selection: after eight 8-bit passes `prefix` is the key of the wanted element and `k`
// its rank among the elements with that key (in scan direction).
struct SelState {
    unsigned long long prefix;
    long long k;
    long long count;   // candidates (threshold mode: weights above the threshold)
    long long keep;    // entries to keep
    int shift;
    int descending;
    int skip;          // 1: nothing to select (all candidates are kept, or none)
    int pad;
    double value[2];   // selected values (median passes)
    unsigned int hist[256];
};

// |w - mu| of weight t as an order-preserving key (non-negative doubles order like their bit patterns).
struct SrcAbsDev {
    const float* W;
    const double* ms;
    const uint8_t* mask;  // candidates only where mask != 0 (NULL: every weight)
    __device__ bool valid(int64_t t) const { return mask == nullptr || mask[t] != 0; }
    __device__ unsigned long long key(int64_t t, double mu) const {
        return (unsigned long long)__double_as_longlong(fabs(__dsub_rn((double)W[t], mu)));
    }
    __device__ double mu() const { return ms[0]; }
};

// Any doubles: flip so that unsigned order equals numeric order.
struct SrcDouble {
    const double* v;
    __device__ bool valid(int64_t) const { return true; }
    __device__ unsigned long long key(int64_t t, double) const {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v[t]);
        return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
    }
    __device__ double mu() const { return 0.0; }
};
__device__ __forceinline__ double unflip(unsigned long long k) {
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

template <class Src>
__global__ void __launch_bounds__(256) sel_hist(Src src, int64_t n, SelState* st) {
    __shared__ unsigned int h[256];
    if (st->skip) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const int shift = st->shift;
    const unsigned long long prefix = st->prefix;
    const double mu = src.mu();
    // runs of one digit (the high bytes of similar magnitudes) are counted in a register first
    unsigned int run_bin = 0, run = 0;
    for (int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x; t < n; t += (int64_t)gridDim.x * 256) {
        if (!src.valid(t)) continue;
        const unsigned long long key = src.key(t, mu);
        if (shift == 56 || ((key ^ prefix) >> (shift + 8)) == 0) {
            const unsigned int bin = (unsigned int)(key >> shift) & 255u;
            if (bin != run_bin && run) { atomicAdd(&h[run_bin], run); run = 0; }
            run_bin = bin;
            ++run;
        }
    }
    if (run) atomicAdd(&h[run_bin], run);
    __syncthreads();
    if (h[threadIdx.x]) atomicAdd(&st->hist[threadIdx.x], h[threadIdx.x]);
}

__global__ void sel_pick(SelState* st) {
    if (st->skip) return;
    long long k = st->k;
    const int shift = st->shift;
    int d;
    if (st->descending) {
        for (d = 255; d > 0; --d) {
            const long long c = st->hist[d];
            if (k < c) break;
            k -= c;
        }
    } else {
        for (d = 0; d < 255; ++d) {
            const long long c = st->hist[d];
            if (k < c) break;
            k -= c;
        }
    }
    st->k = k;
    st->prefix |= (unsigned long long)d << shift;
    st->shift = shift - 8;
    for (int j = 0; j < 256; ++j) st->hist[j] = 0;
}

__global__ void sel_begin(SelState* st, long long k, int descending) {
    st->prefix = 0;
    st->k = k;
    st->shift = 56;
    st->descending = descending;
    st->skip = 0;
    for (int j = 0; j < 256; ++j) st->hist[j] = 0;
}

// value[slot] = the selected double (SrcDouble keys)
__global__ void sel_store_double(SelState* st, int slot) { st->value[slot] = unflip(st->prefix); }
// value[slot] = the selected |w - mu|
__global__ void sel_store_absdev(SelState* st, int slot) { st->value[slot] = __longlong_as_double((long long)st->prefix); }

__global__ void median_finish(const SelState* st, int64_t n, double scale, double* out) {
    const double m = (n & 1) ? st->value[1] : __dmul_rn(0.5, __dadd_rn(st->value[0], st->value[1]));
    *out = scale == 1.0 ? m : __dmul_rn(scale, m);
}

// Median of a short array (the per-channel cosines), one block, one launch: the keys' range is cut into 2048 equal steps
// and counted, and the members of the one or two steps that hold the middle values are ranked against each other.  Where
// those steps hold more than a block's worth of keys (many equal values) their range is cut again.
__device__ __forceinline__ void median_small(const double* __restrict__ v, int n, double* out) {
    constexpr int kBins = 2048, kCand = 1024;
    __shared__ unsigned int hist[kBins];
    __shared__ unsigned long long cand[kCand], s_lo, s_hi, s_val[2];
    __shared__ int sh[32];
    __shared__ int total, s_n, s_bin[2], s_before;
    const SrcDouble src{v};
    const int tid = threadIdx.x;
    unsigned long long lo = ~0ull, hi = 0ull;
    for (int t = tid; t < n; t += 1024) { const unsigned long long k = src.key(t, 0.0); lo = k < lo ? k : lo; hi = k > hi ? k : hi; }
    if (tid == 0) { s_lo = ~0ull; s_hi = 0ull; }
    __syncthreads();
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, lo, d), b = __shfl_xor_sync(0xffffffffu, hi, d);
        lo = a < lo ? a : lo; hi = b > hi ? b : hi;
    }
    if ((tid & 31) == 0) { atomicMin(&s_lo, lo); atomicMax(&s_hi, hi); }
    __syncthreads();
    lo = s_lo; hi = s_hi;
    int k0 = (n - 1) / 2, k1 = n / 2;        // ranks of the middle values among the keys of [lo, hi]
    for (;;) {
        if (lo == hi) { if (tid == 0) s_val[0] = s_val[1] = lo; break; }
        const unsigned long long span = hi - lo;
        const int sft = 64 - __clzll((long long)span) > 11 ? 64 - __clzll((long long)span) - 11 : 0;   // span >> sft < 2048
        for (int i = tid; i < kBins; i += 1024) hist[i] = 0;
        if (tid == 0) s_n = 0;
        __syncthreads();
        for (int t = tid; t < n; t += 1024) {
            const unsigned long long k = src.key(t, 0.0);
            if (k >= lo && k <= hi) atomicAdd(&hist[(k - lo) >> sft], 1u);
        }
        __syncthreads();
        const int h0 = (int)hist[2 * tid], h1 = (int)hist[2 * tid + 1];
        const int off = block_excl_scan(h0 + h1, sh, &total);
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            const int k = w ? k1 : k0;
            if (k >= off && k < off + h0) { s_bin[w] = 2 * tid; if (w == 0) s_before = off; }
            else if (k >= off + h0 && k < off + h0 + h1) { s_bin[w] = 2 * tid + 1; if (w == 0) s_before = off + h0; }
        }
        __syncthreads();
        const unsigned long long a = lo + ((unsigned long long)s_bin[0] << sft);
        const unsigned long long bb = lo + (((unsigned long long)s_bin[1] + 1ull) << sft) - 1ull, b = bb < hi ? bb : hi;
        k0 -= s_before; k1 -= s_before;
        for (int t = tid; t < n; t += 1024) {
            const unsigned long long k = src.key(t, 0.0);
            if (k >= a && k <= b) { const int at = atomicAdd(&s_n, 1); if (at < kCand) cand[at] = k; }
        }
        __syncthreads();
        const int c = s_n;
        if (c <= kCand) {
            if (tid < c) {
                const unsigned long long mine = cand[tid];
                int rank = 0;
                for (int j = 0; j < c; ++j) rank += cand[j] < mine || (cand[j] == mine && j < tid);
                if (rank == k0) s_val[0] = mine;
                if (rank == k1) s_val[1] = mine;
            }
            break;
        }
        if (s_bin[0] != s_bin[1]) {
            // the middle falls between two crowded steps: the largest key of the first and the smallest of the next
            const unsigned long long edge = lo + ((unsigned long long)(s_bin[0] + 1) << sft);
            unsigned long long l = 0ull, h = ~0ull;
            for (int t = tid; t < n; t += 1024) {
                const unsigned long long k = src.key(t, 0.0);
                if (k < edge) l = k > l ? k : l; else h = k < h ? k : h;
            }
            if (tid == 0) { s_val[0] = 0ull; s_val[1] = ~0ull; }
            __syncthreads();
            atomicMax(&s_val[0], l); atomicMin(&s_val[1], h);
            break;
        }
        // the common step, narrowed to the keys it holds
        unsigned long long l = ~0ull, h = 0ull;
        for (int t = tid; t < n; t += 1024) {
            const unsigned long long k = src.key(t, 0.0);
            if (k >= a && k <= b) { l = k < l ? k : l; h = k > h ? k : h; }
        }
        if (tid == 0) { s_lo = ~0ull; s_hi = 0ull; }
        __syncthreads();
        atomicMin(&s_lo, l); atomicMax(&s_hi, h);
        __syncthreads();
        lo = s_lo; hi = s_hi;
    }
    __syncthreads();
    if (tid == 0) *out = (n & 1) ? unflip(s_val[1]) : __dmul_rn(0.5, __dadd_rn(unflip(s_val[0]), unflip(s_val[1])));
}

template <class Src>
static cudaError_t run_select(Src src, int64_t n, SelState* st, cudaStream_t s) {
    int blocks = (int)((n + 256 * 16 - 1) / (256 * 16));
    if (blocks < 1) blocks = 1;
    const int cap = xfp::sm_count() * 8;
    if (blocks > cap) blocks = cap;
    for (int p = 0; p < 8; ++p) {
        sel_hist<Src><<<blocks, 256, 0, s>>>(src, n, st);
        sel_pick<<<1, 1, 0, s>>>(st);
    }
    return cudaGetLastError();
}

// median of the keys of src (even n: mean of the two middle ones), times `scale`, to *out
template <class Src>
static cudaError_t run_median(Src src, int64_t n, double scale, bool absdev, double* out, SelState* st,
                              cudaStream_t s) {
    for (int slot = 0; slot < 2; ++slot) {
        const long long k = slot == 0 ? (n - 1) / 2 : n / 2;
        sel_begin<<<1, 1, 0, s>>>(st, k, 0);
        cudaError_t e = run_select(src, n, st, s);
        if (e != cudaSuccess) return e;
        if (absdev) sel_store_absdev<<<1, 1, 0, s>>>(st, slot);
        else sel_store_double<<<1, 1, 0, s>>>(st, slot);
    }
    // odd n: both passes chose the same element and value[1] is used
    median_finish<<<1, 1, 0, s>>>(st, n, scale, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ outlier mask

// Sixteen weights per thread and step: four 16-byte loads in flight, one 16-byte store of mask bytes.
__global__ void __launch_bounds__(256) mask_threshold(const float* __restrict__ W, int64_t n,
                                                       const double* __restrict__ ms, double k, uint8_t* mask,
                                                       SelState* st) {
    __shared__ int warp_cnt[8];
    const double mu = ms[0];
    const double thresh = __dmul_rn(k, ms[1]);
    int c = 0;
    const int64_t n16 = n >> 4;
    for (int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x; t < n16; t += (int64_t)gridDim.x * 256) {
        const float4* p = (const float4*)W + 4 * t;
        const float4 w[4] = {__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3)};
        uint32_t o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t a = fabs(__dsub_rn((double)w[u].x, mu)) > thresh, b = fabs(__dsub_rn((double)w[u].y, mu)) > thresh,
                           d = fabs(__dsub_rn((double)w[u].z, mu)) > thresh, e = fabs(__dsub_rn((double)w[u].w, mu)) > thresh;
            o[u] = a | (b << 8) | (d << 16) | (e << 24);
            c += (int)(a + b + d + e);
        }
        ((uint4*)mask)[t] = make_uint4(o[0], o[1], o[2], o[3]);
    }
    if (blockIdx.x == 0 && (int64_t)threadIdx.x < (n & 15)) {
        const int64_t t = (n & ~(int64_t)15) + threadIdx.x;
        const int m = fabs(__dsub_rn((double)W[t], mu)) > thresh;
        mask[t] = (uint8_t)m;
        c += m;
    }
    for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
    if ((threadIdx.x & 31) == 0) warp_cnt[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < 8; ++w) tot += warp_cnt[w];
        if (tot) atomicAdd((unsigned long long*)&st->count, (unsigned long long)tot);
    }
}

__global__ void outlier_zero(SelState* st) { st->count = 0; }

// Decide what the selection has to do.  mode 0: keep = floor(cap*n), select only when more qualified.
// mode 1: keep = floor(rate*n) of all weights.  skip_out (may be null): a copy of the decision for the host.
__global__ void outlier_plan(SelState* st, int64_t n, int mode, double frac, int64_t* count_out, int64_t* skip_out) {
    const long long keep = (long long)floor(__dmul_rn(frac, (double)n));
    if (threadIdx.x < 256) st->hist[threadIdx.x] = 0;
    if (threadIdx.x) return;
    st->keep = keep;
    st->prefix = 0;
    st->shift = 56;
    st->descending = 1;
    if (mode == 0) {
        st->skip = st->count <= keep;
        st->k = keep - 1;
        *count_out = st->skip ? st->count : keep;
    } else {
        st->skip = keep <= 0;
        st->count = n;
        st->k = keep - 1;
        *count_out = keep > 0 ? keep : 0;
    }
    if (skip_out) *skip_out = st->skip;
}

__global__ void __launch_bounds__(256) mask_clear(uint8_t* mask, int64_t n) {
    for (int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x; t < n; t += (int64_t)gridDim.x * 256) mask[t] = 0;
}

// Ties of the selected key are kept in position order: count them per chunk ...
template <class Src>
__global__ void __launch_bounds__(256) tie_count(Src src, int64_t n, const SelState* st, int* blockcnt) {
    __shared__ int sh[8];
    __shared__ int total;
    if (st->skip) return;
    const unsigned long long T = st->prefix;
    const double mu = src.mu();
    const int64_t base = (int64_t)blockIdx.x * kTieChunk + (int64_t)threadIdx.x * kTiePer;
    int c = 0;
    for (int e = 0; e < kTiePer; ++e) {
        const int64_t t = base + e;
        if (t < n && src.valid(t) && src.key(t, mu) == T) ++c;
    }
    block_excl_scan(c, sh, &total);
    if (threadIdx.x == 0) blockcnt[blockIdx.x] = total;
}

// ... turn the chunk counts into offsets ...
__global__ void __launch_bounds__(1024) tie_scan(int* blockcnt, int nblk, const SelState* st) {
    __shared__ int sh[32];
    __shared__ int total;
    if (st->skip) return;
    int carry = 0;
    for (int b0 = 0; b0 < nblk; b0 += 1024) {
        const int b = b0 + threadIdx.x;
        const int v = b < nblk ? blockcnt[b] : 0;
        const int off = block_excl_scan(v, sh, &total);
        if (b < nblk) blockcnt[b] = carry + off;
        carry += total;
        __syncthreads();
    }
}

// ... and write the final mask: above the selected key, or one of its first k+1 ties.
template <class Src>
__global__ void __launch_bounds__(256) tie_apply(Src src, int64_t n, const SelState* st, const int* blockcnt,
                                                 uint8_t* mask) {
    __shared__ int sh[8];
    __shared__ int total;
    if (st->skip) return;
    const unsigned long long T = st->prefix;
    const long long need = st->k + 1;
    const double mu = src.mu();
    const int64_t base = (int64_t)blockIdx.x * kTieChunk + (int64_t)threadIdx.x * kTiePer;
    unsigned long long keys[kTiePer];
    int c = 0;
#pragma unroll
    for (int e = 0; e < kTiePer; ++e) {
        const int64_t t = base + e;
        const bool ok = t < n && src.valid(t);
        keys[e] = ok ? src.key(t, mu) : 0ull;
        if (ok && keys[e] == T) ++c;   // slots that are no candidates never count, whatever T is
    }
    long long rank = (long long)blockcnt[blockIdx.x] + block_excl_scan(c, sh, &total);
#pragma unroll
    for (int e = 0; e < kTiePer; ++e) {
        const int64_t t = base + e;
        if (t >= n) break;
        if (!src.valid(t)) continue;   // not a candidate: its mask byte is already 0
        int m = 0;
        if (keys[e] > T) m = 1;
        else if (keys[e] == T) m = rank++ < need;
        mask[t] = (uint8_t)m;
    }
}

// ------------------------------------------------------------------ decoded value of a stored index

struct Unpacked {
    const uint8_t* idx;
    const uint16_t* cb;
    const uint8_t* gid;
    const uint16_t* gscale;
    const uint16_t* gmid;
    int mode, K, E, G, group;
};
__device__ __forceinline__ uint16_t decode16(const Unpacked& u, int row, int k) {
    const int q = u.idx[(int64_t)row * u.K + k];
    if (u.mode == 0) return u.cb[(int64_t)row * u.E + q];
    const int64_t g = (int64_t)row * u.G + k / u.group;
    return v2a_value16(u.gscale[g], u.cb[(int)u.gid[g] * u.E + q], u.gmid[g]);
}

// ------------------------------------------------------------------ residual (CSR)

__global__ void __launch_bounds__(256) row_count_kernel(const uint8_t* __restrict__ mask, int rows, int K, int* cnt) {
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= rows) return;
    const uint32_t* m = (const uint32_t*)(mask + (int64_t)row * K);
    int c = 0;
#pragma unroll 8
    for (int k = lane; k < K / 4; k += 32) c += __popc(__vcmpne4(__ldg(m + k), 0u)) >> 3;
    for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
    if (lane == 0) cnt[row] = c;
}

// One block; every thread owns a run of consecutive rows.
__device__ __forceinline__ void rowptr_block(const int* __restrict__ cnt, int rows, int32_t* rowptr) {
    __shared__ int sh[32];
    __shared__ int total;
    const int per = (rows + 1023) / 1024, b0 = threadIdx.x * per, b1 = b0 + per < rows ? b0 + per : rows;
    int v = 0;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) v += cnt[b];
    int run = block_excl_scan(v, sh, &total);
#pragma unroll 8
    for (int b = b0; b < b1; ++b) { const int x = cnt[b]; rowptr[b] = run; run += x; }
    if (threadIdx.x == 0) rowptr[rows] = total;
}
__global__ void __launch_bounds__(1024) rowptr_scan(const int* __restrict__ cnt, int rows, int32_t* rowptr) { rowptr_block(cnt, rows, rowptr); }

// The median of the cosines, and in a second block the row pointers (`cnt` not null): two serial blocks of about 10 us each at
// 12288 channels, side by side.
__global__ void __launch_bounds__(1024) median_small_kernel(const double* __restrict__ v, int n, double* out, const int* __restrict__ cnt,
                                                            int32_t* rowptr) {
    if (blockIdx.x == 0) median_small(v, n, out);
    else rowptr_block(cnt, n, rowptr);
}

// A warp per channel.  The mask is read 512 weights at a time (four words per lane in flight); the places of the set bytes
// follow from four ballots per word, and their columns are collected in shared memory so that the gathers (weight, index,
// codebook entry: three dependent trips) run with every lane busy instead of with the few lanes that found something.
__global__ void __launch_bounds__(256) residual_kernel(const float* __restrict__ W, const uint8_t* __restrict__ mask,
                                                        Unpacked u, int rows, const int32_t* __restrict__ rowptr,
                                                        int32_t* ocol, uint16_t* oval, int64_t capacity) {
    constexpr int kList = 1024;         // a step adds at most 512 columns, the list is emptied when 512 are waiting
    __shared__ uint16_t s_list[8][kList];
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= rows) return;
    uint16_t* list = s_list[threadIdx.x >> 5];
    int64_t p = rowptr[row];
    if (rowptr[row + 1] == p) return;
    const uint32_t* m4 = (const uint32_t*)(mask + (int64_t)row * u.K);
    const uint32_t below = (1u << lane) - 1u;
    const int words = u.K / 4;          // a multiple of 32
    int n = 0;
    for (int w0 = 0; w0 < words; w0 += 128) {
        uint32_t x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = w0 + 32 * i < words ? __ldg(m4 + w0 + 32 * i + lane) : 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (!__any_sync(0xffffffffu, x[i])) continue;
            int before = 0, tot = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t v = __ballot_sync(0xffffffffu, (x[i] >> (8 * b)) & 0xffu);
                before += __popc(v & below); tot += __popc(v);
            }
            int at = n + before;
            for (int b = 0; b < 4; ++b)
                if ((x[i] >> (8 * b)) & 0xffu) list[at++] = (uint16_t)((w0 + 32 * i + lane) * 4 + b);
            n += tot;
        }
        if (n < 512 && w0 + 128 < words) continue;
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            if (p + i >= capacity) break;
            const int k = list[i];
            ocol[p + i] = k;
            oval[p + i] = d2h(__dsub_rn((double)W[(int64_t)row * u.K + k], h2d(decode16(u, row, k))));
        }
        p += n;
        n = 0;
        __syncwarp();
    }
}

// ------------------------------------------------------------------ per-channel cosine

// A warp per channel, four weights per lane and step; fp64 sums.
__global__ void __launch_bounds__(256) cosine_kernel(const float* __restrict__ W, const uint8_t* __restrict__ mask,
                                                      Unpacked u, int rows, double* cosv) {
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= rows) return;
    const float4* w4 = (const float4*)(W + (int64_t)row * u.K);
    const uint32_t* i4 = (const uint32_t*)(u.idx + (int64_t)row * u.K);
    const uint8_t* mrow = mask ? mask + (int64_t)row * u.K : nullptr;
    const bool words = ((uintptr_t)mask & 3u) == 0;      // the public call takes a mask at any address
    double ab = 0.0, aa = 0.0, bb = 0.0;
#pragma unroll 4
    for (int q = lane; q < u.K / 4; q += 32) {
        const float4 w = __ldg(w4 + q);
        const uint32_t ix = __ldg(i4 + q);
        uint32_t x = 0;
        if (mrow) {
            if (words) x = __ldg((const uint32_t*)mrow + q);
            else for (int i = 0; i < 4; ++i) x |= (uint32_t)mrow[4 * q + i] << (8 * i);
        }
        const float f[4] = {w.x, w.y, w.z, w.w};
        const uint16_t* book = u.cb + (int64_t)row * u.E;
        uint16_t sc = 0, mid = 0;
        if (u.mode) {
            const int64_t g = (int64_t)row * u.G + q * 4 / u.group;      // four weights never straddle two groups
            book = u.cb + (int)u.gid[g] * u.E; sc = u.gscale[g]; mid = u.gmid[g];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint16_t e = __ldg(book + ((ix >> (8 * i)) & 0xffu));
            const double a = (double)f[i];
            double b = h2d(u.mode ? v2a_value16(sc, e, mid) : e);
            if ((x >> (8 * i)) & 0xffu) {
                const uint16_t s16 = d2h(__dsub_rn(a, b));           // the stored residual
                b = h2d(d2h(__dadd_rn(b, h2d(s16))));                // W^ = fp16(D16 + S), one rounding
            }
            ab = fma(a, b, ab); aa = fma(a, a, aa); bb = fma(b, b, bb);
        }
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        ab += __shfl_xor_sync(0xffffffffu, ab, d); aa += __shfl_xor_sync(0xffffffffu, aa, d); bb += __shfl_xor_sync(0xffffffffu, bb, d);
    }
    if (lane == 0)
        cosv[row] = (aa == 0.0 || bb == 0.0) ? 1.0 : __ddiv_rn(ab, __dmul_rn(__dsqrt_rn(aa), __dsqrt_rn(bb)));
}

// ------------------------------------------------------------------ host side

struct Workspace {
    double2* part;     // [kRedBlocks]
    SelState* sel;
    int* flags;        // [3] LibFit: did round i change a centroid
    int* tie;          // [ceil(n / kTieChunk)]
    int* rowcnt;       // [rows]
    double* u;         // [rows][64]
    double* nn;        // [rows]
    int* order;        // [rows]
    int* asg;          // [rows]
    double* cen;       // [256][64]
    size_t bytes;
};

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

static Workspace carve(void* base, int64_t rows, int64_t cols) {
    Workspace w;
    char* p = (char*)base;
    size_t o = 0;
    auto take = [&](size_t bytes) { char* r = p + o; o += align256(bytes); return r; };
    const int64_t n = rows * cols;
    w.part = (double2*)take(sizeof(double2) * kRedBlocks);
    w.sel = (SelState*)take(sizeof(SelState));
    w.flags = (int*)take(sizeof(int) * 3);
    w.tie = (int*)take(sizeof(int) * (size_t)((n + kTieChunk - 1) / kTieChunk + 1));
    w.rowcnt = (int*)take(sizeof(int) * (size_t)rows);
    w.u = (double*)take(sizeof(double) * (size_t)rows * 64);
    w.nn = (double*)take(sizeof(double) * (size_t)rows);
    w.order = (int*)take(sizeof(int) * (size_t)rows);
    w.asg = (int*)take(sizeof(int) * (size_t)rows);
    w.cen = (double*)take(sizeof(double) * 256 * 64);
    const size_t lloyd = lloyd_scratch_bytes((int)rows, (int)cols);   // the Lloyd kernel uses the scratch from its start
    if (o < lloyd) o = align256(lloyd);
    w.bytes = o;
    return w;
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

static int shape_status(int64_t rows, int64_t cols) {
    if (rows < 1 || cols < 128 || cols % 128 != 0) return XFP_ERR_SHAPE;
    if (cols > 65536 || rows > (1 << 24)) return XFP_ERR_UNSUPPORTED;
    return XFP_OK;
}

static Unpacked unpacked_of(const xfp_desc* d, const uint8_t* idx, const uint16_t* cb, const uint8_t* gid,
                            const uint16_t* gscale, const uint16_t* gmid) {
    Unpacked u;
    u.idx = idx; u.cb = cb; u.gid = gid; u.gscale = gscale; u.gmid = gmid;
    u.mode = d->mode; u.K = d->cols; u.E = 1 << d->bits; u.group = d->group_size; u.G = d->cols / d->group_size;
    return u;
}

static int desc_status(const xfp_desc* d) {
    if (!d) return XFP_ERR_NULL;
    if (d->mode != 0 && d->mode != 1) return XFP_ERR_SHAPE;
    if (d->bits < 2 || d->bits > 6) return XFP_ERR_SHAPE;
    if (d->group_size != 64 && d->group_size != 128 && d->group_size != 256)
        return d->group_size > 0 ? XFP_ERR_UNSUPPORTED : XFP_ERR_SHAPE;
    if (d->cols > 0 && d->cols % d->group_size) return XFP_ERR_SHAPE;
    if (d->mode == 1 && (d->lib_size < 1 || d->lib_size > 256)) return XFP_ERR_SHAPE;
    return shape_status(d->rows, d->cols);
}

// Extraction, first half: the candidates in `mask` (mode 0: above the threshold) and the plan of the selection.
static void outliers_candidates(const float* W, int64_t n, const double* ms, int mode, double k_or_rate, double cap_frac,
                                uint8_t* mask, int64_t* count, int64_t* skip_out, const Workspace& w, cudaStream_t s) {
    const int64_t nblk = (n + kTieChunk - 1) / kTieChunk, cap = (int64_t)xfp::sm_count() * 8;
    const int sweep = (int)(nblk < cap ? (nblk < 1 ? 1 : nblk) : cap);
    if (mode == 0) {
        outlier_zero<<<1, 1, 0, s>>>(w.sel);
        mask_threshold<<<sweep, 256, 0, s>>>(W, n, ms, k_or_rate, mask, w.sel);
        outlier_plan<<<1, 256, 0, s>>>(w.sel, n, 0, cap_frac, count, skip_out);
    } else {
        mask_clear<<<sweep, 256, 0, s>>>(mask, n);
        outlier_plan<<<1, 256, 0, s>>>(w.sel, n, 1, k_or_rate, count, skip_out);
    }
}
// Second half: the largest |w - mu| of the candidates, ties by position.  A no-op on the device where the plan says skip.
static cudaError_t outliers_select(const float* W, int64_t n, const double* ms, int mode, uint8_t* mask, const Workspace& w,
                                   cudaStream_t s) {
    const unsigned nblk = (unsigned)((n + kTieChunk - 1) / kTieChunk);
    const SrcAbsDev src{W, ms, mode == 0 ? mask : nullptr};
    const cudaError_t e = run_select(src, n, w.sel, s);
    if (e != cudaSuccess) return e;
    tie_count<SrcAbsDev><<<nblk, 256, 0, s>>>(src, n, w.sel, w.tie);
    tie_scan<<<1, 1024, 0, s>>>(w.tie, (int)nblk, w.sel);
    tie_apply<SrcAbsDev><<<nblk, 256, 0, s>>>(src, n, w.sel, w.tie, mask);
    return cudaGetLastError();
}

}  // namespace xq

using namespace xq;

extern "C" {

int xfp_quant_workspace_size(int32_t rows, int32_t cols, size_t* bytes) {
    if (!bytes) return XFP_ERR_NULL;
    const int st = shape_status(rows, cols);
    if (st) return st;
    *bytes = carve(nullptr, rows, cols).bytes;
    return XFP_OK;
}

int xfp_quant_stats(const float* W, int64_t n, int32_t sigma_mode, double* mu_sigma, void* workspace,
                    size_t workspace_bytes, void* stream) {
    if (!W || !mu_sigma || !workspace) return XFP_ERR_NULL;
    if (!aligned16(W) || !aligned16(mu_sigma) || !aligned16(workspace)) return XFP_ERR_ALIGN;
    if (n < 1 || (sigma_mode != 0 && sigma_mode != 1)) return XFP_ERR_SHAPE;
    if (workspace_bytes < carve(nullptr, 1, 128).bytes) return XFP_ERR_BUFFER_TOO_SMALL;
    cudaStream_t s = (cudaStream_t)stream;
    Workspace w = carve(workspace, 1, 128);
    stats_partial<<<kRedBlocks, kRedThreads, 0, s>>>(W, n, w.part);
    stats_final<<<1, kRedThreads, 0, s>>>(w.part, n, mu_sigma);
    if (sigma_mode == 1) {
        SrcAbsDev src{W, mu_sigma, nullptr};
        if (run_median(src, n, 1.4826, true, mu_sigma + 1, w.sel, s) != cudaSuccess) return XFP_ERR_CUDA;
    }
    return cudaGetLastError() == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quant_outliers(const float* W, int64_t n, const double* mu_sigma, int32_t outlier_mode, double k_or_rate,
                       double cap_frac, uint8_t* mask, int64_t* count, void* workspace, size_t workspace_bytes,
                       void* stream) {
    if (!W || !mu_sigma || !mask || !count || !workspace) return XFP_ERR_NULL;
    if (!aligned16(W) || !aligned16(mask) || !aligned16(workspace)) return XFP_ERR_ALIGN;
    if (n < 1 || (outlier_mode != 0 && outlier_mode != 1)) return XFP_ERR_SHAPE;
    if (!(k_or_rate >= 0.0) || (outlier_mode == 0 && !(cap_frac >= 0.0 && cap_frac <= 1.0)) ||
        (outlier_mode == 1 && k_or_rate > 1.0))
        return XFP_ERR_SHAPE;
    const int64_t nblk = (n + kTieChunk - 1) / kTieChunk;
    // the tie counters are the only part of the scratch that grows with n; they start where the smallest layout puts them
    const size_t tie_offset = (size_t)((char*)carve(nullptr, 1, 128).tie - (char*)nullptr);
    if (workspace_bytes < tie_offset + (size_t)nblk * sizeof(int)) return XFP_ERR_BUFFER_TOO_SMALL;
    cudaStream_t s = (cudaStream_t)stream;
    Workspace w = carve(workspace, 1, 128);   // part, sel, flags, then the tie counters
    outliers_candidates(W, n, mu_sigma, outlier_mode, k_or_rate, cap_frac, mask, count, nullptr, w, s);
    if (outliers_select(W, n, mu_sigma, outlier_mode, mask, w, s) != cudaSuccess) return XFP_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quant_lloyd(const float* W, const uint8_t* mask, const double* mu_sigma, int32_t rows, int32_t cols,
                    int32_t bits, int32_t iters, uint16_t* codebook, uint8_t* idx, void* workspace,
                    size_t workspace_bytes, void* stream) {
    if (!W || !mu_sigma || !codebook || !idx) return XFP_ERR_NULL;
    if (!aligned16(W) || !aligned16(codebook) || !aligned16(idx) || (mask && !aligned16(mask))) return XFP_ERR_ALIGN;
    const int st = shape_status(rows, cols);
    if (st) return st;
    if (bits < 2 || bits > 6 || iters < 0) return XFP_ERR_SHAPE;
    const size_t scratch = lloyd_scratch_bytes(rows, cols);
    if (scratch) {
        if (!workspace) return XFP_ERR_NULL;
        if (!aligned16(workspace)) return XFP_ERR_ALIGN;
        if (workspace_bytes < scratch) return XFP_ERR_BUFFER_TOO_SMALL;
    }
    return launch_lloyd(W, mask, mu_sigma, rows, cols, bits, iters, codebook, idx, nullptr, nullptr, workspace,
                        (cudaStream_t)stream) == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quant_libfit_library(const uint16_t* codebook, int32_t rows, int32_t bits, int32_t L, int32_t iters,
                             uint16_t* lib, void* workspace, size_t workspace_bytes, void* stream) {
    if (!codebook || !lib || !workspace) return XFP_ERR_NULL;
    if (!aligned16(codebook) || !aligned16(lib) || !aligned16(workspace)) return XFP_ERR_ALIGN;
    if (rows < 1 || bits < 2 || bits > 6 || L < 1 || L > 256 || iters < 0) return XFP_ERR_SHAPE;
    if (rows > (1 << 24)) return XFP_ERR_UNSUPPORTED;
    if (workspace_bytes < carve(nullptr, rows, 128).bytes) return XFP_ERR_BUFFER_TOO_SMALL;
    cudaStream_t s = (cudaStream_t)stream;
    Workspace w = carve(workspace, rows, 128);
    const int E = 1 << bits;
    return launch_libfit_library(codebook, rows, E, L, iters, w.u, w.nn, w.order, w.asg, w.cen, w.flags, lib, s) == cudaSuccess
               ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quant_libfit_assign(const float* W, const uint8_t* mask, const double* mu_sigma, int32_t rows, int32_t cols,
                            int32_t bits, int32_t L, int32_t group_size, const uint16_t* lib, uint8_t* idx, uint8_t* gid,
                            uint16_t* gscale, uint16_t* gmid, void* stream) {
    if (!W || !mu_sigma || !lib || !idx || !gid || !gscale || !gmid) return XFP_ERR_NULL;
    if (!aligned16(W) || !aligned16(lib) || !aligned16(idx) || !aligned16(gid) || !aligned16(gscale) ||
        !aligned16(gmid) || (mask && !aligned16(mask)))
        return XFP_ERR_ALIGN;
    const int st = shape_status(rows, cols);
    if (st) return st;
    if (bits < 2 || bits > 6 || L < 1 || L > 256) return XFP_ERR_SHAPE;
    if (group_size != 64 && group_size != 128 && group_size != 256) return group_size > 0 ? XFP_ERR_UNSUPPORTED : XFP_ERR_SHAPE;
    if (cols % group_size) return XFP_ERR_SHAPE;
    const int64_t groups = (int64_t)rows * (cols / group_size);
    if (groups > 0x7fffffff) return XFP_ERR_UNSUPPORTED;
    return launch_libfit_assign(W, mask, mu_sigma, rows, cols, bits, L, group_size, lib, idx, gid, gscale, gmid, nullptr,
                                (cudaStream_t)stream) == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

static int unpacked_args_status(const xfp_desc* desc, const float* W, const uint8_t* idx, const uint16_t* codebook,
                                const uint8_t* gid, const uint16_t* gscale, const uint16_t* gmid) {
    const int st = desc_status(desc);
    if (st) return st;
    if (!W || !idx || !codebook) return XFP_ERR_NULL;
    if (desc->mode == 1 && (!gid || !gscale || !gmid)) return XFP_ERR_NULL;
    if (!aligned16(W) || !aligned16(idx) || !aligned16(codebook)) return XFP_ERR_ALIGN;
    return XFP_OK;
}

int xfp_quant_residual(const xfp_desc* desc, const float* W, const uint8_t* mask, const uint8_t* idx,
                       const uint16_t* codebook, const uint8_t* gid, const uint16_t* gscale, const uint16_t* gmid,
                       int32_t* out_rowptr, int32_t* out_col, uint16_t* out_val, int64_t capacity, void* workspace,
                       size_t workspace_bytes, void* stream) {
    const int st = unpacked_args_status(desc, W, idx, codebook, gid, gscale, gmid);
    if (st) return st;
    if (!mask || !out_rowptr || !workspace || (capacity > 0 && (!out_col || !out_val))) return XFP_ERR_NULL;
    if (!aligned16(mask) || !aligned16(out_rowptr) || !aligned16(workspace)) return XFP_ERR_ALIGN;
    if (capacity < 0) return XFP_ERR_SHAPE;
    if (workspace_bytes < carve(nullptr, desc->rows, desc->cols).bytes) return XFP_ERR_BUFFER_TOO_SMALL;
    cudaStream_t s = (cudaStream_t)stream;
    Workspace w = carve(workspace, desc->rows, desc->cols);
    const unsigned grid = (unsigned)((desc->rows + 7) / 8);
    row_count_kernel<<<grid, 256, 0, s>>>(mask, desc->rows, desc->cols, w.rowcnt);
    rowptr_scan<<<1, 1024, 0, s>>>(w.rowcnt, desc->rows, out_rowptr);
    residual_kernel<<<grid, 256, 0, s>>>(W, mask, unpacked_of(desc, idx, codebook, gid, gscale, gmid), desc->rows, out_rowptr,
                                         out_col, out_val, capacity);
    return cudaGetLastError() == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quant_cosine(const xfp_desc* desc, const float* W, const uint8_t* mask, const uint8_t* idx,
                     const uint16_t* codebook, const uint8_t* gid, const uint16_t* gscale, const uint16_t* gmid,
                     double* cos, void* stream) {
    const int st = unpacked_args_status(desc, W, idx, codebook, gid, gscale, gmid);
    if (st) return st;
    if (!cos) return XFP_ERR_NULL;
    if (!aligned16(cos) || (mask && !aligned16(mask))) return XFP_ERR_ALIGN;
    cosine_kernel<<<(unsigned)((desc->rows + 7) / 8), 256, 0, (cudaStream_t)stream>>>(
        W, mask, unpacked_of(desc, idx, codebook, gid, gscale, gmid), desc->rows, cos);
    return cudaGetLastError() == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quant_median(const double* v, int64_t n, double* median, void* workspace, size_t workspace_bytes,
                     void* stream) {
    if (!v || !median || !workspace) return XFP_ERR_NULL;
    if (!aligned16(v) || !aligned16(workspace)) return XFP_ERR_ALIGN;
    if (n < 1) return XFP_ERR_SHAPE;
    if (workspace_bytes < carve(nullptr, 1, 128).bytes) return XFP_ERR_BUFFER_TOO_SMALL;
    if (n <= (1 << 16)) {
        median_small_kernel<<<1, 1024, 0, (cudaStream_t)stream>>>(v, (int)n, median, nullptr, nullptr);
        return cudaGetLastError() == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
    }
    Workspace w = carve(workspace, 1, 128);
    SrcDouble src{v};
    return run_median(src, n, 1.0, false, median, w.sel, (cudaStream_t)stream) == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

int xfp_quantize(int32_t mode, const float* W, int32_t rows, int32_t cols, const xfp_quant_params* p,
                 const int32_t* candidates, int32_t n_candidates, double tau, int32_t lib_size, uint8_t* mask,
                 uint8_t* idx, uint16_t* codebook, uint16_t* lib, uint8_t* gid, uint16_t* gscale, uint16_t* gmid,
                 int32_t* out_rowptr, int32_t* out_col, uint16_t* out_val, int64_t capacity, double* cos,
                 xfp_quant_result* result, void* workspace, size_t workspace_bytes, void* stream) {
    if (!W || !p || !candidates || !mask || !idx || !codebook || !out_rowptr || !cos || !result || !workspace)
        return XFP_ERR_NULL;
    if (mode != 0 && mode != 1) return XFP_ERR_SHAPE;
    if (mode == 1 && (!lib || !gid || !gscale || !gmid)) return XFP_ERR_NULL;
    if (n_candidates < 1 || n_candidates > 5) return XFP_ERR_SHAPE;
    for (int c = 0; c < n_candidates; ++c) {
        if (candidates[c] < 2 || candidates[c] > 6) return XFP_ERR_SHAPE;
        if (c && candidates[c] <= candidates[c - 1]) return XFP_ERR_SHAPE;
    }
    int st = shape_status(rows, cols);
    if (st) return st;
    size_t need;
    xfp_quant_workspace_size(rows, cols, &need);
    // mu, sigma, the median, the count and the extraction's plan live behind the carved scratch
    if (workspace_bytes < need + 256) return XFP_ERR_BUFFER_TOO_SMALL;
    // everything the stages below would refuse one by one: the kernels are launched past their entry points
    if (!aligned16(W) || !aligned16(mask) || !aligned16(workspace) || !aligned16(codebook) || !aligned16(idx) ||
        !aligned16(out_rowptr) || !aligned16(cos))
        return XFP_ERR_ALIGN;
    if (mode == 1 && (!aligned16(lib) || !aligned16(gid) || !aligned16(gscale) || !aligned16(gmid))) return XFP_ERR_ALIGN;
    if ((reinterpret_cast<uintptr_t>(out_col) & 3u) || (reinterpret_cast<uintptr_t>(out_val) & 1u)) return XFP_ERR_ALIGN;
    if (p->lloyd_iters < 0 || (p->outlier_mode != 0 && p->outlier_mode != 1) || (p->outlier_mode == 0 ? !(p->k_sigma >= 0.0) || !(p->cap_frac >= 0.0 && p->cap_frac <= 1.0)
                                                                              : !(p->rate >= 0.0 && p->rate <= 1.0)))
        return XFP_ERR_SHAPE;
    cudaStream_t s = (cudaStream_t)stream;
    struct Head { double mu, sigma, med, pad; int64_t count, skip; } host;
    Head* dev = (Head*)((char*)workspace + need);
    double* ms = &dev->mu;
    double* med_dev = &dev->med;
    const int64_t n = (int64_t)rows * cols;

    st = xfp_quant_stats(W, n, p->sigma_mode, ms, workspace, need, stream);
    if (st) return st;
    // One read-back tells the host the count and whether the cap (or a fixed rate) calls for a selection at all: the
    // selection is twenty small launches, 2 - 3 us each even where every one of them returns at once.
    const Workspace small = carve(workspace, 1, 128);
    outliers_candidates(W, n, ms, p->outlier_mode, p->outlier_mode ? p->rate : p->k_sigma, p->cap_frac, mask, &dev->count,
                        &dev->skip, small, s);
    if (cudaMemcpyAsync(&host, dev, sizeof(host), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return XFP_ERR_CUDA;
    if (!host.skip && outliers_select(W, n, ms, p->outlier_mode, mask, small, s) != cudaSuccess) return XFP_ERR_CUDA;
    const int64_t host_cnt = host.count;
    if (host_cnt > capacity) return XFP_ERR_BUFFER_TOO_SMALL;

    xfp_desc d;
    d.mode = mode; d.rows = rows; d.cols = cols; d.group_size = p->group_size ? p->group_size : 128;
    d.lib_size = mode ? lib_size : 0;
    if (d.group_size != 64 && d.group_size != 128 && d.group_size != 256) return d.group_size > 0 ? XFP_ERR_UNSUPPORTED : XFP_ERR_SHAPE;
    if (cols % d.group_size) return XFP_ERR_SHAPE;
    if (mode == 1 && (int64_t)rows * (cols / d.group_size) > 0x7fffffff) return XFP_ERR_UNSUPPORTED;
    d.col_bits = 32; d.nnz = host_cnt;
    result->mu = host.mu; result->sigma = host.sigma; result->nnz = host_cnt;
    result->fallback = 1; result->tried = 0; result->reserved = 0;
    if (mode == 1 && (lib_size < 1 || lib_size > 256)) return XFP_ERR_SHAPE;
    // What a channel's Lloyd block has at hand it also delivers: the count of its extracted weights and (V2) its cosine.
    // For V2a its indices are not wanted, LibFit assigns its own.
    const bool fused = lloyd_fuses_cosine(cols);
    int* rowcnt = carve(workspace, rows, cols).rowcnt;
    const unsigned rgrid = (unsigned)((rows + 7) / 8);
    if (!fused) {
        row_count_kernel<<<rgrid, 256, 0, s>>>(mask, rows, cols, rowcnt);
        rowptr_scan<<<1, 1024, 0, s>>>(rowcnt, rows, out_rowptr);
    }
    for (int c = 0; c < n_candidates; ++c) {
        d.bits = candidates[c];
        if (launch_lloyd(W, mask, ms, rows, cols, d.bits, p->lloyd_iters, codebook, mode ? nullptr : idx,
                         mode == 0 && fused ? cos : nullptr, c == 0 && fused ? rowcnt : nullptr, workspace, s) != cudaSuccess)
            return XFP_ERR_CUDA;
        const bool beside = mode == 0 && c == 0 && fused && rows <= (1 << 16);   // the row pointers beside the median (the library's scratch overlaps the counts)
        if (c == 0 && fused && !beside) rowptr_scan<<<1, 1024, 0, s>>>(rowcnt, rows, out_rowptr);
        if (mode == 1) {
            st = xfp_quant_libfit_library(codebook, rows, d.bits, lib_size, p->lloyd_iters, lib, workspace, need, stream);
            if (st) return st;
            if (launch_libfit_assign(W, mask, ms, rows, cols, d.bits, lib_size, d.group_size, lib, idx, gid, gscale, gmid, cos,
                                     s) != cudaSuccess)
                return XFP_ERR_CUDA;
        } else if (!fused) {
            st = xfp_quant_cosine(&d, W, mask, idx, codebook, nullptr, nullptr, nullptr, cos, stream);
            if (st) return st;
        }
        if (beside) median_small_kernel<<<2, 1024, 0, s>>>(cos, rows, med_dev, rowcnt, out_rowptr);
        else if ((st = xfp_quant_median(cos, rows, med_dev, workspace, need, stream))) return st;
        double med = 0.0;
        if (cudaMemcpyAsync(&med, med_dev, sizeof(med), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return XFP_ERR_CUDA;
        result->bits = d.bits;
        result->median_cos = med;
        result->tried = c + 1;
        if (med >= tau) { result->fallback = 0; break; }
    }
    if (capacity > 0 && (!out_col || !out_val)) return XFP_ERR_NULL;
    residual_kernel<<<rgrid, 256, 0, s>>>(W, mask, unpacked_of(&d, idx, mode ? lib : codebook, gid, gscale, gmid), rows,
                                          out_rowptr, out_col, out_val, capacity);
    return cudaGetLastError() == cudaSuccess ? XFP_OK : XFP_ERR_CUDA;
}

}  // extern "C"
