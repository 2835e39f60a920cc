// "Learned Codebook via Lloyd Iteration": one channel per block, the answer of the serial fp64 evaluation bit for bit.
//
// A channel's bulk values (extracted positions hold mu) are put in ascending order, prefix sums are taken in fp64, and every
// round turns 2^N - 1 boundaries into cell means by differences of prefix sums.  lloyd_kernel (channels of up to 16384
// weights) spends a few instructions per weight on that:
//
//   order     the kept weights are dealt to half as many equal-width buckets as there are weights (bounds from the
//             channel's mean and deviation), counted and placed with shared-memory atomics on packed 16-bit counters.
//             Nothing below needs the order inside a bucket except around zero and mu.  A channel whose fullest bucket
//             holds more than kMaxBucket weights (few distinct values) is sorted by a bitonic network instead.
//   prefix    a serial chain of K fp64 additions would be the longest phase.  Where no addition of the chain rounds, any
//             order gives its bits, and that is provable here: with A >= sum |v|, every float of magnitude >= T =
//             2^(ceil(log2 A) - 30) is a multiple of r = 2^(ceil(log2 A) - 53), and a sum of such values stays below
//             2^53 r.  So the values below -T are summed in parallel; the few values around zero and mu (and the run of
//             copies of mu itself) are sorted and added serially; the values above T are summed in parallel again if the
//             sum that the serial part left behind is a multiple of 2^-53 times a power of two above every later partial
//             sum (checked; else the channel is sorted and the chain goes on serially).  Kept: the sum in front of every
//             fourth position ("anchors"); a sum in between continues its anchor.
//   rounds    one warp, a lane per boundary: the sum in front of the boundary's bucket, and the bucket's members (two to
//             five) that are not above it.
//   indices   the nearest-entry rule is monotone in the weight, so every boundary between two stored entries is one
//             float threshold, found by evaluating the rule itself; a weight is placed by N comparisons.
//
// 12288 x 4096 weights, N = 4, 20 rounds, with the cosine, one launch on one B200: 2272 -> 514 us (300 of them without the
// rounds).  Bound by issue slots and by the barriers around the single warp of the rounds, seven blocks per SM.
#include "xfp_quant_common.cuh"
#include "xfp_quant_internal.h"
#include "xfp_internal.h"
#include "../../include/xfp_quant.h"

namespace xq {

namespace {

constexpr int kEpt = 32;            // weights per thread: a block of TH threads takes channels of up to 32 * TH weights
constexpr int kMaxBucket = 128;     // weights in one bucket beyond which the bitonic network is cheaper than looking through it
constexpr int kMid = 4;             // weights around zero and mu that are sorted for the serial part, per thread
constexpr int kShortCols = 16384;   // longest channel that is sorted in shared memory

// Monotone map of a weight to a bucket: one rounding of v * inv + off, clamped; the addition of 2^23 rounds to an integer.
struct Buckets {
    float inv, off, top;
    __device__ __forceinline__ int of(float v) const {
        const float f = fminf(fmaxf(fmaf(v, inv, off), 0.f), top);
        return __float_as_int(f + 8388608.f) & 0x7fffff;
    }
};

// r[0..K) ascending: a bitonic network in its all-ascending form (the first step of a merge compares mirrored
// positions), which tolerates any K: positions beyond it would hold +inf and never move.
__device__ void sort_bitonic(float* r, int K, int tid, int threads) {
    int p2 = 1;
    while (p2 < K) p2 <<= 1;
    for (int size = 2; size <= p2; size <<= 1) {
        const int h = size >> 1;
        for (int p = tid; p < (p2 >> 1); p += threads) {
            const int base = (p / h) * size, o = p & (h - 1), a = base + o, b = base + size - 1 - o;
            if (b < K) { const float x = r[a], y = r[b]; if (x > y) { r[a] = y; r[b] = x; } }
        }
        __syncthreads();
        for (int j = h >> 1; j; j >>= 1) {
            for (int p = tid; p < (p2 >> 1); p += threads) {
                const int a = ((p & ~(j - 1)) << 1) | (p & (j - 1)), b = a + j;
                if (b < K) { const float x = r[a], y = r[b]; if (x > y) { r[a] = y; r[b] = x; } }
            }
            __syncthreads();
        }
    }
}

// number of entries of r[lo, hi) with r <= x (ascending), plus lo
__device__ __forceinline__ int upper_bound(const float* r, int lo, int hi, float x) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (r[mid] <= x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The ordered channel: `r` the kept weights, m copies of mu behind the first p0 of them.
struct Channel {
    const float* r;
    const double* anchor;   // sum in front of position 4 i (mu's copies included once 4 i > p0)
    double p1;              // sum behind mu's copies
    int p0;
    // sum of the first cu kept weights, and of mu's copies when `incl` (then cu >= p0)
    __device__ __forceinline__ double prefix(int cu, bool incl) const {
        int u = cu & ~3;
        double run;
        if (incl && u <= p0) { u = p0; run = p1; } else run = anchor[u >> 2];
        for (; u < cu; ++u) run = __dadd_rn(run, (double)r[u]);
        return run;
    }
};

template <int TH>
__global__ void __launch_bounds__(TH, TH == 128 ? 7 : TH == 256 ? 3 : 2)
lloyd_kernel(const float* __restrict__ W, const uint8_t* __restrict__ mask, const double* __restrict__ ms, int K, int bits,
             int iters, int nb, uint16_t* __restrict__ cb16, uint8_t* __restrict__ idx, double* __restrict__ cosv,
             int* __restrict__ rowcnt) {
    constexpr int NW = TH / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    float* r = (float*)smem;                                    // [K]
    double* anchor = (double*)(smem + (size_t)K * 4);           // [K / 4 + 1], padded to K / 4 + 2
    uint32_t* cnt2 = (uint32_t*)(anchor + K / 4 + 2);           // [nb / 2] two 16-bit bucket counters a word
    __shared__ double s_red[3][NW];
    __shared__ float s_f[4][NW];
    __shared__ int s_i[NW];
    __shared__ double c[64], e16[64], val[65];
    __shared__ float thr[64];
    __shared__ int cut[65];
    __shared__ double s_p1, s_p2, s_s1, s_total;
    __shared__ int s_pos[3], s_shift, s_direct, s_mu_idx, s_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int E = 1 << bits;
    const double mu = ms[0];
    const int64_t row = blockIdx.x, row0 = row * K;
    const float4* w4 = (const float4*)(W + row0);
    const uint32_t* m4 = mask ? (const uint32_t*)(mask + row0) : nullptr;

    // ---- load; moments that bound the buckets and the sums (their own rounding decides nothing) ----
    float v[kEpt];
    float sum = 0.f, sq = 0.f, ab = 0.f, some = 0.f;
    int kept = 0;                                // in its upper half the extracted weights (the mask of xfp_quantize holds 0 and 1)
#pragma unroll
    for (int e = 0; e < kEpt / 4; ++e) {
        const int q = e * TH + tid;
        float4 w = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        uint32_t x = 0x01010101u;
        if (q * 4 < K) { w = __ldg(w4 + q); x = m4 ? __ldg(m4 + q) : 0u; kept += __popc(x) << 16; }
        v[4 * e] = (x & 0xffu) ? INFINITY : w.x; v[4 * e + 1] = (x & 0xff00u) ? INFINITY : w.y;
        v[4 * e + 2] = (x & 0xff0000u) ? INFINITY : w.z; v[4 * e + 3] = (x & 0xff000000u) ? INFINITY : w.w;
    }
    for (int i = tid; i < nb / 2; i += TH) cnt2[i] = 0u;
    // every weight for sum |v| and the count, every fourth for the mean and the deviation
#pragma unroll
    for (int e = 0; e < kEpt; ++e) {
        const bool ok = v[e] < INFINITY;
        const float x = ok ? v[e] : 0.f;
        kept += ok; ab += fabsf(x);
        if ((e & 3) == 0) { some += ok ? 1.f : 0.f; sum += x; sq = fmaf(x, x, sq); }
    }
    sum = warp_sum(sum); sq = warp_sum(sq); ab = warp_sum(ab); some = warp_sum(some);
    kept = __reduce_add_sync(0xffffffffu, kept);
    if (lane == 0) { s_f[0][warp] = sum; s_f[1][warp] = sq; s_f[2][warp] = ab; s_f[3][warp] = some; s_i[warp] = kept; }
    __syncthreads();
    sum = sq = ab = some = 0.f; kept = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) { sum += s_f[0][w]; sq += s_f[1][w]; ab += s_f[2][w]; some += s_f[3][w]; kept += s_i[w]; }
    // weights that are no finite numbers are counted as copies of mu with the extracted ones, but only these have a residual
    const int n = kept & 0xffff, m = K - n, extracted = kept >> 16;
    Buckets bk{0.f, 0.f, (float)(nb - 1)};
    {
        // 3.3 deviations either side of the mean: a bell-shaped channel then puts at most three or four weights in a bucket
        const float mean = sum / some, half = 3.3f * sqrtf(fmaxf(sq / some - mean * mean, 0.f));
        const float lo = mean - half, hi = mean + half, inv = (float)(nb - 1) / (hi - lo);
        if (hi > lo && inv < 1e30f && fabsf(lo * inv) < 1e30f) { bk.inv = inv; bk.off = -lo * inv; }
    }

    // ---- sort ----
#pragma unroll
    for (int e = 0; e < kEpt; ++e)
        if (v[e] < INFINITY) { const int b = bk.of(v[e]); atomicAdd(&cnt2[b >> 1], 1u << ((b & 1) * 16)); }
    __syncthreads();
    int full = 0;
    {
        const int nq = nb / (8 * TH);           // 16-byte vectors (eight counters each) of this thread's share
        uint4* mine = (uint4*)cnt2 + (size_t)tid * nq;
        int tot = 0;
        for (int i = 0; i < nq; ++i) {
            const uint4 t = mine[i];
            const uint32_t u[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int a = (int)(u[k] & 0xffffu), b = (int)(u[k] >> 16);
                tot += a + b;
                full |= (a > kMaxBucket) | (b > kMaxBucket);
            }
        }
        int inc = tot;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= d) inc += t;
        }
        if (lane == 31) s_i[warp] = inc;
        full = __syncthreads_or(full);
        int run = inc - tot;
        for (int w = 0; w < warp; ++w) run += s_i[w];
        for (int i = 0; i < nq; ++i) {           // starts of the buckets in place of their counts
            const uint4 t = mine[i];
            uint32_t u[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t a = u[k] & 0xffffu, b = u[k] >> 16;
                u[k] = (uint32_t)run | ((uint32_t)(run + (int)a) << 16);
                run += (int)(a + b);
            }
            mine[i] = make_uint4(u[0], u[1], u[2], u[3]);
        }
    }
    __syncthreads();
    const uint16_t* ends = (const uint16_t*)cnt2;   // after the placement: bucket b holds positions [ends[b - 1], ends[b])
    const double A = (double)ab * 1.01 + (double)m * fabs(mu);
    const int eA = A > 0.0 ? ilogb(A) + 1 : -1000;
    // the values that are added serially lie in [low, high]: zero within T, and mu
    const double T = ldexp(1.0, eA - 30), low = fmin(-T, mu), high = fmax(T, mu);
    int q0 = 0, q1 = nb - 1;         // buckets whose members are in ascending order (all of them when `sorted`)
    bool sorted = full != 0;
    if (!sorted) {
#pragma unroll
        for (int e = 0; e < kEpt; ++e)
            if (v[e] < INFINITY) {
                const int b = bk.of(v[e]), sh = (b & 1) * 16;
                const uint32_t old = atomicAdd(&cnt2[b >> 1], 1u << sh);
                r[(old >> sh) & 0xffffu] = v[e];
            }
        q0 = bk.of(__double2float_rd(low)); q1 = bk.of(__double2float_ru(high));
        __syncthreads();
        // sort the buckets around zero and mu: a weight counts the smaller members of its own bucket
        const int t0 = q0 ? ends[q0 - 1] : 0, t1 = ends[q1];
        sorted = t1 - t0 > kMid * TH;
        if (!sorted) {
            float x[kMid];
            int to[kMid];
#pragma unroll
            for (int e = 0; e < kMid; ++e) {
                const int t = t0 + e * TH + tid;
                to[e] = -1;
                if (t < t1) {
                    x[e] = r[t];
                    const int b = bk.of(x[e]), b0 = b ? ends[b - 1] : 0, b1 = ends[b];
                    to[e] = b0;
                    for (int u = b0; u < b1; ++u) { const float y = r[u]; to[e] += (y < x[e]) || (y == x[e] && u < t); }
                }
            }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < kMid; ++e)
                if (to[e] >= 0) r[to[e]] = x[e];
        } else {
            sort_bitonic(r, n, tid, TH);
        }
    } else {
        if (tid == 0) s_n = 0;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < kEpt; ++e)
            if (v[e] < INFINITY) r[atomicAdd(&s_n, 1)] = v[e];
        __syncthreads();
        sort_bitonic(r, n, tid, TH);
    }
    __syncthreads();

    // ---- prefix sums (see the head of this file) ----
    if (warp == 0 && lane < 3) {
        const double x = lane == 0 ? low : lane == 1 ? high : mu;
        int lo = 0, hi = n;
        if (!sorted) { lo = q0 ? ends[q0 - 1] : 0; hi = ends[q1]; }
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const double y = (double)r[mid];
            if (lane == 0 ? y < x : y <= x) lo = mid + 1; else hi = mid;
        }
        s_pos[lane] = lo;
    }
    __syncthreads();
    const int pa = s_pos[0], pb = s_pos[1], p0 = s_pos[2];
    {
        // sums over chunks of four weights; every value that takes part is a multiple of r and no partial sum reaches 2^53 r
        double ex[kEpt / 4], carry = 0.0;
        const int w0 = warp * (kEpt / 4) * 32;
#pragma unroll
        for (int e = 0; e < kEpt / 4; ++e) {
            const int q = w0 + e * 32 + lane, u = q * 4;
            double s = 0.0;
            if (u < n) {
                const float4 f = *(const float4*)(r + u);
                const bool edge = u + 4 > n || (u + 4 > pa && u < pb);
                if (!edge) {
                    s = ((double)f.x + (double)f.y) + ((double)f.z + (double)f.w);
                } else {
                    const float g[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (u + i < n && (u + i < pa || u + i >= pb)) s += (double)g[i];
                }
            }
            double inc = s;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const double t = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += t;
            }
            ex[e] = carry + (inc - s);
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) s_red[0][warp] = carry;
        __syncthreads();
        double base = 0.0, total = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) { if (w < warp) base += s_red[0][w]; total += s_red[0][w]; }
#pragma unroll
        for (int e = 0; e < kEpt / 4; ++e) {
            const int q = w0 + e * 32 + lane;
            if (q <= K / 4) anchor[q] = base + ex[e];
        }
        if (tid == 0 && n == K && K == kEpt * TH) anchor[K / 4] = total;   // the one anchor no lane owns
        __syncthreads();
        // the chain over positions [u, end) in ascending order, mu's copies behind position p0
        auto chain = [&](int u, int end, double run) {
            for (;; ++u) {
                if ((u & 3) == 0) anchor[u >> 2] = run;
                if (u == p0) {
                    for (int i = 0; i < m; ++i) run = __dadd_rn(run, mu);
                    s_p1 = run;
                }
                if (u >= end) return run;
                run = __dadd_rn(run, (double)r[u]);
            }
        };
        if (tid == 0) {
            double s1 = anchor[pa >> 2];
            for (int u = pa & ~3; u < pa; ++u) s1 += (double)r[u];
            const double run = chain(pa, pb, s1);
            const double end = run + (total - s1), big = fmax(fabs(run), fabs(end));
            bool direct = true;
            if (big > 0.0) {
                const int k = ilogb(big) + 1;     // no later partial sum reaches 2^k
                const double x = ldexp(run, 53 - k);
                direct = k <= eA && x == rint(x);
            }
            s_s1 = s1; s_p2 = run; s_total = end; s_direct = direct;
        }
        // meanwhile the other warps find the start of the rounds, the (j + 1/2) / 2^N quantiles: P threads to a quantile,
        // each ranks its share of the quantile's bucket
        {
            int P = 1;
            while (2 * P * E <= TH - 32) P *= 2;
            for (int i = tid - 32; i >= 0 && i < E * P; i += TH - 32) {
                const int j = i / P, sub = i % P;
                long long q = (long long)floor(__ddiv_rn(__dmul_rn(__dadd_rn((double)j, 0.5), (double)K), (double)E));
                if (q >= K) q = K - 1;
                int t = (int)q;
                if (t >= p0 && t < p0 + m) { c[j] = mu; continue; }
                if (t >= p0 + m) t -= m;
                if (sorted) { c[j] = (double)r[t]; continue; }
                int lo = 0, hi = nb - 1;          // the bucket of position t
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (ends[mid] > t) hi = mid; else lo = mid + 1;
                }
                const int b0 = lo ? ends[lo - 1] : 0, b1 = ends[lo];
                for (int a = b0 + sub; a < b1; a += P) {
                    const float y = r[a];
                    int less = 0, same = 0;
                    for (int u = b0; u < b1; ++u) { less += r[u] < y; same += r[u] == y; }
                    if (t - b0 >= less && t - b0 < less + same) c[j] = (double)y;
                }
            }
        }
        __syncthreads();
        if (!s_direct) {          // an addition behind mu may round: sort everything and run the whole chain
            if (!sorted) sort_bitonic(r, n, tid, TH);
            sorted = true;
            if (tid == 0) s_total = chain(0, n, 0.0);
        } else {
            const double s1 = s_s1, p2 = s_p2;
#pragma unroll
            for (int e = 0; e < kEpt / 4; ++e) {
                const int q = w0 + e * 32 + lane;
                if (q * 4 > pb && q <= K / 4) anchor[q] = p2 + ((base + ex[e]) - s1);
            }
            if (tid == 0 && n == K && K == kEpt * TH && K > pb) anchor[K / 4] = s_total;
        }
    }
    __syncthreads();

    // ---- rounds: one warp, a lane per boundary and entry ----
    if (warp == 0) {
        const Channel ch{r, anchor, s_p1, p0};
        const double total = s_total;
        constexpr int kWin = 16;        // weights from the boundary's anchor on that are looked at without a loop
        // count of the values <= b and their sum in the chain's order
        auto below = [&](double b, int& cu, double& sum_b) {
            const float bf = __double2float_rd(b);       // a float is <= b when it is <= bf
            const bool incl = mu <= b;
            int lo = 0, hi = n;
            bool look = sorted;
            if (!sorted) {
                const int q = bk.of(bf);
                lo = q ? ends[q - 1] : 0; hi = ends[q];
                look = q >= q0 && q <= q1;
            }
            const int u0 = lo & ~3;
            if (look) {
                lo = upper_bound(r, lo, hi, bf);
                sum_b = ch.prefix(lo, incl);
            } else if (hi <= u0 + kWin && (!incl || (u0 >= pb && u0 > p0))) {     // no addition rounds here, whatever the order
                double part[4] = {anchor[u0 >> 2], 0.0, 0.0, 0.0};
                int in = 0;
#pragma unroll
                for (int i = 0; i < kWin / 4; ++i) {
                    // the window may reach past the channel (into the anchors behind it): masked by `hi`
                    const float4 f4 = *(const float4*)(r + u0 + 4 * i);
                    const float f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int u = u0 + 4 * i + k;
                        const bool take = u < lo || (u < hi && f[k] <= bf);
                        in += take;
                        part[k] += (double)(take ? f[k] : 0.f);
                    }
                }
                sum_b = (part[0] + part[1]) + (part[2] + part[3]);
                lo = u0 + in;
            } else {
                sum_b = ch.prefix(lo, incl);
                const int b0 = lo;
                for (int u = b0; u < hi; ++u) { const float y = r[u]; if (y <= bf) { sum_b += (double)y; ++lo; } }
            }
            cu = lo + (incl ? m : 0);
        };
        // cell j = (b_{j-1}, b_j], b_j the midpoint of entries j and j+1: a lane's cell ends where its boundary lies
        if (E <= 32) {
            double cj = c[lane < E ? lane : E - 1];
            for (int it = 0; it < iters; ++it) {
                const double cn = __shfl_down_sync(0xffffffffu, cj, 1);
                int cu = K;
                double sum_b = total;
                if (lane < E - 1) below(__dmul_rn(0.5, __dadd_rn(cj, cn)), cu, sum_b);
                __syncwarp();
                int c0 = __shfl_up_sync(0xffffffffu, cu, 1);
                double v0 = __shfl_up_sync(0xffffffffu, sum_b, 1);
                if (lane == 0) { c0 = 0; v0 = 0.0; }
                bool changed = false;
                if (lane < E && cu > c0) {
                    const double mean = __ddiv_rn(__dsub_rn(sum_b, v0), (double)(cu - c0));
                    changed = mean != cj;
                    cj = mean;
                }
                if (!__any_sync(0xffffffffu, changed)) break;
            }
            if (lane < E) c[lane] = cj;
        } else {
            if (lane == 0) { cut[0] = 0; val[0] = 0.0; cut[E] = K; val[E] = total; }
            for (int it = 0; it < iters; ++it) {
                for (int j = lane; j < E - 1; j += 32) below(__dmul_rn(0.5, __dadd_rn(c[j], c[j + 1])), cut[j + 1], val[j + 1]);
                __syncwarp();
                bool changed = false;
                for (int j = lane; j < E; j += 32) {
                    if (cut[j + 1] > cut[j]) {
                        const double mean = __ddiv_rn(__dsub_rn(val[j + 1], val[j]), (double)(cut[j + 1] - cut[j]));
                        if (mean != c[j]) { c[j] = mean; changed = true; }
                    }
                }
                if (!__any_sync(0xffffffffu, changed)) break;
                __syncwarp();
            }
        }
        __syncwarp();
        for (int j = lane; j < E; j += 32) {
            const uint16_t h = d2h(c[j]);
            cb16[row * E + j] = h;
            e16[j] = h2d(h);
        }
        __syncwarp();
        bool bad = false;
        for (int j = lane; j < E; j += 32) {
            thr[j] = INFINITY;
            if (j < E - 1) {
                if (e16[j] < e16[j + 1]) thr[j] = last_of_lower(e16[j], e16[j + 1]);
                else bad = true;              // equal (or, by a rounding, descending) entries: the rule itself below
            }
        }
        bad = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            s_direct = !bad;
            bool asc = true;
            for (int j = 1; j < E && bad; ++j) asc = asc && e16[j] >= e16[j - 1];
            s_shift = asc;
            s_mu_idx = m ? nearest_entry(e16, E, mu, asc) : 0;
            if (rowcnt) rowcnt[row] = extracted;
        }
    }
    __syncthreads();

    // ---- every weight to the nearest STORED entry (ties: lower index); the cosine of the reconstruction on the way ----
    if (!idx) return;               // V2a: only the codebooks are wanted
    const bool by_thr = s_direct != 0, asc = s_shift != 0;
    double sab = 0.0, saa = 0.0, sbb = 0.0;
    uint32_t* out4 = (uint32_t*)(idx + row0);
#pragma unroll 2
    for (int q = tid; q * 4 < K; q += TH) {
        const float4 w = __ldg(w4 + q);
        const uint32_t x = m4 ? __ldg(m4 + q) : 0u;
        const float f[4] = {w.x, w.y, w.z, w.w};
        int at[4] = {0, 0, 0, 0};
        if (by_thr) {
            for (int step = E >> 1; step; step >>= 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) at[i] += f[i] > thr[at[i] + step - 1] ? step : 0;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) at[i] = nearest_entry(e16, E, (double)f[i], asc);
        }
        uint32_t o = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool ext = (x >> (8 * i)) & 0xffu;
            if (ext) at[i] = s_mu_idx;
            o |= (uint32_t)at[i] << (8 * i);
            if (cosv) {
                const double a = (double)f[i];
                double b = e16[at[i]];
                if (ext) b = h2d(d2h(__dadd_rn(b, h2d(d2h(__dsub_rn(a, b))))));   // W^ = fp16(D16 + S), S the stored residual
                sab = fma(a, b, sab); saa = fma(a, a, saa); sbb = fma(b, b, sbb);
            }
        }
        out4[q] = o;
    }
    if (cosv) {
        sab = warp_sum(sab); saa = warp_sum(saa); sbb = warp_sum(sbb);
        if (lane == 0) { s_red[0][warp] = sab; s_red[1][warp] = saa; s_red[2][warp] = sbb; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < NW; ++w) { sab += s_red[0][w]; saa += s_red[1][w]; sbb += s_red[2][w]; }
            cosv[row] = (saa == 0.0 || sbb == 0.0) ? 1.0 : __ddiv_rn(sab, __dmul_rn(__dsqrt_rn(saa), __dsqrt_rn(sbb)));
        }
    }
}

// ------------------------------------------------------------------ channels too long for shared memory

constexpr int kLongThreads = 256;

// Compare-exchange of the bitonic network: after it a <= b when `asc`, a >= b otherwise; equal keys stay put.
__device__ __forceinline__ void cswap(float& a, float& b, bool asc) {
    const bool sw = (a > b) == asc;
    const float x = sw ? b : a, y = sw ? a : b;
    a = x;
    b = y;
}
// the stages with partner distance 4, 2, 1 on eight consecutive elements
__device__ __forceinline__ void last3(float (&v)[8], bool asc) {
    cswap(v[0], v[4], asc); cswap(v[1], v[5], asc); cswap(v[2], v[6], asc); cswap(v[3], v[7], asc);
    cswap(v[0], v[2], asc); cswap(v[1], v[3], asc); cswap(v[4], v[6], asc); cswap(v[5], v[7], asc);
    cswap(v[0], v[1], asc); cswap(v[2], v[3], asc); cswap(v[4], v[5], asc); cswap(v[6], v[7], asc);
}
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
    const float4 a = *(const float4*)p, b = *(const float4*)(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
    *(float4*)p = make_float4(v[0], v[1], v[2], v[3]);
    *(float4*)(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}

// The channel's bulk values in ascending order without storing them as doubles: the weights that were not
// extracted, sorted as floats, with the m copies of mu (one per extracted position) inserted at p0.
struct SortedBulk {
    const float* r;
    int p0, m;
    double mu;
    __device__ __forceinline__ double at(int t) const {   // one load, then a select: no branch
        const int u = t < p0 ? t : (t - m > 0 ? t - m : 0);
        const double v = (double)r[u];
        return (t >= p0 && t < p0 + m) ? mu : v;
    }
};

// Channels beyond kShortCols weights: the two arrays live in a slice of global scratch owned by the block (L1/L2 resident;
// the block's own writes are ordered by its barriers) and the resident blocks walk the channels; any length the format
// allows.  Bitonic sort, serial prefix sum, boundaries by a many-way search.
__global__ void __launch_bounds__(kLongThreads, 4) lloyd_long_kernel(const float* __restrict__ W,
                                                               const uint8_t* __restrict__ mask,
                                                               const double* __restrict__ ms, int rows, int K, int Kp2,
                                                               int bits, int iters, uint16_t* __restrict__ cb16,
                                                               uint8_t* __restrict__ idx, double* scratch,
                                                               size_t slice_doubles) {
    double* base = scratch + (size_t)blockIdx.x * slice_doubles;
    double* pre = base;                      // [K + 1] serial prefix sums of the sorted bulk values
    float* r = (float*)(base + ((K + 2) & ~1));   // [Kp2] kept weights, ascending (extracted slots and padding = +inf); 16-byte aligned
    __shared__ double c[64];
    __shared__ double e16[64];
    __shared__ int cut[65];
    __shared__ int s_m, s_p0;
    const int tid = threadIdx.x;
    const int E = 1 << bits;
    const double mu = ms[0];

#pragma unroll 1
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
    const int64_t row0 = (int64_t)row * K;
    if (tid == 0) s_m = 0;
    __syncthreads();
    int extracted = 0;
    for (int kb = tid; kb < Kp2; kb += 8 * kLongThreads) {   // eight loads in flight per thread
        float v[8];
        uint8_t x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = kb + e * kLongThreads;
            v[e] = k < K ? W[row0 + k] : INFINITY;
            x[e] = (k < K && mask != nullptr) ? mask[row0 + k] : (uint8_t)0;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = kb + e * kLongThreads;
            if (k < Kp2) r[k] = x[e] ? INFINITY : v[e];
            extracted += x[e] != 0;
        }
    }
    if (extracted) atomicAdd(&s_m, extracted);
    __syncthreads();
    // bitonic sort, ascending.  The stages with partner distance 4, 2, 1 stay inside blocks of 8 consecutive
    // elements and run in registers (one pass per step instead of three trips through the array); the wider
    // stages go through the array, a thread's eight pairs loaded before any is written back.
    const int half = Kp2 >> 1, nblk8 = Kp2 >> 3;
    for (int b8 = tid; b8 < nblk8; b8 += kLongThreads) {   // steps 2, 4 and 8 entirely in registers
        float v[8];
        load8(r + 8 * b8, v);
        cswap(v[0], v[1], true); cswap(v[2], v[3], false); cswap(v[4], v[5], true); cswap(v[6], v[7], false);
        cswap(v[0], v[2], true); cswap(v[1], v[3], true); cswap(v[4], v[6], false); cswap(v[5], v[7], false);
        cswap(v[0], v[1], true); cswap(v[2], v[3], true); cswap(v[4], v[5], false); cswap(v[6], v[7], false);
        last3(v, ((8 * b8) & 8) == 0);
        store8(r + 8 * b8, v);
    }
    __syncthreads();
    for (int size = 16; size <= Kp2; size <<= 1) {
        for (int j = size >> 1; j >= 8; j >>= 1) {
            for (int pb = tid; pb < half; pb += 8 * kLongThreads) {
                int ia[8];
                float a[8], b[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int p = pb + e * kLongThreads;
                    ia[e] = p < half ? (((p & ~(j - 1)) << 1) | (p & (j - 1))) : -1;
                    if (ia[e] >= 0) { a[e] = r[ia[e]]; b[e] = r[ia[e] + j]; }
                }
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (ia[e] >= 0 && (a[e] > b[e]) == ((ia[e] & size) == 0)) { r[ia[e]] = b[e]; r[ia[e] + j] = a[e]; }
            }
            __syncthreads();
        }
        for (int b8 = tid; b8 < nblk8; b8 += kLongThreads) {
            float v[8];
            load8(r + 8 * b8, v);
            last3(v, ((8 * b8) & size) == 0);
            store8(r + 8 * b8, v);
        }
        __syncthreads();
    }
    if (tid == 0) {   // where mu sits among the kept weights
        int lo = 0, hi = K - s_m;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((double)r[mid] <= mu) lo = mid + 1; else hi = mid;
        }
        s_p0 = lo;
    }
    __syncthreads();
    SortedBulk s{r, s_p0, s_m, mu};
    // serial prefix sums: cell sums below are differences of these, as in a one-pass CPU evaluation.
    // All threads first lay the sorted values out as doubles in pre[1..K]; one thread then scans in place,
    // fetching the next eight values before it starts the current chain of eight dependent adds.
    for (int t = tid; t < K; t += kLongThreads) pre[t + 1] = s.at(t);
    __syncthreads();
    if (tid == 0) {
        double run = 0.0;
        double f[8], g[8];
        pre[0] = 0.0;
#pragma unroll
        for (int e = 0; e < 8; ++e) f[e] = pre[1 + e];
        for (int t = 0; t < K; t += 8) {   // K is a multiple of 128
            if (t + 8 < K) {
#pragma unroll
                for (int e = 0; e < 8; ++e) g[e] = pre[t + 9 + e];
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                run = __dadd_rn(run, f[e]);
                f[e] = run;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) pre[t + 1 + e] = f[e];
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = g[e];
        }
    }
    if (tid >= 32 && tid < 32 + E) {   // a warp other than the one that runs the prefix
        const int j = tid - 32;
        long long q = (long long)floor(__ddiv_rn(__dmul_rn(__dadd_rn((double)j, 0.5), (double)K), (double)E));
        if (q >= K) q = K - 1;
        c[j] = s.at((int)q);
    }
    if (tid == 32) { cut[0] = 0; cut[E] = K; }
    __syncthreads();

    // P lanes share one boundary search (P = 256 / 2^N, at most a warp): each round probes P positions of
    // the remaining range at once, so 4096 values take three rounds at N = 4 instead of twelve steps.
    const int P = (kLongThreads >> bits) > 32 ? 32 : (kLongThreads >> bits);
    const int jb = tid / P, sub = tid % P;
    const unsigned gmask = (P == 32 ? 0xffffffffu : ((1u << P) - 1u)) << ((tid & 31) & ~(P - 1));
    for (int it = 0; it < iters; ++it) {
        // cell j = (b_{j-1}, b_j], b_j the midpoint of entries j and j+1: cut[j+1] = #{t : s[t] <= b_j}
        {
            const bool mine = jb < E - 1;
            const double b = mine ? __dmul_rn(0.5, __dadd_rn(c[jb], c[jb + 1])) : 0.0;
            int lo = 0, hi = mine ? K : 0;   // every t < lo has s[t] <= b, every t >= hi has s[t] > b
            while (__any_sync(0xffffffffu, lo < hi)) {
                const int step = (hi - lo + P - 1) / P;
                const int pos = lo + (sub + 1) * step - 1;
                const bool below = lo < hi && pos < hi && s.at(pos) <= b;
                const int cnt = __popc(__ballot_sync(0xffffffffu, below) & gmask);   // the probes are ordered
                if (lo < hi) {
                    const int nlo = lo + cnt * step;
                    const int nhi = cnt < P ? lo + (cnt + 1) * step - 1 : hi;
                    lo = nlo < hi ? nlo : hi;
                    hi = nhi < hi ? nhi : hi;
                    if (hi < lo) hi = lo;
                }
            }
            if (mine && sub == 0) cut[jb + 1] = lo;
        }
        __syncthreads();
        int changed = 0;
        if (tid < E) {
            const int n = cut[tid + 1] - cut[tid];
            if (n > 0) {
                const double mean = __ddiv_rn(__dsub_rn(pre[cut[tid + 1]], pre[cut[tid]]), (double)n);
                if (mean != c[tid]) { c[tid] = mean; changed = 1; }
            }
        }
        if (!__syncthreads_or(changed)) break;
    }
    if (tid < E) {
        const uint16_t h = d2h(c[tid]);
        cb16[(int64_t)row * E + tid] = h;
        e16[tid] = h2d(h);
    }
    __syncthreads();
    // every weight goes to the nearest STORED entry (ties: lower index), four weights per thread at a time.  Up to
    // 16 entries the plain scan with four chains of compares in flight is the faster form; above, bisection.
    bool e_asc = E > 16;
    for (int j = 1; j < E && e_asc; ++j) e_asc = e16[j] >= e16[j - 1];
    for (int kb = tid; kb < K; kb += 4 * kLongThreads) {
        double v[4], bd[4];
        int best[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = kb + e * kLongThreads;
            v[e] = k < K ? bulk_value(W, mask, row0 + k, mu) : 0.0;
        }
        if (e_asc) {
#pragma unroll
            for (int e = 0; e < 4; ++e) best[e] = nearest_entry(e16, E, v[e], true);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) { bd[e] = fabs(__dsub_rn(v[e], e16[0])); best[e] = 0; }
            for (int j = 1; j < E; ++j) {
                const double ej = e16[j];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const double d = fabs(__dsub_rn(v[e], ej));
                    if (d < bd[e]) { bd[e] = d; best[e] = j; }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = kb + e * kLongThreads;
            if (k < K && idx) idx[row0 + k] = (uint8_t)best[e];
        }
    }
    __syncthreads();   // the arrays and the small tables are reused by the CTA's next channel
    }
}

size_t long_slice_doubles(int cols, int* kp2_out) {
    int kp2 = 1;
    while (kp2 < cols) kp2 <<= 1;
    *kp2_out = kp2;
    return (((size_t)cols + 2) & ~(size_t)1) + (size_t)kp2 / 2;
}

template <int TH>
cudaError_t launch_short(const float* W, const uint8_t* mask, const double* ms, int rows, int cols, int bits, int iters,
                         uint16_t* codebook, uint8_t* idx, double* cosv, int* rowcnt, cudaStream_t s) {
    int nb = 8 * TH;                                   // a counter per two weights, at least the scan's vectors
    while (nb < cols / 2) nb <<= 1;
    const size_t smem = (size_t)cols * 4 + ((size_t)cols / 4 + 2) * 8 + (size_t)nb * 2;
    static xfp::DeviceOnce done;
    const int dev = xfp::DeviceOnce::current();
    if (!done.is_set(dev)) {
        cudaError_t e = cudaFuncSetAttribute(lloyd_kernel<TH>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024 + 256);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(lloyd_kernel<TH>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        done.set(dev);
    }
    lloyd_kernel<TH><<<rows, TH, smem, s>>>(W, mask, ms, cols, bits, iters, nb, codebook, idx, cosv, rowcnt);
    return cudaGetLastError();
}

}  // namespace

bool lloyd_fuses_cosine(int cols) { return cols <= kShortCols; }

// long channels: two resident blocks on each of kSizingSMs SMs at most, each with a slice for its two arrays
size_t lloyd_scratch_bytes(int rows, int cols) {
    if (cols <= kShortCols) return 0;
    int kp2;
    const size_t slice = long_slice_doubles(cols, &kp2);
    return slice * sizeof(double) * (size_t)(rows < 2 * xfp::kSizingSMs ? rows : 2 * xfp::kSizingSMs);
}

cudaError_t launch_lloyd(const float* W, const uint8_t* mask, const double* ms, int rows, int cols, int bits, int iters,
                         uint16_t* codebook, uint8_t* idx, double* cosv, int* rowcnt, void* scratch, cudaStream_t s) {
    if (cols <= 128 * kEpt) return launch_short<128>(W, mask, ms, rows, cols, bits, iters, codebook, idx, cosv, rowcnt, s);
    if (cols <= 256 * kEpt) return launch_short<256>(W, mask, ms, rows, cols, bits, iters, codebook, idx, cosv, rowcnt, s);
    if (cols <= kShortCols) return launch_short<512>(W, mask, ms, rows, cols, bits, iters, codebook, idx, cosv, rowcnt, s);
    int kp2;
    const size_t slice = long_slice_doubles(cols, &kp2);
    const int want = 2 * xfp::sched_sms();
    lloyd_long_kernel<<<rows < want ? rows : want, kLongThreads, 0, s>>>(W, mask, ms, rows, cols, kp2, bits, iters, codebook,
                                                                         idx, (double*)scratch, slice);
    return cudaGetLastError();
}

}  // namespace xq
