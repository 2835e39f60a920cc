// LibFit ("V2a: Shared Codebook Library"): the library (a k-means pass over normalised per-channel codebooks) and the
// assignment of every group of weights to a library entry.  Integers and fp16 values are those of the serial fp64
// evaluation, bit for bit.
#include <cooperative_groups.h>

#include <atomic>

#include "xfp_quant_common.cuh"
#include "xfp_quant_internal.h"
#include "xfp_internal.h"
#include "../../include/xfp_quant.h"

namespace xq {

namespace {

namespace cg = cooperative_groups;

// ------------------------------------------------------------------ the library

constexpr int kLibThreads = 512;
constexpr int kLibTile = 4096;      // channels whose members are compacted at a time
constexpr int kLibVals = 2048;      // member values staged at a time
constexpr size_t kLibSmemU = 160 * 1024;   // normalised codebooks of this size stay in every block's shared memory

// u_j = (c_j - m) / s, m and s the middle and half-width of the codebook's range; returns |u|^2
__device__ __forceinline__ double normalise_channel(const uint16_t* __restrict__ cb, int E, double* u) {
    double lo = INFINITY, hi = -INFINITY;
    for (int j = 0; j < E; ++j) {
        const double c = h2d(cb[j]);
        if (c < lo) lo = c;
        if (c > hi) hi = c;
    }
    const double m = __dmul_rn(0.5, __dadd_rn(hi, lo));
    double s = __dmul_rn(0.5, __dsub_rn(hi, lo));
    if (s == 0.0) s = 1.0;
    double acc = 0.0;
    for (int j = 0; j < E; ++j) {
        const double v = __ddiv_rn(__dsub_rn(h2d(cb[j]), m), s);
        u[j] = v;
        acc = __dadd_rn(acc, __dmul_rn(v, v));
    }
    return acc == acc ? acc : INFINITY;      // a codebook with an infinity has no norm: last, so that `order` is a permutation
}

__global__ void __launch_bounds__(128) libfit_normalise_kernel(const uint16_t* __restrict__ cb, int rows, int E, double* u, double* nn) {
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i < rows) nn[i] = normalise_channel(cb + (int64_t)i * E, E, u + (int64_t)i * E);
}

// order[r] = the channel of rank r by (nn, channel): rank by counting, a warp per channel
__global__ void __launch_bounds__(256) libfit_rank_kernel(const double* __restrict__ nn, int rows, int* order) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= rows) return;
    const double mine = __ldg(nn + i);
    int r = 0;
#pragma unroll 8
    for (int j = lane; j < rows; j += 32) {
        const double o = __ldg(nn + j);
        r += (o < mine) || (o == mine && j < i);
    }
    r = __reduce_add_sync(0xffffffffu, r);
    if (lane == 0) order[r] = i;
}

// seed l of the library: L evenly spaced channels of that order
__device__ __forceinline__ int seed_rank(int l, int rows, int L) {
    long long t = rows >= L ? (long long)floor(__ddiv_rn(__dmul_rn(__dadd_rn((double)l, 0.5), (double)rows), (double)L))
                            : (long long)(l % rows);
    return (int)(t >= rows ? rows - 1 : t);
}

// the centroid's entries c[0..E) in ascending order, fp16 (thread `tid` < E; entries that are no numbers behind the others, so
// that every place of the library is written)
__device__ __forceinline__ void store_ascending(const double* c, int E, int tid, uint16_t* lib) {
    const double x = c[tid];
    int r = 0;
    for (int j = 0; j < E; ++j) {
        const double v = c[j];
        const bool before = v < x || (x != x && v == v), after = x < v || (v != v && x == x);
        r += before || (!before && !after && j < tid);
    }
    lib[r] = d2h(x);
}

// The rounds of the k-means where they fit one cluster of 16 SMs (N = 2: see launch_libfit_library): the channels are dealt to the blocks in runs.
//   assignment  two threads per channel, its E values in registers, centroids in order with a strict "less than"
//   update      half a block per centroid: every block has all assignments (a byte per channel, written to each of them),
//               compacts the members in channel order, fetches their values from the blocks that hold them, and thread j adds
//               entries j one by one: the order of the serial evaluation
// A round costs two cluster barriers instead of two grid barriers with their trips through L2.  Bound by the serial sums (about
// rows / L dependent fp64 additions) and the barriers.  3072 channels, N = 2, L = 32, 20 rounds:
// 186 -> 155 us with the two kernels in front.
constexpr int kClBlocks = 16;
constexpr int kClVals = 2048;                       // member values staged at a time by half a block
constexpr size_t kClSmem = 200 * 1024;
constexpr long long kClTerms = 2000000;
constexpr int kClLib = 40;                          // centroids at most
__host__ __device__ inline int cl_per(int rows) { return ((rows + kClBlocks - 1) / kClBlocks + 3) & ~3; }
inline size_t cl_smem(int rows, int E, int L) {
    const size_t asg = ((size_t)cl_per(rows) * kClBlocks + 15) & ~size_t(15);
    return (size_t)cl_per(rows) * E * 8 + (size_t)L * E * 8 + 2 * kClVals * 8 + asg + 2 * 2 * asg;
}

template <int E>
__global__ void __launch_bounds__(kLibThreads) libfit_cluster_kernel(const double* __restrict__ u, const int* __restrict__ order, int rows,
                                                                     int L, int iters, uint16_t* lib) {
    extern __shared__ __align__(16) double cl[];
    __shared__ int changed;             // the last round, counted from one, in which a centroid of the cluster moved
    __shared__ int wsum[2][8];
    constexpr int HT = kLibThreads / 2;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), per = cl_per(rows);
    const int tid = threadIdx.x, lane = tid & 31, half = tid / HT, ht = tid % HT, hw = ht >> 5;
    double* su = cl;                                    // [E][per] values of this block's channels
    double* cen = su + (size_t)per * E;                 // [L][E]
    double* vals = cen + (size_t)L * E + half * kClVals;
    uint8_t* asg = (uint8_t*)(cen + (size_t)L * E + 2 * kClVals);
    const int asg_bytes = (per * kClBlocks + 15) & ~15;
    uint16_t* member = (uint16_t*)(asg + asg_bytes) + (size_t)half * asg_bytes;
    const int c0 = rank * per, mine = max(0, min(rows - c0, per));
    for (int i = tid; i < mine * E; i += kLibThreads) su[(i % E) * per + i / E] = __ldg(u + (size_t)c0 * E + i);
    for (int i = tid; i < L * E; i += kLibThreads) cen[i] = __ldg(u + (size_t)__ldg(order + seed_rank(i / E, rows, L)) * E + i % E);
    if (tid == 0) changed = 0;
    cluster.sync();
    auto half_sync = [&]() { asm volatile("bar.sync %0, %1;" :: "r"(1 + half), "r"(HT) : "memory"); };
    for (int it = 1; it <= iters; ++it) {
        for (int i0 = 0; i0 < per; i0 += HT) {       // two neighbouring threads to a channel, half of the centroids each
            const int i = i0 + (tid >> 1), sub = tid & 1, h0 = (L + 1) >> 1, l1 = sub ? L : h0;
            double x[E];
#pragma unroll
            for (int j = 0; j < E; ++j) x[j] = i < mine ? su[j * per + i] : 0.0;
            int best = sub ? h0 : 0;
            double bd = INFINITY;
#pragma unroll 4
            for (int l = best; l < l1; ++l) {
                double d = 0.0;
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const double t = __dsub_rn(x[j], cen[l * E + j]);
                    d = __dadd_rn(d, __dmul_rn(t, t));
                }
                if (d < bd) { bd = d; best = l; }
            }
            const double od = __shfl_xor_sync(0xffffffffu, bd, 1);
            const int ob = __shfl_xor_sync(0xffffffffu, best, 1);
            // the upper half's centroid only when strictly nearer
            if (sub ? !(bd < od) : od < bd) best = ob;
            // four channels to a word, a copy to every block
            uint32_t w = (uint32_t)best << (8 * ((lane >> 1) & 3));
            w |= __shfl_xor_sync(0xffffffffu, w, 2);
            w |= __shfl_xor_sync(0xffffffffu, w, 4);
            if (i < per)
#pragma unroll
                for (int r = 0; r < kClBlocks / 8; ++r)
                    *(uint32_t*)(cluster.map_shared_rank(asg, (lane & 7) + 8 * r) + c0 + (i & ~3)) = w;
        }
        cluster.sync();
        for (int l0 = rank; l0 < L; l0 += 2 * kClBlocks) {
            const int l = l0 + half * kClBlocks;
            // members of centroid l, in channel order: a run of words to every thread
            const int words = (rows + 3) / 4, wpt = (words + HT - 1) / HT;
            const uint32_t want = (uint32_t)(l & 0xff) * 0x01010101u;
            auto hits = [&](int q) -> uint32_t {
                if (l >= L || q >= words) return 0u;
                uint32_t h = __vcmpeq4(*(const uint32_t*)(asg + 4 * q), want) & 0x01010101u;
                const int over = 4 * q + 4 - rows;                      // channels of this word beyond the last
                return over > 0 ? h & (0xffffffffu >> (8 * over)) : h;
            };
            int c = 0;
            for (int k = 0; k < wpt; ++k) c += __popc(hits(ht * wpt + k));
            int inc = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= d) inc += t;
            }
            if (lane == 31) wsum[half][hw] = inc;
            half_sync();
            int at = inc - c, n = 0;
#pragma unroll
            for (int k = 0; k < HT / 32; ++k) { if (k < hw) at += wsum[half][k]; n += wsum[half][k]; }
            for (int k = 0; k < wpt; ++k) {
                const int q = ht * wpt + k;
                for (uint32_t h = hits(q); h; h &= h - 1) member[at++] = (uint16_t)(4 * q + (__ffs(h) >> 3));
            }
            half_sync();
            double acc = 0.0;
            for (int m0 = 0; m0 < n; m0 += kClVals / E) {
                const int cnt = min(n - m0, kClVals / E);
                for (int t = ht; t < cnt * E; t += HT) {
                    const int i = member[m0 + t / E], owner = i / per;
                    vals[t] = cluster.map_shared_rank(su, owner)[(t % E) * per + (i - owner * per)];
                }
                half_sync();
                if (ht < E) {
                    // the next eight values travel under the chain of eight additions
                    double v[8], w[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = k < cnt ? vals[k * E + ht] : 0.0;
                    int m = 0;
                    for (; m + 8 <= cnt; m += 8) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) w[k] = m + 8 + k < cnt ? vals[(m + 8 + k) * E + ht] : 0.0;
#pragma unroll
                        for (int k = 0; k < 8; ++k) { acc = __dadd_rn(acc, v[k]); v[k] = w[k]; }
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (m + k < cnt) acc = __dadd_rn(acc, v[k]);
                }
                half_sync();
            }
            if (ht < E && n > 0) {
                const double m = __ddiv_rn(acc, (double)n);
                if (m != cen[l * E + ht]) {
                    for (int r = 0; r < kClBlocks; ++r) {
                        cluster.map_shared_rank(cen, r)[l * E + ht] = m;
                        *cluster.map_shared_rank(&changed, r) = it;
                    }
                }
            }
            half_sync();            // (the counts of the next centroid overwrite this one's)
        }
        cluster.sync();
        if (changed != it) break;
    }
    for (int l = rank; l < L; l += kClBlocks)
        if (tid < E) store_ascending(cen + l * E, E, tid, lib + l * E);
}

// The whole k-means in one cooperative launch: normalise, order by norm, seed, `iters` rounds of assignment and update,
// store.  As separate launches (three per round) the rounds were bound by launches and by the update's chain of dependent
// loads: 3072 channels, N = 2, 20 rounds 515 us; here a round costs two grid barriers and the update's serial sums.
//   assignment  a warp per channel, a lane per centroid (32 at a time); every lane sums its squared distance in entry
//               order and the smallest (distance, centroid) pair wins: the answer of a scan with a strict "less than"
//   update      a block per centroid compacts its members in channel order, and thread j adds their entries j one by one:
//               the order of the serial evaluation
// A round is a chain of latencies (the two barriers, L2 round trips, the serial sums).  Where the normalised codebooks fit
// (resident: 3072 channels of N = 2 are 96 KB) every block keeps them in shared memory, which takes the L2 round trip out of
// each channel's assignment and the staging of the members out of the update (quantising 3072 x 4096 at N = 2 in all:
// 723 -> 677 us); larger ones are read from L2.
__global__ void __launch_bounds__(kLibThreads) libfit_library_kernel(const uint16_t* __restrict__ cb, int rows, int E, int L,
                                                                     int iters, double* u, double* nn, int* order, int* asg,
                                                                     double* cen, int* flag, uint16_t* lib, int resident) {
    extern __shared__ double su[];      // resident: u
    __shared__ int sh[32];
    __shared__ int total;
    __shared__ int member[kLibTile];
    __shared__ double vals[kLibVals];
    cg::grid_group grid = cg::this_grid();
    const int tid = threadIdx.x, lane = tid & 31;
    const int gt = blockIdx.x * kLibThreads + tid, nt = gridDim.x * kLibThreads;
    const int gw = gt >> 5, nw = nt >> 5;
    // (the steps of normalise_channel, libfit_rank_kernel, seed_rank and store_ascending stand here in line: called as functions they
    // cost this kernel 3 %, N = 4, 3072 channels 290 -> 298 us)
    // u[i][j] = (c_ij - m_i) / s_i, m and s the middle and half-width of the codebook's range; nn[i] = |u_i|^2
    for (int i = gt; i < rows; i += nt) {
        double lo = INFINITY, hi = -INFINITY;
        for (int j = 0; j < E; ++j) {
            const double c = h2d(cb[(int64_t)i * E + j]);
            if (c < lo) lo = c;
            if (c > hi) hi = c;
        }
        const double m = __dmul_rn(0.5, __dadd_rn(hi, lo));
        double s = __dmul_rn(0.5, __dsub_rn(hi, lo));
        if (s == 0.0) s = 1.0;
        double acc = 0.0;
        for (int j = 0; j < E; ++j) {
            const double v = __ddiv_rn(__dsub_rn(h2d(cb[(int64_t)i * E + j]), m), s);
            u[(int64_t)i * E + j] = v;
            acc = __dadd_rn(acc, __dmul_rn(v, v));
        }
        nn[i] = acc == acc ? acc : INFINITY;     // a codebook with an infinity has no norm: last, so that `order` is a permutation
    }
    if (gt < 3) flag[gt] = 0;
    grid.sync();
    if (resident) {                     // (used behind the next barriers)
        const int n2 = rows * E / 2;    // E is even
#pragma unroll 4
        for (int i = tid; i < n2; i += kLibThreads) ((double2*)su)[i] = __ldcg((const double2*)u + i);
    }
    // order[r] = the channel of rank r by (nn, channel): rank by counting
    for (int i = gw; i < rows; i += nw) {
        const double mine = __ldcg(nn + i);
        int r = 0;
#pragma unroll 4
        for (int j = lane; j < rows; j += 32) {
            const double o = __ldcg(nn + j);
            r += (o < mine) || (o == mine && j < i);
        }
        r = __reduce_add_sync(0xffffffffu, r);
        if (lane == 0) order[r] = i;
    }
    grid.sync();
    for (int i = gt; i < L * E; i += nt) {      // L evenly spaced channels of that order
        const int l = i / E, j = i % E;
        long long t = rows >= L ? (long long)floor(__ddiv_rn(__dmul_rn(__dadd_rn((double)l, 0.5), (double)rows), (double)L))
                                : (long long)(l % rows);
        if (t >= rows) t = rows - 1;
        cen[i] = __ldcg(u + (int64_t)__ldcg(order + t) * E + j);
    }
    grid.sync();
    for (int it = 0; it < iters; ++it) {
        const bool staged = L * E <= kLibVals;
        if (staged) {
            for (int i = tid; i < L * E; i += kLibThreads) vals[(i % E) * L + i / E] = __ldcg(cen + i);   // [entry][centroid]
            __syncthreads();
        }
        for (int i = gw; i < rows; i += nw) {
            int best = 0;
            double bd = INFINITY;
            for (int l0 = 0; l0 < L; l0 += 32) {
                const int l = l0 + lane;
                double d = INFINITY;
                if (l < L) {
                    d = 0.0;
#pragma unroll 4
                    for (int j = 0; j < E; ++j) {
                        const double x = resident ? su[i * E + j] : __ldcg(u + (int64_t)i * E + j);
                        const double t = __dsub_rn(x, staged ? vals[j * L + l] : __ldcg(cen + l * E + j));
                        d = __dadd_rn(d, __dmul_rn(t, t));
                    }
                    if (d != d) d = INFINITY;    // nearest to nothing, as in a scan; no lane may drop what it compares it with
                }
                int bl = l;
#pragma unroll
                for (int o = 16; o; o >>= 1) {   // smallest distance, lower centroid on a tie
                    const double od = __shfl_xor_sync(0xffffffffu, d, o);
                    const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
                    if (od < d || (od == d && ol < bl)) { d = od; bl = ol; }
                }
                if (d < bd) { bd = d; best = bl; }   // a later group of 32 wins only when strictly nearer
            }
            if (lane == 0) asg[i] = best;
        }
        grid.sync();
        if (gt == 0) flag[(it + 1) % 3] = 0;         // last read two barriers ago
        for (int l = blockIdx.x; l < L; l += gridDim.x) {
            double acc = 0.0;
            long long cnt = 0;
            for (int i0 = 0; i0 < rows; i0 += kLibTile) {
                constexpr int per = kLibTile / kLibThreads;
                int hit = 0;
                static_assert(per % 4 == 0, "whole vectors of assignments");
#pragma unroll
                for (int e = 0; e < per; e += 4) {
                    const int i = i0 + tid * per + e;
                    int4 t = make_int4(-1, -1, -1, -1);
                    if (i + 3 < rows) t = __ldcg((const int4*)(asg + i));
                    else if (i < rows) { t.x = __ldcg(asg + i); if (i + 1 < rows) t.y = __ldcg(asg + i + 1); if (i + 2 < rows) t.z = __ldcg(asg + i + 2); }
                    hit |= ((t.x == l) | (t.y == l) << 1 | (t.z == l) << 2 | (t.w == l) << 3) << e;
                }
                int at = block_excl_scan(__popc(hit), sh, &total);
                for (int e = 0; e < per; ++e)
                    if ((hit >> e) & 1) member[at++] = i0 + tid * per + e;
                __syncthreads();
                const int n = total, chunk = kLibVals / E;
                if (resident && tid < E) {
#pragma unroll 8
                    for (int m = 0; m < n; ++m) acc = __dadd_rn(acc, su[member[m] * E + tid]);
                }
                if (!resident)
                for (int m0 = 0; m0 < n; m0 += chunk) {
                    const int c = n - m0 < chunk ? n - m0 : chunk;
                    for (int i = tid; i < c * E; i += kLibThreads) vals[i] = __ldcg(u + (int64_t)member[m0 + i / E] * E + i % E);
                    __syncthreads();
                    if (tid < E) {
#pragma unroll 8
                        for (int m = 0; m < c; ++m) acc = __dadd_rn(acc, vals[m * E + tid]);
                    }
                    __syncthreads();
                }
                cnt += n;
                __syncthreads();
            }
            if (tid < E && cnt > 0) {
                const double m = __ddiv_rn(acc, (double)cnt);
                if (m != __ldcg(cen + l * E + tid)) { cen[l * E + tid] = m; flag[it % 3] = 1; }
            }
        }
        grid.sync();
        if (!__ldcg(flag + it % 3)) break;
    }
    // lib[l] = the centroid's entries in ascending order, fp16
    for (int l = blockIdx.x; l < L; l += gridDim.x) {
        __syncthreads();
        if (tid < E) vals[tid] = __ldcg(cen + l * E + tid);
        __syncthreads();
        if (tid < E) {
            const double x = vals[tid];
            int r = 0;
            // (entries that are no numbers behind the others, so that every place of the library is written)
            for (int j = 0; j < E; ++j) {
                const double v = vals[j];
                const bool before = v < x || (x != x && v == v), after = x < v || (v != v && x == x);
                r += before || (!before && !after && j < tid);
            }
            lib[l * E + r] = d2h(x);
        }
    }
}

// ------------------------------------------------------------------ the assignment of a group

constexpr int kLibSmem = 2048;      // library entries (L * 2^N) staged in shared memory

template <int GS>
struct GroupGeo {
    static constexpr int VPL = GS / 32;                 // consecutive weights of a lane
    static constexpr int WARPS = GS == 256 ? 4 : 8;     // groups of a channel at a time
};

// Ascending over the warp: element lane * VPL + e.
template <int VPL>
__device__ __forceinline__ void warp_sort(float (&a)[VPL], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * VPL; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j; j >>= 1) {
            if (j >= VPL) {
                const bool low = ((lane * VPL) & j) == 0, up = ((lane * VPL) & k) == 0;
#pragma unroll
                for (int e = 0; e < VPL; ++e) {
                    const float o = __shfl_xor_sync(0xffffffffu, a[e], j / VPL);
                    a[e] = low == up ? fminf(a[e], o) : fmaxf(a[e], o);
                }
            } else {
#pragma unroll
                for (int e = 0; e < VPL; ++e) {
                    if (e & j) continue;
                    const bool up = k < VPL ? (e & k) == 0 : ((lane * VPL + e) & k) == 0;
                    const float x = fminf(a[e], a[e | j]), y = fmaxf(a[e], a[e | j]);
                    a[e] = up ? x : y; a[e | j] = up ? y : x;
                }
            }
        }
    }
}

// One block per channel, one warp per group of GS weights.  The squared error of a group against a library entry is, in
// exact arithmetic, a sum over the 2^N cells of (sum v^2 - 2 d sum v + n d^2): with the group sorted once and its prefix
// sums of v and v^2 at hand a lane scores an entry by 2^N - 1 searches instead of GS nearest-entry decisions (3072 x 4096
// weights, N = 2, L = 32: 1065 us with every decision and every square taken in fp64).  Those scores carry a rounding
// error far below the differences between entries: an entry is ruled out when its score less its error bound lies above
// another's score plus bound, and only where more than one entry is left are their errors summed value by value in the
// order the method states.
template <int GS>
__global__ void __launch_bounds__(32 * GroupGeo<GS>::WARPS) libfit_group_kernel(
    const float* __restrict__ W, const uint8_t* __restrict__ mask, const double* __restrict__ ms, int K, int bits, int L,
    const uint16_t* __restrict__ lib, uint8_t* __restrict__ idx, uint8_t* __restrict__ gid, uint16_t* __restrict__ gscale,
    uint16_t* __restrict__ gmid, double* __restrict__ cosv) {
    constexpr int VPL = GroupGeo<GS>::VPL, WARPS = GroupGeo<GS>::WARPS;
    __shared__ uint16_t slib[kLibSmem];                 // [entry of a codebook][codebook]
    __shared__ __align__(16) float s_v[WARPS][GS];
    __shared__ double2 s_p[WARPS][GS + 1];              // sums of v - mid and (v - mid)^2 in front of sorted position i
    __shared__ double s_dec[WARPS][64];
    __shared__ float s_thr[WARPS][64];
    __shared__ double s_red[3][WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int E = 1 << bits;
    const double mu = ms[0];
    const float fmu = (float)mu;
    const int64_t row = blockIdx.x;
    const int G = K / GS;
    const bool staged = L * E <= kLibSmem;
    if (staged)
        for (int i = tid; i < L * E; i += blockDim.x) slib[(i % E) * L + i / E] = lib[i];
    __syncthreads();
    float* sv = s_v[warp];
    double2* sp = s_p[warp];
    double* dec = s_dec[warp];
    float* thr = s_thr[warp];
    double sab = 0.0, saa = 0.0, sbb = 0.0;
    for (int g = warp; g < G; g += nwarps) {
        const int64_t grp = row * G + g, base = grp * GS + lane * VPL;
        float w[VPL];
        uint32_t ext = 0;                               // bit e: weight e of this lane was extracted
#pragma unroll
        for (int e = 0; e < VPL; e += 2) { const float2 t = __ldg((const float2*)(W + base + e)); w[e] = t.x; w[e + 1] = t.y; }
        if (mask) {
#pragma unroll
            for (int e = 0; e < VPL; e += 2) {
                const uint16_t t = __ldg((const uint16_t*)(mask + base + e));
                ext |= ((t & 0xffu) ? 1u << e : 0u) | ((t & 0xff00u) ? 2u << e : 0u);
            }
        }
        float a[VPL];
        float lo = INFINITY, hi = -INFINITY;
#pragma unroll
        for (int e = 0; e < VPL; ++e) {
            const bool x = (ext >> e) & 1u;
            a[e] = x ? fmu : w[e];
            lo = fminf(lo, x ? INFINITY : w[e]); hi = fmaxf(hi, x ? -INFINITY : w[e]);
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, d)); hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, d));
        }
        const int nx = __reduce_add_sync(0xffffffffu, __popc(ext));
        double dlo = (double)lo, dhi = (double)hi;
        if (nx) { dlo = fmin(dlo, mu); dhi = fmax(dhi, mu); }
        const uint16_t mid16 = d2h(__dmul_rn(0.5, __dadd_rn(dhi, dlo))), sc16 = d2h(__dmul_rn(0.5, __dsub_rn(dhi, dlo)));
        const bool flat = dhi == dlo;                   // a constant group: scale 0, entry 0, indices 0
        int best = 0;
        if (!flat) {
            const double mid = h2d(mid16);
            warp_sort<VPL>(a, lane);
            double p1 = 0.0, p2 = 0.0;
            double2 own[VPL];
#pragma unroll
            for (int e = 0; e < VPL; ++e) {
                const double t = (double)a[e] - mid;
                p1 += t; p2 = fma(t, t, p2);
                own[e] = make_double2(p1, p2);
            }
            double i1 = p1, i2 = p2;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const double t1 = __shfl_up_sync(0xffffffffu, i1, d), t2 = __shfl_up_sync(0xffffffffu, i2, d);
                if (lane >= d) { i1 += t1; i2 += t2; }
            }
            __syncwarp();                               // the previous group's readers are done
#pragma unroll
            for (int e = 0; e < VPL; ++e) {
                sv[lane * VPL + e] = a[e];
                sp[lane * VPL + e + 1] = make_double2(i1 - p1 + own[e].x, i2 - p2 + own[e].y);
            }
            if (lane == 0) sp[0] = make_double2(0.0, 0.0);
            __syncwarp();
            const double2 all = sp[GS];
            // Values are sorted as floats, which puts mu's copies off by `delta`: a copy's squared error is then off by at most
            // delta (2 |mu - d| + delta), d the nearest entry, wherever the entries lie (a caller's library may reach far
            // beyond the group, whose own library lies in [-1, 1] of it).
            const double delta = fabs(mu - (double)fmu), off = (double)nx * delta;
            const double slack = 1e-9 * all.y + off * (2.0 * fabs(mu - mid) + delta);
            double score[8], bound[8];
            double least = INFINITY;
#pragma unroll 1
            for (int l0 = 0; l0 < L; l0 += 32) {
                const int l = l0 + lane;
                double sc = INFINITY, bd = 0.0;
                if (l < L) {
                    bool asc = true;
                    double far = 0.0, prev = 0.0;
                    double2 at = make_double2(0.0, 0.0);
                    int cut = 0;
                    sc = 0.0;
                    for (int j = 0; j <= E; ++j) {
                        double d = 0.0, x = INFINITY;
                        if (j < E) {
                            d = h2d(v2a_value16(sc16, staged ? slib[j * L + l] : __ldg(lib + l * E + j), mid16));
                            far = fmax(far, fabs(d - mid));
                            if (j == 0) { prev = d; continue; }
                            if (d < prev) asc = false;
                            x = 0.5 * (prev + d);
                        }
                        int c = GS;
                        if (j < E) {
                            const float xf = __double2float_rd(x);
                            c = 0;
#pragma unroll
                            for (int step = GS / 2; step; step >>= 1) c += sv[c + step - 1] <= xf ? step : 0;
                            c += sv[c] <= xf;
                            c = c > cut ? c : cut;
                        }
                        const double2 to = sp[c];
                        const double q = prev - mid;
                        sc += (to.y - at.y) - 2.0 * q * (to.x - at.x) + (double)(c - cut) * q * q;
                        at = to; cut = c; prev = d;
                    }
                    bd = asc ? slack + 2.0 * off * far + 1e-12 * GS * far * far : INFINITY;    // a codebook out of order is always summed exactly
                    least = fmin(least, sc + bd);
                }
                score[l0 >> 5] = sc; bound[l0 >> 5] = bd;
            }
#pragma unroll
            for (int d = 16; d; d >>= 1) least = fmin(least, __shfl_xor_sync(0xffffffffu, least, d));
            int count = 0;
            best = L;
#pragma unroll 1
            for (int l0 = 0; l0 < L; l0 += 32) {
                const bool in = l0 + lane < L && !(score[l0 >> 5] - bound[l0 >> 5] > least);
                const unsigned b = __ballot_sync(0xffffffffu, in);
                count += __popc(b);
                if (b && best == L) best = l0 + __ffs(b) - 1;
            }
            if (count > 1) {                            // too close to call: value by value
                double bs = INFINITY;
                int bl = L;
#pragma unroll 1
                for (int l0 = 0; l0 < L; l0 += 32) {
                    const int l = l0 + lane;
                    if (l >= L || score[l0 >> 5] - bound[l0 >> 5] > least) continue;
                    double d16[64];
                    bool asc = true;
                    for (int j = 0; j < E; ++j) {
                        d16[j] = h2d(v2a_value16(sc16, __ldg(lib + l * E + j), mid16));
                        if (j && d16[j] < d16[j - 1]) asc = false;
                    }
                    double acc = 0.0;
                    for (int t = 0; t < GS; ++t) {
                        const double x = bulk_value(W, mask, grp * GS + t, mu), d = __dsub_rn(x, d16[nearest_entry(d16, E, x, asc)]);
                        acc = __dadd_rn(acc, __dmul_rn(d, d));
                    }
                    if (acc < bs) { bs = acc; bl = l; }
                }
                __syncwarp();
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    const double os = __shfl_xor_sync(0xffffffffu, bs, o);
                    const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
                    if (os < bs || (os == bs && ol < bl)) { bs = os; bl = ol; }
                }
                best = bl < L ? bl : 0;
            }
        }
        if (lane == 0) {
            gid[grp] = (uint8_t)best;
            gscale[grp] = flat ? (uint16_t)0 : sc16;
            gmid[grp] = mid16;
        }
        // indices against the winner
        __syncwarp();
        for (int j = lane; j < E; j += 32) dec[j] = h2d(v2a_value16(flat ? (uint16_t)0 : sc16, __ldg(lib + best * E + j), mid16));
        __syncwarp();
        bool rise = true;
        for (int j = lane; j < E; j += 32) {
            thr[j] = INFINITY;
            if (j < E - 1) {
                if (dec[j] < dec[j + 1]) thr[j] = last_of_lower(dec[j], dec[j + 1]);
                else rise = false;
            }
        }
        rise = __all_sync(0xffffffffu, rise);
        __syncwarp();
        int at[VPL];
#pragma unroll
        for (int e = 0; e < VPL; ++e) at[e] = 0;
        if (!flat) {
            bool asc = true;
            if (!rise)
                for (int j = 1; j < E; ++j) asc = asc && dec[j] >= dec[j - 1];
            if (rise) {
                for (int step = E >> 1; step; step >>= 1) {
#pragma unroll
                    for (int e = 0; e < VPL; ++e) at[e] += w[e] > thr[at[e] + step - 1] ? step : 0;
                }
            } else {
#pragma unroll 1
                for (int e = 0; e < VPL; ++e) at[e] = nearest_entry(dec, E, (double)w[e], asc);
            }
            if (nx) {
                const int xi = nearest_entry(dec, E, mu, asc);
#pragma unroll
                for (int e = 0; e < VPL; ++e)
                    if ((ext >> e) & 1u) at[e] = xi;
            }
        }
#pragma unroll
        for (int e = 0; e < VPL; e += 2) *(uint16_t*)(idx + base + e) = (uint16_t)(at[e] | (at[e + 1] << 8));
        if (cosv) {
#pragma unroll
            for (int e = 0; e < VPL; ++e) {
                const double x = (double)w[e];
                double b = dec[at[e]];
                if ((ext >> e) & 1u) b = h2d(d2h(__dadd_rn(b, h2d(d2h(__dsub_rn(x, b))))));   // W^ = fp16(D16 + S)
                sab = fma(x, b, sab); saa = fma(x, x, saa); sbb = fma(b, b, sbb);
            }
        }
    }
    if (cosv) {
        sab = warp_sum(sab); saa = warp_sum(saa); sbb = warp_sum(sbb);
        if (lane == 0) { s_red[0][warp] = sab; s_red[1][warp] = saa; s_red[2][warp] = sbb; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < nwarps; ++w) { sab += s_red[0][w]; saa += s_red[1][w]; sbb += s_red[2][w]; }
            cosv[row] = (saa == 0.0 || sbb == 0.0) ? 1.0 : __ddiv_rn(sab, __dmul_rn(__dsqrt_rn(saa), __dsqrt_rn(sbb)));
        }
    }
}

template <int GS>
cudaError_t launch_groups(const float* W, const uint8_t* mask, const double* ms, int rows, int cols, int bits, int L,
                          const uint16_t* lib, uint8_t* idx, uint8_t* gid, uint16_t* gscale, uint16_t* gmid, double* cosv,
                          cudaStream_t s) {
    const int groups = cols / GS, warps = groups < GroupGeo<GS>::WARPS ? groups : GroupGeo<GS>::WARPS;
    libfit_group_kernel<GS><<<rows, warps * 32, 0, s>>>(W, mask, ms, cols, bits, L, lib, idx, gid, gscale, gmid, cosv);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_libfit_assign(const float* W, const uint8_t* mask, const double* ms, int rows, int cols, int bits, int L,
                                 int group_size, const uint16_t* lib, uint8_t* idx, uint8_t* gid, uint16_t* gscale,
                                 uint16_t* gmid, double* cosv, cudaStream_t s) {
    if (group_size == 64) return launch_groups<64>(W, mask, ms, rows, cols, bits, L, lib, idx, gid, gscale, gmid, cosv, s);
    if (group_size == 128) return launch_groups<128>(W, mask, ms, rows, cols, bits, L, lib, idx, gid, gscale, gmid, cosv, s);
    return launch_groups<256>(W, mask, ms, rows, cols, bits, L, lib, idx, gid, gscale, gmid, cosv, s);
}

namespace {

template <int E>
cudaError_t launch_cluster(const uint16_t* codebook, int rows, int L, int iters, double* u, double* nn, int* order, uint16_t* lib,
                           cudaStream_t s, bool* taken) {
    static std::atomic<int> fits[256] = {};       // per device: 1 a cluster of this size can be resident, 2 it can not
    const int dev = xfp::DeviceOnce::current();
    const size_t smem = cl_smem(rows, E, L);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kClBlocks);
    cfg.blockDim = dim3(kLibThreads);
    cfg.dynamicSmemBytes = kClSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kClBlocks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int f = fits[dev].load(std::memory_order_acquire);
    if (f == 0) {
        cudaError_t e = cudaFuncSetAttribute(libfit_cluster_kernel<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(libfit_cluster_kernel<E>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        int n = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, libfit_cluster_kernel<E>, &cfg);
        if (e != cudaSuccess) cudaGetLastError();
        f = e == cudaSuccess && n > 0 ? 1 : 2;
        fits[dev].store(f, std::memory_order_release);
    }
    *taken = f == 1;
    if (f != 1) return cudaSuccess;
    libfit_normalise_kernel<<<(rows + 127) / 128, 128, 0, s>>>(codebook, rows, E, u, nn);
    libfit_rank_kernel<<<(rows + 7) / 8, 256, 0, s>>>(nn, rows, order);
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, libfit_cluster_kernel<E>, (const double*)u, (const int*)order, rows, L, iters, lib);
}

}  // namespace

cudaError_t launch_libfit_library(const uint16_t* codebook, int rows, int E, int L, int iters, double* u, double* nn,
                                  int* order, int* asg, double* cen, int* flags, uint16_t* lib, cudaStream_t s) {
    // One cluster at N = 2 while its assignment step (rows L E terms on 16 SMs) costs less than the grid barriers it saves: at few
    // centroids whatever the rows, at many only where rows are many too.  us, 20 rounds at most, one cluster | all SMs:
    //   3072 channels  L = 8 203 | 248, 32 146 | 173, 40 192 | 197, 64 196 | 183, 128 270 | 204, 256 315 | 219
    //   1024 channels  L = 8 91 | 136, 32 99 | 128, 40 93 | 101, 64 103 | 96, 128 134 | 93, 256 177 | 102
    //   12288 channels L = 8 641 | 791, 32 472 | 522, 40 561 | 606, 64 552 | 576, 128 790 | 744
    // N = 3 and 4 lose from 32 centroids on: 3072 channels N = 3 230 | 237, N = 4 369 | 290, 6144 N = 3 443 | 396
    bool taken = false;
    if (E == 4 && L <= kClLib && (long long)rows * L * E <= kClTerms && rows <= 65535 && cl_smem(rows, E, L) <= kClSmem) {
        const cudaError_t e = launch_cluster<4>(codebook, rows, L, iters, u, nn, order, lib, s, &taken);
        if (taken || e != cudaSuccess) return e;
    }
    // a warp per channel, within one block per SM (the blocks wait for one another)
    const int want = (rows + kLibThreads / 32 - 1) / (kLibThreads / 32), sms = xfp::sm_count();
    int blocks = want > L ? want : L;
    if (blocks > sms) blocks = sms;
    size_t smem = (size_t)rows * E * sizeof(double);
    int resident = smem <= kLibSmemU;
    if (!resident) smem = 0;
    static xfp::DeviceOnce attr_done;
    const int dev = xfp::DeviceOnce::current();
    if (!attr_done.is_set(dev)) {
        const cudaError_t e = cudaFuncSetAttribute(libfit_library_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLibSmemU);
        if (e != cudaSuccess) return e;
        attr_done.set(dev);
    }
    void* args[] = {&codebook, &rows, &E, &L, &iters, &u, &nn, &order, &asg, &cen, &flags, &lib, &resident};
    return cudaLaunchCooperativeKernel((const void*)libfit_library_kernel, dim3((unsigned)blocks), dim3(kLibThreads), args, smem, s);
}

}  // namespace xq
