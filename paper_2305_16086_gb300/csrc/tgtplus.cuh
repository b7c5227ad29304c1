// TGT+ (Algorithm 4) kernels: column statistics for CalChi (Alg. 3), the
// per-entry range chi (Eq. 17 / Eq. 15) and walk count R (Eq. 13), the
// switch rule (Eq. 14) and the random-walk tail (Eq. 11).
//
// Notation: X = p_tt(., s_b) for the sources s_b of a launch (the block after
// tt hops), L = tau_k - tt the walk length of entry k = (i -> j).
#pragma once

#include "philox.cuh"
#include "propagate.cuh"

namespace sc {

constexpr int kGammaMax = 16;        // largest supported candidate count (Alg. 3)
constexpr int kChiScanThreads = 128;
constexpr int kChiRowsPerCta = 64;
constexpr uint32_t kWalkTag = 0x57414C4Bu;
constexpr long long kWalkCountCap = 1ll << 40;

// strict total order of (value, node): larger value first, then smaller id
template <typename V>
__device__ __forceinline__ bool better(V v, int32_t x, V w, int32_t y) {
    return v > w || (v == w && x < y);
}

// a := the kGammaMax best of the two sorted (descending) lists a and b; list
// element s of a sits at av[s * as] (strided, so that the lists of the threads
// of a warp interleave across shared-memory banks)
template <typename V>
__device__ __forceinline__ void merge_sorted(V *av, int32_t *ai, int as, const V *bv, const int32_t *bi, int bs) {
    V ov[kGammaMax];
    int32_t oi[kGammaMax];
    int x = 0, y = 0;
#pragma unroll
    for (int s = 0; s < kGammaMax; ++s) {
        const V xa = av[x * as], yb = bv[y * bs];
        const int32_t ia = ai[x * as], ib = bi[y * bs];
        const bool ta = better(xa, ia, yb, ib);
        ov[s] = ta ? xa : yb;
        oi[s] = ta ? ia : ib;
        x += ta ? 1 : 0;
        y += ta ? 0 : 1;
    }
#pragma unroll
    for (int s = 0; s < kGammaMax; ++s) {
        av[s * as] = ov[s];
        ai[s * as] = oi[s];
    }
}

// Per CTA and column: the kGammaMax largest (value, node), min, max and the
// frontier volume sum_{x: X[x,b] != 0} d_x over kChiRowsPerCta rows.
// partial layout: [slice][cta][B] entries, lists of kGammaMax.
template <typename T, int B>
__global__ void __launch_bounds__(kChiScanThreads)
    k_chi_scan(const int32_t *__restrict__ row_ptr, const T *__restrict__ x, int32_t n, double *__restrict__ pval,
               int32_t *__restrict__ pid, double *__restrict__ pmin, double *__restrict__ pmax,
               long long *__restrict__ pvol) {
    constexpr int TPC = kChiScanThreads / B;  // threads per column
    constexpr int BATCH = 8;                 // rows in flight per thread
    const int c = threadIdx.x % B, sub = threadIdx.x / B;
    const int32_t r0 = blockIdx.x * kChiRowsPerCta;
    const int32_t r1 = min(n, r0 + kChiRowsPerCta);
    const T *xs = x + static_cast<int64_t>(blockIdx.y) * n * B;
    constexpr int NT = kChiScanThreads;  // list element s of thread t at [s * NT + t]
    __shared__ double sv[kGammaMax * NT];
    __shared__ int32_t si[kGammaMax * NT];
    __shared__ double smin[NT], smax[NT];
    __shared__ long long svol[NT];
    double *val = sv + threadIdx.x;
    int32_t *id = si + threadIdx.x;
    for (int s = 0; s < kGammaMax; ++s) {
        val[s * NT] = -INFINITY;
        id[s * NT] = INT32_MAX;
    }
    // the scan compares in the block's arithmetic type V (widening to double is
    // exact and order-preserving, so every decision is the one in double; this
    // keeps the FP64 units, slow on this GPU, out of the per-element loop)
    using V = typename AccOf<T>::type;
    V vmin = V(INFINITY), vmax = V(-INFINITY), thr = V(-INFINITY);  // thr: the list's last value
    long long vol = 0;
    for (int32_t rb = r0 + sub; rb < r1; rb += TPC * BATCH) {
        V v[BATCH];
        int32_t d[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int32_t r = rb + u * TPC;
            v[u] = r < r1 ? to_acc(xs[static_cast<int64_t>(r) * B + c]) : V(-INFINITY);
            d[u] = r < r1 ? row_ptr[r + 1] - row_ptr[r] : 0;
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int32_t r = rb + u * TPC;
            if (r < r1) {
                vmin = min(vmin, v[u]);
                vmax = max(vmax, v[u]);
                if (v[u] != V(0)) vol += d[u];
                // rows arrive in increasing order: a tie never beats the last slot
                if (v[u] > thr) {
                    double cv = static_cast<double>(v[u]);
                    int32_t ci = r;
#pragma unroll 1
                    for (int s = 0; s < kGammaMax; ++s) {
                        if (better(cv, ci, val[s * NT], id[s * NT])) {
                            const double tv = val[s * NT];
                            const int32_t ti = id[s * NT];
                            val[s * NT] = cv;
                            id[s * NT] = ci;
                            cv = tv;
                            ci = ti;
                        }
                    }
                    thr = static_cast<V>(val[(kGammaMax - 1) * NT]);  // exact: list values come from V
                }
            }
        }
    }
    smin[threadIdx.x] = static_cast<double>(vmin);
    smax[threadIdx.x] = static_cast<double>(vmax);
    svol[threadIdx.x] = vol;
    __syncthreads();
    for (int half = TPC / 2; half > 0; half >>= 1) {  // tree of sorted merges over the column's threads
        if (sub < half) {
            const int o = threadIdx.x + half * B;
            merge_sorted(val, id, NT, sv + o, si + o, NT);
            smin[threadIdx.x] = fmin(smin[threadIdx.x], smin[o]);
            smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[o]);
            svol[threadIdx.x] += svol[o];
        }
        __syncthreads();
    }
    if (sub == 0) {
        const int64_t base = (static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * B + c;
        for (int s = 0; s < kGammaMax; ++s) {
            pval[base * kGammaMax + s] = val[s * NT];
            pid[base * kGammaMax + s] = id[s * NT];
        }
        pmin[base] = smin[threadIdx.x];
        pmax[base] = smax[threadIdx.x];
        pvol[base] = svol[threadIdx.x];
    }
}

// One CTA per column (slice * B + b): threads merge strided CTA partials, then
// a tree of sorted merges in shared memory. The order is total, so the result
// does not depend on the merge order.
template <int B>
__global__ void __launch_bounds__(kChiScanThreads)
    k_chi_merge(int nct, int ncols, const double *__restrict__ pval, const int32_t *__restrict__ pid,
                const double *__restrict__ pmin, const double *__restrict__ pmax,
                const long long *__restrict__ pvol, double *__restrict__ cval, int32_t *__restrict__ cid,
                double *__restrict__ cmin, double *__restrict__ cmax, long long *__restrict__ cvol) {
    const int q = blockIdx.x;
    if (q >= ncols) return;
    const int slice = q / B, c = q % B, t = threadIdx.x;
    constexpr int NT = kChiScanThreads;
    __shared__ double sv[kGammaMax * NT];
    __shared__ int32_t si[kGammaMax * NT];
    __shared__ double smin[NT], smax[NT];
    __shared__ long long svol[NT];
    double *val = sv + t;
    int32_t *id = si + t;
    for (int s = 0; s < kGammaMax; ++s) {
        val[s * NT] = -INFINITY;
        id[s * NT] = INT32_MAX;
    }
    double vmin = INFINITY, vmax = -INFINITY;
    long long vol = 0;
    double bv[kGammaMax];
    int32_t bi[kGammaMax];
    for (int p = t; p < nct; p += kChiScanThreads) {
        const int64_t base = (static_cast<int64_t>(slice) * nct + p) * B + c;
#pragma unroll
        for (int s = 0; s < kGammaMax; ++s) {
            bv[s] = pval[base * kGammaMax + s];
            bi[s] = pid[base * kGammaMax + s];
        }
        merge_sorted(val, id, NT, bv, bi, 1);
        vmin = fmin(vmin, pmin[base]);
        vmax = fmax(vmax, pmax[base]);
        vol += pvol[base];
    }
    smin[t] = vmin;
    smax[t] = vmax;
    svol[t] = vol;
    __syncthreads();
    for (int half = kChiScanThreads / 2; half > 0; half >>= 1) {
        if (t < half) {
            merge_sorted(val, id, NT, sv + t + half, si + t + half, NT);
            smin[t] = fmin(smin[t], smin[t + half]);
            smax[t] = fmax(smax[t], smax[t + half]);
            svol[t] += svol[t + half];
        }
        __syncthreads();
    }
    if (t == 0) {
        for (int s = 0; s < kGammaMax; ++s) {
            cval[static_cast<int64_t>(q) * kGammaMax + s] = val[s * NT];
            cid[static_cast<int64_t>(q) * kGammaMax + s] = id[s * NT];
        }
        cmin[q] = smin[0];
        cmax[q] = smax[0];
        cvol[q] = svol[0];
    }
}

// ---------------------------------------------------------------------------
// Threshold form of the same column statistics (the default): the top-gamma
// list of a column needs only the entries at or above thr = the gamma-th
// largest of its tile maxima (tiles of kTileRows rows). The gamma tiles with
// the largest maxima hold gamma entries >= thr, so the gamma-th largest entry
// is >= thr, and every entry of the top-gamma list lies in a tile whose
// maximum reaches thr. Two launches: tile maxima, minima and volumes
// (k_chi_tiles); per column thr, min, max and volume, the entries >= thr of the
// tiles reaching it, and the top-gamma list among them in the total order
// (k_chi_column). thr = 0 (fewer than gamma tiles hold a positive entry) takes
// the positive entries of those tiles and
// the gamma smallest-id zero rows (the ties at 0 go to smaller ids). A column
// with more than kCandMax candidates (many ties at thr) is scanned in full.
// The first gamma entries of each list equal the full scan's; entries past
// gamma are not read.
// The statistics stay in the block's arithmetic type V (float for FP32 and BF16
// blocks): widening is exact and keeps the order, so every comparison falls out
// as in double, and a comparison in double takes a warp 16 cycles of an SM's FP64
// pipe here. A test of 192 columns of a 40,000-node Barabasi-Albert graph:
// 137 us with the statistics in double, 89 us so (62 with k_chi_column).
// ---------------------------------------------------------------------------
constexpr int kTileRows = 256;
constexpr int kCandMax = 2048;

// a 16-byte vector of stored values as accumulator-type elements, in memory order
__device__ __forceinline__ void unpack16(const uint4 &v, float (&a)[4]) {
    a[0] = __uint_as_float(v.x);
    a[1] = __uint_as_float(v.y);
    a[2] = __uint_as_float(v.z);
    a[3] = __uint_as_float(v.w);
}
__device__ __forceinline__ void unpack16(const uint4 &v, double (&a)[2]) {
    a[0] = __hiloint2double(static_cast<int>(v.y), static_cast<int>(v.x));
    a[1] = __hiloint2double(static_cast<int>(v.w), static_cast<int>(v.z));
}
__device__ __forceinline__ void unpack16(const uint4 &v, float (&a)[8]) {  // bf16 pairs, low half first
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        a[2 * q] = __uint_as_float(w[q] << 16);
        a[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
    }
}

// Per tile of kTileRows rows and column: maximum, minimum and frontier volume
// (sum of d_x over the rows with X[x, c] != 0). Rows are read as 16-byte
// vectors: LG lanes cover a row (VPL vectors each), a warp reads 32 / LG rows
// per load and keeps UR such loads in flight; the lanes holding the same
// columns are combined by shuffles, the warps through shared memory. Maxima,
// minima and integer sums do not depend on the order of combination.
template <typename T, int B>
__global__ void __launch_bounds__(kChiScanThreads)
    k_chi_tiles(const int32_t *__restrict__ row_ptr, const T *__restrict__ x, int32_t n,
                typename AccOf<T>::type *__restrict__ tmax, typename AccOf<T>::type *__restrict__ tmin,
                long long *__restrict__ tvol) {
    using V = typename AccOf<T>::type;
    constexpr int E = 16 / static_cast<int>(sizeof(T));  // elements per 16-byte vector
    constexpr int NV = B / E;                            // vectors per row
    constexpr int LG = NV < 32 ? NV : 32;                // lanes per row
    constexpr int VPL = NV / LG;                         // vectors per lane
    constexpr int RPW = 32 / LG;                         // rows per warp load
    constexpr int NW = kChiScanThreads / 32;
    constexpr int UR = 8 / VPL;                          // row loads in flight per lane
    constexpr int C = VPL * E;                           // columns per lane
    static_assert(NV % LG == 0 && 32 % LG == 0, "row layout");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gl = lane % LG, rsub = lane / LG;
    const int32_t r0 = blockIdx.x * kTileRows, r1 = min(n, r0 + kTileRows);
    const uint4 *xs = reinterpret_cast<const uint4 *>(x + static_cast<int64_t>(blockIdx.y) * n * B);
    V vmax[C], vmin[C];
    long long vol[C];
#pragma unroll
    for (int e = 0; e < C; ++e) {
        vmax[e] = V(-INFINITY);
        vmin[e] = V(INFINITY);
        vol[e] = 0;
    }
    constexpr int STEP = NW * RPW;  // rows per round of the CTA's warps
    for (int32_t rb = r0 + warp * RPW + rsub; rb < r1; rb += STEP * UR) {
        uint4 v[UR][VPL];
        int32_t d[UR];
#pragma unroll
        for (int u = 0; u < UR; ++u) {
            const int32_t r = rb + u * STEP;
            const bool in = r < r1;
            d[u] = in ? row_ptr[r + 1] - row_ptr[r] : 0;
#pragma unroll
            for (int p = 0; p < VPL; ++p)
                v[u][p] = in ? __ldg(xs + static_cast<int64_t>(r) * NV + gl + p * LG) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < UR; ++u) {
            if (rb + u * STEP >= r1) continue;
#pragma unroll
            for (int p = 0; p < VPL; ++p) {
                V a[E];
                unpack16(v[u][p], a);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int k = p * E + e;
                    vmax[k] = max(vmax[k], a[e]);
                    vmin[k] = min(vmin[k], a[e]);
                    if (a[e] != V(0)) vol[k] += d[u];
                }
            }
        }
    }
    // lanes rsub = 0 .. RPW-1 hold the same columns: combine them
#pragma unroll
    for (int o = LG; o < 32; o <<= 1) {
#pragma unroll
        for (int k = 0; k < C; ++k) {
            vmax[k] = max(vmax[k], __shfl_xor_sync(0xffffffffu, vmax[k], o));
            vmin[k] = min(vmin[k], __shfl_xor_sync(0xffffffffu, vmin[k], o));
            vol[k] += __shfl_xor_sync(0xffffffffu, vol[k], o);
        }
    }
    __shared__ V smax[NW][B], smin[NW][B];
    __shared__ long long svol[NW][B];
    if (rsub == 0) {
#pragma unroll
        for (int p = 0; p < VPL; ++p)
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int c = (gl + p * LG) * E + e;
                smax[warp][c] = vmax[p * E + e];
                smin[warp][c] = vmin[p * E + e];
                svol[warp][c] = vol[p * E + e];
            }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < B; c += kChiScanThreads) {
        V a = smax[0][c], b = smin[0][c];
        long long w = svol[0][c];
#pragma unroll
        for (int q = 1; q < NW; ++q) {
            a = max(a, smax[q][c]);
            b = min(b, smin[q][c]);
            w += svol[q][c];
        }
        const int64_t o = (static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * B + c;
        tmax[o] = a;
        tmin[o] = b;
        tvol[o] = w;
    }
}

__device__ __forceinline__ bool has_edge(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                         int32_t a, int32_t b) {
    int32_t lo = row_ptr[a], hi = row_ptr[a + 1];
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        const int32_t c = col[mid];
        if (c == b) return true;
        if (c < b) lo = mid + 1;
        else hi = mid;
    }
    return false;
}

struct ChiArgs {
    const int32_t *row_ptr, *col, *src, *tau;
    int32_t n, nsrc, ell, gamma;
    const double *cval, *cmin, *cmax;
    const int32_t *cid;
    double eps, log_2m_delta;
    long long *walk_count;   // per CSR entry (0 = no walks)
    long long *rhs;          // [0] sum of the launch's walk counts (Eq. 14 right side), [1] left side, [2] walk steps
    const long long *cvol;   // per column: frontier volume
    int32_t *src_chunks;     // per column: chunks of kWalkChunk walk pairs of its entries
};

constexpr int kWalkChunk = 128;  // walk pairs per warp-sized chunk

__host__ __device__ __forceinline__ long long walk_chunks(long long pairs) {
    return pairs > 0 ? (pairs + kWalkChunk - 1) / kWalkChunk : 0;
}

// Source s of column q, by a CTA of kChiScanThreads threads: rho_hat (Alg. 3) and
// min / max of p over N(s), into stat[3 q .. 3 q + 2]; cv / ci: the column's
// top-gamma list. Also counts the column's frontier volume into Eq. 14's left side.
template <typename T, int B, typename CV>
__device__ __forceinline__ void source_stats(const T *__restrict__ x, const ChiArgs &a, int32_t q, int32_t s,
                                             const CV *cv, const int32_t *ci, long long volume,
                                             double *__restrict__ stat) {
    using V = typename AccOf<T>::type;
    constexpr int NT = kChiScanThreads, NW = NT / 32;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const T *xs = x + static_cast<int64_t>(q / B) * a.n * B + (q % B);
    const int g = a.gamma;
    // rho_hat = max(max over edges inside C of p(c_a) + p(c_b), p(c_1) + p(c_gamma))
    double best = -INFINITY;
    for (int e = t; e < g * g; e += NT) {
        const int u = e / g, v = e % g;
        if (u < v && has_edge(a.row_ptr, a.col, ci[u], ci[v]))
            best = fmax(best, __dadd_rn(static_cast<double>(cv[u]), static_cast<double>(cv[v])));
    }
    V nmin = V(INFINITY), nmax = V(-INFINITY);
    for (int32_t k = a.row_ptr[s] + t; k < a.row_ptr[s + 1]; k += NT) {
        const V v = to_acc(xs[static_cast<int64_t>(a.col[k]) * B]);
        nmin = min(nmin, v);
        nmax = max(nmax, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
        nmin = min(nmin, __shfl_xor_sync(0xffffffffu, nmin, o));
        nmax = max(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
    }
    __shared__ double wbest[NW];
    __shared__ V wmin[NW], wmax[NW];
    if (lane == 0) {
        wbest[warp] = best;
        wmin[warp] = nmin;
        wmax[warp] = nmax;
    }
    __syncthreads();
    if (t != 0) return;
    for (int w = 1; w < NW; ++w) {
        best = fmax(best, wbest[w]);
        nmin = min(nmin, wmin[w]);
        nmax = max(nmax, wmax[w]);
    }
    stat[3 * q] = g > 0 ? fmax(best, __dadd_rn(static_cast<double>(cv[0]), static_cast<double>(cv[g - 1]))) : 0.0;
    stat[3 * q + 1] = static_cast<double>(nmin);
    stat[3 * q + 2] = static_cast<double>(nmax);
    atomicAdd(reinterpret_cast<unsigned long long *>(a.rhs + 1), static_cast<unsigned long long>(volume));
}

// The full scan's last step: one CTA per column of the launch
template <typename T, int B>
__global__ void __launch_bounds__(kChiScanThreads)
    k_chi_source(const T *__restrict__ x, const ChiArgs a, double *__restrict__ stat) {
    const int32_t q = blockIdx.x;
    const int32_t s = a.src[q];
    if (threadIdx.x == 0) a.src_chunks[q] = 0;
    if (s < 0) return;
    source_stats<T, B>(x, a, q, s, a.cval + static_cast<int64_t>(q) * kGammaMax,
                       a.cid + static_cast<int64_t>(q) * kGammaMax, a.cvol[q], stat);
}

// A column from its tiles' statistics to its source's, one CTA per column of the
// launch. (1) min, max, volume and thr: thread t takes tiles t, t + 128, ... and
// keeps their largest maximum; thr = the gamma-th largest of those 128 maxima (0
// if fewer than gamma are positive): they are maxima of distinct tiles, so at
// least gamma tiles reach thr, every top-gamma entry is >= thr, and thr is at
// most the gamma-th largest tile maximum (a few more candidate tiles than that,
// no merge of sorted lists). (2) The candidates (entries >= thr in the tiles whose
// maximum reaches thr; for thr = 0 the positive entries of the tiles holding one,
// and the gamma smallest-id zero rows), then the top-kGammaMax list among them: up
// to kRankMax candidates by counting each one's betters (a thread per candidate,
// broadcast reads), more by sorted lists per thread and a tree of merges, whose
// chain of dependent shared-memory reads is the longer one below that. (3) The
// source's statistics. Latency bound: a CTA's dependent steps, not its bytes; as
// three kernels, the last with a warp per source and all lists merged, a test of
// 192 columns of a 40,000-node Barabasi-Albert graph took 81 us, so 62.
constexpr int kRankMax = 2 * kChiScanThreads;

template <typename T, int B>
__global__ void __launch_bounds__(kChiScanThreads)
    k_chi_column(int ntiles, const T *__restrict__ x, const ChiArgs a,
                 const typename AccOf<T>::type *__restrict__ tmax, const typename AccOf<T>::type *__restrict__ tmin,
                 const long long *__restrict__ tvol, double *__restrict__ cmin, double *__restrict__ cmax,
                 long long *__restrict__ cvol, double *__restrict__ stat) {
    using V = typename AccOf<T>::type;
    const int q = blockIdx.x, n = a.n, gamma = a.gamma;
    const int32_t s = a.src[q];
    const int slice = q / B, c = q % B, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) a.src_chunks[q] = 0;
    if (s < 0) return;
    constexpr int NT = kChiScanThreads, NW = kChiScanThreads / 32;
    const T *xs = x + static_cast<int64_t>(slice) * n * B + c;
    __shared__ V cand_v[kCandMax];
    __shared__ int32_t cand_i[kCandMax];
    __shared__ int ncand;
    __shared__ V sthr, top_v[kGammaMax];
    __shared__ int32_t top_i[kGammaMax];
    __shared__ long long volume;
    __shared__ V sv[kGammaMax * NT];
    __shared__ int32_t si[kGammaMax * NT];
    // ---- thr, min, max, volume ----
    {
        V *smax = sv, *smin = sv + NT;
        long long *svol = reinterpret_cast<long long *>(si);
        static_assert(sizeof(si) >= NT * sizeof(long long), "the lists' ids hold the threads' volumes");
        V vmax = V(-INFINITY), vmin = V(INFINITY);
        long long vol = 0;
        for (int p = t; p < ntiles; p += NT) {
            const int64_t o = (static_cast<int64_t>(slice) * ntiles + p) * B + c;
            vmax = max(vmax, tmax[o]);
            vmin = min(vmin, tmin[o]);
            vol += tvol[o];
        }
        smax[t] = vmax;
        smin[t] = vmin;
        svol[t] = vol;
        if (t == 0) {
            ncand = 0;
            sthr = V(0);
        }
        __syncthreads();
        // rank of each thread's maximum among the 128 (ties by thread index); rank gamma - 1 is thr
        int rank = 0;
        for (int u = 0; u < NT; ++u) rank += (smax[u] > vmax || (smax[u] == vmax && u < t)) ? 1 : 0;
        if (rank == gamma - 1 && vmax > V(0)) sthr = vmax;  // (gamma <= kGammaMax < NT)
        if (rank == 0) cmax[q] = static_cast<double>(vmax);
        for (int half = NT / 2; half > 0; half >>= 1) {
            if (t < half) {
                smin[t] = min(smin[t], smin[t + half]);
                svol[t] += svol[t + half];
            }
            __syncthreads();
        }
        if (t == 0) {
            cmin[q] = static_cast<double>(smin[0]);
            cvol[q] = volume = svol[0];
        }
        __syncthreads();
    }
    if (gamma <= 0) {  // no list: Eq. 15
        source_stats<T, B>(x, a, q, s, top_v, top_i, volume, stat);
        return;
    }
    const V thr = sthr;
    const bool zero_thr = !(thr > V(0));
    // candidates: each warp tests 32 tile maxima at once, then takes the tiles that reach thr
    // one by one, 32 rows at a time
    for (int pb = warp * 32; pb < ntiles; pb += NW * 32) {
        const int pl = pb + lane;
        const V tml = pl < ntiles ? tmax[(static_cast<int64_t>(slice) * ntiles + pl) * B + c] : V(-1);
        uint32_t tiles = __ballot_sync(0xffffffffu, zero_thr ? (tml > V(0)) : (tml >= thr));
        while (tiles) {  // warp-uniform
            const int p = pb + __ffs(tiles) - 1;
            tiles &= tiles - 1u;
            const int32_t r0 = p * kTileRows, r1 = min(n, r0 + kTileRows);
            constexpr int RR = kTileRows / 32;  // the tile's rows, 32 per round, loaded together
            V vals[RR];
#pragma unroll
            for (int u = 0; u < RR; ++u) {
                const int32_t r = r0 + u * 32 + lane;
                vals[u] = r < r1 ? to_acc(xs[static_cast<int64_t>(r) * B]) : V(-1);
            }
#pragma unroll
            for (int u = 0; u < RR; ++u) {
                const int32_t r = r0 + u * 32 + lane;
                const V v = vals[u];
                const bool take = zero_thr ? (v > V(0)) : (v >= thr);
                const uint32_t bal = __ballot_sync(0xffffffffu, take);
                int base = 0;
                if (lane == 0 && bal) base = atomicAdd(&ncand, __popc(bal));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (take) {
                    const int slot = base + __popc(bal & ((1u << lane) - 1u));
                    if (slot < kCandMax) {
                        cand_v[slot] = v;
                        cand_i[slot] = r;
                    }
                }
            }
        }
    }
    __syncthreads();
    if (zero_thr && warp == 0) {
        // the gamma smallest-id zero rows, in id order
        int need = gamma;
        for (int p = 0; p < ntiles && need > 0; ++p) {
            if (tmin[(static_cast<int64_t>(slice) * ntiles + p) * B + c] > V(0)) continue;
            const int32_t r0 = p * kTileRows, r1 = min(n, r0 + kTileRows);
            for (int32_t rb = r0; rb < r1 && need > 0; rb += 32) {
                const int32_t r = rb + lane;
                const bool z = r < r1 && to_acc(xs[static_cast<int64_t>(r) * B]) == V(0);
                uint32_t bal = __ballot_sync(0xffffffffu, z);
                int base = 0;
                while (bal && need > 0) {  // warp-uniform
                    const int l = __ffs(bal) - 1;
                    bal &= bal - 1u;
                    if (lane == 0) {
                        base = ncand;
                        if (base < kCandMax) {
                            cand_v[base] = V(0);
                            cand_i[base] = rb + l;
                        }
                        ncand = base + 1;
                    }
                    --need;
                }
                __syncwarp();
            }
        }
    }
    __syncthreads();
    const int count = ncand;
    if (count <= kRankMax) {
        if (t < kGammaMax) {
            top_v[t] = V(-INFINITY);
            top_i[t] = INT32_MAX;
        }
        __syncthreads();
        for (int e = t; e < count; e += NT) {
            const V v = cand_v[e];
            const int32_t i = cand_i[e];
            int rank = 0;
#pragma unroll 4
            for (int u = 0; u < count; ++u) rank += u != e && better(cand_v[u], cand_i[u], v, i) ? 1 : 0;
            if (rank < kGammaMax) {
                top_v[rank] = v;
                top_i[rank] = i;
            }
        }
    } else {
        V *val = sv + t;
        int32_t *id = si + t;
        for (int r = 0; r < kGammaMax; ++r) {
            val[r * NT] = V(-INFINITY);
            id[r * NT] = INT32_MAX;
        }
        V bv[kGammaMax];
        int32_t bi[kGammaMax];
#pragma unroll
        for (int r = 1; r < kGammaMax; ++r) {
            bv[r] = V(-INFINITY);
            bi[r] = INT32_MAX;
        }
        if (count <= kCandMax) {
            for (int e = t; e < count; e += NT) {
                bv[0] = cand_v[e];
                bi[0] = cand_i[e];
                merge_sorted(val, id, NT, bv, bi, 1);
            }
        } else {
            // too many ties at thr for the buffer: every row of the column
            for (int32_t r = t; r < n; r += NT) {
                bv[0] = to_acc(xs[static_cast<int64_t>(r) * B]);
                bi[0] = r;
                merge_sorted(val, id, NT, bv, bi, 1);
            }
        }
        __syncthreads();
        for (int half = NT / 2; half > 0; half >>= 1) {
            if (t < half) merge_sorted(val, id, NT, sv + t + half, si + t + half, NT);
            __syncthreads();
        }
        if (t < kGammaMax) {
            top_v[t] = sv[t * NT];
            top_i[t] = si[t * NT];
        }
    }
    __syncthreads();
    source_stats<T, B>(x, a, q, s, top_v, top_i, volume, stat);
}

// Per entry k = (i -> j) of source q = blockIdx.x, kChiEntries of them to a
// warp over a (source, entry range) grid so that a hub source spreads over many
// CTAs: for each, the lanes stride over N(j) for its smallest and largest value
// (in the block's arithmetic type), and then a lane per entry evaluates chi (Eq.
// 17, or Eq. 15 for gamma = 0) and R (Eq. 13) for the walk length L = tau_k -
// ell, so that the FP64 expressions, 100 instructions of 16 cycles, run once a
// warp. They follow the oracle's evaluation order (no FMA contraction).
constexpr int kChiEntries = 4;

template <typename T, int B>
__global__ void k_chi_entries(const T *__restrict__ x, const ChiArgs a, const double *__restrict__ stat) {
    using V = typename AccOf<T>::type;
    const int32_t q = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (q >= a.nsrc) return;
    const int32_t s = a.src[q];
    if (s < 0) return;
    const T *xs = x + static_cast<int64_t>(q / B) * a.n * B + (q % B);
    auto px = [&](int32_t v) { return to_acc(xs[static_cast<int64_t>(v) * B]); };
    const int g = a.gamma;
    const int32_t rb = a.row_ptr[s], re = a.row_ptr[s + 1];
    if (rb + static_cast<int32_t>(blockIdx.y) * nw * kChiEntries >= re) return;  // CTA-uniform
    __shared__ unsigned long long sh_cnt[3];
    if (threadIdx.x < 3) sh_cnt[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long local = 0, steps = 0, chunks = 0;
    for (int32_t k0 = rb + (static_cast<int32_t>(blockIdx.y) * nw + warp) * kChiEntries; k0 < re;
         k0 += static_cast<int32_t>(gridDim.y) * nw * kChiEntries) {
        const bool in = lane < kChiEntries && k0 + lane < re;
        const int32_t k = k0 + lane;
        const int32_t L = in ? a.tau[k] - a.ell : 0;
        const int32_t j = in ? a.col[k] : 0;
        V nmin_j = V(INFINITY), nmax_j = V(-INFINITY);
        if (g > 0) {
            const int32_t jb = in && L > 0 ? a.row_ptr[j] : 0, je = in && L > 0 ? a.row_ptr[j + 1] : 0;
#pragma unroll
            for (int e = 0; e < kChiEntries; ++e) {
                const int32_t b0 = __shfl_sync(0xffffffffu, jb, e), b1 = __shfl_sync(0xffffffffu, je, e);
                V lo = V(INFINITY), hi = V(-INFINITY);
#pragma unroll 4
                for (int32_t t = b0 + lane; t < b1; t += 32) {
                    const V v = px(a.col[t]);
                    lo = min(lo, v);
                    hi = max(hi, v);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                }
                if (lane == e) {
                    nmin_j = lo;
                    nmax_j = hi;
                }
            }
        }
        if (!in) continue;
        if (L <= 0) {
            a.walk_count[k] = 0;
            continue;
        }
        const double vmin = a.cmin[q], vmax = a.cmax[q];
        const double rho = stat[3 * q], nmin_i = stat[3 * q + 1], nmax_i = stat[3 * q + 2];
        const double d_i = static_cast<double>(re - rb);
        const double denom = __dmul_rn(__dmul_rn(__dmul_rn(d_i, d_i), a.eps), a.eps);
        double chi;
        if (g == 0) {
            chi = __dmul_rn(__dmul_rn(2.0, static_cast<double>(L)), __dsub_rn(vmax, vmin));  // Eq. 15
        } else {
            const double Lm1 = static_cast<double>(L - 1);
            const double lb_i = __dadd_rn(nmin_i, __dmul_rn(Lm1, vmin));
            const double lb_j = __dadd_rn(static_cast<double>(nmin_j), __dmul_rn(Lm1, vmin));
            const double tail = __ddiv_rn(__dmul_rn(Lm1, rho), 2.0);
            const double ub_i = __dadd_rn(__dadd_rn(__ddiv_rn(nmax_i, 2.0), __ddiv_rn(vmax, 2.0)), tail);
            const double ub_j =
                __dadd_rn(__dadd_rn(__ddiv_rn(static_cast<double>(nmax_j), 2.0), __ddiv_rn(vmax, 2.0)), tail);
            chi = __dsub_rn(__dsub_rn(__dadd_rn(ub_i, ub_j), lb_i), lb_j);  // Eq. 17
        }
        const double r = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(8.0, chi), chi), a.log_2m_delta), denom);
        const double rc = ceil(r);
        const long long R =
            rc < 1.0 ? 1 : (rc > static_cast<double>(kWalkCountCap) ? kWalkCountCap : static_cast<long long>(rc));
        a.walk_count[k] = R;
        local += static_cast<unsigned long long>(R);
        steps += static_cast<unsigned long long>(R) * 2ull * static_cast<unsigned long long>(L);
        chunks += static_cast<unsigned long long>(walk_chunks(R));
    }
    if (local) {
        atomicAdd(&sh_cnt[0], local);
        atomicAdd(&sh_cnt[1], steps);
        atomicAdd(&sh_cnt[2], chunks);
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh_cnt[0]) {
        atomicAdd(reinterpret_cast<unsigned long long *>(a.rhs), sh_cnt[0]);
        atomicAdd(reinterpret_cast<unsigned long long *>(a.rhs + 2), sh_cnt[1]);
        // (a count past 32 bits belongs to a test whose walks are not drawn)
        atomicAdd(&a.src_chunks[q], static_cast<int32_t>(min(sh_cnt[2], 0x7fffffffull)));
    }
}

struct WalkArgs {
    const int32_t *row_ptr, *col, *src, *tau;
    int32_t n, nsrc, tt;
    const long long *walk_count;
    uint32_t key0, key1;
};

// The walks of Algorithm 4's second phase run without the host: it knows their
// number from the test that chose them, which bounds the chunks, and the plan is
// made on the device: for 192 sources of a 40,000-node Barabasi-Albert graph the
// phase took 81 us planned on the host, of which its kernels 19, and takes 31 so
// (events on both sides included). The walks themselves are bound by the latency
// of a step's three dependent loads, so a pair's two walks advance together.

// The plan, one CTA per column of `list` (-1: draws none): its entries' chunks
// follow those of the columns before it, in CSR order. chunk0[k]: the first chunk
// of entry k; chunk_q / chunk_k: a chunk's column and entry; *total: all chunks.
static __global__ void __launch_bounds__(128) k_walk_plan(const int32_t *__restrict__ row_ptr,
                                                          const int32_t *__restrict__ list, int32_t nsrc,
                                                          const int32_t *__restrict__ src_chunks,
                                                          const long long *__restrict__ walk_count,
                                                          int32_t *__restrict__ chunk0, int32_t *__restrict__ chunk_q,
                                                          int32_t *__restrict__ chunk_k, int32_t *__restrict__ total) {
    __shared__ int32_t part[4], warp_sum[4];
    const int32_t q = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t before = 0;
    for (int32_t p = threadIdx.x; p < q; p += 128)
        if (list[p] >= 0) before += src_chunks[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lane == 0) part[warp] = before;
    __syncthreads();
    int32_t at = part[0] + part[1] + part[2] + part[3];
    const int32_t s = list[q];
    if (q == nsrc - 1 && threadIdx.x == 0) *total = at + (s >= 0 ? src_chunks[q] : 0);
    if (s < 0) return;
    const int32_t rb = row_ptr[s], re = row_ptr[s + 1];
    for (int32_t k0 = rb; k0 < re; k0 += 128) {  // CTA-uniform
        const int32_t k = k0 + static_cast<int32_t>(threadIdx.x);
        const int32_t mine = k < re ? static_cast<int32_t>(walk_chunks(walk_count[k])) : 0;
        int32_t inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t up = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += up;
        }
        if (lane == 31) warp_sum[warp] = inc;
        __syncthreads();
        int32_t here = at + inc - mine;
        for (int w = 0; w < warp; ++w) here += warp_sum[w];
        if (k < re) chunk0[k] = here;
        for (uint32_t todo = __ballot_sync(0xffffffffu, mine > 0); todo; todo &= todo - 1u) {  // warp-uniform
            const int l = __ffs(todo) - 1;
            const int32_t first = __shfl_sync(0xffffffffu, here, l), count = __shfl_sync(0xffffffffu, mine, l);
            const int32_t kl = __shfl_sync(0xffffffffu, k, l);
            for (int32_t c = lane; c < count; c += 32) {
                chunk_q[first + c] = q;
                chunk_k[first + c] = kl;
            }
        }
        at += warp_sum[0] + warp_sum[1] + warp_sum[2] + warp_sum[3];
        __syncthreads();
    }
}

struct WalkChunkArgs {
    const int32_t *chunk_q, *chunk_k, *chunk0;  // of k_walk_plan
    const int32_t *total;                       // chunks
    double *chunk_sum;                          // per chunk: sum over its walks of (S_i - S_j)
};

// Walk pair w of entry k: sum_{t=1..L} X[W[t]] from both ends (Eq. 11), their difference
template <typename T, int B>
__device__ __forceinline__ double walk_pair(const WalkArgs &a, const T *__restrict__ xs, int32_t i, int32_t j,
                                            int32_t L, uint32_t k, uint32_t w) {
    int32_t cur[2] = {i, j};
    double sum[2] = {0.0, 0.0};
    Philox4 words[2] = {};
    for (int32_t t = 1; t <= L; ++t) {
        const int r = (t - 1) & 3;
        if (r == 0) {
#pragma unroll
            for (uint32_t side = 0; side < 2; ++side)
                words[side] = philox4x32_10(k, w, (side << 31) | static_cast<uint32_t>((t - 1) >> 2), kWalkTag, a.key0,
                                            a.key1);
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const int32_t b = a.row_ptr[cur[side]];
            const uint32_t d = static_cast<uint32_t>(a.row_ptr[cur[side] + 1] - b);
            const uint32_t word = r == 0 ? words[side].v[0] : r == 1 ? words[side].v[1]
                                : r == 2 ? words[side].v[2] : words[side].v[3];
            cur[side] = a.col[b + static_cast<uint32_t>((static_cast<uint64_t>(word) * d) >> 32)];
        }
#pragma unroll
        for (int side = 0; side < 2; ++side)
            sum[side] += static_cast<double>(to_acc(xs[static_cast<int64_t>(cur[side]) * B]));
    }
    return sum[0] - sum[1];
}

// One warp per chunk of walk pairs of one entry; lanes take walks w0 + lane,
// w0 + lane + 32, ... in the chunk; the chunk sum is reduced by a fixed tree.
template <typename T, int B>
__global__ void k_walk_chunks(const T *__restrict__ x, const WalkArgs a, const WalkChunkArgs c) {
    const int64_t ch = blockIdx.x * static_cast<int64_t>(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (ch >= *c.total) return;
    const int32_t q = c.chunk_q[ch], k = c.chunk_k[ch];
    const int32_t s = a.src[q];
    const T *xs = x + static_cast<int64_t>(q / B) * a.n * B + (q % B);
    const long long R = a.walk_count[k];
    const long long w0 = (ch - c.chunk0[k]) * kWalkChunk;
    const long long w1 = min(R, w0 + kWalkChunk);
    const int32_t L = a.tau[k] - a.tt;
    const int32_t j = a.col[k];
    double acc = 0.0;
    for (long long w = w0 + lane; w < w1; w += 32)
        acc += walk_pair<T, B>(a, xs, s, j, L, static_cast<uint32_t>(k), static_cast<uint32_t>(w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) c.chunk_sum[ch] = acc;
}

// g[k] += (sum of the entry's chunk sums, in chunk order) / R_k  (Algorithm 4's
// walk estimate); one CTA per column of `list`
static __global__ void __launch_bounds__(128) k_walk_finish(const int32_t *__restrict__ row_ptr,
                                                            const int32_t *__restrict__ list,
                                                            const int32_t *__restrict__ chunk0,
                                                            const double *__restrict__ chunk_sum,
                                                            const long long *__restrict__ walk_count,
                                                            double *__restrict__ g) {
    const int32_t s = list[blockIdx.x];
    if (s < 0) return;
    for (int32_t k = row_ptr[s] + static_cast<int32_t>(threadIdx.x); k < row_ptr[s + 1]; k += 128) {
        const long long R = walk_count[k];
        if (R <= 0) continue;
        const int32_t c0 = chunk0[k], c1 = c0 + static_cast<int32_t>(walk_chunks(R));
        double t = 0.0;
        for (int32_t ch = c0; ch < c1; ++ch) t += chunk_sum[ch];
        g[k] += t / static_cast<double>(R);
    }
}

// Per source (one warp each; 0 for an empty slot): out[q] = Eq. 14's right side,
// the sum of the walk counts of its entries; out[nsrc + q] = their walk steps
// 2 R (tau_k - ell)
static __global__ void k_walks_per_source(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ src,
                                          int32_t nsrc, const long long *__restrict__ walk_count,
                                          const int32_t *__restrict__ tau, int32_t ell, long long *__restrict__ out) {
    const int32_t q = blockIdx.x;
    const int lane = threadIdx.x & 31;
    if (q >= nsrc) return;
    const int32_t s = src[q];
    long long acc = 0, steps = 0;
    if (s >= 0)
        for (int32_t k = row_ptr[s] + lane; k < row_ptr[s + 1]; k += 32) {
            const long long R = walk_count[k];
            const int32_t L = tau[k] - ell;
            acc += R;
            if (R > 0 && L > 0) steps += 2ll * R * static_cast<long long>(L);
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        steps += __shfl_xor_sync(0xffffffffu, steps, o);
    }
    if (lane == 0) {
        out[q] = acc;
        out[nsrc + q] = steps;
    }
}

// tau[k] = min(tau[k], cap) over the rows of the listed nodes (entries < 0
// skipped): a source that switched to walks at hop cap gathers no later hop
static __global__ void k_cap_rows(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ list,
                                  int32_t count, int32_t cap, int32_t *__restrict__ tau) {
    const int32_t q = blockIdx.x;
    if (q >= count) return;
    const int32_t v = list[q];
    if (v < 0) return;
    for (int32_t k = row_ptr[v] + static_cast<int32_t>(threadIdx.x); k < row_ptr[v + 1]; k += blockDim.x)
        tau[k] = min(tau[k], cap);
}

}  // namespace sc
