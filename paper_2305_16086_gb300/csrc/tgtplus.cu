// Host side of TGT+ (Algorithm 4): the switch test of Eq. 14 after a hop and
// the random-walk tail, dispatched over (precision, B).
#include <algorithm>
#include <cmath>

#include "tgtplus.cuh"

namespace sc {

template <typename T, int B>
static void chi_check_t(sc_graph *g, const void *x, int slices, const int32_t *src, int nsrc, int max_deg,
                        const int32_t *tau, int ell, int gamma, double eps, double log2md, bool full_scan,
                        cudaStream_t s) {
    gamma = std::min(gamma, g->n);  // a list holds the graph's nodes at most
    const int ncols = slices * B;
    double *pmin = g->tp_pmin.get(), *pmax = g->tp_pmax.get();
    long long *pvol = g->tp_pvol.get();
    ChiArgs a{};
    a.row_ptr = g->row_ptr.get();
    a.col = g->col_idx.get();
    a.src = src;
    a.tau = tau;
    a.n = g->n;
    a.nsrc = nsrc;
    a.ell = ell;
    a.gamma = gamma;
    a.cval = g->tp_cval.get();
    a.cmin = g->tp_cmin.get();
    a.cmax = g->tp_cmax.get();
    a.cid = g->tp_cid.get();
    a.eps = eps;
    a.log_2m_delta = log2md;
    a.walk_count = g->tp_walks.get();
    a.rhs = g->tp_counters.get();
    a.cvol = g->tp_cvol.get();
    a.src_chunks = g->tp_src_chunks.get();
    if (full_scan) {
        // every row of a column through a sorted list per 64-row tile, lists merged per column
        const int nct = ceil_div(g->n, kChiRowsPerCta);
        k_chi_scan<T, B><<<dim3(nct, slices), kChiScanThreads, 0, s>>>(
            g->row_ptr.get(), static_cast<const T *>(x), g->n, g->tp_pval.get(), g->tp_pid.get(), pmin, pmax, pvol);
        k_chi_merge<B><<<ncols, kChiScanThreads, 0, s>>>(nct, ncols, g->tp_pval.get(), g->tp_pid.get(), pmin, pmax,
                                                            pvol, g->tp_cval.get(), g->tp_cid.get(), g->tp_cmin.get(),
                                                            g->tp_cmax.get(), g->tp_cvol.get());
        k_chi_source<T, B><<<nsrc, kChiScanThreads, 0, s>>>(static_cast<const T *>(x), a, g->tp_srcstat.get());
    } else {
        // tile maxima, then per column the threshold and the candidates at or above it
        using V = typename AccOf<T>::type;
        const int ntiles = ceil_div(g->n, kTileRows);
        V *tmax = reinterpret_cast<V *>(pmax), *tmin = reinterpret_cast<V *>(pmin);  // room for doubles
        k_chi_tiles<T, B><<<dim3(ntiles, slices), kChiScanThreads, 0, s>>>(g->row_ptr.get(),
                                                                          static_cast<const T *>(x), g->n, tmax,
                                                                          tmin, pvol);
        k_chi_column<T, B><<<nsrc, kChiScanThreads, 0, s>>>(ntiles, static_cast<const T *>(x), a, tmax, tmin, pvol,
                                                               g->tp_cmin.get(), g->tp_cmax.get(), g->tp_cvol.get(),
                                                               g->tp_srcstat.get());
    }
    const int nw = 256 / 32;
    dim3 grid(nsrc, std::min(ceil_div(std::max(max_deg, 1), nw * kChiEntries), 65535));
    k_chi_entries<T, B><<<grid, 256, 0, s>>>(static_cast<const T *>(x), a, g->tp_srcstat.get());
}

template <typename T, int B>
static void walks_t(sc_graph *g, const void *x, const int32_t *src, int nsrc, const int32_t *tau, int tt,
                    uint64_t seed, const WalkChunkArgs &c, int64_t max_chunks, cudaStream_t s) {
    WalkArgs a{};
    a.row_ptr = g->row_ptr.get();
    a.col = g->col_idx.get();
    a.src = src;
    a.tau = tau;
    a.n = g->n;
    a.nsrc = nsrc;
    a.tt = tt;
    a.walk_count = g->tp_walks.get();
    a.key0 = static_cast<uint32_t>(seed);
    a.key1 = static_cast<uint32_t>(seed >> 32);
    k_walk_chunks<T, B><<<ceil_div(max_chunks, 8), 256, 0, s>>>(static_cast<const T *>(x), a, c);
}

#define SC_DISPATCH_TB(prec, B, FN, ...)                                                   \
    do {                                                                                   \
        if ((prec) == SC_PREC_FP64) {                                                      \
            if ((B) == 32) FN<double, 32>(__VA_ARGS__);                                    \
            else if ((B) == 64) FN<double, 64>(__VA_ARGS__);                               \
            else FN<double, 128>(__VA_ARGS__);                                             \
        } else if ((prec) == SC_PREC_FP32) {                                               \
            if ((B) == 32) FN<float, 32>(__VA_ARGS__);                                     \
            else if ((B) == 64) FN<float, 64>(__VA_ARGS__);                                \
            else FN<float, 128>(__VA_ARGS__);                                              \
        } else {                                                                           \
            if ((B) == 32) FN<__nv_bfloat16, 32>(__VA_ARGS__);                             \
            else if ((B) == 64) FN<__nv_bfloat16, 64>(__VA_ARGS__);                        \
            else FN<__nv_bfloat16, 128>(__VA_ARGS__);                                      \
        }                                                                                  \
    } while (0)

void tgtplus_reserve(sc_graph *g, int slices, int B) {
    const int nct = ceil_div(g->n, kChiRowsPerCta);
    const size_t cols = static_cast<size_t>(slices) * B;
    g->tp_pval.reserve(cols * nct * kGammaMax);
    g->tp_pid.reserve(cols * nct * kGammaMax);
    g->tp_pmin.reserve(cols * nct);
    g->tp_pmax.reserve(cols * nct);
    g->tp_pvol.reserve(cols * nct);
    g->tp_cval.reserve(cols * kGammaMax);
    g->tp_cid.reserve(cols * kGammaMax);
    g->tp_cmin.reserve(cols);
    g->tp_cmax.reserve(cols);
    g->tp_cvol.reserve(cols);
    g->tp_srcstat.reserve(3 * cols);
    g->tp_src_rhs.reserve(2 * cols);
    g->tp_src_chunks.reserve(cols + 1);  // and their total
    g->tp_cap_list.reserve(cols);
    g->tp_walks.reserve(g->nnz);
    g->tp_chunk0.reserve(g->nnz);
    g->tp_counters.reserve(4);
    if (!g->h_counters) SC_CUDA(cudaMallocHost(reinterpret_cast<void **>(&g->h_counters), 4 * sizeof(long long)));
}

// Eq. 14 after hop `ell` for the launch's sources: returns the two sides
// (frontier volume, sum of walk counts); the per-entry walk counts for
// L = tau_k - ell stay in g->tp_walks for the walk kernel, and *steps is their
// number of walk steps. per_source (may be null): the two sides and the walk
// steps per source (nsrc each, in turn).
void tgtplus_check(sc_graph *g, int prec, int B, const void *x, int slices, const int32_t *src, const int32_t *h_src,
                   int nsrc, const int32_t *tau, int ell, int gamma, double eps, double log2md, bool full_scan,
                   long long *lhs, long long *rhs, long long *steps, cudaStream_t s,
                   std::vector<long long> *per_source) {
    SC_CUDA(cudaMemsetAsync(g->tp_counters.get(), 0, 4 * sizeof(long long), s));
    int max_deg = 0;
    for (int q = 0; q < nsrc; ++q)
        if (h_src[q] >= 0) max_deg = std::max(max_deg, g->h_row_ptr[h_src[q] + 1] - g->h_row_ptr[h_src[q]]);
    SC_DISPATCH_TB(prec, B, chi_check_t, g, x, slices, src, nsrc, max_deg, tau, ell, gamma, eps, log2md, full_scan, s);
    SC_LAUNCH_CHECK();
    SC_CUDA(cudaMemcpyAsync(g->h_counters, g->tp_counters.get(), 3 * sizeof(long long), cudaMemcpyDeviceToHost, s));
    if (per_source) {
        per_source->assign(3 * static_cast<size_t>(nsrc), 0);
        k_walks_per_source<<<nsrc, 32, 0, s>>>(g->row_ptr.get(), src, nsrc, g->tp_walks.get(), tau, ell,
                                               g->tp_src_rhs.get());
        SC_LAUNCH_CHECK();
        SC_CUDA(cudaMemcpyAsync(per_source->data(), g->tp_cvol.get(), nsrc * sizeof(long long), cudaMemcpyDeviceToHost, s));
        SC_CUDA(cudaMemcpyAsync(per_source->data() + nsrc, g->tp_src_rhs.get(), 2 * nsrc * sizeof(long long),
                                cudaMemcpyDeviceToHost, s));
    }
    SC_CUDA(cudaStreamSynchronize(s));
    if (per_source)
        for (int q = 0; q < nsrc; ++q)
            if (h_src[q] < 0) (*per_source)[q] = 0;
    *rhs = g->h_counters[0];
    *lhs = g->h_counters[1];
    *steps = g->h_counters[2];
}

// Algorithm 4's walk phase for the launch's sources, or (now not null, on the
// host) those of them it lists, -1 for the others: the entries' walk pairs are cut
// into chunks of kWalkChunk, one warp per chunk, and each entry adds its chunk
// sums in chunk order. pairs: their walk pairs, from the test. Nothing waits for
// the host.
void tgtplus_walks(sc_graph *g, int prec, int B, const void *x, const int32_t *src, const int32_t *h_src, int nsrc,
                   const int32_t *now, long long pairs, const int32_t *tau, int tt, uint64_t seed, double *acc_g,
                   cudaStream_t s) {
    if (pairs <= 0) return;
    int64_t max_chunks = pairs / kWalkChunk;  // an entry's last chunk may be short
    for (int q = 0; q < nsrc; ++q) {
        const int32_t v = now ? now[q] : h_src[q];
        if (v >= 0) max_chunks += g->h_row_ptr[v + 1] - g->h_row_ptr[v];
    }
    if (max_chunks > INT32_MAX) SC_FAIL(SC_ERR_UNSUPPORTED, "too many walks in a launch");
    if (static_cast<size_t>(max_chunks) > g->tp_chunk_sum.count) {  // with room for the launches to come
        const size_t room = static_cast<size_t>(max_chunks) + static_cast<size_t>(max_chunks) / 2;
        g->tp_chunk_q.reserve(room);
        g->tp_chunk_k.reserve(room);
        g->tp_chunk_sum.reserve(room);
    }
    const int32_t *list = src;
    if (now) {
        SC_CUDA(cudaMemcpyAsync(g->tp_cap_list.get(), now, nsrc * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        list = g->tp_cap_list.get();
    }
    int32_t *total = g->tp_src_chunks.get() + g->tp_src_chunks.count - 1;
    k_walk_plan<<<nsrc, 128, 0, s>>>(g->row_ptr.get(), list, nsrc, g->tp_src_chunks.get(), g->tp_walks.get(),
                                     g->tp_chunk0.get(), g->tp_chunk_q.get(), g->tp_chunk_k.get(), total);
    SC_LAUNCH_CHECK();
    WalkChunkArgs c{g->tp_chunk_q.get(), g->tp_chunk_k.get(), g->tp_chunk0.get(), total, g->tp_chunk_sum.get()};
    SC_DISPATCH_TB(prec, B, walks_t, g, x, src, nsrc, tau, tt, seed, c, max_chunks, s);
    SC_LAUNCH_CHECK();
    k_walk_finish<<<nsrc, 128, 0, s>>>(g->row_ptr.get(), list, g->tp_chunk0.get(), g->tp_chunk_sum.get(),
                                       g->tp_walks.get(), acc_g);
    SC_LAUNCH_CHECK();
}

// Caps tau at `cap` on the rows of the listed nodes (host list of count, -1 = skip).
void tgtplus_cap_rows(sc_graph *g, const int32_t *h_list, int count, int32_t cap, int32_t *tau, cudaStream_t s) {
    SC_CUDA(cudaMemcpyAsync(g->tp_cap_list.get(), h_list, count * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    k_cap_rows<<<count, 128, 0, s>>>(g->row_ptr.get(), g->tp_cap_list.get(), count, cap, tau);
    SC_LAUNCH_CHECK();
    SC_CUDA(cudaStreamSynchronize(s));  // h_list may be reused by the caller
}

}  // namespace sc
