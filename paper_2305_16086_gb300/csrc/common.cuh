// Internal helpers shared by the libsc translation units (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdarg>
#include <cstdio>
#include <map>
#include <set>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/sc.h"

namespace sc {

// ---------------------------------------------------------------------------
// Error reporting: every ABI call returns a status; the detail string is
// thread-local and describes the last failing call of the calling thread.
// ---------------------------------------------------------------------------
void set_detail(const char *fmt, ...);
void clear_detail();

struct Failure {
    sc_status status;
};

#define SC_CUDA(call)                                                                     \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) {                                                          \
            ::sc::set_detail("%s:%d %s: %s", __FILE__, __LINE__, #call,                   \
                             cudaGetErrorString(e_));                                     \
            throw ::sc::Failure{e_ == cudaErrorMemoryAllocation ? SC_ERR_OOM : SC_ERR_CUDA}; \
        }                                                                                 \
    } while (0)

#define SC_FAIL(status, ...)                     \
    do {                                         \
        ::sc::set_detail(__VA_ARGS__);           \
        throw ::sc::Failure{status};             \
    } while (0)

#define SC_LAUNCH_CHECK() SC_CUDA(cudaGetLastError())

// Wraps the body of an ABI function: converts Failure / std::bad_alloc into
// a status so no exception leaves the library.
template <typename F>
sc_status guarded(F &&body) {
    try {
        clear_detail();
        body();
        return SC_OK;
    } catch (const Failure &f) {
        return f.status;
    } catch (const std::bad_alloc &) {
        set_detail("host allocation failed");
        return SC_ERR_OOM;
    } catch (...) {
        set_detail("unexpected internal error");
        return SC_ERR_CUDA;
    }
}

// ---------------------------------------------------------------------------
// Device buffer with RAII ownership (plain cudaMalloc / cudaFree).
// ---------------------------------------------------------------------------
template <typename T>
struct DevBuf {
    T *ptr = nullptr;
    size_t count = 0;
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
    ~DevBuf() { release(); }
    void release() {
        if (ptr) cudaFree(ptr);
        ptr = nullptr;
        count = 0;
    }
    // grow-only: keeps the old allocation if it is large enough
    void reserve(size_t n) {
        if (n <= count && ptr) return;
        release();
        if (n == 0) return;
        SC_CUDA(cudaMalloc(reinterpret_cast<void **>(&ptr), n * sizeof(T)));
        count = n;
    }
    T *get() const { return ptr; }
};

// ---------------------------------------------------------------------------
// Element types of the propagated block.
// ---------------------------------------------------------------------------
template <typename T>
struct AccOf {
    using type = float;
};
template <>
struct AccOf<double> {
    using type = double;
};

__device__ __forceinline__ float to_acc(float v) { return v; }
__device__ __forceinline__ double to_acc(double v) { return v; }
__device__ __forceinline__ float to_acc(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T>
__device__ __forceinline__ T from_acc(typename AccOf<T>::type v);
template <>
__device__ __forceinline__ float from_acc<float>(float v) { return v; }
template <>
__device__ __forceinline__ double from_acc<double>(double v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_acc<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

inline int ceil_div(long long a, long long b) { return static_cast<int>((a + b - 1) / b); }

// a launch shape of the propagation: block width, 16-byte vectors per lane
// (0 = the TMA-gather kernel) and the measured time of one hop per source
struct TuneResult {
    int B, vpl;
    double ms_per_source_hop;
};

}  // namespace sc

// ---------------------------------------------------------------------------
// The graph object behind the opaque sc_graph handle.
// ---------------------------------------------------------------------------
struct sc_graph {
    int device = 0;
    cudaStream_t stream = nullptr;
    int32_t n = 0;
    int64_t nnz = 0;
    int32_t min_degree = 0, max_degree = 0;
    int32_t bipartite = 0;
    int32_t bfs_depth = 0;
    int num_sms = 0;
    size_t l2_bytes = 0;

    sc::DevBuf<int32_t> row_ptr, col_idx, rev, level;
    sc::DevBuf<float> inv_deg_f;
    sc::DevBuf<double> inv_deg_d;
    std::vector<int32_t> h_row_ptr;  // host copy of the row pointers (degrees, scheduling)

    std::vector<int32_t> h_walk2;    // per node: sum of its neighbours' degrees, empty until needed

    // row schedule of the SIMT propagation kernel: heavy rows (degree above
    // the threshold, one CTA each, longest first) then light rows in order
    sc::DevBuf<int32_t> row_order;
    int32_t heavy_threshold_cached = -1;
    int32_t n_heavy = 0;
    // the heavy rows again, sorted by id (windowed launches), and on the host
    sc::DevBuf<int32_t> heavy_ids;
    std::vector<int32_t> h_heavy_ids;
    // bandwidth max |i - j| over the entries (i -> j); -1 until computed
    int32_t bandwidth = -1;
    // per-slice windows of windowed launches
    sc::DevBuf<unsigned char> win_list;
    // bit mask of the block's first-hop rows (hop 2 from the sources alone); behind it the
    // non-zero columns of X_2 and the counters of the sparse hops
    sc::DevBuf<uint32_t> mask;
    // the sparse hops: chunks of the long rows and runs of the others (laid out once), partial sums, X_2's
    // sector masks, the work lists of the ball hop
    sc::DevBuf<int32_t> fr_hi_row, fr_hi_k0, fr_hv_id, fr_hv_first, fr_run_lo, fr_run_hi, fr_rows;
    sc::DevBuf<uint32_t> fr_pairs;
    sc::DevBuf<unsigned char> fr_part, fr_sec;
    int32_t front_hchunks = 0, front_hrows = 0, front_runs = 0;
    int32_t front_pair_rows[3] = {0, 0, 0};  // rows of up to 1, 2 and 4 chunks
    bool front_ready = false;
    // row runs of about equal CSR entries, one per warp, for the TMA kernel
    sc::DevBuf<int32_t> part;
    int32_t nparts = 0;
    int32_t part_target = -1;
    // autotuned (block width, lane split) per request key, and its measured ms per source-hop
    std::map<long long, std::pair<int, int>> tuned;
    std::map<long long, double> tuned_cost;
    // per request key: the best lane split of each block width, and the launch shape chosen
    // by timing one real block of each (the block loop's own kernels, see pick_block_width)
    std::map<long long, std::vector<sc::TuneResult>> tuned_per_b;
    std::map<long long, sc::TuneResult> tuned_block;

    // learned length: features (n x 6) and the loaded model
    sc::DevBuf<float> features, mlp;
    bool features_ready = false, mlp_loaded = false;

    // cached eigenvalue estimate
    bool has_lambda = false;
    sc_lambda lam{};

    // CalTau: the pairs of the last sc_eigenpairs (f_k node-major, n x eig_P,
    // their eigenvalues and the bound r on the rest) and the last sc_caltau lengths
    sc::DevBuf<double> eig_Fn;
    std::vector<double> eig_lam;
    double eig_rest = 1.0;
    int32_t eig_P = 0;
    bool eig_ready = false;
    sc::DevBuf<int32_t> caltau_tau;
    double caltau_eps = 0.0;
    bool caltau_ready = false;

    // work buffers (grow-only)
    sc::DevBuf<unsigned char> xa, xb;   // probability blocks
    sc::DevBuf<double> acc_g, acc_t1, acc_t2;
    sc::DevBuf<int32_t> tau_entry, src_list, status;
    sc::DevBuf<double> scratch_d;
    // sc_all_edges / sc_some_edges: a cudaMalloc and its cudaFree cost a small query more than its
    // kernels (16 edges of a 400-node graph: 216 us with, 201 us without)
    sc::DevBuf<int32_t> ws_tau_src, ws_active, ws_flag, ws_rows;
    sc::DevBuf<int64_t> ws_entries;
    sc::DevBuf<double> ws_pre, ws_s, ws_b, ws_sub_s, ws_sub_b;
    // TGT+ work buffers: CalChi partial and per-column statistics, walk counts
    sc::DevBuf<double> tp_pval, tp_pmin, tp_pmax, tp_cval, tp_cmin, tp_cmax;
    sc::DevBuf<int32_t> tp_pid, tp_cid;
    sc::DevBuf<long long> tp_pvol, tp_cvol, tp_walks, tp_counters;
    sc::DevBuf<int32_t> tp_src_chunks, tp_chunk0;  // per column, per CSR entry: chunks of walks, the first one
    sc::DevBuf<int32_t> tp_chunk_q, tp_chunk_k;    // per chunk: its column and CSR entry
    sc::DevBuf<double> tp_chunk_sum;
    sc::DevBuf<double> tp_srcstat;  // per column: rho_hat, min and max of p over N(s)
    sc::DevBuf<long long> tp_src_rhs;  // per column: Eq. 14's right side (per-source switch)
    sc::DevBuf<int32_t> tp_cap_list;   // the sources that switch at a test (per-source switch)
    // resident traversal (resident.cu): neighbour ids in rows of res_width, the
    // groups of sources per kind of segment (0: bipartite, 1: not), work lists
    sc::DevBuf<int32_t> res_ell, res_len, res_list, res_over, res_single, res_order_dev[2];
    sc::DevBuf<unsigned long long> res_count;
    std::vector<int32_t> res_order[2];
    int res_order_width[2] = {0, 0};
    int res_width = 0;
    bool res_ready = false;
    // what samples of its balls said, by (fp64, longest and mean run): the first class, and whether
    // the class without the adjacency pays
    std::map<std::tuple<bool, int32_t, int32_t>, int> res_first, res_global;
    // as a member of batches: (fp64, hops) of runs in which none of its sources ran resident
    std::set<std::pair<bool, int32_t>> res_batch_none;
    sc::DevBuf<unsigned char> res_scratch;
    sc::DevBuf<uint16_t> res_marks;  // per CTA a local id per node, 0xffff between launches
    std::vector<cudaEvent_t> hop_events;  // pairs bracketing timed propagation launches
    std::vector<cudaEvent_t> walk_events;  // pairs bracketing TGT+ walk phases
    long long *h_counters = nullptr;       // page-locked: a switch test's sums
    ~sc_graph() {
        for (cudaEvent_t e : hop_events) cudaEventDestroy(e);
        for (cudaEvent_t e : walk_events) cudaEventDestroy(e);
        if (h_counters) cudaFreeHost(h_counters);
    }
};

namespace sc {
void ensure_row_order(sc_graph *g, int32_t heavy_threshold);
int32_t ensure_bandwidth(sc_graph *g);
void ensure_partition(sc_graph *g, int32_t target);
void fill_i32(int32_t *p, int64_t count, int32_t v, cudaStream_t s);
}
