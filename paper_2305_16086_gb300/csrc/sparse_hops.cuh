// The sparse ends of a block's traversal, for the single-graph block loop
// (Algorithm 2 visits only the nodes its frontier reaches): hop 2 from the
// sources' neighbour bits (k_front2), hop 3 from X_2's non-zero values
// (k_front3) and hop L - 1 on the sources' two-hop balls (k_ball), which the
// last hop reads. All keep k_spmm_hop's summation order (chunks of 32
// consecutive CSR entries summed in order, chunk sums added in chunk order, one
// scale by 1/d), so every value they store is bit for bit the full hop's; a
// value they skip is a zero, which changes no sum, or is never read.
//
// On a power-law graph (Barabasi-Albert, 200,000 nodes, 128 sources of middle
// ids) X_2 holds 0.5% non-zeros: half of a row's neighbours have none, the
// others 1.3 of their 16 sectors on average, and hop L - 1 is read at 114,000 of
// 25.6 M values. What is left is bound by round trips to L2 (ids, masks, values)
// and by instruction issue, so:
//  - X_2 is stored in the 32-byte sectors that hold a non-zero value only, with
//    a sector mask per row (two bytes for 128 FP32 columns) that hop 3 tests in
//    place of 512 bytes of values, and a bit per value for the ball hop;
//  - hop 2 goes through the entries of a run of rows as one stream and stops only
//    at the few that count;
//  - hop 3 gives a warp a row, 32 neighbours at a time, the ones with a non-zero
//    sector packed first; the next rows' bounds, ids and masks are in flight while
//    a row's values are;
//  - the ball hop works from lists of (row, column): a lane sums one chunk of at
//    most 32 entries, 1, 2, 4 or 8 lanes a value by the row's degree; rows with
//    many marked columns are computed whole;
//  - rows above kFrontHeavy entries are cut into chunks, one warp each, whose
//    sums the last of them to finish adds in order.
// Measured there, per block of 128 sources: hop 2 48 us (with the zeroing and the
// marks; full form 65), hop 3 88 us (full hop 137), the ball hop 54 us (137): a
// call at learned lengths 617 -> 359 ms. Hop 3 keeps no unit busy (issue 50%, L1
// 41%, L2 30%, DRAM 18%): it waits for loads across the two halves of L2 with 32
// warps per SM of 64 registers. Tried without gain: more loads in flight per warp
// (U = 6, 8: fewer warps), 40 warps with U = 4 (spills), a lane per sector and two
// rows per warp (as fast, fewer instructions), sectors fetched into L1 a row ahead
// (slower), a lane per chunk with accumulators in shared memory (587 us: the few
// neighbours with a hundred columns stall the other lanes).
#pragma once

#include <type_traits>

#include "propagate.cuh"

namespace sc {

constexpr int kFrontHeavy = 256;    // entries of a row; longer rows go chunk by chunk through partial sums
constexpr int kFrontRun = 192;      // entries of a run of rows
constexpr int kFrontRunRows = 8;    // and its rows: the sources' own rows, whose neighbours are all marked, set the longest run
constexpr int kBallSparseCols = 16; // marked columns of a row up to which they are computed one by one
constexpr int kBallLists = 5;       // pairs of rows of 1, 2, 3-4 and 5-8 chunks, and whole rows

// CPL = B/32 consecutive elements of a row: the share of one lane when a warp
// covers the B columns
template <typename T, int CPL>
struct alignas(CPL * sizeof(T)) LaneVec {
    T v[CPL];
};

template <int W>
__device__ __forceinline__ void load_words(const uint32_t *p, uint32_t *w) {
    if constexpr (W == 4) {
        const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p));
        w[0] = q.x, w[1] = q.y, w[2] = q.z, w[3] = q.w;
    } else if constexpr (W == 2) {
        const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
        w[0] = q.x, w[1] = q.y;
    } else {
        w[0] = __ldg(p);
    }
}

// a lane's vector from L2 (written by another SM during this launch)
template <typename V>
__device__ __forceinline__ V load_cg(const V *p) {
    V out;
    if constexpr (sizeof(V) >= 16) {
#pragma unroll
        for (size_t q = 0; q < sizeof(V) / 16; ++q) reinterpret_cast<uint4 *>(&out)[q] = __ldcg(reinterpret_cast<const uint4 *>(p) + q);
    } else if constexpr (sizeof(V) == 8) {
        *reinterpret_cast<uint2 *>(&out) = __ldcg(reinterpret_cast<const uint2 *>(p));
    } else {
        *reinterpret_cast<uint32_t *>(&out) = __ldcg(reinterpret_cast<const uint32_t *>(p));
    }
    return out;
}

// one bit per 32-byte sector of a row of X_2
template <typename T, int B>
struct SectorMask {
    static constexpr int COUNT = B * static_cast<int>(sizeof(T)) / 32;
    using Word = typename std::conditional<COUNT <= 8, uint8_t,
                                           typename std::conditional<COUNT <= 16, uint16_t, uint32_t>::type>::type;
    static_assert(COUNT <= 32, "sectors of a row");
};

template <typename T>
struct FrontArgs {
    using Acc = typename AccOf<T>::type;
    const int32_t *row_ptr, *col;
    const Acc *inv_deg;
    const T *x_prev;       // X_{l-1}, slices x n x B
    T *x_next;             // X_l
    // per slice, zeroed before hop 2: mask: bit b of row j marks j in N(s_b) (B/32 words a row);
    // nz: bit b of row j set iff X_2[j, b] != 0; any: bit j marks a row with a mask bit
    uint32_t *mask, *nz, *any;
    void *sectors;         // per slice and row: X_2's sector mask (SectorMask)
    int32_t n;
    int32_t light_ctas;
    // chunks of the rows above kFrontHeavy entries: heavy row index and first entry; per heavy row
    // its id and first chunk
    const int32_t *hi_row, *hi_k0, *hv_id, *hv_first;
    int32_t nhchunks, nhrows;
    // runs of consecutive rows without the heavy ones (kFrontRunRows, kFrontRun)
    const int32_t *run_lo, *run_hi;
    int32_t nruns;
    Acc *part;             // slices x nhchunks x B chunk sums
    int32_t *arrived;      // slices x nhrows (zeroed before hop 2, one set a hop)
    // work lists of hop L-1, per slice: pairs row * B + column by chunks of the row, rows (capacity n);
    // their lengths (zeroed before hop 2; nullable: none made). A row's kind is a matter of its degree, so
    // the four lists of pairs lie end to end, kBallSparseCols times the rows of each: pair_rows[k], the
    // rows of the kinds before k + 1
    uint32_t *pairs;       // slices x kBallSparseCols x n
    int32_t pair_rows[3];
    int32_t *rows;         // slices x n
    int32_t *lists;        // slices x kBallLists
    int32_t list_ctas;     // hop 3: CTAs that make them
    // fused gather of X_{l-1} (hop gather_ell) for the slice's sources, one CTA each
    int32_t gather_ctas;
    const int32_t *src;
    int32_t nsrc;
    const int32_t *tau;
    int32_t gather_ell;
    double *g, *t1, *t2;
    GatherRec rec;
};

// the list of pairs of one kind and slice
template <typename T>
__device__ __forceinline__ uint32_t *pair_list(const FrontArgs<T> &a, int kind, int64_t slice) {
    const int32_t before = kind == 0 ? 0 : kind == 1 ? a.pair_rows[0] : kind == 2 ? a.pair_rows[1] : a.pair_rows[2];
    return a.pairs + (slice * a.n + before) * kBallSparseCols;
}

// The chunk sums of a heavy row meet: the warp stores its E values per lane
// (lanes past B / E hold none), and the last warp of the row to arrive adds all
// of them in chunk order. Returns whether this warp did, with the row's total in
// tot[].
template <typename T, int B, int E>
__device__ __forceinline__ bool heavy_total(const FrontArgs<T> &a, int32_t hc, int32_t h,
                                            const typename AccOf<T>::type *chunk, typename AccOf<T>::type *tot) {
    using Acc = typename AccOf<T>::type;
    using Vec = LaneVec<Acc, E>;
    const int lane = threadIdx.x & 31;
    const bool on = lane < B / E;
    Acc *part = a.part + static_cast<int64_t>(blockIdx.y) * a.nhchunks * B + lane * E;
    Vec mine;
#pragma unroll
    for (int c = 0; c < E; ++c) mine.v[c] = chunk[c];
    if (on) *reinterpret_cast<Vec *>(part + static_cast<int64_t>(hc) * B) = mine;
    __threadfence();
    __syncwarp();
    const int32_t c0 = a.hv_first[h], c1 = a.hv_first[h + 1];
    int32_t got = 0;
    if (lane == 0) got = atomicAdd(a.arrived + static_cast<int64_t>(blockIdx.y) * a.nhrows + h, 1);
    got = __shfl_sync(0xffffffffu, got, 0);
    if (got != c1 - c0 - 1) return false;
    __threadfence();
#pragma unroll
    for (int c = 0; c < E; ++c) tot[c] = Acc(0);
    constexpr int U = 4;
    for (int32_t q = c0; q < c1 && on; q += U) {
        Vec v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (q + u < c1) v[u] = load_cg(reinterpret_cast<const Vec *>(part + static_cast<int64_t>(q + u) * B));
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (q + u < c1) {
#pragma unroll
                for (int c = 0; c < E; ++c) tot[c] += v[u].v[c];
            }
    }
    return true;
}

// marks N(s_b): bit b of mask[j], and bit j of any
template <int B>
__global__ void k_front_scatter(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                const int32_t *__restrict__ src, int32_t nsrc, uint32_t *__restrict__ mask,
                                uint32_t *__restrict__ any, int32_t n) {
    const int32_t q = blockIdx.x;
    if (q >= nsrc) return;
    const int32_t s = src[q];
    if (s < 0) return;
    const int b = q % B;
    uint32_t *m = mask + static_cast<int64_t>(q / B) * n * (B / 32) + b / 32;
    any += static_cast<int64_t>(q / B) * ((n + 31) / 32);
    for (int32_t k = row_ptr[s] + threadIdx.x; k < row_ptr[s + 1]; k += blockDim.x) {
        const int32_t j = col[k];
        atomicOr(m + static_cast<int64_t>(j) * (B / 32), 1u << (b % 32));
        atomicOr(any + j / 32, 1u << (j % 32));
    }
}

// ---------------------------------------------------------------------------
// Hop 2 from the neighbour bits: X_2[r, b] sums the stored 1/d_j over the
// neighbours j of r marked for b. Stores X_2's non-zero sectors, their masks and
// nz. CTAs [0, gather_ctas): the gather of hop 1; then a warp per heavy chunk;
// then a warp per run of at most kFrontRunRows rows and kFrontRun entries. A warp
// goes through its run's entries as one stream, testing each neighbour's bit of
// `any` (25 KB for 200,000 nodes, held by L1), and collects the few that pass;
// 32 of them at a time, their masks and 1/d are loaded together, and they are
// added in order, a lane per CPL columns, a row being stored when it ends.
// ---------------------------------------------------------------------------
template <typename T, int B>
__global__ void __launch_bounds__(kSpmmWarps * 32, 10) k_front2(const FrontArgs<T> a) {
    using Acc = typename AccOf<T>::type;
    using SM = SectorMask<T, B>;
    constexpr int W = B / 32, CPL = B / 32, GW = 32 / W;
    using Vec = LaneVec<T, CPL>;
    __shared__ int32_t hit_k[kSpmmWarps][64], hit_j[kSpmmWarps][64];
    __shared__ uint32_t hit_m[kSpmmWarps][32 * W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *__restrict__ row_ptr = a.row_ptr;
    const int32_t *__restrict__ col = a.col;
    auto x1 = [&](int32_t j) { return to_acc(from_acc<T>(a.inv_deg[j])); };  // the stored X_1 value
    if (static_cast<int32_t>(blockIdx.x) < a.gather_ctas) {
        const int32_t q = static_cast<int32_t>(blockIdx.y) * B + static_cast<int32_t>(blockIdx.x);
        if (q < a.nsrc) {
            const int32_t s = a.src[q];
            if (s >= 0)
                for (int32_t k = row_ptr[s] + threadIdx.x; k < row_ptr[s + 1]; k += blockDim.x)
                    gather_term(k, 0.0 - static_cast<double>(x1(col[k])), a.tau, 1, a.g, a.t1, a.t2, a.rec);
        }
        return;
    }
    const int32_t n = a.n;
    const int64_t slice = blockIdx.y;
    T *xn = a.x_next + slice * n * B;
    const uint32_t *__restrict__ mrow = a.mask + slice * n * W;
    const uint32_t *__restrict__ any = a.any + slice * ((n + 31) / 32);
    uint32_t *nz = a.nz + slice * n * W;
    typename SM::Word *sec = static_cast<typename SM::Word *>(a.sectors) + slice * n;
    const int lc0 = lane * CPL, lw = lane / GW, lshift = lc0 % 32;
    auto is_marked = [&](int32_t j) { return (__ldg(any + j / 32) >> (j % 32)) & 1u; };
    auto store_row = [&](int32_t r, Acc sc, const Acc *sum) {
        Vec out;
        uint32_t bits = 0u;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            out.v[c] = from_acc<T>(sum[c] * sc);
            bits |= (to_acc(out.v[c]) != Acc(0) ? 1u : 0u) << (lshift + c);
        }
        constexpr int LS = 32 / SM::COUNT;  // lanes of a sector
        uint32_t lanes = __ballot_sync(0xffffffffu, bits != 0u);
#pragma unroll
        for (int o = 1; o < LS; o <<= 1) lanes |= lanes >> o;  // bit LS q: sector q (higher lanes folded down)
        if ((lanes >> (lane / LS * LS)) & 1u) *reinterpret_cast<Vec *>(xn + static_cast<int64_t>(r) * B + lc0) = out;
        uint32_t word = 0u;
#pragma unroll
        for (int q = 0; q < SM::COUNT; ++q) word |= ((lanes >> (q * LS)) & 1u) << q;
#pragma unroll
        for (int o = GW / 2; o > 0; o >>= 1) bits |= __shfl_xor_sync(0xffffffffu, bits, o);
        if (lane % GW == 0) nz[static_cast<int64_t>(r) * W + lw] = bits;
        if (lane == 0) sec[r] = static_cast<typename SM::Word>(word);
    };
    // lane t: marked entry t's id; its mask words into hit_m, its stored X_1 value returned
    auto load_hits = [&](int32_t j, int count) -> Acc {
        __syncwarp();
        Acc x = Acc(0);
        if (lane < count) {
            uint32_t w[W];
            load_words<W>(mrow + static_cast<int64_t>(j) * W, w);
            x = x1(j);
#pragma unroll
            for (int q = 0; q < W; ++q) hit_m[warp][lane * W + q] = w[q];
        }
        __syncwarp();
        return x;
    };
    auto add_hit = [&](int t, Acc x, Acc *chunk) {
        const uint32_t m = hit_m[warp][t * W + lw];
        const Acc xv = __shfl_sync(0xffffffffu, x, t);
#pragma unroll
        for (int c = 0; c < CPL; ++c) chunk[c] += ((m >> (lshift + c)) & 1u) ? xv : Acc(0);
    };
    int32_t job = (static_cast<int32_t>(blockIdx.x) - a.gather_ctas) * kSpmmWarps + warp;
    if (job < a.nhchunks) {
        const int32_t h = a.hi_row[job], r = a.hv_id[h], k0 = a.hi_k0[job];
        const bool in = lane < row_ptr[r + 1] - k0;
        int32_t j = in ? col[k0 + lane] : 0;
        const uint32_t hit = __ballot_sync(0xffffffffu, in && is_marked(j));
        const int count = __popc(hit);
        j = __shfl_sync(0xffffffffu, j, __fns(hit, 0, lane + 1) & 31);  // the marked entries to the first lanes
        Acc chunk[CPL], tot[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) chunk[c] = Acc(0);
        const Acc x = load_hits(j, count);
        for (int t = 0; t < count; ++t) add_hit(t, x, chunk);
        if (heavy_total<T, B, CPL>(a, job, h, chunk, tot)) store_row(r, a.inv_deg[r], tot);
        return;
    }
    job -= a.nhchunks;
    if (job >= a.nruns) return;
    const int32_t r0 = a.run_lo[job], nr = a.run_hi[job] - r0;
    const int32_t lb = row_ptr[r0 + min(lane, nr)];  // first entry of row r0 + lane
    const int32_t kb = __shfl_sync(0xffffffffu, lb, 0), ke = row_ptr[r0 + nr];
    const Acc inv = lane < nr ? a.inv_deg[r0 + lane] : Acc(0);
    if (lane < nr) sec[r0 + lane] = 0;
    __syncwarp();
    Acc sum[CPL], chunk[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) sum[c] = chunk[c] = Acc(0);
    int cur = -1;  // row of the run * 8 + chunk being added
    auto close_chunk = [&] {
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            sum[c] += chunk[c];
            chunk[c] = Acc(0);
        }
    };
    auto close_row = [&] {
        if (cur < 0) return;
        close_chunk();
        store_row(r0 + cur / 8, __shfl_sync(0xffffffffu, inv, cur / 8), sum);
#pragma unroll
        for (int c = 0; c < CPL; ++c) sum[c] = Acc(0);
    };
    // the first `count` collected entries (all of them in order)
    auto take = [&](int count) {
        const int32_t k = lane < count ? hit_k[warp][lane] : 0, j = lane < count ? hit_j[warp][lane] : 0;
        int r = 0;  // the row of entry k
#pragma unroll
        for (int o = kFrontRunRows / 2; o > 0; o >>= 1) {
            const int32_t v = __shfl_sync(0xffffffffu, lb, r + o);
            if (r + o < nr && v <= k) r += o;
        }
        const int tag = r * 8 + ((k - __shfl_sync(0xffffffffu, lb, r)) / kChunk & 7);
        const Acc x = load_hits(j, count);
        for (int t = 0; t < count; ++t) {  // warp-uniform
            const int to = __shfl_sync(0xffffffffu, tag, t);
            if (to != cur) {
                if (to / 8 != cur / 8) close_row();
                else close_chunk();
                cur = to;
            }
            add_hit(t, x, chunk);
        }
    };
    int have = 0;
    constexpr int U = 4;
    for (int32_t k0 = kb; k0 < ke; k0 += U * 32) {
        int32_t j[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) j[u] = k0 + u * 32 + lane < ke ? col[k0 + u * 32 + lane] : -1;
#pragma unroll
        for (int u = 0; u < U; ++u) in[u] = j[u] >= 0 && is_marked(j[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t hit = __ballot_sync(0xffffffffu, in[u]);
            if (!hit) continue;
            if (in[u]) {
                const int at = have + __popc(hit & ((1u << lane) - 1u));
                hit_k[warp][at] = k0 + u * 32 + lane;
                hit_j[warp][at] = j[u];
            }
            have += __popc(hit);
            __syncwarp();
            if (have >= 32) {
                take(32);
                have -= 32;
                const int32_t k = hit_k[warp][32 + lane], jj = hit_j[warp][32 + lane];
                __syncwarp();
                hit_k[warp][lane] = k;
                hit_j[warp][lane] = jj;
                __syncwarp();
            }
        }
    }
    if (have) take(have);
    close_row();
}

// what hop L-1 computes of row `row` (lane per row): its marked columns (nz or mask) go to the
// lists by the row's degree, up to kBallSparseCols of them; a row with more is taken whole
template <typename T, int B>
__device__ __forceinline__ void list_row(const FrontArgs<T> &a, int64_t slice, int32_t row) {
    constexpr int W = B / 32;
    const int lane = threadIdx.x & 31;
    uint32_t need[W];
    int marked = 0, degree = 0;
    if (row < a.n) {
        uint32_t w[W];
        load_words<W>(a.mask + (slice * a.n + row) * W, w);
        load_words<W>(a.nz + (slice * a.n + row) * W, need);
#pragma unroll
        for (int q = 0; q < W; ++q) {
            need[q] |= w[q];
            marked += __popc(need[q]);
        }
        degree = a.row_ptr[row + 1] - a.row_ptr[row];
        if (degree > kFrontHeavy) marked = 0;  // its chunks see to it
    }
    const int kind = marked > kBallSparseCols ? 4 : degree <= kChunk ? 0 : degree <= 2 * kChunk ? 1 : degree <= 4 * kChunk ? 2 : 3;
    int32_t *lists = a.lists + slice * kBallLists;
    int first = 0;
#pragma unroll
    for (int k = 0; k < kBallLists; ++k) {
        const int count = marked && kind == k ? (k == 4 ? 1 : marked) : 0;
        if (!__any_sync(0xffffffffu, count)) continue;
        int at = count;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, at, o);
            if (lane >= o) at += up;
        }
        const int all = __shfl_sync(0xffffffffu, at, 31);
        int base = 0;
        if (lane == 0) base = atomicAdd(lists + k, all);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (kind == k) first = base + at - count;
    }
    if (!marked) return;
    if (kind == 4) {
        a.rows[slice * a.n + first] = row;
        return;
    }
    uint32_t *out = pair_list(a, kind, slice) + first;
#pragma unroll
    for (int q = 0; q < W; ++q) {
        uint32_t bits = need[q];
        while (bits) {
            *out++ = static_cast<uint32_t>(row) * B + q * 32 + __ffs(bits) - 1;
            bits &= bits - 1u;
        }
    }
}

// ---------------------------------------------------------------------------
// Hop 3 from X_2's non-zero sectors: X_3 is stored in full. CTAs [0,
// gather_ctas): the gather of X_2 (a value whose sector was not stored is a
// zero); then a warp per heavy chunk; then list_ctas CTAs that make hop L-1's
// work lists; then a warp per row, striding over the rows. Lane l covers columns
// l * CPL .. and loads them from the neighbours whose sector there has values.
// ---------------------------------------------------------------------------
template <typename T, int B>
__global__ void __launch_bounds__(kSpmmWarps * 32, 8) k_front3(const FrontArgs<T> a) {
    using Acc = typename AccOf<T>::type;
    __shared__ uint2 packs[kSpmmWarps][32 + 8];
    using SM = SectorMask<T, B>;
    constexpr int CPL = B / 32, LS = 32 / SM::COUNT;
    constexpr int U = 4;  // loads in flight
    using Vec = LaneVec<T, CPL>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *__restrict__ row_ptr = a.row_ptr;
    const int32_t *__restrict__ col = a.col;
    const int32_t n = a.n;
    const int64_t slice = blockIdx.y;
    const T *__restrict__ xp = a.x_prev + slice * n * B;
    T *__restrict__ xn = a.x_next + slice * n * B;
    const typename SM::Word *__restrict__ sec = static_cast<const typename SM::Word *>(a.sectors) + slice * n;
    if (static_cast<int32_t>(blockIdx.x) < a.gather_ctas) {
        const int b = blockIdx.x, bs = b * static_cast<int>(sizeof(T)) / 32;
        const int32_t q = static_cast<int32_t>(slice) * B + b;
        if (q >= a.nsrc) return;
        const int32_t s = a.src[q];
        if (s < 0) return;
        auto value = [&](int32_t j) {
            return (sec[j] >> bs) & 1u ? static_cast<double>(to_acc(xp[static_cast<int64_t>(j) * B + b])) : 0.0;
        };
        const double diag = value(s);
        for (int32_t k = row_ptr[s] + threadIdx.x; k < row_ptr[s + 1]; k += blockDim.x)
            gather_term(k, diag - value(col[k]), a.tau, a.gather_ell, a.g, a.t1, a.t2, a.rec);
        return;
    }
    const uint32_t mine = 1u << (lane / LS);
    const T *xl = xp + lane * CPL;
    uint2 *pack = packs[warp];
    // a chunk's entries (lane t: entry t's id and sector mask, 0: none) added to chunk[] in order:
    // those with a sector packed (offset, mask), then U loads in flight
    auto add_chunk = [&](int32_t j, uint32_t m, Acc *chunk) {
        const uint32_t any = __ballot_sync(0xffffffffu, m != 0u);
        const int count = __popc(any);
        __syncwarp();  // the last chunk's entries are read
        if (m) pack[__popc(any & ((1u << lane) - 1u))] = make_uint2(static_cast<uint32_t>(j) * B, m);
        if (lane < U) pack[count + lane] = make_uint2(0u, 0u);
        __syncwarp();
        for (int t = 0; t < count; t += U) {
            Vec v[U];
            bool in[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint2 e = pack[t + u];
                in[u] = (e.y & mine) != 0u;
                if (in[u]) v[u] = *reinterpret_cast<const Vec *>(xl + e.x);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (in[u]) {
#pragma unroll
                    for (int c = 0; c < CPL; ++c) chunk[c] += to_acc(v[u].v[c]);
                }
        }
    };
    auto store_row = [&](int32_t r, Acc sc, const Acc *sum) {
        Vec out;
#pragma unroll
        for (int c = 0; c < CPL; ++c) out.v[c] = from_acc<T>(sum[c] * sc);
        *reinterpret_cast<Vec *>(xn + static_cast<int64_t>(r) * B + lane * CPL) = out;
    };
    int32_t job = (static_cast<int32_t>(blockIdx.x) - a.gather_ctas) * kSpmmWarps + warp;
    const int32_t hwarps = (a.nhchunks + kSpmmWarps - 1) / kSpmmWarps * kSpmmWarps;
    if (job < hwarps) {
        if (job >= a.nhchunks) return;
        const int32_t h = a.hi_row[job], r = a.hv_id[h], k0 = a.hi_k0[job];
        const bool in = lane < row_ptr[r + 1] - k0;
        const int32_t j = in ? col[k0 + lane] : 0;
        Acc chunk[CPL], tot[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) chunk[c] = Acc(0);
        add_chunk(j, in ? sec[j] : 0u, chunk);
        if (heavy_total<T, B, CPL>(a, job, h, chunk, tot)) store_row(r, a.inv_deg[r], tot);
        return;
    }
    job -= hwarps;
    if (job < a.list_ctas * kSpmmWarps) {
        for (int64_t r = static_cast<int64_t>(job) * 32; r < n; r += static_cast<int64_t>(a.list_ctas) * kSpmmWarps * 32)
            list_row<T, B>(a, slice, static_cast<int32_t>(r) + lane);
        return;
    }
    // rows idx, idx + stride, ...: bounds three rows ahead, ids two, sector masks and 1/d one
    const uint32_t stride = static_cast<uint32_t>(a.light_ctas) * kSpmmWarps, rows = static_cast<uint32_t>(n);
    uint32_t idx = static_cast<uint32_t>(job - a.list_ctas * kSpmmWarps);
    int32_t rb = 0, re = 0, b1 = 0, e1 = 0, b2 = 0, e2 = 0;
    if (idx < rows) rb = row_ptr[idx], re = row_ptr[idx + 1];
    if (idx + stride < rows) b1 = row_ptr[idx + stride], e1 = row_ptr[idx + stride + 1];
    if (idx + 2 * stride < rows) b2 = row_ptr[idx + 2 * stride], e2 = row_ptr[idx + 2 * stride + 1];
    int32_t j = lane < re - rb ? col[rb + lane] : -1;
    int32_t j1 = lane < e1 - b1 ? col[b1 + lane] : -1;
    uint32_t m = j >= 0 ? sec[j] : 0u;
    Acc sc = idx < rows ? a.inv_deg[idx] : Acc(0);
    for (; idx < rows; idx += stride) {
        const int32_t j2 = lane < e2 - b2 ? col[b2 + lane] : -1;
        const uint32_t m1 = j1 >= 0 ? sec[j1] : 0u;
        const Acc sc1 = idx + stride < rows ? a.inv_deg[idx + stride] : Acc(0);
        int32_t b3 = 0, e3 = 0;
        if (idx + 3 * stride < rows) b3 = row_ptr[idx + 3 * stride], e3 = row_ptr[idx + 3 * stride + 1];
        if (re - rb <= kFrontHeavy) {
            Acc sum[CPL], chunk[CPL];
#pragma unroll
            for (int c = 0; c < CPL; ++c) sum[c] = Acc(0);
            for (int32_t k0 = rb; k0 < re; k0 += kChunk) {
                if (k0 > rb) {
                    j = lane < re - k0 ? col[k0 + lane] : -1;
                    m = j >= 0 ? sec[j] : 0u;
                }
#pragma unroll
                for (int c = 0; c < CPL; ++c) chunk[c] = Acc(0);
                add_chunk(j, m, chunk);
#pragma unroll
                for (int c = 0; c < CPL; ++c) sum[c] += chunk[c];
            }
            store_row(static_cast<int32_t>(idx), sc, sum);
        }
        rb = b1, re = e1, b1 = b2, e1 = e2, b2 = b3, e2 = e3;
        j = j1, j1 = j2, m = m1, sc = sc1;
    }
}

// the work lists alone (a block whose hop 3 is the ball hop itself, or runs in full)
template <typename T, int B>
__global__ void __launch_bounds__(kSpmmWarps * 32) k_front_lists(const FrontArgs<T> a) {
    const int64_t r = (static_cast<int64_t>(blockIdx.x) * kSpmmWarps + (threadIdx.x >> 5)) * 32;
    if (r < a.n) list_row<T, B>(a, blockIdx.y, static_cast<int32_t>(r) + (threadIdx.x & 31));
}

// ---------------------------------------------------------------------------
// Hop L-1 at the values of the work lists: X_{L-1}[y, b] for y in N(s_b) or
// N(N(s_b)), which is where the last hop (k_last_hop) and its gather read it;
// nothing else is stored. k_ball_rows: whole rows, a warp per chunk of a heavy
// row (when any column of it is marked), then a CTA per row with many marked
// columns, a warp per chunk. k_ball: CTAs [0, gather_ctas) gather X_{L-2}; the
// warps of the rest take the single values, a lane per chunk of at most 32
// entries: 4 values of 8 chunks to a warp, 8 of 4, 16 of 2, 32 of 1. In two
// launches because the second needs a third of the first's registers, and with
// them the warps that hide its loads.
// ---------------------------------------------------------------------------
template <typename T, int B>
__global__ void __launch_bounds__(kSpmmWarps * 32) k_ball_rows(const FrontArgs<T> a) {
    using Acc = typename AccOf<T>::type;
    constexpr int W = B / 32, CPL = B / 32;
    constexpr int U = CPL * static_cast<int>(sizeof(Acc)) > 16 ? 4 : 8;
    using Vec = LaneVec<T, CPL>;
    __shared__ Acc part[kSpmmWarps][B];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *__restrict__ row_ptr = a.row_ptr;
    const int32_t *__restrict__ col = a.col;
    const int64_t slice = blockIdx.y;
    const T *__restrict__ xp = a.x_prev + slice * a.n * B;
    T *__restrict__ xn = a.x_next + slice * a.n * B;
    const int lc0 = lane * CPL;
    // the lane's CPL columns of the entries [k0, k1), one chunk, in CSR order
    auto chunk_of = [&](int32_t k0, int32_t k1, Acc *chunk) {
#pragma unroll
        for (int c = 0; c < CPL; ++c) chunk[c] = Acc(0);
        const int32_t j = lane < k1 - k0 ? col[k0 + lane] : 0;
        const int cnt = k1 - k0;
        for (int t = 0; t < cnt; t += U) {
            Vec v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)  // past the end: the last entry again, not added
                v[u] = *reinterpret_cast<const Vec *>(xp + static_cast<int64_t>(__shfl_sync(0xffffffffu, j, min(t + u, cnt - 1))) * B + lc0);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (t + u < cnt) {
#pragma unroll
                    for (int c = 0; c < CPL; ++c) chunk[c] += to_acc(v[u].v[c]);
                }
        }
    };
    const int32_t hctas = (a.nhchunks + kSpmmWarps - 1) / kSpmmWarps;
    if (static_cast<int32_t>(blockIdx.x) < hctas) {
        const int32_t job = static_cast<int32_t>(blockIdx.x) * kSpmmWarps + warp;
        if (job >= a.nhchunks) return;
        const int32_t h = a.hi_row[job], r = a.hv_id[h], k0 = a.hi_k0[job];
        uint32_t any = 0u;
#pragma unroll
        for (int w = 0; w < W; ++w) any |= a.mask[(slice * a.n + r) * W + w] | a.nz[(slice * a.n + r) * W + w];
        if (!any) return;  // the same for every chunk of the row
        Acc chunk[CPL], tot[CPL];
        chunk_of(k0, min(k0 + kChunk, row_ptr[r + 1]), chunk);
        if (heavy_total<T, B, CPL>(a, job, h, chunk, tot)) {
            const Acc sc = a.inv_deg[r];
            Vec out;
#pragma unroll
            for (int c = 0; c < CPL; ++c) out.v[c] = from_acc<T>(tot[c] * sc);
            *reinterpret_cast<Vec *>(xn + static_cast<int64_t>(r) * B + lc0) = out;
        }
        return;
    }
    const int32_t *rows = a.rows + slice * a.n;
    const int32_t nr = a.lists[slice * kBallLists + 4];
    for (int32_t q = static_cast<int32_t>(blockIdx.x) - hctas; q < nr; q += static_cast<int32_t>(gridDim.x) - hctas) {
        const int32_t r = rows[q], rb = row_ptr[r], re = row_ptr[r + 1];
        const int nch = (re - rb + kChunk - 1) / kChunk;
        Acc total = Acc(0);  // thread t < B owns column t
        for (int c0 = 0; c0 < nch; c0 += kSpmmWarps) {
            const int c = c0 + warp;
            if (c < nch) {
                Acc chunk[CPL];
                chunk_of(rb + c * kChunk, min(rb + (c + 1) * kChunk, re), chunk);
#pragma unroll
                for (int e = 0; e < CPL; ++e) part[warp][lc0 + e] = chunk[e];
            }
            __syncthreads();
            if (threadIdx.x < B)
                for (int w = 0; w < min(kSpmmWarps, nch - c0); ++w) total += part[w][threadIdx.x];
            __syncthreads();
        }
        if (threadIdx.x < B) xn[static_cast<int64_t>(r) * B + threadIdx.x] = from_acc<T>(total * a.inv_deg[r]);
    }
}

template <typename T, int B>
__global__ void __launch_bounds__(kSpmmWarps * 32) k_ball(const FrontArgs<T> a) {
    using Acc = typename AccOf<T>::type;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t *__restrict__ row_ptr = a.row_ptr;
    const int32_t *__restrict__ col = a.col;
    const int64_t slice = blockIdx.y;
    const T *__restrict__ xp = a.x_prev + slice * a.n * B;
    T *__restrict__ xn = a.x_next + slice * a.n * B;
    if (static_cast<int32_t>(blockIdx.x) < a.gather_ctas) {
        const int32_t q = static_cast<int32_t>(slice) * B + static_cast<int32_t>(blockIdx.x);
        if (q < a.nsrc && a.src[q] >= 0)
            gather_source<T, B>(row_ptr, col, xp + blockIdx.x, 0, a.src[q], a.tau, a.gather_ell, a.g, a.t1, a.t2,
                                threadIdx.x, kSpmmWarps * 32, a.rec);
        return;
    }
    const int32_t *lists = a.lists + slice * kBallLists;
    int32_t np[4], njob[4], jobs = 0;  // values and warp jobs of the lists
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        np[k] = lists[k];
        njob[k] = (np[k] + (32 >> k) - 1) / (32 >> k);
        jobs += njob[k];
    }
    const int32_t nwarps = (static_cast<int32_t>(gridDim.x) - a.gather_ctas) * kSpmmWarps;
    for (int32_t q = (static_cast<int32_t>(blockIdx.x) - a.gather_ctas) * kSpmmWarps + warp; q < jobs; q += nwarps) {
        int32_t job = q;
        int kind = 3;
        int32_t count = np[3];
#pragma unroll
        for (int k = 3; k > 0; --k)
            if (kind == k && job >= njob[k]) {
                job -= njob[k];
                kind = k - 1;
                count = np[k - 1];
            }
        // 1 << kind lanes a value
        const int64_t at = static_cast<int64_t>(job) * (32 >> kind) + (lane >> kind);
        uint32_t pr = 0;
        int32_t r = 0, k0 = 0, cnt = 0;
        Acc sc = Acc(0);
        if (at < count) {
            pr = pair_list(a, kind, slice)[at];
            r = static_cast<int32_t>(pr / B);
            k0 = row_ptr[r] + (lane & ((1 << kind) - 1)) * kChunk;
            cnt = min(kChunk, row_ptr[r + 1] - k0);
            sc = a.inv_deg[r];
        }
        const T *xb = xp + pr % B;
        Acc chunk = Acc(0);
        for (int t = 0; t < cnt; t += 8) {
            int32_t j[8];
            Acc v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) j[u] = t + u < cnt ? col[k0 + t + u] : -1;
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = j[u] >= 0 ? to_acc(xb[static_cast<int64_t>(j[u]) * B]) : Acc(0);
#pragma unroll
            for (int u = 0; u < 8; ++u) chunk += v[u];
        }
        __syncwarp();
        Acc sum = Acc(0);
        for (int c = 0; c < 1 << kind; ++c) sum += __shfl_sync(0xffffffffu, chunk, (lane >> kind << kind) + c);
        if (at < count && (lane & ((1 << kind) - 1)) == 0) xn[pr] = from_acc<T>(sum * sc);
    }
}

}  // namespace sc
