// Resident traversal: a few sources' whole traversal (Algorithm 2, every hop
// and every gather of Eq. 9) by one CTA, the probabilities in shared memory.
//
// On graphs of small degree whose balls grow slowly (lattices, road networks,
// paths) a source's walk reaches few nodes: within l hops of it the support of
// p_l, and since the outputs read p_l at the source and its neighbours only,
// hop l of L needs the rows within min(l, L - l + 1) hops (a row further out
// no longer reaches them). A ball of radius (L + 1) / 2 holds all of it: 2,450
// nodes of a square lattice at L = 69, against the 150 * 69 rows and more of a
// block's id interval. So each CTA takes C sources next to each other, walks
// the ball around them breadth first into a list of nodes in level order
// (shared-memory hash table), turns their adjacency into 16-bit local ids, and
// runs all hops on the ball: the rows of hop l are a prefix of the list. No
// launch per hop, no block in global memory.
//
// Every value is bit for bit the block kernels': a row's neighbours are summed
// in CSR order (degrees up to 8, one chunk), scaled once by 1/d and rounded to
// the storage type where the block would store it; rows outside the ball are
// exact zeros or are never read.
//
// On a bipartite graph the sources of a CTA have one colour, hop l touches the
// levels of its own parity only, and one buffer serves both X_{l-1} and X_l
// (they lie on different levels); otherwise two buffers alternate.
//
// What bounds it: shared-memory bandwidth in the hops. 32 rows of 4 neighbours
// and a 16-byte vector of columns move 23 wavefronts of 128 bytes (4 neighbour
// vectors, the result, the ids, 1/d): 5.6 values a clock per SM at best, against
// 2.3 measured for the windowed block kernel, which streams its rows through
// HBM. Small balls are bound by the latency of a level (one dependent global
// load and a table insert, then a barrier) and of a hop (one barrier), which is
// why several CTAs share an SM when the ball is small. Whole calls, windowed
// blocks against this: 150 x 613 strip at 67 + 2 hops 94 -> 8.4 ms, 400 x 400
// lattice at learned lengths (37 to 353 hops) 625 -> 30 ms, 24 mixed graphs with
// lattices of 1,000 to 5,000 nodes at 1,003 hops 223 -> 85 ms. On graphs whose balls
// grow fast (expanders, trees) nothing fits within a few hops; what a sample of the
// balls says decides which class, if any, runs (res_first, global_class_pays).
#include <algorithm>
#include <numeric>

#include "budget.h"
#include "resident.cuh"

namespace sc {

constexpr int kResDegMax = 8;       // largest degree taken (neighbour ids kept per row)
constexpr int kResClasses = 4;      // shared-memory sizes tried in turn; the last keeps the adjacency in global memory
constexpr int kResIdOrder = 4;      // hops per level from which the lists are kept in id order,
constexpr int kResIdHops = 64;      // and hops: the ranks cost an SM 40 us on 4,200 nodes, six of its hops
constexpr int kResSample = 128;     // groups whose ball is measured to choose the first class

// what a measuring launch counts: the largest list, the groups that did not fit; of the others the
// nodes, the rows of all hops and the levels
enum ResCount { kResLargest, kResOver, kResNodes, kResRows, kResLevels, kResCounts };

struct ResArgs {
    const int32_t *row_ptr;
    const int32_t *ell;      // n x W neighbour ids in CSR order, -1 past the degree
    int32_t n;
    const int32_t *order;    // groups of C sources (-1: empty slot)
    const int32_t *groups;   // the launch's groups (nullable: all of 0 .. ngroups)
    int32_t ngroups;
    const int32_t *len;      // per node: hops its traversal takes (<= 0: not run)
    int32_t cap;             // nodes a list holds
    int32_t levels;          // level bounds held
    int32_t hash;            // slots of the hash table
    int32_t h0;              // first hop whose values are rounded to bf16
    const int32_t *tau;
    double *g, *t1, *t2;
    GatherRec rec;
    int32_t *over;           // [0]: groups that did not fit, [1 ..]: their ids
    unsigned long long *count;  // nullable: measure the balls only (ResCount)
    // global-adjacency class: per CTA adjacency, 1/d and nodes, and a local id per node of the graph
    // (0xffff between launches: a CTA takes its ball's back)
    unsigned char *scratch;
    size_t scratch_cta;
    uint16_t *marks;
    size_t marks_cta;
    int32_t ctas;            // (host) its CTAs
};

template <typename Acc, int C>
struct alignas(C * sizeof(Acc)) ResVec {
    Acc v[C];
};

template <int W>
struct alignas(2 * W) ResAdj {
    uint16_t v[W];
};

// the last CTA-wide layout: adjacency, 1/d, level bounds, then X, which the build's tables overlay
template <typename Acc, int C, int W, bool BIP, bool GADJ>
struct ResLayout {
    static constexpr int NBUF = BIP ? 1 : 2;
    static constexpr size_t row_bytes = (GADJ ? 0 : 2 * W + sizeof(Acc)) + static_cast<size_t>(NBUF) * C * sizeof(Acc);
    static __host__ __device__ size_t up(size_t x) { return (x + 15) / 16 * 16; }
    static __host__ __device__ size_t adj_bytes(int N) { return up(static_cast<size_t>(N) * 2 * W); }
    static __host__ __device__ size_t inv_bytes(int N) { return up(static_cast<size_t>(N) * sizeof(Acc)); }
    static __host__ __device__ size_t x_bytes(int N) { return up(static_cast<size_t>(NBUF) * (N + 1) * C * sizeof(Acc)); }
};

template <typename Acc, int C, int W, bool BIP, bool GADJ>
__global__ void __launch_bounds__(1024) k_resident(const ResArgs a) {
    using L = ResLayout<Acc, C, W, BIP, GADJ>;
    using Vec = ResVec<Acc, C>;
    using Adj = ResAdj<W>;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int32_t cnt[2], span[2], spos[C];
    __shared__ Acc recip[kResDegMax + 1];  // 1/d as the graph stores it
    if (threadIdx.x >= 1 && threadIdx.x <= kResDegMax)
        recip[threadIdx.x] = static_cast<Acc>(1.0 / static_cast<double>(static_cast<int>(threadIdx.x)));
    const int T = blockDim.x, tid = threadIdx.x;
    const int cap = a.cap, N = (BIP ? 2 : 1) * cap;  // local ids; id N: a cell that stays zero
    int32_t *lvl = reinterpret_cast<int32_t *>(sm);  // lvl[k]: nodes of its list up to level k
    unsigned char *p = sm + L::up(static_cast<size_t>(a.levels) * sizeof(int32_t));
    Adj *adj;
    Acc *inv;
    int32_t *nodes;
    uint32_t *hkey = nullptr;
    uint16_t *hval;  // shared: value of a hash slot; global-adjacency class: local id per node of the graph
    if constexpr (GADJ) {
        unsigned char *q = a.scratch + blockIdx.x * a.scratch_cta;
        adj = reinterpret_cast<Adj *>(q);
        inv = reinterpret_cast<Acc *>(q + L::adj_bytes(N));
        nodes = reinterpret_cast<int32_t *>(q + L::adj_bytes(N) + L::inv_bytes(N));
        hval = a.marks + blockIdx.x * a.marks_cta;
    } else {
        adj = reinterpret_cast<Adj *>(p);
        inv = reinterpret_cast<Acc *>(p + L::adj_bytes(N));
        p += L::adj_bytes(N) + L::inv_bytes(N);
        nodes = reinterpret_cast<int32_t *>(p);
        hkey = reinterpret_cast<uint32_t *>(p + L::up(static_cast<size_t>(N) * 4));
        hval = reinterpret_cast<uint16_t *>(hkey + a.hash);
    }
    Vec *X = reinterpret_cast<Vec *>(p);  // NBUF x (N + 1)

    for (int32_t gi = blockIdx.x; gi < a.ngroups; gi += gridDim.x) {
        const int32_t gid = a.groups ? a.groups[gi] : gi;
        const int32_t *src = a.order + static_cast<int64_t>(gid) * C;
        int32_t Lg = 0;
#pragma unroll
        for (int q = 0; q < C; ++q) Lg = max(Lg, src[q] >= 0 ? a.len[src[q]] : 0);
        if (Lg <= 0) continue;  // CTA-uniform
        const int32_t R = (Lg + 1) / 2;

        // ---- the ball: nodes in level order, sources first ----
        if constexpr (!GADJ)
            for (int t = tid; t < a.hash; t += T) hkey[t] = 0u;
        if (tid == 0) {
            cnt[0] = C;
            cnt[1] = 0;
            lvl[0] = C;
        }
        __syncthreads();
        bool fits = true;
        // claims node v for `list` unless it is known; false: it does not fit
        auto visit = [&](int32_t v, int list) -> bool {
            if constexpr (GADJ) {
                unsigned short *m = reinterpret_cast<unsigned short *>(hval) + v;
                if (*reinterpret_cast<volatile unsigned short *>(m) != 0xffffu) return true;
                if (atomicCAS(m, static_cast<unsigned short>(0xffffu), static_cast<unsigned short>(0xfffeu)) != 0xffffu) return true;
                const int32_t at = atomicAdd(&cnt[list], 1);
                if (at >= cap) {
                    *m = 0xffffu;
                    return false;
                }
                *m = static_cast<unsigned short>(list * cap + at);
                nodes[list * cap + at] = v;
                return true;
            } else {
                const uint32_t key = static_cast<uint32_t>(v) + 1u;
                uint32_t slot = __umulhi(key * 2654435761u, static_cast<uint32_t>(a.hash));
                for (int probe = 0; probe < a.hash; ++probe) {
                    const uint32_t old = atomicCAS(&hkey[slot], 0u, key);
                    if (old == key) return true;
                    if (old == 0u) {
                        // the next level reads this node's neighbours
                        asm volatile("prefetch.global.L1 [%0];" ::"l"(a.ell + static_cast<int64_t>(v) * W));
                        const int32_t at = atomicAdd(&cnt[list], 1);
                        if (at >= cap) return false;
                        hval[slot] = static_cast<uint16_t>(list * cap + at);
                        nodes[list * cap + at] = v;
                        return true;
                    }
                    slot = slot + 1 == static_cast<uint32_t>(a.hash) ? 0 : slot + 1;
                }
                return false;
            }
        };
        if (tid == 0) {
            for (int q = 0; q < C; ++q) {
                const int32_t s = src[q];
                const bool on = s >= 0 && a.len[s] > 0;
                nodes[q] = on ? s : -1;
                if (!on) continue;
                if constexpr (GADJ) {
                    hval[s] = static_cast<uint16_t>(q);
                } else {
                    const uint32_t key = static_cast<uint32_t>(s) + 1u;
                    uint32_t slot = __umulhi(key * 2654435761u, static_cast<uint32_t>(a.hash));
                    while (hkey[slot]) slot = slot + 1 == static_cast<uint32_t>(a.hash) ? 0 : slot + 1;  // < C keys in the table
                    hkey[slot] = key;
                    hval[slot] = static_cast<uint16_t>(q);
                }
            }
        }
        __syncthreads();
        // One barrier a level, which also carries the overflow marks. The level's bounds are in
        // registers: on a bipartite graph a level's inserts go to the other list, so its count is
        // not touched again before every thread has read it; with one list a second barrier is
        // needed for that.
        int32_t top = 0;                 // last level
        int32_t low[2] = {C, 0};         // BIP: nodes of each list so far
        int32_t f0 = 0, f1 = C;          // the frontier in its list
        for (int32_t k = 0; k < R; ++k) {
            const int from = BIP ? (k & 1) : 0, to = BIP ? 1 - from : 0;
            bool over = false;
            for (int32_t t = tid; t < (f1 - f0) * W; t += T) {
                const int32_t v = nodes[from * cap + f0 + t / W];
                if (v < 0) continue;
                const int32_t nb = a.ell[static_cast<int64_t>(v) * W + t % W];
                if (nb >= 0 && !visit(nb, to)) {
                    over = true;
                    break;
                }
            }
            if (k + 1 >= a.levels) over = true;  // too deep for the level bounds
            if (__syncthreads_or(over)) {
                fits = false;
                break;
            }
            const int32_t before = BIP ? low[to] : f1, now = cnt[to];
            if (now == before) break;
            if (tid == 0) lvl[k + 1] = now;
            top = k + 1;
            low[to] = now;
            f0 = before;
            f1 = now;
            if constexpr (!BIP) __syncthreads();
        }
        __syncthreads();
        const int32_t n0 = min(cnt[0], cap), n1 = BIP ? min(cnt[1], cap) : 0;
        auto forget = [&] {  // the global-adjacency class: the nodes' local ids back to "unknown"
            if constexpr (GADJ) {
                for (int32_t t = tid; t < n0 + n1; t += T) {
                    const int32_t v = nodes[t < n0 ? t : cap + t - n0];
                    if (v >= 0) hval[v] = 0xffffu;
                }
            }
        };
        if (a.count || !fits) {
            if (tid == 0) {
                if (a.count) {
                    atomicMax(&a.count[kResLargest], static_cast<unsigned long long>(max(n0, n1)));
                    if (!fits) {
                        atomicAdd(&a.count[kResOver], 1ull);
                    } else {
                        unsigned long long rows = 0;
                        for (int32_t h = 1; h <= Lg; ++h) {
                            int32_t lim = min(min(h, Lg - h + 1), top);
                            if (BIP) lim -= (lim ^ h) & 1;
                            rows += lim >= 0 ? lvl[lim] : 0;
                        }
                        atomicAdd(&a.count[kResNodes], static_cast<unsigned long long>(n0 + n1));
                        atomicAdd(&a.count[kResRows], rows);
                        atomicAdd(&a.count[kResLevels], static_cast<unsigned long long>(top));
                    }
                } else {
                    a.over[1 + atomicAdd(&a.over[0], 1)] = gid;
                }
            }
            forget();
            __syncthreads();
            continue;
        }

        // ---- a run of many more hops than levels: the lists in id order ----
        // The level prefixes save little there; in id order the neighbours of consecutive rows of a
        // row-major lattice are consecutive too, and their 16-byte values free of bank conflicts.
        // Ranks by a bitmap of the ids per list, over the adjacency and 1/d, not yet written.
        int32_t m0 = n0, m1 = n1;  // list lengths (in id order the empty source slots are gone)
        bool by_id = false;
        if constexpr (!GADJ) {
            if (Lg >= kResIdOrder * top && Lg >= kResIdHops) {
                if (tid == 0) span[0] = INT32_MAX, span[1] = -1;
                __syncthreads();
                for (int32_t t = tid; t < n0 + n1; t += T) {
                    const int32_t v = nodes[t < n0 ? t : cap + t - n0];
                    if (v >= 0) {
                        atomicMin(&span[0], v);
                        atomicMax(&span[1], v);
                    }
                }
                __syncthreads();
                const int32_t first = span[0], words = (span[1] - first) / 32 + 1;
                constexpr int LISTS = BIP ? 2 : 1;
                by_id = static_cast<size_t>(LISTS) * words * 8 <= L::adj_bytes(N);
                if (by_id) {  // CTA-uniform
                    uint32_t *bits = reinterpret_cast<uint32_t *>(adj);
                    int32_t *pre = reinterpret_cast<int32_t *>(bits + LISTS * words);
                    int32_t *moved = reinterpret_cast<int32_t *>(inv);
                    for (int32_t t = tid; t < LISTS * words; t += T) bits[t] = 0u;
                    __syncthreads();
                    for (int32_t t = tid; t < n0 + n1; t += T) {
                        const int32_t v = nodes[t < n0 ? t : cap + t - n0];
                        if (v >= 0) atomicOr(&bits[(t < n0 ? 0 : words) + (v - first) / 32], 1u << ((v - first) % 32));
                    }
                    __syncthreads();
                    if (tid < LISTS * 32) {  // a warp per list: running counts over its words
                        const int32_t l = tid / 32, lane = tid % 32;
                        int32_t run = 0;
                        for (int32_t w = 0; w < words; w += 32) {
                            const int32_t c = w + lane < words ? __popc(bits[l * words + w + lane]) : 0;
                            int32_t inc = c;
#pragma unroll
                            for (int o = 1; o < 32; o <<= 1) {
                                const int32_t up = __shfl_up_sync(0xffffffffu, inc, o);
                                if (lane >= o) inc += up;
                            }
                            if (w + lane < words) pre[l * words + w + lane] = run + inc - c;
                            run += __shfl_sync(0xffffffffu, inc, 31);
                        }
                        if (lane == 0) cnt[l] = run;
                    }
                    __syncthreads();
                    for (int32_t t = tid; t < n0 + n1; t += T) {
                        const int32_t v = nodes[t < n0 ? t : cap + t - n0];
                        if (v < 0) continue;
                        const int32_t l = t < n0 ? 0 : 1, w = l * words + (v - first) / 32;
                        const int32_t at = l * cap + pre[w] + __popc(bits[w] & ((1u << ((v - first) % 32)) - 1u));
                        moved[at] = v;
                        if (t < C) spos[t] = at;
                        const uint32_t key = static_cast<uint32_t>(v) + 1u;
                        uint32_t slot = __umulhi(key * 2654435761u, static_cast<uint32_t>(a.hash));
                        for (int probe = 0; probe < a.hash && hkey[slot] != key; ++probe)
                            slot = slot + 1 == static_cast<uint32_t>(a.hash) ? 0 : slot + 1;
                        hval[slot] = static_cast<uint16_t>(at);
                    }
                    m0 = cnt[0];
                    if (BIP) m1 = cnt[1];
                    __syncthreads();
                    for (int32_t t = tid; t < m0 + m1; t += T) {
                        const int32_t i = t < m0 ? t : cap + t - m0;
                        nodes[i] = moved[i];
                    }
                    __syncthreads();
                }
            }
        }
        if (!by_id && tid < C) spos[tid] = tid;

        // ---- adjacency in local ids (past the ball or the degree: the zero cell), 1/d ----
#pragma unroll 2
        for (int32_t t = tid; t < m0 + m1; t += T) {
            const int32_t i = t < m0 ? t : cap + t - m0;
            const int32_t v = nodes[i];
            Adj out;
            int4 row[W / 4];
#pragma unroll
            for (int w = 0; w < W / 4; ++w)
                row[w] = v >= 0 ? *reinterpret_cast<const int4 *>(a.ell + static_cast<int64_t>(v) * W + 4 * w)
                                : make_int4(-1, -1, -1, -1);
            int degree = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const int32_t nb = w % 4 == 0 ? row[w / 4].x : w % 4 == 1 ? row[w / 4].y : w % 4 == 2 ? row[w / 4].z : row[w / 4].w;
                degree += nb >= 0;
                uint16_t id = static_cast<uint16_t>(N);
                if (nb >= 0) {
                    if constexpr (GADJ) {
                        const uint16_t m = *reinterpret_cast<volatile uint16_t *>(&hval[nb]);
                        if (m != 0xffffu) id = m;
                    } else {
                        const uint32_t key = static_cast<uint32_t>(nb) + 1u;
                        uint32_t slot = __umulhi(key * 2654435761u, static_cast<uint32_t>(a.hash));
                        for (int probe = 0; probe < a.hash; ++probe) {
                            const uint32_t have = hkey[slot];
                            if (have == key) id = hval[slot];
                            if (have == key || have == 0u) break;
                            slot = slot + 1 == static_cast<uint32_t>(a.hash) ? 0 : slot + 1;
                        }
                    }
                }
                out.v[w] = id;
            }
            adj[i] = out;
            inv[i] = v >= 0 ? recip[degree] : Acc(0);
        }
        __syncthreads();
        forget();
        __syncthreads();

        // ---- X_0 = e_s ----
        {
            Vec z;
#pragma unroll
            for (int c = 0; c < C; ++c) z.v[c] = Acc(0);
            for (int b = 0; b < L::NBUF; ++b) {
                Vec *xb = X + static_cast<size_t>(b) * (N + 1);
                for (int32_t t = tid; t < m0 + m1; t += T) xb[t < m0 ? t : cap + t - m0] = z;
                if (tid == 0) xb[N] = z;
            }
        }
        __syncthreads();
        if (tid < C && src[tid] >= 0 && a.len[src[tid]] > 0) X[spos[tid]].v[tid] = Acc(1);
        // the last warp gathers and computes no rows, so that the FP64 chain of a term (two
        // conversions, a difference, a sum) runs beside the hop instead of behind it: lane gt holds
        // entry `gk` of source column `gq`
        const int TR = T - 32, gt = tid - TR;
        const int gq = gt < 0 ? 0 : gt / W;
        int32_t gk = -1, glen = 0, gtau = 0;
        uint32_t gj = 0;
        double acc = 0.0, r1 = 0.0, r2 = 0.0;
        int32_t gs = 0;
        if (gt >= 0 && gt < C * W && src[gq] >= 0 && a.len[src[gq]] > 0) {
            const int32_t s = src[gq], b = a.row_ptr[s];
            if (gt % W < a.row_ptr[s + 1] - b) {
                gk = b + gt % W;
                glen = a.len[s];
                gtau = a.tau[gk];
                gs = spos[gq];
                gj = adj[gs].v[gt % W];
                acc = a.g[gk];
                r1 = a.t1[gk];
                r2 = a.t2[gk];
            }
        }
        auto gather = [&](int32_t h) {  // the hop-h term of Eq. 9 (gather_term, the sums in registers)
            if (gk < 0 || h > glen) return;
            const Vec *xb = X + (BIP ? 0 : static_cast<size_t>(h & 1) * (N + 1));
            const double diag = BIP && (h & 1) ? 0.0 : static_cast<double>(xb[gs].v[gq]);
            const double xj = BIP && !(h & 1) ? 0.0 : static_cast<double>(xb[gj].v[gq]);
            const double term = diag - xj;
            if (h <= gtau) {
                acc += term;
                if (a.rec.mode == 1) {
                    if (h == gtau - 1) r1 = term;
                    else if (h == gtau) r2 = term;
                }
            } else if (a.rec.mode == 0 || a.rec.mode == 3) {
                if (h == gtau + 1) r1 = term;
                else if (h == gtau + 2) r2 = term;
            }
            if (a.rec.all) {
                if (a.rec.mode == 3) {
                    if (h == gtau - 1 || h == gtau) a.rec.all[static_cast<int64_t>(gk) * 2 + (h - gtau + 1)] = term;
                } else {
                    a.rec.all[static_cast<int64_t>(gk) * a.rec.stride + h] = term;
                }
            }
        };
        __syncthreads();

        // ---- the hops ----
        for (int32_t h = 1; h <= Lg; ++h) {
            int32_t lim = min(min(h, Lg - h + 1), top);
            const int par = BIP ? (h & 1) : 0;
            if (BIP) lim -= (lim ^ h) & 1;
            const int32_t rows = by_id ? (par ? m1 : m0) : lim >= 0 ? lvl[lim] : 0;
            const Vec *xp = X + (BIP ? 0 : static_cast<size_t>((h - 1) & 1) * (N + 1));
            Vec *xn = X + (BIP ? 0 : static_cast<size_t>(h & 1) * (N + 1));
            const bool to_bf16 = h >= a.h0;
            const int32_t base = par * cap;
            if (gt >= 0 && h >= 2) gather(h - 1);
#pragma unroll 2
            for (int32_t t = gt >= 0 ? rows : tid; t < rows; t += TR) {
                const Adj id = adj[base + t];
                Vec sum = xp[id.v[0]];
#pragma unroll
                for (int w = 1; w < W; ++w) {
                    const Vec x = xp[id.v[w]];
#pragma unroll
                    for (int c = 0; c < C; ++c) sum.v[c] += x.v[c];
                }
                const Acc d = inv[base + t];
#pragma unroll
                for (int c = 0; c < C; ++c) sum.v[c] *= d;
                if constexpr (sizeof(Acc) == 4)
                    if (to_bf16) {
#pragma unroll
                        for (int c = 0; c < C; ++c) sum.v[c] = __bfloat162float(__float2bfloat16_rn(sum.v[c]));
                    }
                xn[base + t] = sum;
            }
            __syncthreads();
        }
        gather(Lg);
        if (gk >= 0) {
            a.g[gk] = acc;
            a.t1[gk] = r1;
            a.t2[gk] = r2;
        }
        __syncthreads();  // X and the lists are the next group's
    }
}

// neighbour ids in rows of W, -1 past the degree (rows of larger degree: all -1, never taken)
__global__ void k_res_ell(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col, int32_t n, int W,
                          int32_t *__restrict__ ell) {
    const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (t >= static_cast<int64_t>(n) * W) return;
    const int32_t r = static_cast<int32_t>(t / W), w = static_cast<int32_t>(t % W);
    const int32_t b = row_ptr[r], d = row_ptr[r + 1] - b;
    ell[t] = d <= W && w < d ? col[b + w] : -1;
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
struct ResClass {
    size_t smem;  // dynamic shared memory of a CTA
    int threads, levels, per_sm;
};
// four, two and one CTA per SM (1 KB of an SM's 228 KB goes with each CTA, a few words are static)
static const ResClass kResClass[kResClasses] = {{55 * 1024, 256, 256, 4},
                                                {112 * 1024, 512, 1024, 2},
                                                {226 * 1024, 1024, 1024, 1},
                                                {226 * 1024, 1024, 1024, 1}};

template <typename Acc, int W, bool BIP, bool GADJ>
static int32_t res_capacity(int cls) {
    constexpr int C = GADJ ? 1 : 16 / static_cast<int>(sizeof(Acc));
    using L = ResLayout<Acc, C, W, BIP, GADJ>;
    const size_t room = kResClass[cls].smem - kResClass[cls].levels * sizeof(int32_t) - 6 * 16 - 2 * 16;
    size_t rows = room / L::row_bytes;
    rows = std::min<size_t>(rows, 65000);  // 16-bit ids, and room for the marks 0xfffe, 0xffff
    return static_cast<int32_t>(BIP ? rows / 2 : rows);
}

static size_t marks_stride(int32_t n) { return (static_cast<size_t>(n) + 127) / 128 * 128; }

template <typename Acc, int W, bool BIP, bool GADJ>
static void res_launch(sc_graph *g, ResArgs a, int cls, cudaStream_t s) {
    constexpr int C = GADJ ? 1 : 16 / static_cast<int>(sizeof(Acc));
    using L = ResLayout<Acc, C, W, BIP, GADJ>;
    const ResClass &k = kResClass[cls];
    a.cap = res_capacity<Acc, W, BIP, GADJ>(cls);
    a.levels = k.levels;
    const int N = (BIP ? 2 : 1) * a.cap;
    // the tables lie over X: 4 bytes a node for the list, 6 a slot
    a.hash = GADJ ? 0 : std::min<int>(2 * N, static_cast<int>((L::x_bytes(N) - L::up(static_cast<size_t>(N) * 4)) / 6));
    int grid = a.ngroups;
    if (GADJ) {
        grid = std::min(grid, a.ctas);
        a.scratch_cta = L::adj_bytes(N) + L::inv_bytes(N) + L::up(static_cast<size_t>(N) * 4);
        g->res_scratch.reserve(a.scratch_cta * a.ctas);
        a.scratch = g->res_scratch.get();
        a.marks_cta = marks_stride(g->n);
        if (g->res_marks.count < a.marks_cta * a.ctas) {
            g->res_marks.reserve(a.marks_cta * a.ctas);
            SC_CUDA(cudaMemsetAsync(g->res_marks.get(), 0xff, g->res_marks.count * sizeof(uint16_t), s));
        }
        a.marks = g->res_marks.get();
    }
    auto *fn = k_resident<Acc, C, W, BIP, GADJ>;
    SC_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(k.smem)));
    fn<<<grid, k.threads, k.smem, s>>>(a);
    SC_LAUNCH_CHECK();
}

template <typename Acc, int W>
static void res_dispatch(sc_graph *g, const ResArgs &a, int cls, bool bip, cudaStream_t s) {
    if (cls == kResClasses - 1) {
        if (bip) res_launch<Acc, W, true, true>(g, a, cls, s);
        else res_launch<Acc, W, false, true>(g, a, cls, s);
    } else {
        if (bip) res_launch<Acc, W, true, false>(g, a, cls, s);
        else res_launch<Acc, W, false, false>(g, a, cls, s);
    }
}

static void res_dispatch(sc_graph *g, const ResArgs &a, bool fp64, int W, int cls, bool bip, cudaStream_t s) {
    if (fp64) {
        if (W == 4) res_dispatch<double, 4>(g, a, cls, bip, s);
        else res_dispatch<double, 8>(g, a, cls, bip, s);
    } else {
        if (W == 4) res_dispatch<float, 4>(g, a, cls, bip, s);
        else res_dispatch<float, 8>(g, a, cls, bip, s);
    }
}

template <typename Acc>
static int32_t res_cap_of(int W, int cls, bool bip) {
    if (W == 4) return bip ? res_capacity<Acc, 4, true, false>(cls) : res_capacity<Acc, 4, false, false>(cls);
    return bip ? res_capacity<Acc, 8, true, false>(cls) : res_capacity<Acc, 8, false, false>(cls);
}

// nodes the global-adjacency class holds
template <typename Acc>
static int32_t res_global_rows(int W) {
    constexpr int c = kResClasses - 1;
    return 2 * (W == 4 ? res_capacity<Acc, 4, true, true>(c) : res_capacity<Acc, 8, true, true>(c));
}

// The global-adjacency class runs a source and its ball alone on an SM, where a block shares each row
// of ids among 32 to 128 sources, so it pays for long runs on balls that are small against the graph
// and not for short ones on most of it: an SM's time for the measured sources, predicted from counts,
// against the blocks' (ResidentRun::block_ns). Fitted on lattices, trees and random regular graphs of
// 10,000 to 100,000 nodes at 15 to 201 hops: 3.5 ns a node and slot to build a ball (slots: the mean
// of the degree and the width of a row of ids; in vain where it does not fit), 1 us a level, 0.4 ns a
// row and hop at four slots and 0.6 at eight, 0.2 us a hop. Calls, FP32, blocks against this class:
// random 4-regular bipartite of 20,000 nodes at 15 hops 12.8 and 22.6 ms, 51 hops 44 and 73, 201 hops
// 175 and 149; 8-regular of 40,000 at 9 hops 37 and 83; renamed lattice of 40,000 at 201 hops 720 and
// 170. Within kResGain the blocks are taken.
constexpr double kResGain = 1.1;

// h: the measured sources' counts, of ns sources of `hops` hops together and `blocks_ns` in blocks
static bool global_class_pays(const unsigned long long *h, int32_t ns, double hops, double blocks_ns, int W,
                              double degree, int32_t cap_rows, int sms) {
    const double over = static_cast<double>(h[kResOver]), fit = (ns - over) / ns;
    const double build = 3.5 * 0.5 * (degree + W) * (static_cast<double>(h[kResNodes]) + over * cap_rows);
    const double run = (0.2 + 0.05 * W) * static_cast<double>(h[kResRows]) +
                       1000.0 * static_cast<double>(h[kResLevels]) + 200.0 * fit * hops;
    return kResGain * (build + run) < fit * blocks_ns * sms;
}

bool resident_degree_ok(int32_t max_degree) { return max_degree <= kResDegMax; }

// Groups of `width` sources with neighbouring ids, one segment (and, on a
// bipartite one, one colour) to a group, segments of more nodes first; only
// segments of the wanted kind whose degrees fit.
static std::vector<int32_t> res_groups(const sc_graph *g, const std::vector<int32_t> &level,
                                       const std::vector<int32_t> &seg_start, const std::vector<char> &seg_take,
                                       const std::vector<char> &seg_bip, bool bip, int width) {
    const int nseg = static_cast<int>(seg_start.size()) - 1;
    std::vector<int> segs;
    for (int i = 0; i < nseg; ++i)
        if (seg_take[i] && (seg_bip[i] != 0) == bip) segs.push_back(i);
    std::stable_sort(segs.begin(), segs.end(), [&](int x, int y) {
        return seg_start[x + 1] - seg_start[x] > seg_start[y + 1] - seg_start[y];
    });
    std::vector<int32_t> out;
    for (int i : segs)
        for (int colour = 0; colour < (bip ? 2 : 1); ++colour) {
            for (int32_t v = seg_start[i]; v < seg_start[i + 1]; ++v)
                if (!bip || (level[v] & 1) == colour) out.push_back(v);
            while (out.size() % width) out.push_back(-1);
        }
    return out;
}

// The traversal of `sources` (len + extra hops each) as far as their balls fit;
// returns the sources that are left for the block kernels. seg_take marks the
// segments to handle here (degrees up to kResDegMax).
std::vector<int32_t> run_resident(const ResidentRun &r, const std::vector<int32_t> &sources,
                                  const std::vector<int32_t> &len, const std::vector<int32_t> &seg_start,
                                  const std::vector<char> &seg_take, const std::vector<char> &seg_bip,
                                  ResidentStats *st) {
    sc_graph *g = r.g;
    cudaStream_t s = r.s;
    const int32_t n = g->n;
    const bool fp64 = r.prec == SC_PREC_FP64;
    const int W = g->res_width;
    std::vector<int32_t> h_len(n, 0), left;
    int32_t longest = 0;
    int64_t total = 0, count = 0;
    for (int32_t v : sources) {
        const int32_t l = std::max(len[v] + r.extra, 0);
        h_len[v] = l;
        longest = std::max(longest, l);
        total += l;
        count += l > 0;
    }
    const std::tuple<bool, int32_t, int32_t> key(fp64, longest, static_cast<int32_t>(total / std::max<int64_t>(count, 1)));
    auto kept = [&](const std::map<std::tuple<bool, int32_t, int32_t>, int> &m) {  // a graph's own, -1: not asked
        const auto it = seg_start.size() == 2 ? m.find(key) : m.end();
        return it == m.end() ? -1 : it->second;
    };
    const int kept_first = kept(g->res_first), kept_global = kept(g->res_global);
    if (kept_first == kResClasses - 1 && (!seg_bip[0] || kept_global == 0)) {  // none runs
        for (int32_t v : sources)
            if (h_len[v] > 0) left.push_back(v);
        return left;
    }
    g->res_len.reserve(n);
    SC_CUDA(cudaMemcpyAsync(g->res_len.get(), h_len.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    if (!g->res_ready) {
        g->res_ell.reserve(static_cast<size_t>(n) * W);
        k_res_ell<<<ceil_div(static_cast<int64_t>(n) * W, 256), 256, 0, s>>>(g->row_ptr.get(), g->col_idx.get(), n, W,
                                                                           g->res_ell.get());
        SC_LAUNCH_CHECK();
        ++st->launches;
        g->res_ready = true;
    }
    for (int kind = 0; kind < 2; ++kind) {
        const bool bip = kind == 0;
        bool any = false;
        for (size_t i = 0; i + 1 < seg_start.size(); ++i) any = any || (seg_take[i] && (seg_bip[i] != 0) == bip);
        if (!any) continue;
        // groups of the widest class, and the same sources one by one for the last class
        const int width = fp64 ? 2 : 4;
        std::vector<int32_t> &order = g->res_order[kind];
        DevBuf<int32_t> &d_order = g->res_order_dev[kind];
        if (g->res_order_width[kind] != width) {
            std::vector<int32_t> level(n);
            SC_CUDA(cudaMemcpyAsync(level.data(), g->level.get(), n * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            SC_CUDA(cudaStreamSynchronize(s));
            order = res_groups(g, level, seg_start, seg_take, seg_bip, bip, width);
            d_order.reserve(order.size());
            SC_CUDA(cudaMemcpyAsync(d_order.get(), order.data(), order.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
            g->res_order_width[kind] = width;
        }
        const int32_t ngroups = static_cast<int32_t>(order.size() / width);
        std::vector<int32_t> list;
        for (int32_t q = 0; q < ngroups; ++q) {
            int32_t Lg = 0;
            for (int c = 0; c < width; ++c) {
                const int32_t v = order[static_cast<size_t>(q) * width + c];
                if (v >= 0) Lg = std::max(Lg, h_len[v]);
            }
            if (Lg > 0) {
                list.push_back(q);
                st->hops += Lg;
            }
        }
        if (list.empty()) continue;
        g->res_list.reserve(list.size());
        g->res_over.reserve(list.size() + 1);
        g->res_count.reserve(kResCounts);
        // (a copy from host memory may still read it when the call returns)
        bool copying = false;
        auto put_list = [&] {
            SC_CUDA(cudaMemcpyAsync(g->res_list.get(), list.data(), list.size() * sizeof(int32_t),
                                    cudaMemcpyHostToDevice, s));
            copying = true;
        };
        auto free_list = [&] {  // before `list` changes
            if (copying) SC_CUDA(cudaStreamSynchronize(s));
            copying = false;
        };
        put_list();
        ResArgs a{};
        a.row_ptr = g->row_ptr.get();
        a.ell = g->res_ell.get();
        a.n = n;
        a.order = d_order.get();
        a.groups = g->res_list.get();
        a.ngroups = static_cast<int32_t>(list.size());
        a.len = g->res_len.get();
        a.h0 = r.prec == SC_PREC_BF16 ? r.h0 : INT32_MAX;
        a.tau = g->tau_entry.get();
        a.g = g->acc_g.get();
        a.t1 = g->acc_t1.get();
        a.t2 = g->acc_t2.get();
        a.rec = r.rec;
        a.over = g->res_over.get();
        // the first class: the one that holds the largest ball of a sample of the groups. It is kept
        // when the sample was of a graph's whole request: measured again at every call it cost a
        // third of a short one (random 8-regular, 5,000 nodes, 7 hops: 0.84 ms, 0.60 without)
        int cls = 0;
        const bool keep = seg_start.size() == 2 && static_cast<int32_t>(list.size()) == ngroups;
        auto measure = [&](ResArgs m, int c, unsigned long long *h) {  // the balls of m's groups
            SC_CUDA(cudaMemsetAsync(g->res_count.get(), 0, kResCounts * sizeof(unsigned long long), s));
            m.count = g->res_count.get();
            res_dispatch(g, m, fp64, W, c, bip, s);
            ++st->launches;
            SC_CUDA(cudaMemcpyAsync(h, g->res_count.get(), kResCounts * sizeof(unsigned long long),
                                    cudaMemcpyDeviceToHost, s));
            SC_CUDA(cudaStreamSynchronize(s));
        };
        auto cap_of = [&](int c) { return fp64 ? res_cap_of<double>(W, c, bip) : res_cap_of<float>(W, c, bip); };
        int32_t seg_max = 0;
        for (size_t i = 0; i + 1 < seg_start.size(); ++i)
            if (seg_take[i] && (seg_bip[i] != 0) == bip) seg_max = std::max(seg_max, seg_start[i + 1] - seg_start[i]);
        if (kept_first >= 0) {
            cls = kept_first;
        } else if (seg_max + width > cap_of(0)) {
            std::vector<int32_t> pick;
            const int32_t ns = std::min<int32_t>(kResSample, a.ngroups);
            for (int32_t q = 0; q < ns; ++q) pick.push_back(list[static_cast<size_t>(q) * a.ngroups / ns]);
            SC_CUDA(cudaMemcpyAsync(g->res_over.get(), pick.data(), ns * sizeof(int32_t), cudaMemcpyHostToDevice, s));
            ResArgs m = a;
            m.groups = g->res_over.get();
            m.ngroups = ns;
            unsigned long long h[kResCounts];
            measure(m, kResClasses - 2, h);
            while (cls < kResClasses - 2 && h[kResLargest] > static_cast<unsigned long long>(cap_of(cls))) ++cls;
            // no ball of the sample fits with its adjacency
            if (h[kResOver] == static_cast<unsigned long long>(ns)) cls = kResClasses - 1;
        }
        if (keep) g->res_first[key] = cls;
        // groups of small segments need no more than the class that holds the segment, which leaves
        // room for more CTAs per SM: `list` starts with the smallest class in use, later classes get
        // their own groups and the ones that did not fit
        std::vector<int32_t> later[kResClasses];
        if (cls < kResClasses - 1) {
            std::vector<int32_t> seg_class(seg_start.size() - 1, cls);
            int lowest = cls;
            for (size_t i = 0; i + 1 < seg_start.size(); ++i) {
                int &c = seg_class[i];
                while (c > 0 && seg_start[i + 1] - seg_start[i] + width <= cap_of(c - 1)) --c;
                if (seg_take[i] && (seg_bip[i] != 0) == bip) lowest = std::min(lowest, c);
            }
            if (lowest < cls) {
                std::vector<int32_t> first;
                for (int32_t q : list) {
                    const int32_t v = order[static_cast<size_t>(q) * width];  // a group's first slot is taken
                    const size_t i = std::upper_bound(seg_start.begin(), seg_start.end(), v) - seg_start.begin() - 1;
                    (seg_class[i] == lowest ? first : later[seg_class[i]]).push_back(q);
                }
                free_list();
                list.swap(first);
                cls = lowest;
                put_list();
            }
        }
        auto more = [&](int c) {
            for (int q = c; q < kResClasses; ++q)
                if (!later[q].empty()) return true;
            return false;
        };
        for (; cls < kResClasses && (!list.empty() || more(cls)); ++cls) {
            if (!later[cls].empty()) {  // with what earlier classes left over
                free_list();
                list.insert(list.end(), later[cls].begin(), later[cls].end());
                later[cls].clear();
                put_list();
            }
            if (list.empty()) continue;
            if (cls == kResClasses - 1) {
                // one source to a group, adjacency in global memory: bipartite graphs only (one
                // buffer, half the rows a hop; without that the block kernels are as fast), and only
                // where it pays
                if (!bip) break;
                std::vector<int32_t> single;
                for (int32_t q : list)
                    for (int c = 0; c < width; ++c) {
                        const int32_t v = order[static_cast<size_t>(q) * width + c];
                        if (v >= 0 && h_len[v] > 0) single.push_back(v);
                    }
                g->res_single.reserve(single.size());
                g->res_over.reserve(single.size() + 1);
                SC_CUDA(cudaMemcpyAsync(g->res_single.get(), single.data(), single.size() * sizeof(int32_t),
                                        cudaMemcpyHostToDevice, s));
                SC_CUDA(cudaStreamSynchronize(s));  // `single` goes out of scope
                a.order = g->res_single.get();
                a.groups = nullptr;
                a.ngroups = static_cast<int32_t>(single.size());
                a.over = g->res_over.get();
                const size_t marks = marks_stride(n) * sizeof(uint16_t), held = g->res_marks.count * sizeof(uint16_t);
                a.ctas = global_class_ctas(marks, single.size(), g->num_sms, held, 0);
                if (a.ctas == 0) {
                    size_t free_b = 0, total_b = 0;
                    SC_CUDA(cudaMemGetInfo(&free_b, &total_b));
                    a.ctas = global_class_ctas(marks, single.size(), g->num_sms, held, free_b);
                }
                if (a.ctas == 0) {  // (2 bytes a node and SM: 14 million nodes in 4 GB)
                    left.insert(left.end(), single.begin(), single.end());
                    list.clear();
                    break;
                }
                const int32_t ns = kResSample;
                // few sources run about as soon as measured, and a call's later runs (the same sources at
                // longer lengths, in which this class does better) take the first one's answer
                int pays = kept_global >= 0 ? kept_global : *r.global;
                if (pays < 0 && a.ngroups > 4 * ns) {
                    std::vector<int32_t> pick;
                    double blocks_ns = 0.0, hops = 0.0;
                    for (int32_t q = 0; q < ns; ++q) {
                        pick.push_back(static_cast<int32_t>(static_cast<int64_t>(q) * a.ngroups / ns));
                        const int32_t v = single[pick.back()];
                        blocks_ns += r.block_ns(v, h_len[v]);
                        hops += h_len[v];
                    }
                    SC_CUDA(cudaMemcpyAsync(g->res_over.get(), pick.data(), ns * sizeof(int32_t), cudaMemcpyHostToDevice, s));
                    ResArgs m = a;
                    m.groups = g->res_over.get();
                    m.ngroups = ns;
                    unsigned long long h[kResCounts];
                    measure(m, cls, h);
                    const int32_t cap_rows = fp64 ? res_global_rows<double>(W) : res_global_rows<float>(W);
                    pays = global_class_pays(h, ns, hops, blocks_ns, W, static_cast<double>(g->nnz) / n, cap_rows,
                                             g->num_sms > 0 ? g->num_sms : 148);
                    if (seg_start.size() == 2) g->res_global[key] = pays;
                    *r.global = pays;
                }
                if (pays == 0) {
                    left.insert(left.end(), single.begin(), single.end());
                    list.clear();
                    break;
                }
                SC_CUDA(cudaMemsetAsync(g->res_over.get(), 0, sizeof(int32_t), s));
                r.timed([&] { res_dispatch(g, a, fp64, W, cls, bip, s); });
                ++st->launches;
                std::vector<int32_t> over(single.size() + 1);
                SC_CUDA(cudaMemcpyAsync(over.data(), g->res_over.get(), over.size() * sizeof(int32_t),
                                        cudaMemcpyDeviceToHost, s));
                SC_CUDA(cudaStreamSynchronize(s));
                list.clear();
                for (int32_t t = 0; t < over[0]; ++t) left.push_back(single[over[1 + t]]);
                break;
            }
            SC_CUDA(cudaMemsetAsync(g->res_over.get(), 0, sizeof(int32_t), s));
            a.groups = g->res_list.get();
            a.ngroups = static_cast<int32_t>(list.size());
            r.timed([&] { res_dispatch(g, a, fp64, W, cls, bip, s); });
            ++st->launches;
            int32_t nover = 0;
            SC_CUDA(cudaMemcpyAsync(&nover, g->res_over.get(), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            SC_CUDA(cudaStreamSynchronize(s));
            copying = false;
            list.resize(nover);
            if (nover > 0) {
                SC_CUDA(cudaMemcpyAsync(list.data(), g->res_over.get() + 1, nover * sizeof(int32_t),
                                        cudaMemcpyDeviceToHost, s));
                SC_CUDA(cudaStreamSynchronize(s));
                std::sort(list.begin(), list.end());
                put_list();
            }
        }
        free_list();
        for (int32_t q : list)
            for (int c = 0; c < width; ++c) {
                const int32_t v = order[static_cast<size_t>(q) * width + c];
                if (v >= 0 && h_len[v] > 0) left.push_back(v);
            }
    }
    SC_CUDA(cudaStreamSynchronize(s));  // host vectors behind the async copies
    std::sort(left.begin(), left.end());
    return left;
}

}  // namespace sc
