// Host interface of the resident traversal (resident.cu).
#pragma once

#include <functional>
#include <vector>

#include "propagate.cuh"

namespace sc {

struct ResidentRun {
    sc_graph *g;
    cudaStream_t s;
    int prec;
    int32_t h0;  // SC_PREC_BF16: first hop stored in bf16
    int extra;   // hops past each source's length (records)
    GatherRec rec;
    std::function<void(const std::function<void()> &)> timed;  // runs one traversal launch, with its events
    std::function<double(int32_t, int32_t)> block_ns;  // source, hops: its share of the blocks' time, estimated
    int *global;  // whether the class without the adjacency pays, from one run of a call to the next (-1: not asked)
};

struct ResidentStats {
    int64_t launches = 0;
    int64_t hops = 0;  // summed over the groups
};

bool resident_degree_ok(int32_t max_degree);
std::vector<int32_t> run_resident(const ResidentRun &r, const std::vector<int32_t> &sources,
                                  const std::vector<int32_t> &len, const std::vector<int32_t> &seg_start,
                                  const std::vector<char> &seg_take, const std::vector<char> &seg_bip,
                                  ResidentStats *st);

}  // namespace sc
