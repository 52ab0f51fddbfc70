// ExtractSG state shared by the pipeline stages.
#pragma once

#include "graph.cuh"

namespace lds {

struct SgState {
    int64_t D = 0;                        // denominator of the loads
    DevBuf<int32_t> order;                // [n] internal ids by (load desc, id asc)
    DevBuf<int32_t> pos;                  // [n] position of each internal id
    int64_t ncut = 0;
    DevBuf<int64_t> cuts;                 // [ncut] 1-based cut positions (ascending)
    int32_t ng = 0;                       // accepted groups
    DevBuf<int64_t> gend;                 // [ng] exclusive end position of each accepted group
    DevBuf<int64_t> lo, hi;               // [ng] min / max modified load of each group (over D)
    int32_t windows = 0, steps = 0;       // of the candidate walk
};

// Alg. 2 on the last Frank-Wolfe run of g (g->fw_*).
void extract_sg(lds_graph* g, SgState& st);

}  // namespace lds
