// FP64 PCG of one component with its vectors on chip, one persistent kernel (resident.cu).
#pragma once

#include "graph.h"

namespace nvd {

struct ResidentPlan;

// Estimated microseconds of one iteration of a tile of KT columns.
double resident_iter_us(int64_t n, int64_t nnz, int KT);

// Plan for tiles of KT columns, or *out = NULL where the graph is not one component (besides
// isolated nodes), its vectors do not fit, or KT is not 1, 4, 8 or 16.
int resident_plan_for(nvd_graph_s *g, int KT, ResidentPlan **out);

// Columns per tile of a plan, and its kernel variant: 1 x in global memory.
int32_t resident_width(const ResidentPlan *pl);
int32_t resident_variant(const ResidentPlan *pl);

// Solve k columns, tile after tile (own: x, y, z at column 0).  d2dev: [k] device or NULL.
// Synchronises s and reads the [k] results back into a buffer of the handle, valid until its
// next solve: a bounded wait that gave up is reported by this call or not at all.  NVD_ERR_OOM
// comes before anything is launched.
int resident_solve(nvd_graph_s *g, ResidentPlan *pl, const nvd_solve_opts &o, const Owner &own, int k, int xdt,
                   double *d2dev, ColResult **res, cudaStream_t s);

// New weights in the cached plans (nvd_graph_set_weights).
int resident_refill(nvd_graph_s *g, cudaStream_t s);

}  // namespace nvd
