// One cluster per (component, pair): FP64 PCG of small and mid-sized graphs (cluster.cu).
#pragma once

#include "graph.h"

namespace nvd {

struct ClusterPlan;

// Plan for solving `cols` columns per component with one cluster each, or *out = NULL
// where the components do not fit or the host-driven loop (gen_tiles tiles of gen_kt
// columns) is estimated to be faster.
int cluster_plan_for(nvd_graph_s *g, int64_t cols, int gen_kt, int gen_tiles, ClusterPlan **out);

// Solve K columns for every owner (owners_dev: device table of n_owner, or NULL: own0);
// the owners' x, y, z point at column 0 and hold kc columns.  d2dev: [K] device, one
// owner only, or NULL.  want_res: read the [n_owner][K] results back (synchronises s)
// into a buffer of the handle, valid until its next solve.
int cluster_solve(nvd_graph_s *g, ClusterPlan *pl, const nvd_solve_opts &o, const Owner *owners_dev, const Owner &own0,
                  int n_owner, int K, int xdt, bool write_z, double *d2dev, bool want_res, ColResult **res,
                  cudaStream_t s);

// New weights in the cached plans (nvd_graph_set_weights).
int cluster_refill(nvd_graph_s *g, cudaStream_t s);

}  // namespace nvd
