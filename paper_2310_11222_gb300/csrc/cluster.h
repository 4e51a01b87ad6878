// One cluster per (component, pair): FP64 PCG of small and mid-sized graphs (cluster.cu).
#pragma once

#include "graph.h"

namespace nvd {

struct ClusterPlan;

// Estimated microseconds of one iteration of `cols` columns per component with one cluster
// each, and the cluster size that takes them; *cs = 0 where the components do not fit.
int cluster_estimate(nvd_graph_s *g, int64_t cols, int *cs, double *us);
// The plan for that cluster size (after cluster_estimate), or *out = NULL if it does not fit.
int cluster_plan_get(nvd_graph_s *g, int cs, ClusterPlan **out);
// The largest component's cluster size and kernel variant: 1 p gathered from L2, 2 matrix in
// shared memory, 4 one slot per thread, 8 p published through L2.
void cluster_variant(const ClusterPlan *pl, int32_t *cs, int32_t *variant);
// Estimated microseconds of one iteration of the host-driven loop on `tiles` tiles of kt FP64
// columns, fitted to runs from 3 * 10^4 to 10^6 rows: three launches and their block reductions,
// and 1.35 times the FP64 instructions (a multiply-add per entry and 10 operations per row, at 2
// lanes per SM and clock).
inline double tiles_iter_us(int64_t n, int64_t nnz, int kt, int tiles) {
    return tiles * (32.0 + 0.6 * kt + 1.35 * kt * ((double)nnz + 10.0 * (double)n) / 6.3e5);
}

// Solve K columns for every owner (owners_dev: device table of n_owner, or NULL: own0);
// the owners' x, y, z point at column 0 and hold kc columns.  d2dev: [K] device, one
// owner only, or NULL.  want_res: read the [n_owner][K] results back (synchronises s)
// into a buffer of the handle, valid until its next solve.  NVD_ERR_OOM comes before anything
// is launched.
int cluster_solve(nvd_graph_s *g, ClusterPlan *pl, const nvd_solve_opts &o, const Owner *owners_dev, const Owner &own0,
                  int n_owner, int K, int xdt, bool write_z, double *d2dev, bool want_res, ColResult **res,
                  cudaStream_t s);

// New weights in the cached plans (nvd_graph_set_weights).
int cluster_refill(nvd_graph_s *g, cudaStream_t s);

}  // namespace nvd
