// Device helpers shared by the solves that keep their vectors on chip (cluster.cu,
// resident.cu; internal).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "graph.h"

namespace nvd {
namespace onchip {

// Tests on the bits: a comparison is an FP64 instruction too.
__device__ __forceinline__ bool finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool pos_finite(double v) { return __double_as_longlong(v) > 0 && finite(v); }

__device__ __forceinline__ double butterfly(double v, int width) {
    for (int off = width / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// One warp's rows: `steps` steps of H entries (one per lane group) from e (relative to the
// CTA's first), stored in groups of 4 steps so that a lane reads its 4 columns with one
// 16-byte load and its 4 weights with two; lane group g works for local slot
// slot + (g >> lg).
struct Item {
    int32_t e, steps, slot, lg;
};
// Place of step t of lane group g relative to the item's first entry: columns
// [group of steps][g][4], weights [group of steps][2][g][2].
__host__ __device__ constexpr int64_t col_at(int64_t t, int g, int H) { return (t >> 2) * 4 * H + g * 4 + (t & 3); }
__host__ __device__ constexpr int64_t w_at(int64_t t, int g, int H) {
    return (t >> 2) * 4 * H + ((t >> 1) & 1) * 2 * H + g * 2 + (t & 1);
}

// Entries of a plan from the CSR, one warp per task.  A task is a run of a row's entries
// [first, first + len) whose consecutive entries go to `width` consecutive lane groups from
// g0 on, step by step, of the item at e; padding up to pad entries has weight 0 on the row's
// own slot `self`.
struct FillTask {
    int64_t e, first;
    int32_t len, pad, width_g0, self;   // width | g0 << 8
};
template <class TW>
__global__ void k_fill(int64_t n, int H, const FillTask *__restrict__ task, const int32_t *__restrict__ slot_of,
                       const int32_t *__restrict__ colidx, const TW *__restrict__ w, int32_t *__restrict__ col,
                       double *__restrict__ wo) {
    const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int lane = threadIdx.x & 31;
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < n; t += nwarp) {
        const FillTask f = task[t];
        const int width = f.width_g0 & 255, g0 = f.width_g0 >> 8;
        for (int32_t j = lane; j < f.pad; j += 32) {
            const bool in = j < f.len;
            const int g = g0 + j % width;
            col[f.e + col_at(j / width, g, H)] = in ? slot_of[colidx[f.first + j]] : f.self;
            wo[f.e + w_at(j / width, g, H)] = in ? (double)w[f.first + j] : 0.0;
        }
    }
}
// Per slot its row's degree and inverse (0 without a row).
static __global__ void k_fill_deg(int64_t n, const int32_t *__restrict__ row, const double *__restrict__ deg64,
                                  const double *__restrict__ dinv64, double *__restrict__ deg,
                                  double *__restrict__ dinv) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = row[t];
        deg[t] = r >= 0 ? deg64[r] : 0.0;
        dinv[t] = r >= 0 ? dinv64[r] : 0.0;
    }
}

// Fill a plan's entries and degrees from the graph (at creation and for new weights).
inline int fill_onchip(const nvd_graph_s *g, int64_t n_tasks, int H, const FillTask *tasks, const int32_t *slot_of,
                       int32_t *col, double *w, int64_t n_slots, const int32_t *slot_row, double *deg, double *dinv,
                       cudaStream_t s) {
    if (n_slots == 0) return NVD_OK;
    const int64_t warps = n_tasks > n_slots ? n_tasks : n_slots;
    const int64_t cap = (int64_t)g->num_sms * 16, want = (warps + 7) / 8;
    const int grid = (int)(want < cap ? want : cap);
    auto go = [&](auto *wg) {
        k_fill<<<grid, 256, 0, s>>>(n_tasks, H, tasks, slot_of, g->colidx.as<int32_t>(), wg, col, w);
    };
    if (g->wdtype == NVD_F64) go(g->w.as<double>());
    else go(g->w.as<float>());
    k_fill_deg<<<grid, 256, 0, s>>>(n_slots, slot_row, g->deg64.as<double>(), g->dinv64.as<double>(), deg, dinv);
    NVD_TRY_CUDA(cudaGetLastError());
    return NVD_OK;
}

// Pinned read-back buffer of at least n results.
inline int pinned_results(ColResult **h, size_t *cap, size_t n) {
    if (*cap >= n) return NVD_OK;
    if (*h) cudaFreeHost(*h);
    *h = nullptr;
    *cap = 0;
    if (cudaHostAlloc((void **)h, n * sizeof(ColResult), cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        *h = nullptr;
        set_error("no pinned memory for %zu results", n);
        return NVD_ERR_OOM;
    }
    *cap = n;
    return NVD_OK;
}

}  // namespace onchip
}  // namespace nvd
