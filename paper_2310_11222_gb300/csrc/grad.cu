// C ABI: nvd_ge_grad -- adjoint of d^2 = delta^T L^+ delta (no new solve).
//
// With z = L^+ delta (mean-zero per component) and upstream weights gbar_j:
//   d(d^2)/dx = 2 z,  d(d^2)/dy = -2 z                       (L^+ symmetric)
//   d(d^2)/dW_uv = -z^T (dL/dW_uv) z = -1/2 (z_u - z_v)^2    per stored entry,
// from dL^+ = -L^+ dL L^+ (the null space is fixed while weights stay positive)
// and dL/dW_uv = 1/2 (e_u - e_v)(e_u - e_v)^T for the operator built from
// W_sym = (W + W^T)/2.  The two stored entries of an undirected edge thus sum to
// -(z_u - z_v)^2, the derivative with respect to the edge weight.
//
// The weight gradient is a gather over the undirected edges: z is first laid out as
// [n][KT] tiles (one 16-byte aligned row per node); an edge reads its two nodes' rows and
// writes its two stored entries, which have the same derivative.  The edge list (its nodes
// and the places of its entries) is made from the CSR once per handle; without memory for it
// the stored entries are taken one by one.
#include <algorithm>
#include <cstring>
#include <utility>

#include "graph.h"
#include "kernels.cuh"

using namespace nvd;

namespace {

// zt[i][j] = z[c0 + j][user(i)] (0 beyond k), 32 rows per CTA through shared memory.
template <class TZ, int KT>
__global__ void k_z_tile(const TZ *__restrict__ z, int64_t n, int k, int c0, const int32_t *__restrict__ perm,
                         TZ *__restrict__ zt) {
    __shared__ TZ tile[32][KT + 1];
    const int64_t i0 = (int64_t)blockIdx.x * 32;
    for (int t = threadIdx.x; t < 32 * KT; t += blockDim.x) {
        const int li = t % 32, j = t / 32;
        const int64_t i = i0 + li;
        TZ v = 0;
        if (i < n && c0 + j < k) {
            const int64_t u = perm ? (int64_t)perm[i] : i;
            v = z[(int64_t)(c0 + j) * n + u];
        }
        tile[li][j] = v;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 32 * KT; t += blockDim.x) {
        const int j = t % KT, li = t / KT;
        const int64_t i = i0 + li;
        if (i < n) zt[i * KT + j] = tile[li][j];
    }
}

// The edge list from the CSR: one edge for every stored entry (u, v), u < v, with the place of
// (v, u) beside its own (rev; -1 if it is not stored), and one for every entry u > v whose
// mirror is not stored (a pattern the caller vouched for).  A block takes 256 rows, a warp a
// row at a time: once to count, then (WRITE), with the block's range of the list reserved, to write.
__device__ __forceinline__ int64_t find_entry(const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colidx,
                                              int32_t row, int32_t col) {
    int64_t lo = __ldg(rowptr + row), hi = __ldg(rowptr + row + 1);
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(colidx + mid) < col) lo = mid + 1;
        else hi = mid;
    }
    return lo < __ldg(rowptr + row + 1) && __ldg(colidx + lo) == col ? lo : -1;
}
template <bool WRITE>
__global__ void __launch_bounds__(256) k_edge_list(int64_t n, const int64_t *__restrict__ rowptr,
                                                   const int32_t *__restrict__ colidx, bool symmetric,
                                                   unsigned long long *total, int2 *__restrict__ uv,
                                                   longlong2 *__restrict__ at) {
    __shared__ unsigned cnt[256];
    __shared__ unsigned long long base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t r0 = (int64_t)blockIdx.x * 256; r0 < n; r0 += (int64_t)gridDim.x * 256) {
        for (int pass = 0; pass < (WRITE ? 2 : 1); ++pass) {
            for (int q = warp; q < 256 && r0 + q < n; q += 8) {
                const int32_t u = (int32_t)(r0 + q);
                const int64_t e0 = __ldg(rowptr + u), e1 = __ldg(rowptr + u + 1);
                unsigned done = 0;
                for (int64_t eb = e0; eb < e1; eb += 32) {
                    const int64_t e = eb + lane;
                    int32_t v = -1;
                    int64_t rev = -1;
                    bool take = false;
                    if (e < e1) {
                        v = __ldg(colidx + e);
                        // counting needs only the mirrors of entries below the diagonal, and
                        // those only where the pattern was not checked
                        if (v > u ? WRITE && pass == 1 : !symmetric) rev = find_entry(rowptr, colidx, v, u);
                        take = v > u || (!symmetric && rev < 0);
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, take);
                    if (pass && take) {
                        const unsigned long long o = base + cnt[q] + done + __popc(m & ((1u << lane) - 1u));
                        uv[o] = make_int2(u, v);
                        at[o] = make_longlong2(e, rev);
                    }
                    done += __popc(m);
                }
                if (!pass && lane == 0) cnt[q] = done;
            }
            __syncthreads();
            if (!pass && warp == 0) {   // running sums of the 256 counts, 8 per lane
                unsigned c[8], s = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    c[q] = r0 + lane * 8 + q < n ? cnt[lane * 8 + q] : 0u;
                    s += c[q];
                }
                unsigned incl = s;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const unsigned o = __shfl_up_sync(0xffffffffu, incl, off);
                    if (lane >= off) incl += o;
                }
                unsigned run = incl - s;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    cnt[lane * 8 + q] = run;
                    run += c[q];
                }
                if (lane == 31) base = atomicAdd(total, (unsigned long long)incl);
            }
            __syncthreads();
        }
    }
}

template <class T> __device__ __forceinline__ double to_f64(T v) {
    if constexpr (sizeof(T) == 4) return dev::f2d(v);
    else return v;
}

// For every edge (u, v): g[entries of the edge] (+)= -1/2 sum_j gbar_j (zt[u][j] - zt[v][j])^2.
// One lane per edge, two from 8 columns on, each taking every second 16 bytes of the rows.
// Bound by the FP64 pipe: three operations per edge and column and, per 16 edges, one to add
// the lane pair and one to scale.  A warp per row that took every stored entry with a lane group
// per entry did each edge twice and spent 5 of 11 instructions on adding and scaling 4 entries
// at 16 FP64 columns: 10^6 edges of a BA graph took 644 us, this way 106 us; 5 * 10^6 edges and 32
// columns 4,824 us, this way 950 us.
template <class TZ, class TG, int KT, bool ACC>
__global__ void __launch_bounds__(256) k_grad_edges(int64_t n_edges, const int2 *__restrict__ uv,
                                                    const longlong2 *__restrict__ at, const TZ *__restrict__ zt,
                                                    const double *__restrict__ gb, TG *__restrict__ g) {
    constexpr int VEC = dev::VecCfg<TZ, KT>::VEC, LPE = KT >= 8 ? 2 : 1, P = KT / (VEC * LPE);
    static_assert(P >= 1, "columns fill the lanes");
    const int lane = threadIdx.x & 31, sub = lane % LPE;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; b * (32 / LPE) < n_edges; b += nw) {
        const int64_t e = b * (32 / LPE) + lane / LPE;
        double s = 0.0;
        longlong2 pos = make_longlong2(-1, -1);
        if (e < n_edges) {
            const int2 nd = __ldcs(uv + e);
            pos = __ldcs(at + e);
            const TZ *zu = zt + (int64_t)nd.x * KT, *zv = zt + (int64_t)nd.y * KT;
#pragma unroll(P < 4 ? P : 4)
            for (int i = 0; i < P; ++i) {
                const int c0 = (i * LPE + sub) * VEC;
                TZ a[VEC], c[VEC];
                dev::ldv<dev::LdRO, TZ, VEC>(zu + c0, a);
                dev::ldv<dev::LdRO, TZ, VEC>(zv + c0, c);
#pragma unroll
                for (int q = 0; q < VEC; ++q) {
                    const double d = to_f64(a[q]) - to_f64(c[q]);
                    s += __ldg(gb + c0 + q) * d * d;
                }
            }
        }
        if (LPE == 2) s += __shfl_xor_sync(0xffffffffu, s, 1);
        const double val = -0.5 * s;
        // two lanes: one entry each
        if (sub == 0 && pos.x >= 0) {
            if (ACC) g[pos.x] = (TG)((double)g[pos.x] + val);
            else g[pos.x] = (TG)val;
        }
        if (sub == LPE - 1 && pos.y >= 0) {
            if (ACC) g[pos.y] = (TG)((double)g[pos.y] + val);
            else g[pos.y] = (TG)val;
        }
    }
}

// The same without the edge list (24 bytes per edge), for a handle that has no memory for it:
// one warp per row, a lane group per stored entry.
template <class TZ, class TG, int KT, bool ACC>
__global__ void __launch_bounds__(256) k_grad_rows(int64_t n, const int64_t *__restrict__ rowptr,
                                                   const int32_t *__restrict__ colidx, const TZ *__restrict__ zt,
                                                   const double *__restrict__ gb, TG *__restrict__ g) {
    constexpr int VEC = dev::VecCfg<TZ, KT>::VEC, LPR = KT / VEC, G = 32 / LPR;
    const int lane = threadIdx.x & 31, gi = lane / LPR, col0 = (lane % LPR) * VEC;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += nw) {
        const int64_t e1 = __ldg(rowptr + u + 1);
        TZ own[VEC];
        dev::ldv<dev::LdRO, TZ, VEC>(zt + u * KT + col0, own);
        for (int64_t eb = __ldg(rowptr + u); eb < e1; eb += G) {
            const int64_t e = eb + gi;
            double s = 0.0;
            if (e < e1) {
                TZ zv[VEC];
                dev::ldv<dev::LdRO, TZ, VEC>(zt + (int64_t)__ldcs(colidx + e) * KT + col0, zv);
#pragma unroll
                for (int q = 0; q < VEC; ++q) {
                    const double d = to_f64(own[q]) - to_f64(zv[q]);
                    s += __ldg(gb + col0 + q) * d * d;
                }
            }
#pragma unroll
            for (int off = 1; off < LPR; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (e < e1 && col0 == 0) {
                const double val = -0.5 * s;
                if (ACC) g[e] = (TG)((double)g[e] + val);
                else g[e] = (TG)val;
            }
        }
    }
}

// grad_w[e] = g_int[uent[e]] (0 for dropped self-loops), converted to TW.
template <class TW>
__global__ void k_grad_scatter(const double *__restrict__ gint, const int64_t *__restrict__ uent,
                               int64_t nnz_user, TW *__restrict__ gw) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz_user;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t m = uent ? uent[e] : e;
        gw[e] = m >= 0 ? (TW)gint[m] : (TW)0;
    }
}

// grad_x = 2 gbar_j z, grad_y = -grad_x.  Column j of [k][n] on blockIdx.y (and its
// grid stride): the factor 2 gbar_j is one value per column, so an element costs one
// multiply and no index division (the FP64 unit, 1/64 of the FP32 rate, had bounded
// the per-element form).
template <class TZ>
__global__ void k_grad_xy(const TZ *__restrict__ z, int64_t n, int k, const double *__restrict__ gbar,
                          TZ *gx, TZ *gy) {
    for (int j = blockIdx.y; j < k; j += gridDim.y) {
        const double cj = 2.0 * gbar[j];
        const TZ *zj = z + (int64_t)j * n;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
            const double v = cj * (double)zj[i];
            if (gx) gx[(int64_t)j * n + i] = (TZ)v;
            if (gy) gy[(int64_t)j * n + i] = (TZ)(-v);
        }
    }
}

int grid_cap(int64_t work, int num_sms) {
    int64_t b = (work + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)num_sms * 32));
}

// The handle's edge list, made on first use.
int edge_list(nvd_graph_s *g, cudaStream_t s) {
    if (g->grad_uv.p) return NVD_OK;
    int st = NVD_OK;
    unsigned long long *total = (unsigned long long *)g->wsp("grad_total", 8, &st);
    if (st) return st;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((g->n + 255) / 256, (int64_t)g->num_sms * 8));
    auto run = [&](auto kern, int2 *uv, longlong2 *at, unsigned long long *out) -> int {
        NVD_TRY_CUDA(cudaMemsetAsync(total, 0, 8, s));
        kern<<<grid, 256, 0, s>>>(g->n, g->rowptr.as<int64_t>(), g->colidx.as<int32_t>(), g->sym_checked, total, uv, at);
        NVD_TRY_CUDA(cudaGetLastError());
        NVD_TRY_CUDA(cudaMemcpyAsync(out, total, 8, cudaMemcpyDeviceToHost, s));
        NVD_TRY_CUDA(cudaStreamSynchronize(s));
        return NVD_OK;
    };
    unsigned long long ne = 0, written = 0;
    NVD_TRY(run(k_edge_list<false>, nullptr, nullptr, &ne));
    DevBuf uv, at;
    NVD_TRY(g->grow(uv, (size_t)ne * sizeof(int2)));
    NVD_TRY(g->grow(at, (size_t)ne * sizeof(longlong2)));
    NVD_TRY(run(k_edge_list<true>, uv.as<int2>(), at.as<longlong2>(), &written));
    std::swap(g->grad_uv.p, uv.p);
    std::swap(g->grad_uv.bytes, uv.bytes);
    std::swap(g->grad_at.p, at.p);
    std::swap(g->grad_at.bytes, at.bytes);
    g->grad_edges = (int64_t)ne;
    return NVD_OK;
}

template <class TZ, class TW, int KT>
int grad_w_impl(nvd_graph_s *g, int k, const TZ *z, const double *gbar, TW *grad_w, cudaStream_t s) {
    int st = NVD_OK;
    const int ntile = (k + KT - 1) / KT;
    double *gbp = (double *)g->wsp("grad_gbar", (size_t)ntile * KT * 8, &st);
    TZ *zt = (TZ *)g->wsp("grad_zt", (size_t)g->n * KT * sizeof(TZ), &st);
    if (st) return st;
    NVD_TRY_CUDA(cudaMemsetAsync(gbp, 0, (size_t)ntile * KT * 8, s));
    NVD_TRY_CUDA(cudaMemcpyAsync(gbp, gbar, (size_t)k * 8, cudaMemcpyDeviceToDevice, s));
    const bool direct = (ntile == 1) && !g->uent.p;
    double *gint = nullptr;
    if (!direct) {
        gint = (double *)g->wsp("grad_gint", (size_t)std::max<int64_t>(g->nnz, 1) * 8, &st);
        if (st) return st;
    }
    const int zgrid = (int)((g->n + 31) / 32);
    NVD_TRY(unless_oom(edge_list(g, s)));
    const bool list = g->grad_uv.p != nullptr;
    const int64_t ne = g->grad_edges;
    const int2 *uv = g->grad_uv.as<int2>();
    const longlong2 *at = g->grad_at.as<longlong2>();
    const int64_t *rp = g->rowptr.as<int64_t>();
    const int32_t *ci = g->colidx.as<int32_t>();
    const int egrid = grid_cap(list ? ne * (KT >= 8 ? 2 : 1) : g->n * 32, g->num_sms);
    for (int t = 0; t < ntile; ++t) {
        const double *gbt = gbp + t * KT;
        k_z_tile<TZ, KT><<<zgrid, 256, 0, s>>>(z, g->n, k, t * KT, g->perm.as<int32_t>(), zt);
        if (direct) {
            if (list) k_grad_edges<TZ, TW, KT, false><<<egrid, 256, 0, s>>>(ne, uv, at, zt, gbt, grad_w);
            else k_grad_rows<TZ, TW, KT, false><<<egrid, 256, 0, s>>>(g->n, rp, ci, zt, gbt, grad_w);
        } else if (t == 0) {
            if (list) k_grad_edges<TZ, double, KT, false><<<egrid, 256, 0, s>>>(ne, uv, at, zt, gbt, gint);
            else k_grad_rows<TZ, double, KT, false><<<egrid, 256, 0, s>>>(g->n, rp, ci, zt, gbt, gint);
        } else {
            if (list) k_grad_edges<TZ, double, KT, true><<<egrid, 256, 0, s>>>(ne, uv, at, zt, gbt, gint);
            else k_grad_rows<TZ, double, KT, true><<<egrid, 256, 0, s>>>(g->n, rp, ci, zt, gbt, gint);
        }
        NVD_TRY_CUDA(cudaGetLastError());
    }
    if (!direct) {
        k_grad_scatter<TW><<<grid_cap(g->nnz_user, g->num_sms), 256, 0, s>>>(gint, g->uent.as<int64_t>(),
                                                                             g->nnz_user, grad_w);
        NVD_TRY_CUDA(cudaGetLastError());
    }
    return NVD_OK;
}

template <class TZ, class TW>
int grad_w_kt(nvd_graph_s *g, int k, const TZ *z, const double *gbar, TW *grad_w, cudaStream_t s) {
    if (k <= 1) return grad_w_impl<TZ, TW, 1>(g, k, z, gbar, grad_w, s);
    if (k <= 4) return grad_w_impl<TZ, TW, 4>(g, k, z, gbar, grad_w, s);
    if (k <= 8) return grad_w_impl<TZ, TW, 8>(g, k, z, gbar, grad_w, s);
    if (k <= 16) return grad_w_impl<TZ, TW, 16>(g, k, z, gbar, grad_w, s);
    return grad_w_impl<TZ, TW, 32>(g, k, z, gbar, grad_w, s);
}

int grad_impl(nvd_graph_t g, int32_t k, const void *z, int32_t zdt, const double *gbar, void *grad_w,
              void *grad_x, void *grad_y, cudaStream_t s) {
    if (!g || k < 0 || (zdt != NVD_F32 && zdt != NVD_F64) || (k > 0 && (!z || !gbar))) {
        set_error("nvd_ge_grad: invalid argument");
        return NVD_ERR_INVALID_ARG;
    }
    if (k == 0) return NVD_OK;
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != g->device) cudaSetDevice(g->device);
    int rc = NVD_OK;
    if (grad_x || grad_y) {
        // about 32 CTAs per SM in all, spread over the columns
        const int gy = std::min(k, 65535);
        const int gx = (int)std::max<int64_t>(1, std::min<int64_t>((g->n + 255) / 256,
                                                                   ((int64_t)g->num_sms * 32 + gy - 1) / gy));
        const dim3 grid((unsigned)gx, (unsigned)gy);
        if (zdt == NVD_F64)
            k_grad_xy<double><<<grid, 256, 0, s>>>((const double *)z, g->n, k, gbar, (double *)grad_x,
                                                   (double *)grad_y);
        else
            k_grad_xy<float><<<grid, 256, 0, s>>>((const float *)z, g->n, k, gbar, (float *)grad_x,
                                                  (float *)grad_y);
        if (cudaGetLastError() != cudaSuccess) rc = NVD_ERR_CUDA;
    }
    if (rc == NVD_OK && grad_w && g->nnz_user > 0) {
        if (g->nnz == 0) {
            rc = cudaMemsetAsync(grad_w, 0, (size_t)g->nnz_user * (g->wdtype == NVD_F64 ? 8 : 4), s) == cudaSuccess
                     ? NVD_OK : NVD_ERR_CUDA;
        } else if (zdt == NVD_F64) {
            rc = g->wdtype == NVD_F64 ? grad_w_kt<double, double>(g, k, (const double *)z, gbar, (double *)grad_w, s)
                                      : grad_w_kt<double, float>(g, k, (const double *)z, gbar, (float *)grad_w, s);
        } else {
            rc = g->wdtype == NVD_F64 ? grad_w_kt<float, double>(g, k, (const float *)z, gbar, (double *)grad_w, s)
                                      : grad_w_kt<float, float>(g, k, (const float *)z, gbar, (float *)grad_w, s);
        }
    }
    if (rc == NVD_OK) {
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            set_error("nvd_ge_grad: %s", cudaGetErrorString(e));
            rc = NVD_ERR_CUDA;
        }
    }
    if (prev >= 0 && prev != g->device) cudaSetDevice(prev);
    return rc;
}

}  // namespace

extern "C" int nvd_ge_grad(nvd_graph_t g, int32_t k, const void *z, int32_t zdtype, const double *gbar,
                           void *grad_w, void *grad_x, void *grad_y, nvd_stream_t stream) {
    clear_error();
    TraceRange trace("nvd_ge_grad");
    try {
        return grad_impl(g, k, z, zdtype, gbar, grad_w, grad_x, grad_y, (cudaStream_t)stream);
    } catch (...) {
        set_error("nvd_ge_grad: unexpected host exception");
        return NVD_ERR_CUDA;
    }
}
