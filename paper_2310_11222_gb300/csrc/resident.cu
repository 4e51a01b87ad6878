// FP64 PCG of one component with its vectors on chip: one persistent cooperative kernel,
// one CTA per SM (internal).
//
// For components too large for one cluster (cluster.cu) and tiles small enough for the SMs'
// shared memory (rows x columns up to about 1.3 million): each CTA owns a range of rows and
// keeps its r, q, p and, while they fit, x in shared memory for the whole solve, so the
// vector passes move nothing but the new p, which goes to global memory and is gathered from
// L2.  CTAs meet at a grid barrier three times per iteration (p^T q, the residual sums, the
// new p).  Around a barrier each CTA publishes its partial sums and then adds all CTAs'
// itself, in a fixed order: no second meeting, and every CTA takes the same scalars.
//
// Against the three launches of the host-driven loop this saves their ramps, tails and block
// reductions and the vectors' trips to L2.  Microseconds per iteration (host-driven): ER graph
// of 30,000 nodes, mean degree 10: 1 / 4 / 8 / 16 columns 15 / 18 / 23 / 30 (32 / 41 / 45 / 57);
// of 100,000 nodes 1 / 4 / 8 columns 19 / 27 / 40 (39 / 50 / 67); BA graph of 300,000, one column
// 36 (66).  One column of 10^6 nodes is left to the host-driven loop (116 against 89): with
// 174 KB of vectors in shared memory L1 holds too few of the gathers in flight.  What bounds it:
// the FP64 pipe from 8 columns on (100,000 nodes: row sums 33,600 of 80,000 clocks, vector
// passes 17,000); below, the two sums (9,000 clocks each, 4,000 of them the meeting) and the
// chain of dependent loads in the row sums.
//
// The grid barrier's wait is bounded (2 s): a CTA that gives up records NVD_ERR_TIMEOUT in
// the error word and leaves; all CTAs are co-resident (cooperative launch), so this can
// only follow a failure elsewhere, and the others then leave the same way.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <vector>

#include "dispatch.h"
#include "onchip.cuh"
#include "resident.h"

namespace nvd {

void note_launch(int64_t n);
int allow_dynamic_smem(const void *kern, int bytes);

namespace {

using namespace onchip;

constexpr int RS_NT = 1024;
constexpr size_t RS_SMEM_MAX = 224 * 1024;   // dynamic shared memory per CTA (227 KB less the static part)
constexpr int RS_MAX_KT = 16;
constexpr int64_t RS_PART_STEPS = 64;        // a longer row's entries are split over several items

constexpr int rs_lpr(int KT) { return KT == 1 ? 1 : KT / 2; }   // lanes per row (2 columns each)
constexpr int rs_groups(int KT) { return 32 / rs_lpr(KT); }

// A CTA's share: local slots 0 .. nslot - 1 (a row each), items, entries, split rows.
struct RsCta {
    int64_t slot0, item0, e0, split0;
    int32_t nslot, nitem, nsplit, nextra;
};
// A row whose items write partial sums to extra slots nslot + first .. of the CTA.
struct RsSplit {
    int32_t slot, first, count, pad;
};

struct RsArgs {
    const RsCta *ctas;
    const Item *items;
    const RsSplit *splits;
    const int32_t *col;        // slots of the whole component
    const double *w;
    const int32_t *node;       // slot -> user node
    const double *deg, *dinv;
    Owner own;                 // x, y, z at the tile's first column, kc columns
    int64_t n;                 // rows of the component
    double *pg;                // [slots][KT] published p
    double *xg;                // [slots][KT] x, or NULL: in shared memory
    double *part;              // [2][CTAs][2 * KT] partial sums
    unsigned *bar;             // arrivals, zero at launch
    int32_t *err;
    ColResult *res;            // [KT]
    double *d2dev;             // [kc] or NULL
    double rtol2, d2stop;
    int32_t max_iter, xdt, write_z;
    int32_t bar_extra;         // arrivals a meeting waits for beyond the grid's (NVD_SOLVE_TEST_TIMEOUT)
};

// Scalars per column, the same in every CTA.
struct RsState {
    double mean[RS_MAX_KT], alpha[RS_MAX_KT], beta[RS_MAX_KT], rho[RS_MAX_KT], rr[RS_MAX_KT], rr0[RS_MAX_KT],
        d2[RS_MAX_KT], hs_sum[RS_MAX_KT], hist[RS_MAX_KT][d2_window()];
    int32_t iters[RS_MAX_KT], status[RS_MAX_KT], active[RS_MAX_KT];
    int32_t go, fail, next;
};

__device__ __forceinline__ uint64_t timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// All CTAs; every thread's writes before it are seen after it.  target: arrivals so far.
// `meanwhile` runs between this CTA's arrival and its wait (work no other CTA asks for).
template <class W>
__device__ __forceinline__ bool grid_meet(const RsArgs &a, RsState &st, unsigned &target, W meanwhile) {
    target += gridDim.x;
    __syncthreads();
    // release and acquire at GPU scope order the whole CTA's writes and reads through the
    // block barriers around them
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    meanwhile();
    if (threadIdx.x == 0) {
        unsigned seen;
        const uint64_t t0 = timer_ns();
        for (unsigned spin = 1;; ++spin) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.bar) : "memory");
            if ((int)(seen - target) >= a.bar_extra) break;
            if ((spin & 1023u) == 0 && (__ldcg(a.err) != 0 || timer_ns() - t0 > 2000000000ull)) {
                atomicCAS(a.err, 0, (int)NVD_ERR_TIMEOUT);
                st.fail = 1;
                break;
            }
        }
    }
    __syncthreads();
    return st.fail == 0;
}

// Barrier `id` (1..15) among the first `n` threads of a group of warps.
__device__ __forceinline__ void part_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// Sums over 256 values, laid out [256 / S][S] in red, by the 8 warps of group `id` (thread t of
// 0..255, whose value is v): lanes l < S of its first warp return sum l.  Barriers of 8 and 2
// warps: one of all 32 costs about 150 clocks, and a sum has five steps.
template <int S>
__device__ __forceinline__ double sum256(double *red, int id, int t, double v) {
    red[t] = v;
    part_sync(1 + 2 * id, 256);
    if (t >= 64) return 0.0;
    v = (red[t] + red[t + 64]) + (red[t + 128] + red[t + 192]);
    red[t] = v;              // read by this thread alone so far
    part_sync(2 + 2 * id, 64);
    if (t >= 32) return 0.0;
    v = red[t] + red[t + 32];
#pragma unroll
    for (int off = 16; off >= S; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Column sums over the grid of every thread's v0 (and v1), the thread's column being
// threadIdx.x % KT; fin(j, s0, s1) runs in thread j < KT of every CTA, with the same values.
// Returns false if a wait gave up.  `red` holds NV * RS_NT doubles.
template <int KT, int NV, class F, class W>
__device__ __forceinline__ bool grid_sum(const RsArgs &a, RsState &st, double *red, unsigned &target, int &par, double v0,
                                         double v1, F fin, W meanwhile) {
    constexpr int S = NV * KT;
    const int t = threadIdx.x;
    double *part = a.part + (int64_t)par * gridDim.x * 2 * KT;
    par ^= 1;
    red[t] = v0;
    if (NV == 2) red[RS_NT + t] = v1;
    __syncthreads();
    if (t < NV * 256) {      // 8 warps per sum
        const int v = t >> 8, tt = t & 255;
        double *rv = red + v * RS_NT;
        const double m = (rv[tt] + rv[tt + 256]) + (rv[tt + 512] + rv[tt + 768]);
        const double s = sum256<KT>(rv, v, tt, m);
        if (tt < KT) part[(int64_t)blockIdx.x * S + v * KT + tt] = s;
    }
    if (!grid_meet(a, st, target, meanwhile)) return false;
    if (t < 256) {
        // all CTAs' sums: thread t adds sum t % S of CTAs t / S, t / S + 256 / S, ...
        double s = 0.0;
        const int n = (int)gridDim.x * S;
        int i = t;
        for (; i + 3 * 256 < n; i += 4 * 256) {
            const double b0 = __ldcg(part + i), b1 = __ldcg(part + i + 256), b2 = __ldcg(part + i + 512),
                         b3 = __ldcg(part + i + 768);
            s += (b0 + b1) + (b2 + b3);
        }
        for (; i < n; i += 256) s += __ldcg(part + i);
        const double sum = sum256<S>(red, 0, t, s);
        if (t < 32) {
            const double s1 = NV == 2 ? __shfl_sync(0xffffffffu, sum, (t + KT) & 31) : 0.0;
            if (t < KT) fin(t, sum, s1);
        }
    }
    __syncthreads();
    return true;
}

template <int KT>
__global__ void __launch_bounds__(RS_NT, 1) k_resident_pcg(const __grid_constant__ RsArgs a) {
    extern __shared__ __align__(16) double sm[];
    __shared__ RsState st;
    constexpr int VEC = KT == 1 ? 1 : 2, LPR = rs_lpr(KT), H = rs_groups(KT);
    constexpr int LH = H == 32 ? 5 : H == 16 ? 4 : H == 8 ? 3 : 2;   // log2 H
    const int tid = threadIdx.x, lane = tid & 31, j = tid % KT;
    const RsCta ct = a.ctas[blockIdx.x];
    const int ne = ct.nslot * KT;                   // this CTA's elements, [slot][column]
    double *r = sm, *q = r + ne, *p = q + ne + (int64_t)ct.nextra * KT, *red = p + ne;
    double *x = a.xg ? a.xg + ct.slot0 * KT : red + 2 * RS_NT;
    double *pg = a.pg + ct.slot0 * KT;
    const int32_t *__restrict__ node = a.node + ct.slot0;
    const double *__restrict__ deg = a.deg + ct.slot0;
    const double *__restrict__ dinv = a.dinv + ct.slot0;
    const Item *__restrict__ items = a.items + ct.item0;
    const RsSplit *__restrict__ splits = a.splits + ct.split0;
    const int32_t *__restrict__ cv = a.col + ct.e0;
    const double *__restrict__ wv = a.w + ct.e0;
    unsigned target = 0;
    int par = 0;
    auto nothing = []() {};

    auto delta_at = [&](int s) -> double {
        if (j >= a.own.kc) return 0.0;
        const int64_t u = __ldg(node + s) - a.own.base;
        if (a.own.idx & 1)
            return (double)(u == (int64_t)__ldg((const int32_t *)a.own.x + j)) -
                   (double)(u == (int64_t)__ldg((const int32_t *)a.own.y + j));
        const int64_t o = (int64_t)j * a.own.ld + u;
        return a.xdt ? __ldg((const double *)a.own.x + o) - __ldg((const double *)a.own.y + o)
                     : (double)__ldg((const float *)a.own.x + o) - (double)__ldg((const float *)a.own.y + o);
    };

    if (tid < KT) {
        st.iters[tid] = 0;
        st.status[tid] = NVD_OK;
        st.hs_sum[tid] = 0.0;
        for (int k = 0; k < d2_window(); ++k) st.hist[tid][k] = 0.0;
    }
    if (tid == 0) {
        st.fail = 0;
        st.next = 0;
    }
    // delta projected mean-zero, r = delta, u = D^-1 r, p = u, x = 0
    double s0 = 0.0, s1 = 0.0;
    for (int e = tid; e < ne; e += RS_NT) {
        const double d = delta_at(e / KT);
        r[e] = d;
        s0 += d;
    }
    __syncthreads();
    if (!(grid_sum<KT, 1>(a, st, red, target, par, s0, 0.0, [&](int c, double s, double) { st.mean[c] = s / (double)a.n; }, nothing)))
        return;
    s0 = 0.0;
    for (int e = tid; e < ne; e += RS_NT) {
        const double rv = r[e] - st.mean[j];
        const double u = __ldg(dinv + e / KT) * rv;
        r[e] = rv;
        x[e] = 0.0;
        p[e] = u;
        pg[e] = u;
        s0 = fma(rv, u, s0);
        s1 = fma(rv, rv, s1);
    }
    if (!(grid_sum<KT, 2>(a, st, red, target, par, s0, s1, [&](int c, double rho, double rr) {
            st.rho[c] = rho;
            st.rr[c] = rr;
            st.rr0[c] = rr;
            const bool valid = c < a.own.kc;
            if (valid && (!finite(rr) || !finite(rho))) st.status[c] = NVD_ERR_NUMERIC;
            const int act = valid && pos_finite(rr) && pos_finite(rho);
            st.active[c] = act;
            const unsigned all = (1u << KT) - 1u;
            const unsigned any = __ballot_sync(all, act);
            if (c == 0) st.go = any != 0;
        }, nothing)))
        return;
    while (st.go) {
        // row sums of W p: warps take the CTA's items, longest first
        for (;;) {
            int i = 0;
            if (lane == 0) i = atomicAdd(&st.next, 1);
            i = __shfl_sync(0xffffffffu, i, 0);
            if (i >= ct.nitem) break;
            const int4 iv = __ldg(reinterpret_cast<const int4 *>(items + i));
            const Item it{iv.x, iv.y, iv.z, iv.w};
            const int g = lane / LPR, c0 = (lane % LPR) * VEC;
            const int4 *cp = reinterpret_cast<const int4 *>(cv + it.e) + g;
            const double2 *wp = reinterpret_cast<const double2 *>(wv + it.e) + g;
            const int L = it.steps;
            double acc[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) acc[v] = 0.0;
            auto gather = [&](int c, double (&o)[VEC]) {
                if constexpr (VEC == 1) {
                    o[0] = __ldcg(a.pg + c);
                } else {
                    const double2 t = __ldcg(reinterpret_cast<const double2 *>(a.pg + (int64_t)c * KT + c0));
                    o[0] = t.x;
                    o[1] = t.y;
                }
            };
            int4 c = __ldg(cp);
            double2 wa = __ldg(wp), wb = __ldg(wp + H);
            for (int e = 0; e < L; e += 4) {
                double g0[VEC], g1[VEC], g2[VEC], g3[VEC];
                gather(c.x, g0);
                if (e + 1 < L) gather(c.y, g1);
                if (e + 2 < L) gather(c.z, g2);
                if (e + 3 < L) gather(c.w, g3);
                const double2 ua = wa, ub = wb;
                if (e + 4 < L) {
                    cp += H;
                    wp += 2 * H;
                    c = __ldg(cp);
                    wa = __ldg(wp);
                    wb = __ldg(wp + H);
                }
#pragma unroll
                for (int v = 0; v < VEC; ++v) {
                    acc[v] = fma(ua.x, g0[v], acc[v]);
                    if (e + 1 < L) acc[v] = fma(ua.y, g1[v], acc[v]);
                    if (e + 2 < L) acc[v] = fma(ub.x, g2[v], acc[v]);
                    if (e + 3 < L) acc[v] = fma(ub.y, g3[v], acc[v]);
                }
            }
            for (int off = LPR; off < (LPR << it.lg); off <<= 1)
#pragma unroll
                for (int v = 0; v < VEC; ++v) acc[v] += __shfl_xor_sync(0xffffffffu, acc[v], off);
            if ((g & ((1 << it.lg) - 1)) == 0) {
                const int s = it.slot + (g >> it.lg);
                if (it.lg < LH ? s < ct.nslot : true) {
#pragma unroll
                    for (int v = 0; v < VEC; ++v) q[s * KT + c0 + v] = acc[v];
                }
            }
        }
        __syncthreads();
        if (tid == 0) st.next = 0;
        if (ct.nsplit) {
            for (int e = tid; e < ct.nsplit * KT; e += RS_NT) {
                const RsSplit sp = splits[e / KT];
                double s = 0.0;
                for (int k = 0; k < sp.count; ++k) s += q[(ct.nslot + sp.first + k) * KT + j];
                q[sp.slot * KT + j] = s;
            }
            __syncthreads();
        }
        // q = D p - W p and p^T q
        s0 = 0.0;
        for (int e = tid; e < ne; e += RS_NT) {
            const double own = p[e];
            const double y = fma(__ldg(deg + e / KT), own, -q[e]);
            q[e] = y;
            s0 = fma(own, y, s0);
        }
        if (!(grid_sum<KT, 1>(a, st, red, target, par, s0, 0.0, [&](int c, double pq, double) {
                if (!st.active[c]) {
                    st.alpha[c] = 0.0;
                } else if (pos_finite(pq)) {
                    st.alpha[c] = st.rho[c] / pq;
                } else {
                    st.alpha[c] = 0.0;
                    st.status[c] = NVD_ERR_NUMERIC;
                }
            }, nothing)))
            return;
        // r -= alpha q, u = D^-1 r (kept in q); r^T u and |r|^2; x += alpha p while the CTAs meet
        const double al = st.alpha[j];
        s0 = s1 = 0.0;
        for (int e = tid; e < ne; e += RS_NT) {
            const double rv = fma(-al, q[e], r[e]);
            const double u = __ldg(dinv + e / KT) * rv;
            r[e] = rv;
            q[e] = u;
            s0 = fma(rv, u, s0);
            s1 = fma(rv, rv, s1);
        }
        if (!(grid_sum<KT, 2>(a, st, red, target, par, s0, s1, [&](int c, double rho_new, double rr) {
                int act = st.active[c];
                if (act) {
                    const int it = st.iters[c] + 1;
                    st.iters[c] = it;
                    st.rr[c] = rr;
                    const bool d2_done = a.d2stop > 0.0 && d2_settled(it, st.alpha[c] * st.rho[c], a.d2stop, st.hs_sum[c], st.hist[c]);
                    int end = -1;
                    if (st.status[c] == NVD_ERR_NUMERIC || !finite(rr) || !finite(rho_new)) end = NVD_ERR_NUMERIC;
                    else if (rr <= a.rtol2 * st.rr0[c] || d2_done) end = NVD_OK;
                    else if (it >= a.max_iter) end = NVD_ERR_NOT_CONVERGED;
                    if (end >= 0) {
                        st.status[c] = end;
                        st.active[c] = act = 0;
                    } else {
                        st.beta[c] = rho_new / st.rho[c];
                        st.rho[c] = rho_new;
                    }
                }
                const unsigned all = (1u << KT) - 1u;
                const unsigned any = __ballot_sync(all, act);
                if (c == 0) st.go = any != 0;
            },
            [&]() {
                for (int e = tid; e < ne; e += RS_NT) x[e] = fma(al, p[e], x[e]);
            })))
            return;
        if (!st.go) break;
        if (st.active[j]) {
            const double be = st.beta[j];
            for (int e = tid; e < ne; e += RS_NT) {
                const double v = fma(be, p[e], q[e]);
                p[e] = v;
                pg[e] = v;
            }
        }
        if (!grid_meet(a, st, target, nothing)) return;
    }
    // d^2 = delta^T x (delta projected), the mean of x, z = x - mean
    s0 = s1 = 0.0;
    for (int e = tid; e < ne; e += RS_NT) {
        const double xv = x[e];
        s0 += xv;
        s1 = fma(delta_at(e / KT) - st.mean[j], xv, s1);
    }
    if (!(grid_sum<KT, 2>(a, st, red, target, par, s0, s1, [&](int c, double sx, double dx) {
            st.beta[c] = sx / (double)a.n;
            st.d2[c] = dx;
        }, nothing)))
        return;
    if (a.write_z && j < a.own.kc) {
        const double mu = st.beta[j];
        for (int e = tid; e < ne; e += RS_NT) {
            const int64_t o = (int64_t)j * a.own.ld + (__ldg(node + e / KT) - a.own.base);
            if (a.xdt) ((double *)a.own.z)[o] = x[e] - mu;
            else ((float *)a.own.z)[o] = (float)(x[e] - mu);
        }
    }
    if (blockIdx.x == 0 && tid < KT) {
        a.res[tid] = ColResult{st.d2[tid], st.rr[tid], st.rr0[tid], st.iters[tid], st.status[tid]};
        if (a.d2dev && tid < a.own.kc) a.d2dev[tid] = st.d2[tid];
    }
}

}  // namespace

struct ResidentPlan {
    int KT = 0, ncta = 0;
    bool x_global = false, fits = false;
    size_t smem = 0;
    int64_t n_slots = 0;
    // two allocations and one copy: with one each, a new graph's first call took 10 ms instead
    // of 4 at 100,000 nodes (the rest of that was a comparison sort; 2.6 since only the plan that
    // is used is built)
    DevBuf meta, data;
    RsCta *ctas = nullptr;
    Item *items = nullptr;
    RsSplit *splits = nullptr;
    int32_t *node = nullptr, *col = nullptr;
    double *w = nullptr, *deg = nullptr, *dinv = nullptr;
    FillTask *tasks = nullptr;         // with slot_row, slot_of: what the weight updates need
    int32_t *slot_row = nullptr, *slot_of = nullptr;
    int64_t n_tasks = 0;
};

struct ResidentState {
    std::map<int, std::unique_ptr<ResidentPlan>> plans;   // by KT
    ColResult *h_res = nullptr;                           // pinned read-back
    size_t h_cap = 0;
    ~ResidentState() {
        if (h_res) cudaFreeHost(h_res);
    }
};
void resident_state_delete(ResidentState *c) { delete c; }

int64_t resident_state_bytes(const ResidentState *c) {
    int64_t b = 0;
    if (c)
        for (auto &kv : c->plans)
            b += (int64_t)(kv.second->meta.bytes + kv.second->data.bytes);
    return b;
}

namespace {

int fill_plan(nvd_graph_s *g, ResidentPlan *pl, cudaStream_t s) {
    return fill_onchip(g, pl->n_tasks, rs_groups(pl->KT), pl->tasks, pl->slot_of, pl->col, pl->w, pl->n_slots,
                       pl->slot_row, pl->deg, pl->dinv, s);
}

size_t rs_smem(int64_t rows, int64_t extra, int KT, bool x_global) {
    return ((size_t)(x_global ? 3 : 4) * rows * KT + (size_t)extra * KT + 2 * RS_NT) * 8;
}

int build_resident_plan(nvd_graph_s *g, int KT, ResidentPlan **out) {
    std::unique_ptr<ResidentPlan> pl(new ResidentPlan());
    pl->KT = KT;
    pl->ncta = g->num_sms;
    const int H = rs_groups(KT), P = pl->ncta;
    const std::vector<int64_t> &rp = g->h_rowptr;
    const int64_t a = g->h_seg_begin[0], n = g->h_seg_end[0] - a;
    std::vector<int32_t> perm;
    if (g->perm.p) {
        perm.resize(g->n);
        NVD_TRY_CUDA(cudaMemcpy(perm.data(), g->perm.p, (size_t)g->n * 4, cudaMemcpyDeviceToHost));
    }
    auto len_of = [&](int64_t r) { return rp[r + 1] - rp[r]; };
    std::vector<RsCta> ctas(P);
    std::vector<Item> items;
    std::vector<RsSplit> splits;
    std::vector<FillTask> tasks;
    std::vector<int32_t> node, slot_row, slot_of(g->n, 0);
    std::vector<int64_t> ord;
    tasks.reserve(n + n / 16);
    node.reserve(n);
    slot_row.reserve(n);
    // Rows of more than 32 entries are dealt to the CTAs back and forth, longest first (hubs
    // often come together in the node order, and the CTAs meet after the row sums and after the
    // vector passes: each needs its share of both; by running work alone the CTAs with the hubs
    // of a BA graph took twice the others' time in the row sums).  The rest in node order, cut
    // where the running work (a multiply-add per entry, 9 operations per row) reaches each CTA's
    // share.
    const int lg_all = H == 32 ? 5 : H == 16 ? 4 : H == 8 ? 3 : 2;
    std::vector<int64_t> wide;
    double total = 0.0;
    for (int64_t i = a; i < a + n; ++i) {
        if (len_of(i) > 32) wide.push_back(i);
        else total += (double)len_of(i) + 9.0;
    }
    std::stable_sort(wide.begin(), wide.end(), [&](int64_t x, int64_t y) { return len_of(x) > len_of(y); });
    int64_t r = a, ne = 0, max_rows = 0, max_extra = 0;
    double done = 0.0;
    for (int c = 0; c < P; ++c) {
        ord.clear();
        for (int64_t round = 0; round * P < (int64_t)wide.size(); ++round) {
            const int64_t at = round * P + ((round & 1) ? P - 1 - c : c);
            if (at < (int64_t)wide.size()) ord.push_back(wide[at]);
        }
        // the light rows of its range by length, longest first (at most 32 entries: counting sort)
        const double until = total * (c + 1) / P;
        const int64_t r0 = r;
        int64_t at[34] = {0};
        for (; r < a + n; ++r) {
            const int64_t d = len_of(r);
            if (d > 32) continue;
            const double work = (double)d + 9.0;
            if (c < P - 1 && done + 0.5 * work > until) break;
            done += work;
            ++at[33 - d];
        }
        for (int d = 1; d < 34; ++d) at[d] += at[d - 1];
        const int64_t nwide = (int64_t)ord.size();
        ord.resize(nwide + at[33]);
        for (int64_t i = r0; i < r; ++i) {
            const int64_t d = len_of(i);
            if (d <= 32) ord[nwide + at[32 - d]++] = i;
        }
        const int64_t nr = (int64_t)ord.size();
        RsCta &ct = ctas[c];
        ct = RsCta{};
        ct.slot0 = (int64_t)slot_row.size();
        ct.item0 = (int64_t)items.size();
        ct.split0 = (int64_t)splits.size();
        ct.e0 = ne;
        ct.nslot = (int32_t)nr;
        for (int64_t i = 0; i < nr; ++i) {
            const int64_t row = ord[i];
            slot_of[row] = (int32_t)(ct.slot0 + i);
            slot_row.push_back((int32_t)row);
            node.push_back(perm.empty() ? (int32_t)row : perm[row]);
        }
        int32_t extra = 0;
        for (int64_t i = 0; i < nr;) {
            const int64_t d = len_of(ord[i]);
            // lane groups per row: all of them for rows of more than 32 entries
            const bool all = d > 32;
            const int width = all ? H : 1;
            const int64_t parts = all ? std::max<int64_t>(1, (d + RS_PART_STEPS * H - 1) / (RS_PART_STEPS * H)) : 1;
            if (parts > 1) splits.push_back(RsSplit{(int32_t)i, extra, (int32_t)parts, 0});
            for (int64_t k = 0; k < parts; ++k) {
                const int64_t first = k * RS_PART_STEPS * H;
                const int64_t len = std::min<int64_t>(d - first, parts > 1 ? RS_PART_STEPS * H : d);
                const int64_t steps = (len + width - 1) / width;
                const int64_t room = std::max<int64_t>((steps + 3) / 4 * 4, 4);
                const int32_t slot = parts > 1 ? (int32_t)(nr + extra + k) : (int32_t)i;
                items.push_back(Item{(int32_t)(ne - ct.e0), (int32_t)steps, slot, all ? lg_all : 0});
                for (int l = 0; l < H / width; ++l) {
                    const bool in = i + l < nr;
                    const int64_t row = in ? ord[i + l] : ord[i];
                    tasks.push_back(FillTask{ne, rp[row] + (all ? first : 0),
                                             in ? (int32_t)(all ? len : len_of(row)) : 0, (int32_t)(room * width),
                                             width | (l * width) << 8, slot_of[row]});
                }
                ne += room * H;
            }
            if (parts > 1) extra += (int32_t)parts;
            i += H / width;
        }
        ct.nitem = (int32_t)(items.size() - ct.item0);
        ct.nsplit = (int32_t)(splits.size() - ct.split0);
        ct.nextra = extra;
        max_rows = std::max(max_rows, nr);
        max_extra = std::max<int64_t>(max_extra, extra);
    }
    pl->n_slots = (int64_t)slot_row.size();
    pl->n_tasks = (int64_t)tasks.size();
    pl->x_global = rs_smem(max_rows, max_extra, KT, false) > RS_SMEM_MAX;
    pl->smem = rs_smem(max_rows, max_extra, KT, pl->x_global);
    pl->fits = pl->smem <= RS_SMEM_MAX;
    if (pl->fits) {
        std::vector<char> host;
        size_t off[7];
        auto add = [&](int i, const void *h, size_t bytes) {
            off[i] = host.size();
            host.resize(off[i] + (bytes + 255) / 256 * 256);
            if (bytes) memcpy(host.data() + off[i], h, bytes);
        };
        add(0, ctas.data(), ctas.size() * sizeof(RsCta));
        add(1, items.data(), items.size() * sizeof(Item));
        add(2, splits.data(), splits.size() * sizeof(RsSplit));
        add(3, tasks.data(), tasks.size() * sizeof(FillTask));
        add(4, node.data(), node.size() * 4);
        add(5, slot_row.data(), slot_row.size() * 4);
        add(6, slot_of.data(), slot_of.size() * 4);
        NVD_TRY(pl->meta.alloc(host.size()));
        NVD_TRY_CUDA(cudaMemcpy(pl->meta.p, host.data(), host.size(), cudaMemcpyHostToDevice));
        char *m = pl->meta.as<char>();
        pl->ctas = (RsCta *)(m + off[0]);
        pl->items = (Item *)(m + off[1]);
        pl->splits = (RsSplit *)(m + off[2]);
        pl->tasks = (FillTask *)(m + off[3]);
        pl->node = (int32_t *)(m + off[4]);
        pl->slot_row = (int32_t *)(m + off[5]);
        pl->slot_of = (int32_t *)(m + off[6]);
        // weights, degrees, columns: entries come in multiples of 4 per lane group
        NVD_TRY(pl->data.alloc((size_t)ne * 12 + (size_t)pl->n_slots * 16 + 64));
        pl->w = pl->data.as<double>();
        pl->col = (int32_t *)(pl->w + ne);
        pl->deg = (double *)(pl->col + ne);
        pl->dinv = pl->deg + pl->n_slots;
        NVD_TRY(fill_plan(g, pl.get(), 0));
        NVD_TRY_CUDA(cudaDeviceSynchronize());
    }
    *out = pl.release();
    return NVD_OK;
}

template <int KT>
int launch(const ResidentPlan *pl, const RsArgs &a, cudaStream_t s) {
    auto kern = k_resident_pcg<KT>;
    NVD_TRY(allow_dynamic_smem((const void *)kern, (int)RS_SMEM_MAX));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)pl->ncta);
    cfg.blockDim = dim3(RS_NT);
    cfg.dynamicSmemBytes = pl->smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    NVD_TRY_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
    note_launch(1);
    return NVD_OK;
}

}  // namespace

// Fitted to measured runs: three meetings and two sums 16 us; the FP64 instructions, 15% of the
// entries and 35% in all lost to padding and imbalance (20% on ER graphs, 45% on BA); one column is bound by its gathers, 1.3
// clocks each, and from about 150,000 rows on by the loads L1 can keep in flight beside the
// vectors in shared memory.
double resident_iter_us(int64_t n, int64_t nnz, int KT) {
    const double mhz = 2000.0, sms = 152.0;
    if (KT == 1)
        return 16.0 + 9.0 * (double)n / (2.0 * sms) / mhz + 1.3 * (double)nnz / sms / mhz * (n > 150000 ? 1.8 : 1.0);
    return 16.0 + 1.35 * KT * (1.15 * (double)nnz + 9.0 * (double)n) / (2.0 * sms) / mhz;
}

int resident_plan_for(nvd_graph_s *g, int KT, ResidentPlan **out) {
    *out = nullptr;
    if (g->nseg != 1 || !(KT == 1 || KT == 4 || KT == 8 || KT == 16)) return NVD_OK;
    const int64_t n = g->h_seg_end[0] - g->h_seg_begin[0];
    if (rs_smem((n + g->num_sms - 1) / g->num_sms, 0, KT, true) > RS_SMEM_MAX) return NVD_OK;
    if (!g->resident) g->resident.reset(new ResidentState());
    auto &slot = g->resident->plans[KT];
    if (!slot) {
        ResidentPlan *p = nullptr;
        const int rc = build_resident_plan(g, KT, &p);
        if (rc != NVD_OK) {
            g->resident->plans.erase(KT);
            return rc;
        }
        slot.reset(p);
    }
    if (slot->fits) *out = slot.get();
    return NVD_OK;
}

int32_t resident_width(const ResidentPlan *pl) { return pl->KT; }
int32_t resident_variant(const ResidentPlan *pl) { return pl->x_global ? 1 : 0; }

int resident_refill(nvd_graph_s *g, cudaStream_t s) {
    if (!g->resident) return NVD_OK;
    for (auto &kv : g->resident->plans)
        if (kv.second->fits) NVD_TRY(fill_plan(g, kv.second.get(), s));
    return NVD_OK;
}

int resident_solve(nvd_graph_s *g, ResidentPlan *pl, const nvd_solve_opts &o, const Owner &own, int k, int xdt,
                   double *d2dev, ColResult **res, cudaStream_t s) {
    ResidentState *rst = g->resident.get();
    const int KT = pl->KT, ntiles = (k + KT - 1) / KT;
    const size_t xsz = own.idx ? 4 : xdt == NVD_F64 ? 8 : 4, zsz = xdt == NVD_F64 ? 8 : 4;
    int st = NVD_OK;
    const size_t vec = (size_t)pl->n_slots * KT * 8;
    double *pg = (double *)g->wsp("rs_p", vec, &st);
    double *xg = pl->x_global ? (double *)g->wsp("rs_x", vec, &st) : nullptr;
    double *part = (double *)g->wsp("rs_part", (size_t)2 * pl->ncta * 2 * KT * 8, &st);
    // the error word, then the barrier words of the tiles
    unsigned *bar = (unsigned *)g->wsp("rs_bar", (size_t)(1 + ntiles) * 4, &st);
    ColResult *rd = (ColResult *)g->wsp("rs_res", (size_t)ntiles * KT * sizeof(ColResult), &st);
    if (st) return st;
    const size_t need = (size_t)ntiles * KT + 1;
    NVD_TRY(pinned_results(&rst->h_res, &rst->h_cap, need));   // the last thing that can lack memory
    NVD_TRY_CUDA(cudaMemsetAsync(bar, 0, (size_t)(1 + ntiles) * 4, s));
    for (int t = 0; t < ntiles; ++t) {
        const int c0 = t * KT, kc = std::min(KT, k - c0);
        const size_t off = own.idx ? (size_t)c0 * xsz : (size_t)c0 * own.ld * xsz;
        RsArgs a{};
        a.ctas = pl->ctas;
        a.items = pl->items;
        a.splits = pl->splits;
        a.col = pl->col;
        a.w = pl->w;
        a.node = pl->node;
        a.deg = pl->deg;
        a.dinv = pl->dinv;
        a.own = own;
        a.own.x = (const char *)own.x + off;
        a.own.y = (const char *)own.y + off;
        a.own.z = own.z ? (char *)own.z + (size_t)c0 * own.ld * zsz : nullptr;
        a.own.kc = kc;
        a.n = pl->n_slots;
        a.pg = pg;
        a.xg = xg;
        a.part = part;
        a.err = (int32_t *)bar;
        a.bar = bar + 1 + t;
        a.res = rd + (size_t)t * KT;
        a.d2dev = d2dev ? d2dev + c0 : nullptr;
        a.rtol2 = o.rtol * o.rtol;
        a.d2stop = (o.flags & NVD_SOLVE_D2_STOP) ? o.d2_rtol : 0.0;
        a.max_iter = o.max_iter;
        a.xdt = xdt == NVD_F64 ? 1 : 0;
        a.write_z = own.z ? 1 : 0;
        a.bar_extra = (o.flags & NVD_SOLVE_TEST_TIMEOUT) ? 1 : 0;
        switch (KT) {
            case 1: NVD_TRY(launch<1>(pl, a, s)); break;
            case 4: NVD_TRY(launch<4>(pl, a, s)); break;
            case 8: NVD_TRY(launch<8>(pl, a, s)); break;
            default: NVD_TRY(launch<16>(pl, a, s)); break;
        }
    }
    int32_t *err = (int32_t *)(rst->h_res + (need - 1));
    NVD_TRY_CUDA(cudaMemcpyAsync(rst->h_res, rd, (need - 1) * sizeof(ColResult), cudaMemcpyDeviceToHost, s));
    NVD_TRY_CUDA(cudaMemcpyAsync(err, bar, 4, cudaMemcpyDeviceToHost, s));
    NVD_TRY_CUDA(cudaStreamSynchronize(s));
    if (*err) {
        set_error("nvd_ge_distance: a bounded device wait gave up (status %d)", *err);
        return *err;
    }
    *res = rst->h_res;
    return NVD_OK;
}

}  // namespace nvd
