// FP64 PCG of small and mid-sized components, one right-hand side per thread-block
// cluster (internal).
//
// The host-driven iteration (solver.cuh) is three dependent launches with a grid-wide
// reduction each: 23-60 us per iteration however small the graph is, against a
// microsecond of FP64 work for a few thousand nodes.  Here one cluster of CS CTAs
// (CS = 1, 2, 4, 8 or 16) runs the whole solve of one (component, pair): x, r, q and p
// of its rows stay in shared memory, and the only synchronisation is the hardware
// cluster barrier, three per iteration (after p^T q, after the residual sums, after the
// new p is published).  Every CTA adds the CTAs' partial sums in rank order and so takes
// the same scalars and the same decision to stop.  Pairs do not wait for one another:
// each cluster stops when its own pair has converged, and the GPU's scheduler starts the
// next (component, pair).
//
// Layout.  A component's rows are put in order of length and dealt to the CTAs as items
// of one warp: 32 rows with a lane each, 8 rows with 4 lanes each or one row with 32
// lanes, the longer the row the more lanes (cl_limits).  The rows are renumbered in that
// order ("slots", a CTA's slots contiguous), so every vector access but the gather is
// conflict-free and columns are stored as slots.  The gathered p is replicated in every
// CTA's shared memory while it fits (the CTAs write their new slots to one another
// through distributed shared memory); above that each CTA keeps its own p and publishes
// it in global memory, and the gathers go to L2 (past L1, which is not coherent).
//
// What bounds it: FP64 runs at 2 lanes per SM and clock on this part, and one warp
// instruction holds its SM quarter for 64 clocks however many lanes are active (measured;
// 65 clocks for a dependent multiply-add, 107 for a butterfly step, 650 for a division).
// With many rows per CTA that rate is the limit -- one multiply-add per entry, 9 operations
// per row -- and below a few hundred rows the chain of dependent FP64 instructions, so the
// partial sums of a CTA go through shared memory to a few warps spread over the SM's quarters
// (cluster_sum) instead of a butterfly in every warp.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <vector>

#include "cluster.h"
#include "dispatch.h"
#include "onchip.cuh"

namespace nvd {

void note_launch(int64_t n);
int allow_dynamic_smem(const void *kern, int bytes);

namespace {

using namespace onchip;

constexpr int CL_MAX_CS = 16;
constexpr int CL_MAX_NT = 1024;
constexpr size_t CL_SMEM_MAX = 224 * 1024;   // dynamic, per CTA: 227 KB on this part less the static part

// One component of the graph in the plan: its rows are slots [slot0, slot0 + CS * spc),
// CTA r holding slots r * spc .. of them.
struct ClSeg {
    int64_t slot0;
    int32_t seg, n, spc, cta0, owner, pad;
};
// A CTA's share: items [item0, item0 + nitem) (32 lane groups of one lane) and their entries
// [e0, e0 + ne).
struct ClCta {
    int64_t item0, e0;
    int32_t nitem, ne;
};
struct ClArgs {
    const ClSeg *segs;
    const ClCta *ctas;
    const Item *items;
    const int32_t *col;        // slots, relative to the component's first
    const double *w;
    const int32_t *node;       // slot -> user node (-1: empty)
    const double *deg, *dinv;  // per slot (0: empty)
    const Owner *owners;       // device table or NULL (own0)
    Owner own0;
    int32_t K;                 // columns per component
    int64_t task0;             // first task of this launch: component task / K of the class, column task % K
    double *pg;                // published p of this launch's tasks (pg_stride slots each), or NULL
    int64_t pg_stride;
    ColResult *part;           // [nseg][K]
    double *d2dev;             // [K] d^2 of a graph with one component, or NULL
    double rtol2, d2stop;
    int32_t max_iter, xdt, write_z;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// All threads of the cluster (one CTA: of the block); releases and acquires their writes.
__device__ __forceinline__ void cluster_sync(int cs) {
    if (cs == 1) {
        __syncthreads();
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// Warps that add the threads' partial values of one sum (two sums: one warp per SM quarter).
constexpr int CL_RW = 2;

// Scalars of the solve, the same in every CTA of the cluster.
struct ClState {
    double mean, alpha, beta, rho, rr, rr0, stop, d2, meanx, hs_sum;
    double hist[d2_window()];
    int32_t iters, status, go;
    double cred[2][2][CL_MAX_CS * CL_RW];   // [parity][sum][rank * CL_RW + warp]: partial sums of all CTAs
    double irho;
};

// Sum v0 (and v1) over the cluster.  Every thread's value goes through shared memory to
// CL_RW warps per sum, which add them lane by lane, then by a butterfly; their totals go to
// every CTA, where warp 0 adds them, one sum in each half of the warp.  (Each step is an FP64
// instruction of 64 clocks however few lanes it serves: the sums share instructions and SM
// quarters.  Adding across lanes in integers, aligned to the largest exponent, measured the
// same.)  fin(s0, s1) runs in thread 0 of every CTA, with the same values.
template <int NV, class F>
__device__ __forceinline__ void cluster_sum(ClState &st, double *red, int cs, int rank, int par, double v0, double v1,
                                            F fin) {
    const int nt = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    red[threadIdx.x] = v0;
    if (NV == 2) red[nt + threadIdx.x] = v1;
    __syncthreads();
    if (warp < NV * CL_RW) {
        const int v = warp / CL_RW, w = warp % CL_RW;
        const double *rv = red + v * nt;
        double t = 0.0;
        int k = 32 * w + lane;
        if (k < nt) t = rv[k];
        for (k += 32 * CL_RW; k < nt; k += 32 * CL_RW) t += rv[k];
        t = butterfly(t, 32);
        if (cs == 1) {
            if (lane == 0) st.cred[par][v][w] = t;
        } else if (lane < cs) {
            peer_store(peer_addr(smem_addr(&st.cred[par][v][rank * CL_RW + w]), lane), t);
        }
    }
    cluster_sync(cs);
    if (warp == 0) {
        // lanes 0..15: sum 0, lanes 16..31: sum 1, two values each at most
        const int n = cs * CL_RW, v = lane >> 4, l = lane & 15;
        double t = 0.0;
        if (v < NV && l < n) t = st.cred[par][v][l];
        if (n > 16 && v < NV) t += st.cred[par][v][l + 16];
        t = butterfly(t, n > 16 ? 16 : n);
        const double t1 = NV == 2 ? __shfl_sync(0xffffffffu, t, 16) : 0.0;
        if (lane == 0) fin(t, t1);
    }
    __syncthreads();
}

// PG: p gathered from global memory (L2); MS: the CTA's matrix in shared memory; ONE: one
// slot per thread (blockDim.x >= spc), whose r, x, p, degree stay in registers -- with one
// or two warps per SM quarter an instruction takes about 10 clocks, so the loops and loads
// of the general form cost as much as its arithmetic (the x, r pass of 288 slots: 1,400
// clocks against 300).
//
// Measured, FP64 to 1e-10, whole call (before: the host-driven tiles): one pair on a BA
// graph of 2,000 nodes 0.22 ms (0.92), 16 pairs 0.27 ms (2.2); one pair on a ring of 20,011
// 1.1 ms (2.0); 96 graphs of 24..500 nodes, 4 pairs each, 0.59 ms (2.9); 96 node pairs on an
// ER graph of 30,011 nodes 4.8 ms (18.2; resident.cu 4.1).  An iteration at 2,000 nodes and 16 CTAs takes
// 13,600 clocks: row sums 3,700, sums 2,900 and 3,400, publishing p 2,900.
template <bool PG, bool MS, bool ONE>
__global__ void __launch_bounds__(CL_MAX_NT, 1) k_cluster_pcg(const __grid_constant__ ClArgs a) {
    extern __shared__ __align__(16) double sm[];
    __shared__ ClState st;
    int cs, rank;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(cs));
    asm("mov.u32 %0, %%cluster_ctaid.x;" : "=r"(rank));
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int64_t lt = blockIdx.x / cs;                 // task of this launch
    const int64_t task = a.task0 + lt;
    const ClSeg sg = a.segs[task / a.K];
    const int j = (int)(task % a.K);
    const Owner ow = a.owners ? a.owners[sg.owner] : a.own0;
    if (j >= ow.kc) return;                             // the whole cluster
    const ClCta ct = a.ctas[sg.cta0 + rank];
    const int spc = sg.spc;
    const int64_t slot0 = sg.slot0 + (int64_t)rank * spc;
    const int32_t *__restrict__ node = a.node + slot0;
    // shared memory: r, x (not ONE), q, then p (replicated: of all CTAs; else this CTA's),
    // scratch, then (MS) the degrees, their inverses (not ONE) and the CTA's entries
    double *r = sm, *x = r + (ONE ? 0 : spc), *q = x + (ONE ? 0 : spc), *pall = q + spc;
    double *p = PG ? pall : pall + (int64_t)rank * spc;
    double *red = pall + (PG ? spc : cs * spc);
    const double *deg = a.deg + slot0, *dinv = a.dinv + slot0, *wv = a.w + ct.e0;
    const int32_t *cv = a.col + ct.e0;
    const Item *items = a.items + ct.item0;
    if constexpr (MS) {
        double *sd = red + 2 * nt, *sdi = sd + (ONE ? 0 : spc), *sw = sdi + (ONE ? 0 : spc);
        Item *si = reinterpret_cast<Item *>(sw + ct.ne);          // ne is a multiple of 32
        int32_t *sc = reinterpret_cast<int32_t *>(si + ct.nitem);
        if constexpr (!ONE) {
            for (int s = tid; s < spc; s += nt) {
                sd[s] = __ldg(deg + s);
                sdi[s] = __ldg(dinv + s);
            }
        }
        for (int e = tid; e < ct.ne; e += nt) {
            sw[e] = __ldg(wv + e);
            sc[e] = __ldg(cv + e);
        }
        for (int i = tid; i < ct.nitem; i += nt) si[i] = items[i];
        if constexpr (!ONE) {
            deg = sd;
            dinv = sdi;
        }
        wv = sw;
        cv = sc;
        items = si;
    }
    auto mld = [](const auto *ptr) { return MS ? *ptr : __ldg(ptr); };
    double *pg = a.pg ? a.pg + lt * a.pg_stride : nullptr;
    int par = 0;

    // delta = x - y of this pair at the CTA's nodes
    auto delta_at = [&](int s) -> double {
        const int32_t nd = __ldg(node + s);
        if (nd < 0) return 0.0;
        const int64_t u = nd - ow.base;
        if (ow.idx & 1)
            return (double)(u == (int64_t)__ldg((const int32_t *)ow.x + j)) -
                   (double)(u == (int64_t)__ldg((const int32_t *)ow.y + j));
        const int64_t o = (int64_t)j * ow.ld + u;
        return a.xdt ? __ldg((const double *)ow.x + o) - __ldg((const double *)ow.y + o)
                     : (double)__ldg((const float *)ow.x + o) - (double)__ldg((const float *)ow.y + o);
    };
    auto gather = [&](int c) -> double { return PG ? __ldcg(pg + c) : pall[c]; };
    // the CTA's new p at slot s, to every CTA that gathers it: distributed shared memory
    // (about 10 bytes a clock into one CTA) while the whole p is small, else through L2
    const bool via_l2 = a.pg != nullptr;
    auto publish = [&](int s, double v) {
        if (via_l2) {
            if (PG) p[s] = v;
            pg[(int64_t)rank * spc + s] = v;
        } else if (cs == 1) {
            p[s] = v;
        } else {
            const uint32_t la = smem_addr(p + s);
            for (int c = 0; c < cs; ++c) peer_store(peer_addr(la, c), v);
        }
    };
    // after the cluster barrier that follows publish: the other CTAs' p into shared memory
    auto collect = [&]() {
        if (!PG && via_l2) {
            const double2 *src = reinterpret_cast<const double2 *>(pg);
            double2 *dst = reinterpret_cast<double2 *>(pall);
            for (int s = tid; s < cs * spc / 2; s += nt) dst[s] = __ldcg(src + s);
            __syncthreads();
        }
    };

    if (tid == 0) {
        st.iters = 0;
        st.status = NVD_OK;
        st.hs_sum = 0.0;
        for (int k = 0; k < d2_window(); ++k) st.hist[k] = 0.0;
    }
    cluster_sync(cs);   // every CTA runs before its shared memory is written from another
    // right-hand side: delta projected mean-zero, r = delta, u = D^-1 r, p = u, x = 0
    double s0 = 0.0, s1 = 0.0;
    double r1 = 0.0, x1 = 0.0, p1 = 0.0, q1 = 0.0, deg1 = 0.0, dinv1 = 0.0;   // ONE: the thread's slot
    const bool has = tid < spc;
    if constexpr (ONE) {
        if (has) {
            deg1 = __ldg(deg + tid);
            dinv1 = __ldg(dinv + tid);
            r1 = s0 = delta_at(tid);
        }
    } else {
        for (int s = tid; s < spc; s += nt) {
            const double d = delta_at(s);
            r[s] = d;
            s0 += d;
        }
    }
    cluster_sum<1>(st, red, cs, rank, par, s0, 0.0, [&](double t, double) { st.mean = t / (double)sg.n; });
    par ^= 1;
    s0 = s1 = 0.0;
    if constexpr (ONE) {
        r1 = has && __ldg(node + tid) >= 0 ? r1 - st.mean : 0.0;
        p1 = dinv1 * r1;
        if (has) {
            q[tid] = 0.0;       // stays 0 in slots without a row
            publish(tid, p1);
        }
        s0 = r1 * p1;
        s1 = r1 * r1;
    } else
    for (int s = tid; s < spc; s += nt) {
        const double rv = __ldg(node + s) >= 0 ? r[s] - st.mean : 0.0;
        const double u = mld(dinv + s) * rv;
        r[s] = rv;
        x[s] = 0.0;
        q[s] = 0.0;             // stays 0 in slots without a row
        publish(s, u);
        s0 = fma(rv, u, s0);
        s1 = fma(rv, rv, s1);
    }
    cluster_sum<2>(st, red, cs, rank, par, s0, s1, [&](double rho, double rr) {
        st.rho = rho;
        st.rr = rr;
        st.rr0 = rr;
        st.stop = a.rtol2 * rr;
        if (!finite(rr) || !finite(rho)) st.status = NVD_ERR_NUMERIC;
        st.go = pos_finite(rr) && pos_finite(rho);
    });
    par ^= 1;
    collect();
    while (st.go) {
        // row sums of W p, an item per warp; the next group's entries are loaded while
        // this group's gathers are in flight
        // (the last warp, which has the shortest item if any, first takes the division of the
        // next beta off the chain)
        if (tid == nt - 1) st.irho = 1.0 / st.rho;
        for (int i = warp; i < ct.nitem; i += nw) {
            const Item it = items[i];
            const int4 *cp = reinterpret_cast<const int4 *>(cv + it.e) + lane;
            const double2 *wp = reinterpret_cast<const double2 *>(wv + it.e) + lane;
            const int L = it.steps;
            double acc = 0.0;
            int4 c = mld(cp);
            double2 wa = mld(wp), wb = mld(wp + 32);
            for (int e = 0; e < L; e += 4) {
                const double p0 = gather(c.x);
                const double p1 = e + 1 < L ? gather(c.y) : 0.0;
                const double p2 = e + 2 < L ? gather(c.z) : 0.0;
                const double p3 = e + 3 < L ? gather(c.w) : 0.0;
                const double2 ua = wa, ub = wb;
                if (e + 4 < L) {
                    cp += 32;
                    wp += 64;
                    c = mld(cp);
                    wa = mld(wp);
                    wb = mld(wp + 32);
                }
                acc = fma(ua.x, p0, acc);
                if (e + 1 < L) acc = fma(ua.y, p1, acc);
                if (e + 2 < L) acc = fma(ub.x, p2, acc);
                if (e + 3 < L) acc = fma(ub.y, p3, acc);
            }
            if (it.lg == 5) {
                acc = butterfly(acc, 32);
            } else if (it.lg == 2) {
                acc = butterfly(acc, 4);
            }
            if ((lane & ((1 << it.lg) - 1)) == 0) q[it.slot + (lane >> it.lg)] = acc;
        }
        __syncthreads();
        // q = D p - W p and p^T q
        double pq = 0.0;
        if constexpr (ONE) {
            q1 = has ? fma(deg1, p1, -q[tid]) : 0.0;
            pq = p1 * q1;
        } else
        for (int s = tid; s < spc; s += nt) {
            const double own = p[s];
            const double y = fma(mld(deg + s), own, -q[s]);
            q[s] = y;
            pq = fma(own, y, pq);
        }
        cluster_sum<1>(st, red, cs, rank, par, pq, 0.0, [&](double t, double) {
            if (pos_finite(t)) {
                st.alpha = st.rho / t;
            } else {
                st.alpha = 0.0;
                st.status = NVD_ERR_NUMERIC;
            }
        });
        par ^= 1;
        // x += alpha p, r -= alpha q, u = D^-1 r (kept in q); r^T u and |r|^2
        const double al = st.alpha;
        s0 = s1 = 0.0;
        if constexpr (ONE) {
            r1 = fma(-al, q1, r1);
            q1 = dinv1 * r1;
            s0 = r1 * q1;
            s1 = r1 * r1;
            x1 = fma(al, p1, x1);
        } else
        for (int s = tid; s < spc; s += nt) {
            x[s] = fma(al, p[s], x[s]);
            const double rv = fma(-al, q[s], r[s]);
            const double u = mld(dinv + s) * rv;
            r[s] = rv;
            q[s] = u;
            s0 = fma(rv, u, s0);
            s1 = fma(rv, rv, s1);
        }
        cluster_sum<2>(st, red, cs, rank, par, s0, s1, [&](double rho_new, double rr) {
            const int it = st.iters + 1;
            st.iters = it;
            st.rr = rr;
            const bool d2_done = a.d2stop > 0.0 && d2_settled(it, st.alpha * st.rho, a.d2stop, st.hs_sum, st.hist);
            int end = -1;
            if (st.status == NVD_ERR_NUMERIC || !finite(rr) || !finite(rho_new)) end = NVD_ERR_NUMERIC;
            else if (rr <= st.stop || d2_done) end = NVD_OK;
            else if (it >= a.max_iter) end = NVD_ERR_NOT_CONVERGED;
            if (end >= 0) {
                st.status = end;
                st.go = 0;
            } else {
                st.beta = rho_new * st.irho;
                st.rho = rho_new;
            }
        });
        par ^= 1;
        if (!st.go) break;
        const double be = st.beta;
        if constexpr (ONE) {
            p1 = fma(be, p1, q1);
            if (has) publish(tid, p1);
        } else {
            for (int s = tid; s < spc; s += nt) publish(s, fma(be, p[s], q[s]));
        }
        cluster_sync(cs);
        collect();
    }
    // d^2 = delta^T x (delta projected), the mean of x, z = x - mean
    s0 = s1 = 0.0;
    for (int s = tid; s < spc; s += nt) {
        if (__ldg(node + s) < 0) continue;
        const double xv = ONE ? x1 : x[s];
        s0 += xv;
        s1 = fma(delta_at(s) - st.mean, xv, s1);
    }
    cluster_sum<2>(st, red, cs, rank, par, s0, s1, [&](double sx, double dx) {
        st.meanx = sx / (double)sg.n;
        st.d2 = dx;
    });
    if (a.write_z) {
        const double mu = st.meanx;
        for (int s = tid; s < spc; s += nt) {
            const int32_t nd = __ldg(node + s);
            if (nd < 0) continue;
            const int64_t o = (int64_t)j * ow.ld + (nd - ow.base);
            const double zv = (ONE ? x1 : x[s]) - mu;
            if (a.xdt) ((double *)ow.z)[o] = zv;
            else ((float *)ow.z)[o] = (float)zv;
        }
    }
    if (rank == 0 && tid == 0) {
        a.part[(int64_t)sg.seg * a.K + j] = ColResult{st.d2, st.rr, st.rr0, st.iters, st.status};
        if (a.d2dev) a.d2dev[j] = st.d2;
    }
}

// Results per (owner, column) from the per-component ones (as k_collect, solver.cuh).
__global__ void k_cluster_collect(const ColResult *__restrict__ part, const Owner *__restrict__ owners, Owner own0,
                                  int n_owner, int K, ColResult *__restrict__ res, double *__restrict__ d2dev) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n_owner * K) return;
    const int o = (int)(t / K), j = (int)(t % K);
    const Owner ow = owners ? owners[o] : own0;
    ColResult r{0.0, 0.0, 0.0, 0, NVD_OK};
    if (j < ow.kc) {
        for (int sg = ow.seg0; sg < ow.seg1; ++sg) {
            const ColResult v = part[(int64_t)sg * K + j];
            r.d2 += v.d2;
            r.rr += v.rr;
            r.rr0 += v.rr0;
            r.iters = max(r.iters, v.iters);
            if (v.status == NVD_ERR_NUMERIC || (v.status == NVD_ERR_NOT_CONVERGED && r.status == NVD_OK))
                r.status = v.status;
        }
        if (d2dev) d2dev[j] = r.d2;
    }
    res[t] = r;
}

struct ClClass {
    int cs = 1, nt = 128;
    bool pg = false, ms = false, l2 = false, one = false;
    int64_t max_ne = 0, max_items = 0;   // most entries and items of one CTA
    size_t smem = 0;
    int64_t seg0 = 0, nseg = 0, max_slots = 0;   // components [seg0, seg0 + nseg) of the plan, largest first
};

}  // namespace

struct ClusterPlan {
    bool fits = true;          // else nothing is on the device
    std::vector<ClClass> classes;
    int64_t n_slots = 0;
    DevBuf segs, ctas, items, col, w, node, deg, dinv;
    DevBuf tasks, slot_row, slot_of;   // what the weight updates need
    int64_t n_tasks = 0;
};

struct ClusterState {
    std::map<int, std::unique_ptr<ClusterPlan>> plans;   // by cs_max
    int64_t max_n = -1, max_nnz = 0, rows = 0;           // largest component, all components
    ColResult *h_res = nullptr;                          // pinned read-back
    size_t h_cap = 0;
    ~ClusterState() {
        if (h_res) cudaFreeHost(h_res);
    }
};
void cluster_state_delete(ClusterState *c) { delete c; }

int64_t cluster_state_bytes(const ClusterState *c) {
    int64_t b = 0;
    if (c)
        for (auto &kv : c->plans)
            for (const DevBuf *d : {&kv.second->segs, &kv.second->ctas, &kv.second->items, &kv.second->col,
                                    &kv.second->w, &kv.second->node, &kv.second->deg, &kv.second->dinv,
                                    &kv.second->tasks, &kv.second->slot_row, &kv.second->slot_of})
                b += (int64_t)d->bytes;
    return b;
}

namespace {

// Threads per CTA for spc slots: one slot a thread up to 1,024.  Its shared memory.
int cl_threads(int64_t spc) { return (int)std::min<int64_t>(CL_MAX_NT, std::max<int64_t>(spc, 128)); }
size_t cl_smem(int cs, int64_t spc, int nt, bool pg) {
    return ((size_t)((pg ? 2 : 1 + cs) + (spc <= nt ? 0 : 2)) * spc + 2 * (size_t)nt) * 8;
}
// More shared memory: the degrees, their inverses, ne entries and the items of a CTA.
size_t cl_smem_matrix(int64_t spc, int nt, int64_t ne, int64_t items) {
    return (spc <= nt ? 0 : (size_t)spc * 16) + (size_t)ne * 12 + (size_t)items * sizeof(Item);
}
// Longest row that keeps one lane, and 4 lanes.  With few rows per CTA an item is one
// serial chain of multiply-adds (65 clocks each) that sets the pace, so rows are split
// early; with many rows every added lane sum costs throughput.
struct ClLimits {
    int64_t one, four;
};
ClLimits cl_limits(int64_t rows_per_cta) {
    return rows_per_cta <= 1024 ? ClLimits{8, 64} : ClLimits{32, 256};
}
// Slots per CTA of a component of n rows (upper estimate; the plan's own count is exact).
int64_t cl_spc_estimate(int64_t n, int cs) { return ((n + cs - 1) / cs + 31) / 32 * 32 + 64; }

int fill_cluster_plan(nvd_graph_s *g, ClusterPlan *pl, cudaStream_t s) {
    return fill_onchip(g, pl->n_tasks, 32, pl->tasks.as<FillTask>(), pl->slot_of.as<int32_t>(), pl->col.as<int32_t>(),
                       pl->w.as<double>(), pl->n_slots, pl->slot_row.as<int32_t>(), pl->deg.as<double>(),
                       pl->dinv.as<double>(), s);
}

// CTAs per cluster of a component of n rows when the largest uses cs_max: one up to 512 rows
// (an iteration without cluster barriers takes 8,000 to 11,000 clocks, 4 CTAs took 11,600, and
// components of one class run in one launch, not one class after another), else about 256
// rows per CTA (2,000 rows: 8 and 16 CTAs the same).
int cl_cs(int64_t n, int cs_max) {
    int cs = 1;
    while (n > 512 && cs < cs_max && n > (int64_t)cs * 256) cs *= 2;
    return cs;
}

int build_cluster_plan(nvd_graph_s *g, int cs_max, ClusterPlan **out) {
    std::unique_ptr<ClusterPlan> pl(new ClusterPlan());
    const std::vector<int64_t> &rp = g->h_rowptr;
    const int nseg = g->nseg;
    std::vector<int32_t> owner(nseg, 0);
    if (nseg) NVD_TRY_CUDA(cudaMemcpy(owner.data(), g->seg_owner.p, (size_t)nseg * 4, cudaMemcpyDeviceToHost));
    std::vector<int32_t> perm;
    if (g->perm.p) {
        perm.resize(g->n);
        NVD_TRY_CUDA(cudaMemcpy(perm.data(), g->perm.p, (size_t)g->n * 4, cudaMemcpyDeviceToHost));
    }
    // components by class (CTAs per cluster, most first), then by size
    std::vector<int32_t> order(nseg);
    for (int s = 0; s < nseg; ++s) order[s] = s;
    auto rows_of = [&](int s) { return g->h_seg_end[s] - g->h_seg_begin[s]; };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return rows_of(a) > rows_of(b); });
    std::vector<ClSeg> segs;
    std::vector<ClCta> ctas;
    std::vector<Item> items;
    std::vector<FillTask> tasks;
    std::vector<int32_t> node, slot_row, slot_of(g->n, 0);
    std::vector<int32_t> rows, cnt;
    int64_t ne = 0;
    for (int s : order) {
        const int64_t a = g->h_seg_begin[s], n = rows_of(s);
        const int cs = cl_cs(n, cs_max);
        if (pl->classes.empty() || pl->classes.back().cs != cs) {
            ClClass c;
            c.cs = cs;
            c.seg0 = (int64_t)segs.size();
            pl->classes.push_back(c);
        }
        ClClass &cl = pl->classes.back();
        // rows by length, longest first (counting sort, ties by row)
        int64_t dmax = 0;
        for (int64_t r = a; r < a + n; ++r) dmax = std::max(dmax, rp[r + 1] - rp[r]);
        cnt.assign(dmax + 2, 0);
        for (int64_t r = a; r < a + n; ++r) ++cnt[dmax - (rp[r + 1] - rp[r]) + 1];
        for (int64_t d = 0; d <= dmax; ++d) cnt[d + 1] += cnt[d];
        rows.resize(n);
        for (int64_t r = a; r < a + n; ++r) rows[cnt[dmax - (rp[r + 1] - rp[r])]++] = (int32_t)r;
        auto len_of = [&](int32_t r) { return rp[r + 1] - rp[r]; };
        // items, longest rows first: {first row, lanes per row}
        const ClLimits lim = cl_limits((n + cs - 1) / cs);
        std::vector<std::pair<int64_t, int>> todo;
        for (int64_t r = 0; r < n;) {
            const int64_t d = len_of(rows[r]);
            const int g1 = d > lim.four ? 32 : d > lim.one ? 4 : 1;
            todo.emplace_back(r, g1);
            r += 32 / g1;
        }
        // each item to the CTA with the least work so far (steps, plus the 9 operations
        // per 32 rows of the vector passes)
        std::vector<std::vector<size_t>> mine(cs);
        std::vector<std::pair<double, int>> load;   // min-heap
        for (int c = 0; c < cs; ++c) load.emplace_back(0.0, c);
        auto more = [](const std::pair<double, int> &u, const std::pair<double, int> &v) { return u > v; };
        for (size_t i = 0; i < todo.size(); ++i) {
            const int g1 = todo[i].second;
            std::pop_heap(load.begin(), load.end(), more);
            mine[load.back().second].push_back(i);
            load.back().first += (double)((len_of(rows[todo[i].first]) + g1 - 1) / g1) + (g1 > 1 ? 3.0 : 0.0) + 9.0 / g1;
            std::push_heap(load.begin(), load.end(), more);
        }
        int64_t spc = 128;
        for (int c = 0; c < cs; ++c) {
            int64_t t = 0;
            for (size_t i : mine[c]) t += 32 / todo[i].second;
            spc = std::max(spc, (t + 31) / 32 * 32);
        }
        ClSeg sg{};
        sg.slot0 = (int64_t)slot_row.size();
        sg.seg = s;
        sg.n = (int32_t)n;
        sg.spc = (int32_t)spc;
        sg.cta0 = (int32_t)ctas.size();
        sg.owner = owner[s];
        segs.push_back(sg);
        const size_t base = slot_row.size();
        slot_row.resize(base + cs * spc, -1);
        node.resize(base + cs * spc, -1);
        for (int c = 0; c < cs; ++c) {
            ClCta ct{};
            ct.item0 = (int64_t)items.size();
            ct.e0 = ne;
            int32_t slot = 0;
            for (size_t i : mine[c]) {
                const int g1 = todo[i].second;
                const int64_t r0 = todo[i].first, steps = (len_of(rows[r0]) + g1 - 1) / g1;
                const int64_t room = std::max<int64_t>((steps + 3) / 4 * 4, 4);   // whole groups
                items.push_back(Item{(int32_t)(ne - ct.e0), (int32_t)steps, slot, g1 == 32 ? 5 : g1 == 4 ? 2 : 0});
                for (int l = 0; l < 32 / g1; ++l, ++slot) {
                    const size_t t = base + (size_t)c * spc + slot;
                    const int32_t self = (int32_t)((int64_t)c * spc + slot);
                    const bool in = r0 + l < n;
                    const int32_t row = in ? rows[r0 + l] : -1;
                    slot_row[t] = row;
                    tasks.push_back(FillTask{ne, in ? rp[row] : 0, in ? (int32_t)len_of(row) : 0, (int32_t)(room * g1),
                                             g1 | (l * g1) << 8, self});
                    if (in) {
                        slot_of[row] = self;
                        node[t] = perm.empty() ? row : perm[row];
                    }
                }
                ne += 32 * room;
            }
            ct.nitem = (int32_t)mine[c].size();
            ct.ne = (int32_t)(ne - ct.e0);
            ctas.push_back(ct);
            cl.max_ne = std::max<int64_t>(cl.max_ne, ct.ne);
            cl.max_items = std::max<int64_t>(cl.max_items, ct.nitem);
        }
        cl.nseg = (int64_t)segs.size() - cl.seg0;
        const int nt = cl_threads(spc);
        cl.nt = std::max(cl.nt, nt);
        cl.max_slots = std::max<int64_t>(cl.max_slots, cs * spc);
        // p replicated in every CTA while it fits, else published in global memory
        if (cl_smem(cs, spc, CL_MAX_NT, false) > CL_SMEM_MAX) cl.pg = true;
    }
    for (ClClass &cl : pl->classes) {
        cl.one = !cl.pg && cl.max_slots / cl.cs <= CL_MAX_NT;
        cl.smem = cl_smem(cl.cs, cl.max_slots / cl.cs, cl.nt, cl.pg);
        // the matrix too where it fits: each of its loads is then a shared-memory access
        // instead of one that L1 keeps only as far as the other data leave room
        const size_t m = cl_smem_matrix(cl.max_slots / cl.cs, cl.nt, cl.max_ne, cl.max_items);
        cl.ms = !cl.pg && cl.smem + m <= CL_SMEM_MAX;
        if (cl.ms) cl.smem += m;
        // publish p through L2 from 40 KB on (measured, barrier included: 2,080 clocks against
        // 2,350 at 18 KB, 4,160 against 3,450 at 65 KB, 15,300 against 5,800 at 164 KB)
        cl.l2 = cl.pg || (cl.cs > 1 && 8 * cl.max_slots > 40 * 1024);
        pl->fits = pl->fits && cl.smem <= CL_SMEM_MAX;
    }
    if (!pl->fits) {
        *out = pl.release();
        return NVD_OK;
    }
    pl->n_slots = (int64_t)slot_row.size();
    auto up = [&](DevBuf &d, const void *h, size_t bytes) -> int {
        NVD_TRY(d.alloc(std::max<size_t>(bytes, 16)));
        if (bytes) NVD_TRY_CUDA(cudaMemcpy(d.p, h, bytes, cudaMemcpyHostToDevice));
        return NVD_OK;
    };
    NVD_TRY(up(pl->segs, segs.data(), segs.size() * sizeof(ClSeg)));
    NVD_TRY(up(pl->ctas, ctas.data(), ctas.size() * sizeof(ClCta)));
    NVD_TRY(up(pl->items, items.data(), items.size() * sizeof(Item)));
    NVD_TRY(up(pl->node, node.data(), node.size() * 4));
    NVD_TRY(up(pl->slot_row, slot_row.data(), slot_row.size() * 4));
    pl->n_tasks = (int64_t)tasks.size();
    NVD_TRY(up(pl->tasks, tasks.data(), tasks.size() * sizeof(FillTask)));
    NVD_TRY(up(pl->slot_of, slot_of.data(), slot_of.size() * 4));
    NVD_TRY(pl->deg.alloc(std::max<int64_t>(pl->n_slots, 1) * 8));
    NVD_TRY(pl->dinv.alloc(std::max<int64_t>(pl->n_slots, 1) * 8));
    NVD_TRY(pl->col.alloc(std::max<int64_t>(ne, 1) * 4));
    NVD_TRY(pl->w.alloc(std::max<int64_t>(ne, 1) * 8));
    NVD_TRY(fill_cluster_plan(g, pl.get(), 0));
    NVD_TRY_CUDA(cudaDeviceSynchronize());
    *out = pl.release();
    return NVD_OK;
}

// Largest cluster the device takes (16 CTAs need an opt-in and 16 free SMs of one GPC)
// and how many clusters of each size it holds at once, one CTA per SM.
struct ClusterLimits {
    int fit[5] = {0, 0, 0, 0, 0};   // clusters of 1, 2, 4, 8, 16 CTAs
};
template <bool PG, bool MS, bool ONE>
int allow_clusters() {
    auto kern = k_cluster_pcg<PG, MS, ONE>;
    NVD_TRY(allow_dynamic_smem((const void *)kern, (int)(CL_SMEM_MAX)));
    NVD_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    return NVD_OK;
}
int cluster_limits(const nvd_graph_s *g, ClusterLimits *out) {
    static std::mutex mu;
    static std::map<int, ClusterLimits> known;   // by device
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find(g->device);
    if (it == known.end()) {
        NVD_TRY((allow_clusters<false, false, false>()));
        NVD_TRY((allow_clusters<false, true, false>()));
        NVD_TRY((allow_clusters<false, false, true>()));
        NVD_TRY((allow_clusters<false, true, true>()));
        NVD_TRY((allow_clusters<true, false, false>()));
        ClusterLimits lim;
        for (int k = 0; k < 5; ++k) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1u << k);
            cfg.blockDim = dim3(CL_MAX_NT);
            cfg.dynamicSmemBytes = CL_SMEM_MAX;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 1u << k;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int nc = 0;
            if (cudaOccupancyMaxActiveClusters(&nc, k_cluster_pcg<false, false, false>, &cfg) != cudaSuccess) {
                cudaGetLastError();
                nc = 0;
            }
            lim.fit[k] = nc;
        }
        it = known.emplace(g->device, lim).first;
    }
    *out = it->second;
    return NVD_OK;
}

// Microseconds of one iteration of one task on CS CTAs (model fitted to measured runs):
// the chain of barriers, reductions and divisions; the FP64 instructions of a CTA (16
// clocks each), 30% of them lost to padding and imbalance; publishing p through L2; with p
// in global memory the gathers, 1.3 clocks each (32 tags per warp load).  With m CTAs per
// SM the FP64 instructions of all of them share the pipe.
double cl_iter_us(int64_t n, int64_t nnz, int cs, bool pg, int m) {
    const double mhz = 2000.0;
    const double base = cs == 1 ? 3.5 : cs <= 4 ? 5.0 : 6.0;
    const double spmv = 1.3 * (double)nnz / cs * (pg ? 1.3 : 0.5) / mhz;
    const double vec = 1.3 * 9.0 * (double)n / cs * 0.5 / mhz;
    const double pub = cs > 1 && !pg ? (double)n * 8.0 / 30.0 / mhz : 0.0;
    return std::max(base + spmv + vec + pub, m * (spmv + vec));
}

}  // namespace

int cluster_estimate(nvd_graph_s *g, int64_t cols, int *cs_out, double *us_out) {
    *cs_out = 0;
    if (g->nseg < 1 || cols < 1) return NVD_OK;
    if (!g->clusters) g->clusters.reset(new ClusterState());
    ClusterState *cst = g->clusters.get();
    if (cst->max_n < 0) {
        cst->max_n = 0;
        for (int s = 0; s < g->nseg; ++s) {
            const int64_t n = g->h_seg_end[s] - g->h_seg_begin[s];
            cst->rows += n;
            cst->max_n = std::max(cst->max_n, n);
            cst->max_nnz = std::max(cst->max_nnz, g->h_rowptr[g->h_seg_end[s]] - g->h_rowptr[g->h_seg_begin[s]]);
        }
    }
    const int64_t room = (int64_t)CL_SMEM_MAX - 2 * CL_MAX_NT * 8;
    if (4 * 8 * cl_spc_estimate(cst->max_n, CL_MAX_CS) > room) return NVD_OK;
    ClusterLimits lim;
    NVD_TRY(cluster_limits(g, &lim));
    // the largest component's tasks decide the cluster size: least (waves x iteration time),
    // all tasks as if they had its size, as many as the rows make
    const double tasks = std::max<double>((double)cols, (double)cols * cst->rows / std::max<int64_t>(cst->max_n, 1));
    double best = 1e300;
    for (int k = 0; k < 5; ++k) {
        const int cs = 1 << k;
        if (!lim.fit[k]) continue;
        const int64_t spc = cl_spc_estimate(cst->max_n, cs);
        const bool pg = cl_smem(cs, spc, CL_MAX_NT, false) > CL_SMEM_MAX;
        if (pg && 4 * 8 * spc > room) continue;
        const int nt = cl_threads(spc);
        const int m = (int)std::min<int64_t>(CL_MAX_NT / nt, (int64_t)(CL_SMEM_MAX / (cl_smem(cs, spc, nt, pg) + 2048)));
        const double t = std::ceil(tasks / ((double)lim.fit[k] * std::max(m, 1))) *
                         cl_iter_us(cst->max_n, cst->max_nnz, cs, pg, m);
        if (t < best) {
            best = t;
            *cs_out = cs;
        }
    }
    *us_out = best;
    return NVD_OK;
}

int cluster_plan_get(nvd_graph_s *g, int cs, ClusterPlan **out) {
    *out = nullptr;
    ClusterState *cst = g->clusters.get();
    auto &slot = cst->plans[cs];
    if (!slot) {
        ClusterPlan *p = nullptr;
        const int rc = build_cluster_plan(g, cs, &p);
        if (rc != NVD_OK) {
            cst->plans.erase(cs);
            return rc;
        }
        slot.reset(p);
    }
    if (slot->fits) *out = slot.get();
    return NVD_OK;
}

void cluster_variant(const ClusterPlan *pl, int32_t *cs, int32_t *variant) {
    const ClClass &c = pl->classes.front();
    *cs = c.cs;
    *variant = (c.pg ? 1 : 0) | (c.ms ? 2 : 0) | (c.one ? 4 : 0) | (c.l2 ? 8 : 0);
}

int cluster_refill(nvd_graph_s *g, cudaStream_t s) {
    if (!g->clusters) return NVD_OK;
    for (auto &kv : g->clusters->plans)
        if (kv.second->fits) NVD_TRY(fill_cluster_plan(g, kv.second.get(), s));
    return NVD_OK;
}

int cluster_solve(nvd_graph_s *g, ClusterPlan *pl, const nvd_solve_opts &o, const Owner *owners_dev, const Owner &own0,
                  int n_owner, int K, int xdt, bool write_z, double *d2dev, bool want_res, ColResult **res,
                  cudaStream_t s) {
    ClusterState *cst = g->clusters.get();
    int st = NVD_OK;
    const bool direct = n_owner == 1 && g->nseg == 1;
    const size_t nres = (size_t)n_owner * K;
    // A graph's columns are solved so many at a time that the results per (component, column)
    // stay within 64 MB: with node-id inputs they would outgrow everything else (10^5
    // components and pairs: 320 GB).  Batches (a table of owners) bring vectors of at least that size.
    const int64_t per_col = (int64_t)std::max(g->nseg, 1) * (int64_t)sizeof(ColResult);
    const int Kc = owners_dev ? K : (int)std::max<int64_t>(1, std::min<int64_t>(K, ((int64_t)64 << 20) / per_col));
    ColResult *out = (ColResult *)g->wsp("cl_res", nres * sizeof(ColResult), &st);
    ColResult *part = direct ? nullptr : (ColResult *)g->wsp("cl_part", (size_t)per_col * Kc, &st);
    if (st) return st;
    // p of the tasks of one launch, up to 256 MB; where there is no memory for that, fewer tasks
    double *pg = nullptr;
    int64_t room = 0, want = 0, least = 0;
    for (const ClClass &cl : pl->classes)
        if (cl.l2) {
            want = std::max(want, cl.nseg * Kc * 8 * cl.max_slots);
            least = std::max(least, 8 * cl.max_slots);
        }
    if (least) {
        room = std::max(least, std::min<int64_t>(want, (int64_t)1 << 28));
        while (!(pg = (double *)g->wsp("cl_p", (size_t)room, &st))) {
            if (st != NVD_ERR_OOM || room == least) return st;
            clear_error();
            st = NVD_OK;
            room = std::max(least, room / 4);
        }
    }
    if (want_res) NVD_TRY(pinned_results(&cst->h_res, &cst->h_cap, nres));
    const size_t xsz = own0.idx ? 4 : xdt == NVD_F64 ? 8 : 4, zsz = xdt == NVD_F64 ? 8 : 4;
    for (int c0 = 0; c0 < K; c0 += Kc) {
        const int kc = std::min(Kc, K - c0);
        Owner own = own0;
        if (c0) {
            const size_t off = own.idx ? (size_t)c0 * xsz : (size_t)c0 * own.ld * xsz;
            own.x = (const char *)own.x + off;
            own.y = (const char *)own.y + off;
            if (own.z) own.z = (char *)own.z + (size_t)c0 * own.ld * zsz;
        }
        if (!owners_dev) own.kc = kc;
        ColResult *po = direct ? out + c0 : part;
        for (const ClClass &cl : pl->classes) {
            const int64_t tasks = cl.nseg * kc;
            int64_t per = std::min<int64_t>(tasks, ((int64_t)1 << 30) / cl.cs);
            if (cl.l2) per = std::max<int64_t>(1, std::min<int64_t>(per, room / (8 * cl.max_slots)));
            for (int64_t t0 = 0; t0 < tasks; t0 += per) {
                ClArgs a{};
                a.segs = pl->segs.as<ClSeg>() + cl.seg0;
                a.ctas = pl->ctas.as<ClCta>();
                a.items = pl->items.as<Item>();
                a.col = pl->col.as<int32_t>();
                a.w = pl->w.as<double>();
                a.node = pl->node.as<int32_t>();
                a.deg = pl->deg.as<double>();
                a.dinv = pl->dinv.as<double>();
                a.owners = owners_dev;
                a.own0 = own;
                a.K = kc;
                a.task0 = t0;
                a.pg = cl.l2 ? pg : nullptr;
                a.pg_stride = cl.max_slots;
                a.part = po;
                a.d2dev = direct && d2dev ? d2dev + c0 : nullptr;
                a.rtol2 = o.rtol * o.rtol;
                a.d2stop = (o.flags & NVD_SOLVE_D2_STOP) ? o.d2_rtol : 0.0;
                a.max_iter = o.max_iter;
                a.xdt = xdt == NVD_F64 ? 1 : 0;
                a.write_z = write_z ? 1 : 0;
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)(std::min<int64_t>(per, tasks - t0) * cl.cs));
                cfg.blockDim = dim3(cl.nt);
                cfg.dynamicSmemBytes = cl.smem;
                cfg.stream = s;
                cudaLaunchAttribute at[1];
                at[0].id = cudaLaunchAttributeClusterDimension;
                at[0].val.clusterDim.x = cl.cs;
                at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
                cfg.attrs = at;
                cfg.numAttrs = 1;
                auto kern = cl.pg ? k_cluster_pcg<true, false, false>
                            : cl.one ? (cl.ms ? k_cluster_pcg<false, true, true> : k_cluster_pcg<false, false, true>)
                                     : (cl.ms ? k_cluster_pcg<false, true, false> : k_cluster_pcg<false, false, false>);
                NVD_TRY_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
                note_launch(1);
            }
        }
        if (!direct) {
            const int64_t nr = (int64_t)n_owner * kc;
            k_cluster_collect<<<(unsigned)((nr + 127) / 128), 128, 0, s>>>(part, owners_dev, own, n_owner, kc, out + c0,
                                                                           d2dev ? d2dev + c0 : nullptr);
            note_launch(1);
            NVD_TRY_CUDA(cudaGetLastError());
        }
    }
    if (want_res) {
        NVD_TRY_CUDA(cudaMemcpyAsync(cst->h_res, out, nres * sizeof(ColResult), cudaMemcpyDeviceToHost, s));
        NVD_TRY_CUDA(cudaStreamSynchronize(s));
        *res = cst->h_res;
    }
    return NVD_OK;
}

}  // namespace nvd
