// Cluster-resident solver of the shifted Laplacian: one thread-block cluster
// takes one right-hand side from the task queue and solves it to the end on
// chip.  Its CTAs hold the inner CG vectors of the whole lattice (p, t = H p
// and e in shared memory, r and q in registers; neighbours in another CTA's
// slice come through distributed shared memory), so an inner iteration moves
// no byte of HBM, and the FP64 solution, residual and source of the outer
// defect correction are touched once per outer step.  One launch does a whole
// pt_solve / pt_trace_PAinv call: sources, inner CG, FP64 outer steps,
// convergence tests, contractions and copy-out.
//
// Why: the batched engine streams every Krylov vector through HBM (28 bytes
// per lattice site and iteration on the even Schur complement, 16^4: 0.35 us
// per right-hand side and iteration at 5.3 TB/s) and needs 12 launches per
// iteration, which is all that small lattices spend their time on.  Measured
// on one GB300, batched engine -> this kernel: 16^4, 4216 right-hand sides
// (twenty colourings, eight sets) 107.8 -> 45.5 ms; 9 x 7 x 11 x 15, full
// system, 48 right-hand sides 4.02 -> 1.00 ms; 4^4, 16 right-hand sides
// 880 -> 86 us; 16^4, 24 solves in FP64 4.20 -> 2.21 ms.
//
// What bounds it now: an iteration needs about 18 shared-memory wavefronts of
// 128 bytes per 32 entries (two hops of 7.25, and p, t, e), 0.34 of the SMs'
// shared-memory bandwidth at 16^4; the rest is latency (four cluster barriers
// and two serial sums per iteration, 16 warps per SM to cover them and the
// loads) and the FP64 pipe (0.28 busy: the outer steps' two hops).  So a
// cluster is as small as its registers allow: two CTAs of 256 threads and 128
// registers per SM, 32 entries per thread, four CTAs for 16^4.  Measured and
// not taken at 16^4: eight CTAs of 16 entries per thread, three per SM,
// 63 ms; two CTAs of 512 threads, one per SM, 49 ms.  The t neighbours that
// lie in another CTA cost 1.6 ms of 46.4 (with each slab closed on itself
// instead: 44.8 ms; before the last trims).
//
// The steps and the per-entry arithmetic are the engine's (k_eo_hop, k_eo_apply,
// k_cg_update, k_eo_outer_*, k_cg_apply, k_outer_residual, k_contract): FP32 or
// BF16-rounded inner values with FP32 arithmetic inside FP64 defect correction,
// or FP64 throughout; dot products as sums of eight entries and warp trees in
// the arithmetic type, then FP64 sums in a fixed order.  Different on purpose:
// CG keeps its direction across a residual replacement, and a last cycle that
// kept it ends at an eighth of the tolerance (PT_CG_KEEP, PT_CG_LAST2); the
// engine restarts and ends at the tolerance.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>

#include "engine.cuh"

// CTAs per cluster: above 8 by opt-in, only for lattices that 8 cannot hold
// (measured against the batched engine, ms: 24 x 22 x 10 x 22, 64 solves 2.7 : 5.3;
// 16^3 x 64, 64 solves 5.3 : 11.1; 16^2 x 24^2, 200 solves 7.7 : 14.4; 14 x 12 x 18^2
// in FP64, 20 solves 2.4 : 4.6)
#define RES_MAXC 16
#define RES_PORTC 8                 // the portable limit
#define RES_MAXW 16                 // warps per CTA

struct ResP {
    Geom g;
    int nh, n_loc, C;               // entries of a field (N/2 even-odd, N full), per CTA, CTAs per cluster
    int Te;                         // threads at work: whole xy planes of units
    int nt, nt_last;                // t planes per CTA, and of the last one
    int row, sy, sz, st;            // entries of an x row; entry offsets of the y, z, t neighbours
    double diag, inv_dd;            // d = 8 + m2 and 1 / d, formed on the host: a division costs the FP64 pipe
    float diag_f, inv_df;
    int mode;
    const int32_t *col;
    uint64_t seed;
    int mu, n_p;
    int p[PT_MAX_P];
    int n_lev, n_pr, m_fin;
    const int32_t *lev_cols;
    const int *lev_anc;
    const Task *tasks;
    int n_tasks;
    const double *B_user;
    double *X_user;
    double *x64, *t64, *b64;        // [clusters][nh] scratch of the task in flight
    int *head, *flags;
    TaskStat *tstat;
    double *task_out;
    double tol, delta;
    int maxit, max_inner;
    long long max_steps;            // inner iterations + outer steps of one task before it gives up
};

// scalars of the task in flight: every CTA of the cluster computes the same
// values from the same sums (thread 0), the other threads read them
enum { RS_INNER = 0, RS_OUTER = 1, RS_DONE = 2 };
struct ResSh {
    double red[2][3][RES_MAXC * RES_MAXW];   // warp sums of every CTA, double-buffered
    double part[RES_MAXC][PT_MAX_P];         // contraction sums of every CTA (used in CTA 0)
    double alpha, beta;                      // in the arithmetic type: FP32 uses the first half
    double rr, rr_rec, target2, b2;          // rr_rec: |r|^2 the recursion had when its cycle ended
    long long steps;
    int inner_it, total_it, outer_it, phase, task, fresh;   // fresh: the next direction is r itself
    int cnt[RES_MAXW];
};

// the Z2 noise of a site as the sign bit of its hash (pt_noise without the FP64 pipe)
__device__ __forceinline__ bool res_minus(uint64_t key, int site) {
    return (pt_mix64(key + ((uint64_t)site + 1ULL) * PT_GAMMA) >> 63) != 0;
}

__device__ __forceinline__ uint32_t res_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t res_remote(const void *p, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(res_smem(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ int res_ctarank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ int res_clusterid() {
    uint32_t r;
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ void res_sync(int C) {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
// volatile keeps these between the cluster barriers, which order them; without a memory
// clobber the compiler may move this CTA's own shared-memory loads past them
template <int V>
__device__ __forceinline__ void res_ldr(const float *p, int rank, float v[V]) {
    if constexpr (V == 4)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(res_remote(p, rank)));
    else
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[0]) : "r"(res_remote(p, rank)));
}
template <int V>
__device__ __forceinline__ void res_ldr(const double *p, int rank, double v[V]) {
    if constexpr (V == 4) {
        const uint32_t a = res_remote(p, rank);
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(a));
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2 + 16];" : "=d"(v[2]), "=d"(v[3]) : "r"(a));
    } else {
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[0]) : "r"(res_remote(p, rank)));
    }
}
__device__ __forceinline__ void res_str(double *p, int rank, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(res_remote(p, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void res_str(float2 *p, int rank, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(res_remote(p, rank)), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void res_str(int *p, int rank, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(res_remote(p, rank)), "r"(v) : "memory");
}
__device__ __forceinline__ void res_ld4(const float *p, float v[4]) {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
__device__ __forceinline__ void res_ld4(const double *p, double v[4]) {
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void res_st4(float *p, const float v[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void res_st4(double *p, const double v[4]) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
template <int V, typename F>
__device__ __forceinline__ void res_ld(const F *p, F v[V]) {
    if constexpr (V == 4) res_ld4(p, v);
    else v[0] = p[0];
}
template <int V, typename F>
__device__ __forceinline__ void res_st(F *p, const F v[V]) {
    if constexpr (V == 4) res_st4(p, v);
    else p[0] = v[0];
}

// What a thread knows of its units' neighbours, once per launch.  A CTA holds
// nt whole t planes; thread tid takes the units tid, tid + Te, ... with Te a
// multiple of the xy plane, so that its x and y, and with them the x and y
// neighbour offsets, are the same for all its units, and one bit per unit
// says the rest: the row's parity and whether z or t is at its lower or upper
// end (for t: of the CTA's slab, where the neighbour is another CTA's).
struct ResNb {
    int l0;                     // first unit's entry (beyond the slice for a thread without work)
    int yf, yb, xl, xr;         // offsets: y+, y-, and the entry left / right of the unit (wrapped in its row)
    uint32_t par, zl, zh, tl, th;
};

template <int EO, int V, int U>
__device__ __forceinline__ ResNb res_neighbours(const ResP &P, int base, int nv, int nt_mine) {
    ResNb n;
    const int tid = threadIdx.x;
    n.l0 = tid < P.Te ? V * tid : 0x3fffffff;
    n.yf = n.yb = n.xl = n.xr = 0;
    n.par = n.zl = n.zh = n.tl = n.th = 0;
#pragma unroll 1
    for (int u = 0; u < U; ++u) {
        const int l = n.l0 + u * V * P.Te;
        if (tid >= P.Te || l >= nv) break;
        int x[4];
        site_coords(P.g, EO ? 2 * (base + l) : base + l, x);
        const int c = EO ? x[0] >> 1 : x[0];
        n.xl = c == 0 ? P.row - 1 : -1;
        n.xr = c + V == P.row ? V - P.row : V;
        n.yf = x[1] == P.g.D[1] - 1 ? -(P.g.D[1] - 1) * P.sy : P.sy;
        n.yb = x[1] == 0 ? (P.g.D[1] - 1) * P.sy : -P.sy;
        const int tt = x[3] - base / P.st;
        n.par |= (uint32_t)((x[1] + x[2] + x[3]) & 1) << u;
        n.zl |= (uint32_t)(x[2] == 0) << u;
        n.zh |= (uint32_t)(x[2] == P.g.D[2] - 1) << u;
        n.tl |= (uint32_t)(tt == 0) << u;
        n.th |= (uint32_t)(tt == nt_mine - 1) << u;
    }
    return n;
}

__device__ __forceinline__ ResNb res_opaque(ResNb n) {
    asm volatile("" : "+r"(n.l0), "+r"(n.yf), "+r"(n.yb), "+r"(n.xl), "+r"(n.xr));
    asm volatile("" : "+r"(n.par), "+r"(n.zl), "+r"(n.zh), "+r"(n.tl), "+r"(n.th));
    return n;
}

// Sum over the eight neighbours of the unit at l (a thread's unit u), added in
// the engine's order x+, x-, y+, y-, z+, z-, t+, t-.  Even-odd: the unit's
// sites have parity par and `buf` holds the other parity (the x neighbours of
// entry k are entries k and k - 1 of the row, or k + 1 and k, by the site's x
// parity).
template <int EO, int V, typename F>
__device__ __forceinline__ void res_nbsum(const ResP &P, const F *buf, const ResNb &n, int u, int l, int rank,
                                          int nt_mine, int par, F acc[V]) {
    const F *own = buf + l;
    const uint32_t bit = 1u << u;
    // The t neighbours first: at the slab's ends they are another CTA's, the
    // longest way (t+: the next CTA's first plane, t-: the last plane of the one
    // before).  Both are loaded through the cluster's address space wherever they
    // lie: a branch around a remote load kept the loads of the next unit behind
    // it (16^4: 46.4 ms with the branch, 43.9 without).
    F tf[V], tb[V], t[V];
    {
        const int prev = rank == 0 ? P.C - 1 : rank - 1, next = rank + 1 == P.C ? 0 : rank + 1;
        const bool hi = (n.th & bit) != 0, lo = (n.tl & bit) != 0;
        res_ldr<V>(own + (hi ? -(nt_mine - 1) * P.st : P.st), hi ? next : rank, tf);
        res_ldr<V>(own + (lo ? ((prev == P.C - 1 ? P.nt_last : P.nt) - 1) * P.st : -P.st), lo ? prev : rank, tb);
    }
    if constexpr (EO) {
        const bool odd_x = ((n.par >> u) ^ (uint32_t)par) & 1u;
        F Q[V], sW;
        res_ld<V>(own, Q);
        const F W = own[odd_x ? n.xr : n.xl];
        if constexpr (V == 4) {
            const F s01 = Q[1] + Q[0], s12 = Q[2] + Q[1], s23 = Q[3] + Q[2];
            sW = W + (odd_x ? Q[3] : Q[0]);
            acc[0] = odd_x ? s01 : sW;
            acc[1] = odd_x ? s12 : s01;
            acc[2] = odd_x ? s23 : s12;
            acc[3] = odd_x ? sW : s23;
        } else {
            acc[0] = Q[0] + W;
        }
    } else {
        static_assert(EO || V == 1, "the full system takes one site per unit");
        acc[0] = own[n.xr];
        acc[0] += own[n.xl];
    }
    res_ld<V>(own + n.yf, t);
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += t[k];
    res_ld<V>(own + n.yb, t);
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += t[k];
    res_ld<V>(own + ((n.zh & bit) ? -(P.g.D[2] - 1) * P.sz : P.sz), t);
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += t[k];
    res_ld<V>(own + ((n.zl & bit) ? (P.g.D[2] - 1) * P.sz : -P.sz), t);
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += t[k];
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += tf[k];
#pragma unroll
    for (int k = 0; k < V; ++k) acc[k] += tb[k];
}

// Sums over a CTA's entries.  FP32 chains stay as short as the engine's, whose
// warps add eight entries per lane and the 32 lanes in FP32: one sum per eight
// entries of a thread (NG of them), each added over the warp by a tree of its
// own; what is added beyond that is an unevaluated pair hi + lo (Knuth's
// two-sum).  This and FP64 sums of |r|^2 on the full system against one FP32
// chain over a thread's 16 or 32 entries: 16^4, 4216 solves 44.4 -> 45.6 ms;
// 9 x 7 x 11 x 15, 48 solves 0.97 -> 1.02 ms.
template <typename R, int KPT>
struct ResAcc {
    static constexpr int NG = std::is_same<R, float>::value && KPT > 8 ? KPT / 8 : 1;
    R g[NG];
    __device__ __forceinline__ ResAcc() {
#pragma unroll
        for (int i = 0; i < NG; ++i) g[i] = R(0);
    }
    // entry k of the thread (known where it is unrolled)
    __device__ __forceinline__ void add(int k, R v) { g[NG == 1 ? 0 : k / 8] += v; }
    __device__ __forceinline__ double total() const {
        double s = (double)g[0];
#pragma unroll
        for (int i = 1; i < NG; ++i) s += (double)g[i];
        return s;
    }
};

__device__ __forceinline__ void res_pair(float &hi, float &lo, float h, float l) {
    const float s = hi + h, b = s - hi;
    lo = (lo + l) + ((hi - (s - b)) + (h - b));
    hi = s;
}
__device__ __forceinline__ float res_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
// half of the lanes go on with a, half with b, each taking the other half's
__device__ __forceinline__ float res_split(float a, float b, int o) {
    const bool h = (threadIdx.x & o) != 0;
    return (h ? b : a) + res_xor(h ? a : b, o);
}
template <int KPT>
__device__ __forceinline__ float2 res_warp(const ResAcc<float, KPT> &a) {
    constexpr int NG = ResAcc<float, KPT>::NG;
    static_assert(NG == 1 || NG == 2 || NG == 4, "sums of eight entries");
    float hi, lo = 0.f;
    if constexpr (NG == 4) hi = res_split(res_split(a.g[0], a.g[2], 16), res_split(a.g[1], a.g[3], 16), 8);
    else if constexpr (NG == 2) hi = res_split(a.g[0], a.g[1], 16);
    else hi = a.g[0];
#pragma unroll
    for (int o = 16 / NG; o > 0; o >>= 1) hi += res_xor(hi, o);
    if constexpr (NG == 4) res_pair(hi, lo, res_xor(hi, 8), 0.f);
    if constexpr (NG > 1) res_pair(hi, lo, res_xor(hi, 16), res_xor(lo, 16));
    return make_float2(hi, lo);
}

template <typename R>
__device__ __forceinline__ R &res_scalar(double &d) { return *reinterpret_cast<R *>(&d); }

// shuffles that add up n values, one per lane or several, at lane 0
__device__ __forceinline__ int res_span(int n) { return n > 16 ? 16 : n > 8 ? 8 : n > 4 ? 4 : n > 2 ? 2 : n > 1 ? 1 : 0; }

// Sums of K FP64 values over the cluster, in thread 0 of every CTA (which alone
// uses them: the upper lanes of its warp hold parts): warp trees, the warp sums
// of all CTAs gathered in each, added in a fixed order.  One cluster barrier.
template <int K>
__device__ __forceinline__ void res_totals(ResSh &sh, int &buf, int C, int rank, double (&v)[K], double (&tot)[K]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (C == 1) {
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; ++k) sh.red[buf][k][warp] = v[k];
    } else if (lane < C) {
#pragma unroll
        for (int k = 0; k < K; ++k) res_str(sh.red[buf][k] + rank * nw + warp, lane, v[k]);
    }
    res_sync(C);
    if (warp == 0) {
        const int n = C * nw;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double s = 0.0;
            for (int i = lane; i < n; i += 32) s += sh.red[buf][k][i];
            for (int o = res_span(n); o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            tot[k] = s;
        }
    }
    buf ^= 1;
}

// the same for one sum in the inner solve's arithmetic
template <int KPT>
__device__ __forceinline__ double res_total(ResSh &sh, int &buf, int C, int rank, const ResAcc<double, KPT> &a) {
    double v[1] = {a.g[0]}, tot[1];
    res_totals<1>(sh, buf, C, rank, v, tot);
    return tot[0];
}
template <int KPT>
__device__ __forceinline__ double res_total(ResSh &sh, int &buf, int C, int rank, const ResAcc<float, KPT> &a) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const float2 v = res_warp(a);
    float2 *const red = reinterpret_cast<float2 *>(sh.red[buf][0]);
    if (C == 1) {
        if (lane == 0) red[warp] = v;
    } else if (lane < C) {
        res_str(red + rank * nw + warp, lane, v);
    }
    res_sync(C);
    double s = 0.0;
    if (warp == 0) {
        const int n = C * nw;
        for (int i = lane; i < n; i += 32) {
            const float2 w = red[i];
            s += (double)w.x;
            if constexpr (ResAcc<float, KPT>::NG > 1) s += (double)w.y;
        }
        for (int o = res_span(n); o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    buf ^= 1;
    return s;
}

// the engine's k_fin_outer (thread 0 of every CTA; CTA 0 reports)
template <typename R>
__device__ __forceinline__ void res_outer_step(const ResP &P, ResSh &sh, int rank, bool start, const double tot[3]) {
    if (start) {
        sh.b2 = tot[1];
        sh.total_it = 0;
        sh.outer_it = 0;
        sh.steps = 0;
    }
    const double rel = sh.b2 > 0.0 ? sqrt(tot[0] / sh.b2) : 0.0;
    sh.outer_it += 1;
    sh.steps += 1;
    const bool finite = isfinite(tot[0]);
    const bool conv = sh.b2 == 0.0 || rel <= P.tol;
    const bool late = sh.steps >= P.max_steps;
    if (conv || !finite || sh.total_it >= P.maxit || late) {
        if (rank == 0) {
            if (!finite) atomicOr(&P.flags[FLAG_NUMERIC], 1);
            else if (!conv && sh.total_it >= P.maxit) atomicAdd(&P.flags[FLAG_NOCONV], 1);
            else if (!conv) atomicOr(&P.flags[FLAG_TIMEOUT], 1);
            P.tstat[sh.task] = TaskStat{sh.total_it, sh.outer_it, rel};
        }
        sh.phase = RS_DONE;
    } else {
        sh.phase = RS_INNER;
        sh.inner_it = 0;
        sh.fresh = start || !(tot[2] <= PT_CG_KEEP * sh.rr_rec);
        res_scalar<R>(sh.beta) = (R)(sh.fresh ? 0.0 : tot[2] / sh.rr);
        sh.rr = tot[2];
        sh.target2 = fmax(P.delta * P.delta * tot[2], 0.25 * P.tol * P.tol * sh.b2);
        // a last cycle that keeps its direction goes on to an eighth of the tolerance (PT_CG_KEEP)
        if (!sh.fresh && sh.target2 <= P.tol * P.tol * sh.b2)
            sh.target2 = fmin(sh.target2, PT_CG_LAST2 * P.tol * P.tol * sh.b2);
    }
}

template <typename S, typename R>
__device__ __forceinline__ R res_rnd(R v) {
    if constexpr (std::is_same<S, __nv_bfloat16>::value) return __bfloat162float(__float2bfloat16_rn(v));
    else return v;
}

// S: storage type of the inner vectors (BF16: FP32 values rounded to BF16);
// EO: even Schur complement; V: entries per unit (4: D_0 a multiple of 8);
// KPT: entries per thread; TMAX: threads per CTA
template <typename S, int EO, int V, int KPT, int TMAX, int MINB>
__global__ void __launch_bounds__(TMAX, MINB) k_lap_resident(const __grid_constant__ ResP P) {
    typedef typename std::conditional<std::is_same<S, double>::value, double, float>::type R;
    constexpr int U = KPT / V;
    extern __shared__ __align__(16) unsigned char res_dyn[];
    __shared__ ResSh sh;
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    const int C = P.C, rank = C == 1 ? 0 : res_ctarank();
    const int cl = C == 1 ? (int)blockIdx.x : res_clusterid();
    const int n_cap = T * KPT;
    R *const ps = reinterpret_cast<R *>(res_dyn);
    R *const ts = ps + n_cap;
    R *const es = ts + n_cap;
    double *const xs = reinterpret_cast<double *>(res_dyn);      // over p (and t): n_cap doubles
    int *const lst = reinterpret_cast<int *>(res_dyn);           // over the same: 2 n_cap ints
    const int base = rank * P.n_loc;
    const int nv = max(0, min(P.n_loc, P.nh - base));            // entries of this CTA (a multiple of V)
    double *const x64 = P.x64 + (size_t)cl * P.nh + base;
    double *const t64 = P.t64 + (size_t)cl * P.nh + base;
    double *const b64 = P.b64 + (size_t)cl * P.nh + base;
    R diag, inv_d;
    if constexpr (std::is_same<R, double>::value) { diag = P.diag; inv_d = P.inv_dd; }
    else { diag = P.diag_f; inv_d = P.inv_df; }
    const double inv_dd = P.inv_dd;
    const int nt_mine = rank == C - 1 ? P.nt_last : P.nt;
    const ResNb nb0 = res_neighbours<EO, V, U>(P, base, nv, nt_mine);
    int buf = 0;
    // Each sweep over the units starts from a copy of nb that the compiler
    // cannot trace back: it would otherwise keep every unit's addresses and
    // selected offsets in registers from one sweep to the next, and spill.
#define RES_UNITS                                                              \
    {                                                                          \
        const ResNb nb = res_opaque(nb0);                                      \
        _Pragma("unroll") for (int u = 0; u < U; ++u) {                        \
            const int l = nb.l0 + u * V * P.Te;                                \
            if (l >= nv) continue;
#define RES_UNITS_END                                                          \
        }                                                                      \
    }

    R r[U][V];
    res_sync(C);                         // every CTA of the cluster runs before its shared memory is addressed
    while (true) {
        if (rank == 0 && tid == 0) {
            const int t = atomicAdd(P.head, 1);
            for (int c = 0; c < C; ++c) {
                if (C == 1) sh.task = t;
                else res_str(&sh.task, c, t);
            }
        }
        res_sync(C);
        if (sh.task >= P.n_tasks) break;
        const Task tk = P.tasks[sh.task];
        const uint64_t key = P.mode == MODE_SOLVE ? 0 : pt_set_key(P.seed, tk.set);
        const int32_t *col = P.mode == MODE_SOLVE ? nullptr : P.col + (size_t)tk.cidx * P.g.N;
        const double *bu = P.mode == MODE_SOLVE ? P.B_user + (size_t)tk.set * P.g.N : nullptr;
        auto probe_at = [&](int site) -> float {       // the probe's entry: 0 or +-1
            return col[site] == tk.colour ? (res_minus(key, site) ? -1.f : 1.f) : 0.f;
        };

        // -------- source: b' (x = 0, so r = b'), |b|^2, and the rounded r
        {
            double v[3] = {0.0, 0.0, 0.0};
            ResAcc<R, KPT> v2;
            if constexpr (EO) {
                if (P.mode == MODE_SOLVE) {
                    RES_UNITS
                        const int b = (int)((nb.par >> u) & 1u);
                        double o[V];
#pragma unroll
                        for (int k = 0; k < V; ++k) o[k] = bu[2 * (base + l + k) + 1 - b];
                        res_st<V>(xs + l, o);
                    RES_UNITS_END
                } else {
                    RES_UNITS
                        const int b = (int)((nb.par >> u) & 1u);
                        R o[V], e[V];
#pragma unroll
                        for (int k = 0; k < V; ++k) {
                            e[k] = (R)probe_at(2 * (base + l + k) + b);
                            o[k] = (R)probe_at(2 * (base + l + k) + 1 - b);
                        }
                        res_st<V>(ps + l, e);
                        res_st<V>(ts + l, o);
                    RES_UNITS_END
                }
                res_sync(C);
            }
            float v1f = 0.f;
            RES_UNITS
                double bp[V];
                if constexpr (EO) {
                    if (P.mode == MODE_SOLVE) {
                        const int b = (int)((nb.par >> u) & 1u);
                        double hs[V], o[V];
                        res_ld<V>(xs + l, o);
                        res_nbsum<EO, V, double>(P, xs, nb, u, l, rank, nt_mine, 0, hs);
#pragma unroll
                        for (int k = 0; k < V; ++k) {
                            const double be = bu[2 * (base + l + k) + b];
                            v[1] += be * be + o[k] * o[k];
                            bp[k] = be + hs[k] * inv_dd;
                        }
                    } else {                            // 0 and +-1: the sums are exact in R
                        R hs[V], e[V], o[V];
                        res_ld<V>(ps + l, e);
                        res_ld<V>(ts + l, o);
                        res_nbsum<EO, V, R>(P, ts, nb, u, l, rank, nt_mine, 0, hs);
#pragma unroll
                        for (int k = 0; k < V; ++k) {
                            v1f += (float)(e[k] * e[k] + o[k] * o[k]);
                            bp[k] = 0.0;
                            if (e[k] != R(0) || hs[k] != R(0)) bp[k] = (double)e[k] + (double)hs[k] * inv_dd;
                        }
                    }
                } else {
                    bp[0] = P.mode == MODE_SOLVE ? bu[base + l] : (double)probe_at(base + l);
                    v[1] += bp[0] * bp[0];
                }
                double zero[V];
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    zero[k] = 0.0;
                    v[0] += bp[k] * bp[k];
                    r[u][k] = res_rnd<S, R>((R)bp[k]);
                    if constexpr (EO) v2.add(u * V + k, r[u][k] * r[u][k]);
                    else v[2] += (double)r[u][k] * (double)r[u][k];
                }
                res_st<V>(b64 + l, bp);
                res_st<V>(x64 + l, zero);
                if constexpr (EO) res_st<V>(t64 + l, zero);
            RES_UNITS_END
            v[1] += (double)v1f;
            v[2] += v2.total();
            double tot[3];
            res_totals<3>(sh, buf, C, rank, v, tot);
            if (tid == 0) res_outer_step<R>(P, sh, rank, true, tot);
            __syncthreads();
        }

        // At the start of a cycle the e array holds the kept direction p (the outer step uses the
        // p and t arrays for FP64 values); the first iteration takes it from there and sets e = 0.
        // The update e += alpha p of an iteration is left to the next one, which reads p anyway.
        bool resume = true, pending = false;
        R al = R(0);
        while (sh.phase != RS_DONE) {
            // -------- inner CG on S e = r
            while (true) {
                const bool first = sh.fresh != 0;
                const R be = res_scalar<R>(sh.beta);
                RES_UNITS
                    R po[V], pn[V], e[V];
                    if (resume) {
                        res_ld<V>(es + l, po);
#pragma unroll
                        for (int k = 0; k < V; ++k) e[k] = R(0);
                    } else {
                        res_ld<V>(ps + l, po);
                        res_ld<V>(es + l, e);
#pragma unroll
                        for (int k = 0; k < V; ++k) e[k] = res_rnd<S, R>(e[k] + al * po[k]);
                    }
                    res_st<V>(es + l, e);
#pragma unroll
                    for (int k = 0; k < V; ++k) pn[k] = first ? r[u][k] : res_rnd<S, R>(r[u][k] + be * po[k]);
                    res_st<V>(ps + l, pn);
                RES_UNITS_END
                pending = false;
                resume = false;
                res_sync(C);
                if constexpr (EO) {
                    RES_UNITS
                        R hs[V];
                        res_nbsum<EO, V, R>(P, ps, nb, u, l, rank, nt_mine, 1, hs);
#pragma unroll
                        for (int k = 0; k < V; ++k) hs[k] = res_rnd<S, R>(hs[k]);
                        res_st<V>(ts + l, hs);
                    RES_UNITS_END
                    res_sync(C);
                }
                R q[U][V];
                ResAcc<R, KPT> pq;
                RES_UNITS
                    R hs[V], pc[V];
                    res_nbsum<EO, V, R>(P, EO ? ts : ps, nb, u, l, rank, nt_mine, 0, hs);
                    res_ld<V>(ps + l, pc);
#pragma unroll
                    for (int k = 0; k < V; ++k) {
                        q[u][k] = res_rnd<S, R>(EO ? diag * pc[k] - hs[k] * inv_d : diag * pc[k] - hs[k]);
                        pq.add(u * V + k, pc[k] * q[u][k]);
                    }
                RES_UNITS_END
                double tot = res_total(sh, buf, C, rank, pq);
                if (tid == 0) {
                    if (!(tot > 0.0) || !isfinite(tot)) {            // restart from the true residual
                        if (rank == 0) atomicOr(&P.flags[FLAG_NUMERIC], 2);
                        sh.rr_rec = -1.0;
                        sh.phase = RS_OUTER;
                    } else {
                        res_scalar<R>(sh.alpha) = (R)(sh.rr / tot);
                    }
                }
                __syncthreads();
                if (sh.phase == RS_OUTER) break;
                al = res_scalar<R>(sh.alpha);
                pending = true;
                ResAcc<R, KPT> rn;
                RES_UNITS
#pragma unroll
                    for (int k = 0; k < V; ++k) {
                        r[u][k] = res_rnd<S, R>(r[u][k] - al * q[u][k]);
                        rn.add(u * V + k, r[u][k] * r[u][k]);
                    }
                RES_UNITS_END
                tot = res_total(sh, buf, C, rank, rn);
                if (tid == 0) {
                    sh.inner_it += 1;
                    sh.total_it += 1;
                    sh.steps += 1;
                    if (tot <= sh.target2 || sh.inner_it >= P.max_inner || sh.total_it >= P.maxit ||
                        !isfinite(tot) || sh.steps >= P.max_steps) {
                        sh.rr_rec = tot;
                        sh.phase = RS_OUTER;
                    } else {
                        sh.fresh = 0;
                        res_scalar<R>(sh.beta) = (R)(tot / sh.rr);
                        sh.rr = tot;
                    }
                }
                __syncthreads();
                if (sh.phase == RS_OUTER) break;
            }

            // -------- outer step: x64 += e, r = b' - S x64 (FP64), e = 0
            double v[3] = {0.0, 0.0, 0.0};
            ResAcc<R, KPT> v2;
            // every read of p and t by another CTA is past a barrier of res_totals
            RES_UNITS
                R e[V], pc[V];
                double x[V];
                res_ld<V>(x64 + l, x);
                res_ld<V>(es + l, e);
                res_ld<V>(ps + l, pc);
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    if (pending) e[k] = res_rnd<S, R>(e[k] + al * pc[k]);
                    x[k] += (double)e[k];
                }
                res_st<V>(x64 + l, x);
                res_st<V>(es + l, pc);
            RES_UNITS_END
            __syncthreads();             // p is saved: x64 may take its place in shared memory
            RES_UNITS
                double x[V];
                res_ld<V>(x64 + l, x);
                res_st<V>(xs + l, x);
            RES_UNITS_END
            res_sync(C);
            if constexpr (EO) {
                RES_UNITS
                    double th[V];
                    res_nbsum<EO, V, double>(P, xs, nb, u, l, rank, nt_mine, 1, th);
                    res_st<V>(t64 + l, th);
                RES_UNITS_END
                res_sync(C);
                RES_UNITS
                    double th[V];
                    res_ld<V>(t64 + l, th);
                    res_st<V>(xs + l, th);
                RES_UNITS_END
                res_sync(C);
            }
            RES_UNITS
                double hs[V], x[V], bp[V];
                res_nbsum<EO, V, double>(P, xs, nb, u, l, rank, nt_mine, 0, hs);
                res_ld<V>(x64 + l, x);
                res_ld<V>(b64 + l, bp);
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    // b' - d x + H t / d, two fused multiply-adds
                    const double rx = fma(-P.diag, x[k], bp[k]);
                    const double rv = EO ? fma(hs[k], inv_dd, rx) : rx + hs[k];
                    v[0] += rv * rv;
                    r[u][k] = res_rnd<S, R>((R)rv);
                    if constexpr (EO) v2.add(u * V + k, r[u][k] * r[u][k]);
                    else v[2] += (double)r[u][k] * (double)r[u][k];
                }
            RES_UNITS_END
            resume = true;
            v[2] += v2.total();
            double tot[3];
            res_totals<3>(sh, buf, C, rank, v, tot);
            if (tid == 0) res_outer_step<R>(P, sh, rank, false, tot);
            __syncthreads();
        }

        // -------- copy-out, or contraction v^H P x.  Even-odd: x_o = (b_o + t64) / d with the
        // t64 = H_oe x64 of the last outer step (zero for a task that converged with x = 0)
        if (P.mode == MODE_SOLVE) {
            double *X = P.X_user + (size_t)tk.set * P.g.N;
            RES_UNITS
                double x[V];
                res_ld<V>(x64 + l, x);
                if constexpr (EO) {
                    double th[V];
                    res_ld<V>(t64 + l, th);
                    const int b = (int)((nb.par >> u) & 1u);
#pragma unroll
                    for (int k = 0; k < V; ++k) {
                        const int s2 = 2 * (base + l + k);
                        const double bo = bu[s2 + 1 - b];
                        X[s2 + b] = x[k];
                        X[s2 + 1 - b] = (bo + th[k]) * inv_dd;
                    }
                } else {
                    X[base + l] = x[0];
                }
            RES_UNITS_END
            res_sync(C);                 // the next task overwrites the shared buffers and the scalars
            continue;
        }
        // (every read of the shared field is past the barrier in res_totals: the lists take its place)
        // members of the probe's class (nested: of its coarsest ancestor), per warp in a fixed order;
        // bit 30: the noise is -1
        constexpr int W2 = EO ? 2 : 1;
        int *const my = lst + (size_t)warp * 32 * KPT * W2;
        int n_my = 0;
#pragma unroll 1
        for (int u = 0; u < U; ++u) {
            const int l = nb0.l0 + u * V * P.Te;
#pragma unroll 1
            for (int k = 0; k < V * W2; ++k) {
                int site = 0;                        // (l of a thread without work is beyond what W2 l may be)
                bool in = false;
                if (l < nv) {
                    site = W2 * (base + l) + k;
                    in = P.n_lev ? P.lev_cols[site] == P.lev_anc[tk.colour] : col[site] == tk.colour;
                }
                const unsigned m = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const bool neg = res_minus(key, site);
                    my[n_my + __popc(m & ((1u << lane) - 1u))] = site | (neg ? 1 << 30 : 0);
                }
                n_my += __popc(m);
            }
        }
        if (lane == 0) sh.cnt[warp] = n_my;
        res_sync(C);                     // lists and counts for the CTA; x64 and t64 for the cluster
        const double *xg = P.x64 + (size_t)cl * P.nh, *tg = P.t64 + (size_t)cl * P.nh;
        for (int n = warp; n < P.n_p; n += nw) {
            double acc = 0.0;
            const int lev = P.n_lev ? n / P.n_pr : 0;
            for (int w = 0; w < nw; ++w) {
                const int *li = lst + (size_t)w * 32 * KPT * W2;
                for (int i = lane; i < sh.cnt[w]; i += 32) {
                    const int site = li[i] & 0x3fffffff;
                    if (lev > 0 && P.lev_cols[(size_t)lev * P.g.N + site] != P.lev_anc[(size_t)lev * P.m_fin + tk.colour])
                        continue;
                    int x[4], cm;
                    site_coords(P.g, site, x);
                    const int y = shift_fwd(P.g, site, x, P.mu, P.p[n], &cm);
                    double xv;
                    if constexpr (EO) {
                        const int sum = x[0] + x[1] + x[2] + x[3] - x[P.mu] + cm;
                        if (sum & 1) xv = ((double)probe_at(y) + __ldcg(tg + (y >> 1))) * inv_dd;
                        else xv = __ldcg(xg + (y >> 1));
                    } else {
                        xv = __ldcg(xg + y);
                    }
                    acc += (li[i] >> 30) ? -xv : xv;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) {
                if (C == 1) sh.part[0][n] = acc;
                else res_str(&sh.part[rank][n], 0, acc);
            }
        }
        res_sync(C);
        static_assert(PT_MAX_P <= 32, "one thread per output: a CTA has a warp at least");
        if (rank == 0 && tid < P.n_p) {
            double s = 0.0;
            for (int c = 0; c < C; ++c) s += sh.part[c][tid];
            double *dst = P.task_out + ((size_t)sh.task * P.n_p + tid) * 2;
            dst[0] = s;
            dst[1] = 0.0;
        }
        if (C == 1) __syncthreads();     // the next task's number overwrites sh.task
        else res_sync(C);
    }
    res_sync(C);                         // no CTA leaves while another may still address its shared memory
#undef RES_UNITS
#undef RES_UNITS_END
}

// ------------------------------------------------------------------ host
// Entries per thread of the two builds of each kind: the small one keeps more
// threads on short slices, the large one fills the registers.  One-entry
// units (V = 1) take 512 threads with 16 entries each instead of 256 with 32:
// xy planes up to 512 entries fit, and the code stays short.
struct ResCfg {
    int C, T, Te, big, n_loc, nt, nt_last;
    size_t smem;
};

template <typename S> constexpr int res_big(int V) { return std::is_same<S, double>::value ? (V == 4 ? 16 : 8) : (V == 4 ? 32 : 16); }
template <typename S> constexpr int res_small(int) { return 4; }
template <typename S> constexpr int res_minb(int V) { return 2; }
constexpr int res_tmax(int V) { return V == 4 ? 256 : 512; }

// CTAs per cluster, threads and build; false where an xy plane exceeds a CTA's
// threads or sixteen CTAs cannot hold a slab of t planes each
static bool res_config(int elem, int V, int kbig, int ksmall, int tmax, const Geom &g, int div, ResCfg *cf) {
    const int plane = g.D[0] / div * g.D[1] / V, st = g.stride[3] / div, Dt = g.D[3];
    if (plane > tmax) return false;
    const int zs = tmax / plane;                                 // xy planes of units per step of the CTA
    auto steps = [&](int nt, int z) { return (nt * g.D[2] + z - 1) / z; };
    auto fits = [&](int c) { return steps((Dt + c - 1) / c, zs) * V <= kbig; };
    int C = 1;
    while (C <= RES_MAXC && !(C <= Dt && fits(C))) C *= 2;
    if (C > RES_MAXC) return false;
    // The cluster depends on the lattice, the precision and the form, never on the
    // number of right-hand sides: its CTAs fix the order in which a solve's sums
    // are added, so that a solve has the same bits in a call of one as in a call of
    // a thousand.  Wider clusters while CTA slots are free would speed up calls of
    // a few solves (one on 9 x 7 x 11 x 15: 0.95 -> 0.52 ms, on 16^4 0.61 -> 0.47
    // ms) and give nothing from 48 on (0.94 and 0.95 ms; 0.86 and 0.85 ms).
    cf->nt = (Dt + C - 1) / C;
    cf->C = (Dt + cf->nt - 1) / cf->nt;                          // no CTA without a plane
    cf->nt_last = Dt - (cf->C - 1) * cf->nt;
    cf->n_loc = cf->nt * st;
    cf->big = steps(cf->nt, zs) * V > ksmall;
    const int z = std::min(zs, cf->nt * g.D[2]);
    cf->Te = z * plane;
    cf->T = (cf->Te + 31) / 32 * 32;
    const int kpt = cf->big ? kbig : ksmall;
    cf->smem = (size_t)3 * cf->T * kpt * elem;
    return steps(cf->nt, z) * V <= kpt;
}

static bool res_shape(const pt_op *op, const EngineRequest &rq, bool eo, int *V, ResCfg *cf) {
    const bool f64 = rq.prec == PT_PREC_FP64;
    *V = eo && op->g.D[0] % 8 == 0 ? 4 : 1;
    const int kb = f64 ? res_big<double>(*V) : res_big<float>(*V), ks = f64 ? res_small<double>(*V) : res_small<float>(*V);
    return res_config(f64 ? 8 : 4, *V, kb, ks, res_tmax(*V), op->g, eo ? 2 : 1, cf);
}

bool pt_lap_resident_fits(const pt_op *op, const EngineRequest &rq, bool eo) {
    int V;
    ResCfg cf;
    return op->kind == 0 && rq.mode != MODE_GRAD && rq.R_force <= 0 && rq.n_tasks >= 1 &&
           res_shape(op, rq, eo, &V, &cf);
}

typedef void (*ResKernel)(const ResP);

// Dynamic shared memory that a build may ask for: three arrays of its most
// entries.  The kernel's limit is set to this, and never to one call's own
// need: it belongs to the device, and contexts of other host threads launch
// the same build at other sizes in between.
static size_t res_smem_limit(int elem, int V, bool big, int kbig, int ksmall) {
    return (size_t)3 * res_tmax(V) * (big ? kbig : ksmall) * elem;
}

template <typename S>
static ResKernel res_kernel(bool eo, int V, bool big) {
    if (eo && V == 4)
        return big ? k_lap_resident<S, 1, 4, res_big<S>(4), res_tmax(4), res_minb<S>(4)> : k_lap_resident<S, 1, 4, res_small<S>(4), res_tmax(4), res_minb<S>(4)>;
    if (eo)
        return big ? k_lap_resident<S, 1, 1, res_big<S>(1), res_tmax(1), res_minb<S>(1)> : k_lap_resident<S, 1, 1, res_small<S>(1), res_tmax(1), res_minb<S>(1)>;
    return big ? k_lap_resident<S, 0, 1, res_big<S>(1), res_tmax(1), res_minb<S>(1)> : k_lap_resident<S, 0, 1, res_small<S>(1), res_tmax(1), res_minb<S>(1)>;
}

int pt_lap_resident_run(const pt_op *op, EngineRequest &rq, const LapResidentPlan &plan, pt_stats *stats) {
    pt_ctx *c = op->ctx;
    const Geom &g = op->g;
    int V;
    ResCfg cf;
    if (!res_shape(op, rq, plan.eo, &V, &cf)) {
        pt_set_error("the lattice does not fit the resident solver");
        return PT_ERR_ARG;
    }
    ResKernel kern = rq.prec == PT_PREC_FP64 ? res_kernel<double>(plan.eo, V, cf.big)
                     : rq.prec == PT_PREC_MIXED_FP32 ? res_kernel<float>(plan.eo, V, cf.big)
                                                     : res_kernel<__nv_bfloat16>(plan.eo, V, cf.big);
    const size_t smem_limit = rq.prec == PT_PREC_FP64
                                  ? res_smem_limit(8, V, cf.big, res_big<double>(V), res_small<double>(V))
                                  : res_smem_limit(4, V, cf.big, res_big<float>(V), res_small<float>(V));
    PT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_limit));
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof(lc));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cf.C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    lc.blockDim = dim3(cf.T);
    lc.dynamicSmemBytes = cf.smem;
    lc.stream = c->stream;
    lc.attrs = at;
    lc.numAttrs = cf.C > 1 ? 1 : 0;
    lc.gridDim = dim3(cf.C);
    int n_cl = 0;
    if (cf.C > 1) {
        if (cf.C > RES_PORTC) PT_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        PT_CUDA(cudaOccupancyMaxActiveClusters(&n_cl, kern, &lc));
        if (n_cl < 1) return PT_RES_NO_ROOM;                     // (no GPC with that many free SMs)
    } else {
        PT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n_cl, kern, cf.T, cf.smem));
        n_cl *= c->num_sms;
    }
    // clusters in flight: what the GPU holds, the tasks, and the caller's caps
    const int nh = plan.eo ? g.N / 2 : g.N;
    n_cl = std::max(1, std::min(n_cl, rq.n_tasks));
    if (c->max_slots > 0) n_cl = std::min(n_cl, c->max_slots);
    n_cl = (int)std::max<size_t>(1, std::min<size_t>((size_t)n_cl, c->mem_budget / ((size_t)nh * 3 * sizeof(double))));
    lc.gridDim = dim3(n_cl * cf.C);

    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
    const size_t o_x = take((size_t)n_cl * nh * sizeof(double));
    const size_t o_t = take((size_t)n_cl * nh * sizeof(double));
    const size_t o_b = take((size_t)n_cl * nh * sizeof(double));
    const size_t o_head = take(16 * sizeof(int));
    const size_t o_tasks = take((size_t)rq.n_tasks * sizeof(Task));
    const size_t o_stat = take((size_t)rq.n_tasks * sizeof(TaskStat));
    const size_t o_out = take((size_t)rq.n_tasks * std::max(rq.n_p, 1) * 2 * sizeof(double));
    void *ws;
    int rc = pt_workspace(c, off, &ws);
    if (rc) return rc;
    char *b = (char *)ws;
    ResP P;
    memset(&P, 0, sizeof(P));
    P.g = g;
    P.nh = nh;
    P.n_loc = cf.n_loc;
    P.C = cf.C;
    const int div = plan.eo ? 2 : 1;
    P.Te = cf.Te;
    P.nt = cf.nt;
    P.nt_last = cf.nt_last;
    P.row = g.D[0] / div;
    P.sy = g.stride[1] / div;
    P.sz = g.stride[2] / div;
    P.st = g.stride[3] / div;
    P.diag = 8.0 + op->m2;
    P.inv_dd = 1.0 / P.diag;
    P.diag_f = (float)P.diag;
    P.inv_df = (float)P.inv_dd;
    P.mode = rq.mode;
    P.col = rq.col;
    P.seed = rq.seed;
    P.mu = rq.mu;
    P.n_p = rq.n_p;
    for (int n = 0; n < rq.n_p && n < PT_MAX_P; ++n) {
        const int D = g.D[rq.mu];
        P.p[n] = ((rq.p_list[n] % D) + D) % D;
    }
    P.n_lev = rq.n_lev;
    P.n_pr = rq.n_pr;
    P.m_fin = rq.m_fin;
    P.lev_cols = rq.lev_cols;
    P.lev_anc = rq.lev_anc;
    P.tasks = (const Task *)(b + o_tasks);
    P.n_tasks = rq.n_tasks;
    P.B_user = rq.B_user;
    P.X_user = rq.X_user;
    P.x64 = (double *)(b + o_x);
    P.t64 = (double *)(b + o_t);
    P.b64 = (double *)(b + o_b);
    P.head = (int *)(b + o_head);
    P.flags = P.head + 8;
    P.tstat = (TaskStat *)(b + o_stat);
    P.task_out = (double *)(b + o_out);
    P.tol = rq.tol;
    P.delta = plan.delta;
    P.maxit = rq.maxit;
    P.max_inner = plan.max_inner;
    P.max_steps = 2LL * rq.maxit + 400;
    cudaStream_t st = c->stream;
    PT_CUDA(cudaMemcpyAsync((void *)P.tasks, rq.h_tasks, (size_t)rq.n_tasks * sizeof(Task), cudaMemcpyHostToDevice, st));
    PT_CUDA(cudaMemsetAsync(P.head, 0, 16 * sizeof(int), st));
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (c->prof) {
        for (auto &e : ev) PT_CUDA(cudaEventCreate(&e));
        PT_CUDA(cudaEventRecord(ev[0], st));
    }
    PT_CUDA(cudaLaunchKernelEx(&lc, kern, P));
    ++pt_kernel_launch_count;
    if (c->prof) PT_CUDA(cudaEventRecord(ev[1], st));
    int *hf = c->h_flags;
    rq.tstat.resize(rq.n_tasks);
    PT_CUDA(cudaMemcpyAsync(hf, P.flags, 8 * sizeof(int), cudaMemcpyDeviceToHost, st));
    PT_CUDA(cudaMemcpyAsync(rq.tstat.data(), P.tstat, (size_t)rq.n_tasks * sizeof(TaskStat), cudaMemcpyDeviceToHost, st));
    if (rq.mode == MODE_TRACE) {
        rq.task_out.resize((size_t)rq.n_tasks * rq.n_p * 2);
        PT_CUDA(cudaMemcpyAsync(rq.task_out.data(), P.task_out, rq.task_out.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    }
    PT_CUDA(cudaStreamSynchronize(st));
    if (c->prof) {       // one kernel does all of an engine iteration's work: the whole-iteration class
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, ev[0], ev[1]) == cudaSuccess) {
            c->prof_ms[3] += ms;
            c->prof_launches[3] += 1;
        }
        for (auto &e : ev) cudaEventDestroy(e);
    }
    if (hf[FLAG_TIMEOUT]) {
        pt_set_error("the solver did not finish within %lld steps per right-hand side", P.max_steps);
        return PT_ERR_TIMEOUT;
    }
    rq.x64_out = nullptr;
    rq.R_used = n_cl;
    if (stats) {
        memset(stats, 0, sizeof(*stats));
        stats->n_rhs = rq.n_tasks;
        stats->n_slots = n_cl;
        stats->kernel_launches = 1;
        for (auto &t : rq.tstat) {
            stats->inner_iters += t.iters;
            stats->outer_iters += t.outer;
            stats->max_relres = std::max(stats->max_relres, t.relres);
        }
        stats->engine_iters = stats->inner_iters;
        stats->site_rhs_applies = (stats->inner_iters + stats->outer_iters - stats->n_rhs) * (int64_t)g.N;
        stats->n_noconv = hf[FLAG_NOCONV];
    }
    if (hf[FLAG_NUMERIC] & 1) {
        pt_set_error("non-finite residual (NaN/Inf) in the solve");
        return PT_ERR_NUMERIC;
    }
    if (hf[FLAG_NOCONV]) {
        pt_set_error("%d right-hand side(s) did not reach tol %.3g within maxit %d", hf[FLAG_NOCONV], rq.tol, rq.maxit);
        return PT_ERR_NOCONV;
    }
    return PT_OK;
}
