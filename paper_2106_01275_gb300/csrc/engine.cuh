// Definitions shared by the batched solver engine (engine.cu) and the
// cluster-resident Laplacian solver (lap_resident.cu).
#pragma once

#include <vector>

#include "pt_common.cuh"

enum { MODE_TRACE = 0, MODE_SOLVE = 1, MODE_GRAD = 2 };
enum { TASK_ADJ = 1 };      // source is P^T v (with g5 for Wilson)

struct Task {
    int set, colour, comp, flags;
    int cidx, pad0, pad1, pad2;   // cidx: which colouring (multi-colouring runs)
};

struct TaskStat {
    int iters, outer;
    double relres;
};

#define FLAG_DONE 0
#define FLAG_NUMERIC 1
#define FLAG_NOCONV 2
#define FLAG_TIMEOUT 3

struct EngineRequest {
    int mode;
    int n_tasks;
    const Task *h_tasks;
    const int32_t *col;
    uint64_t seed;
    int noise, mu, n_p, dilute, pshift;
    const int *p_list;
    const double *B_user;
    double *X_user;
    double tol;
    int maxit;
    int prec;
    int R_force;               // >0: exact slot count (grad mode)
    int n_lev = 0, n_pr = 0, m_fin = 0;   // nested trace mode (see EP)
    const int32_t *lev_cols = nullptr;
    const int *lev_anc = nullptr;
    // outputs
    std::vector<double> task_out;   // trace: [n_tasks][n_p] complex
    std::vector<TaskStat> tstat;
    double *x64_out;           // grad mode: device pointer to the solutions (valid until next call)
    int R_used;
};

// site index and coordinate along mu of x + p e_mu for 0 <= p < D_mu (the
// engine reduces its displacements once on the host): an add and a
// conditional subtract instead of a modulo
__device__ __forceinline__ int shift_fwd(const Geom &g, int idx, const int x[4], int mu, int p, int *c_out) {
    int c = x[mu] + p;
    if (c >= g.D[mu]) c -= g.D[mu];
    *c_out = c;
    return idx + (c - x[mu]) * g.stride[mu];
}

// CG keeps its search direction across an FP64 residual replacement (the
// direction's weight is |r|^2 of the new residual over that of the last
// iteration) as long as the new residual is the one the recursion had reached
// (within half as much again); a fresh start would build up the Krylov space
// anew at every cycle.  At the same residual a solution reached that way has
// more error left in the smooth modes than a restarted one (8^3 x 16, m^2 =
// 0.16, displacement 5: 1.8e-9 of the estimate against 2.0e-10), so its last
// cycle aims at an eighth of the tolerance: 1.9e-10 there, below the restarted
// solves' error on every lattice tried, for one more iteration (16^4: 50.7
// iterations a solve restarted, 46.7 kept, 48.9 kept and taken further).
#define PT_CG_KEEP 2.25
#define PT_CG_LAST2 0.015625

// The inner tolerance and iteration bounds of a run, as run_engine_t sets them.
struct LapResidentPlan {
    bool eo;                   // even Schur complement (every side even) or the full system
    double delta;
    int max_inner;
};

// Whether a Laplacian run fits the cluster-resident solver (lap_resident.cu).
bool pt_lap_resident_fits(const pt_op *op, const EngineRequest &rq, bool eo);
// Runs it: fills rq.task_out, rq.tstat and *stats as the engine does; PT_RES_NO_ROOM
// (nothing done) where the device cannot schedule a cluster of the size needed.
#define PT_RES_NO_ROOM 1
int pt_lap_resident_run(const pt_op *op, EngineRequest &rq, const LapResidentPlan &plan, pt_stats *stats);
