// kete_adjoint.h -- device buffers and launchers of the adjoint (kete_adjoint.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kete_impl.h"

namespace kete {

// one record per accepted step: t_start, t_end, then the symmetric Newtonian
// da/dx (xx, xy, xz, yy, yz, zz) at the step's 8 Gauss-Radau nodes; a final
// record (t_end = t_start) holds da/dx at the last state in node 0's place
constexpr int kAdjRec = 2 + 8 * 6;
// the full-model extension of a record: 8 nodes x (da/dx beyond Newton, da/dv)
constexpr int kAdjRecX = 8 * 18;
// checkpoint stops per body before the chain gives up (KETE_BODY_STEP_CAP)
constexpr int kAdjMaxCkpt = 1 << 16;

// the problem (caller's arrays; states and grad are [6][n], obs [n][m])
struct AdjProblem {
    const double *states, *epochs;
    int64_t n;
    const kete_obs *obs;
    int32_t m;
    double span, ckpt, inv_ckpt;   // inv_ckpt: 1 / ckpt (0: no grid)
    double cos_eps, sin_eps;
    double *loss, *grad, *pred;
    double *jac;       // [n][m][2][6] d(RA, Dec)/d(x0, v0) per observation, or null
    int32_t *status;
    DevCounters *ctr;
};

// library scratch for one chunk of nc bodies
struct AdjBuffers {
    double *rec;       // [nc][cap][kAdjRec]
    int32_t cap;       // records per body
    int32_t *n_rec;    // [nc] records written (0: no gradient)
    int32_t *nbat;     // [nc] batches
    int32_t *bidx;     // [nc][m] steps taken when batch k's midpoint was reached
    double *yref;      // [nc][m][6] state at batch k's midpoint
    double *gjump;     // [nc][m][6] dL/dy(t_ref) of batch k
    double *phi;       // [nc][m][36] state-transition matrix at batch k's midpoint
                       // (row-major, d y_r(t_ref) / d y0_c), or null
    double *recx;      // [nc][cap][8][18] per record and node: da/dx beyond the Newtonian
                       // part (9, row-major) and da/dv (9) -- the full force model's
                       // Jacobian (calls with non-gravitational terms); null: the
                       // Newtonian da/dx of rec alone
    int32_t *rich;     // [nc] (with recx) 1: the body has non-gravitational terms and
                       // its records carry recx; 0: a body without terms, Newtonian
                       // records only
    int32_t *status;   // [nc]
    double *bfrac;     // [nc][m] where in step bidx[k] batch k's midpoint
                       // lies, (t_ref - t_start) / h; 0: at the step's start
    double *mid;       // [nc][m] batch midpoints (launch_fit_stops), or null
    double *planets;   // [7 n_bodies 6][lanes of the forward grid]: see attempt_sweep
};

// lanes of the forward pass's grid for chunks of nc bodies
int64_t adjoint_forward_lanes(int64_t nc, bool full);

// checkpoints of the grid (one in 1 / inv_ckpt days, none for 0) before t
__device__ __forceinline__ double ckpts_before(double inv_ckpt, double epoch0, double t)
{
    return inv_ckpt > 0.0 && t > epoch0 ? ceil((t - epoch0) * inv_ckpt) - 1.0 : 0.0;
}

// The record limit counts steps that end at every stop, midpoint and checkpoint
// (k_adj_forward's): a step that passes stops is one for each of them, the others
// one.  (Stops and steps added up would refuse arcs whose every step is a leg: 4
// years of 8-day legs, 183 steps there, came to 281.)
__device__ __forceinline__ int steps_with_stops(double ckpts, int midpoints)
{
    const int stops = (int)fmin(ckpts, 1e6) + midpoints;
    return stops > 1 ? stops : 1;
}

// observations in use: those before the first non-finite epoch
__device__ __forceinline__ int obs_count(const kete_obs *o, int m)
{
    int mi = 0;
    while (mi < m && isfinite(o[mi].epoch)) mi++;
    return mi;
}

// batches of one body's observations (the <= span rule of Sec. 2): the batch
// starting at j0 ends before the returned index; tref = midpoint.
__device__ __forceinline__ int next_batch(const kete_obs *o, int mi, int j0, double span,
                                          double &tref)
{
    const double e0 = o[j0].epoch;
    int j = j0;
    while (j + 1 < mi) {
        const double e = o[j + 1].epoch;
        if (!(e == e0 || e - e0 < span)) break;
        j++;
    }
    tref = 0.5 * (e0 + o[j].epoch);
    return j + 1;
}

cudaError_t upload_adjoint_tables(cudaStream_t st);
// kete_warp.cu: the forward pass with one warp per body, without
// non-gravitational terms: steps of the size the step control proposes, the
// batch midpoints inside them from the step polynomial (B.bfrac)
cudaError_t launch_adjoint_forward_warp(const EphemDev &E, const ForceDev &F, const WarpModel &W,
                                        const AdjBuffers &B, const AdjProblem &P, int64_t i0,
                                        int64_t nc, cudaStream_t st, PropQueue q = PropQueue{});
// The lane form of the same for many bodies whose epochs lie close enough for
// one step grid: each body's midpoints, batch count and first status (B.mid,
// B.nbat, B.status; B.n_rec: 1 past the record limit) and the span of all
// chains, [first epoch, last midpoint] as order-preserving keys in range[0..1];
// the lanes (kete_prop.cu), which leave step polynomials in the records and set
// long bodies aside; da/dx in place of the polynomials.
cudaError_t launch_fit_stops(const AdjBuffers &B, const AdjProblem &P, int64_t i0, int64_t nc,
                             unsigned long long *range, cudaStream_t st);
double fit_range_epoch(unsigned long long key);
cudaError_t launch_fit_lanes(const EphemDev &E, const ForceDev &F, const AdjBuffers &B,
                             const AdjProblem &P, int64_t i0, int64_t nc, const GridDev &Q,
                             unsigned long long *next, const int32_t *order,
                             const unsigned long long *order_n, const PropDefer &defer,
                             cudaStream_t st);
cudaError_t launch_fit_jacobian(const EphemDev &E, const ForceDev &F, const AdjBuffers &B,
                                int64_t nc, cudaStream_t st);
// persistent grid with work stealing from the counter *next;
// order != null: lanes take the chunk's bodies in that order
cudaError_t launch_adjoint_forward(const EphemDev &E, const ForceDev &F, const AdjBuffers &B,
                                   const AdjProblem &P, int64_t i0, int64_t nc,
                                   unsigned long long *next, cudaStream_t st,
                                   const int32_t *order = nullptr);
// t_end[i] = the last observation epoch of chunk body i (its epoch if none)
cudaError_t launch_adjoint_last_epoch(const AdjProblem &P, int64_t i0, int64_t nc, double *t_end,
                                      cudaStream_t st);
cudaError_t launch_adjoint_observe(const EphemDev &E, const AdjBuffers &B, const AdjProblem &P,
                                   int64_t i0, int64_t nc, cudaStream_t st);
cudaError_t launch_adjoint_backward(const AdjBuffers &B, const AdjProblem &P, int64_t i0,
                                    int64_t nc, cudaStream_t st);
// the state-transition matrix at every batch midpoint (B.phi), integrated
// forward over the recorded steps
cudaError_t launch_adjoint_stm(const AdjBuffers &B, const AdjProblem &P, int64_t i0, int64_t nc,
                               cudaStream_t st);

}  // namespace kete
