// kete_impl.h -- internal types shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/kete.h"

namespace kete {

// physical constants (App. A.1 units: AU, TDB days)
constexpr double kKmPerAu = 149597870.7;
constexpr double kC = 299792.458 * 86400.0 / kKmPerAu;   // speed of light, AU/day
constexpr double kInvC2 = 1.0 / (kC * kC);
constexpr double kInvC = 1.0 / kC;

// device view of the loaded Chebyshev table
struct EphemDev {
    const double *coef;      // [body][seg][3][n_coef]
    const float *coef32;     // the same table in FP32 (mixed-precision planets)
    double t_start, t_end, seg_len, inv_seg;
    int n_seg, n_coef, n_bodies, pad;
    double gm[KETE_MAX_BODIES];
};

// device view of a force model (derived quantities precomputed on the host)
struct ForceDev {
    uint32_t active_mask;    // body_mask with massless bodies removed
    uint32_t gr_mask, j2_mask;
    int32_t precision;
    double j2k[KETE_MAX_BODIES];        // 1.5 * J2 * mu * R^2
    double pole[KETE_MAX_BODIES][3];    // unit pole, ecliptic J2000
    // per-mass factors of the GR and J2 terms, formed once here (each saves
    // an FP64 multiply per mass and force evaluation): 4 mu, mu / c^2,
    // 4 mu / c^2 and -2 x the pole
    double gm4[KETE_MAX_BODIES], grk[KETE_MAX_BODIES], gr4k[KETE_MAX_BODIES];
    double pole_m2[KETE_MAX_BODIES][3];
    double eps, safety, dt_init;
    double eps_pc;           // the caller's threshold as the analytic start needs it (make_force)
    int32_t max_iter;
    float log2_eps;
    int64_t max_steps;
    // FP32 copies for the mixed-precision planetary terms (rounded once here)
    float gm32[KETE_MAX_BODIES];
    float j2k32[KETE_MAX_BODIES];
    float pole32[KETE_MAX_BODIES][3];
    float gm4_32[KETE_MAX_BODIES], grk32[KETE_MAX_BODIES], gr4k32[KETE_MAX_BODIES];
    float pole_m2_32[KETE_MAX_BODIES][3];
    const kete_nongrav *nongrav;        // per-body non-gravitational terms or null
};

// device counters accumulated by the kernels
struct DevCounters {
    unsigned long long steps, rejected, force_evals, iterations;
    unsigned long long candidates, hits;
    unsigned long long node_evals;   // force evaluations served by batch node rows
    unsigned long long deferred;     // bodies set aside for the split second phase
    int error_flags;         // bit 0: unsorted epochs, 1: exposure mismatch, 2: bad observer,
                             // 3: bad n_edges, 4: non-finite frame, 5: batch epoch outside table
    int pad;
};

// Step grid of a propagation: epochs g[0..J] that every body's steps meet, and
// the planet states at the 8 Gauss-Radau node epochs of the steps g[j] ->
// g[j + len[q]] (rows of step (j, q) at (j n_len + q) 8 nb 6), shared by every
// body that takes that step.  ok[j n_len + q] is 0 where a node lies outside
// the table or the grid.
constexpr int kGridLens = 25;
struct GridDev {
    const double *g;
    const double *row64;   // [step][8][nb][6] FP64 barycentric pos, vel
    const float *row32;    // [step][8][nb][6] FP32 heliocentric pos, vel
    const uint8_t *ok;     // [step]
    double inv_unit;       // 1 / days per grid unit
    int J, n_len, nb, dir; // dir: +1 forward in time, -1 backward
    int chain;             // the call has more than one stop
    int len[kGridLens];    // step lengths in grid units, ascending from 1
};
// stop_row of a mark: no stop of the caller's but where a launch ends.  Bodies
// on their way wait there for the next launch; one that starts past it (its
// epoch is its own) stays where it is.
constexpr int32_t kMarkRow = -2;

// per-body working state of a propagation chain: [8][n] = x,y,z,vx,vy,vz,t,dt;
// kstop[n] (may be null): the stop a set-aside body resumes at
struct ChainState {
    double *w;
    int32_t *status;
    int64_t n;
    int32_t *kstop = nullptr;
    int64_t *tries = nullptr;   // step attempts made toward the next stop (max_steps
                                // counts them over launches; null: not kept)
};

// where a propagation launch takes its bodies from (see k_propagate)
struct PropQueue {
    const int32_t *list = nullptr;               // bodies to take; null: 0..n-1
    const unsigned long long *list_n = nullptr;  // how many (device)
    int resume = 0;                              // bodies resume at cs.kstop (else stop 0)
    int32_t *defer = nullptr;                    // set-aside bodies are appended here
    unsigned long long *defer_n = nullptr;
    int budget = 0;                              // step attempts per stop reached ...
    int budget0 = 0;                             // ... and besides
};

// Masses by lane of the one-warp-per-body kernel (kete_warp.cu): slot s of lane r (of four)
// holds body list[4 s + r]; the masses with GR or J2 terms fill slot 0, whose
// code evaluates both without branches.
constexpr int kWarpSlots = 3;
struct WarpModel {
    int list[4 * kWarpSlots];   // -1: none
    int gr, j2;                 // any GR / J2 mass
};

// scratch of the two-phase launch (long bodies set aside)
struct PropDefer {
    int32_t *list;                 // [n]
    unsigned long long *count;     // set-aside bodies
    int budget0;                   // PropQueue::budget0
    WarpModel model;               // masses of the second phase
};

// launch helpers implemented in the .cu files ---------------------------------
void upload_radau_tables(cudaStream_t st);            // kete_prop.cu
cudaError_t launch_ephem_eval(const EphemDev &E, const double *t, int64_t n, int body,
                              double *pos, double *vel, cudaStream_t st);
cudaError_t launch_chain_init(ChainState cs, const double *states, const double *epochs,
                              const ForceDev &F, cudaStream_t st);
// fill the rows and flags of a grid whose points are at grid.g
cudaError_t launch_grid_rows(const EphemDev &E, const GridDev &grid, double *row64, float *row32,
                             uint8_t *ok, cudaStream_t st);
// how the propagation kernel is launched (chosen by the autotuner)
enum PropKind { PROP_STATIC = 0, PROP_WORK_STEALING = 1 };
struct PropVariant {
    int kind;         // PropKind
    int block;        // threads per block (<= 128)
    int split = 0;    // > 1: the explicit budget below (the values 4, 8, 16 act alike)
    int budget = 0;   // step attempts per stop after which a body is set aside
    int order = 0;    // take bodies most expensive first (kete_order.cu)
    double grid_scale = 1.0;   // persistent grids scaled by this (<= 1: a sample of the
                               // bodies run with as many bodies per lane as the whole)
    int64_t population = 0;    // bodies of the whole, which the form (lanes or warps) and the
                               // set-aside budget follow (0: those of the call)
};
// stop_row (device, may be null): output row of each stop, -1: not written
// (null: stop k is row k).  grid (may be null): the step grid to follow.
cudaError_t launch_propagate(const EphemDev &E, const ForceDev &F, ChainState cs,
                             const double *stops_dev, const int32_t *stop_row, int n_stops,
                             double *out, int64_t out_stride, bool keep_on_fail, DevCounters *ctr,
                             cudaStream_t st, const GridDev *grid = nullptr,
                             PropVariant var = PropVariant{PROP_STATIC, 128},
                             unsigned long long *next_body = nullptr,
                             PropDefer *defer = nullptr, const int32_t *order = nullptr,
                             const unsigned long long *order_n = nullptr, bool out_aos = false);
int propagate_ws_blocks(int block, int mode);
// kete_warp.cu: one warp per body.
// false: the model does not fit (the Sun inactive, more than 12 masses, more
// than 4 with GR or J2 terms)
bool warp_model(const EphemDev &E, const ForceDev &F, WarpModel &W);
cudaError_t upload_warp_tables(cudaStream_t st);
// q: bodies 0..n-1, or q.list (resuming at their saved stops if q.resume)
cudaError_t launch_propagate_warp(const EphemDev &E, const ForceDev &F, const WarpModel &W,
                                  ChainState cs, const double *stops, const int32_t *row,
                                  int n_stops, double *out, int64_t stride, bool keep_on_fail,
                                  DevCounters *ctr, cudaStream_t st, PropQueue q, bool out_aos);
cudaError_t launch_gather_bodies(const double *st, const double *ep, int64_t n, int64_t m,
                                 double *dst, double *dep, cudaStream_t s);
cudaError_t launch_chain_finish(ChainState cs, double *states, double *epochs,
                                int32_t *status, cudaStream_t st);
// kete_noalloc.cu: propagation with the chain scratch in a fixed device array
int noalloc_propagate(int device, cudaStream_t st, const EphemDev &E, const ForceDev &F,
                      double *states, double *epochs, int64_t n, double t_target,
                      int32_t *status, const char **why);

}  // namespace kete
