// kete_prop.cu -- n-body propagation of massless bodies (Sec. 3.2, App. A, App. A.6).
//
// Each lane integrates one body at a time along its chain of stops (the
// body's epoch, then every stop in order).  With a step grid a body takes the
// steps its own step control proposes, rounded down to whole grid units, and
// the states at the stops inside a step come from the step's collocation
// polynomial; without one its steps end at every stop.  Each step is a 15th-order Gauss-Radau step in the
// IAS15 form (Newton-basis coefficients g, power-basis coefficients b, 8
// spacings).  The corrector starts from two-body motion, then from the previous
// step's polynomial (see CorrectorStart), and iterates until max|db6|/max|a| <
// eps_pc, the error stops falling (after 3 iterations) or max_iter is reached.  Step control follows IAS15:
// dt_new = dt (eps / (max|b6|/max|a|))^(1/7), reject below safety*dt, grow at
// most 1/safety.  Every loop is bounded: max_iter corrector iterations,
// max_steps step attempts per leg, after which the body gets a status code.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "kete_adjoint.h"
#include "kete_step.cuh"

namespace kete {

void upload_radau_tables(cudaStream_t st) { upload_step_tables(st); }

#ifndef KETE_PROP_MIN_BLOCKS
#define KETE_PROP_MIN_BLOCKS 1   // resident blocks per SM asked of the register allocator
#endif

// the state (x, v) of body i at stop k (component c at o[c * s])
__device__ __forceinline__ void write_stop(double *__restrict__ out,
                                           const int32_t *__restrict__ stop_row, int k, int64_t i,
                                           int64_t out_stride, int out_aos, const double x[3],
                                           const double v[3])
{
    const int row = stop_row ? stop_row[k] : k;
    if (row < 0) return;
    double *o = out_aos ? out + ((int64_t)row * out_stride + i) * 6
                        : out + (int64_t)row * 6 * out_stride + i;
    const int64_t s = out_aos ? 1 : out_stride;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        o[c * s] = x[c];
        o[(3 + c) * s] = v[c];
    }
}

// The propagation kernel.  Each lane owns one body at a time and advances it
// along its chain of stops, writing the state at every stop k (row =
// stop_row[k], or k without stop_row; -1: not written) to out[row][c][i] (stride
// out_stride between rows; out_aos: to out[row][i][c] with out_stride bodies per
// stop, one contiguous 48-byte record per body and stop) and the chain state
// back when it is done.
// Q (use_grid): the step grid.  A body whose next stop lies in the grid's
// direction follows it (step_begin_grid); FP64 issue bounds this kernel, so the
// count of force evaluations is what to save: stopping at every third day of a
// survey chain took 121 steps of 22 evaluations a year, the proposed steps of
// a main-belt body (~16 days) are 24 of 15-16 evaluations, and the rows keep those evaluations
// at the shared-planet cost (about 250 FP64 instructions against 650).  A body
// whose step past a stop fails takes plain steps, stop by stop, from there on,
// so that the stops before the failure still get their states.  A mark
// (kMarkRow) ends the launch for a body on its way and none of its own.
// A pass of the loop is one corrector sweep (7 force evaluations) for every
// lane inside a step attempt.  An FP64 warp instruction costs the same
// whatever its active lanes, so the work between attempts (step control, the
// stops inside the step, the next body, the acceleration at the next step's
// start: about a third of a sweep) waits until kSyncLanes lanes have reached
// it or none is left in an attempt (400,000 main-belt bodies over 60 days: 40.8
// ms for 8 lanes, 39.1 for 16, 40.2 for 24, 40.3 for 32).
//   refill = 0 (static): lane j of the grid takes body j and then idles;
//   refill = 1 (work stealing, persistent grid): a lane whose body is done
//   takes the next one from an atomic counter (warp-aggregated), so a body
//   needing hundreds of steps no longer idles the rest of its warp.
// Every body sees the same arithmetic in the same order whatever the
// schedule and whatever its warp-mates do: results are identical.
// Queue q: the bodies come from q.list (q.list_n of them, device) instead of
// 0..n-1, resuming at their saved stops cs.kstop[i] if q.resume; with q.defer
// set, a body that has made more than q.budget step attempts per stop reached,
// plus q.budget0, is set aside at its next step boundary (state and stop saved,
// index appended to q.defer) for a second launch with one warp per body, and
// with q.budget0 so is one whose proposed step falls below a grid unit: its
// per-thread planet sums would be paid by the whole warp.
// NG: bodies may carry non-gravitational terms (F.nongrav); the instantiation
// without them has those branches compiled out.
constexpr int kSyncLanes = 16;
// REC (k_propagate): the bodies are those of an orbit fit.  The stops are each body's batch
// midpoints (B.mid, B.nbat), kept with the step each lies in; every accepted
// step leaves its epochs and polynomial in its record.  A body set aside
// starts again in the warp form.  100,000 fits over 90 days: forward pass 42.1
// ms one warp per body, 25.3 with lanes and k_fit_jacobian (the planets from the
// grid's rows, a full lane grid's issue per step).
struct FitRecord {
    AdjBuffers B;
    AdjProblem P;
    int64_t i0;
};

__device__ __forceinline__ void fit_stop(const FitRecord &R, int k, int64_t i, int count, double frac,
                                         const double x[3], const double v[3])
{
    const size_t at = (size_t)i * R.P.m + k;
    double *y = R.B.yref + at * 6;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        y[c] = x[c];
        y[3 + c] = v[c];
    }
    R.B.bidx[at] = count;
    R.B.bfrac[at] = frac;
}

// the body's last record (its final state) and status; used: its steps counted
// toward the record limit (steps_with_stops)
__device__ __forceinline__ void fit_done(const EphemDev &E, const FitRecord &R, int64_t i, int status, bool capped,
                                         int count, int used, double t, const double x[3],
                                         double *rec)
{
    if (R.P.ckpt > 0.0 && used > R.B.cap - 1) capped = true;
    Seg g;
    if (status == KETE_BODY_OK && capped) status = KETE_BODY_ADJ_CAP;
    else if (status == KETE_BODY_OK && !ephem_seg(E, t, 0.0, g)) status = KETE_BODY_OUT_OF_SPAN;
    if (status == KETE_BODY_OK) {
        double *r = rec + (size_t)count * kAdjRec;
        r[0] = r[1] = t;
#pragma unroll
        for (int c = 0; c < 3; c++) r[2 + c] = x[c];
        count++;
    }
    R.B.n_rec[i] = status == KETE_BODY_OK ? count : 0;
    R.B.status[i] = status;
}

template <int MODE, bool NG, bool V32 = false, bool REC = false>
__global__ void __launch_bounds__(128, KETE_PROP_MIN_BLOCKS)
k_propagate(EphemDev E, ForceDev F, ChainState cs, const double *__restrict__ stops_in,
            const int32_t *__restrict__ stop_row, int n_stops_in, double *__restrict__ out,
            int64_t out_stride, int out_aos, int keep_on_fail, DevCounters *ctr, GridDev Q,
            int use_grid, unsigned long long *__restrict__ next_body, int refill, PropQueue q,
            FitRecord R)
{
    const int64_t n = cs.n;
    const unsigned long long n_items = q.list ? *q.list_n : (unsigned long long)n;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    Cnt cnt = {0, 0, 0, 0, 0};
    int64_t i = 0;            // current body
    const double *stops = stops_in;   // its stops
    int n_stops = n_stops_in;
    double *rec = nullptr, epoch0 = 0.0;   // REC: its records
    int count = 0, used = 0;
    bool capped = false;
    int k = 0;                // next stop of the body
    double x[3], v[3], t = 0.0, dt = 0.0;
    int status = KETE_BODY_OK;
    long long attempts = 0, body_attempts = 0;
    StepState S;
    S.have_a0 = S.chained = false;
    S.start = START_A0;
    S.ng = nullptr;
    S.ng_chi = 0.0;
    bool plain = true, careful = false;   // steps end at the stops; for good after a failure
    int j = 0, jn = 0;                    // grid point stood on or ahead, and the attempt's
    Attempt A;
    enum { TAKE, BOUNDARY, SWEEP, SWEPT, DRAINED };
    int phase = TAKE;
    bool first = true;
    for (;;) {
        const unsigned sweeping = __ballot_sync(FULL, phase == SWEEP);
        const unsigned waiting = __ballot_sync(FULL, phase != SWEEP && phase != DRAINED);
        if (!(sweeping | waiting)) break;
        if (waiting && (!sweeping || __popc(waiting) >= kSyncLanes)) {
            if (phase == SWEPT) {
                phase = BOUNDARY;
                if (status == KETE_BODY_OK) {
                    const double proposed = dt;
                    double x1[3], v1[3];
                    bool accepted;
                    status = step_control<MODE>(F, A, x, v, dt, S, cnt, x1, v1, accepted);
                    if (accepted) {
                        const int k_from = k;
                        if (!plain) {
                            // stops inside the step, from its polynomial
                            while (k < n_stops && (Q.dir > 0 ? stops[k] < A.t_new : stops[k] > A.t_new)) {
                                double xs[3], vs[3];
                                attempt_dense(A, t, x, v, S.a0, stops[k], xs, vs);
                                if (REC) fit_stop(R, k, i, count, (stops[k] - t) / A.h, xs, vs);
                                else write_stop(out, stop_row, k, i, out_stride, out_aos, xs, vs);
                                k++;
                                attempts = 0;
                            }
                            j = jn;
                            // a step cut short by the grid says little about the next
                            // (its b6 is rounding, 1e-13 |a|, a growth of 3.7 at
                            // eps 1e-9) unless its own error holds the next one back
                            if (fabs(A.h) < 0.5 * fabs(proposed) && fabs(dt) < fabs(proposed) &&
                                fabs(dt) >= 2.0 * fabs(A.h))
                                dt = proposed;
                        }
                        if (REC) {   // the step's polynomial (k_fit_jacobian turns it into da/dx)
                            const double ck = ckpts_before(R.P.inv_ckpt, epoch0, A.t_new) -
                                              ckpts_before(R.P.inv_ckpt, epoch0, t);
                            used += steps_with_stops(ck, k - k_from + (k < n_stops && stops[k] == A.t_new));
                            if (ck > 0.0) attempts = 0;   // max_steps counts the attempts of a leg
                            if (count < R.B.cap - 1) {
                                double *r = rec + (size_t)count * kAdjRec;
                                r[0] = t;
                                r[1] = A.t_new;
#pragma unroll
                                for (int c = 0; c < 3; c++) {
                                    r[2 + c] = x[c];
                                    r[5 + c] = v[c];
                                    r[8 + c] = S.a0[c];
#pragma unroll
                                    for (int m = 0; m < 7; m++) r[11 + 3 * m + c] = A.b[m][c];
                                }
                                count++;
                            } else {
                                capped = true;
                            }
                        }
#pragma unroll
                        for (int c = 0; c < 3; c++) {
                            x[c] = x1[c];
                            v[c] = v1[c];
                        }
                        t = A.t_new;
                        S.have_a0 = false;
                        S.chained = fabs(dt) <= kNextMost * fabs(A.h);
                    } else {
                        S.start = MODE == KETE_MIXED ? START_A0 : START_RETRY;
                    }
                }
                if (status != KETE_BODY_OK && !plain && k < n_stops && stops[k] != A.t_new) {
                    careful = plain = true;   // a step past a stop failed: plain steps from here
                    status = KETE_BODY_OK;
                    S.start = START_A0;       // (its polynomial is of no use)
                    S.chained = false;
                }
            }
            // lanes without a body take the next ones; a body may already be
            // done when it is taken (no stops ahead, a bad state)
            for (;;) {
                const bool need = phase == TAKE;
                const unsigned m = __ballot_sync(FULL, need);
                if (m) {
                    unsigned long long base = 0;
                    const int leader = __ffs(m) - 1;
                    if (refill) {
                        if (lane == leader) base = atomicAdd(next_body, (unsigned long long)__popc(m));
                        base = __shfl_sync(FULL, base, leader);
                    }
                    if (need) {
                        // needing lanes before this one
                        unsigned long long mine = base + (unsigned long long)__popc(m & ((1u << lane) - 1u));
                        if (!refill)   // static: one body per lane, taken on the first pass
                            mine = first ? (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x : n_items;
                        if (mine < n_items) {
                            i = q.list ? (int64_t)q.list[mine] : (int64_t)mine;
                            attempts = 0;
                            if (REC) {
                                const AdjProblem &P = R.P;
                                const int64_t gi = R.i0 + i;
#pragma unroll
                                for (int c = 0; c < 3; c++) {
                                    x[c] = P.states[c * P.n + gi];
                                    v[c] = P.states[(3 + c) * P.n + gi];
                                }
                                t = epoch0 = P.epochs[gi];
                                dt = 0.0;
                                status = R.B.status[i];
                                k = 0;
                                stops = R.B.mid + (size_t)i * P.m;
                                n_stops = R.B.nbat[i];
                                capped = R.B.n_rec[i] != 0;
                                rec = R.B.rec + (size_t)i * R.B.cap * kAdjRec;
                                count = used = 0;
                            } else {
#pragma unroll
                                for (int c = 0; c < 3; c++) {
                                    x[c] = cs.w[c * n + i];
                                    v[c] = cs.w[(3 + c) * n + i];
                                }
                                t = cs.w[6 * n + i];
                                dt = cs.w[7 * n + i];
                                status = cs.status[i];
                                k = q.resume ? cs.kstop[i] : 0;
                                if (cs.tries) attempts = cs.tries[i];
                            }
                            body_attempts = 0;
                            S.have_a0 = false;
                            S.chained = false;
                            S.ng = (NG && F.nongrav) ? F.nongrav + i : nullptr;
                            S.ng_chi = 0.0;
                            plain = true;
                            careful = !use_grid;
                            if (!REC && use_grid)   // past a mark
                                while (k < n_stops && stop_row && stop_row[k] == kMarkRow &&
                                       (Q.dir > 0 ? t >= stops[k] : t <= stops[k]))
                                    k++;
                            if (status == KETE_BODY_OK && k < n_stops) {
                                aim_step(F, t, stops[k], dt);
                                plain = careful || (stops[k] >= t) != (Q.dir > 0);
                                if (!plain) j = grid_locate(Q, t);
                            }
                            phase = BOUNDARY;
                        } else {
                            phase = DRAINED;
                        }
                    }
                }
                first = false;
                if (phase == BOUNDARY) {
                    // stops the body stands at, or all of them if it failed
                    while (k < n_stops && (status != KETE_BODY_OK || t == stops[k])) {
                        const double nan = __longlong_as_double(0x7ff8000000000000ll);
                        const double none[3] = {nan, nan, nan};
                        if (REC) {
                            if (status == KETE_BODY_OK) fit_stop(R, k, i, count, 0.0, x, v);
                        } else if (status == KETE_BODY_OK)
                            write_stop(out, stop_row, k, i, out_stride, out_aos, x, v);
                        else if (!keep_on_fail) write_stop(out, stop_row, k, i, out_stride, out_aos, none, none);
                        if (!(use_grid && stop_row && stop_row[k] == kMarkRow)) attempts = 0;
                        k++;
                        S.have_a0 = false;
                        if (k < n_stops && status == KETE_BODY_OK) {
                            aim_step(F, t, stops[k], dt);
                            if (plain && !careful && (stops[k] >= t) == (Q.dir > 0)) {
                                plain = false;
                                j = grid_locate(Q, t);
                            }
                        }
                    }
                    bool aside = false;
                    if (q.defer && k < n_stops && !S.have_a0)
                        aside = body_attempts >= (long long)q.budget * (k + 1) + q.budget0 ||
                                (q.budget0 > 0 && body_attempts > 0 && !plain &&
                                 fabs(dt) * Q.inv_unit < 1.0 && F.dt_init * Q.inv_unit >= 1.0);
                    if (REC && (k >= n_stops || aside)) {
                        if (aside) {
                            q.defer[atomicAdd(q.defer_n, 1ull)] = (int32_t)i;
                            atomicAdd(&ctr->deferred, 1ull);
                            R.B.n_rec[i] = 0;
                        } else {
                            fit_done(E, R, i, status, capped, count, used, t, x, rec);
                        }
                        phase = TAKE;
                    } else if (k >= n_stops || aside) {
                        // write the chain state back and free the lane
#pragma unroll
                        for (int c = 0; c < 3; c++) {
                            cs.w[c * n + i] = x[c];
                            cs.w[(3 + c) * n + i] = v[c];
                        }
                        cs.w[6 * n + i] = t;
                        cs.w[7 * n + i] = dt;
                        cs.status[i] = status;
                        if (cs.tries) cs.tries[i] = attempts;
                        if (aside) {
                            cs.kstop[i] = k;
                            q.defer[atomicAdd(q.defer_n, 1ull)] = (int32_t)i;
                            atomicAdd(&ctr->deferred, 1ull);
                        }
                        phase = TAKE;
                    }
                }
                if (!__any_sync(FULL, phase == TAKE)) break;
            }
            if (phase == BOUNDARY) {
                body_attempts++;
                if (++attempts > F.max_steps) {
                    status = KETE_BODY_STEP_CAP;
                } else {
                    status = plain ? step_begin<MODE>(E, F, x, v, t, dt, stops[k], S, A, cnt)
                                   : step_begin_grid<MODE>(E, F, Q, j, jn, x, v, t, dt, S, A, cnt);
                    if (status == KETE_BODY_OK) {
                        phase = SWEEP;
                    } else if (!plain) {   // plain steps from here, as after a failed sweep
                        careful = plain = true;
                        status = KETE_BODY_OK;
                    }
                }
            }
        }
        // the lanes that have just begun a step and the others sweep together (they
        // left the branches above apart: 757,000 bodies over 60 days 108 ms
        // without this, 85 with it)
        __syncwarp(FULL);
        if (phase == SWEEP) {   // one corrector sweep
            bool done = false;
            status = attempt_sweep<MODE, false, V32>(E, F, t, x, v, S.a0, S.as0, S.close, S.enc, A,
                                                     done, cnt, nullptr, S.ng, &S.ng_chi);
            if (done || status != KETE_BODY_OK) phase = SWEPT;
        }
    }
    flush_counters(cnt, ctr);
}

// Grid rows: thread per (step, node n, body m); step = (start j, length q).
// The node epoch is (g[j], h_n h) with h the exact difference of the grid
// points, as the integrator forms it.
__global__ void k_grid_rows(EphemDev E, GridDev Q, double *__restrict__ row64,
                            float *__restrict__ row32, uint8_t *__restrict__ okf)
{
    const int nb = Q.nb;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int m = (int)(idx % nb);
    const int n = (int)((idx / nb) % 8);
    const int64_t step = idx / (8 * nb);
    if (step >= (int64_t)Q.J * Q.n_len) return;
    const int j = (int)(step / Q.n_len), q = (int)(step % Q.n_len);
    const int je = j + Q.len[q];
    if (je > Q.J) {
        if (m == 0 && n == 0) okf[step] = 0;
        return;
    }
    const double ts = Q.g[j], h = Q.g[je] - ts;
    if (m == 0 && n == 0) {
        // no node lies past the step's ends
        Seg a, b;
        okf[step] = ephem_seg(E, ts, 0.0, a) && ephem_seg(E, ts, h, b) ? 1 : 0;
    }
    Seg g;
    if (!ephem_seg(E, ts, g_rt.h[n] * h, g)) return;
    double st[6], sun[6];
    double *o64 = row64 + (step * 8 + n) * nb * 6 + 6 * m;
    float *o32 = row32 + (step * 8 + n) * nb * 6 + 6 * m;
    cheb_pos_vel(ephem_coef(E, m, g.s), E.n_coef, g.tau, 2.0 * E.inv_seg, st, st + 3);
    cheb_pos_vel(ephem_coef(E, 0, g.s), E.n_coef, g.tau, 2.0 * E.inv_seg, sun, sun + 3);
    for (int c = 0; c < 6; c++) o64[c] = st[c];
    for (int c = 0; c < 3; c++) {
        o32[c] = (float)(st[c] - sun[c]);
        o32[3 + c] = (float)st[3 + c];
    }
}

__global__ void k_chain_init(ChainState cs, const double *__restrict__ states,
                             const double *__restrict__ epochs)
{
    const int64_t n = cs.n;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    bool ok = true;
    for (int c = 0; c < 6; c++) {
        double q = states[c * n + i];
        cs.w[c * n + i] = q;
        ok = ok && isfinite(q);
    }
    double t = epochs[i];
    cs.w[6 * n + i] = t;
    cs.w[7 * n + i] = 0.0;
    cs.status[i] = (ok && isfinite(t)) ? KETE_BODY_OK : KETE_BODY_NONFINITE;
    if (cs.tries) cs.tries[i] = 0;
}

__global__ void k_chain_finish(ChainState cs, double *__restrict__ epochs,
                               int32_t *__restrict__ status)
{
    const int64_t n = cs.n;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int s = cs.status[i];
    if (epochs && s == KETE_BODY_OK) epochs[i] = cs.w[6 * n + i];
    if (status) status[i] = s;
}

__global__ void k_ephem_eval(EphemDev E, const double *__restrict__ t, int64_t n, int body,
                             double *__restrict__ pos, double *__restrict__ vel)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Seg g;
    double p[3], v[3];
    if (!ephem_seg(E, t[i], 0.0, g)) {
        for (int c = 0; c < 3; c++) {
            pos[3 * i + c] = __longlong_as_double(0x7ff8000000000000ll);
            if (vel) vel[3 * i + c] = __longlong_as_double(0x7ff8000000000000ll);
        }
        return;
    }
    cheb_pos_vel(ephem_coef(E, body, g.s), E.n_coef, g.tau, 2.0 * E.inv_seg, p, v);
    for (int c = 0; c < 3; c++) {
        pos[3 * i + c] = p[c];
        if (vel) vel[3 * i + c] = v[c];
    }
}

// evenly spread sample of m of the n bodies: dst[c][j] = src[c][floor(j n / m)]
// (autotuner)
__global__ void k_gather_bodies(const double *__restrict__ st, const double *__restrict__ ep,
                                int64_t n, int64_t m, double *__restrict__ dst,
                                double *__restrict__ dep)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int64_t i = (j * n) / m;
    for (int c = 0; c < 6; c++) dst[c * m + j] = st[c * n + i];
    dep[j] = ep[i];
}

static unsigned grid_for(int64_t n, int block) { return (unsigned)((n + block - 1) / block); }

cudaError_t launch_ephem_eval(const EphemDev &E, const double *t, int64_t n, int body,
                              double *pos, double *vel, cudaStream_t st)
{
    if (n > 0) k_ephem_eval<<<grid_for(n, 256), 256, 0, st>>>(E, t, n, body, pos, vel);
    return cudaGetLastError();
}

cudaError_t launch_chain_init(ChainState cs, const double *states, const double *epochs,
                              const ForceDev &, cudaStream_t st)
{
    if (cs.n > 0) k_chain_init<<<grid_for(cs.n, 256), 256, 0, st>>>(cs, states, epochs);
    return cudaGetLastError();
}

cudaError_t launch_grid_rows(const EphemDev &E, const GridDev &grid, double *row64, float *row32,
                             uint8_t *ok, cudaStream_t st)
{
    const int64_t tot = (int64_t)grid.J * grid.n_len * 8 * grid.nb;
    if (tot > 0) k_grid_rows<<<grid_for(tot, 128), 128, 0, st>>>(E, grid, row64, row32, ok);
    return cudaGetLastError();
}

template <int MODE>
static int ws_blocks(int block)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_propagate<MODE, false>, block, 0);
    return (sms > 0 ? sms : 152) * (per_sm > 0 ? per_sm : 1);
}

int propagate_ws_blocks(int block, int mode)
{
    return mode == KETE_MIXED ? ws_blocks<KETE_MIXED>(block) : ws_blocks<KETE_FP64>(block);
}

template <int MODE>
static void launch_k(int64_t grid, int block, cudaStream_t st, const EphemDev &E,
                     const ForceDev &F, ChainState cs, const double *stops, const int32_t *row,
                     int n_stops, double *out, int64_t stride, int aos, int kof, DevCounters *ctr,
                     GridDev Q, int ug, unsigned long long *next, int refill, PropQueue q)
{
    // mixed precision along a chain of stops: the node velocity in FP32 (V32)
    if (F.nongrav) {
        k_propagate<MODE, true><<<(unsigned)grid, block, 0, st>>>(
            E, F, cs, stops, row, n_stops, out, stride, aos, kof, ctr, Q, ug, next, refill, q, FitRecord{});
        return;
    }
    if constexpr (MODE == KETE_MIXED) {
        if (ug && Q.chain) {
            k_propagate<MODE, false, true><<<(unsigned)grid, block, 0, st>>>(
                E, F, cs, stops, row, n_stops, out, stride, aos, kof, ctr, Q, ug, next, refill, q, FitRecord{});
            return;
        }
    }
    k_propagate<MODE, false><<<(unsigned)grid, block, 0, st>>>(
        E, F, cs, stops, row, n_stops, out, stride, aos, kof, ctr, Q, ug, next, refill, q, FitRecord{});
}

cudaError_t launch_propagate(const EphemDev &E, const ForceDev &F, ChainState cs,
                             const double *stops_dev, const int32_t *stop_row, int n_stops,
                             double *out, int64_t out_stride, bool keep_on_fail, DevCounters *ctr,
                             cudaStream_t st, const GridDev *grid_in, PropVariant var,
                             unsigned long long *next_body, PropDefer *defer,
                             const int32_t *order, const unsigned long long *order_n,
                             bool out_aos)
{
    const int aos = out_aos ? 1 : 0;
    if (cs.n <= 0 || n_stops <= 0) return cudaGetLastError();
    GridDev Q{};
    if (grid_in) Q = *grid_in;
    const int kof = keep_on_fail ? 1 : 0, ug = grid_in ? 1 : 0;
    const int block = (var.block > 0 && var.block <= 128) ? var.block : 128;
    const bool mixed = F.precision == KETE_MIXED;
    int refill = 0;
    int64_t grid = (cs.n + block - 1) / block;
    if (var.kind == PROP_WORK_STEALING && next_body) {
        cudaError_t e = cudaMemsetAsync(next_body, 0, sizeof(unsigned long long), st);
        if (e != cudaSuccess) return e;
        refill = 1;
        int64_t persistent = propagate_ws_blocks(block, F.precision);
        if (var.grid_scale < 1.0)
            persistent = std::max<int64_t>(1, (int64_t)(persistent * var.grid_scale + 0.5));
        if (grid > persistent) grid = persistent;
    }
    // phase 1: one lane per body; bodies past their budget of attempts are set aside
    PropQueue q{};
    if (order && order_n) {
        q.list = order;
        q.list_n = order_n;
    }
    const bool split = defer && cs.kstop && (var.budget > 0 || defer->budget0 > 0);
    if (split) {
        cudaError_t e = cudaMemsetAsync(defer->count, 0, sizeof(unsigned long long), st);
        if (e != cudaSuccess) return e;
        q.defer = defer->list;
        q.defer_n = defer->count;
        q.budget = var.budget;
        q.budget0 = defer->budget0;
    }
    if (mixed)
        launch_k<KETE_MIXED>(grid, block, st, E, F, cs, stops_dev, stop_row, n_stops, out, out_stride, aos, kof, ctr, Q, ug, next_body, refill, q);
    else
        launch_k<KETE_FP64>(grid, block, st, E, F, cs, stops_dev, stop_row, n_stops, out, out_stride, aos, kof, ctr, Q, ug, next_body, refill, q);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !split) return e;
    // phase 2: the set-aside bodies, one warp each
    PropQueue q2{};
    q2.list = defer->list;
    q2.list_n = defer->count;
    q2.resume = 1;
    return launch_propagate_warp(E, F, defer->model, cs, stops_dev, stop_row, n_stops, out,
                                 out_stride, keep_on_fail, ctr, st, q2, out_aos);
}

cudaError_t launch_fit_lanes(const EphemDev &E, const ForceDev &F, const AdjBuffers &B,
                             const AdjProblem &P, int64_t i0, int64_t nc, const GridDev &Q,
                             unsigned long long *next, const int32_t *order,
                             const unsigned long long *order_n, const PropDefer &defer,
                             cudaStream_t st)
{
    if (nc <= 0) return cudaGetLastError();
    cudaError_t e = cudaMemsetAsync(next, 0, sizeof(unsigned long long), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(defer.count, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    ChainState cs{};
    cs.n = nc;
    PropQueue q{};
    if (order && order_n) {
        q.list = order;
        q.list_n = order_n;
    }
    q.defer = defer.list;
    q.defer_n = defer.count;
    q.budget0 = defer.budget0;
    const int64_t need = (nc + 127) / 128, most = ws_blocks<KETE_FP64>(128);
    k_propagate<KETE_FP64, false, false, true><<<(unsigned)std::min(need, most), 128, 0, st>>>(
        E, F, cs, nullptr, nullptr, 0, nullptr, 0, 0, 0, P.ctr, Q, 1, next, 1, q,
        FitRecord{B, P, i0});
    return cudaGetLastError();
}

cudaError_t launch_gather_bodies(const double *st, const double *ep, int64_t n, int64_t m,
                                 double *dst, double *dep, cudaStream_t s)
{
    if (m > 0) k_gather_bodies<<<grid_for(m, 256), 256, 0, s>>>(st, ep, n, m, dst, dep);
    return cudaGetLastError();
}

cudaError_t launch_chain_finish(ChainState cs, double *states, double *epochs, int32_t *status,
                                cudaStream_t st)
{
    (void)states;
    if (cs.n > 0) k_chain_finish<<<grid_for(cs.n, 256), 256, 0, st>>>(cs, epochs, status);
    return cudaGetLastError();
}

}  // namespace kete
