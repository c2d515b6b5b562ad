// kete_warp.cu -- n-body propagation with one warp per body (Sec. 3.2, App. A,
// App. A.6): the form for few bodies and for the bodies that need far more
// steps than the rest.
//
// An FP64 warp instruction occupies its SM sub-partition's FP64 unit for 64
// cycles whatever its active lanes, so a lane-per-body step is a serial chain
// of 15-16 force evaluations x 250 FP64 instructions on the grid's rows (650
// off it): 0.4 ms, and the slowest body of a call sets its time.  Here the 32 lanes of a warp share one
// body's step: lane 4 n + r holds Gauss-Radau node n (0: the step start) and
// every fourth mass from r on, and coordinate r of the corrector.
//   - The planets at the 8 nodes are summed once per attempt and kept in
//     registers for all its sweeps.
//   - A sweep evaluates the forces at the 7 nodes together from the previous
//     sweep's coefficients (Jacobi order; the lane kernel's sweep updates them
//     node by node).  It converges to the same collocation solution, in about
//     one sweep more.
//   - The divided differences run through the nodes by shuffles, level by
//     level, in the lane kernel's arithmetic; positions and velocities at the
//     nodes come from the Newton coefficients directly (tabulated integrals of
//     the Newton basis), so no power-basis conversion is done.
// About 170 FP64 instructions a sweep, 180 for the planets of an attempt and 85
// to continue the previous step's polynomial (2.0-2.3 sweeps a step; 1,000
// comet clones over 8 years 21.5 ms, 26.5 from the two-body derivatives).
// Steps end only at the last stop of a direction; the stops inside a step come
// from its polynomial, eight at a time (one per node group).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "kete_adjoint.h"
#include "kete_step.cuh"

namespace kete {

struct WarpTables {
    double wx[8][7];    // double integral of Newton basis k+1 at node n, over s_n^2
    double wv[8][7];    // its integral, over s_n
    double wxe[7], wve[7];   // the same at the step end
};
static __constant__ WarpTables g_wt;

static WarpTables warp_tables()
{
    RadauTables t;
    fill_radau_tables(t);
    WarpTables w;
    for (int n = 0; n < 9; n++) {
        const long double s = n < 8 ? (long double)kRadauH[n] : 1.0L;
        for (int k = 0; k < 7; k++) {
            long double ax = 0.0L, av = 0.0L, sp = s;
            for (int m = 0; m <= k; m++) {
                ax += (long double)t.c[k + 1][m] * sp / ((m + 2.0L) * (m + 3.0L));
                av += (long double)t.c[k + 1][m] * sp / (m + 2.0L);
                sp *= s;
            }
            (n < 8 ? w.wx[n] : w.wxe)[k] = (double)ax;
            (n < 8 ? w.wv[n] : w.wve)[k] = (double)av;
        }
    }
    return w;
}

cudaError_t upload_warp_tables(cudaStream_t st)
{
    static const WarpTables w = warp_tables();   // (the copy may read it after the return)
    cudaError_t e = upload_step_tables(st);
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbolAsync(g_wt, &w, sizeof(w), 0, cudaMemcpyHostToDevice, st);
}

constexpr int kSlots = kWarpSlots;
constexpr unsigned kFull = 0xffffffffu;

bool warp_model(const EphemDev &E, const ForceDev &F, WarpModel &W)
{
    int n = 0, special = 0;
    for (int q = 0; q < 4 * kSlots; q++) W.list[q] = -1;
    if (!(F.active_mask & 1u)) return false;   // the Sun leads slot 0
    for (int pass = 0; pass < 2; pass++)
        for (int m = 0; m < E.n_bodies; m++) {
            if (!((F.active_mask >> m) & 1u)) continue;
            const bool sp = m == 0 || (((F.gr_mask | F.j2_mask) >> m) & 1u);
            if (sp != (pass == 0)) continue;
            if (n >= 4 * kSlots) return false;
            W.list[n++] = m;
            if (sp) special++;
        }
    W.gr = F.gr_mask != 0;
    W.j2 = F.j2_mask != 0;
    return special <= 4;
}

// the planets of one lane at its node
struct LaneMasses {
    double mu[kSlots];
    double p[kSlots][3];      // position (the encounter's mass: its displacement since the start)
    double w[3];              // velocity of slot 0's mass
    double mu4, grk, gr4k, j2k, pole[3];   // slot 0
    int id[kSlots];
};

__device__ __forceinline__ bool lane_planets(const EphemDev &E, const WarpModel &W, double t,
                                             double off, LaneMasses &M)
{
    Seg g;
    if (!ephem_seg(E, t, off, g)) return false;
    const double t2 = 2.0 * g.tau;
    const int nc = E.n_coef;
    const double *c0 = ephem_coef(E, M.id[0] < 0 ? 0 : M.id[0], g.s);
    const double *c1 = ephem_coef(E, M.id[1] < 0 ? 0 : M.id[1], g.s);
    const double *c2 = ephem_coef(E, M.id[2] < 0 ? 0 : M.id[2], g.s);
    double Tm1 = 1.0, T = g.tau, Um1 = 1.0, U = t2;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const double k1 = __ldg(c0 + d * nc + 1);
        M.p[0][d] = fma(k1, g.tau, __ldg(c0 + d * nc));
        M.w[d] = k1;
        M.p[1][d] = fma(__ldg(c1 + d * nc + 1), g.tau, __ldg(c1 + d * nc));
        M.p[2][d] = fma(__ldg(c2 + d * nc + 1), g.tau, __ldg(c2 + d * nc));
    }
#pragma unroll 2
    for (int k = 2; k < nc; k++) {
        const double Tn = fma(t2, T, -Tm1);
        Tm1 = T;
        T = Tn;
        const double dk = (double)k * U;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const double a = __ldg(c0 + d * nc + k);
            M.p[0][d] = fma(a, T, M.p[0][d]);
            M.w[d] = fma(a, dk, M.w[d]);
            M.p[1][d] = fma(__ldg(c1 + d * nc + k), T, M.p[1][d]);
            M.p[2][d] = fma(__ldg(c2 + d * nc + k), T, M.p[2][d]);
        }
        const double Un = fma(t2, U, -Um1);
        Um1 = U;
        U = Un;
    }
    const double dtau = 2.0 * E.inv_seg;
#pragma unroll
    for (int d = 0; d < 3; d++) M.w[d] *= dtau;
    return true;
}

__device__ __forceinline__ void newton_term(double mu, const double r[3], double a[3])
{
    const double ri = rsqrt(fma(r[0], r[0], fma(r[1], r[1], r[2] * r[2])));
    const double f = -mu * (ri * ri * ri);
    a[0] = fma(f, r[0], a[0]);
    a[1] = fma(f, r[1], a[1]);
    a[2] = fma(f, r[2], a[2]);
}

// The lane's masses at (x, v) of its node; dx: displacement since the step
// start.  The sum of coordinate r over the group's four lanes is returned in
// lane r (r = 3: nothing).  ng (lane 3 adds it): the body's own terms.
__device__ __forceinline__ double node_force(const WarpModel &W, const LaneMasses &M,
                                             const double x[3], const double v[3],
                                             const double dx[3], int enc_slot, const double d0[3],
                                             int r, const double own[3])
{
    double a[3] = {own[0], own[1], own[2]};
#pragma unroll
    for (int s = kSlots - 1; s >= 0; s--) {   // the Sun last
        double d[3];
#pragma unroll
        for (int c = 0; c < 3; c++)
            d[c] = enc_slot == s ? d0[c] + (dx[c] - M.p[s][c]) : x[c] - M.p[s][c];
        if (s > 0) {
            newton_term(M.mu[s], d, a);
            continue;
        }
        const double rr = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
        const double ri = rsqrt(rr), ri2 = ri * ri, ri3 = ri2 * ri;
        double f = -M.mu[0] * ri3;
        if (W.gr) {
            const double w[3] = {v[0] - M.w[0], v[1] - M.w[1], v[2] - M.w[2]};
            const double ww = fma(w[0], w[0], fma(w[1], w[1], w[2] * w[2]));
            const double rw = fma(d[0], w[0], fma(d[1], w[1], d[2] * w[2]));
            f = fma(M.grk * ri3, fma(M.mu4, ri, -ww), f);
            const double fw = (M.gr4k * ri3) * rw;
#pragma unroll
            for (int c = 0; c < 3; c++) a[c] = fma(fw, w[c], a[c]);
        }
        if (W.j2) {
            const double z = fma(d[0], M.pole[0], fma(d[1], M.pole[1], d[2] * M.pole[2]));
            const double psi = M.j2k * ri3 * ri2;
            f = fma(-psi, fma(-5.0, z * z * ri2, 1.0), f);
            const double fp = -2.0 * (psi * z);
#pragma unroll
            for (int c = 0; c < 3; c++) a[c] = fma(fp, M.pole[c], a[c]);
        }
#pragma unroll
        for (int c = 0; c < 3; c++) a[c] = fma(f, d[c], a[c]);
    }
    // transposed sum: lane r ends with coordinate r
    const bool odd = r & 1;
    const double s0 = odd ? a[0] : a[1], s1 = odd ? a[2] : 0.0;
    const double g0 = __shfl_xor_sync(kFull, s0, 1), g1 = __shfl_xor_sync(kFull, s1, 1);
    const double lo = (odd ? a[1] : a[0]) + g0;        // coordinate r & 1
    const double hi = odd ? 0.0 : a[2] + g1;           // coordinate 2 (even lanes)
    const double snd = r < 2 ? hi : lo;
    const double got = __shfl_xor_sync(kFull, snd, 2);
    return (r < 2 ? lo : hi) + got;
}

__device__ __forceinline__ float warp_max(float v)   // v >= 0 or NaN
{
    return __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(v)));
}

// The Newtonian da/dx (newton_jacobian) at the lane's node from its masses,
// summed over the group's four lanes.
__device__ __forceinline__ void node_jacobian(const LaneMasses &M, const double x[3],
                                              const double dx[3], int enc_slot,
                                              const double d0[3], double J[6])
{
#pragma unroll
    for (int q = 0; q < 6; q++) J[q] = 0.0;
#pragma unroll
    for (int s = 0; s < kSlots; s++) {
        double d[3];
#pragma unroll
        for (int c = 0; c < 3; c++)
            d[c] = enc_slot == s ? d0[c] + (dx[c] - M.p[s][c]) : x[c] - M.p[s][c];
        newton_jacobian(M.mu[s], d, J);
    }
#pragma unroll
    for (int q = 0; q < 6; q++) {
        J[q] += __shfl_xor_sync(kFull, J[q], 1);
        J[q] += __shfl_xor_sync(kFull, J[q], 2);
    }
}

// the forward pass of an orbit fit (REC): its arrays and the chunk's first body
struct WarpRecord {
    AdjBuffers B;
    AdjProblem P;
    int64_t i0;
};

// REC: the bodies are those of an orbit fit.  The stops are each body's batch
// midpoints, kept with the step each lies in, and every accepted step leaves
// its epochs and the Newtonian da/dx at its nodes (see kete_adjoint.cu).
template <bool NG, bool REC>
__global__ void __launch_bounds__(32)
k_propagate_warp(EphemDev E, ForceDev F, WarpModel W, ChainState cs,
                 const double *__restrict__ stops_in, const int32_t *__restrict__ stop_row,
                 int n_stops_in, double *__restrict__ out, int64_t out_stride, int out_aos,
                 int keep_on_fail, DevCounters *ctr, PropQueue q, WarpRecord R)
{
    __shared__ double mid[KETE_ADJ_MAX_OBS];
    const double *stops = REC ? mid : stops_in;
    int n_stops = n_stops_in;
    const int64_t n = cs.n;
    const int lane = threadIdx.x & 31, node = lane >> 2, r = lane & 3;
    const int rc = r < 3 ? r : 2;   // the coordinate this lane computes (lane 3: a copy of 2)
    const unsigned long long n_items = q.list ? *q.list_n : (unsigned long long)n;
    Cnt cnt = {0, 0, 0, 0, 0};
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const double inf = __longlong_as_double(0x7ff0000000000000ll);
    // this lane's constants
    LaneMasses M;
#pragma unroll
    for (int s = 0; s < kSlots; s++) {
        M.id[s] = W.list[4 * s + r];
        M.mu[s] = M.id[s] >= 0 ? E.gm[M.id[s]] : 0.0;
    }
    {
        const int m = M.id[0] < 0 ? 0 : M.id[0];
        const bool gr = M.id[0] >= 0 && ((F.gr_mask >> m) & 1u), j2 = M.id[0] >= 0 && ((F.j2_mask >> m) & 1u);
        M.mu4 = F.gm4[m];
        M.grk = gr ? F.grk[m] : 0.0;
        M.gr4k = gr ? F.gr4k[m] : 0.0;
        M.j2k = j2 ? F.j2k[m] : 0.0;
#pragma unroll
        for (int c = 0; c < 3; c++) M.pole[c] = j2 ? F.pole[m][c] : 0.0;
    }
    const double s_n = g_rt.h[node];
    double wx[7], wv[7], ri[7];
#pragma unroll
    for (int k = 0; k < 7; k++) {
        wx[k] = g_wt.wx[node][k];
        wv[k] = g_wt.wv[node][k];
        ri[k] = node > k ? g_rt.rinv[node][k] : 0.0;
    }
    const int max_sweeps = F.max_iter + 4;
    // the change of F between sweeps at the nodes, relative to |a|: one sweep more
    // contracts what is left by ~1e-3, below the rounding of the positions
    const float tol = (float)(0.3 * F.eps_pc);
    for (unsigned long long item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int64_t i = q.list ? (int64_t)q.list[item] : (int64_t)item;
        // own coordinate of the step-start state
        double x0, v0, t, dt = 0.0;
        int status = KETE_BODY_OK, k = 0, count = 0, used = 0;
        double *rec = nullptr;
        bool capped = false;
        if (REC) {
            const AdjProblem &P = R.P;
            const int64_t gi = R.i0 + i;
            const kete_obs *o = P.obs + gi * P.m;
            x0 = P.states[rc * P.n + gi];
            v0 = P.states[(3 + rc) * P.n + gi];
            t = P.epochs[gi];
            rec = R.B.rec + (size_t)i * R.B.cap * kAdjRec;
            if (!__all_sync(kFull, isfinite(x0) && isfinite(v0) && isfinite(t)))
                status = KETE_BODY_NONFINITE;
            const int mi = obs_count(o, P.m);
            bool sorted = true;
            for (int j = 1; j < mi; j++) sorted = sorted && !(o[j].epoch < o[j - 1].epoch);
            if (!sorted) {
                if (lane == 0) atomicOr(&ctr->error_flags, 1 << 6);
                status = KETE_BODY_NONFINITE;
            }
            n_stops = 0;
            double last = t;
            __syncwarp();
            for (int j0 = 0; j0 < mi; n_stops++) {
                j0 = next_batch(o, mi, j0, P.span, last);
                if (lane == 0) mid[n_stops] = last;
            }
            __syncwarp();
            // the checkpoint grid bounds no step here, but its stops count toward
            // the limits as they do where the steps end at them
            if (P.ckpt > 0.0 && last > t) {
                const double ck = ceil((last - t) / P.ckpt) - 1.0;
                if (ck >= (double)kAdjMaxCkpt) status = KETE_BODY_STEP_CAP;
                else if (ck + n_stops > (double)(R.B.cap - 1)) capped = true;
                count = 0;
            }
        } else {
            x0 = cs.w[rc * n + i];
            v0 = cs.w[(3 + rc) * n + i];
            t = cs.w[6 * n + i];
            dt = cs.w[7 * n + i];
            status = cs.status[i];
            k = q.resume ? cs.kstop[i] : 0;
        }
        const double epoch0 = t;
        const kete_nongrav *ng = (NG && F.nongrav) ? F.nongrav + i : nullptr;
        double ng_chi = 0.0;
        long long attempts = !REC && cs.tries ? cs.tries[i] : 0;
        bool careful = false, have_a0 = false;
        double a0 = 0.0, bound = inf;
        double d1 = 0.0, d2 = 0.0, d3 = 0.0;   // derivatives of a at the step start
        // the last attempt's Newton coefficients, its size, whether it is the
        // accepted step that ended here, and what the next one starts from
        double g[7], h_last = 1.0;
        bool chained = false;
        int start = START_A0;
        int enc_m = -1, enc_slot = -1;
        double d0[3] = {0.0, 0.0, 0.0};
        while (k < n_stops && status == KETE_BODY_OK) {
            const double next_stop = stops[k];
            if (REC && t == next_stop) {
                if (node == 0 && r < 3) {
                    double *y = R.B.yref + ((size_t)i * R.P.m + k) * 6;
                    y[r] = x0;
                    y[3 + r] = v0;
                }
                if (lane == 0) {
                    R.B.bidx[(size_t)i * R.P.m + k] = count;
                    R.B.bfrac[(size_t)i * R.P.m + k] = 0.0;
                }
                k++;
                attempts = 0;
                have_a0 = false;
                continue;
            }
            if (t == next_stop) {
                const int row = stop_row ? stop_row[k] : k;
                if (node == 0 && r < 3 && row >= 0) {
                    double *o = out_aos ? out + ((int64_t)row * out_stride + i) * 6
                                        : out + (int64_t)row * 6 * out_stride + i;
                    const int64_t s = out_aos ? 1 : out_stride;
                    o[r * s] = x0;
                    o[(3 + r) * s] = v0;
                }
                if (row != kMarkRow) attempts = 0;
                k++;
                have_a0 = false;
                continue;
            }
            aim_step(F, t, next_stop, dt);
            const bool fwd = next_stop > t;
            const double target = (careful || !fwd) ? next_stop : stops[n_stops - 1];
            if (++attempts > F.max_steps) {
                status = KETE_BODY_STEP_CAP;
                break;
            }
            double h, t_new;
            double sun[6] = {0, 0, 0, 0, 0, 0};
            bool inside = true;
            auto aim = [&]() {
                double t_stop = target;
                if (have_a0 && (fwd ? bound < target : bound > target)) t_stop = bound;
                t_new = fabs(dt) >= fabs(t_stop - t) ? t_stop : t + dt;
                h = t_new - t;
                inside = lane_planets(E, W, t, s_n * h, M);
            };
            aim();
            int st = __shfl_sync(kFull, (int)inside, 0) ? KETE_BODY_OK : KETE_BODY_OUT_OF_SPAN;
            // full state of the step start in every lane
            const double xs[3] = {__shfl_sync(kFull, x0, 0), __shfl_sync(kFull, x0, 1),
                                  __shfl_sync(kFull, x0, 2)};
            const double vs[3] = {__shfl_sync(kFull, v0, 0), __shfl_sync(kFull, v0, 1),
                                  __shfl_sync(kFull, v0, 2)};
            const double zero[3] = {0.0, 0.0, 0.0};
            // the body's own terms at the lane's node (lane 3 of each group)
            auto own_terms = [&](bool on, const double x[3], const double v[3], double own[3]) -> int {
                own[0] = own[1] = own[2] = 0.0;
                int s2 = KETE_BODY_OK;
                if (NG && ng && on && r == 3) {
                    const double hr[3] = {x[0] - sun[0], x[1] - sun[1], x[2] - sun[2]};
                    const double hw[3] = {v[0] - sun[3], v[1] - sun[4], v[2] - sun[5]};
                    const NgOut o = nongrav_helio(E.gm[0], ng, hr[0], hr[1], hr[2], hw[0], hw[1],
                                                  hw[2], ng_chi);
                    ng_chi = o.chi;
                    s2 = o.status;
                    own[0] = o.a[0]; own[1] = o.a[1]; own[2] = o.a[2];
                }
                return s2;
            };
            auto share_sun = [&]() {
                if (NG && ng) {
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        sun[c] = __shfl_sync(kFull, M.p[0][c], lane & ~3);
                        sun[3 + c] = __shfl_sync(kFull, M.w[c], lane & ~3);
                    }
                }
            };
            if (st == KETE_BODY_OK && !have_a0) {
                // acceleration at the step start and the nearest planet: node 0's lanes
                share_sun();
                double best = kEncounterAu * kEncounterAu;
                int bm = -1;
#pragma unroll
                for (int s = 0; s < kSlots; s++) {
                    const double e0 = xs[0] - M.p[s][0], e1 = xs[1] - M.p[s][1], e2 = xs[2] - M.p[s][2];
                    const double rr = e0 * e0 + e1 * e1 + e2 * e2;
                    if (M.id[s] > 0 && (rr < best || (rr == best && M.id[s] < bm))) {
                        best = rr;
                        bm = M.id[s];
                        d0[0] = e0; d0[1] = e1; d0[2] = e2;
                    }
                }
                double own[3];
                const int s2 = own_terms(node == 0, xs, vs, own);
                const double f = node_force(W, M, xs, vs, zero, -1, d0, r, own);
                a0 = __shfl_sync(kFull, f, r);
                start = chained ? START_NEXT : START_DERIVS;
                if (!chained) {   // two_body_derivs, from the Sun in lane 0
                    double hr[3], hw[3], e1[3], e2[3], e3[3];
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        hr[c] = xs[c] - __shfl_sync(kFull, M.p[0][c], 0);
                        hw[c] = vs[c] - __shfl_sync(kFull, M.w[c], 0);
                    }
                    two_body_derivs(E.gm[0], hr, hw, e1, e2, e3);
                    d1 = rc == 0 ? e1[0] : rc == 1 ? e1[1] : e1[2];
                    d2 = rc == 0 ? e2[0] : rc == 1 ? e2[1] : e2[2];
                    d3 = rc == 0 ? e3[0] : rc == 1 ? e3[1] : e3[2];
                }
                if (NG && ng) st = __shfl_sync(kFull, s2, 3);
                cnt.evals++;
#pragma unroll
                for (int o = 1; o <= 2; o <<= 1) {   // within the group of four
                    const double ob = __shfl_xor_sync(kFull, best, o);
                    const int om = __shfl_xor_sync(kFull, bm, o);
                    double od[3];
#pragma unroll
                    for (int c = 0; c < 3; c++) od[c] = __shfl_xor_sync(kFull, d0[c], o);
                    if (om >= 0 && (bm < 0 || ob < best || (ob == best && om < bm))) {
                        best = ob;
                        bm = om;
                        d0[0] = od[0]; d0[1] = od[1]; d0[2] = od[2];
                    }
                }
                enc_m = __shfl_sync(kFull, bm, 0);
#pragma unroll
                for (int c = 0; c < 3; c++) d0[c] = __shfl_sync(kFull, d0[c], 0);
                bound = fwd ? inf : -inf;
                enc_slot = -1;
                if (enc_m >= 0) {
                    const double kk = floor((t - E.t_start) * E.inv_seg);
                    double b = fwd ? E.t_start + (kk + 1.0) * E.seg_len : E.t_start + kk * E.seg_len;
                    if (!fwd && b == t) b = E.t_start + (kk - 1.0) * E.seg_len;
                    bound = b;
#pragma unroll
                    for (int s = 0; s < kSlots; s++)
                        if (M.id[s] == enc_m) enc_slot = s;
                }
                have_a0 = st == KETE_BODY_OK;
                if (have_a0 && (fwd ? bound < t_new : bound > t_new)) aim();
            }
            if (st == KETE_BODY_OK && !__all_sync(kFull, inside)) st = KETE_BODY_OUT_OF_SPAN;
            if (st == KETE_BODY_OK && h == 0.0) {
                status = KETE_BODY_STEP_CAP;   // step below the epoch resolution
                break;
            }
            double b6 = 0.0, amax = 0.0;
            if (st == KETE_BODY_OK) {
                share_sun();
                if (enc_m >= 0 && enc_slot >= 0) {   // that planet's displacement instead
                    double dp[3];
                    cheb_delta64(E, enc_m, t, s_n * h, dp);
#pragma unroll
                    for (int s = 0; s < kSlots; s++)
                        if (enc_slot == s) {
                            M.p[s][0] = dp[0]; M.p[s][1] = dp[1]; M.p[s][2] = dp[2];
                        }
                }
                const double sh = s_n * h, sh2 = sh * sh, shv = sh * v0;
                double Fo = a0;
                float pc_prev = 0.0f;
                if (start == START_NEXT || start == START_RETRY) {   // as attempt_begin
                    double b[7];
#pragma unroll
                    for (int m = 0; m < 7; m++) {
                        b[m] = 0.0;
#pragma unroll
                        for (int p = 6; p >= m; p--) b[m] = fma(g_rt.c[p + 1][m], g[p], b[m]);
                    }
                    continue_poly(b, h / h_last, start == START_NEXT ? 1.0 : 0.0);
                    double pn = 0.0;
#pragma unroll
                    for (int m = 6; m >= 0; m--) {
                        pn = fma(pn, s_n, b[m]);
                        g[m] = b[m];
                    }
                    newton_form(g);
                    Fo = fma(pn, s_n, a0);   // what the start predicts at the node
                } else {
#pragma unroll
                    for (int m = 3; m < 7; m++) g[m] = 0.0;
                    const double h1 = g_rt.h[1], h2 = g_rt.h[2];
                    const double b0 = h * d1, b1 = 0.5 * h * h * d2, b2 = h * h * h * (1.0 / 6.0) * d3;
                    g[2] = b2;
                    g[1] = fma(h1 + h2, b2, b1);
                    g[0] = fma(h1, g[1], fma(-h1 * h2, b2, b0));
                    // what the start predicts at the node
                    Fo = fma(fma(fma(d3, sh * (1.0 / 3.0), d2), 0.5 * sh, d1), sh, a0);
                }
                for (int it = 1;; it++) {
                    double px = g[6] * wx[6], pv = g[6] * wv[6];
#pragma unroll
                    for (int m = 5; m >= 0; m--) {
                        px = fma(g[m], wx[m], px);
                        pv = fma(g[m], wv[m], pv);
                    }
                    px = fma(a0, 0.5, px);
                    const double dxr = fma(sh2, px, shv);
                    const double vr = fma(sh, pv + a0, v0);
                    double dx[3], xn[3], vn[3];
                    const int b = lane & ~3;
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        dx[c] = __shfl_sync(kFull, dxr, b + c);
                        vn[c] = __shfl_sync(kFull, vr, b + c);
                        xn[c] = xs[c] + dx[c];
                    }
                    double own[3];
                    const int s2 = own_terms(node > 0, xn, vn, own);
                    if (NG && ng) {
                        const unsigned bad = __ballot_sync(kFull, s2 != KETE_BODY_OK);
                        if (bad) st = __shfl_sync(kFull, s2, __ffs(bad) - 1);
                    }
                    const double Fn = node_force(W, M, xn, vn, dx, enc_slot, d0, r, own);
                    // divided differences, node by node
                    double d = (Fn - a0) * ri[0];
#pragma unroll
                    for (int m = 1; m < 7; m++) {
                        g[m - 1] = __shfl_sync(kFull, d, 4 * m + rc);
                        if (node > m) d = (d - g[m - 1]) * ri[m];
                    }
                    g[6] = __shfl_sync(kFull, d, 28 + rc);
                    const float df = (node > 0 && r < 3) ? fabsf((float)(Fn - Fo)) : 0.0f;
                    const float fm = (node == 7 && r < 3) ? fabsf((float)Fn) : 0.0f;
                    const float pc = warp_max(df) / warp_max(fm);
                    Fo = Fn;
                    cnt.iters++;
                    cnt.evals += 7;
                    if (st != KETE_BODY_OK) break;
                    if (!isfinite(pc)) {
                        st = KETE_BODY_NONFINITE;
                        break;
                    }
                    if ((pc < tol && it >= 2) || (it >= 3 && pc >= pc_prev) || it >= max_sweeps) break;
                    pc_prev = pc;
                }
                h_last = h;
                b6 = fabs(g[6]);
                const double f7 = fabs(__shfl_sync(kFull, Fo, 28 + rc));
                b6 = fmax(__shfl_sync(kFull, b6, 0), fmax(__shfl_sync(kFull, b6, 1), __shfl_sync(kFull, b6, 2)));
                amax = fmax(__shfl_sync(kFull, f7, 0), fmax(__shfl_sync(kFull, f7, 1), __shfl_sync(kFull, f7, 2)));
            }
            double x1 = 0.0, v1 = 0.0;
            if (st == KETE_BODY_OK) {
                double px = g[6] * g_wt.wxe[6], pv = g[6] * g_wt.wve[6];
#pragma unroll
                for (int m = 5; m >= 0; m--) {
                    px = fma(g[m], g_wt.wxe[m], px);
                    pv = fma(g[m], g_wt.wve[m], pv);
                }
                px = fma(a0, 0.5, px);
                x1 = fma(h * h, px, fma(h, v0, x0));
                v1 = fma(h, pv + a0, v0);
                if (!__all_sync(kFull, isfinite(x1) && isfinite(v1))) st = KETE_BODY_NONFINITE;
            }
            if (st != KETE_BODY_OK) {
                if (!careful && fwd && t_new != next_stop) {
                    // a step past a stop failed: stop by stop from here
                    careful = true;
                    d1 = d2 = d3 = 0.0;   // (the attempt's polynomial is of no use)
                    start = START_A0;
                    chained = false;
                    continue;
                }
                status = st;
                break;
            }
            const double err = b6 / amax;
            const double factor = step_factor(F, err);
            dt = factor * h;
            if (factor < F.safety) {   // reject: retry from the same a0
                cnt.rejected++;
                start = START_RETRY;
                continue;
            }
            cnt.steps++;
            if (REC) {   // the step's record: da/dx at the nodes of its final polynomial
                double px = g[6] * wx[6];
#pragma unroll
                for (int m = 5; m >= 0; m--) px = fma(g[m], wx[m], px);
                const double sh = s_n * h;
                const double dxr = fma(sh * sh, fma(a0, 0.5, px), sh * v0);
                double dx[3], xn[3], J[6];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    dx[c] = __shfl_sync(kFull, dxr, (lane & ~3) + c);
                    xn[c] = xs[c] + dx[c];
                }
                node_jacobian(M, xn, dx, enc_slot, d0, J);
                if (count < R.B.cap - 1) {
                    double *rr = rec + (size_t)count * kAdjRec;
                    if (lane == 0) {
                        rr[0] = t;
                        rr[1] = t_new;
                    }
                    if (r < 3) {
                        rr[2 + 6 * node + r] = r == 0 ? J[0] : r == 1 ? J[1] : J[2];
                        rr[5 + 6 * node + r] = r == 0 ? J[3] : r == 1 ? J[4] : J[5];
                    }
                } else {
                    capped = true;
                }
            }
            const int k_from = k;
            // stops inside the step, eight at a time (node group q takes stop k + q)
            if (fwd && !careful && stops[k] < t_new) {
                double b[7];
#pragma unroll
                for (int m = 0; m < 7; m++) {
                    b[m] = 0.0;
#pragma unroll
                    for (int p = 6; p >= m; p--) b[m] = fma(g_rt.c[p + 1][m], g[p], b[m]);
                }
                for (;;) {
                    const int kq = k + node;
                    const bool in = kq < n_stops && stops[kq] < t_new;
                    const int row = in ? (!REC && stop_row ? stop_row[kq] : kq) : -1;
                    if (REC && in && r == 3) {
                        R.B.bidx[(size_t)i * R.P.m + kq] = count;
                        R.B.bfrac[(size_t)i * R.P.m + kq] = (stops[kq] - t) / h;
                    }
                    if (row >= 0 && r < 3) {
                        const double off = stops[kq] - t, s = off / h;
                        double px = 0.0, pv = 0.0;   // Horner in s
#pragma unroll
                        for (int m = 6; m >= 0; m--) {
                            px = fma(px, s, b[m] * (1.0 / ((m + 2.0) * (m + 3.0))));
                            pv = fma(pv, s, b[m] * (1.0 / (m + 2.0)));
                        }
                        px = fma(px, s, 0.5 * a0);
                        pv = fma(pv, s, a0);
                        double *o = REC ? R.B.yref + ((size_t)i * R.P.m + row) * 6
                                    : out_aos ? out + ((int64_t)row * out_stride + i) * 6
                                              : out + (int64_t)row * 6 * out_stride + i;
                        const int64_t sd = REC || out_aos ? 1 : out_stride;
                        o[r * sd] = x0 + fma(off * off, px, off * v0);
                        o[(3 + r) * sd] = fma(off, pv, v0);
                    }
                    const int took = __popc(__ballot_sync(kFull, in)) / 4;
                    k += took;
                    if (took < 8) break;
                }
                attempts = 0;
            }
            if (REC) {
                const double ck = ckpts_before(R.P.inv_ckpt, epoch0, t_new) -
                                  ckpts_before(R.P.inv_ckpt, epoch0, t);
                used += steps_with_stops(ck, k - k_from + (k < n_stops && stops[k] == t_new));
                if (ck > 0.0) attempts = 0;   // max_steps counts the attempts of a leg
            }
            x0 = x1;
            v0 = v1;
            t = t_new;
            have_a0 = false;
            chained = factor <= kNextMost;
            if (REC && count < R.B.cap - 1) count++;
        }
        if (REC) {
            if (R.P.ckpt > 0.0 && used > R.B.cap - 1) capped = true;
            if (status == KETE_BODY_OK && !capped) {   // da/dx at the final state closes the last step
                const bool inside = lane_planets(E, W, t, 0.0, M);
                const double zero[3] = {0.0, 0.0, 0.0};
                const double xs[3] = {__shfl_sync(kFull, x0, 0), __shfl_sync(kFull, x0, 1),
                                      __shfl_sync(kFull, x0, 2)};
                double J[6];
                node_jacobian(M, xs, zero, -1, zero, J);
                if (!__all_sync(kFull, inside)) status = KETE_BODY_OUT_OF_SPAN;
                if (lane == 0) {
                    double *rr = rec + (size_t)count * kAdjRec;
                    rr[0] = t;
                    rr[1] = t;
#pragma unroll
                    for (int c = 0; c < 6; c++) rr[2 + c] = J[c];
                }
                count++;
            }
            if (status == KETE_BODY_OK && capped) status = KETE_BODY_ADJ_CAP;
            if (lane == 0) {
                R.B.n_rec[i] = status == KETE_BODY_OK ? count : 0;
                R.B.nbat[i] = n_stops;
                R.B.status[i] = status;
            }
            continue;
        }
        // a failed body: no state at the remaining stops
        if (status != KETE_BODY_OK && !keep_on_fail)
            for (; k < n_stops; k++) {
                const int row = stop_row ? stop_row[k] : k;
                if (row < 0 || node != 0 || r >= 3) continue;
                double *o = out_aos ? out + ((int64_t)row * out_stride + i) * 6
                                    : out + (int64_t)row * 6 * out_stride + i;
                const int64_t s = out_aos ? 1 : out_stride;
                o[r * s] = nan;
                o[(3 + r) * s] = nan;
            }
        if (node == 0 && r < 3) {
            cs.w[r * n + i] = x0;
            cs.w[(3 + r) * n + i] = v0;
        }
        if (lane == 0) {
            cs.w[6 * n + i] = t;
            cs.w[7 * n + i] = dt;
            cs.status[i] = status;
            if (cs.tries) cs.tries[i] = attempts;
        }
    }
    if (lane == 0) {
        atomicAdd(&ctr->steps, cnt.steps);
        atomicAdd(&ctr->rejected, cnt.rejected);
        atomicAdd(&ctr->force_evals, cnt.evals);
        atomicAdd(&ctr->iterations, cnt.iters);
    }
}

static unsigned warp_grid(int64_t n)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t most = (int64_t)(sms > 0 ? sms : 152) * 8;
    return (unsigned)(n < most ? n : most);
}

cudaError_t launch_adjoint_forward_warp(const EphemDev &E, const ForceDev &F, const WarpModel &W,
                                        const AdjBuffers &B, const AdjProblem &P, int64_t i0,
                                        int64_t nc, cudaStream_t st, PropQueue q)
{
    if (nc <= 0) return cudaGetLastError();
    ChainState cs{};
    cs.n = nc;
    k_propagate_warp<false, true><<<warp_grid(nc), 32, 0, st>>>(
        E, F, W, cs, nullptr, nullptr, 0, nullptr, 0, 0, 0, P.ctr, q, WarpRecord{B, P, i0});
    return cudaGetLastError();
}

cudaError_t launch_propagate_warp(const EphemDev &E, const ForceDev &F, const WarpModel &W,
                                  ChainState cs, const double *stops, const int32_t *row,
                                  int n_stops, double *out, int64_t stride, bool keep_on_fail,
                                  DevCounters *ctr, cudaStream_t st, PropQueue q, bool out_aos)
{
    if (cs.n <= 0 || n_stops <= 0) return cudaGetLastError();
    const unsigned grid = warp_grid(cs.n);
    const int aos = out_aos ? 1 : 0, kof = keep_on_fail ? 1 : 0;
    if (F.nongrav)
        k_propagate_warp<true, false><<<grid, 32, 0, st>>>(E, F, W, cs, stops, row, n_stops, out, stride, aos, kof, ctr, q, WarpRecord{});
    else
        k_propagate_warp<false, false><<<grid, 32, 0, st>>>(E, F, W, cs, stops, row, n_stops, out, stride, aos, kof, ctr, q, WarpRecord{});
    return cudaGetLastError();
}

}  // namespace kete
