// kete_step.cuh -- one Gauss-Radau 15th-order step in the IAS15 form (Sec. 3.2,
// App. A.6), shared by the propagation kernel and the adjoint's forward pass.
// The paper removes the predictor; here the corrector starts from what is known
// of the motion (CorrectorStart), which changes its sweeps, not its solution.
//
// Each translation unit that includes this header holds its own copy of the
// node tables g_rt in constant memory and must fill it with
// upload_step_tables() before its first launch.
#pragma once

#include <cuda_runtime.h>

#include <cstring>

#include "kete_device.cuh"

namespace kete {
static __constant__ RadauTables g_rt;

// Gauss-Radau spacings on [0, 1] (Everhart 1985, 30 published digits)
static const double kRadauH[8] = {
    0.0,
    0.0562625605369221464656521910318,
    0.180240691736892364987579942780,
    0.352624717113169637373907769648,
    0.547153626330555383001448554766,
    0.734210177215410531523210605558,
    0.885320946839095768090359771030,
    0.977520613561287501891174488626,
};

static inline void fill_radau_tables(RadauTables &t)
{
    std::memset(&t, 0, sizeof(t));
    for (int n = 0; n < 8; n++) t.h[n] = kRadauH[n];
    for (int n = 0; n < 8; n++)
        for (int k = 0; k < n; k++) t.rinv[n][k] = 1.0 / (kRadauH[n] - kRadauH[k]);
    // Newton basis N_n(s) = s (s-h_1)...(s-h_{n-1}); c[n][m] = coefficient of
    // s^(m+1) in N_n, built by the recurrence N_n = N_{n-1} (s - h_{n-1}).
    double poly[8] = {1, 0, 0, 0, 0, 0, 0, 0};   // coefficients of prod (s-h_i), s^0 first
    for (int n = 1; n <= 7; n++) {
        if (n >= 2) {
            double nxt[8] = {0};
            for (int p = 0; p < 7; p++) {
                nxt[p + 1] += poly[p];
                nxt[p] -= kRadauH[n - 1] * poly[p];
            }
            std::memcpy(poly, nxt, sizeof(poly));
        }
        for (int m = 0; m < 7; m++) {
            t.c[n][m] = (m < n) ? poly[m] : 0.0;
            t.cf[n][m] = (float)t.c[n][m];
        }
    }
    // predictor weights of the power-basis coefficients at each node
    for (int n = 0; n < 8; n++) {
        double sp = kRadauH[n];
        for (int k = 0; k < 7; k++) {
            t.wx[n][k] = sp / ((k + 2.0) * (k + 3.0));
            t.wv[n][k] = sp / (k + 2.0);
            t.wvf[n][k] = (float)t.wv[n][k];
            sp *= kRadauH[n];
        }
    }
    // leading coefficient of the interpolant through the 8 nodes
    for (int n = 0; n < 8; n++) {
        double p = 1.0;
        for (int k = 0; k < 8; k++)
            if (k != n) p *= (kRadauH[n] - kRadauH[k]);
        t.w7[n] = 1.0 / p;
    }
}

// fill this translation unit's copy of g_rt
static inline cudaError_t upload_step_tables(cudaStream_t st)
{
    // (static: the copy may read it after the return)
    static const RadauTables t = [] { RadauTables r; fill_radau_tables(r); return r; }();
    return cudaMemcpyToSymbolAsync(g_rt, &t, sizeof(t), 0, cudaMemcpyHostToDevice, st);
}

struct Cnt {
    unsigned long long steps, rejected, evals, iters, node_evals;
};

// Planet rows of the 8 nodes of one step (null: the planets are summed per
// thread).
struct StepRows {
    const double *r64;
    const float *r32;
    int stride;   // elements per node
};

// Force evaluation dispatch by precision mode.
// detect: the evaluation at a step start, which also finds the planets near
// the body (see accel_fp64 / accel_mixed).
// JAC (FP64 only): also store the Newtonian da/dx at this point to jout[0..5].
template <int MODE, bool JAC = false>
__device__ __forceinline__ int accel(const EphemDev &E, const ForceDev &F, double t0, double off,
                                     const double *row64, const float *row32, uint32_t &close,
                                     const double x[3], const double v[3], double a[3],
                                     double as[3], Encounter &enc, const double dx[3], bool detect,
                                     double *jout = nullptr, const kete_nongrav *ng = nullptr,
                                     const float *vf = nullptr, double *ng_chi = nullptr,
                                     double *helio = nullptr,
                                     PlanetCache cache = PlanetCache{nullptr, 0, false})
{
    static_assert(!(JAC && MODE == KETE_MIXED), "Jacobian capture is FP64 only");
    if (MODE == KETE_MIXED)
        return accel_mixed(E, F, t0, off, row64, row32, close, x, v, a, as, enc, dx, detect, ng,
                           vf, ng_chi, helio);
    double J[6];
    int st = accel_fp64<JAC>(E, F, t0, off, row64, x, v, a, enc, dx, detect, J, ng, ng_chi, helio,
                             cache);
    as[0] = a[0]; as[1] = a[1]; as[2] = a[2];
    if (JAC) {
#pragma unroll
        for (int q = 0; q < 6; q++) jout[q] = J[q];
    }
    return st;
}

// Corrector state of one Gauss-Radau step attempt of size h (from t to
// t_new) between corrector sweeps; one sweep is one corrector iteration over
// the 7 substep nodes.  rows.r64 != null: a grid step, the planets come from
// its rows (node n at rows.r64 + n * stride).
struct Attempt {
    double b[7][3], g[7][3];
    float bf[7][3];         // mixed precision: b in FP32, for the node velocity
    double gs7[3];          // mixed precision: b6 of the FP64 part, last sweep
    double amax, pc_prev;   // max|a| at the last node and the last convergence measure
    double h, t_new;
    StepRows rows;
    int it;                 // sweeps done
};

// What a step's corrector starts from.  START_DERIVS: A.b[0..2] hold estimates
// of the first three time derivatives of a at the step start (two_body_derivs),
// the polynomial is a0 + b0 s + b1 s^2 + b2 s^3.  START_NEXT: A holds the
// accepted step that ended here, its polynomial is continued past its end.
// START_RETRY: A holds the rejected attempt from the same start, whose
// polynomial is cut to the new step.  START_A0: the constant a0.
// A main-belt step's continued polynomial is off by ~1e-8 of a where the
// two-body one is off by ~1e-5, one sweep's contraction: 250,000 mixed bodies
// over a year 224 -> 167 ms, 757,000 over 60 days 87 -> 71.  Not in mixed
// precision: the FP32 terms' rounding in b6 grows 2^7-fold over the next step
// (100,003 bodies with terms over 180 days 65.5 ms without, 69 with it).
// (FP64 only: START_NEXT, START_RETRY)
// START_NEXT only for a step of at most kNextMost times the last one: continued
// q steps far, b6 grows q^7-fold, and after a short step (to a grid point, to a
// segment boundary) its b6 is rounding, 1e-13 |a|.  The sweeps correct b by
// increments, so what rounding leaves of an absurd start stays in the solution:
// 400 bodies whose first step is 0.0015 days and whose second is 1 day ended 60
// days on 1e-6 AU off, 1e-15 within this bound.  At 16 the start is 3e-5 |a| off, no
// more than the two-body one; step control grows a step by at most 1 / safety, 4
// by default (a bound of 4, met by steps to grid points, cost 99,000 mixed bodies
// over 400 days 82.8 ms, 16 costs 77.3).
enum CorrectorStart { START_A0, START_DERIVS, START_NEXT, START_RETRY };
constexpr double kNextMost = 16.0;

// coefficients b of sum b_k s^(k+1) in s' of s = next + q s' (next 1 or 0), the
// constant dropped: b'_k = q^(k+1) (b_k + next sum_{j>k} C(j+1, k+1) b_j)
__device__ __forceinline__ void continue_poly(double b[7], double q, double next)
{
    constexpr double binom[7][7] = {{1, 2, 3, 4, 5, 6, 7},    {0, 1, 3, 6, 10, 15, 21},
                                    {0, 0, 1, 4, 10, 20, 35}, {0, 0, 0, 1, 5, 15, 35},
                                    {0, 0, 0, 0, 1, 6, 21},   {0, 0, 0, 0, 0, 1, 7},
                                    {0, 0, 0, 0, 0, 0, 1}};
    double qp = q;
#pragma unroll
    for (int k = 0; k < 7; k++) {
        double c = 0.0;
#pragma unroll
        for (int j = 6; j > k; j--) c = fma(binom[k][j], b[j], c);
        b[k] = qp * fma(next, c, b[k]);
        qp *= q;
    }
}

// power-basis b -> Newton-basis g in place: repeated synthetic division by s - h_n
__device__ __forceinline__ void newton_form(double g[7])
{
#pragma unroll
    for (int n = 0; n < 6; n++)
#pragma unroll
        for (int m = 5; m >= n; m--) g[m] = fma(g_rt.h[n + 1], g[m + 1], g[m]);
}

__device__ __forceinline__ void attempt_begin(Attempt &A, double h, double t_new, StepRows rows,
                                              int start)
{
    if (start == START_NEXT || start == START_RETRY) {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            double c[7];
#pragma unroll
            for (int k = 0; k < 7; k++) c[k] = A.b[k][i];
            continue_poly(c, h / A.h, start == START_NEXT ? 1.0 : 0.0);
#pragma unroll
            for (int k = 0; k < 7; k++) A.b[k][i] = c[k];
            newton_form(c);
#pragma unroll
            for (int k = 0; k < 7; k++) A.g[k][i] = c[k];
        }
    } else {
        const double h1 = g_rt.h[1], h2 = g_rt.h[2];
        const bool fresh = start == START_DERIVS;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const double b0 = fresh ? h * A.b[0][i] : 0.0;
            const double b1 = fresh ? (0.5 * h * h) * A.b[1][i] : 0.0;
            const double b2 = fresh ? (h * h * h * (1.0 / 6.0)) * A.b[2][i] : 0.0;
            // Newton basis: s, s (s - h1), s (s - h1) (s - h2)
            const double g1 = fma(h1 + h2, b2, b1);
            A.g[0][i] = fma(h1, g1, fma(-h1 * h2, b2, b0));
            A.g[1][i] = g1;
            A.g[2][i] = b2;
            A.b[0][i] = b0;
            A.b[1][i] = b1;
            A.b[2][i] = b2;
        }
#pragma unroll
        for (int m = 3; m < 7; m++)
#pragma unroll
            for (int i = 0; i < 3; i++) A.b[m][i] = A.g[m][i] = 0.0;
    }
#pragma unroll
    for (int m = 0; m < 7; m++)
#pragma unroll
        for (int i = 0; i < 3; i++) A.bf[m][i] = m < 3 ? (float)A.b[m][i] : 0.0f;
    A.gs7[0] = A.gs7[1] = A.gs7[2] = 0.0;
    A.amax = 0.0;
    A.pc_prev = 0.0;
    A.h = h;
    A.t_new = t_new;
    A.rows = rows;
    A.it = 0;
}

// The corrector update at node N (compile-time): Newton divided difference
// g_{N-1} from the node's force and the earlier g, then the power-basis
// coefficients b.
template <int MODE, int N, bool V32 = false>
__device__ __forceinline__ void node_update(Attempt &A, const double Fn[3], const double Fs[3],
                                            const double a0[3], double F7[3])
{
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double gn = (Fn[i] - a0[i]) * g_rt.rinv[N][0];
#pragma unroll
        for (int k = 1; k < N; k++) gn = (gn - A.g[k - 1][i]) * g_rt.rinv[N][k];
        double dg = gn - A.g[N - 1][i];
        A.g[N - 1][i] = gn;
#pragma unroll
        for (int m = 0; m < N; m++) A.b[m][i] = fma(g_rt.c[N][m], dg, A.b[m][i]);
        if (MODE == KETE_MIXED && V32) {
            const float dgf = (float)dg;
#pragma unroll
            for (int m = 0; m < N; m++) A.bf[m][i] = fmaf(g_rt.cf[N][m], dgf, A.bf[m][i]);
        }
        if (N == 7) F7[i] = Fn[i];
        if (MODE == KETE_MIXED) A.gs7[i] = fma(g_rt.w7[N], Fs[i], A.gs7[i]);
    }
}

// One corrector sweep of the attempt from (t, x0, v0) with a0 = a(t, x0, v0)
// (as0: its FP64 part).  V32: see vel32 below.  Sets done when the corrector has converged
// (max|db6|/max|a| < eps_pc), stopped improving (from the third sweep) or
// reached max_iter sweeps.  JAC: every node evaluation also stores da/dx at
// node n to jrec[6n..6n+5]; the last sweep's values remain.
// planets (FP64, no rows): this lane's scratch of 7 E.n_bodies 6 doubles, pstride
// apart, where the first sweep keeps the planets for the others.
template <int MODE, bool JAC = false, bool V32 = false>
__device__ __forceinline__ int attempt_sweep(const EphemDev &E, const ForceDev &F, double t,
                                             const double x0[3], const double v0[3],
                                             const double a0[3], const double as0[3],
                                             uint32_t close, Encounter enc, Attempt &A, bool &done,
                                             Cnt &cnt, double *jrec = nullptr,
                                             const kete_nongrav *ng = nullptr,
                                             double *ng_chi = nullptr, double *planets = nullptr,
                                             int64_t pstride = 0)
{
    const double h = A.h;
    double b6o[3] = {A.b[6][0], A.b[6][1], A.b[6][2]};
    double F7[3];
    // V32 (mixed precision, launches with node rows): without non-gravitational
    // terms the node velocity feeds only FP32 terms, so it is predicted in FP32
    // from A.bf (kept only in these launches: the extra registers cost the
    // per-thread-ephemeris launches more than the FP64 work they save)
    const bool vel32 = (MODE == KETE_MIXED) && V32 && !ng;
    float v0f[3], a0f[3];
    if (MODE == KETE_MIXED) {
#pragma unroll
        for (int i = 0; i < 3; i++) A.gs7[i] = g_rt.w7[0] * as0[i];
        if (vel32) {
#pragma unroll
            for (int i = 0; i < 3; i++) {
                v0f[i] = (float)v0[i];
                a0f[i] = (float)a0[i];
            }
        }
    }
    // one copy of the force evaluation: the node index is the same for every
    // lane of the sweep (uniform table reads, uniform guards below)
#pragma unroll 1
    for (int n = 1; n <= 7; n++) {
        const double s = g_rt.h[n];
        const double sh = s * h;
        double xn[3], vn[3], dxn[3];
        float vnf[3];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            // x(s) = x0 + s h v0 + (s h)^2 [a0/2 + sum_k b_k s^(k+1) / ((k+2)(k+3))]
            // v(s) = v0 + s h [a0 + sum_k b_k s^(k+1) / (k+2)]
            // with the node's weights from the table (smallest terms first)
            double px = A.b[6][i] * g_rt.wx[n][6];
#pragma unroll
            for (int k = 5; k >= 0; k--) px = fma(A.b[k][i], g_rt.wx[n][k], px);
            px = fma(a0[i], 0.5, px);
            dxn[i] = fma(sh * sh, px, sh * v0[i]);   // displacement since the step start
            xn[i] = x0[i] + dxn[i];
            if (vel32) {
                float pv = A.bf[6][i] * g_rt.wvf[n][6];
#pragma unroll
                for (int k = 5; k >= 0; k--) pv = fmaf(A.bf[k][i], g_rt.wvf[n][k], pv);
                vnf[i] = fmaf((float)sh, pv + a0f[i], v0f[i]);
                vn[i] = 0.0;
            } else {
                double pv = A.b[6][i] * g_rt.wv[n][6];
#pragma unroll
                for (int k = 5; k >= 0; k--) pv = fma(A.b[k][i], g_rt.wv[n][k], pv);
                pv = pv + a0[i];
                vn[i] = fma(sh, pv, v0[i]);
            }
        }
        double Fn[3], Fs[3];
        const double *r64 = A.rows.r64 ? A.rows.r64 + n * A.rows.stride : nullptr;
        const float *r32 = A.rows.r32 ? A.rows.r32 + n * A.rows.stride : nullptr;
        PlanetCache cache = {nullptr, pstride, A.it == 0};
        if (planets) cache.p = planets + (int64_t)(n - 1) * E.n_bodies * 6 * pstride;
        int st = accel<MODE, JAC>(E, F, t, sh, r64, r32, close, xn, vn, Fn, Fs, enc, dxn,
                                     false, JAC ? jrec + 6 * n : nullptr, ng,
                                     vel32 ? vnf : nullptr, ng_chi, nullptr, cache);
        cnt.evals++;
        if (r64) cnt.node_evals++;
        if (st != KETE_BODY_OK) return st;
        switch (n) {
        case 1: node_update<MODE, 1, V32>(A, Fn, Fs, a0, F7); break;
        case 2: node_update<MODE, 2, V32>(A, Fn, Fs, a0, F7); break;
        case 3: node_update<MODE, 3, V32>(A, Fn, Fs, a0, F7); break;
        case 4: node_update<MODE, 4, V32>(A, Fn, Fs, a0, F7); break;
        case 5: node_update<MODE, 5, V32>(A, Fn, Fs, a0, F7); break;
        case 6: node_update<MODE, 6, V32>(A, Fn, Fs, a0, F7); break;
        default: node_update<MODE, 7, V32>(A, Fn, Fs, a0, F7); break;
        }
    }
    cnt.iters++;
    A.it++;
    double db = 0.0, amax = 0.0;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        db = fmax(db, fabs(A.b[6][i] - b6o[i]));
        amax = fmax(amax, fabs(F7[i]));
    }
    A.amax = amax;
    const double pc = db / amax;
    if (!isfinite(pc)) return KETE_BODY_NONFINITE;
    // (a continued polynomial's b6 can agree by chance in the first sweep)
    done = (pc < F.eps_pc && (JAC || MODE == KETE_MIXED || A.it >= 2)) || (A.it >= 3 && pc >= A.pc_prev) ||
           (A.it >= F.max_iter);
    A.pc_prev = pc;
    return KETE_BODY_OK;
}

// The attempt's end state and its IAS15 error estimate max|b6| / max|a| (in
// mixed precision b6 of the smooth FP64 part: FP32 rounding is not smooth and
// b6 would amplify it).
template <int MODE>
__device__ __forceinline__ int attempt_end(const Attempt &A, const double x0[3], const double v0[3],
                                           const double a0[3], double x1[3], double v1[3],
                                           double &err)
{
    const double h = A.h;
    double bmax = (MODE == KETE_MIXED)
                      ? fmax(fabs(A.gs7[0]), fmax(fabs(A.gs7[1]), fabs(A.gs7[2])))
                      : fmax(fabs(A.b[6][0]), fmax(fabs(A.b[6][1]), fabs(A.b[6][2])));
    err = bmax / A.amax;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double px = fma(A.b[6][i], 1.0 / 72.0, A.b[5][i] * (1.0 / 56.0));
        px = fma(A.b[4][i], 1.0 / 42.0, px);
        px = fma(A.b[3][i], 1.0 / 30.0, px);
        px = fma(A.b[2][i], 1.0 / 20.0, px);
        px = fma(A.b[1][i], 1.0 / 12.0, px);
        px = fma(A.b[0][i], 1.0 / 6.0, px);
        px = fma(a0[i], 0.5, px);
        double pv = fma(A.b[6][i], 0.125, A.b[5][i] * (1.0 / 7.0));
        pv = fma(A.b[4][i], 1.0 / 6.0, pv);
        pv = fma(A.b[3][i], 0.2, pv);
        pv = fma(A.b[2][i], 0.25, pv);
        pv = fma(A.b[1][i], 1.0 / 3.0, pv);
        pv = fma(A.b[0][i], 0.5, pv);
        pv = pv + a0[i];
        x1[i] = fma(h * h, px, fma(h, v0[i], x0[i]));
        v1[i] = fma(h, pv, v0[i]);
    }
    if (!(isfinite(x1[0]) && isfinite(x1[1]) && isfinite(x1[2]) && isfinite(v1[0]) &&
          isfinite(v1[1]) && isfinite(v1[2])))
        return KETE_BODY_NONFINITE;
    return KETE_BODY_OK;
}

// Per-body integrator state between step attempts.
struct StepState {
    double a0[3], as0[3];   // acceleration at the step start (and its FP64 part)
    uint32_t close;         // planets near the body at the step start (mixed precision)
    Encounter enc;          // nearest planet within kEncounterAu (close-encounter path)
    double bound;           // epoch no step may pass: the next table segment boundary
                            // during an encounter, else infinite
    int start;              // what the next attempt's corrector starts from (CorrectorStart)
    bool chained;           // the Attempt holds an accepted step that ended here, and the
                            // next one is proposed within kNextMost times its length
    bool have_a0;           // a0 valid for (x, v, t): kept across a rejection
    const kete_nongrav *ng; // the body's non-gravitational terms (null: none)
    double ng_chi;          // the thermal lag's last two-body solution (0: none yet)
};

// The first three time derivatives of the acceleration of two-body motion at
// heliocentric (r, w): r^(k) = A_k r + B_k w with u = mu / r^3, p = r.w / r^2,
// q = w.w / r^2 (u' = -3 u p, p' = q - u - 2 p^2, q' = -2 p (u + q)):
//   A_3 = 3 u p,                     B_3 = -u,
//   A_4 = u (3 q - 15 p^2 - 2 u),     B_4 = 6 u p,
//   A_5 = u p (105 p^2 - 45 q + 30 u), B_5 = u (9 q - 45 p^2 - 8 u).
// They start a step's corrector: from the constant a0 the first sweep's nodes
// are off by ~(n h)^3 of a, with these by what the planets change over the
// step, for ~60 operations against a sweep's ~2,700 (main belt: 3.7 sweeps a
// step without, 3.0 with them at a ten times tighter threshold).  Used where no
// step of like length went before (START_NEXT) and in mixed precision.
__device__ __forceinline__ void two_body_derivs(double mu, const double r[3], const double w[3],
                                                double d1[3], double d2[3], double d3[3])
{
    const double rr = fma(r[0], r[0], fma(r[1], r[1], r[2] * r[2]));
    const double ri = rsqrt(rr), ri2 = ri * ri;
    const double u = mu * ri2 * ri;
    const double p = fma(r[0], w[0], fma(r[1], w[1], r[2] * w[2])) * ri2;
    const double q = fma(w[0], w[0], fma(w[1], w[1], w[2] * w[2])) * ri2;
    const double pp = p * p, up = u * p;
    const double a3 = 3.0 * up, b4 = 6.0 * up;
    const double a4 = u * fma(3.0, q, fma(-15.0, pp, -2.0 * u));
    const double a5 = up * fma(105.0, pp, fma(-45.0, q, 30.0 * u));
    const double b5 = u * fma(9.0, q, fma(-45.0, pp, -8.0 * u));
#pragma unroll
    for (int i = 0; i < 3; i++) {
        d1[i] = fma(a3, r[i], -u * w[i]);
        d2[i] = fma(a4, r[i], b4 * w[i]);
        d3[i] = fma(a5, r[i], b5 * w[i]);
    }
}

// The acceleration at the start of a step attempt of (x, v, t) if it is not
// known yet (kept across a rejection), from node-0 rows when given,
// what its corrector starts from (S.start; the derivatives in A.b), and the
// epoch no step toward `dir` may pass: during an encounter no step straddles
// a boundary of the planet polynomials (S.bound; infinite otherwise).
template <int MODE, bool JAC>
__device__ __forceinline__ int step_start(const EphemDev &E, const ForceDev &F, const double *r64,
                                          const float *r32, const double x[3], const double v[3],
                                          double t, bool forward, StepState &S, Attempt &A,
                                          Cnt &cnt, double *jrec)
{
    if (S.have_a0) {
        S.start = JAC ? START_A0 : S.start;
        return KETE_BODY_OK;
    }
    const double zero[3] = {0.0, 0.0, 0.0};
    double helio[6];
    int st = accel<MODE, JAC>(E, F, t, 0.0, r64, r32, S.close, x, v, S.a0, S.as0, S.enc, zero,
                              true, jrec, S.ng, nullptr, &S.ng_chi, helio);
    cnt.evals++;
    if (r64) cnt.node_evals++;
    if (st != KETE_BODY_OK) return st;
    S.bound = forward ? __longlong_as_double(0x7ff0000000000000ll)
                      : __longlong_as_double(0xfff0000000000000ll);
    if (S.enc.m >= 0) {
        const double k = floor((t - E.t_start) * E.inv_seg);
        double b = forward ? E.t_start + (k + 1.0) * E.seg_len : E.t_start + k * E.seg_len;
        if (!forward && b == t) b = E.t_start + (k - 1.0) * E.seg_len;
        S.bound = b;
    }
    S.start = START_A0;
    if (!JAC && MODE == KETE_FP64 && S.chained) {
        S.start = START_NEXT;
    } else if (!JAC && (F.active_mask & 1u)) {
        S.start = START_DERIVS;
        two_body_derivs(E.gm[0], helio, helio + 3, A.b[0], A.b[1], A.b[2]);
    }
    S.have_a0 = true;
    return KETE_BODY_OK;
}

// Begin the attempt of size dt, clamped at `target` (or the encounter's
// boundary when that is nearer), planets per thread.
__device__ __forceinline__ int step_aim(double t, double dt, double target, const StepState &S,
                                        Attempt &A)
{
    double t_stop = target;
    if ((target > t && S.bound < target) || (target < t && S.bound > target)) t_stop = S.bound;
    const bool clamped = fabs(dt) >= fabs(t_stop - t);
    // the step is the exact difference of the representable epochs it joins
    const double t_new = clamped ? t_stop : t + dt;
    const double h = t_new - t;
    if (h == 0.0) return KETE_BODY_STEP_CAP;   // step below the epoch resolution
    attempt_begin(A, h, t_new, StepRows{nullptr, nullptr, 0}, S.start);
    return KETE_BODY_OK;
}

// Start a step attempt of (x, v, t) toward `target` (t != target): the
// acceleration at the step start, the step size, the corrector state A.
// Returns a KETE_BODY_* status.  JAC: as attempt_sweep (jrec[0..5] at t).
template <int MODE, bool JAC = false>
__device__ __forceinline__ int step_begin(const EphemDev &E, const ForceDev &F, const double x[3],
                                          const double v[3], double t, double dt, double target,
                                          StepState &S, Attempt &A, Cnt &cnt,
                                          double *jrec = nullptr)
{
    const int st = step_start<MODE, JAC>(E, F, nullptr, nullptr, x, v, t, target > t, S, A,
                                            cnt, jrec);
    return st != KETE_BODY_OK ? st : step_aim(t, dt, target, S, A);
}

// Index of the first grid point at or past t in the grid's direction.
__device__ __forceinline__ int grid_locate(const GridDev &Q, double t)
{
    int lo = 0, hi = Q.J;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const double g = __ldg(Q.g + mid);
        if (Q.dir > 0 ? g >= t : g <= t) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// As step_begin for a body that follows the grid Q (j: the grid point it
// stands on or the next one): from a grid point the longest tabulated step
// that does not exceed the proposed dt, its planets read from the rows; off the
// grid a step up to the next grid point, and with a proposal below one unit a
// step of dt, the planets summed per thread.  jn: the first grid point at or
// past the step's end.
template <int MODE>
__device__ __forceinline__ int step_begin_grid(const EphemDev &E, const ForceDev &F,
                                               const GridDev &Q, int j, int &jn,
                                               const double x[3], const double v[3], double t,
                                               double dt, StepState &S, Attempt &A, Cnt &cnt)
{
    const bool on = t == __ldg(Q.g + j);
    const int stride = Q.nb * 6;
    const size_t cell = (size_t)8 * stride;
    const bool row0 = on && j < Q.J && __ldg(Q.ok + (size_t)j * Q.n_len);
    const size_t at0 = (size_t)j * Q.n_len * cell;
    const int st = step_start<MODE, false>(E, F, row0 ? Q.row64 + at0 : nullptr,
                                              row0 ? Q.row32 + at0 : nullptr, x, v, t, Q.dir > 0, S, A,
                                              cnt, nullptr);
    if (st != KETE_BODY_OK) return st;
    if (on) {
        const double units = fabs(dt) * Q.inv_unit * (1.0 + 1e-12);
        const int most = units < (double)(Q.J - j) ? (int)units : Q.J - j;
        int best = -1;
        for (int q = 0; q < Q.n_len; q++) {
            const int len = Q.len[q];
            if (len > most) break;
            const double t_new = __ldg(Q.g + j + len);
            if (Q.dir > 0 ? t_new > S.bound : t_new < S.bound) break;
            if (__ldg(Q.ok + (size_t)j * Q.n_len + q)) best = q;
        }
        if (best >= 0) {
            jn = j + Q.len[best];
            const double t_new = __ldg(Q.g + jn);
            const size_t at = ((size_t)j * Q.n_len + best) * cell;
            attempt_begin(A, t_new - t, t_new, StepRows{Q.row64 + at, Q.row32 + at, stride}, S.start);
            return KETE_BODY_OK;
        }
    }
    // (at the grid's end with stops past it: a step of length zero, which the
    // caller answers with plain steps)
    jn = on && j < Q.J ? j + 1 : j;
    if (fabs(dt) * Q.inv_unit >= 1.0) return step_aim(t, dt, __ldg(Q.g + jn), S, A);
    // (a grid of single-unit legs: no step passes one)
    const int st2 = step_aim(t, dt, __ldg(Q.g + (Q.n_len == 1 ? jn : Q.J)), S, A);
    while (jn < Q.J && (Q.dir > 0 ? __ldg(Q.g + jn) < A.t_new : __ldg(Q.g + jn) > A.t_new)) jn++;
    return st2;
}

// The body's state at epoch ts inside the attempt A from (t, x0, v0, a0): the
// collocation polynomial of the corrector (the node predictor's sums at
// s = (ts - t) / h instead of a node).  The polynomial interpolates the
// acceleration through the 8 nodes; with b6 / |a| held near 1e-9 by the step
// control its interpolation error, times h^2 |a|, stays orders of magnitude
// below the rounding of the position.
__device__ __forceinline__ void attempt_dense(const Attempt &A, double t, const double x0[3],
                                              const double v0[3], const double a0[3], double ts,
                                              double xs[3], double vs[3])
{
    const double sh = ts - t;
    const double s = sh / A.h;
    double wx[7], wv[7], sp = s;
    constexpr double cx[7] = {1.0 / 6.0,  1.0 / 12.0, 1.0 / 20.0, 1.0 / 30.0,
                              1.0 / 42.0, 1.0 / 56.0, 1.0 / 72.0};
    constexpr double cv[7] = {1.0 / 2.0, 1.0 / 3.0, 1.0 / 4.0, 1.0 / 5.0,
                              1.0 / 6.0, 1.0 / 7.0, 1.0 / 8.0};
#pragma unroll
    for (int k = 0; k < 7; k++) {
        wx[k] = sp * cx[k];
        wv[k] = sp * cv[k];
        sp *= s;
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double px = A.b[6][i] * wx[6], pv = A.b[6][i] * wv[6];
#pragma unroll
        for (int k = 5; k >= 0; k--) {
            px = fma(A.b[k][i], wx[k], px);
            pv = fma(A.b[k][i], wv[k], pv);
        }
        px = fma(a0[i], 0.5, px);
        xs[i] = x0[i] + fma(sh * sh, px, sh * v0[i]);
        vs[i] = fma(sh, pv + a0[i], v0[i]);
    }
}

// The adjoint's forward pass (JAC) keeps the constant start and the FP64 step
// factor: its loss is made of residuals ~1e-7 of the predicted angles, so a
// step sequence that differs in the last bits moves a gradient by up to 1e-9 of
// itself, and nothing but those bits is to be gained.
//
// IAS15's step factor (eps / err)^(1/7), at most 1 / safety (also for an err
// of zero or none).  The power in FP32: a step proposal needs no more than its
// 1e-7, and the FP64 pow cost as much issue time as a force evaluation.
template <bool JAC = false>
__device__ __forceinline__ double step_factor(const ForceDev &F, double err)
{
    const double most = 1.0 / F.safety;
    if (JAC) {
        if (isfinite(err) && err >= 2.2250738585072014e-308) return pow(F.eps / err, 1.0 / 7.0);
        return most;
    }
    if (!(isfinite(err) && err > 1e-37)) return most;
    const float e = (float)fmin(err, 1e37);
    return fmin((double)exp2f((F.log2_eps - log2f(e)) * (1.0f / 7.0f)), most);
}

// End a step attempt whose corrector is done: IAS15 step control.  Accepted:
// (x1, v1) is the state at the step end and dt holds the next proposal.
// Rejected: dt shrinks and a0 is kept.  Returns a KETE_BODY_* status.
template <int MODE, bool JAC = false>
__device__ __forceinline__ int step_control(const ForceDev &F, const Attempt &A, const double x[3],
                                            const double v[3], double &dt, const StepState &S,
                                            Cnt &cnt, double x1[3], double v1[3], bool &accepted)
{
    double err;
    accepted = false;
    int st = attempt_end<MODE>(A, x, v, S.a0, x1, v1, err);
    if (st != KETE_BODY_OK) return st;
    const double h = A.h;
    const double factor = step_factor<JAC>(F, err);
    dt = factor * h;
    if (fabs(dt / h) < F.safety) {   // reject: retry from the same a0
        cnt.rejected++;
        return KETE_BODY_OK;
    }
    if (JAC && fabs(dt / h) > 1.0 / F.safety) dt = h / F.safety;
    accepted = true;
    cnt.steps++;
    return KETE_BODY_OK;
}

// step_control, and the state advanced when the step was accepted
template <int MODE, bool JAC = false>
__device__ __forceinline__ int step_end(const ForceDev &F, const Attempt &A, double x[3],
                                        double v[3], double &t, double &dt, StepState &S, Cnt &cnt)
{
    double x1[3], v1[3];
    bool accepted;
    const int st = step_control<MODE, JAC>(F, A, x, v, dt, S, cnt, x1, v1, accepted);
    if (st != KETE_BODY_OK || !accepted) return st;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        x[i] = x1[i];
        v[i] = v1[i];
    }
    t = A.t_new;
    S.have_a0 = false;
    return KETE_BODY_OK;
}

// orient the carried step toward the next stop (|dt| kept; dt_init to start)
__device__ __forceinline__ void aim_step(const ForceDev &F, double t, double target, double &dt)
{
    const double dir = (target >= t) ? 1.0 : -1.0;
    if (dt == 0.0 || ((dt > 0.0) != (dir > 0.0))) dt = dir * fabs(dt == 0.0 ? F.dt_init : dt);
}

// warp sums of the lanes' counters into ctr
__device__ __forceinline__ void flush_counters(const Cnt &c, DevCounters *ctr)
{
    unsigned long long s = c.steps, r = c.rejected, e = c.evals, it = c.iters, ne = c.node_evals;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        r += __shfl_xor_sync(0xffffffffu, r, o);
        e += __shfl_xor_sync(0xffffffffu, e, o);
        it += __shfl_xor_sync(0xffffffffu, it, o);
        ne += __shfl_xor_sync(0xffffffffu, ne, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&ctr->steps, s);
        atomicAdd(&ctr->rejected, r);
        atomicAdd(&ctr->force_evals, e);
        atomicAdd(&ctr->iterations, it);
        atomicAdd(&ctr->node_evals, ne);
    }
}


}  // namespace kete
