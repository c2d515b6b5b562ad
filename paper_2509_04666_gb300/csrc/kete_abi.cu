// kete_abi.cu -- the C ABI of libkete_gpu.so (declared in include/kete.h).
//
// Host orchestration only: argument checks, device scratch, launch order on
// the context stream, the few host reads the survey driver needs (exposure and
// batch counts, candidate and hit counts per chunk of batches).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "kete_adjoint.h"
#include "kete_fov.h"
#include "kete_impl.h"
#include "kete_order.h"

using namespace kete;

namespace {

enum Slot {
    S_CHAIN, S_STATUS, S_STOPS, S_STOPSTATES, S_ISSTART, S_EX, S_SCANTMP, S_FCEN, S_FAUX,
    S_EXPFIRST, S_XEPOCH, S_XOBS, S_XCEN, S_XCENF, S_XRAD, S_XCS, S_XBATCH, S_NEXT, S_BFIRST, S_BTREF,
    S_BO, S_BROBS, S_BTSPAN, S_BRMAX, S_BSUN, S_NBATCH, S_BANDS, S_CELLKEY, S_CELLCNT,
    S_CELLSTART, S_CELLCUR, S_CELLEXP, S_CAND, S_EXPCNT, S_EXPOFF, S_EXPCUR, S_CANDBODY,
    S_HITTMP, S_FRAMECNT, S_FRAMEOFF, S_FRAMECUR, S_HITGROUP, S_MAXRAD, S_GRID, S_GRID_OK,
    S_GRID_R64, S_GRID_R32, S_STOPROW, S_XSUN, S_XOBSREL, S_NEXTBODY, S_TUNE_ST, S_TUNE_EP, S_TUNE_OUT,
    S_ADJ_REC, S_ADJ_NREC, S_ADJ_NBAT, S_ADJ_BIDX, S_ADJ_YREF, S_ADJ_GJUMP, S_ADJ_STATUS,
    S_KSTOP, S_TRIES, S_DEFER_LIST, S_DEFER_CNT, S_ORDER, S_ORDER_KEY, S_ORDER_HIST, S_ORDER_OFF,
    S_ORDER_SCAN, S_ORDER_N, S_ADJ_TEND,
    S_EXT_START, S_EXT_EX, S_EXT_TMP, S_EXT_FIRST, S_EXT_SUB, S_EXT_PARENT, S_EXT_CNT,
    S_EXT_OFF, S_EXT_CUR, S_EXT_GROUP, S_EXT_KEEP, S_EXT_KCNT, S_EXT_KOFF, S_ADJ_PHI, S_ADJ_RECX,
    S_PRE_KEEP, S_PRE_N, S_ADJ_RICH, S_ADJ_PLANETS, S_ADJ_BFRAC, S_ADJ_MID, S_ADJ_RANGE,
    S_NSLOTS
};

struct Scratch {
    void *p = nullptr;
    size_t bytes = 0;
};

}  // namespace

struct kete_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::string err;
    bool have_ephem = false;
    double *d_coef = nullptr;
    float *d_coef32 = nullptr;
    EphemDev E{};
    Scratch slot[S_NSLOTS];
    DevCounters *d_ctr = nullptr;
    DevCounters *h_ctr = nullptr;   // pinned
    kete_stats stats{};
    std::vector<cudaEvent_t> ev;    // pool: [0] start, [1] end, then pairs for propagation
    int n_sm = 152;
    int pending_prop_pairs = 0;
    int64_t extra_launches = 0;     // ordering and second-phase launches of this call
    std::vector<std::shared_ptr<const void>> uploads;   // host arrays that copies in flight read
    // phase timers: pairs of events per phase (prep, candidates, exact, order)
    std::vector<cudaEvent_t> phase_ev[4];
    int phase_n[4] = {0, 0, 0, 0};
    PropVariant var[2] = {{PROP_WORK_STEALING, 128, 0, 0, 1},
                          {PROP_WORK_STEALING, 128, 0, 0, 1}};   // per precision
};

enum Phase { PH_PREP = 0, PH_CAND = 1, PH_EXACT = 2, PH_ORDER = 3 };

static void phase_mark(kete_ctx *ctx, int ph, bool begin)
{
    size_t idx = 2 * (size_t)ctx->phase_n[ph] + (begin ? 0 : 1);
    auto &v = ctx->phase_ev[ph];
    while (v.size() <= idx) {
        cudaEvent_t e;
        cudaEventCreate(&e);
        v.push_back(e);
    }
    cudaEventRecord(v[idx], ctx->stream);
    if (!begin) ctx->phase_n[ph]++;
}

static int fail(kete_ctx *c, int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    if (c) c->err = buf;
    return code;
}

#define CUDA_TRY(x)                                                                       \
    do {                                                                                  \
        cudaError_t _e = (x);                                                             \
        if (_e != cudaSuccess)                                                            \
            return fail(ctx, KETE_ERR_CUDA, "%s failed: %s", #x, cudaGetErrorString(_e)); \
    } while (0)

static cudaError_t ensure(kete_ctx *ctx, int s, size_t bytes, void **out)
{
    Scratch &b = ctx->slot[s];
    if (bytes == 0) bytes = 16;
    if (b.bytes < bytes) {
        if (b.p) {
            cudaError_t e = cudaStreamSynchronize(ctx->stream);
            if (e != cudaSuccess) return e;
            cudaFree(b.p);
            b.p = nullptr;
            b.bytes = 0;
        }
        size_t want = bytes + bytes / 4;
        cudaError_t e = cudaMalloc(&b.p, want);
        if (e != cudaSuccess) {
            cudaGetLastError();
            e = cudaMalloc(&b.p, bytes);
            if (e != cudaSuccess) return e;
            want = bytes;
        }
        b.bytes = want;
    }
    *out = b.p;
    return cudaSuccess;
}

template <typename T>
static int get(kete_ctx *ctx, int s, size_t count, T **out)
{
    void *p = nullptr;
    cudaError_t e = ensure(ctx, s, count * sizeof(T), &p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(ctx, KETE_ERR_NOMEM, "device allocation of %zu bytes failed: %s",
                    count * sizeof(T), cudaGetErrorString(e));
    }
    *out = (T *)p;
    return KETE_OK;
}

#define GET(slot, n, ptr)                                  \
    do {                                                   \
        int _r = get(ctx, slot, (size_t)(n), &(ptr));      \
        if (_r != KETE_OK) return _r;                      \
    } while (0)

// Copy a host array to the device.  A copy from pageable memory may read it as
// late as the stream gets to it (where the GPU reads host memory through the
// host's page tables nothing is staged), so the context keeps it until it has
// synchronised the stream.
template <typename T>
static cudaError_t upload(kete_ctx *ctx, T *dst, std::shared_ptr<const std::vector<T>> src)
{
    const cudaError_t e = cudaMemcpyAsync(dst, src->data(), src->size() * sizeof(T),
                                          cudaMemcpyHostToDevice, ctx->stream);
    ctx->uploads.push_back(std::move(src));
    return e;
}

static cudaEvent_t event_at(kete_ctx *ctx, size_t i)
{
    while (ctx->ev.size() <= i) {
        cudaEvent_t e;
        cudaEventCreate(&e);
        ctx->ev.push_back(e);
    }
    return ctx->ev[i];
}

static void stats_begin(kete_ctx *ctx)
{
    if (!ctx->uploads.empty()) {   // left by a call that failed
        cudaStreamSynchronize(ctx->stream);
        ctx->uploads.clear();
    }
    std::memset(&ctx->stats, 0, sizeof(ctx->stats));
    ctx->pending_prop_pairs = 0;
    ctx->extra_launches = 0;
    for (int q = 0; q < 4; q++) ctx->phase_n[q] = 0;
    cudaMemsetAsync(ctx->d_ctr, 0, sizeof(DevCounters), ctx->stream);
    cudaEventRecord(event_at(ctx, 0), ctx->stream);
}

static void prop_event(kete_ctx *ctx, bool begin)
{
    size_t idx = 2 + 2 * (size_t)ctx->pending_prop_pairs + (begin ? 0 : 1);
    cudaEventRecord(event_at(ctx, idx), ctx->stream);
    if (!begin) ctx->pending_prop_pairs++;
}

static int stats_end(kete_ctx *ctx)
{
    cudaEventRecord(event_at(ctx, 1), ctx->stream);
    CUDA_TRY(cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost,
                             ctx->stream));
    return KETE_OK;
}

static void stats_collect(kete_ctx *ctx)
{
    cudaStreamSynchronize(ctx->stream);
    ctx->uploads.clear();
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, ctx->ev[0], ctx->ev[1]);
    ctx->stats.total_ms = ms;
    double p = 0.0;
    for (int k = 0; k < ctx->pending_prop_pairs; k++) {
        float m = 0.0f;
        cudaEventElapsedTime(&m, ctx->ev[2 + 2 * k], ctx->ev[3 + 2 * k]);
        p += m;
    }
    ctx->stats.prop_ms = p;
    ctx->stats.fov_ms = ctx->stats.total_ms - p;
    ctx->stats.steps = (int64_t)ctx->h_ctr->steps;
    ctx->stats.rejected = (int64_t)ctx->h_ctr->rejected;
    ctx->stats.force_evals = (int64_t)ctx->h_ctr->force_evals;
    ctx->stats.iterations = (int64_t)ctx->h_ctr->iterations;
    ctx->stats.node_evals = (int64_t)ctx->h_ctr->node_evals;
    ctx->stats.deferred = (int64_t)ctx->h_ctr->deferred;
    ctx->stats.prop_launches = ctx->pending_prop_pairs;
    ctx->stats.launches += ctx->extra_launches;
    ctx->pending_prop_pairs = 0;
    double *dst[4] = {&ctx->stats.prep_ms, &ctx->stats.cand_ms, &ctx->stats.exact_ms,
                      &ctx->stats.order_ms};
    for (int q = 0; q < 4; q++) {
        double acc = 0.0;
        for (int k = 0; k < ctx->phase_n[q]; k++) {
            float m = 0.0f;
            cudaEventElapsedTime(&m, ctx->phase_ev[q][2 * k], ctx->phase_ev[q][2 * k + 1]);
            acc += m;
        }
        *dst[q] = acc;
        ctx->phase_n[q] = 0;
    }
}

extern "C" {

void kete_force_model_default(kete_force_model *fm)
{
    if (!fm) return;
    std::memset(fm, 0, sizeof(*fm));
    const double deg = 3.14159265358979323846 / 180.0;
    const double au = 149597870.7;
    fm->body_mask = 0x1FFu;
    fm->gr_mask = (1u << 0) | (1u << 3) | (1u << 5);   // Sun, Earth, Jupiter (App. A.2)
    fm->j2_mask = (1u << 0) | (1u << 5);               // Sun, Jupiter (App. A.3)
    fm->precision = KETE_FP64;
    fm->j2[0] = 2.1961e-7;
    fm->radius[0] = 696000.0 / au;
    fm->pole_ra[0] = 286.13 * deg;
    fm->pole_dec[0] = 63.87 * deg;
    fm->j2[5] = 0.014736;
    fm->radius[5] = 71492.0 / au;
    fm->pole_ra[5] = 268.056595 * deg;
    fm->pole_dec[5] = 64.495303 * deg;
    fm->eps = 1e-9;
    fm->eps_pc = 1e-10;
    fm->safety = 0.25;
    fm->dt_init = 4.0;
    fm->max_iter = 12;
    fm->max_steps = 100000;
}

void kete_survey_opts_default(kete_survey_opts *opt)
{
    if (!opt) return;
    opt->batch_span = 3.0;
    opt->twobody_max = 1.5;
    opt->cell_deg = 0.0;
    opt->mem_budget_gb = 0.0;
}

int kete_create(kete_ctx **out, int device, void *cuda_stream)
{
    if (!out) return KETE_ERR_BAD_ARG;
    *out = nullptr;
    kete_ctx *ctx = new kete_ctx();
    ctx->device = device;
    ctx->stream = (cudaStream_t)cuda_stream;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->d_ctr, sizeof(DevCounters));
    if (e == cudaSuccess) e = cudaMallocHost(&ctx->h_ctr, sizeof(DevCounters));
    if (e != cudaSuccess) {
        delete ctx;
        return KETE_ERR_CUDA;
    }
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) == cudaSuccess && sms > 0)
        ctx->n_sm = sms;
    std::memset(ctx->h_ctr, 0, sizeof(DevCounters));
    upload_radau_tables(ctx->stream);
    e = upload_adjoint_tables(ctx->stream);
    if (e == cudaSuccess) e = upload_warp_tables(ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) {
        kete_destroy(ctx);
        return KETE_ERR_CUDA;
    }
    *out = ctx;
    return KETE_OK;
}

void kete_destroy(kete_ctx *ctx)
{
    if (!ctx) return;
    cudaSetDevice(ctx->device);
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    else cudaDeviceSynchronize();
    for (auto &s : ctx->slot)
        if (s.p) cudaFree(s.p);
    if (ctx->d_coef) cudaFree(ctx->d_coef);
    if (ctx->d_coef32) cudaFree(ctx->d_coef32);
    if (ctx->d_ctr) cudaFree(ctx->d_ctr);
    if (ctx->h_ctr) cudaFreeHost(ctx->h_ctr);
    for (auto e : ctx->ev) cudaEventDestroy(e);
    for (auto &v : ctx->phase_ev)
        for (auto e : v) cudaEventDestroy(e);
    delete ctx;
}

int kete_set_stream(kete_ctx *ctx, void *cuda_stream)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    ctx->stream = (cudaStream_t)cuda_stream;
    return KETE_OK;
}

const char *kete_last_error(const kete_ctx *ctx) { return ctx ? ctx->err.c_str() : "null context"; }

int kete_get_stats(const kete_ctx *ctx, kete_stats *out)
{
    if (!ctx || !out) return KETE_ERR_BAD_ARG;
    *out = ctx->stats;
    return KETE_OK;
}

int kete_load_ephem(kete_ctx *ctx, const void *buf, size_t nbytes)
{
    if (!ctx || !buf) return fail(ctx, KETE_ERR_BAD_ARG, "null context or buffer");
    const unsigned char *p = (const unsigned char *)buf;
    if (nbytes < 256 || std::memcmp(p, "KETECHB1", 8) != 0)
        return fail(ctx, KETE_ERR_BAD_ARG, "not a KETECHB1 table");
    int32_t hdr[4];
    double td[2];
    std::memcpy(hdr, p + 8, sizeof(hdr));
    std::memcpy(td, p + 24, sizeof(td));
    if (hdr[0] != 1) return fail(ctx, KETE_ERR_BAD_ARG, "unsupported table version %d", hdr[0]);
    int nb = hdr[1], nc = hdr[2], ns = hdr[3];
    if (nb < 1 || nb > KETE_MAX_BODIES || nc < 2 || nc > 64 || ns < 1)
        return fail(ctx, KETE_ERR_BAD_ARG, "bad table sizes (bodies %d, coef %d, seg %d)", nb, nc, ns);
    if (!(td[1] > 0.0) || !std::isfinite(td[0]))
        return fail(ctx, KETE_ERR_BAD_ARG, "bad table span");
    size_t ncoef = (size_t)nb * ns * 3 * nc;
    if (nbytes < 256 + ncoef * sizeof(double))
        return fail(ctx, KETE_ERR_BAD_ARG, "table truncated: %zu bytes, need %zu", nbytes,
                    256 + ncoef * sizeof(double));
    CUDA_TRY(cudaSetDevice(ctx->device));
    if (ctx->d_coef) {
        cudaStreamSynchronize(ctx->stream);
        cudaFree(ctx->d_coef);
        cudaFree(ctx->d_coef32);
        ctx->d_coef = nullptr;
        ctx->d_coef32 = nullptr;
    }
    ctx->have_ephem = false;
    std::vector<float> f32(ncoef);
    const double *src = (const double *)(p + 256);
    std::vector<double> f64(src, src + ncoef);
    for (size_t i = 0; i < ncoef; i++) f32[i] = (float)f64[i];
    CUDA_TRY(cudaMalloc(&ctx->d_coef, ncoef * sizeof(double)));
    CUDA_TRY(cudaMalloc(&ctx->d_coef32, ncoef * sizeof(float)));
    CUDA_TRY(cudaMemcpyAsync(ctx->d_coef, f64.data(), ncoef * sizeof(double), cudaMemcpyHostToDevice, ctx->stream));
    CUDA_TRY(cudaMemcpyAsync(ctx->d_coef32, f32.data(), ncoef * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
    CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    EphemDev E{};
    E.coef = ctx->d_coef;
    E.coef32 = ctx->d_coef32;
    E.t_start = td[0];
    E.seg_len = td[1];
    E.inv_seg = 1.0 / td[1];
    E.t_end = td[0] + ns * td[1];
    E.n_seg = ns;
    E.n_coef = nc;
    E.n_bodies = nb;
    std::memcpy(E.gm, p + 48, sizeof(double) * KETE_MAX_BODIES);
    ctx->E = E;
    ctx->have_ephem = true;
    return KETE_OK;
}

}  // extern "C"

// The corrector starts from the two-body derivatives of a, so b6 settles
// before the rest of the polynomial does: its threshold is taken ten times
// tighter than from a constant start.  A chain of 20 stops over 60 days then
// ends 3e-17 AU rms from full convergence (3.5e-16 untightened, 9.5e-18 from the
// constant start, rounding 3.4e-16), and an orbit-fit gradient 2.5e-10 from its
// converged value (2.9e-9 and 3.1e-10), in 3.0 sweeps a step instead of 3.7.
constexpr double kStartTighter = 0.1;

static int make_force(kete_ctx *ctx, const kete_force_model *fm_in, ForceDev &F)
{
    kete_force_model fm;
    if (fm_in) fm = *fm_in;
    else kete_force_model_default(&fm);
    if (!(fm.eps > 0) || !(fm.safety > 0 && fm.safety < 1) || fm.max_iter < 1 || fm.max_iter > 100 ||
        fm.max_steps < 1 || !(fm.dt_init > 0) || !(fm.eps_pc >= 0))
        return fail(ctx, KETE_ERR_BAD_ARG, "invalid force-model controls");
    if (fm.precision != KETE_FP64 && fm.precision != KETE_MIXED)
        return fail(ctx, KETE_ERR_BAD_ARG, "unknown precision mode %d", fm.precision);
    std::memset(&F, 0, sizeof(F));
    const double eps_obl = 84381.448 / 3600.0 * 3.14159265358979323846 / 180.0;
    const double ce = std::cos(eps_obl), se = std::sin(eps_obl);
    uint32_t act = 0;
    for (int m = 0; m < ctx->E.n_bodies; m++)
        if (((fm.body_mask >> m) & 1u) && ctx->E.gm[m] != 0.0) act |= 1u << m;
    F.active_mask = act;
    F.gr_mask = fm.gr_mask & act;
    F.j2_mask = fm.j2_mask & act;
    F.precision = fm.precision;
    for (int m = 0; m < KETE_MAX_BODIES; m++) {
        F.j2k[m] = 1.5 * fm.j2[m] * ctx->E.gm[m] * fm.radius[m] * fm.radius[m];
        double ra = fm.pole_ra[m], de = fm.pole_dec[m];
        double ex = std::cos(de) * std::cos(ra), ey = std::cos(de) * std::sin(ra), ez = std::sin(de);
        F.pole[m][0] = ex;
        F.pole[m][1] = ce * ey + se * ez;
        F.pole[m][2] = -se * ey + ce * ez;
    }
    for (int m = 0; m < KETE_MAX_BODIES; m++) {
        const double gm = ctx->E.gm[m];
        F.gm4[m] = 4.0 * gm;
        F.grk[m] = gm * kInvC2;
        F.gr4k[m] = 4.0 * F.grk[m];
        for (int c = 0; c < 3; c++) F.pole_m2[m][c] = -2.0 * F.pole[m][c];
        F.gm32[m] = (float)gm;
        F.j2k32[m] = (float)F.j2k[m];
        for (int c = 0; c < 3; c++) F.pole32[m][c] = (float)F.pole[m][c];
        F.gm4_32[m] = (float)F.gm4[m];
        F.grk32[m] = (float)F.grk[m];
        F.gr4k32[m] = (float)F.gr4k[m];
        for (int c = 0; c < 3; c++) F.pole_m2_32[m][c] = (float)F.pole_m2[m][c];
    }
    F.eps = fm.eps;
    F.log2_eps = (float)std::log2(fm.eps);
    F.eps_pc = kStartTighter * fm.eps_pc;
    F.safety = fm.safety;
    F.dt_init = fm.dt_init;
    F.max_iter = fm.max_iter;
    F.max_steps = fm.max_steps;
    if (fm.nongrav && (reinterpret_cast<uintptr_t>(fm.nongrav) & 7u))
        return fail(ctx, KETE_ERR_BAD_ARG, "nongrav must be 8-byte aligned");
    F.nongrav = fm.nongrav;
    return KETE_OK;
}

extern "C" int kete_ephem_eval(kete_ctx *ctx, const double *t, int64_t n, int body, double *pos,
                               double *vel)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n < 0 || (n > 0 && (!t || !pos)) || body < 0 || body >= ctx->E.n_bodies)
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments");
    CUDA_TRY(cudaSetDevice(ctx->device));
    CUDA_TRY(launch_ephem_eval(ctx->E, t, n, body, pos, vel, ctx->stream));
    return KETE_OK;
}

// Bodies (states [6][stride] SoA, epochs [n], device) most expensive first
// over [epoch, end]: end = t_end, or t_end_i[i] (device) per body.  *order_n receives a device copy of n, the kernels'
// queue length.
static int cost_order(kete_ctx *ctx, const double *states, int64_t stride, const double *epochs,
                      int64_t n, double t_end, const double *t_end_i, const kete_nongrav *ng, int32_t **order, unsigned long long **order_n)
{
    OrderScratch s;
    const size_t nh = order_hist_elems(n);
    GET(S_ORDER, n, *order);
    GET(S_ORDER_KEY, n, s.key);
    GET(S_ORDER_HIST, nh, s.hist);
    GET(S_ORDER_OFF, nh + 1, s.off);
    GET(S_ORDER_SCAN, scan_tmp_elems((int64_t)nh), s.scan_tmp);
    GET(S_ORDER_N, 1, *order_n);
    CUDA_TRY(upload(ctx, *order_n, std::make_shared<const std::vector<unsigned long long>>(1, n)));
    CUDA_TRY(order_by_cost(ctx->E, states, stride, epochs, n, t_end, t_end_i, ng, s, *order,
                           ctx->stream));
    ctx->extra_launches += order_launches(n, ng);
    return KETE_OK;
}

// Whether a call takes one warp per body throughout.  A step takes a lane 0.4
// ms and the full lane grid 0.016 us, a warp 0.025 ms and the full grid of warps
// 0.06 us, and the lanes wait for their last warps.  Measured (ms, warps /
// lanes), catalogue bodies: 10 days 30,000 3.2 / 3.7, 60,000 6.0 / 4.2; 30 days
// 20,000 3.7 / 4.3, 30,000 5.7 / 4.7; 90 days 12,000 6.1 / 6.7, 20,000 8.5 / 7.3;
// a year 12,000 17.9 / 19.2, 20,000 25.6 / 19.4; mixed precision (lanes faster):
// 10 days 20,000 2.2 / 2.6, 30,000 3.2 / 2.9; a year 12,000 17.9 / 18.3.  The steps
// of a body are taken as 3 to start plus one in 14 days.
constexpr int64_t kWarpBodies = 13000;
static bool takes_warps(int64_t n, double span, bool mixed)
{
    const double steps = (double)n * (3.0 + std::fabs(span) / 14.0);
    return n <= (mixed ? 12000 : kWarpBodies) || steps <= (mixed ? 95e3 : 125e3);
}

// Bodies that need far more steps than the rest would set the time of a whole
// launch: past this many attempts they finish with one warp each (the main belt
// takes 24 steps a year).  The more bodies there are to a lane, and the slower
// lanes are, the longer lanes can go on with them.  Measured (ms), attempts a
// day beyond the first six: 250,000 mixed bodies over a year 0.3 158.0, 0.6
// 152.5; 30,011 over 120 days 0.05 8.5, 0.1 9.6, 0.3 15.5; mixed precision: 100,003
// over 180 days 0.05 58.2, 0.1 59.4, 0.3 73.6, 250,000 over 20 days 0.15 11.3, 0.6
// 12.8.  Below 0.075 main-belt bodies themselves are set aside.
static int attempts_budget(const kete_ctx *ctx, int64_t n, double span, bool mixed)
{
    const double load = (double)n / (512.0 * ctx->n_sm);
    const double per_day = std::min(mixed ? 0.4 : 0.6, std::max(0.075, (mixed ? 0.05 : 0.19) * load));
    return 6 + (int)std::min(1e6, std::fabs(span) * per_day);
}

// One propagation launch (and the set-aside bodies' second one) of the chain
// state along stops (device) with the context's variant for F's precision.
static int propagate_launch(kete_ctx *ctx, const ForceDev &F, ChainState cs, double t_start,
                            double t_end, const double *stops_dev, const int32_t *row, int n_stops,
                            double *out, int64_t stride, bool keep_on_fail, const GridDev *grid,
                            bool out_aos)
{
    PropVariant var = ctx->var[F.precision == KETE_MIXED ? 1 : 0];
    unsigned long long *next = nullptr;
    if (var.kind == PROP_WORK_STEALING) GET(S_NEXTBODY, 1, next);
    PropDefer defer{}, *dp = nullptr;
    // (not on a grid of single-unit legs: a set-aside body would step past them)
    if (!(grid && grid->n_len == 1 && grid->J > 1) && warp_model(ctx->E, F, defer.model)) {
        GET(S_DEFER_LIST, cs.n, defer.list);
        GET(S_DEFER_CNT, 1, defer.count);
        defer.budget0 = var.budget > 0 ? 0 : attempts_budget(ctx, var.population ? var.population : cs.n,
                                                             t_end - t_start, F.precision == KETE_MIXED);
        dp = &defer;
    }
    int32_t *order = nullptr;
    unsigned long long *order_n = nullptr;
    if (var.order) {
        int r = cost_order(ctx, cs.w, cs.n, cs.w + 6 * cs.n, cs.n, t_end, nullptr, F.nongrav,
                           &order, &order_n);
        if (r != KETE_OK) return r;
    }
    CUDA_TRY(launch_propagate(ctx->E, F, cs, stops_dev, row, n_stops, out, stride, keep_on_fail,
                              ctx->d_ctr, ctx->stream, grid, var, next, dp, order, order_n,
                              out_aos));
    if (dp) ctx->extra_launches += 1;   // the second phase
    return KETE_OK;
}

// Step lengths of a grid, in units of about a day: every whole number up to 16
// (the main belt's steps are 10-25 days, so rounding a proposal down costs a
// few per cent of it), then about 10-25 % apart.
static const int kGridLen[kGridLens] = {1,  2,  3,  4,  5,  6,  7,  8,  9,  10, 11, 12, 13,
                                        14, 15, 16, 18, 20, 22, 24, 28, 32, 40, 48, 64};
constexpr int kGridUnits = 512;   // units of one grid: 512 x 25 steps x 9 bodies are 66 MB of rows
constexpr double kGridMaxLaunches = 4096.0;   // grids of one call (5,700 years); longer spans take plain steps
// The grid of one launch: points pts[0..J] (host, monotonic).  single: steps
// of one unit only.
static int make_grid(kete_ctx *ctx, std::vector<double> &&points, double unit, bool single,
                     GridDev &Q)
{
    const auto shared = std::make_shared<const std::vector<double>>(std::move(points));
    const std::vector<double> &pts = *shared;
    const int J = (int)pts.size() - 1;
    Q = GridDev{};
    Q.J = J;
    Q.nb = ctx->E.n_bodies;
    Q.dir = pts[J] >= pts[0] ? 1 : -1;
    Q.inv_unit = 1.0 / unit;
    Q.n_len = 0;
    for (int q = 0; q < (single ? 1 : kGridLens) && kGridLen[q] <= J; q++)
        Q.len[Q.n_len++] = kGridLen[q];
    const size_t steps = (size_t)J * Q.n_len, elems = steps * 8 * Q.nb * 6;
    double *g, *r64;
    float *r32;
    uint8_t *ok;
    GET(S_GRID, J + 1, g);
    GET(S_GRID_R64, elems, r64);
    GET(S_GRID_R32, elems, r32);
    GET(S_GRID_OK, steps, ok);
    CUDA_TRY(upload(ctx, g, shared));
    Q.g = g;
    Q.row64 = r64;
    Q.row32 = r32;
    Q.ok = ok;
    CUDA_TRY(launch_grid_rows(ctx->E, Q, r64, r32, ok, ctx->stream));
    ctx->extra_launches += 1;
    return KETE_OK;
}

// Propagate the chain state along the stops (host), stop k to row k of out.
// t_from: the first body's epoch, or where an earlier call left the chain
// (NaN: not known).  use_grid: follow a step grid from t_from (from the first
// stop where t_from is not known or lies past it) in units of about a day;
// Marks (kMarkRow) between stops far apart cut the span into launches of at
// most kGridUnits units.  Grid and marks lie on the table: an epoch off it fails
// its own body.  leg_days > 0 (one stop, t_from known): stops that are not
// written every leg_days from t_from on, which are the grid's points.
static int propagate(kete_ctx *ctx, const ForceDev &F, ChainState cs, const double *stops,
                     int n_stops, double t_from, double *out, int64_t stride, bool keep_on_fail,
                     bool use_grid, double leg_days = 0.0, bool out_aos = false)
{
    std::vector<double> at(stops, stops + n_stops);
    std::vector<int32_t> row((size_t)n_stops);
    for (int k = 0; k < n_stops; k++) row[k] = k;
    double *d_stops;
    int32_t *d_row;
    const PropVariant &var = ctx->var[F.precision == KETE_MIXED ? 1 : 0];
    ctx->stats.prop_kind = var.kind;
    ctx->stats.prop_block = var.block;
    ctx->stats.prop_split = var.split;
    ctx->stats.prop_budget = var.budget;
    ctx->stats.prop_order = var.order;
    WarpModel model;
    const bool few = takes_warps(var.population ? var.population : cs.n, stops[n_stops - 1] - t_from, F.precision == KETE_MIXED) &&
                     var.budget == 0 && leg_days == 0.0 && F.max_iter >= 8 &&
                     warp_model(ctx->E, F, model);
    if (few) use_grid = false;
    const double unit = leg_days > 0.0 ? leg_days : 1.0;
    double start = t_from;
    const double last = stops[n_stops - 1];
    if (!std::isfinite(t_from) || (last > stops[0] && t_from > stops[0])) start = stops[0];
    const auto on_table = [&](double t) { return std::min(std::max(t, ctx->E.t_start), ctx->E.t_end); };
    if (leg_days == 0.0) start = on_table(start);
    const bool forward = last > start;
    if (last == start) use_grid = false;
    if (leg_days == 0.0) {
        // a target off the table fails every body; spans of millennia (and chains
        // with stops far off the table) would be cut into too many launches
        if (n_stops == 1 && !(last >= ctx->E.t_start && last <= ctx->E.t_end)) use_grid = false;
        if (!(std::fabs(last - start) <= kGridMaxLaunches * kGridUnits * unit)) use_grid = false;
    }
    if (use_grid) {
        // internal marks where a gap exceeds one launch
        std::vector<double> m2;
        std::vector<int32_t> r2;
        double prev = start;
        for (int k = 0; k < n_stops; k++) {
            const double from = leg_days > 0.0 ? prev : on_table(prev);
            const double gap = (leg_days > 0.0 ? stops[k] : on_table(stops[k])) - from;
            const double most = leg_days > 0.0 ? leg_days : unit * kGridUnits;
            const int64_t parts = (gap > 0.0) == forward ? (int64_t)std::ceil(std::fabs(gap) / most) : 0;
            for (int64_t p = 1; p < parts; p++) {
                const double step = leg_days > 0.0 ? (forward ? most : -most) : gap / (double)parts;
                m2.push_back(from + step * (double)p);
                r2.push_back(leg_days > 0.0 ? -1 : kMarkRow);
            }
            m2.push_back(stops[k]);
            r2.push_back(k);
            prev = stops[k];
        }
        at.swap(m2);
        row.swap(r2);
    }
    const auto marks = std::make_shared<const std::vector<double>>(std::move(at));
    const std::vector<double> &mark = *marks;
    const int n_marks = (int)mark.size();
    GET(S_STOPS, n_marks, d_stops);
    GET(S_STOPROW, n_marks, d_row);
    CUDA_TRY(upload(ctx, d_stops, marks));
    CUDA_TRY(upload(ctx, d_row, std::make_shared<const std::vector<int32_t>>(std::move(row))));
    if (few) {
        CUDA_TRY(launch_propagate_warp(ctx->E, F, model, cs, d_stops, d_row, n_marks, out, stride,
                                       keep_on_fail, ctx->d_ctr, ctx->stream, PropQueue{}, out_aos));
        return KETE_OK;
    }
    if (!use_grid)
        return propagate_launch(ctx, F, cs, t_from, stops[n_stops - 1], d_stops, d_row, n_marks, out, stride,
                                keep_on_fail, nullptr, out_aos);
    for (int k0 = 0; k0 < n_marks;) {
        int k1 = k0 + 1;   // the marks of this launch
        while (k1 < n_marks && (leg_days > 0.0 ? k1 - k0 < kGridUnits
                                               : std::fabs(mark[k1] - start) <= unit * kGridUnits * (1.0 + 1e-12)))
            k1++;
        const double end = mark[k1 - 1], span = std::fabs(end - start);
        GridDev Q;
        const bool grid = end != start;
        if (grid) {
            const int J = leg_days > 0.0 ? k1 - k0
                                         : (int)std::max(1.0, std::min((double)kGridUnits, std::ceil(span / unit - 1e-9)));
            const double u = leg_days > 0.0 ? leg_days : span / J;
            std::vector<double> pts((size_t)J + 1);
            for (int j = 0; j <= J; j++)
                pts[j] = leg_days > 0.0 && j > 0 ? mark[k0 + j - 1] : start + (end > start ? u : -u) * j;
            pts[J] = end;
            const int r = make_grid(ctx, std::move(pts), u, leg_days > 0.0, Q);
            if (r != KETE_OK) return r;
            Q.chain = n_stops > 1 || leg_days > 0.0;
        }
        const int r = propagate_launch(ctx, F, cs, start, end, d_stops + k0, d_row + k0, k1 - k0, out, stride,
                                       keep_on_fail, grid ? &Q : nullptr, out_aos);
        if (r != KETE_OK) return r;
        if (k1 < n_marks) ctx->extra_launches += 1;
        start = end;
        k0 = k1;
    }
    return KETE_OK;
}

// the first body's epoch (device)
static int first_epoch(kete_ctx *ctx, const double *epochs, double &e0)
{
    CUDA_TRY(cudaMemcpyAsync(&e0, epochs, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    return KETE_OK;
}

static int run_chain(kete_ctx *ctx, const ForceDev &F, const double *states, const double *epochs,
                     int64_t n, ChainState &cs)
{
    GET(S_CHAIN, 8 * n, cs.w);
    GET(S_STATUS, n, cs.status);
    GET(S_KSTOP, n, cs.kstop);
    GET(S_TRIES, n, cs.tries);
    cs.n = n;
    CUDA_TRY(launch_chain_init(cs, states, epochs, F, ctx->stream));
    return KETE_OK;
}

extern "C" int kete_propagate(kete_ctx *ctx, double *states, double *epochs, int64_t n,
                              double t_target, const kete_force_model *fm, int32_t *status)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n < 0 || n > INT32_MAX || (n > 0 && (!states || !epochs)) || !std::isfinite(t_target))
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments");
    ForceDev F;
    int r = make_force(ctx, fm, F);
    if (r != KETE_OK) return r;
    CUDA_TRY(cudaSetDevice(ctx->device));
    stats_begin(ctx);
    if (n > 0) {
        ChainState cs;
        r = run_chain(ctx, F, states, epochs, n, cs);
        if (r != KETE_OK) return r;
        prop_event(ctx, true);
        double e0;
        if ((r = first_epoch(ctx, epochs, e0)) != KETE_OK) return r;
        r = propagate(ctx, F, cs, &t_target, 1, e0, states, n, true, true);
        if (r != KETE_OK) return r;
        prop_event(ctx, false);
        CUDA_TRY(launch_chain_finish(cs, states, epochs, status, ctx->stream));
        ctx->stats.launches = 4;
    }
    r = stats_end(ctx);
    if (r != KETE_OK) return r;
    stats_collect(ctx);
    return KETE_OK;
}

extern "C" int kete_propagate_legs(kete_ctx *ctx, double *states, double *epochs, int64_t n,
                                   double t_target, double leg_days, const kete_force_model *fm,
                                   int32_t *status)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n < 0 || n > INT32_MAX || (n > 0 && (!states || !epochs)) || !std::isfinite(t_target) ||
        !(leg_days > 0.0) || !std::isfinite(leg_days))
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments (leg_days must be positive and finite)");
    ForceDev F;
    int r = make_force(ctx, fm, F);
    if (r != KETE_OK) return r;
    CUDA_TRY(cudaSetDevice(ctx->device));
    stats_begin(ctx);
    if (n > 0) {
        // the grid starts at the first body's epoch
        double e0 = 0.0;
        CUDA_TRY(cudaMemcpyAsync(&e0, epochs, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
        CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        if (!std::isfinite(e0)) return fail(ctx, KETE_ERR_BAD_ARG, "epochs[0] is not finite");
        const double span = t_target - e0;
        const double n_legs = std::ceil(std::fabs(span) / leg_days);
        if (n_legs > 1e7) return fail(ctx, KETE_ERR_BAD_ARG, "more than 10,000,000 legs");
        ChainState cs;
        r = run_chain(ctx, F, states, epochs, n, cs);
        if (r != KETE_OK) return r;
        prop_event(ctx, true);
        r = propagate(ctx, F, cs, &t_target, 1, e0, states, n, true, true,
                      n_legs > 1.0 ? leg_days : 0.0);   // one leg: as kete_propagate
        if (r != KETE_OK) return r;
        prop_event(ctx, false);
        CUDA_TRY(launch_chain_finish(cs, states, epochs, status, ctx->stream));
        ctx->stats.launches = 3;
    }
    r = stats_end(ctx);
    if (r != KETE_OK) return r;
    stats_collect(ctx);
    return KETE_OK;
}

extern "C" int kete_propagate_stops(kete_ctx *ctx, const double *states, const double *epochs,
                                    int64_t n, const double *stops, int64_t n_stops,
                                    const kete_force_model *fm, double *out, int32_t *status)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n < 0 || n > INT32_MAX || n_stops < 0 || n_stops > INT32_MAX ||
        (n > 0 && (!states || !epochs)) || (n_stops > 0 && (!stops || !out)))
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments");
    for (int64_t k = 0; k < n_stops; k++)
        if (!std::isfinite(stops[k]) || (k > 0 && stops[k] < stops[k - 1]))
            return fail(ctx, KETE_ERR_BAD_ARG, "stops must be finite and ascending");
    ForceDev F;
    int r = make_force(ctx, fm, F);
    if (r != KETE_OK) return r;
    CUDA_TRY(cudaSetDevice(ctx->device));
    stats_begin(ctx);
    if (n > 0 && n_stops > 0) {
        ChainState cs;
        r = run_chain(ctx, F, states, epochs, n, cs);
        if (r != KETE_OK) return r;
        prop_event(ctx, true);
        double e0;
        if ((r = first_epoch(ctx, epochs, e0)) != KETE_OK) return r;
        r = propagate(ctx, F, cs, stops, (int)n_stops, e0, out, n, false, true);
        if (r != KETE_OK) return r;
        prop_event(ctx, false);
        CUDA_TRY(launch_chain_finish(cs, nullptr, nullptr, status, ctx->stream));
        ctx->stats.launches = 4;
    }
    r = stats_end(ctx);
    if (r != KETE_OK) return r;
    stats_collect(ctx);
    return KETE_OK;
}

// Union of the sub-frames' hits (tmp, nh in any order; parent[sub-frame]) per
// parent frame: one hit per (frame, body), the earliest sub-frame's, sorted by
// (frame, body) into hits.  CAPACITY leaves the merged count in *n_hits.
static int merge_extended(kete_ctx *ctx, const kete_hit *tmp, unsigned long long nh,
                          const int32_t *parent, int64_t np, kete_hit *hits, int64_t capacity,
                          int64_t *n_hits, int64_t &launches)
{
    cudaStream_t st = ctx->stream;
    int32_t *cnt, *cur, *kcnt; int64_t *off, *koff, *scan_tmp; kete_hit *grp; int8_t *keep;
    GET(S_EXT_CNT, np, cnt);
    GET(S_EXT_CUR, np, cur);
    GET(S_EXT_KCNT, np, kcnt);
    GET(S_EXT_OFF, np + 1, off);
    GET(S_EXT_KOFF, np + 1, koff);
    GET(S_EXT_TMP, scan_tmp_elems(np), scan_tmp);
    GET(S_EXT_GROUP, nh, grp);
    GET(S_EXT_KEEP, nh, keep);
    phase_mark(ctx, PH_ORDER, true);
    CUDA_TRY(cudaMemsetAsync(cnt, 0, np * sizeof(int32_t), st));
    CUDA_TRY(cudaMemsetAsync(cur, 0, np * sizeof(int32_t), st));
    CUDA_TRY(fov_merge_count(tmp, nh, parent, cnt, nullptr, nullptr, nullptr, false, st));
    CUDA_TRY(exclusive_scan(cnt, np, off, scan_tmp, st));
    CUDA_TRY(fov_merge_count(tmp, nh, parent, cnt, off, cur, grp, true, st));
    CUDA_TRY(fov_merge_keep(grp, off, np, keep, kcnt, ctx->n_sm, st));
    CUDA_TRY(exclusive_scan(kcnt, np, koff, scan_tmp, st));
    int64_t merged = 0;
    CUDA_TRY(cudaMemcpyAsync(&merged, koff + np, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    launches += 3 + 2 * scan_launches(np);
    *n_hits = merged;
    if (merged > capacity) {
        phase_mark(ctx, PH_ORDER, false);
        return fail(ctx, KETE_ERR_CAPACITY, "hit buffer holds %lld, %lld needed", (long long)capacity,
                    (long long)merged);
    }
    if (merged > 0) {
        CUDA_TRY(fov_merge_place(grp, off, keep, koff, np, hits, ctx->n_sm, st));
        launches++;
    }
    phase_mark(ctx, PH_ORDER, false);
    return KETE_OK;
}

// sky-cell grid: bands of height ~cell, cells of width >= cell along each band
static void make_bands(double cell, std::vector<int32_t> &off, std::vector<int32_t> &cnt,
                       double &hb, int &n_bands, int &n_cells)
{
    const double pi = 3.14159265358979323846;
    n_bands = std::max(1, (int)std::ceil(pi / cell));
    hb = pi / n_bands;
    off.assign(n_bands + 1, 0);
    cnt.assign(n_bands, 1);
    for (int j = 0; j < n_bands; j++) {
        double lo = -0.5 * pi + j * hb, hi = lo + hb;
        double closest = (lo <= 0.0 && hi >= 0.0) ? 0.0 : std::min(std::fabs(lo), std::fabs(hi));
        int nj = (int)std::floor(2.0 * pi * std::cos(closest) / cell);
        cnt[j] = std::max(1, nj);
        off[j + 1] = off[j] + cnt[j];
    }
    n_cells = off[n_bands];
}

// The survey driver.  ext_nsub > 0: the frames are extended exposures of
// ext_dur[f] days each (device), replaced by ext_nsub instantaneous sub-frames
// (fov_ext_expand) whose hits are merged back per frame at the end.
static int fov_check_impl(kete_ctx *ctx, const double *states, const double *epochs,
                          int64_t n, const kete_frame *frames, int64_t n_frames,
                          const double *observers, int64_t n_obs,
                          const kete_force_model *fm, const kete_survey_opts *opt_in,
                          const kete_mag_params *mag, kete_hit *hits, int64_t capacity,
                          int64_t *n_hits, int32_t *status, const double *ext_dur = nullptr,
                          int ext_nsub = 0)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (!n_hits || n < 0 || n > INT32_MAX || n_frames < 0 || n_frames >= INT32_MAX || n_obs < 0 ||
        capacity < 0 || (n > 0 && (!states || !epochs)) ||
        (n_frames > 0 && (!frames || !observers || n_obs == 0)) || (capacity > 0 && !hits))
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments");
    kete_survey_opts opt;
    if (opt_in) opt = *opt_in;
    else kete_survey_opts_default(&opt);
    if (!(opt.batch_span >= 0) || !(opt.twobody_max >= 0) || !(opt.cell_deg >= 0) ||
        !(opt.mem_budget_gb >= 0))
        return fail(ctx, KETE_ERR_BAD_ARG, "invalid survey options");
    ForceDev F;
    int r = make_force(ctx, fm, F);
    if (r != KETE_OK) return r;
    const bool ext = ext_nsub > 0;
    if (ext && (ext_nsub > KETE_EXT_MAX_SUB || (n_frames > 0 && !ext_dur) ||
                n_frames * (int64_t)ext_nsub >= INT32_MAX))
        return fail(ctx, KETE_ERR_BAD_ARG, "extended exposures: n_sub must be 1..%d, durations "
                    "given, n_frames * n_sub below 2^31", KETE_EXT_MAX_SUB);
    *n_hits = 0;
    CUDA_TRY(cudaSetDevice(ctx->device));
    cudaStream_t st = ctx->stream;
    stats_begin(ctx);
    int64_t launches = 0;
    int32_t *ext_parent = nullptr;
    if (ext && n_frames > 0) {
        // sub-frames of the extended exposures (Sec. 3.1)
        int32_t *pst, *pfirst; int64_t *pex, *ptmp; kete_frame *sub;
        GET(S_EXT_START, n_frames, pst);
        GET(S_EXT_EX, n_frames + 1, pex);
        GET(S_EXT_TMP, scan_tmp_elems(n_frames), ptmp);
        GET(S_EXT_FIRST, n_frames + 1, pfirst);
        GET(S_EXT_SUB, n_frames * ext_nsub, sub);
        GET(S_EXT_PARENT, n_frames * ext_nsub, ext_parent);
        CUDA_TRY(fov_ext_expand(frames, ext_dur, n_frames, ext_nsub, n_obs, pst, pex, ptmp, pfirst,
                                sub, ext_parent, ctx->d_ctr, st));
        launches += 3 + scan_launches(n_frames);
        CUDA_TRY(cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost, st));
        CUDA_TRY(cudaStreamSynchronize(st));
        const int fl = ctx->h_ctr->error_flags;
        if (fl & 1) return fail(ctx, KETE_ERR_BAD_ARG, "frames are not sorted by epoch");
        if (fl & 2) return fail(ctx, KETE_ERR_BAD_ARG, "frames of one exposure differ in epoch, observer or duration");
        if (fl & 4) return fail(ctx, KETE_ERR_BAD_ARG, "observer_idx + n_sub exceeds the observer rows");
        if (fl & 64) return fail(ctx, KETE_ERR_BAD_ARG, "exposure durations must be finite and >= 0");
        frames = sub;
        n_frames *= ext_nsub;
    }
    const int64_t nf = n_frames;
    ChainState cs{};
    if (n > 0) {
        r = run_chain(ctx, F, states, epochs, n, cs);
        if (r != KETE_OK) return r;
        launches++;
    }
    if (nf == 0 || n == 0) {
        if (n > 0) CUDA_TRY(launch_chain_finish(cs, nullptr, nullptr, status, st));
        r = stats_end(ctx);
        if (r != KETE_OK) return r;
        stats_collect(ctx);
        return KETE_OK;
    }
    // ---- frames -> exposures ------------------------------------------------
    int32_t *is_start; int64_t *ex, *scan_tmp; double *fcen; float4 *faux; int32_t *exp_first;
    GET(S_ISSTART, nf, is_start);
    GET(S_EX, nf + 1, ex);
    GET(S_FCEN, 4 * nf, fcen);
    GET(S_FAUX, nf, faux);
    phase_mark(ctx, PH_PREP, true);
    CUDA_TRY(fov_frame_prep(frames, nf, n_obs, is_start, fcen, faux, ctx->d_ctr, st));
    GET(S_SCANTMP, scan_tmp_elems(nf), scan_tmp);
    CUDA_TRY(exclusive_scan(is_start, nf, ex, scan_tmp, st));
    GET(S_EXPFIRST, nf + 1, exp_first);
    CUDA_TRY(fov_exposure_first(is_start, ex, nf, exp_first, st));
    launches += 3 + 2;
    int64_t h_ne = 0;
    CUDA_TRY(cudaMemcpyAsync(&h_ne, ex + nf, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    int flags = ctx->h_ctr->error_flags;
    if ((flags & 1) && ext)
        return fail(ctx, KETE_ERR_BAD_ARG, "sub-frame epochs are not sorted: extended exposures overlap in time");
    if (flags & 1) return fail(ctx, KETE_ERR_BAD_ARG, "frames are not sorted by epoch");
    if (flags & 2) return fail(ctx, KETE_ERR_BAD_ARG, "frames of one exposure differ in epoch or observer");
    if (flags & 4) return fail(ctx, KETE_ERR_BAD_ARG, "observer_idx out of range");
    if (flags & 8) return fail(ctx, KETE_ERR_BAD_ARG, "n_edges must be 3 or 4 (polygon) or 0 (cone)");
    if (flags & 16) return fail(ctx, KETE_ERR_BAD_ARG, "non-finite or degenerate frame");
    const int64_t ne = h_ne;
    ExpArrays X;
    GET(S_XEPOCH, ne, X.epoch);
    GET(S_XOBS, 3 * ne, X.obs);
    GET(S_XCEN, 3 * ne, X.cen);
    GET(S_XRAD, ne, X.rad);
    GET(S_XCS, ne, X.cs);
    GET(S_XCENF, ne, X.cenf);
    GET(S_XBATCH, ne, X.batch);
    GET(S_XSUN, 6 * ne, X.sun);
    GET(S_XOBSREL, ne, X.obs_rel);
    unsigned int *d_maxrad;
    GET(S_MAXRAD, 1, d_maxrad);
    CUDA_TRY(cudaMemsetAsync(d_maxrad, 0, sizeof(unsigned int), st));
    CUDA_TRY(fov_exposure_prep(ctx->E, frames, nf, observers, fcen, exp_first, ne, X, d_maxrad,
                               ctx->d_ctr, st));
    // ---- batches (Sec. 2) ---------------------------------------------------
    double span = std::min(opt.batch_span, 2.0 * opt.twobody_max);
    int32_t *next, *d_nb;
    BatchArrays B;
    GET(S_NEXT, ne, next);
    GET(S_BFIRST, ne + 1, B.first);
    GET(S_BTREF, ne, B.t_ref);
    GET(S_NBATCH, 1, d_nb);
    CUDA_TRY(fov_batches(X.epoch, ne, span, next, B, d_nb, st));
    launches += 3;
    int32_t h_nb = 0;
    unsigned int h_maxrad = 0;
    CUDA_TRY(cudaMemcpyAsync(&h_nb, d_nb, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(&h_maxrad, d_maxrad, sizeof(unsigned int), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    const int32_t nb = h_nb;
    std::vector<int32_t> h_first(nb + 1);
    std::vector<double> h_tref(nb);
    double chain_at = 0.0;   // where the chain of midpoints stands
    CUDA_TRY(cudaMemcpyAsync(h_first.data(), B.first, (nb + 1) * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(h_tref.data(), B.t_ref, nb * sizeof(double), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(&chain_at, epochs, sizeof(double), cudaMemcpyDeviceToHost, st));
    GET(S_BO, 3 * nb, B.O);
    GET(S_BROBS, nb, B.robs);
    GET(S_BTSPAN, nb, B.tspan);
    GET(S_BRMAX, nb, B.rmax);
    GET(S_BSUN, 6 * nb, B.sun);
    CUDA_TRY(fov_batch_info(ctx->E, X, B, nb, ctx->d_ctr, st));
    phase_mark(ctx, PH_PREP, false);
    launches++;
    // ---- sky cells -------------------------------------------------------------
    float maxrad;
    std::memcpy(&maxrad, &h_maxrad, sizeof(float));
    const double pi = 3.14159265358979323846;
    double cell = opt.cell_deg > 0 ? opt.cell_deg * pi / 180.0
                                   : std::min(20.0 * pi / 180.0, std::max(0.5 * pi / 180.0, 2.0 * (double)maxrad));
    std::vector<int32_t> boff, bcnt;
    CellGrid G;
    int n_bands, n_cells;
    make_bands(cell, boff, bcnt, G.hb, n_bands, n_cells);
    G.n_bands = n_bands;
    G.n_cells = n_cells;
    int32_t *d_bands;
    GET(S_BANDS, 2 * n_bands + 1, d_bands);
    CUDA_TRY(cudaMemcpyAsync(d_bands, boff.data(), (n_bands + 1) * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemcpyAsync(d_bands + n_bands + 1, bcnt.data(), n_bands * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    G.band_off = d_bands;
    G.band_n = d_bands + n_bands + 1;
    // ---- chunks of batches ----------------------------------------------------
    double budget = (opt.mem_budget_gb > 0 ? opt.mem_budget_gb : 8.0) * 1e9;
    int64_t per_batch = 48 * n;
    int32_t C = (int32_t)std::max<int64_t>(1, std::min<int64_t>(nb, (int64_t)(budget / per_batch)));
    // keep the cell CSR of a chunk modest
    C = (int32_t)std::max<int64_t>(1, std::min<int64_t>(C, 200000000LL / std::max(1, n_cells)));
    double *stop_states;
    GET(S_STOPSTATES, (size_t)C * 6 * n, stop_states);
    int32_t *frame_cnt;
    GET(S_FRAMECNT, nf, frame_cnt);
    CUDA_TRY(cudaMemsetAsync(frame_cnt, 0, nf * sizeof(int32_t), st));
    unsigned long long cand_cap = ctx->slot[S_CAND].bytes / sizeof(uint2);
    if (cand_cap < (unsigned long long)(4 * n + 1024)) cand_cap = 4 * n + 1024;
    unsigned long long hit_cap = ctx->slot[S_HITTMP].bytes / sizeof(kete_hit);
    if (hit_cap < (unsigned long long)(nf + 1024)) hit_cap = nf + 1024;
    kete_hit *hit_tmp;
    GET(S_HITTMP, hit_cap, hit_tmp);
    hit_cap = ctx->slot[S_HITTMP].bytes / sizeof(kete_hit);
    CUDA_TRY(cudaStreamSynchronize(st));
    unsigned long long hits_total = 0, cands_total = 0, exact_total = 0;
    for (int32_t k0 = 0; k0 < nb; k0 += C) {
        const int32_t k1 = std::min(nb, k0 + C), nk = k1 - k0;
        const int32_t e0 = h_first[k0], e1 = h_first[k1];
        const int32_t nek = e1 - e0;
        // propagation to the batch midpoints of this chunk
        prop_event(ctx, true);
        r = propagate(ctx, F, cs, h_tref.data() + k0, nk, chain_at, stop_states, n, false, true, 0.0,
                      true);
        if (r != KETE_OK) return r;
        chain_at = h_tref[k1 - 1];
        prop_event(ctx, false);
        launches++;
        // exposures of the chunk into sky cells
        const int64_t nkeys = (int64_t)nk * n_cells;
        int32_t *ckey, *ccnt, *ccur, *cexp; int64_t *cstart;
        GET(S_CELLKEY, nek, ckey);
        GET(S_CELLCNT, nkeys, ccnt);
        GET(S_CELLCUR, nkeys, ccur);
        GET(S_CELLSTART, nkeys + 1, cstart);
        GET(S_CELLEXP, nek, cexp);
        GET(S_SCANTMP, std::max(scan_tmp_elems(nkeys), scan_tmp_elems(nf)), scan_tmp);
        phase_mark(ctx, PH_CAND, true);
        CUDA_TRY(cudaMemsetAsync(ccnt, 0, nkeys * sizeof(int32_t), st));
        CUDA_TRY(cudaMemsetAsync(ccur, 0, nkeys * sizeof(int32_t), st));
        CUDA_TRY(fov_cell_keys(X, G, e0, e1, k0, ckey, ccnt, st));
        CUDA_TRY(exclusive_scan(ccnt, nkeys, cstart, scan_tmp, st));
        CUDA_TRY(fov_cell_scatter(e0, e1, ckey, cstart, ccur, cexp, st));
        launches += 4;
        // candidate (exposure, body) pairs
        int32_t *exp_cnt;
        GET(S_EXPCNT, ne, exp_cnt);
        unsigned long long ncand = 0;
        for (int attempt = 0; attempt < 3; attempt++) {
            uint2 *cand;
            GET(S_CAND, cand_cap, cand);
            cand_cap = ctx->slot[S_CAND].bytes / sizeof(uint2);
            CUDA_TRY(cudaMemsetAsync(exp_cnt + e0, 0, nek * sizeof(int32_t), st));
            CUDA_TRY(cudaMemsetAsync(&ctx->d_ctr->candidates, 0, sizeof(unsigned long long), st));
            CandArgs ca;
            ca.X = X; ca.B = B; ca.G = G; ca.stop_states = stop_states; ca.n = n; ca.k0 = k0;
            ca.nk = nk; ca.cell_start = cstart; ca.cell_exp = cexp; ca.cand = cand;
            ca.cap = cand_cap; ca.exp_cnt = exp_cnt; ca.ctr = ctx->d_ctr; ca.mu_sun = ctx->E.gm[0];
            CUDA_TRY(fov_candidates(ca, st));
            launches++;
            CUDA_TRY(cudaMemcpyAsync(&ncand, &ctx->d_ctr->candidates, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
            CUDA_TRY(cudaStreamSynchronize(st));
            if (ncand <= cand_cap) break;
            cand_cap = ncand + ncand / 2 + 1024;
        }
        if (ncand > cand_cap)
            return fail(ctx, KETE_ERR_NOMEM, "candidate buffer could not grow to %llu pairs", ncand);
        cands_total += ncand;
        int64_t *exp_off; int32_t *exp_cur, *cand_body;
        GET(S_EXPOFF, nek + 1, exp_off);
        GET(S_EXPCUR, nek, exp_cur);
        GET(S_CANDBODY, ncand, cand_body);
        CUDA_TRY(exclusive_scan(exp_cnt + e0, nek, exp_off, scan_tmp, st));
        CUDA_TRY(cudaMemsetAsync(exp_cur, 0, nek * sizeof(int32_t), st));
        CUDA_TRY(fov_cand_scatter((const uint2 *)ctx->slot[S_CAND].p, ncand, exp_off, e0, exp_cur, cand_body, st));
        phase_mark(ctx, PH_CAND, false);
        launches += 3;
        // exact two-body + light time + polygon test, after the FP32 prefilter
        uint32_t *pre_keep;
        unsigned long long *pre_n;
        GET(S_PRE_KEEP, ncand, pre_keep);
        GET(S_PRE_N, 1, pre_n);
        for (int attempt = 0; attempt < 3; attempt++) {
            CUDA_TRY(cudaMemcpyAsync(&ctx->d_ctr->hits, &hits_total, sizeof(unsigned long long), cudaMemcpyHostToDevice, st));
            ExactArgs xa;
            xa.E = ctx->E; xa.X = X; xa.B = B; xa.frames = frames; xa.faux = faux;
            xa.stop_states = stop_states; xa.n = n; xa.k0 = k0; xa.e_begin = e0; xa.e_end = e1;
            xa.exp_off = exp_off; xa.n_cand = (int64_t)ncand; xa.cand_body = cand_body;
            xa.exp_first = exp_first;
            xa.hits = hit_tmp; xa.cap = hit_cap; xa.frame_cnt = frame_cnt; xa.status = cs.status;
            xa.ctr = ctx->d_ctr;
            xa.mag = mag;
            xa.keep = pre_keep;
            xa.n_keep = pre_n;
            phase_mark(ctx, PH_EXACT, true);
            CUDA_TRY(fov_exact(xa, ctx->n_sm, st));
            phase_mark(ctx, PH_EXACT, false);
            if (ncand > 0 && nek > 0) launches += ncand <= 0xffffffffull ? 2 : 1;
            unsigned long long nh = 0, nkept = ncand;
            CUDA_TRY(cudaMemcpyAsync(&nh, &ctx->d_ctr->hits, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
            if (ncand > 0 && nek > 0 && ncand <= 0xffffffffull)
                CUDA_TRY(cudaMemcpyAsync(&nkept, pre_n, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
            CUDA_TRY(cudaStreamSynchronize(st));
            if (nh <= hit_cap) {
                hits_total = nh;
                exact_total += nkept;
                break;
            }
            // grow the hit buffer, keep earlier chunks' hits, redo this chunk
            int32_t fa = 0, fb = 0;
            CUDA_TRY(cudaMemcpy(&fa, exp_first + e0, sizeof(int32_t), cudaMemcpyDeviceToHost));
            CUDA_TRY(cudaMemcpy(&fb, exp_first + e1, sizeof(int32_t), cudaMemcpyDeviceToHost));
            CUDA_TRY(cudaMemsetAsync(frame_cnt + fa, 0, (size_t)(fb - fa) * sizeof(int32_t), st));
            unsigned long long want = nh + nh / 2 + 1024;
            kete_hit *bigger = nullptr;
            CUDA_TRY(cudaMalloc(&bigger, want * sizeof(kete_hit)));
            if (hits_total)
                CUDA_TRY(cudaMemcpyAsync(bigger, hit_tmp, hits_total * sizeof(kete_hit), cudaMemcpyDeviceToDevice, st));
            CUDA_TRY(cudaStreamSynchronize(st));
            cudaFree(ctx->slot[S_HITTMP].p);
            ctx->slot[S_HITTMP].p = bigger;
            ctx->slot[S_HITTMP].bytes = want * sizeof(kete_hit);
            hit_tmp = bigger;
            hit_cap = want;
        }
        if (hits_total > hit_cap)
            return fail(ctx, KETE_ERR_NOMEM, "hit buffer could not grow to %llu hits", hits_total);
    }
    ctx->stats.n_batches = nb;
    ctx->stats.n_exposures = ne;
    ctx->stats.n_candidates = (int64_t)cands_total;
    ctx->stats.n_exact = (int64_t)exact_total;
    ctx->stats.n_hits = (int64_t)hits_total;
    *n_hits = (int64_t)hits_total;
    CUDA_TRY(launch_chain_finish(cs, nullptr, nullptr, status, st));
    launches++;
    CUDA_TRY(cudaMemcpyAsync(ctx->h_ctr, ctx->d_ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    if (ctx->h_ctr->error_flags & 32) {
        ctx->stats.launches = launches;
        return fail(ctx, KETE_ERR_EPHEM_SPAN, "a batch midpoint or frame epoch lies outside the ephemeris table");
    }
    if (ext) {
        r = merge_extended(ctx, hit_tmp, hits_total, ext_parent, nf / ext_nsub, hits, capacity,
                           n_hits, launches);
        if (r != KETE_OK) return r;
        r = stats_end(ctx);
        if (r != KETE_OK) return r;
        stats_collect(ctx);
        ctx->stats.n_batches = nb;
        ctx->stats.n_exposures = ne;
        ctx->stats.n_candidates = (int64_t)cands_total;
    ctx->stats.n_exact = (int64_t)exact_total;
        ctx->stats.n_hits = *n_hits;
        ctx->stats.launches = launches + ctx->extra_launches;
        return KETE_OK;
    }
    if ((int64_t)hits_total > capacity) {
        r = stats_end(ctx);
        stats_collect(ctx);
        ctx->stats.launches = launches + ctx->extra_launches;
        return fail(ctx, KETE_ERR_CAPACITY, "hit buffer holds %lld, %llu needed", (long long)capacity,
                    hits_total);
    }
    if (hits_total > 0) {
        int64_t *frame_off; int32_t *frame_cur; kete_hit *grouped;
        GET(S_FRAMEOFF, nf + 1, frame_off);
        GET(S_FRAMECUR, nf, frame_cur);
        GET(S_HITGROUP, hits_total, grouped);
        phase_mark(ctx, PH_ORDER, true);
        CUDA_TRY(exclusive_scan(frame_cnt, nf, frame_off, scan_tmp, st));
        CUDA_TRY(cudaMemsetAsync(frame_cur, 0, nf * sizeof(int32_t), st));
        CUDA_TRY(fov_order_hits(hit_tmp, hits_total, frame_off, nf, frame_cur, grouped, hits, ctx->n_sm, st));
        phase_mark(ctx, PH_ORDER, false);
        launches += 4;
    }
    r = stats_end(ctx);
    if (r != KETE_OK) return r;
    stats_collect(ctx);
    ctx->stats.n_batches = nb;
    ctx->stats.n_exposures = ne;
    ctx->stats.n_candidates = (int64_t)cands_total;
    ctx->stats.n_exact = (int64_t)exact_total;
    ctx->stats.n_hits = (int64_t)hits_total;
    ctx->stats.launches = launches + ctx->extra_launches;
    return KETE_OK;
}

extern "C" int kete_fov_check(kete_ctx *ctx, const double *states, const double *epochs,
                              int64_t n, const kete_frame *frames, int64_t n_frames,
                              const double *observers, int64_t n_obs,
                              const kete_force_model *fm, const kete_survey_opts *opt,
                              kete_hit *hits, int64_t capacity, int64_t *n_hits, int32_t *status)
{
    return fov_check_impl(ctx, states, epochs, n, frames, n_frames, observers, n_obs, fm, opt,
                          nullptr, hits, capacity, n_hits, status);
}

extern "C" int kete_fov_check_mag(kete_ctx *ctx, const double *states, const double *epochs,
                                  int64_t n, const kete_frame *frames, int64_t n_frames,
                                  const double *observers, int64_t n_obs,
                                  const kete_force_model *fm, const kete_survey_opts *opt,
                                  const kete_mag_params *mag_params, kete_hit *hits,
                                  int64_t capacity, int64_t *n_hits, int32_t *status)
{
    return fov_check_impl(ctx, states, epochs, n, frames, n_frames, observers, n_obs, fm, opt,
                          mag_params, hits, capacity, n_hits, status);
}

extern "C" int kete_fov_check_extended(kete_ctx *ctx, const double *states, const double *epochs,
                                       int64_t n, const kete_frame *frames, int64_t n_frames,
                                       const double *durations, int32_t n_sub,
                                       const double *observers, int64_t n_obs,
                                       const kete_force_model *fm, const kete_survey_opts *opt,
                                       const kete_mag_params *mag_params, kete_hit *hits,
                                       int64_t capacity, int64_t *n_hits, int32_t *status)
{
    if (ctx && n_sub < 1)
        return fail(ctx, KETE_ERR_BAD_ARG, "extended exposures: n_sub must be 1..%d", KETE_EXT_MAX_SUB);
    return fov_check_impl(ctx, states, epochs, n, frames, n_frames, observers, n_obs, fm, opt,
                          mag_params, hits, capacity, n_hits, status, durations, n_sub);
}

// Propagation whose chain scratch is a fixed device array (see kete.h): no
// cudaMalloc, cudaFree, scratch slot or event is touched on this path.
extern "C" int kete_propagate_noalloc(kete_ctx *ctx, double *states, double *epochs, int64_t n,
                                      double t_target, const kete_force_model *fm,
                                      int32_t *status)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n < 0 || (n > 0 && (!states || !epochs)) || !std::isfinite(t_target))
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments");
    if (n > KETE_NOALLOC_MAX_BODIES)
        return fail(ctx, KETE_ERR_BAD_ARG, "n = %lld exceeds KETE_NOALLOC_MAX_BODIES = %d",
                    (long long)n, KETE_NOALLOC_MAX_BODIES);
    ForceDev F;
    int r = make_force(ctx, fm, F);
    if (r != KETE_OK) return r;
    CUDA_TRY(cudaSetDevice(ctx->device));
    const char *why = "";
    r = noalloc_propagate(ctx->device, ctx->stream, ctx->E, F, states, epochs, n, t_target,
                          status, &why);
    if (r != KETE_OK) return fail(ctx, r, "kete_propagate_noalloc: %s", why);
    return KETE_OK;
}

extern "C" int kete_set_propagation(kete_ctx *ctx, int precision, int kind, int block,
                                    int split_lanes, int defer_steps, int cost_order_on)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    const bool split_ok = split_lanes == 0 || split_lanes == 1 || split_lanes == 4 ||
                          split_lanes == 8 || split_lanes == 16;
    if ((precision != KETE_FP64 && precision != KETE_MIXED) ||
        (kind != KETE_PROP_STATIC && kind != KETE_PROP_WORK_STEALING) || block < 32 ||
        block > 128 || block % 32 != 0 || !split_ok || defer_steps < 0)
        return fail(ctx, KETE_ERR_BAD_ARG,
                    "bad propagation variant (precision %d, kind %d, block %d, split %d, defer %d)",
                    precision, kind, block, split_lanes, defer_steps);
    PropVariant v{kind, block};
    v.split = split_lanes > 1 ? split_lanes : 0;
    v.budget = v.split ? defer_steps : 0;
    v.order = cost_order_on ? 1 : 0;
    ctx->var[precision == KETE_MIXED ? 1 : 0] = v;
    return KETE_OK;
}

extern "C" int kete_autotune(kete_ctx *ctx, const double *states, const double *epochs, int64_t n,
                             const double *stops, int64_t n_stops, const kete_force_model *fm,
                             int64_t max_sample, int32_t *kind, int32_t *block,
                             int32_t *split_lanes, int32_t *defer_steps, int32_t *cost_order)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n <= 0 || n > INT32_MAX || !states || !epochs || n_stops <= 0 || n_stops > INT32_MAX ||
        !stops || max_sample <= 0)
        return fail(ctx, KETE_ERR_BAD_ARG, "bad arguments");
    for (int64_t k = 0; k < n_stops; k++)
        if (!std::isfinite(stops[k]) || (k > 0 && stops[k] < stops[k - 1]))
            return fail(ctx, KETE_ERR_BAD_ARG, "stops must be finite and ascending");
    ForceDev F;
    int r = make_force(ctx, fm, F);
    if (r != KETE_OK) return r;
    F.nongrav = nullptr;   // the sample is gathered: body indices differ from the caller's
    CUDA_TRY(cudaSetDevice(ctx->device));
    stats_begin(ctx);
    cudaStream_t st = ctx->stream;
    // The sample (spread evenly over the bodies) runs in the form the whole would
    // take and on persistent grids scaled
    // down by m / n, so that each lane works through as many bodies as in the
    // whole run: on the full grid a sample would leave a lane a few bodies and
    // be dominated by its longest-lived ones, which favours the split variants.
    const int64_t m = std::min(n, max_sample);
    const double scale = (double)m / (double)n;
    double *sst, *sep, *out, e_first;
    GET(S_TUNE_ST, 6 * m, sst);
    GET(S_TUNE_EP, m, sep);
    GET(S_TUNE_OUT, (size_t)n_stops * 6 * m, out);
    if ((r = first_epoch(ctx, epochs, e_first)) != KETE_OK) return r;
    CUDA_TRY(launch_gather_bodies(states, epochs, n, m, sst, sep, st));
    // schedules x cost order, then the split variants (with cost order)
    PropVariant cands[8];
    const int kinds[3][2] = {{PROP_STATIC, 128}, {PROP_WORK_STEALING, 64}, {PROP_WORK_STEALING, 128}};
    int n_cands = 0;
    for (int o = 0; o < 2; o++)
        for (int q = 0; q < 3; q++) {
            cands[n_cands] = PropVariant{kinds[q][0], kinds[q][1]};
            cands[n_cands++].order = o;
        }
    for (int budget : {64, 24}) {
        cands[n_cands] = PropVariant{PROP_WORK_STEALING, 128};
        cands[n_cands].split = 8;
        cands[n_cands].budget = budget;
        cands[n_cands++].order = 1;
    }
    // (the values of split act alike)
    const auto alike = [](const PropVariant &a, const PropVariant &b) {
        return a.kind == b.kind && a.block == b.block && (a.split > 0) == (b.split > 0) &&
               a.budget == b.budget && a.order == b.order;
    };
    const int slot = F.precision == KETE_MIXED ? 1 : 0;
    const PropVariant saved = ctx->var[slot];
    float best_ms = 1e30f, saved_ms = -1.0f;
    PropVariant best = saved;
    event_at(ctx, 3);
    cudaEvent_t e0 = event_at(ctx, 2), e1 = event_at(ctx, 3);
    // time variant v on cnt bodies (states st, epochs ep; output rows out),
    // the best of reps runs after one that warms up
    auto time_variant = [&](const PropVariant &v, const double *st_, const double *ep_,
                            int64_t cnt, double *out_, int reps, float &ms) -> int {
        ctx->var[slot] = v;
        ms = 1e30f;
        for (int rep = 0; rep <= reps; rep++) {
            ChainState cs;
            int r2 = run_chain(ctx, F, st_, ep_, cnt, cs);
            if (r2 != KETE_OK) return r2;
            CUDA_TRY(cudaEventRecord(e0, st));
            r2 = propagate(ctx, F, cs, stops, (int)n_stops, e_first, out_, cnt, false, true);
            if (r2 != KETE_OK) return r2;
            CUDA_TRY(cudaEventRecord(e1, st));
            CUDA_TRY(cudaEventSynchronize(e1));
            float t = 0.0f;
            CUDA_TRY(cudaEventElapsedTime(&t, e0, e1));
            if (rep > 0) ms = std::min(ms, t);
        }
        return KETE_OK;
    };
    for (int c = 0; c < n_cands; c++) {
        cands[c].grid_scale = scale;
        cands[c].population = n;
    }
    for (int c = 0; c < n_cands; c++) {
        float ms;
        r = time_variant(cands[c], sst, sep, m, out, 2, ms);
        if (r != KETE_OK) return r;
        if (ms < best_ms) {
            best_ms = ms;
            best = cands[c];
        }
        if (alike(cands[c], saved)) saved_ms = ms;
    }
    // a sample ranks variants that differ by a few per cent unreliably (its
    // scaled-down grid holds fewer warps per SM than the real launch): the
    // variant in use stays unless another beats it by more than 5 %, and a
    // pick that does is checked against it on all the bodies when their
    // output rows fit in 2 GB
    if (saved_ms > 0.0f && best_ms > 0.95f * saved_ms) best = saved;
    if (!alike(best, saved) && m < n && saved_ms > 0.0f && (double)n_stops * 48.0 * (double)n <= 2e9) {
        double *full_out;
        GET(S_TUNE_OUT, (size_t)n_stops * 6 * n, full_out);
        PropVariant pick = best, cur = saved;
        pick.grid_scale = cur.grid_scale = 1.0;
        // the best of two runs each (run-to-run spread ~1-2 %); the pick must
        // win by 2 %
        float ms_pick, ms_cur;
        r = time_variant(cur, states, epochs, n, full_out, 2, ms_cur);
        if (r != KETE_OK) return r;
        r = time_variant(pick, states, epochs, n, full_out, 2, ms_pick);
        if (r != KETE_OK) return r;
        if (!(ms_pick < 0.98f * ms_cur)) best = saved;
    }
    best.grid_scale = 1.0;
    best.population = 0;
    ctx->var[slot] = best;
    if ((r = stats_end(ctx)) != KETE_OK) return r;
    stats_collect(ctx);   // the counters of all its runs
    if (kind) *kind = best.kind;
    if (block) *block = best.block;
    if (split_lanes) *split_lanes = best.split;
    if (defer_steps) *defer_steps = best.budget;
    if (cost_order) *cost_order = best.order;
    return KETE_OK;
}

// The orbit-fit path of kete_adjoint and kete_sky_jacobian: forward pass with
// step records, then (jac) the state-transition matrix at every batch
// midpoint, the observations (loss, predictions, partials), then (grad) the
// backward pass.
static int adjoint_impl(kete_ctx *ctx, const double *states, const double *epochs, int64_t n,
                        const kete_obs *obs, int32_t m, const kete_force_model *fm,
                        const kete_survey_opts *opt_in, double ckpt_days, double *loss,
                        double *grad, double *pred, double *jac, int32_t *status)
{
    if (!ctx) return KETE_ERR_BAD_ARG;
    if (!ctx->have_ephem) return fail(ctx, KETE_ERR_NO_EPHEM, "no ephemeris loaded");
    if (n < 0 || n > INT32_MAX || m < 1 || m > KETE_ADJ_MAX_OBS ||
        (n > 0 && (!states || !epochs || !obs || (!loss && !jac))) ||
        !(ckpt_days == 0.0 || ckpt_days >= 1e-3) || !std::isfinite(ckpt_days))
        return fail(ctx, KETE_ERR_BAD_ARG,
                    "bad arguments (m must lie in 1..%d, ckpt_days 0 or >= 1e-3)", KETE_ADJ_MAX_OBS);
    kete_survey_opts opt;
    if (opt_in) opt = *opt_in;
    else kete_survey_opts_default(&opt);
    if (!(opt.batch_span > 0) || !(opt.twobody_max >= 0) || !(opt.mem_budget_gb >= 0))
        return fail(ctx, KETE_ERR_BAD_ARG, "invalid survey options");
    kete_force_model fm64;
    if (fm) fm64 = *fm;
    else kete_force_model_default(&fm64);
    fm64.precision = KETE_FP64;
    ForceDev F;
    int r = make_force(ctx, &fm64, F);
    if (r != KETE_OK) return r;
    F.eps_pc = fm64.eps_pc;   // constant start (see step_factor)
    CUDA_TRY(cudaSetDevice(ctx->device));
    stats_begin(ctx);
    if (n > 0) {
        const double eps_obl = 84381.448 / 3600.0 * 3.14159265358979323846 / 180.0;
        AdjProblem P;
        P.states = states;
        P.epochs = epochs;
        P.n = n;
        P.obs = obs;
        P.m = m;
        P.span = std::min(opt.batch_span, 2.0 * opt.twobody_max);
        P.ckpt = ckpt_days;
        P.inv_ckpt = ckpt_days > 0.0 ? 1.0 / ckpt_days : 0.0;
        P.cos_eps = std::cos(eps_obl);
        P.sin_eps = std::sin(eps_obl);
        P.loss = loss;
        P.grad = grad;
        P.pred = pred;
        P.jac = jac;
        P.status = status;
        P.ctr = ctx->d_ctr;
        // scratch per chunk of bodies within the memory budget
        const int cap = KETE_ADJ_MAX_STEPS;
        // with non-gravitational terms the records carry the full model's Jacobian
        const bool full = fm64.nongrav != nullptr;
        const size_t per_body = (size_t)cap * (kAdjRec + (full ? kAdjRecX : 0)) * sizeof(double) +
                                (size_t)m * (sizeof(int32_t) + 12 * sizeof(double)) +
                                (jac ? (size_t)m * 36 * sizeof(double) : 0) +
                                (size_t)m * sizeof(double) + 3 * sizeof(int32_t);
        const double budget = (opt.mem_budget_gb > 0 ? opt.mem_budget_gb : 8.0) * 1073741824.0;
        int64_t chunk = (int64_t)(budget / (double)per_body);
        chunk = std::max<int64_t>(1, std::min<int64_t>(chunk, n));
        const int64_t n_chunks = (n + chunk - 1) / chunk;   // even chunks
        chunk = (n + n_chunks - 1) / n_chunks;
        // one warp per body (kete_warp.cu); the lanes serve what that form does not
        WarpModel model;
        const bool warps = !full && F.max_iter >= 8 && warp_model(ctx->E, F, model);
        if (warps) F.eps_pc = kStartTighter * fm64.eps_pc;
        AdjBuffers B;
        B.cap = cap;
        GET(S_ADJ_REC, (size_t)chunk * cap * kAdjRec, B.rec);
        GET(S_ADJ_NREC, chunk, B.n_rec);
        GET(S_ADJ_NBAT, chunk, B.nbat);
        GET(S_ADJ_BIDX, (size_t)chunk * m, B.bidx);
        GET(S_ADJ_YREF, (size_t)chunk * m * 6, B.yref);
        GET(S_ADJ_GJUMP, (size_t)chunk * m * 6, B.gjump);
        GET(S_ADJ_STATUS, chunk, B.status);
        GET(S_ADJ_BFRAC, (size_t)chunk * m, B.bfrac);
        B.phi = nullptr;
        if (jac) GET(S_ADJ_PHI, (size_t)chunk * m * 36, B.phi);
        B.recx = nullptr;
        B.rich = nullptr;
        if (full) {
            GET(S_ADJ_RECX, (size_t)chunk * cap * kAdjRecX, B.recx);
            GET(S_ADJ_RICH, chunk, B.rich);
        }
        B.planets = nullptr;
        if (!warps)
            GET(S_ADJ_PLANETS, (size_t)adjoint_forward_lanes(chunk, full) * 7 * ctx->E.n_bodies * 6,
                B.planets);
        unsigned long long *next = nullptr;
        GET(S_NEXTBODY, 1, next);
        int launches = 0;
        double *t_end;
        GET(S_ADJ_TEND, chunk, t_end);
        const bool order_on = ctx->var[0].order != 0;
        for (int64_t i0 = 0; i0 < n; i0 += chunk) {
            const int64_t nc = std::min(chunk, n - i0);
            prop_event(ctx, true);
            int32_t *order = nullptr;
            // many bodies whose chains share one step grid: lanes (see takes_warps)
            unsigned long long *order_n = nullptr;
            GridDev Q{};
            double span = 0.0;
            bool lanes = warps && nc > kWarpBodies;
            B.mid = nullptr;
            if (lanes) {
                unsigned long long *range, key[2];
                GET(S_ADJ_MID, (size_t)chunk * m, B.mid);
                GET(S_ADJ_RANGE, 2, range);
                CUDA_TRY(launch_fit_stops(B, P, i0, nc, range, ctx->stream));
                CUDA_TRY(cudaMemcpyAsync(key, range, sizeof(key), cudaMemcpyDeviceToHost, ctx->stream));
                CUDA_TRY(cudaStreamSynchronize(ctx->stream));
                launches++;
                const double lo = std::max(ctx->E.t_start, fit_range_epoch(key[0]));
                const double hi = std::min(ctx->E.t_end, fit_range_epoch(key[1]));
                span = hi - lo;
                lanes = span > 0.0 && span <= (double)kGridUnits && !takes_warps(nc, span, false);
                if (lanes) {
                    const int J = (int)std::max(1.0, std::ceil(span - 1e-9));
                    std::vector<double> pts((size_t)J + 1);
                    for (int j = 0; j <= J; j++) pts[j] = lo + span / J * j;
                    pts[J] = hi;
                    if ((r = make_grid(ctx, std::move(pts), span / J, false, Q)) != KETE_OK) return r;
                }
            }
            if (order_on && (!warps || lanes)) {   // most expensive bodies first (schedule only)
                CUDA_TRY(launch_adjoint_last_epoch(P, i0, nc, t_end, ctx->stream));
                // bodies with and without non-gravitational terms in separate
                // ranges, so that the full-model records rarely share a warp
                int r2 = cost_order(ctx, states + i0, n, epochs + i0, nc, 0.0, t_end,
                                    F.nongrav ? F.nongrav + i0 : nullptr, &order, &order_n);
                if (r2 != KETE_OK) return r2;
                launches += 1;
            }
            if (lanes) {
                PropDefer defer{};
                GET(S_DEFER_LIST, nc, defer.list);
                GET(S_DEFER_CNT, 1, defer.count);
                // (lengths rounded down to the grid's can double a body's steps: one
                // near the record limit takes its own in a warp)
                defer.budget0 = std::min(attempts_budget(ctx, nc, span, false), KETE_ADJ_MAX_STEPS / 2);
                CUDA_TRY(launch_fit_lanes(ctx->E, F, B, P, i0, nc, Q, next, order, order_n, defer,
                                          ctx->stream));
                CUDA_TRY(launch_fit_jacobian(ctx->E, F, B, nc, ctx->stream));
                PropQueue q{};
                q.list = defer.list;
                q.list_n = defer.count;
                CUDA_TRY(launch_adjoint_forward_warp(ctx->E, F, model, B, P, i0, nc, ctx->stream, q));
                launches += 2;
            } else if (warps)
                CUDA_TRY(launch_adjoint_forward_warp(ctx->E, F, model, B, P, i0, nc, ctx->stream));
            else CUDA_TRY(launch_adjoint_forward(ctx->E, F, B, P, i0, nc, next, ctx->stream, order));
            prop_event(ctx, false);
            if (jac) {
                CUDA_TRY(launch_adjoint_stm(B, P, i0, nc, ctx->stream));
                launches++;
            }
            CUDA_TRY(launch_adjoint_observe(ctx->E, B, P, i0, nc, ctx->stream));
            launches += 2;
            if (grad) {
                CUDA_TRY(launch_adjoint_backward(B, P, i0, nc, ctx->stream));
                launches++;
            }
        }
        ctx->stats.launches = launches;
    }
    r = stats_end(ctx);
    if (r != KETE_OK) return r;
    stats_collect(ctx);
    if (ctx->h_ctr->error_flags & (1 << 6))
        return fail(ctx, KETE_ERR_BAD_ARG, "observations of a body are not sorted by epoch");
    return KETE_OK;
}

extern "C" int kete_adjoint(kete_ctx *ctx, const double *states, const double *epochs, int64_t n,
                            const kete_obs *obs, int32_t m, const kete_force_model *fm,
                            const kete_survey_opts *opt, double ckpt_days, double *loss,
                            double *grad, double *pred, int32_t *status)
{
    if (ctx && n > 0 && !loss) return fail(ctx, KETE_ERR_BAD_ARG, "loss is required");
    return adjoint_impl(ctx, states, epochs, n, obs, m, fm, opt, ckpt_days, loss, grad, pred,
                        nullptr, status);
}

extern "C" int kete_sky_jacobian(kete_ctx *ctx, const double *states, const double *epochs,
                                 int64_t n, const kete_obs *obs, int32_t m,
                                 const kete_force_model *fm, const kete_survey_opts *opt,
                                 double ckpt_days, double *jac, double *pred, int32_t *status)
{
    if (ctx && n > 0 && !jac) return fail(ctx, KETE_ERR_BAD_ARG, "jac is required");
    return adjoint_impl(ctx, states, epochs, n, obs, m, fm, opt, ckpt_days, nullptr, nullptr,
                        pred, jac, status);
}
