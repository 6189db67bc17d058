// C-ABI runtime of liblbm (declared in include/lbm.h): parameter set-up of
// Section 4, state buffers, CUDA-graph replay of long step sequences and the
// observables round trip.
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_internal.h"

using namespace lbm;

namespace {

constexpr int kGraphSteps = 64;  // steps per captured graph (an even number of launches: keeps buffer parity)

thread_local std::string g_init_error;

}  // namespace

struct lbm_handle_s {
    lbm_params p;
    Derived dv;
    CoefSet coef;
    Geom gm;
    int precision;
    size_t buf_bytes;
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;
    void* buf[2] = {nullptr, nullptr};
    int cur = 0;  // buf[cur] holds B_n, buf[cur ^ 1] holds B_{n-1}
    long t = 0;
    void* phi = nullptr;
    void* snap = nullptr;
    int snap_valid = 0;
    double* partials = nullptr;
    double* obs_dev = nullptr;
    double* obs_host = nullptr;
    int* status_dev = nullptr;
    unsigned* nu_counter = nullptr;  // block counter of the row-parallel Nusselt kernel
    double* nu_dev = nullptr;        // its two results
    double* wall_cols = nullptr;     // two halves of kObsCols temperatures per row, written by observing steps
    cudaStream_t nu_stream = nullptr;  // lbm_step_nusselt's reductions, beside the next step
    cudaEvent_t nu_step[2] = {nullptr, nullptr};  // observing step done, per half of wall_cols
    cudaEvent_t nu_red[2] = {nullptr, nullptr};   // its reduction done
    cudaGraphExec_t gexec[2] = {nullptr, nullptr};
    cudaGraphExec_t steady_exec = nullptr;
    long steady_key[4] = {0, 0, 0, 0};  // K, parity, max_checks, tol bits
    double* steady_dev = nullptr;       // 8 doubles of loop state
    double* extrema_dev = nullptr;      // 3 doubles per column
    int bx = 128, by = 2, npt = 1;
    TileShape tile;     // several steps per launch on chip (steps = 0: not on this lattice)
    DuoShape duo;       // two steps per launch (threads = 0: not on this lattice)
    std::string err;
};

namespace {

int fail(lbm_handle h, int code, const std::string& msg) {
    if (h) h->err = msg;
    else g_init_error = msg;
    return code;
}

int cuda_fail(lbm_handle h, cudaError_t e, const char* where) {
    return fail(h, LBM_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

#define CK(h, expr)                                          \
    do {                                                     \
        cudaError_t e_ = (expr);                             \
        if (e_ != cudaSuccess) return cuda_fail(h, e_, #expr); \
    } while (0)

// Section 4 set-up: Eq. 37 (second occurrence) for tau_nu and tau_T,
// Eq. 24 for nu_e, J = nu_e / nu, U = sqrt(g beta dT L) = Ma c_s, Da = K/L^2,
// Eq. 5 for F_phi.
int derive(const lbm_params* p, Derived* dv, std::string* why) {
    if (p->nx < 5 || p->ny < 5) return *why = "nx and ny must be >= 5", LBM_ERR_ARG;
    if (!(p->phi > 0.0 && p->phi <= 1.0)) return *why = "phi must lie in (0, 1]", LBM_ERR_ARG;
    const bool cooled = p->thermal_bc == LBM_BC_COOLED;
    if (!(p->Da > 0.0) || !(p->Pr > 0.0) || !(p->J > 0.0) || !(p->Ma > 0.0) || !(p->RaI >= 0.0))
        return *why = "Da, Pr, J and Ma must be positive and RaI non-negative", LBM_ERR_ARG;
    if (cooled ? !(p->RaI > 0.0) : !(p->Ra > 0.0))
        return *why = "Ra must be positive (RaI for LBM_BC_COOLED)", LBM_ERR_ARG;
    if (!(p->sigma > 0.0) || !(p->varpi < 1.0) || !(p->varpi > -4.0))
        return *why = "sigma must be positive and varpi in (-4, 1)", LBM_ERR_ARG;
    if (!(p->Th > p->Tc)) return *why = "Th must exceed Tc (with LBM_BC_COOLED, Th - Tc is the scale dT)", LBM_ERR_ARG;
    if (p->precision < LBM_F64 || p->precision > LBM_F32_FRAMED) return *why = "bad precision", LBM_ERR_ARG;
    if (p->use_phi_field && !(p->phi < 1.0))
        return *why = "a porosity field needs a mean porosity below 1", LBM_ERR_ARG;
    if (p->adiabatic_order != 1 && p->adiabatic_order != 2) return *why = "adiabatic_order is 1 or 2", LBM_ERR_ARG;
    if (p->thermal_bc != LBM_BC_SIDE_HEATED && p->thermal_bc != LBM_BC_COOLED)
        return *why = "unknown thermal_bc", LBM_ERR_ARG;
    if (p->collision != LBM_MRT && p->collision != LBM_LBGK) return *why = "unknown collision", LBM_ERR_ARG;
    const double cs2 = 1.0 / 3.0, cs = sqrt(cs2);
    const double L = (double)(p->nx - 1);
    const double cT2 = (4.0 + p->varpi) / 10.0;
    dv->L = L;
    // Eq. 37 (second occurrence); Section 4.2 replaces Ra by Ra_I when Ra = 0
    const double Rs = cooled ? p->RaI : p->Ra;
    dv->tau_nu = 0.5 + p->Ma * p->J * L / cs * sqrt(p->Pr / Rs);
    dv->tau_T = 0.5 + cs2 * (dv->tau_nu - 0.5) / (p->sigma * cT2 * p->Pr);
    if (!(dv->tau_nu > 0.5) || !(dv->tau_T > 0.5)) return *why = "relaxation time not above 1/2", LBM_ERR_ARG;
    dv->nu = cs2 * (dv->tau_nu - 0.5) / p->J;
    dv->dT = p->Th - p->Tc;
    const double U = p->Ma * cs;
    dv->gbeta = U * U / (dv->dT * L);
    dv->K = p->Da * L * L;
    dv->Fphi = p->forchheimer ? 1.75 / sqrt(150.0 * p->phi * p->phi * p->phi) : 0.0;
    // buoyancy reference: the mean wall temperature (Section 4.1), T_c with internal heating only (Section 4.2)
    dv->T0 = cooled ? p->Tc : 0.5 * (p->Th + p->Tc);
    // heat source: Ra_I / Ra = Q L^2 / (alpha_e dT) (Section 2), alpha_e from A9
    const double alpha = p->sigma * cT2 * (dv->tau_T - 0.5);
    if (cooled) dv->Q = dv->dT * alpha / (L * L);
    else if (p->RaI > 0.0) dv->Q = p->RaI / p->Ra * alpha * dv->dT / (L * L);
    else dv->Q = p->Qppp;
    return LBM_OK;
}

struct Rates {
    double s[9], z[5];  // of the flow and thermal moments (Eq. 20, 31)
};
Rates rates_of(const lbm_params* p, const Derived& dv) {
    Rates r;
    if (p->collision == LBM_LBGK) {
        for (int k = 0; k < 9; ++k) r.s[k] = 1.0 / dv.tau_nu;
        for (int k = 0; k < 5; ++k) r.z[k] = 1.0 / dv.tau_T;
    } else {  // Section 4 choices
        r = {{1.0, 1.1, 1.1, 1.0, 1.2, 1.0, 1.2, 1.0 / dv.tau_nu, 1.0 / dv.tau_nu},
             {1.0, 1.0 / dv.tau_T, 1.0 / dv.tau_T, 1.5, 1.5}};
    }
    return r;
}

// Per-cell Ergun (Eq. 5) with d_p^2 fixed by K(phi_bar) = K_bar:
// phi nu / K(phi) = 150 nu (1-phi)^2 / (phi^2 d_p^2), phi F_phi / sqrt K = 1.75 (1-phi) / (phi^2 d_p)
struct Ergun {
    double lin = 0.0, quad = 0.0;
};
Ergun ergun_of(const lbm_params* p, const Derived& dv) {
    Ergun a;
    if (p->phi < 1.0) {
        const double pb = p->phi;
        const double dp2 = 150.0 * dv.K * (1.0 - pb) * (1.0 - pb) / (pb * pb * pb);
        a.lin = 150.0 * dv.nu / dp2;
        a.quad = p->forchheimer ? 1.75 / sqrt(dp2) : 0.0;
    }
    return a;
}

// 8-bit temperature frames: the power of two fq whose 128 steps span the
// largest |T - T0| expected, the wall temperatures plus the conduction
// maximum Q L^2 / (8 alpha_e) of a heat source (alpha_e from A9); a
// larger |T - T0| only saturates the frame, which costs precision, not
// correctness
double frame_quantum(const lbm_params* p, const Derived& dv) {
    const double alpha = p->sigma * (4.0 + p->varpi) / 10.0 * (dv.tau_T - 0.5);
    const double tspan = fmax(fabs(p->Th - dv.T0), fabs(p->Tc - dv.T0)) + fabs(dv.Q) * dv.L * dv.L / (8.0 * alpha);
    return exp2(ceil(log2(tspan / 128.0)));
}

// The direct form's coefficients (FP16 flow storage).
void fill_direct(const lbm_params* p, const Derived& dv, Direct* c) {
    const Rates r = rates_of(p, dv);
    for (int k = 0; k < 9; ++k) {
        c->s[k] = (float)r.s[k];
        c->hs[k] = (float)(1.0 - 0.5 * r.s[k]);
    }
    for (int k = 0; k < 5; ++k) {
        c->z[k] = (float)r.z[k];
        c->hz[k] = (float)(1.0 - 0.5 * r.z[k]);
    }
    c->gbeta = (float)dv.gbeta;
    c->T0 = (float)dv.T0;
    c->dTh = (float)(p->Th - dv.T0);
    c->dTc = (float)(p->Tc - dv.T0);
    c->inv_sigma = (float)(1.0 / p->sigma);
    c->varpi = (float)p->varpi;
    c->inv_csT2 = (float)(10.0 / (4.0 + p->varpi));
    c->wt0 = (float)((1.0 - p->varpi) / 5.0);
    c->wt1 = (float)((4.0 + p->varpi) / 20.0);
    c->psi0 = (float)(dv.Q / p->sigma);
    c->psi3 = (float)(p->varpi * dv.Q / p->sigma);
    c->qhalf = (float)(0.5 * dv.Q / p->sigma);
    c->phi = (float)p->phi;
    c->c_lin = (float)(p->phi * dv.nu / dv.K);  // 0 when Da = INFINITY
    c->c_quad = (float)(p->phi * dv.Fphi / sqrt(dv.K));
    const Ergun a = ergun_of(p, dv);
    c->a_lin = (float)a.lin;
    c->a_quad = (float)a.quad;
    const double fq = frame_quantum(p, dv);
    c->fq = (float)fq;
    c->ifq = (float)(1.0 / fq);
    c->wt1fq = (float)((4.0 + p->varpi) / 20.0) * (float)fq;
}

template <class R>
void fill_coef(const lbm_params* p, const Derived& dv, Coef<R>* c) {
    const Rates r = rates_of(p, dv);
    const double(&s)[9] = r.s, (&z)[5] = r.z;
    c->T0 = (R)dv.T0;
    c->dTh = (R)(p->Th - dv.T0);
    c->dTc = (R)(p->Tc - dv.T0);
    c->varpi = (R)p->varpi;
    c->qhalf = (R)(0.5 * dv.Q / p->sigma);
    c->phi = (R)p->phi;
    const Ergun a = ergun_of(p, dv);
    const double fq = frame_quantum(p, dv);

    // the constants of lbm_core.cuh (see there for the rearranged formulas),
    // formed in FP64; with a porosity field 1 / phi comes with the products
    Coll<R>& k = c->k;
    const bool field = p->use_phi_field != 0;
    const double ip = field ? 1.0 : 1.0 / p->phi;
    const double hs[9] = {1 - s[0] / 2, 1 - s[1] / 2, 1 - s[2] / 2, 1 - s[3] / 2, 1 - s[4] / 2,
                          1 - s[5] / 2, 1 - s[6] / 2, 1 - s[7] / 2, 1 - s[8] / 2};
    double c_lin = p->phi * dv.nu / dv.K, c_quad = p->phi * dv.Fphi / sqrt(dv.K);
    if (sizeof(R) == 4) c_lin = std::min(c_lin, 4.0 * (double)kMostDrag);  // see Por
    k.hb = (R)(0.5 * dv.gbeta * (field ? 1.0 : p->phi));
    k.gb = (R)dv.gbeta;
    k.cc = (R)(0.25 * (field ? (double)(R)a.lin : c_lin));
    k.ec = field ? (R)0 : (R)(0.25 * c_lin + 0.0625 * c_lin * c_lin);
    k.l1 = (R)(0.5 * (field ? (double)(R)a.quad : c_quad));
    k.iphi = (R)(1.0 / p->phi);
    k.niphi = (R)(-1.0 / p->phi);
    k.qhalf = c->qhalf;
    k.a0 = (R)(-(s[0] + 4 * s[1] + 4 * s[2]) / 9);
    k.b0 = (R)((-s[0] - s[1] + 2 * s[2]) / 9);
    k.c0 = (R)((-s[0] + 2 * s[1] - s[2]) / 9);
    k.a1 = (R)((s[1] - s[2]) / 15);
    k.b1 = (R)((s[1] + 2 * s[2]) / 60);
    k.c1 = (R)(-(2 * s[1] + s[2]) / 60);
    k.a2 = (R)(-(hs[1] + hs[2]) * 12 / 9 * ip);
    k.b2 = (R)((2 * hs[2] - hs[1]) / 3 * ip);
    k.c2 = (R)((2 * hs[1] - hs[2]) / 3 * ip);
    k.k7 = (R)(-s[7] / 4);
    k.f7 = (R)(hs[7] * ip);
    k.k8 = (R)(-s[8] / 4);
    k.f8 = (R)(hs[8] / 2 * ip);
    k.s4d = (R)(-s[4] / 12);  // the axis part is exactly -2 times the diagonal one
    k.s4a = (R)-2 * k.s4d;
    k.s6d = (R)(-s[6] / 12);
    k.s6a = (R)-2 * k.s6d;
    k.s3 = (R)(s[3] / 6);
    k.s4 = (R)(s[4] / 6);
    k.s5 = (R)(s[5] / 6);
    k.s6 = (R)(s[6] / 6);
    k.f5 = (R)(hs[5] / 6);
    k.f6 = (R)(hs[6] / 6);
    k.is = (R)(1.0 / p->sigma);
    k.Tis = (R)(dv.T0 / p->sigma);
    k.nis = -k.is;
    k.nTis = -k.Tis;
    const double psi = dv.Q / p->sigma, wt0 = (1.0 - p->varpi) / 5.0, wt1 = (4.0 + p->varpi) / 20.0;
    k.q0 = (R)(wt0 * psi);
    k.q1 = (R)(wt1 * psi);
    k.t1 = (R)(-z[3] / 20 * (1.0 - p->varpi));
    k.h1 = (R)(z[3] / 20 * (4.0 + p->varpi));
    k.t4 = (R)-4 * k.t1;
    k.h4 = (R)-4 * k.h1;
    k.z1 = (R)(-z[1] / 2);
    k.z2 = (R)(-z[2] / 2);
    k.z4 = (R)(-z[4] / 4);
    k.nz4 = -k.z4;
    const double fu = p->precision == LBM_F32 || p->precision == LBM_F32_STORE_F16 ? fq : 1.0;
    k.fu = (R)fu;
    k.ifu = (R)(1.0 / fu);
    k.w1 = (R)wt1 * (R)fu;
    k.nw0 = -(R)wt0 * (R)fu;
    k.nw1 = -k.w1;
    k.wt0 = (R)wt0;
    k.wt1 = (R)wt1;
    k.dTh = c->dTh;
    k.dTc = c->dTc;
}

}  // namespace

#ifdef LBM_BOUNDS_CHECK
// Bounds-checked build: the count of skipped out-of-plane accesses of every
// kernel of this process on this device (the symbol's device address is
// looked up on the host, so that nothing is allocated for it).
__device__ int g_oob_count;
#endif

namespace lbm {
void set_global_error(const std::string& msg) { g_init_error = msg; }

int* oob_counter() {
#ifdef LBM_BOUNDS_CHECK
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_oob_count) != cudaSuccess) return nullptr;
    return (int*)p;
#else
    return nullptr;
#endif
}

int setup_lattice(const lbm_params* p, Derived* dv, CoefSet* cs, Geom* gm, std::string* why) {
    int rc = derive(p, dv, why);
    if (rc != LBM_OK) return rc;
    // row pitch in elements: rows of the flow planes and of the thermal planes
    // both start on 128-byte boundaries (FP64: 16, FP32: 32, FP16 flow: 64)
    const int align = p->precision == LBM_F64 ? 16 : (p->precision == LBM_F32_STORE_F16 ? 64 : 32);
    const long pitch = ((long)p->nx + align - 1) / align * align;
    const long plane = pitch * (long)p->ny;
    if (plane * NPOP >= (1L << 31)) return *why = "lattice too large for 32-bit offsets", LBM_ERR_ARG;
    gm->nx = p->nx;
    gm->ny = p->ny;
    gm->pitch = (int)pitch;
    gm->plane = (int)plane;
    gm->thermal_bc = p->thermal_bc;
    gm->adi_order = p->adiabatic_order;
#ifdef LBM_BOUNDS_CHECK
    gm->oob = oob_counter();
    if (!gm->oob) return *why = "bounds-checked build: no device counter", LBM_ERR_CUDA;
#endif
    fill_coef<double>(p, *dv, &cs->d);
    fill_coef<float>(p, *dv, &cs->f);
    fill_direct(p, *dv, &cs->h);
    return LBM_OK;
}
}  // namespace lbm

namespace {

void free_handle(lbm_handle h) {
    if (!h) return;
    for (int k = 0; k < 2; ++k) {
        if (h->gexec[k]) cudaGraphExecDestroy(h->gexec[k]);
        if (h->buf[k]) cudaFree(h->buf[k]);
    }
    if (h->steady_exec) cudaGraphExecDestroy(h->steady_exec);
    if (h->steady_dev) cudaFree(h->steady_dev);
    if (h->extrema_dev) cudaFree(h->extrema_dev);
    if (h->phi) cudaFree(h->phi);
    if (h->snap) cudaFree(h->snap);
    if (h->partials) cudaFree(h->partials);
    if (h->obs_dev) cudaFree(h->obs_dev);
    if (h->status_dev) cudaFree(h->status_dev);
    if (h->nu_counter) cudaFree(h->nu_counter);
    if (h->nu_dev) cudaFree(h->nu_dev);
    if (h->wall_cols) cudaFree(h->wall_cols);
    for (int b = 0; b < 2; ++b) {
        if (h->nu_step[b]) cudaEventDestroy(h->nu_step[b]);
        if (h->nu_red[b]) cudaEventDestroy(h->nu_red[b]);
    }
    if (h->nu_stream) cudaStreamDestroy(h->nu_stream);
    if (h->obs_host) cudaFreeHost(h->obs_host);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    delete h;
}

StepLaunch step_launch(lbm_handle h, int src, cudaStream_t s) {
    StepLaunch L;
    L.precision = h->precision;
    L.src = h->buf[src];
    L.dst = h->buf[src ^ 1];
    L.phi = h->p.use_phi_field ? h->phi : nullptr;
    L.gm = h->gm;
    L.bx = h->bx;
    L.by = h->by;
    L.npt = h->npt;
    L.status = h->status_dev;
    L.stream = s;
    return L;
}

// The most steps that one launch takes on this lattice where the states
// between are not needed: tiles on chip (lbm_tile.cu), two steps per launch
// (lbm_duo.cu), or one.
int most_steps(lbm_handle h) { return h->tile.steps ? h->tile.steps : h->duo.threads ? 2 : 1; }

// Picks the way (FP32 storage only: FP64 is bound by its arithmetic unit, and FP16
// flow has no such kernels).  Measured, us per step
// with one step per launch / a tile on chip: 64^2 2.2 / 1.0, 128^2 1.9 / 1.3, 200^2
// 2.2 / 1.7, 230^2 2.1 / 1.9, 240^2 2.1 / 2.1, 260^2 2.3 / 2.5, 400^2 3.0 / 3.8, 500 x 100
// 2.1 / 1.9, 1000 x 60 2.1 / 2.1; one / two: 700^2 6.1 / 7.4, 800^2 7.6 / 8.8, 850^2 9.4 /
// 9.2, 900^2 12.0 / 10.8, 1024^2 16.5 / 13.7, 4096^2 272 / 170.
//
// Two steps per launch lose on lattices of a few rows, whose wall tiles outweigh the
// marches (one / two, us per step: 93,750 x 8 9.9 / 16.9, 41,666 x 24 15.4 / 16.3, 62,500 x
// 24 25.6 / 23.7, 500,000 x 8 71 / 87, 250,000 x 16 68 / 65; the line below is within 10 % of
// even from 12 rows to 850), and on columns narrower than a march's warps, from 2^21 nodes on, where
// one step has its border beside its rows, more of them (30 x 33,333 38 / 50, 36 x
// 27,777 53 / 47, 80 x 50,000 97 / 105, 100 x 40,000 100 / 88).
bool twos_worth(long nx, long ny) {
    constexpr long kTwosWorth = 712000, kWallRows = 9;
    return nx * (ny - kWallRows) >= kTwosWorth && nx >= (nx * ny < (1L << 21) ? 34 : 90);
}

cudaError_t choose_steps(lbm_handle h) {
    constexpr double kTileWorth = 1.8;  // us per step of tile_shape's model (240^2: 1.6, 250^2: 1.8)
    if (h->precision != PREC_F32 && h->precision != PREC_F32T) return cudaSuccess;
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const bool field = h->p.use_phi_field != 0;
    const TileShape tile = tile_shape(h->p.nx, h->p.ny, nsm);
    if (tile.steps && tile.us < kTileWorth) {
        h->tile = tile;
        return tile_prepare(h->precision, field);
    }
    if (twos_worth(h->p.nx, h->p.ny)) return duo_shape(h->precision, field, h->gm, nsm, &h->duo);
    return cudaSuccess;
}

cudaError_t launch_steps(lbm_handle h, const StepLaunch& Ls, int steps) {
    if (steps == 1) return launch_step(Ls, h->coef);
    if (!h->tile.steps) return launch_duo(Ls, h->coef, h->duo);
    TileShape s = h->tile;
    s.steps = steps;
    return launch_tile(Ls, h->coef, s);
}

// nsteps steps from buf[cur] on stream s, several per launch where possible;
// the first is launched as a programmatic dependent when pdl_first (a step
// kernel right before it), the others when pdl.  keep_prev: the last step is
// one of its own, so that buf[cur ^ 1] ends up holding B_{n-1}, from which the
// post-stream state is rebuilt.  even: in an even number of launches, which
// leaves cur as it was (nsteps even).
cudaError_t enqueue_steps(lbm_handle h, long nsteps, cudaStream_t s, bool pdl_first, bool pdl, bool keep_prev,
                          bool even) {
    if (nsteps <= 0) return cudaSuccess;
    const long alone = keep_prev ? 1 : 0, together = nsteps - alone;
    long launches = (together + most_steps(h) - 1) / most_steps(h);
    if (even && ((launches + alone) & 1)) ++launches;
    cudaError_t e = cudaSuccess;
    for (long k = 0; k < launches + alone && e == cudaSuccess; ++k) {
        // the steps taken together, shared out evenly
        const int steps = k < launches ? (int)(together * (k + 1) / launches - together * k / launches) : 1;
        StepLaunch Ls = step_launch(h, h->cur, s);
        Ls.pdl = k == 0 ? pdl_first : pdl;
        if ((e = launch_steps(h, Ls, steps)) == cudaSuccess) h->cur ^= 1;
    }
    return e;
}

// The same on the handle's stream, in the handle's launch shape.
int advance(lbm_handle h, long nsteps, bool pdl_first, bool keep_prev) {
    CK(h, enqueue_steps(h, nsteps, h->stream, pdl_first, true, keep_prev, false));
    return LBM_OK;
}

// State B_{-1} = rest everywhere (zero deviations) in both buffers, then one
// step: pulling the rest state and applying the wall rule gives the initial
// post-stream state S_0, whose collision is B_0.
int reset_state(lbm_handle h) {
    CK(h, cudaMemsetAsync(h->buf[0], 0, h->buf_bytes, h->stream));
    CK(h, cudaMemsetAsync(h->buf[1], 0, h->buf_bytes, h->stream));
    CK(h, cudaMemsetAsync(h->status_dev, 0, sizeof(int), h->stream));
    h->cur = 0;
    CK(h, launch_step(step_launch(h, 0, h->stream), h->coef));
    h->cur = 1;
    h->t = 0;
    h->snap_valid = 0;
    return LBM_OK;
}

int capture_graph(lbm_handle h, int parity) {
    cudaGraph_t g = nullptr;
    CK(h, cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
    const int cur = h->cur;
    h->cur = parity;
    cudaError_t e = enqueue_steps(h, kGraphSteps, h->cap_stream, false, true, false, true);
    h->cur = cur;
    cudaError_t e2 = cudaStreamEndCapture(h->cap_stream, &g);
    if (e != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(h, e, "capture step");
    }
    if (e2 != cudaSuccess) return cuda_fail(h, e2, "cudaStreamEndCapture");
    e = cudaGraphInstantiate(&h->gexec[parity], g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaGraphInstantiate");
    return LBM_OK;
}

void drop_graphs(lbm_handle h) {
    for (int k = 0; k < 2; ++k)
        if (h->gexec[k]) {
            cudaGraphExecDestroy(h->gexec[k]);
            h->gexec[k] = nullptr;
        }
    if (h->steady_exec) {
        cudaGraphExecDestroy(h->steady_exec);
        h->steady_exec = nullptr;
    }
}

// The steady-state graph: while (cond) { K steps; check }.
int build_steady_graph(lbm_handle h, long K, long max_checks, double tol) {
    cudaGraph_t g = nullptr;
    CK(h, cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle cond;
    cudaError_t e = cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault);
    cudaGraphNodeParams cp = {};
    cudaGraphNode_t node;
    if (e == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = cond;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        e = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &cp);
    }
    if (e == cudaSuccess) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        e = cudaStreamBeginCaptureToGraph(h->cap_stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            // an even number of launches: every turn of the loop starts from the same buffer
            const int cur = h->cur;
            e = enqueue_steps(h, K, h->cap_stream, false, true, true, true);
            h->cur = cur;
            if (e == cudaSuccess) {
                SteadyCheckLaunch L;
                L.precision = h->precision;
                L.prev = h->buf[h->cur ^ 1];
                L.gm = h->gm;
                L.L = h->dv.L;
                L.dT = h->dv.dT;
                L.status = h->status_dev;
                L.tol = tol;
                L.max_checks = max_checks;
                L.state = h->steady_dev;
                L.cond = cond;
                L.stream = h->cap_stream;
                e = launch_steady_check(L, h->coef);
            }
            cudaGraph_t out = nullptr;
            cudaError_t e2 = cudaStreamEndCapture(h->cap_stream, &out);
            if (e == cudaSuccess) e = e2;
        }
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&h->steady_exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(h, e, "steady-state graph");
    return LBM_OK;
}

}  // namespace

extern "C" {

void lbm_params_default(lbm_params* p, int nx, int ny, double Ra, double Da, double phi) {
    memset(p, 0, sizeof(*p));
    p->nx = nx;
    p->ny = ny;
    p->Ra = Ra;
    p->Da = Da;
    p->phi = phi;
    p->Pr = 1.0;
    p->J = 1.0;
    p->Ma = 0.1;
    p->sigma = 1.0;
    p->varpi = -2.0;
    p->Th = 1.0;
    p->Tc = 0.0;
    p->Qppp = 0.0;
    p->precision = LBM_F32;
    p->use_phi_field = 0;
    p->forchheimer = 1;
    p->thermal_bc = LBM_BC_SIDE_HEATED;
    p->adiabatic_order = 1;
    p->collision = LBM_MRT;
    p->block_x = 0;
    p->block_y = 0;
}

int lbm_init(const lbm_params* p, void* stream, lbm_handle* out) {
    if (!out) return fail(nullptr, LBM_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!p) return fail(nullptr, LBM_ERR_ARG, "params is NULL");
    lbm_handle h = new lbm_handle_s();
    std::string why;
    int rc = setup_lattice(p, &h->dv, &h->coef, &h->gm, &why);
    if (rc != LBM_OK) {
        delete h;
        return fail(nullptr, rc, why);
    }
    h->p = *p;
    h->precision = p->precision;
    const long plane = h->gm.plane;
    // defaults, measured in us per step: FP32 arithmetic two nodes side by side
    // along x, in one-warp blocks on small lattices, which share them out evenly
    // (200^2 2.3 against 2.9 with 64 x 2 threads, 450^2 3.6 / 4.1, 4096^2 the same);
    // FP64 one node per thread on the smallest (64^2 8.4 / 10.5 / 26.7 with one / two
    // along y / two in blocks of 64 x 2), else two along y (257^2 21.3 / 46) as long as
    // its blocks, eight to an SM by their registers, all run at once (a fiftieth to
    // spare), or in so many waves that the last does not count; one between (us for
    // two / one: 257^2 21.1 / 23.0, 264^2 34.7 / 25.0, 280^2 36.4 / 25.7, 400^2 57.8 /
    // 46.7, 512^2 78.7 / 71.9, 800^2 176 / 172, 900^2 222 / 222, 1024^2 276 / 278), from
    // 350^2 on in blocks of 32 x 4 (against 32 x 1: 320^2 34.8 / 31.6, 400^2 46.7 / 48.7)
    const long nodes = (long)p->nx * p->ny;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        nsm = 0;  // (an error that persists shows at the first allocation)
    // blocks of two nodes along y, the border's included
    const long by_two = (p->nx + 31L) / 32 * ((p->ny - 1) / 2) + (p->nx + p->ny) / 16;
    const bool two = nodes >= (1L << 14) && (50 * by_two <= 49 * 8L * nsm || nodes >= 800000);
    const bool f64 = p->precision == LBM_F64, f16 = p->precision == LBM_F32_STORE_F16;
    // (a grid has at most 65535 rows of blocks)
    const bool narrow = p->block_x <= 0 && p->block_y <= 0 && p->ny < 60000 && !f16 && (f64 || nodes < (1L << 20));
    h->bx = p->block_x > 0 ? p->block_x : (p->nx <= 128 || narrow ? 32 : 64);
    const int rows = f64 ? (two || nodes < 110000 ? 1 : 4) : nodes < 100000 ? 1 : 2;
    h->by = p->block_y > 0 ? p->block_y : narrow ? rows : (h->bx >= 128 ? 1 : 128 / h->bx);
    h->npt = p->nodes_per_thread > 0 ? p->nodes_per_thread : f64 ? (two ? 2 : 1) : 3;
    if (h->bx * h->by > 256 || h->bx <= 0 || h->by <= 0 || h->npt > 3) {
        delete h;
        return fail(nullptr, LBM_ERR_ARG, "block_x * block_y must be <= 256 and nodes_per_thread 1, 2 or 3");
    }
    h->stream = (cudaStream_t)stream;
    h->buf_bytes = state_buffer_bytes(p->precision, (int)plane);

    cudaError_t e;
#define CKI(expr)                                                   \
    do {                                                            \
        e = (expr);                                                 \
        if (e != cudaSuccess) {                                     \
            std::string m_ = std::string(#expr) + ": " + cudaGetErrorString(e); \
            free_handle(h);                                         \
            return fail(nullptr, LBM_ERR_CUDA, m_);                 \
        }                                                           \
    } while (0)
    CKI(choose_steps(h));
    CKI(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    CKI(cudaMalloc(&h->buf[0], h->buf_bytes));
    CKI(cudaMalloc(&h->buf[1], h->buf_bytes));
    CKI(cudaMalloc(&h->partials, sizeof(double) * 4 * kReduceBlocks));
    CKI(cudaMalloc(&h->obs_dev, sizeof(double) * 8));
    CKI(cudaMalloc(&h->status_dev, sizeof(int)));
    CKI(cudaMalloc(&h->nu_counter, sizeof(unsigned)));
    CKI(cudaMemsetAsync(h->nu_counter, 0, sizeof(unsigned), h->stream));
    CKI(cudaMalloc(&h->nu_dev, 2 * sizeof(double)));
    CKI(cudaMalloc(&h->wall_cols, sizeof(double) * 2 * kObsCols * (size_t)p->ny));
    CKI(cudaMallocHost(&h->obs_host, sizeof(double) * 8));
    const size_t rsz = p->precision == LBM_F64 ? 8 : 4;
    CKI(cudaMalloc(&h->snap, rsz * 2 * (size_t)p->nx * p->ny));
    if (p->use_phi_field) {
        CKI(cudaMalloc(&h->phi, phi_bytes(p->precision, (int)plane)));
        CKI(cudaMemsetAsync(h->phi, 0, phi_bytes(p->precision, (int)plane), h->stream));
    }
#undef CKI
    if (p->use_phi_field) {
        // until a field is set, every cell holds the mean porosity
        std::string m;
        const size_t n = (size_t)p->nx * p->ny;
        double* tmp = nullptr;
        e = cudaMalloc(&tmp, n * sizeof(double));
        if (e == cudaSuccess) {
            double* host = (double*)malloc(n * sizeof(double));
            for (size_t k = 0; k < n; ++k) host[k] = p->phi;
            e = cudaMemcpyAsync(tmp, host, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
            if (e == cudaSuccess)
                e = launch_convert_phi(tmp, 1, h->phi, h->precision, h->gm, kReduceBlocks, h->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
            free(host);
            cudaFree(tmp);
        }
        if (e != cudaSuccess) {
            m = std::string("porosity fill: ") + cudaGetErrorString(e);
            free_handle(h);
            return fail(nullptr, LBM_ERR_CUDA, m);
        }
    }
    rc = reset_state(h);
    if (rc != LBM_OK) {
        std::string m = h->err;
        free_handle(h);
        return fail(nullptr, rc, m);
    }
    *out = h;
    return LBM_OK;
}

int lbm_set_porous_field(lbm_handle h, const void* phi_dev, int dtype) {
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!h->p.use_phi_field) return fail(h, LBM_ERR_STATE, "handle was created with use_phi_field = 0");
    if (!phi_dev) return fail(h, LBM_ERR_ARG, "phi_dev is NULL");
    if (dtype != LBM_F64 && dtype != LBM_F32) return fail(h, LBM_ERR_ARG, "dtype must be LBM_F64 or LBM_F32");
    // every cell must lie in (0, 1): a 0 would make 1/phi infinite, a 1 or more
    // the Ergun drag zero or negative (Eq. 5); the count lands in the
    // partial-sum scratch, which no other call uses concurrently
    unsigned long long* bad = (unsigned long long*)h->partials;
    unsigned long long nbad = 0;
    CK(h, cudaMemsetAsync(bad, 0, sizeof *bad, h->stream));
    CK(h, launch_count_bad_phi(phi_dev, dtype == LBM_F64, (long)h->p.nx * h->p.ny, bad, kReduceBlocks, h->stream));
    CK(h, cudaMemcpyAsync(h->obs_host, bad, sizeof nbad, cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    memcpy(&nbad, h->obs_host, sizeof nbad);
    if (nbad) return fail(h, LBM_ERR_ARG, std::to_string(nbad) + " porosity values outside (0, 1)");
    CK(h, launch_convert_phi(phi_dev, dtype == LBM_F64, h->phi, h->precision, h->gm, kReduceBlocks, h->stream));
    drop_graphs(h);
    return reset_state(h);
}

int lbm_bounds_check(int* enabled, long* count) {
#ifdef LBM_BOUNDS_CHECK
    if (enabled) *enabled = 1;
    int* p = oob_counter();
    if (!p) return fail(nullptr, LBM_ERR_CUDA, "bounds-checked build: no device counter");
    int v = 0;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(&v, p, sizeof v, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemset(p, 0, sizeof v);
    if (e != cudaSuccess) return fail(nullptr, LBM_ERR_CUDA, std::string("bounds counter: ") + cudaGetErrorString(e));
    if (count) *count = v;
#else
    if (enabled) *enabled = 0;
    if (count) *count = 0;
#endif
    return LBM_OK;
}

int lbm_reset(lbm_handle h) {
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    return reset_state(h);
}

int lbm_tune(lbm_handle h, const char* cache_path, int* block_x, int* block_y, int* nodes_per_thread) {
    TraceRange trace_("lbm_tune");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    char sig[256];
    {
        int dev = 0;
        cudaDeviceProp pr;
        std::string name = "unknown";
        if (cudaGetDevice(&dev) == cudaSuccess && cudaGetDeviceProperties(&pr, dev) == cudaSuccess) name = pr.name;
        for (auto& ch : name)
            if (ch == ' ') ch = '_';
        snprintf(sig, sizeof sig, "step2:%s:p%d:%dx%d:f%d", name.c_str(), h->precision, h->p.nx, h->p.ny,
                 h->p.use_phi_field);
    }
    int best[3] = {h->bx, h->by, h->npt};
    bool cached = false;
    if (cache_path) {
        FILE* fp = fopen(cache_path, "r");
        if (fp) {
            char key[256];
            int a, b, c;
            while (fscanf(fp, "%255s %d %d %d", key, &a, &b, &c) == 4)
                if (strcmp(key, sig) == 0) {
                    best[0] = a;
                    best[1] = b;
                    best[2] = c;
                    cached = true;
                }
            fclose(fp);
        }
    }
    if (!cached) {
        // the shape that the handle has (the library's own, if none was given) first
        const int cand[][3] = {{h->bx, h->by, h->npt},
                               {128, 2, 1}, {64, 4, 1}, {256, 1, 1}, {32, 8, 1}, {32, 1, 1}, {32, 2, 1},
                               {128, 1, 2}, {64, 2, 2}, {128, 2, 2}, {256, 1, 2}, {32, 4, 2}, {32, 1, 2},
                               {32, 2, 2},  {32, 8, 3}, {64, 4, 3}, {128, 2, 3}, {64, 2, 3}, {128, 1, 3},
                               {256, 1, 3}, {32, 1, 3}, {32, 2, 3}};
        // on lattices stepped on chip (lbm_tile.cu) one node per thread or two along y: the
        // one-step kernel takes the last step of a call and the observing ones there
        const bool few = h->tile.steps != 0;
        cudaEvent_t e0, e1;
        CK(h, cudaEventCreate(&e0));
        CK(h, cudaEventCreate(&e1));
        float best_ms = 1e30f;
        drop_graphs(h);
        for (auto& cd : cand) {
            if (few && cd[2] == 3) continue;
            // (a grid has at most 65535 rows of blocks)
            if (h->p.ny / (cd[1] * (cd[2] == 2 ? 2 : 1)) > 65000) continue;
            h->bx = cd[0];
            h->by = cd[1];
            h->npt = cd[2];
            auto singles = [&](long n) {
                for (long k = 0; k < n; ++k) {
                    int r1 = advance(h, 1, k > 0, true);
                    if (r1 != LBM_OK) return r1;
                }
                return (int)LBM_OK;
            };
            int rc = singles(3);
            if (rc != LBM_OK) return rc;
            // 30 steps, or on small lattices as many as take about 2 ms (at most
            // 2000), so that timer resolution and clock ramps do not pick the shape
            long nsteps = 30;
            float ms = 0.f;
            for (int pass = 0; pass < 2; ++pass) {
                CK(h, cudaEventRecord(e0, h->stream));
                if ((rc = singles(nsteps)) != LBM_OK) return rc;
                CK(h, cudaEventRecord(e1, h->stream));
                CK(h, cudaEventSynchronize(e1));
                CK(h, cudaEventElapsedTime(&ms, e0, e1));
                if (pass == 1 || ms >= 2.f) break;
                nsteps = std::min(2000L, (long)(nsteps * 2.f / std::max(ms, 1e-3f)) + 1);
            }
            ms *= 30.f / (float)nsteps;  // per 30 steps
            if (ms < best_ms) {
                best_ms = ms;
                best[0] = cd[0];
                best[1] = cd[1];
                best[2] = cd[2];
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        if (cache_path) {
            FILE* fp = fopen(cache_path, "a");
            if (fp) {
                fprintf(fp, "%s %d %d %d\n", sig, best[0], best[1], best[2]);
                fclose(fp);
            }
        }
    }
    h->bx = best[0];
    h->by = best[1];
    h->npt = best[2];
    drop_graphs(h);
    int rc = reset_state(h);
    if (rc != LBM_OK) return rc;
    if (block_x) *block_x = best[0];
    if (block_y) *block_y = best[1];
    if (nodes_per_thread) *nodes_per_thread = best[2];
    return LBM_OK;
}

int lbm_step(lbm_handle h, long nsteps) {
    TraceRange trace_("lbm_step");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (nsteps < 0) return fail(h, LBM_ERR_ARG, "nsteps < 0");
    long left = nsteps;
    // with several steps per launch the graphs leave no B_{n-1}: at least one step follows them
    const long after = most_steps(h) > 1 ? 1 : 0;
    while (left >= kGraphSteps + after) {
        if (!h->gexec[h->cur]) {
            int rc = capture_graph(h, h->cur);
            if (rc != LBM_OK) return rc;
        }
        CK(h, cudaGraphLaunch(h->gexec[h->cur], h->stream));
        left -= kGraphSteps;  // an even number of launches: cur unchanged
    }
    int rc = advance(h, left, false, true);  // each directly behind the step kernel before it
    if (rc != LBM_OK) return rc;
    h->t += nsteps;
    return LBM_OK;
}

int lbm_observables(lbm_handle h, lbm_obs* out, void* ux_dev, void* uy_dev, void* T_dev, void* p_dev) {
    TraceRange trace_("lbm_observables");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    ObserveLaunch L;
    L.precision = h->precision;
    L.prev = h->buf[h->cur ^ 1];
    L.phi = h->p.use_phi_field ? h->phi : nullptr;
    L.gm = h->gm;
    L.ux = ux_dev;
    L.uy = uy_dev;
    L.T = T_dev;
    L.p = p_dev;
    L.snap = h->snap;
    L.snap_valid = h->snap_valid;
    L.partials = h->partials;
    L.nblocks = kReduceBlocks;
    L.L = h->dv.L;
    L.dT = h->dv.dT;
    L.status = h->status_dev;
    L.out = h->obs_dev;
    L.counter = h->nu_counter;
    L.stream = h->stream;
    CK(h, launch_observe(L, h->coef));
    CK(h, cudaMemcpyAsync(h->obs_host, h->obs_dev, sizeof(double) * 7, cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    h->snap_valid = 1;
    const double* o = h->obs_host;
    const double n = (double)h->p.nx * (double)h->p.ny;
    const int status = o[6] != 0.0 ? LBM_ERR_DIVERGED : LBM_OK;
    if (out) {
        out->t = h->t;
        out->nu_hot = o[0];
        out->nu_cold = o[1];
        out->umax = o[2];
        out->residual = o[2] > 0.0 ? o[3] / o[2] : 0.0;
        out->mass = n + o[4];  // sum_i w_i rho0 = 1 per node
        out->heat = n * h->dv.T0 + o[5];
        out->status = status;
    }
    if (status != LBM_OK) return fail(h, status, "divergence flag raised (non-finite value or |u| >= 1/2)");
    return LBM_OK;
}

namespace {
// The address a kernel writes to for p: p itself for device and managed
// memory, the mapped device address for page-locked host memory, nullptr for
// pageable host memory or a pointer not aligned for doubles.
double* device_writable(double* p) {
    if ((uintptr_t)p % alignof(double) != 0) return nullptr;
    cudaPointerAttributes a;
    memset(&a, 0, sizeof a);
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return p;
    if (a.type == cudaMemoryTypeHost && a.devicePointer) return (double*)a.devicePointer;
    return nullptr;
}

// out: where the kernel writes (nu_hot, nu_cold); device-accessible memory
int enqueue_nusselt(lbm_handle h, double* out) {
    if (4 * kReduceBlocks < 2 * ((h->p.ny + 31) / 32)) return fail(h, LBM_ERR_ARG, "too many rows for the reduction");
    ObserveLaunch L;
    memset(&L, 0, sizeof(L));
    L.precision = h->precision;
    L.prev = h->buf[h->cur ^ 1];
    L.gm = h->gm;
    L.partials = h->partials;
    L.L = h->dv.L;
    L.dT = h->dv.dT;
    L.status = h->status_dev;
    L.out = out;
    L.counter = h->nu_counter;
    L.stream = h->stream;
    CK(h, launch_nusselt(L, h->coef));
    return LBM_OK;
}
}  // namespace

int lbm_nusselt(lbm_handle h, double* nu_hot, double* nu_cold) {
    TraceRange trace_("lbm_nusselt");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    int rc = enqueue_nusselt(h, h->nu_dev);
    if (rc != LBM_OK) return rc;
    CK(h, cudaMemcpyAsync(h->obs_host, h->nu_dev, sizeof(double) * 2, cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    if (nu_hot) *nu_hot = h->obs_host[0];
    if (nu_cold) *nu_cold = h->obs_host[1];
    return LBM_OK;
}

int lbm_nusselt_async(lbm_handle h, double* out2) {
    TraceRange trace_("lbm_nusselt_async");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!out2) return fail(h, LBM_ERR_ARG, "out2 is NULL");
    // device memory and mapped (pinned) host memory: the kernel writes there
    // itself; other host memory gets a copy
    double* direct = device_writable(out2);
    int rc = enqueue_nusselt(h, direct ? direct : h->nu_dev);
    if (rc != LBM_OK) return rc;
    if (!direct) CK(h, cudaMemcpyAsync(out2, h->nu_dev, sizeof(double) * 2, cudaMemcpyDefault, h->stream));
    return LBM_OK;
}

int lbm_step_nusselt(lbm_handle h, long nsteps, double* out) {
    TraceRange trace_("lbm_step_nusselt");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (nsteps < 0) return fail(h, LBM_ERR_ARG, "nsteps < 0");
    if (nsteps == 0) return LBM_OK;
    if (!out) return fail(h, LBM_ERR_ARG, "out is NULL");
    if (4 * kReduceBlocks < 2 * ((h->p.ny + 31) / 32)) return fail(h, LBM_ERR_ARG, "too many rows for the reduction");
    double* dev = device_writable(out);
    if (!dev) return fail(h, LBM_ERR_ARG, "out must be device memory or page-locked host memory, aligned for double");
    if (!h->nu_stream) {
        // the reductions take few blocks: the highest priority lets them in
        // while the next step's blocks are still being dispatched
        int least = 0, greatest = 0;
        CK(h, cudaDeviceGetStreamPriorityRange(&least, &greatest));
        CK(h, cudaStreamCreateWithPriority(&h->nu_stream, cudaStreamNonBlocking, greatest));
        for (int b = 0; b < 2; ++b) {
            CK(h, cudaEventCreateWithFlags(&h->nu_step[b], cudaEventDisableTiming));
            CK(h, cudaEventCreateWithFlags(&h->nu_red[b], cudaEventDisableTiming));
        }
    }
    ObserveLaunch L;
    memset(&L, 0, sizeof(L));
    L.precision = h->precision;
    L.gm = h->gm;
    L.partials = h->partials;
    L.L = h->dv.L;
    L.dT = h->dv.dT;
    L.status = h->status_dev;
    L.counter = h->nu_counter;
    L.stream = h->nu_stream;
    // step k writes half k & 1 of wall_cols; its reduction runs on nu_stream
    // beside step k + 1 (which writes the other half), and step k + 2 waits
    // for it before rewriting the half
    cudaError_t e = cudaSuccess;
    const char* where = "";
    for (long k = 0; k < nsteps; ++k) {
        const int b = (int)(k & 1);
        double* cols = h->wall_cols + (size_t)b * kObsCols * h->p.ny;
        if (k >= 2 && (e = cudaStreamWaitEvent(h->stream, h->nu_red[b], 0)) != cudaSuccess) {
            where = "wait for the reduction two steps back";
            break;
        }
        StepLaunch Ls = step_launch(h, h->cur, h->stream);
        Ls.obs = cols;
        if ((e = launch_step(Ls, h->coef)) != cudaSuccess) {
            where = "observing step";
            break;
        }
        h->cur ^= 1;
        h->t += 1;
        if ((e = cudaEventRecord(h->nu_step[b], h->stream)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(h->nu_stream, h->nu_step[b], 0)) != cudaSuccess) {
            where = "hand-over to the reduction stream";
            break;
        }
        L.prev = h->buf[h->cur ^ 1];
        L.obs = cols;
        L.out = dev + 2 * k;
        if ((e = launch_nusselt(L, h->coef)) != cudaSuccess ||
            (e = cudaEventRecord(h->nu_red[b], h->nu_stream)) != cudaSuccess) {
            where = "wall-column reduction";
            break;
        }
    }
    // the caller's stream reaches this point once the last reduction is done
    // (the reductions run in order on nu_stream)
    if (e == cudaSuccess && (e = cudaStreamWaitEvent(h->stream, h->nu_red[(nsteps - 1) & 1], 0)) != cudaSuccess)
        where = "join of the reduction stream";
    if (e != cudaSuccess) {
        (void)cudaStreamSynchronize(h->nu_stream);  // no reduction keeps running beside later work
        return cuda_fail(h, e, where);
    }
    return LBM_OK;
}

int lbm_adjoint_step(lbm_handle h, long nsteps, long ckpt_every, double* J, void* dJdphi_dev) {
    TraceRange trace_("lbm_adjoint_step");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!h->p.use_phi_field) return fail(h, LBM_ERR_STATE, "the adjoint needs a handle created with use_phi_field = 1");
    if (h->precision != LBM_F64 && h->precision != LBM_F32 && h->precision != LBM_F32_FRAMED)
        return fail(h, LBM_ERR_ARG, "the adjoint runs in LBM_F64, LBM_F32 or LBM_F32_FRAMED");
    if (h->p.adiabatic_order != 1) return fail(h, LBM_ERR_ARG, "the adjoint supports first-order adiabatic walls");
    if (nsteps < 1 || ckpt_every < 1 || !dJdphi_dev) return fail(h, LBM_ERR_ARG, "need nsteps >= 1, ckpt_every >= 1, output");
    // N / K kept states and 2 (K - 1) recomputed ones take the least memory at K =
    // sqrt(N / 2); a longer interval would save the forward sweep's copies, but
    // allocating, mapping and freeing its states takes longer than they do (512^2,
    // N = 600: 1.0 GB at K = 17 against 3.0 GB and 2.2 ms of a call at K = 100)
    const long N = nsteps, best = std::max(1L, std::lround(std::sqrt(0.5 * (double)N)));
    const long K = std::min({ckpt_every, N, best});
    const long nseg = (N + K - 1) / K;
    const size_t rsz = h->precision == LBM_F64 ? sizeof(double) : sizeof(float);
    // one allocation: kept states, two halves of K - 1 recomputed states (one segment
    // is recomputed while the next is reversed), two adjoint states, the gradient
    auto whole = [](size_t bytes) { return (bytes + 255) & ~(size_t)255; };
    const size_t of_ckpt = whole((size_t)nseg * h->buf_bytes), of_seg = whole(2 * (size_t)(K - 1) * h->buf_bytes),
                 of_madj = whole(2 * (size_t)h->gm.plane * NPOP * rsz);
    char* ckpt = nullptr;
    auto release = [&]() { cudaFree(ckpt); };
    cudaError_t e = cudaMalloc(&ckpt, of_ckpt + of_seg + of_madj + sizeof(double) * (size_t)h->p.nx * h->p.ny);
    void *const seg = ckpt + of_ckpt, *const madj = ckpt + of_ckpt + of_seg;
    double* const gphi = (double*)(ckpt + of_ckpt + of_seg + of_madj);
    if (e != cudaSuccess) {
        release();
        return cuda_fail(h, e, "adjoint buffers");
    }
    // forward sweep from the initial state, keeping B_{sK-1} (state index j = sK)
    int rc = reset_state(h);
    if (rc == LBM_OK) {
        e = cudaMemsetAsync(ckpt, 0, h->buf_bytes, h->stream);  // j = 0: the rest state B_{-1}
        if (e != cudaSuccess) rc = cuda_fail(h, e, "adjoint forward sweep");
        // runs of steps between the kept states: before step t (buf[cur] holds
        // B_t, state index j = t + 1) the state is kept when j % K == 0, j < N
        for (long t = 0; t < N && rc == LBM_OK;) {
            const long j = t + 1;
            const bool copy = j % K == 0 && j <= N - 1;
            if (copy && (e = cudaMemcpyAsync(ckpt + (size_t)(j / K) * h->buf_bytes, h->buf[h->cur],
                                             h->buf_bytes, cudaMemcpyDeviceToDevice, h->stream)) != cudaSuccess) {
                rc = cuda_fail(h, e, "adjoint forward sweep");
                break;
            }
            const long next = (j / K + 1) * K - 1;  // the next step that keeps its input state
            const long upto = next <= N - 2 ? next : N;
            // directly behind the previous step kernel; only the last run's B_{N-1} is read
            rc = advance(h, upto - t, t > 0 && !copy, upto == N);
            t = upto;
        }
        h->t = N;
    }
    if (rc == LBM_OK) {
        double nuh = 0.0;
        rc = lbm_nusselt(h, &nuh, nullptr);
        if (rc == LBM_OK && J) *J = nuh;
    }
    if (rc == LBM_OK) {
        AdjointJob A;
        A.precision = h->precision;
        A.gm = h->gm;
        A.coef = h->precision == LBM_F64 ? (const void*)&h->coef.d : (const void*)&h->coef.f;
        A.nsteps = N;
        A.ckpt_every = K;
        A.buf_bytes = h->buf_bytes;
        A.ckpt = ckpt;
        A.seg = seg;
        A.madj = madj;
        A.gphi = gphi;
        A.phi = h->phi;
        A.status = h->status_dev;
        A.L = h->dv.L;
        A.dT = h->dv.dT;
        A.out = dJdphi_dev;
        A.bx = h->bx;  // the handle's (tuned) launch shape, as in the forward sweep
        A.by = h->by;
        A.npt = h->npt;
        A.stream = h->stream;
        e = launch_adjoint_sweep(A);
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) rc = cuda_fail(h, e, "adjoint reverse sweep");
    }
    release();
    return rc;
}

int lbm_run_steady(lbm_handle h, double tol, long check_every, long max_steps, long* steps_taken, double* change) {
    TraceRange trace_("lbm_run_steady");
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!(tol > 0.0) || check_every < 1 || max_steps < 1) return fail(h, LBM_ERR_ARG, "need tol > 0, check_every >= 1, max_steps >= 1");
    const long K = (check_every + 1) / 2 * 2;  // even: the captured buffers return to their parity
    const long max_checks = (max_steps + K - 1) / K;
    if (!h->steady_dev) CK(h, cudaMalloc(&h->steady_dev, 8 * sizeof(double)));
    long tolbits;
    memcpy(&tolbits, &tol, sizeof tolbits);
    const long key[4] = {K, h->cur, max_checks, tolbits};
    if (!h->steady_exec || memcmp(key, h->steady_key, sizeof key) != 0) {
        if (h->steady_exec) cudaGraphExecDestroy(h->steady_exec);
        h->steady_exec = nullptr;
        int rc = build_steady_graph(h, K, max_checks, tol);
        if (rc != LBM_OK) return rc;
        memcpy(h->steady_key, key, sizeof key);
    }
    CK(h, cudaMemsetAsync(h->steady_dev, 0, 8 * sizeof(double), h->stream));
    CK(h, cudaGraphLaunch(h->steady_exec, h->stream));
    double st[8];
    CK(h, cudaMemcpyAsync(st, h->steady_dev, sizeof st, cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    const long steps = (long)st[3] * K;
    h->t += steps;
    h->snap_valid = 0;
    if (steps_taken) *steps_taken = steps;
    if (change) *change = st[2];
    if ((int)st[4] == 2) return fail(h, LBM_ERR_DIVERGED, "divergence flag raised during the steady-state loop");
    return LBM_OK;
}

int lbm_field_extrema(lbm_handle h, double* T_max, double* psi_min, double* psi_max) {
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!h->extrema_dev) CK(h, cudaMalloc(&h->extrema_dev, 3 * sizeof(double) * (size_t)h->p.nx));
    CK(h, launch_extrema(h->precision, h->buf[h->cur ^ 1], h->p.use_phi_field ? h->phi : nullptr, h->gm, h->coef,
                         h->extrema_dev, h->stream));
    std::vector<double> col(3 * (size_t)h->p.nx);
    CK(h, cudaMemcpyAsync(col.data(), h->extrema_dev, sizeof(double) * col.size(), cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    double tm = -INFINITY, pmn = 0.0, pmx = 0.0;
    for (int x = 0; x < h->p.nx; ++x) {
        tm = fmax(tm, col[3 * x]);
        pmn = fmin(pmn, col[3 * x + 1]);
        pmx = fmax(pmx, col[3 * x + 2]);
    }
    if (T_max) *T_max = tm;
    if (psi_min) *psi_min = pmn;
    if (psi_max) *psi_max = pmx;
    return LBM_OK;
}

int lbm_read_state(lbm_handle h, double* f_dev, double* g_dev) {
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    if (!f_dev || !g_dev) return fail(h, LBM_ERR_ARG, "f_dev and g_dev are required");
    ReadStateLaunch L;
    L.precision = h->precision;
    L.prev = h->buf[h->cur ^ 1];
    L.phi = h->p.use_phi_field ? h->phi : nullptr;
    L.gm = h->gm;
    L.f = f_dev;
    L.g = g_dev;
    L.nblocks = kReduceBlocks;
    L.stream = h->stream;
    CK(h, launch_read_state(L, h->coef));
    return LBM_OK;
}

int lbm_checkpoint_size(lbm_handle h, size_t* bytes) {
    if (!h || !bytes) return fail(h, LBM_ERR_ARG, "handle and bytes are required");
    *bytes = sizeof(CkptHeader) + h->buf_bytes;
    return LBM_OK;
}

// Host-to-device copy of a checkpoint's payload.  From pinned memory the copy
// runs about 8 % faster from a 256-byte-aligned host address (211 against
// 194 GB/s measured on GB300 at the 40-byte header's offset), so the bytes
// before the next boundary go first, apart.
static cudaError_t copy_in(void* dst, const char* src, size_t n, cudaStream_t s) {
    size_t head = (256 - ((uintptr_t)src & 255)) & 255;
    if (head > n) head = n;
    if (head) {
        cudaError_t e = cudaMemcpyAsync(dst, src, head, cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) return e;
    }
    return cudaMemcpyAsync((char*)dst + head, src + head, n - head, cudaMemcpyHostToDevice, s);
}

int lbm_save(lbm_handle h, void* host, size_t bytes) {
    TraceRange trace_("lbm_save");
    if (!h || !host) return fail(h, LBM_ERR_ARG, "handle and host buffer are required");
    size_t need = sizeof(CkptHeader) + h->buf_bytes;
    if (bytes < need) return fail(h, LBM_ERR_ARG, "checkpoint buffer too small");
    CkptHeader hd;
    memset(&hd, 0, sizeof hd);
    memcpy(hd.magic, "LBMCKPT", 8);
    hd.version = 3;
    hd.nx = h->p.nx;
    hd.ny = h->p.ny;
    hd.precision = h->precision;
    hd.t = h->t;
    hd.payload = (long)h->buf_bytes;
    memcpy(host, &hd, sizeof hd);
    // B_{n-1} alone: the post-stream state S_n is pulled from it, and B_n is collide(S_n)
    CK(h, cudaMemcpyAsync((char*)host + sizeof hd, h->buf[h->cur ^ 1], h->buf_bytes, cudaMemcpyDeviceToHost,
                          h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

int lbm_load(lbm_handle h, const void* host, size_t bytes) {
    TraceRange trace_("lbm_load");
    if (!h || !host) return fail(h, LBM_ERR_ARG, "handle and host buffer are required");
    CkptHeader hd;
    if (bytes < sizeof hd) return fail(h, LBM_ERR_ARG, "checkpoint buffer too small");
    memcpy(&hd, host, sizeof hd);
    if (memcmp(hd.magic, "LBMCKPT", 8) != 0 || hd.version < 1 || hd.version > 3)
        return fail(h, LBM_ERR_ARG, "not a checkpoint");
    if (!ckpt_layout_current(hd.version, hd.precision))
        return fail(h, LBM_ERR_ARG, "checkpoint written with an older storage layout of this precision");
    const long nbuf = hd.version == 1 ? 2 : 1;
    if (hd.nx != h->p.nx || hd.ny != h->p.ny || hd.precision != h->precision ||
        hd.payload != (long)(nbuf * h->buf_bytes) || bytes < sizeof hd + nbuf * h->buf_bytes)
        return fail(h, LBM_ERR_ARG, "checkpoint does not match this handle");
    const char* src = (const char*)host + sizeof hd;
    for (long k = 0; k < nbuf; ++k) CK(h, copy_in(h->buf[k], src + k * h->buf_bytes, h->buf_bytes, h->stream));
    if (nbuf == 1) {
        // B_n = collide(pull(B_{n-1}) + wall rule): the step this handle would have taken
        CK(h, launch_step(step_launch(h, 0, h->stream), h->coef));
    }
    CK(h, cudaStreamSynchronize(h->stream));
    h->cur = 1;
    h->t = hd.t;
    h->snap_valid = 0;
    return LBM_OK;
}

int lbm_query(lbm_handle h, long* t, int* status) {
    if (!h) return fail(nullptr, LBM_ERR_ARG, "handle is NULL");
    int st = 0;
    CK(h, cudaMemcpyAsync(&st, h->status_dev, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    if (t) *t = h->t;
    if (status) *status = st ? LBM_ERR_DIVERGED : LBM_OK;
    return LBM_OK;
}

int lbm_destroy(lbm_handle h) {
    if (!h) return LBM_OK;
    cudaError_t e = cudaStreamSynchronize(h->stream);
    free_handle(h);
    if (e != cudaSuccess) return fail(nullptr, LBM_ERR_CUDA, cudaGetErrorString(e));
    return LBM_OK;
}

const char* lbm_last_error(lbm_handle h) { return h ? h->err.c_str() : g_init_error.c_str(); }

}  // extern "C"
