// sgpe_api.cu -- the C ABI of libsgpe (see include/sgpe.h): context, workspace
// layout, parameter checks, step orchestration and CUDA-graph replay.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <algorithm>
#include <complex>
#include <vector>
#include <tuple>

#include "../../include/sgpe.h"
#include "sgpe_device.cuh"
#include "sgpe_kernels.cuh"
#include "sgpe_launch.h"
#include "sgpe_socn.cuh"

using namespace sgpe;

namespace sgpe {
Geometry make_geometry(int dim, int nx, int ny, int esz) {
    Geometry g;
    g.dim = dim;
    g.nx = nx;
    g.ny = ny;
    g.esz = esz;
    // x sweep: register kernel (one warp per line) up to kRegMaxN points; longer
    // lines: one block of long_warps(nx) warps per line, the line staged in
    // shared memory (32 * nw chunks of kLongC + 1 entries)
    g.reg_x = nx <= kRegMaxN;
    g.fused = dim == 2 && g.reg_x;
    g.wx = long_warps(nx);  // (the register kernels take one warp a line)
    g.smem_x = (size_t)32 * g.wx * (kLongC + 1) * esz;
    g.blocks_x = 3 * ny;
    // y sweep: register kernel up to kRegMaxN points; longer columns: tiles of wy
    // adjacent columns (a 32-byte row segment where the block stays within
    // kLongMaxWarps warps), long_warps(ny) warps per column
    g.reg_y = ny <= kRegMaxN;
    const int nwy = long_warps(ny);
    // a power of two (the kernel splits a staging index into row and column by shift and mask)
    int wy = std::max(1, std::min(32 / esz, kLongMaxWarps / nwy));
    while (wy & (wy - 1)) wy &= wy - 1;
    g.wy = g.reg_y ? 1 : wy;
    g.smem_y = g.reg_y ? 0 : (size_t)g.wy * (32 * nwy * (kLongC + 1) + long_col_pad(esz, g.wy)) * esz;
    g.blocks_y = dim == 2 ? 3 * ceil_div(nx, g.reg_y ? cny_cols_per_warp(chunk_len(ny), esz) : g.wy) : 0;
    const int mid_min = esz == 8 ? kMidMinN : kMidMinN16;
    g.tiled = dim == 2 && nx >= mid_min && ny >= mid_min && g.reg_x && g.reg_y;
    g.tile_rt = ny <= kTileShortMaxN ? kTileRealShort : kTileReal;
    g.blocks_yt = dim == 2 && (!g.reg_y || g.tiled) ? 3 * ceil_div(nx, 32) * ceil_div(ny, kLongC * g.tile_rt) : 0;
    g.blocks_pair = dim == 2 && esz == 16 ? 3 * pair_parts(nx, ny) : 0;
    g.blocks_obs = ceil_div(nx, 32) * ceil_div(ny, 4);
    g.blocks_norm = kNormBlocks;
    return g;
}
}  // namespace sgpe

// Call f with a value of the arithmetic type of precision p (double, float or
// the double-float pair).
template <typename F> static auto with_prec(sgpe_precision p, F&& f) {
    if (p == SGPE_C128) return f(double(0));
    if (p == SGPE_C64) return f(float(0));
    return f(df(0));
}

struct GraphKey {
    int imag, count;
    const double* omega;
    bool operator<(const GraphKey& o) const {
        return std::tie(imag, count, omega) < std::tie(o.imag, o.count, o.omega);
    }
};

struct sgpe_ctx {
    int dim, nx, ny;
    double dx, dy;
    sgpe_precision prec;
    int esz;
    cudaStream_t stream;
    int device;
    Geometry geo;
    // caller-owned buffers
    void* psi;
    unsigned char* work;
    // workspace carve-up
    DevScalars* sc;
    void* mid;
    TabSet tabs[3][2];  // [mode: 0 imag, 1 real, 2 real with -dt (adjoint)][axis: 0 x, 1 y]
    void* us[3][2];     // the start corrections of the constant-factor form (long lines)
    double* partials;
    // SO by Crank-Nicolson (params.so_mode = 1): skew tables [mode: 0 imag, 1 real][axis][m: +1, -1][4]
    // and the line families [mode][axis]
    void* tabs_so[2][2][2][4];
    SoCnLines socn[2][2];
    bool socn_y;  // 2D with eta != 0: a y part
    // parameters
    bool have_params;
    sgpe_params params;
    KParams kp;
    KParams kp_half;  // the same with dt/2 (Strang splitting)
    // graph cache
    std::map<GraphKey, cudaGraphExec_t> graphs;
    bool graphs_ok;
    char err[512];
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Message of the last failed sgpe_init_grid on this host thread (no context exists then).
static thread_local char g_init_err[256] = "";

namespace sgpe {
void set_thread_error(const char* msg) { snprintf(g_init_err, sizeof(g_init_err), "%s", msg); }
}  // namespace sgpe

static sgpe_status fail(sgpe_ctx* c, sgpe_status st, const char* fmt, ...) {
    if (c) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(c->err, sizeof(c->err), fmt, ap);
        va_end(ap);
    }
    return st;
}

static sgpe_status cuda_fail(sgpe_ctx* c, cudaError_t e, const char* where) {
    return fail(c, SGPE_ECUDA, "%s: %s", where, cudaGetErrorString(e));
}

#define CK(expr, where)                                   \
    do {                                                  \
        cudaError_t e_ = (expr);                          \
        if (e_ != cudaSuccess) return cuda_fail(c, e_, where); \
    } while (0)

struct Layout {
    size_t sc, mid, tabs[3][2][4], us[3][2], tabs_so[2][2][2][4], partials, total;
};

static Layout layout_of(const sgpe_ctx* c) {
    Layout L;
    size_t off = 0;
    L.sc = off;
    off = align256(off + sizeof(DevScalars));
    L.mid = off;
    off = align256(off + (size_t)3 * c->nx * c->ny * c->esz);
    for (int m = 0; m < 3; m++)
        for (int a = 0; a < 2; a++) {
            int n = a == 0 ? c->nx : c->ny;
            for (int k = 0; k < 4; k++) {
                L.tabs[m][a][k] = off;
                off = align256(off + (size_t)table_len(n) * c->esz);
            }
            L.us[m][a] = off;
            off = align256(off + (size_t)(n > kRegMaxN || c->geo.tiled ? kUniMaxS : 1) * c->esz);
        }
    for (int m = 0; m < 2; m++)
        for (int a = 0; a < 2; a++) {
            const int n = a == 0 ? c->nx : c->ny;
            for (int q = 0; q < 2; q++)
                for (int k = 0; k < 4; k++) {
                    L.tabs_so[m][a][q][k] = off;
                    off = align256(off + (size_t)table_len(n) * c->esz);
                }
        }
    L.partials = off;
    size_t np = 0;
    const Geometry& g = c->geo;
    size_t cand[6] = {(size_t)g.blocks_x * 3, (size_t)g.blocks_y * 3, (size_t)g.blocks_obs * kObsAcc,
                      (size_t)g.blocks_norm * 3, (size_t)g.blocks_yt * 3, (size_t)g.blocks_pair};
    for (int i = 0; i < 6; i++)
        if (cand[i] > np) np = cand[i];
    off = align256(off + np * sizeof(double));
    L.total = off;
    return L;
}

static void invalidate_graphs(sgpe_ctx* c) {
    for (auto& kv : c->graphs) cudaGraphExecDestroy(kv.second);
    c->graphs.clear();
}

namespace sgpe {
const char* check_params(const sgpe_params* p) {
    if (!(p->dt > 0.0) || !isfinite(p->dt)) return "dt must be positive and finite";
    if (p->so_type < 0 || p->so_type > 3) return "so_type must be 0..3";
    if (p->renorm < 0 || p->renorm > 2) return "renorm must be 0, 1 or 2";
    if (p->renorm == 2 && !(fabs(p->mag) < 1.0)) return "renorm 2 needs |mag| < 1";
    if (p->split != 0 && p->split != 1) return "split must be 0 (Lie) or 1 (Strang)";
    if (p->so_mode != 0 && p->so_mode != 1) return "so_mode must be 0 (Euler) or 1 (Crank-Nicolson)";
    const double vals[] = {p->c0, p->c2, p->gamma, p->omega, p->wx, p->wy, p->mag};
    for (double v : vals)
        if (!isfinite(v)) return "non-finite parameter";
    return nullptr;
}

KParams make_kparams(int dim, int nx, int ny, double dx, double dy, const sgpe_params* p) {
    KParams k;
    memset(&k, 0, sizeof(k));
    k.dim = dim;
    k.nx = nx;
    k.ny = ny;
    k.dx = dx;
    k.dy = dy;
    k.dt = p->dt;
    const double gt = p->gamma / sqrt(2.0);
    k.so_case = 0;
    if (p->so_type != 0 && p->gamma != 0.0) {
        if (dim == 1) {
            k.so_case = p->so_type;
            k.sx = (p->so_type == 3 ? p->gamma : gt) / (2.0 * dx);
            k.sy = 0.0;
        } else {
            double eta = p->so_type == 1 ? 1.0 : (p->so_type == 2 ? -1.0 : 0.0);
            k.so_case = 4;
            k.sx = gt / (2.0 * dx);
            k.sy = gt * eta / (2.0 * dy);
        }
    }
    k.hx = p->dt * k.sx;
    k.hy = p->dt * k.sy;
    k.c0 = p->c0;
    k.c2 = p->c2;
    k.wx2h = 0.5 * p->wx * p->wx;
    k.wy2h = dim == 2 ? 0.5 * p->wy * p->wy : 0.0;
    k.vx = k.wx2h * dx * dx;
    k.vy = k.wy2h * dy * dy;
    k.omega_t = p->omega / sqrt(2.0);
    k.wx = p->wx;
    k.wy = dim == 2 ? p->wy : 0.0;
    k.cell = dim == 2 ? dx * dy : dx;
    k.renorm = p->renorm;
    k.mag = p->mag;
    k.split = p->split;
    k.so_mode = p->so_mode;
    return k;
}
}  // namespace sgpe

namespace sgpe {
// The pivot limit: the root u of u^2 - (1 + 2bt) u + bt^2 with |u| > |bt| (as Launcher::uni).
static std::complex<double> pivot_limit(std::complex<double> b) {
    using C = std::complex<double>;
    const C d = 1.0 + 2.0 * b, disc = std::sqrt(d * d - 4.0 * b * b), alt = (d - disc) * 0.5;
    C u = (d + disc) * 0.5;
    if (std::abs(alt) > std::abs(u)) u = alt;
    for (int k = 0; k < 8; k++) u = d - b * b / u;
    return u;
}

// v0 g^k into wr, wi until |g|^k < 2^-bits: the taps needed, or 0 where room does not hold
// them. kp (nullable): those with |g|^k >= 2^-26.
static int geometric_taps(std::complex<double> v, std::complex<double> g, int bits, int room, double* wr, double* wi,
                          int* kp) {
    double w = 1.0;
    int kt = 0;
    for (; kt < room && !(w < std::ldexp(1.0, -bits)); kt++) {
        if (kp && !(w < std::ldexp(1.0, -26))) *kp = kt + 1;
        wr[kt] = v.real();
        wi[kt] = v.imag();
        v *= g;
        w *= std::abs(g);
    }
    return w < std::ldexp(1.0, -bits) ? kt : 0;
}

// (lines shorter than the taps would need images of images)
PairHost pair_form(int n, double bre, double bim) {
    PairHost h{};
    const std::complex<double> b(bre, bim), u = pivot_limit(b), g = b / u;
    const int kt = geometric_taps(2.0 * b / (u * (1.0 + g)), g, 56, kPairTaps, h.wr, h.wi, &h.kp);
    if (h.kp <= kPairPairTaps && n > kPairTaps) h.kt = kt;
    return h;
}
ConvHost conv_form(int n, double bre, double bim) {
    ConvHost h{};
    const std::complex<double> b(bre, bim), u = pivot_limit(b), g = b / u;
    const int kt = geometric_taps(2.0 * b / (u * (1.0 - g * g)), g, 34, kConvTaps, h.wr, h.wi, nullptr);
    if (n > kConvTaps) h.kt = kt;
    return h;
}
}  // namespace sgpe

// The SO-CN line families and their skew tables for the current parameters:
// the SO time step is dt (dt/2 with Strang splitting); along each family the
// operator is g S p (1D: gamma Sigma_(x|y|z); 2D: -gamma Sigma_y along x,
// eta gamma Sigma_x along y) and a_(+1) = -i z g / (4 h).
static void spin_eigvecs(int which, double* ur, double* ui) {
    // columns: eigenvectors of m = +1, 0, -1 (U[j][k] at 3j + k)
    const double r = 0.70710678118654752440;
    for (int q = 0; q < 9; q++) ur[q] = ui[q] = 0.0;
    if (which == 0) {  // Sigma_x
        const double u[9] = {0.5, r, 0.5, r, 0.0, -r, 0.5, -r, 0.5};
        for (int q = 0; q < 9; q++) ur[q] = u[q];
    } else if (which == 1) {  // Sigma_y
        const double u[9] = {0.5, r, 0.5, 0.0, 0.0, 0.0, -0.5, r, -0.5};
        for (int q = 0; q < 9; q++) ur[q] = u[q];
        ui[3] = r;   // U[1][0] = i/sqrt2
        ui[5] = -r;  // U[1][2] = -i/sqrt2
    } else {  // Sigma_z
        ur[0] = ur[4] = ur[8] = 1.0;
    }
}

// The table job of an n-point line with tables t.
static CoefJob coef_job(void* const* t, int n, double bre, double bim, int skew) {
    return CoefJob{t[0], t[1], t[2], t[3], n, chunk_len(n), table_len(n), n > kRegMaxN ? 1 : 0, skew, bre, bim};
}

// (its table jobs are added to jobs)
static sgpe_status build_socn(sgpe_ctx* c, CoefJob* jobs, int* njobs) {
    const sgpe_params& p = c->params;
    c->socn_y = false;
    if (c->kp.so_case == 0 || c->nx > kRegMaxN || (c->dim == 2 && c->ny > kRegMaxN)) return SGPE_OK;
    const double dts = p.split ? 0.5 * p.dt : p.dt;
    const double eta = p.so_type == 1 ? 1.0 : (p.so_type == 2 ? -1.0 : 0.0);
    c->socn_y = c->dim == 2 && eta != 0.0;
    for (int a = 0; a < c->dim; a++) {
        int which;
        double g, h = a == 0 ? c->dx : c->dy;
        if (c->dim == 1) {
            which = p.so_type - 1;
            g = p.gamma;
        } else if (a == 0) {
            which = 1;
            g = -p.gamma;
        } else {
            which = 0;
            g = eta * p.gamma;
        }
        for (int m = 0; m < 2; m++) {
            SoCnLines& L = c->socn[m][a];
            spin_eigvecs(which, L.ur, L.ui);
            L.which = which;
            const double q = dts * g / (4.0 * h);
            L.are = m == 0 ? 0.0 : q;   // imaginary time: a = -i dt g/(4h)
            L.aim = m == 0 ? -q : 0.0;  // real time: a = dt g/(4h)
            L.plane = (long long)c->nx * c->ny;
            if (a == 0) {
                L.n = c->nx;
                L.nlines = c->ny;
                L.stride = 1;
                L.lstride = c->nx;
            } else {
                L.n = c->ny;
                L.nlines = c->nx;
                L.stride = c->nx;
                L.lstride = 1;
            }
            if (a == 1 && !c->socn_y) continue;
            jobs[(*njobs)++] = coef_job(c->tabs_so[m][a][0], L.n, L.are, L.aim, 1);
            jobs[(*njobs)++] = coef_job(c->tabs_so[m][a][1], L.n, -L.are, -L.aim, 1);
        }
    }
    return SGPE_OK;
}

extern "C" {

sgpe_status sgpe_init_grid(sgpe_ctx** out, int dim, int nx, int ny, double dx, double dy, sgpe_precision prec,
                           void* cuda_stream) {
    if (!out) return SGPE_EINVAL;
    *out = nullptr;
    if (dim != 1 && dim != 2) return SGPE_EINVAL;
    if (dim == 1) {
        ny = 1;
        dy = dx;
    }
    if (nx < 3 || (dim == 2 && ny < 3)) return SGPE_EINVAL;
    if (!(dx > 0.0) || !(dy > 0.0) || !isfinite(dx) || !isfinite(dy)) return SGPE_EINVAL;
    if (prec != SGPE_C128 && prec != SGPE_C64 && prec != SGPE_CDF) return SGPE_EINVAL;
    int nmax = prec == SGPE_C64 ? 8192 : 4096;
    if (nx > nmax || ny > nmax) return SGPE_EUNSUPPORTED;
    sgpe_ctx* c = new (std::nothrow) sgpe_ctx();
    if (!c) return SGPE_ENOMEM;
    c->dim = dim;
    c->nx = nx;
    c->ny = ny;
    c->dx = dx;
    c->dy = dy;
    c->prec = prec;
    c->esz = prec == SGPE_C64 ? 8 : 16;
    c->stream = (cudaStream_t)cuda_stream;
    c->geo = make_geometry(dim, nx, ny, c->esz);
    c->psi = nullptr;
    c->work = nullptr;
    c->have_params = false;
    c->graphs_ok = true;
    c->err[0] = 0;
    cudaError_t e = cudaGetDevice(&c->device);
    if (e == cudaSuccess) e = with_prec(prec, [](auto r) { return Launcher<decltype(r)>::setup(); });
    if (e != cudaSuccess) {
        snprintf(g_init_err, sizeof(g_init_err), "sgpe_init_grid: %s", cudaGetErrorString(e));
        delete c;
        return SGPE_ECUDA;
    }
    *out = c;
    return SGPE_OK;
}

sgpe_status sgpe_workspace_bytes(const sgpe_ctx* c, size_t* bytes) {
    if (!c || !bytes) return SGPE_EINVAL;
    *bytes = layout_of(c).total;
    return SGPE_OK;
}

sgpe_status sgpe_bind(sgpe_ctx* c, void* psi_dev, void* workspace_dev) {
    if (!c) return SGPE_EINVAL;
    if (!psi_dev || !workspace_dev) return fail(c, SGPE_EINVAL, "sgpe_bind: null buffer");
    if (((uintptr_t)psi_dev & 15) != 0) return fail(c, SGPE_EINVAL, "sgpe_bind: psi not 16-byte aligned");
    if (((uintptr_t)workspace_dev & 255) != 0) return fail(c, SGPE_EINVAL, "sgpe_bind: workspace not 256-byte aligned");
    invalidate_graphs(c);
    c->psi = psi_dev;
    c->work = (unsigned char*)workspace_dev;
    Layout L = layout_of(c);
    c->sc = (DevScalars*)(c->work + L.sc);
    c->mid = c->work + L.mid;
    for (int m = 0; m < 3; m++)
        for (int a = 0; a < 2; a++) {
            for (int k = 0; k < 4; k++) c->tabs[m][a].t[k] = c->work + L.tabs[m][a][k];
            c->tabs[m][a].u = UniHost{};
            c->tabs[m][a].pair = PairHost{};
            c->tabs[m][a].conv = ConvHost{};
            c->us[m][a] = c->work + L.us[m][a];
        }
    for (int m = 0; m < 2; m++)
        for (int a = 0; a < 2; a++)
            for (int q = 0; q < 2; q++)
                for (int k = 0; k < 4; k++) c->tabs_so[m][a][q][k] = c->work + L.tabs_so[m][a][q][k];
    c->partials = (double*)(c->work + L.partials);
    c->have_params = false;
    CK(cudaMemsetAsync(c->sc, 0, sizeof(DevScalars), c->stream), "sgpe_bind memset");
    CK(reset_scale(c->stream, c->sc), "sgpe_bind reset_scale");
    return SGPE_OK;
}

sgpe_status sgpe_set_params(sgpe_ctx* c, const sgpe_params* p) {
    if (!c || !p) return SGPE_EINVAL;
    if (!c->psi) return fail(c, SGPE_ESTATE, "sgpe_set_params: no buffers bound");
    if (const char* why = check_params(p)) return fail(c, SGPE_EINVAL, "%s", why);
    if (p->so_mode && p->so_type != 0 && (c->nx > kRegMaxN || (c->dim == 2 && c->ny > kRegMaxN)))
        return fail(c, SGPE_EUNSUPPORTED, "so_mode 1 needs lines of at most %d points", kRegMaxN);
    invalidate_graphs(c);
    c->params = *p;
    c->kp = make_kparams(c->dim, c->nx, c->ny, c->dx, c->dy, p);
    sgpe_params ph = *p;
    ph.dt = 0.5 * p->dt;
    c->kp_half = make_kparams(c->dim, c->nx, c->ny, c->dx, c->dy, &ph);
    CoefJob jobs[8 + 6];  // SO by Crank-Nicolson: [mode][axis][m]; kinetic: [mode][axis]
    int njobs = 0;
    if (sgpe_status st = build_socn(c, jobs, &njobs)) return st;
    // COEF: Crank-Nicolson tables, bt = z/(4 h^2), z = dt (imaginary), i dt (real), -i dt (adjoint)
    for (int m = 0; m < 3; m++)
        for (int a = 0; a < (c->dim == 2 ? 2 : 1); a++) {
            double h = a == 0 ? c->dx : c->dy;
            int n = a == 0 ? c->nx : c->ny;
            double b = p->dt / (4.0 * h * h);
            double bre = m == 0 ? b : 0.0, bim = m == 0 ? 0.0 : (m == 1 ? b : -b);
            jobs[njobs++] = coef_job(c->tabs[m][a].t, n, bre, bim, 0);
            // lines longer than kRegMaxN (and the lines of a tiled grid): the constant-factor
            // form of the same solve
            c->tabs[m][a].u = UniHost{};
            c->tabs[m][a].conv = c->dim == 1 && c->prec == SGPE_C64 ? conv_form(n, bre, bim) : ConvHost{};
            c->tabs[m][a].pair = c->dim == 2 && c->prec != SGPE_C64 ? pair_form(n, bre, bim) : PairHost{};
            if (n > kRegMaxN || c->geo.tiled) {
                cudaError_t e = with_prec(c->prec, [&](auto r) {
                    return Launcher<decltype(r)>::uni(c->stream, n, bre, bim, c->us[m][a], &c->tabs[m][a].u);
                });
                CK(e, "constant-factor form");
            }
        }
    cudaError_t e = with_prec(
        c->prec, [&](auto r) { return Launcher<decltype(r)>::coef(c->stream, jobs, njobs); });
    CK(e, "COEF kernel");
    c->have_params = true;
    return SGPE_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Step orchestration
// ---------------------------------------------------------------------------
// The fused 2D step with the register y sweep ends without a finalize launch:
// each step's head kernel derives the pending scale from the previous y
// sweep's norm partials, and end_steps publishes it after the last step.
// Strang splitting or the SO substep by Crank-Nicolson: the unfused step of
// enqueue_step_general.
static bool general_path(const sgpe_ctx* c) { return c->params.split != 0 || c->params.so_mode != 0; }

// The step of a complex128 or double-float 2D grid in the given time mode (0
// imaginary, 1 real) as increments in FP32 pairs (sgpe_pair.cuh), where both axes'
// sweeps are short convolutions (bt up to about 0.08, lines of more than 16 points).
// Double-float grids of 320..~630 points an axis keep the tiled step in imaginary time, where it
// is the faster one (us a step, tiled against pair: 320^2 29.3 / 31.1, 512^2 55.6 / 66.6, 700^2 107 /
// 95; in real time 400 x 330 53 / 37).
constexpr long long kPairCdfTiledMax = 400000;
// Grids of fewer points keep the register kernels. (24 x 20, us a step, register / pair: 15.6 / 17.6 when the
// line was drawn, 14.4 / 11.3 since the head kernel's chains were shortened; the line has not followed.)
// So do complex128 steps longer than kPairMaxDt, whose dt mu passes 2^-5 where the state lives so often that most
// blocks leave the increments: dx = 0.2, c0 = 50, imaginary time 100 x 120 at dt = 4e-3 18.0 / 19.4, at 0.01 17.7 /
// 24.5, 64^2 at 0.01 15.7 / 18.8. (Grids that fill the GPU would gain there too: 256^2 47.5 / 32.5 and 47.7 /
// 45.1; the line has not been split by size.)
constexpr long long kPairMinPoints = 1536;
constexpr double kPairMaxDt = 2.5e-3;
static bool pair_mode(const sgpe_ctx* c, int mode) {
    if (c->prec == SGPE_CDF && mode == 0 && (long long)c->nx * c->ny <= kPairCdfTiledMax && c->geo.tiled &&
        tiled_step(c->geo, c->tabs[0][0], c->tabs[0][1]))
        return false;
    if ((long long)c->nx * c->ny < kPairMinPoints || (c->prec == SGPE_C128 && c->params.dt > kPairMaxDt)) return false;
    return c->dim == 2 && c->prec != SGPE_C64 && !general_path(c) && c->tabs[mode][0].pair.kt > 0 &&
           c->tabs[mode][1].pair.kt > 0;
}
static int pair_parts(const sgpe_ctx* c) { return sgpe::pair_parts(c->nx, c->ny); }

// A tiled grid's step in the given time mode (0 imaginary, 1 real) on the kernels of long lines.
static bool tiled_mode(const sgpe_ctx* c, int mode) {
    return c->geo.tiled && !general_path(c) && tiled_step(c->geo, c->tabs[mode][0], c->tabs[mode][1]);
}
// The fused head kernel of a complex64 step on the long-line kernels (tiled grids,
// or rows of 1025..2048 points) forms the pending scale from the row tiles' partials
// itself instead of a finalize block: with renormalisation, where there are at most
// kHeadMaxParts partials a component (2048^2, 1024 a component: every block summing
// them measured 108.5 -> 126.4 us/step); without it (real time) the y tiles store
// the scale 1 and nothing is summed (2048^2 real time 126.5 -> 124.9).
constexpr int kHeadMaxParts = 256;
static bool tiled_head(const sgpe_ctx* c, int mode) {
    if (general_path(c) || !pwx_long_fits(c->geo, c->tabs[mode][0])) return false;
    if (c->geo.tiled ? !tiled_mode(c, mode) : c->geo.reg_x) return false;
    const int renorm = mode == 0 ? c->params.renorm : 0;
    return y_tiled(c->geo, c->tabs[mode][1], c->mid, c->psi) &&
           (renorm == 0 || c->geo.blocks_yt / 3 <= kHeadMaxParts);
}
static bool head_scale(const sgpe_ctx* c, int mode) {
    if (general_path(c)) return false;
    if (pair_mode(c, mode)) return (mode == 0 ? c->params.renorm : 0) == 0 || pair_parts(c) <= kHeadMaxParts;
    return (c->geo.fused && c->geo.reg_y && !tiled_mode(c, mode)) || tiled_head(c, mode);
}

// The y sweeps (2D) and the long x sweep (1D) of the complex64 and double-float
// forms leave their norm partials as double-float pairs (summed on the FP32
// pipe); the 1D register x sweep, every complex128 sweep and the pair step leave FP64 sums.
static int parts_df(const sgpe_ctx* c, int mode) {
    return c->prec != SGPE_C128 && !pair_mode(c, mode) && (c->dim == 2 || !c->geo.reg_x);
}

// The end-of-step launch: norms, next pending scale, step counter (advance).
static cudaError_t finalize(sgpe_ctx* c, int mode, int advance) {
    const int renorm = mode == 0 ? c->params.renorm : 0;
    const int nblk = pair_mode(c, mode) ? 3 * pair_parts(c)
                     : c->dim == 2      ? y_parts(c->geo, c->tabs[mode][1], c->mid, c->psi)
                                        : 3 * c->ny;  // 1D: one partial per line
    return finalize_step(c->stream, c->partials, nblk, c->kp.cell, renorm, c->kp.mag, advance, c->sc,
                         parts_df(c, mode));
}

static cudaError_t end_steps(sgpe_ctx* c, bool imag) {
    const int mode = imag ? 0 : 1;
    return head_scale(c, mode) ? finalize(c, mode, 0) : cudaSuccess;
}

// The SO substep by Crank-Nicolson on the line families of the grid, in -> out:
// x lines then y lines (reverse: y then x); scale: apply the pending scale.
template <typename R>
static cudaError_t so_cn_pass(sgpe_ctx* c, int mode, const void* in, void* out, bool reverse, bool scale) {
    const SoCnLines* L = c->socn[mode];
    if (!c->socn_y)
        return Launcher<R>::socn(c->stream, in, out, L[0], c->tabs_so[mode][0][0], c->tabs_so[mode][0][1], c->sc,
                                 scale ? 1 : 0);
    const int a0 = reverse ? 1 : 0, a1 = 1 - a0;
    cudaError_t e = Launcher<R>::socn(c->stream, in, out, L[a0], c->tabs_so[mode][a0][0], c->tabs_so[mode][a0][1],
                                      c->sc, scale ? 1 : 0);
    if (e) return e;
    return Launcher<R>::socn(c->stream, out, out, L[a1], c->tabs_so[mode][a1][0], c->tabs_so[mode][a1][1], c->sc, 0);
}

// One step with Strang splitting (params.split = 1: the pointwise and SO
// substeps with dt/2 before the Crank-Nicolson sweeps, then again in the
// reverse order) and / or the SO substep by Crank-Nicolson (params.so_mode = 1):
// unfused kernels, A -> B -> A, the norms and the next pending scale at the end.
template <typename R>
static cudaError_t enqueue_step_general(sgpe_ctx* c, bool imag, const double* omega_tab) {
    cudaError_t e;
    const int mode = imag ? 0 : 1;
    const int renorm = imag ? c->params.renorm : 0;
    const bool strang = c->params.split != 0;
    const bool socn = c->params.so_mode != 0 && c->kp.so_case != 0;
    const KParams& kh = strang ? c->kp_half : c->kp;
    void* A = c->psi;
    void* B = c->mid;
    int mask = 7;
    if (socn) {
        if ((e = so_cn_pass<R>(c, mode, A, A, false, true))) return e;
        mask = 2 | 4 | kMaskNoScale;
    }
    if ((e = Launcher<R>::pointwise(c->stream, imag, A, B, kh, c->sc, omega_tab, mask))) return e;
    if (c->dim == 2) {
        if ((e = Launcher<R>::cn_x(c->stream, imag, false, B, B, c->kp, c->tabs[mode][0], c->geo, c->partials, c->sc,
                                   renorm, 0)))
            return e;
        if ((e = Launcher<R>::cn_y(c->stream, imag, B, A, c->kp, c->tabs[mode][1], c->geo, c->partials, c->sc, renorm,
                                   0, 0)))
            return e;
    } else {
        if ((e = Launcher<R>::cn_x(c->stream, imag, false, B, A, c->kp, c->tabs[mode][0], c->geo, c->partials, c->sc,
                                   renorm, 0)))
            return e;
    }
    if (strang) {
        if ((e = Launcher<R>::pointwise(c->stream, imag, A, B, kh, c->sc, omega_tab,
                                        2 | 4 | kMaskReverse | kMaskNoScale)))
            return e;
        if (socn)
            e = so_cn_pass<R>(c, mode, B, A, true, false);
        else
            e = Launcher<R>::pointwise(c->stream, imag, B, A, kh, c->sc, omega_tab, 1 | kMaskNoScale);
        if (e) return e;
    }
    return Launcher<R>::norms(c->stream, A, (size_t)c->nx * c->ny, c->kp.cell, renorm, c->kp.mag, c->partials, c->sc,
                              1);
}

template <typename R>
static cudaError_t enqueue_step(sgpe_ctx* c, bool imag, const double* omega_tab) {
    cudaError_t e;
    const int mode = imag ? 0 : 1;
    const int renorm = imag ? c->params.renorm : 0;
    if (general_path(c)) return enqueue_step_general<R>(c, imag, omega_tab);
    if (pair_mode(c, mode)) {
        const bool head = head_scale(c, mode);
        if ((e = Launcher<R>::pair_x(c->stream, imag, c->psi, c->mid, c->kp, c->sc, omega_tab, c->tabs[mode][0].pair,
                                     head ? c->partials : nullptr, pair_parts(c), renorm)))
            return e;
        if ((e = Launcher<R>::pair_y(c->stream, imag, c->mid, c->psi, c->kp, c->tabs[mode][1].pair, c->partials, c->sc,
                                     renorm, 1, head)))
            return e;
        return head ? cudaSuccess : finalize(c, mode, 1);
    }
    if (c->geo.fused && !tiled_mode(c, mode)) {
        if ((e = Launcher<R>::pwx(c->stream, imag, c->psi, c->mid, c->kp, c->sc, omega_tab, c->tabs[mode][0].t,
                                  c->partials, c->geo.blocks_y / 3, renorm)))
            return e;
        const bool head = head_scale(c, mode);
        if ((e = Launcher<R>::cn_y(c->stream, imag, c->mid, c->psi, c->kp, c->tabs[mode][1], c->geo, c->partials,
                                   c->sc, renorm, 1, 1, head)))
            return e;
        if (head) return cudaSuccess;  // the next head kernel (or end_steps) takes the scale from the partials
        return finalize(c, mode, 1);
    }
    if (tiled_head(c, mode)) {
        // tiled complex64 grid: the fused kernel forms the pending scale from the row
        // tiles' partials, the y sweep marks them and moves the step counter on
        if ((e = Launcher<R>::pwx_long(c->stream, imag, c->psi, c->mid, c->kp, c->sc, omega_tab, c->tabs[mode][0], 7,
                                       c->partials, c->geo.blocks_yt / 3, renorm)))
            return e;
        return Launcher<R>::cn_y(c->stream, imag, c->mid, c->psi, c->kp, c->tabs[mode][1], c->geo, c->partials,
                                 c->sc, renorm, 1, 1, true);
    }
    if (pwx_long_fits(c->geo, c->tabs[mode][0]) && (!c->geo.reg_x || tiled_mode(c, mode))) {
        // complex64 rows of 1025..2048 points (and tiled grids outside the head path): pointwise
        // substeps and x sweep in one kernel
        if ((e = Launcher<R>::pwx_long(c->stream, imag, c->psi, c->mid, c->kp, c->sc, omega_tab, c->tabs[mode][0],
                                       7)))
            return e;
    } else {
        if ((e = Launcher<R>::pointwise(c->stream, imag, c->psi, c->mid, c->kp, c->sc, omega_tab, 7))) return e;
        if (c->dim == 2 && (e = Launcher<R>::cn_x(c->stream, imag, false, c->mid, c->mid, c->kp, c->tabs[mode][0],
                                                  c->geo, c->partials, c->sc, renorm, 1)))
            return e;
    }
    if (c->dim == 2) {
        if ((e = Launcher<R>::cn_y(c->stream, imag, c->mid, c->psi, c->kp, c->tabs[mode][1], c->geo, c->partials,
                                   c->sc, renorm, 1, 1)))
            return e;
        return finalize(c, mode, 1);
    }
    if ((e = Launcher<R>::cn_x(c->stream, imag, true, c->mid, c->psi, c->kp, c->tabs[mode][0], c->geo, c->partials,
                               c->sc, renorm, 1)))
        return e;
    return finalize(c, mode, 1);
}

static cudaError_t enqueue_steps(sgpe_ctx* c, int n, bool imag, const double* omega_tab) {
    for (int i = 0; i < n; i++) {
        cudaError_t e = with_prec(c->prec, [&](auto r) { return enqueue_step<decltype(r)>(c, imag, omega_tab); });
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static const int kGraphSteps = 32;

// 1D grids run the whole step loop in one launch: lines of at most 1024 points
// in the complex64 and double-float forms in one block (the FP32-pipe forms fit
// one SM); complex128 lines of at most 256 points in one cluster of up to 8
// CTAs with the FP64 work of a point split over three threads.
static bool one_block_1d(const sgpe_ctx* c) {
    return c->dim == 1 && c->nx <= kRegMaxN && (c->prec != SGPE_C128 || c->nx <= kCl1dMaxN) && !general_path(c);
}

static sgpe_status run_steps(sgpe_ctx* c, int nsteps, bool imag, const double* omega_tab) {
    if (omega_tab) CK(cudaMemsetAsync(&c->sc->step_idx, 0, sizeof(int), c->stream), "step_idx reset");
    if (one_block_1d(c)) {
        if (nsteps == 0) return SGPE_OK;
        const int mode = imag ? 0 : 1;
        const int renorm = imag ? c->params.renorm : 0;
        cudaError_t e = with_prec(c->prec, [&](auto r) {
            return Launcher<decltype(r)>::step1d(c->stream, imag, c->psi, c->kp, c->sc, omega_tab, c->tabs[mode][0],
                                                 nsteps, renorm);
        });
        CK(e, "1D step loop");
        return SGPE_OK;
    }
    int G = nsteps < kGraphSteps ? nsteps : kGraphSteps;
    int reps = G > 0 ? nsteps / G : 0;
    int rem = G > 0 ? nsteps - reps * G : 0;
    cudaGraphExec_t exec = nullptr;
    if (c->graphs_ok && c->stream != nullptr && reps > 0 && G >= 4) {
        GraphKey key{imag ? 1 : 0, G, omega_tab};
        auto it = c->graphs.find(key);
        if (it != c->graphs.end()) {
            exec = it->second;
        } else {
            cudaGraph_t graph = nullptr;
            cudaError_t e = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                cudaError_t e2 = enqueue_steps(c, G, imag, omega_tab);
                e = cudaStreamEndCapture(c->stream, &graph);
                if (e2 != cudaSuccess) e = e2;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
            if (graph) cudaGraphDestroy(graph);
            if (e != cudaSuccess) {
                cudaGetLastError();
                exec = nullptr;
                c->graphs_ok = false;
            } else {
                c->graphs[key] = exec;
            }
        }
    }
    if (exec) {
        for (int r = 0; r < reps; r++) CK(cudaGraphLaunch(exec, c->stream), "cudaGraphLaunch");
        CK(enqueue_steps(c, rem, imag, omega_tab), "step kernels");
    } else {
        CK(enqueue_steps(c, nsteps, imag, omega_tab), "step kernels");
    }
    if (nsteps > 0) CK(end_steps(c, imag), "end of steps");
    return SGPE_OK;
}

static sgpe_status check_ready(sgpe_ctx* c) {
    if (!c) return SGPE_EINVAL;
    if (!c->psi) return fail(c, SGPE_ESTATE, "no buffers bound");
    if (!c->have_params) return fail(c, SGPE_ESTATE, "no parameters set");
    return SGPE_OK;
}

template <typename R> static cudaError_t flush_scale(sgpe_ctx* c) {
    cudaError_t e = Launcher<R>::flush(c->stream, c->psi, (size_t)c->nx * c->ny, c->sc);
    if (e) return e;
    return reset_scale(c->stream, c->sc);
}
static cudaError_t flush_any(sgpe_ctx* c) {
    return with_prec(c->prec, [&](auto r) { return flush_scale<decltype(r)>(c); });
}

static sgpe_status read_err(sgpe_ctx* c) {
    int err = 0;
    CK(cudaMemcpyAsync(&err, &c->sc->err, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "read err");
    CK(cudaStreamSynchronize(c->stream), "sync");
    if (err) {
        CK(cudaMemsetAsync(&c->sc->err, 0, sizeof(int), c->stream), "clear err");
        return fail(c, SGPE_ENONFINITE, "non-finite norm of the state");
    }
    return SGPE_OK;
}

extern "C" {

sgpe_status sgpe_step_imag(sgpe_ctx* c, int nsteps) {
    sgpe_status st = check_ready(c);
    if (st) return st;
    if (nsteps < 0) return fail(c, SGPE_EINVAL, "nsteps < 0");
    if (nsteps == 0) return SGPE_OK;
    return run_steps(c, nsteps, true, nullptr);
}

sgpe_status sgpe_step_real(sgpe_ctx* c, int nsteps, const double* omega_dev) {
    sgpe_status st = check_ready(c);
    if (st) return st;
    if (nsteps < 0) return fail(c, SGPE_EINVAL, "nsteps < 0");
    if (((uintptr_t)omega_dev & 7) != 0) return fail(c, SGPE_EINVAL, "omega table not 8-byte aligned");
    if (nsteps == 0) return SGPE_OK;
    return run_steps(c, nsteps, false, omega_dev);
}

sgpe_status sgpe_normalize(sgpe_ctx* c, double* norms_out) {
    sgpe_status st = check_ready(c);
    if (st) return st;
    CK(flush_any(c), "flush");
    size_t plane = (size_t)c->nx * c->ny;
    cudaError_t e = with_prec(c->prec, [&](auto r) {
        return Launcher<decltype(r)>::norms(c->stream, c->psi, plane, c->kp.cell, 0, 0.0, c->partials, c->sc);
    });
    CK(e, "norms kernel");
    double n[4];
    CK(cudaMemcpyAsync(n, c->sc->norms, sizeof(n), cudaMemcpyDeviceToHost, c->stream), "copy norms");
    st = read_err(c);
    if (norms_out) memcpy(norms_out, n, 3 * sizeof(double));
    return st;
}

sgpe_status sgpe_energy(sgpe_ctx* c, double* out) {
    sgpe_status st = check_ready(c);
    if (st) return st;
    if (!out) return fail(c, SGPE_EINVAL, "null output");
    CK(flush_any(c), "flush");
    cudaError_t e = with_prec(c->prec, [&](auto r) {
        return Launcher<decltype(r)>::observables(c->stream, c->psi, c->kp, c->kp.omega_t, c->partials, c->sc);
    });
    CK(e, "observables kernel");
    CK(cudaMemcpyAsync(out, c->sc->obs, SGPE_NOBS * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "copy obs");
    return read_err(c);
}

// complex128 <-> double-float layout (hi, lo per real part), on the host.
static void cdf_split(const double* in, float* out, size_t nreal) {
    for (size_t i = 0; i < nreal; i++) {
        const df v = df_from(in[i]);
        out[2 * i] = v.hi;
        out[2 * i + 1] = v.lo;
    }
}
static void cdf_join(const float* in, double* out, size_t nreal) {
    for (size_t i = 0; i < nreal; i++) out[i] = (double)in[2 * i] + (double)in[2 * i + 1];
}

sgpe_status sgpe_set_state(sgpe_ctx* c, const void* host_psi) {
    if (!c || !host_psi) return SGPE_EINVAL;
    if (!c->psi) return fail(c, SGPE_ESTATE, "no buffers bound");
    size_t bytes = (size_t)3 * c->nx * c->ny * c->esz;
    if (c->prec == SGPE_CDF) {
        const size_t nreal = (size_t)6 * c->nx * c->ny;
        std::vector<float> tmp(2 * nreal);
        cdf_split((const double*)host_psi, tmp.data(), nreal);
        CK(cudaMemcpyAsync(c->psi, tmp.data(), bytes, cudaMemcpyHostToDevice, c->stream), "set_state copy");
        CK(reset_scale(c->stream, c->sc), "reset scale");
        CK(cudaMemsetAsync(&c->sc->err, 0, sizeof(int), c->stream), "clear err");
        CK(cudaStreamSynchronize(c->stream), "sync");  // tmp must outlive the copy
        return SGPE_OK;
    }
    CK(cudaMemcpyAsync(c->psi, host_psi, bytes, cudaMemcpyHostToDevice, c->stream), "set_state copy");
    CK(reset_scale(c->stream, c->sc), "reset scale");
    CK(cudaMemsetAsync(&c->sc->err, 0, sizeof(int), c->stream), "clear err");
    CK(cudaStreamSynchronize(c->stream), "sync");
    return SGPE_OK;
}

sgpe_status sgpe_load_state(sgpe_ctx* c, const void* psi_dev) {
    if (!c || !psi_dev) return SGPE_EINVAL;
    if (!c->psi) return fail(c, SGPE_ESTATE, "no buffers bound");
    size_t bytes = (size_t)3 * c->nx * c->ny * c->esz;
    if (c->prec == SGPE_CDF)
        CK(cdf_from_c128(c->stream, psi_dev, c->psi, (size_t)3 * c->nx * c->ny), "load_state split");
    else
        CK(cudaMemcpyAsync(c->psi, psi_dev, bytes, cudaMemcpyDeviceToDevice, c->stream), "load_state copy");
    CK(reset_scale(c->stream, c->sc), "reset scale");
    CK(cudaMemsetAsync(&c->sc->err, 0, sizeof(int), c->stream), "clear err");
    return SGPE_OK;
}

sgpe_status sgpe_get_state(sgpe_ctx* c, void* host_psi) {
    if (!c || !host_psi) return SGPE_EINVAL;
    if (!c->psi) return fail(c, SGPE_ESTATE, "no buffers bound");
    CK(flush_any(c), "flush");
    size_t bytes = (size_t)3 * c->nx * c->ny * c->esz;
    if (c->prec == SGPE_CDF) {
        const size_t nreal = (size_t)6 * c->nx * c->ny;
        std::vector<float> tmp(2 * nreal);
        CK(cudaMemcpyAsync(tmp.data(), c->psi, bytes, cudaMemcpyDeviceToHost, c->stream), "get_state copy");
        CK(cudaStreamSynchronize(c->stream), "sync");
        cdf_join(tmp.data(), (double*)host_psi, nreal);
        return SGPE_OK;
    }
    CK(cudaMemcpyAsync(host_psi, c->psi, bytes, cudaMemcpyDeviceToHost, c->stream), "get_state copy");
    CK(cudaStreamSynchronize(c->stream), "sync");
    return SGPE_OK;
}

sgpe_status sgpe_substep(sgpe_ctx* c, int which, int imag, double omega) {
    sgpe_status st = check_ready(c);
    if (st) return st;
    if (which < 0 || which > 7) return fail(c, SGPE_EINVAL, "which must be 0..7");
    if (which >= 6 && c->kp.so_case != 0 && (c->nx > kRegMaxN || (c->dim == 2 && c->ny > kRegMaxN)))
        return fail(c, SGPE_EUNSUPPORTED, "SO by Crank-Nicolson needs lines of at most %d points", kRegMaxN);
    if (which == 4 && c->dim != 2) return fail(c, SGPE_EINVAL, "no y sweep in 1D");
    if (!isfinite(omega)) return fail(c, SGPE_EINVAL, "non-finite omega");
    CK(flush_any(c), "flush");
    const bool im = imag != 0;
    const int mode = im ? 0 : 1;
    const size_t bytes = (size_t)3 * c->nx * c->ny * c->esz;
    cudaError_t e = cudaSuccess;
    if (which <= 2) {
        KParams k = c->kp;
        k.omega_t = omega / sqrt(2.0);
        e = with_prec(c->prec, [&](auto r) {
            return Launcher<decltype(r)>::pointwise(c->stream, im, c->psi, c->mid, k, c->sc, nullptr, 1 << which);
        });
        CK(e, "pointwise kernel");
        CK(cudaMemcpyAsync(c->psi, c->mid, bytes, cudaMemcpyDeviceToDevice, c->stream), "copy back");
    } else if (which == 3) {
        CK(cudaMemcpyAsync(c->mid, c->psi, bytes, cudaMemcpyDeviceToDevice, c->stream), "copy");
        e = with_prec(c->prec, [&](auto r) {
            return Launcher<decltype(r)>::cn_x(c->stream, im, false, c->mid, c->psi, c->kp, c->tabs[mode][0], c->geo,
                                               c->partials, c->sc, 0, 0);
        });
        CK(e, "cn_x kernel");
    } else if (which == 4) {
        CK(cudaMemcpyAsync(c->mid, c->psi, bytes, cudaMemcpyDeviceToDevice, c->stream), "copy");
        e = with_prec(c->prec, [&](auto r) {
            return Launcher<decltype(r)>::cn_y(c->stream, im, c->mid, c->psi, c->kp, c->tabs[mode][1], c->geo,
                                               c->partials, c->sc, 0, 0, 0);
        });
        CK(e, "cn_y kernel");
    } else if (which >= 6) {
        if (c->kp.so_case != 0) {
            e = with_prec(c->prec, [&](auto r) {
                return so_cn_pass<decltype(r)>(c, mode, c->psi, c->psi, which == 7, false);
            });
            CK(e, "SO Crank-Nicolson kernel");
        }
    } else {
        size_t plane = (size_t)c->nx * c->ny;
        int rn = c->params.renorm ? c->params.renorm : 1;
        e = with_prec(c->prec, [&](auto r) {
            return Launcher<decltype(r)>::norms(c->stream, c->psi, plane, c->kp.cell, rn, c->kp.mag, c->partials,
                                                c->sc);
        });
        CK(e, "norms kernel");
        CK(flush_any(c), "flush");
    }
    return SGPE_OK;
}

sgpe_status sgpe_profile_steps(sgpe_ctx* c, int nsteps, int imag, double* ms_out, int* launches_out) {
    sgpe_status st = check_ready(c);
    if (st) return st;
    if (nsteps < 0 || !ms_out || !launches_out) return fail(c, SGPE_EINVAL, "bad profile arguments");
    if (general_path(c)) return fail(c, SGPE_EUNSUPPORTED, "profile_steps: Lie splitting with the Euler SO only");
    const bool im = imag != 0;
    const int mode = im ? 0 : 1;
    const int renorm = im ? c->params.renorm : 0;
    // kinds: 0 pointwise, 1 CN along x, 2 CN along y, 3 end-of-step norm / scale;
    // with the fused 2D head, kind 0 is the fused pointwise + CN-x kernel and
    // kind 1 has no launches.
    // Steps are enqueued in batches of kBatch with their events and synchronised
    // once per batch, so the intervals measure the GPU, not host submission.
    const int kBatch = 64;
    cudaEvent_t evs[kBatch][5];
    for (int b = 0; b < kBatch; b++)
        for (int k = 0; k < 5; k++) CK(cudaEventCreate(&evs[b][k]), "cudaEventCreate");
    double acc[4] = {0, 0, 0, 0};
    int cnt[4] = {0, 0, 0, 0};
    const bool two = c->dim == 2;
    const bool pair = pair_mode(c, mode);
    const bool fused = !pair && c->geo.fused && !tiled_mode(c, mode);
    const bool long_fused = !pair && !general_path(c) && !fused && pwx_long_fits(c->geo, c->tabs[mode][0]) &&
                            (!c->geo.reg_x || tiled_mode(c, mode));
    const bool head = head_scale(c, mode);
    sgpe_status out = SGPE_OK;
    for (int i0 = 0; i0 < nsteps && out == SGPE_OK; i0 += kBatch) {
      const int nb = nsteps - i0 < kBatch ? nsteps - i0 : kBatch;
      cudaError_t e = cudaSuccess;
      for (int bi = 0; bi < nb && !e; bi++) {
        cudaEvent_t* ev = evs[bi];
        e = cudaEventRecord(ev[0], c->stream);
        if (!e && pair)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::pair_x(c->stream, im, c->psi, c->mid, c->kp, c->sc, nullptr,
                                                     c->tabs[mode][0].pair, head ? c->partials : nullptr,
                                                     pair_parts(c), renorm);
            });
        if (!e && fused)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::pwx(c->stream, im, c->psi, c->mid, c->kp, c->sc, nullptr,
                                                  c->tabs[mode][0].t, c->partials, c->geo.blocks_y / 3, renorm);
            });
        if (!e && long_fused)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::pwx_long(c->stream, im, c->psi, c->mid, c->kp, c->sc, nullptr,
                                                       c->tabs[mode][0], 7, head ? c->partials : nullptr,
                                                       c->geo.blocks_yt / 3, renorm);
            });
        if (!e && !pair && !fused && !long_fused)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::pointwise(c->stream, im, c->psi, c->mid, c->kp, c->sc, nullptr, 7);
            });
        if (!e) e = cudaEventRecord(ev[1], c->stream);
        void* xout = two ? c->mid : c->psi;
        if (!e && !pair && !fused && !long_fused)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::cn_x(c->stream, im, !two, c->mid, xout, c->kp, c->tabs[mode][0], c->geo,
                                                   c->partials, c->sc, renorm, 1);
            });
        if (!e) e = cudaEventRecord(ev[2], c->stream);
        if (!e && pair)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::pair_y(c->stream, im, c->mid, c->psi, c->kp, c->tabs[mode][1].pair,
                                                     c->partials, c->sc, renorm, 1, head);
            });
        if (!e && two && !pair)
            e = with_prec(c->prec, [&](auto r) {
                return Launcher<decltype(r)>::cn_y(c->stream, im, c->mid, c->psi, c->kp, c->tabs[mode][1], c->geo,
                                                   c->partials, c->sc, renorm, 1, 1, head);
            });
        if (!e) e = cudaEventRecord(ev[3], c->stream);
        if (!e && !head)
            e = finalize(c, mode, 1);
        if (!e) e = cudaEventRecord(ev[4], c->stream);
      }
      if (!e) e = cudaEventSynchronize(evs[nb - 1][4]);
      if (e) {
          out = cuda_fail(c, e, "profile");
          break;
      }
      for (int bi = 0; bi < nb; bi++)
          for (int k = 0; k < 4; k++) {
              if ((k == 2 && !two) || (k == 1 && (pair || fused || long_fused)) || (k == 3 && head)) continue;
              float ms = 0.f;
              cudaEventElapsedTime(&ms, evs[bi][k], evs[bi][k + 1]);
              acc[k] += ms;
              cnt[k] += 1;
          }
    }
    for (int b = 0; b < kBatch; b++)
        for (int k = 0; k < 5; k++) cudaEventDestroy(evs[b][k]);
    if (out == SGPE_OK && nsteps > 0) CK(end_steps(c, im), "end of steps");
    for (int k = 0; k < 4; k++) {
        ms_out[k] = acc[k];
        launches_out[k] = cnt[k];
    }
    return out;
}

int sgpe_launches_per_step(const sgpe_ctx* c) {
    if (!c) return 0;
    if (general_path(c)) {
        const int so = (c->params.so_mode && c->kp.so_case) ? (c->socn_y ? 2 : 1) : 0;
        const int sweeps = c->dim == 2 ? 2 : 1;
        return so + 1 + sweeps + (c->params.split ? 1 + (so ? so : 1) : 0) + 1;
    }
    if (one_block_1d(c)) return 0;  // one launch per step call
    if (head_scale(c, 0)) return 2;  // plus one end-of-steps launch per step call
    if (pair_mode(c, 0)) return 3;
    if (c->geo.fused && !tiled_mode(c, 0)) return 3;
    if (c->dim == 2 && pwx_long_fits(c->geo, c->tabs[0][0]) && (!c->geo.reg_x || tiled_mode(c, 0))) return 3;
    return c->dim == 2 ? 4 : 3;
}

const char* sgpe_last_error(const sgpe_ctx* c) { return c ? c->err : g_init_err; }

sgpe_status sgpe_destroy(sgpe_ctx* c) {
    if (!c) return SGPE_OK;
    invalidate_graphs(c);
    delete c;
    return SGPE_OK;
}

}  // extern "C"

// Internal access for the adjoint translation unit.
namespace sgpe {
bool ctx_view(sgpe_ctx* c, CtxView* v) {
    if (!c) return false;
    v->dim = c->dim;
    v->nx = c->nx;
    v->ny = c->ny;
    v->esz = c->esz;
    v->dbl = c->prec == SGPE_C128;
    v->prec = c->prec;
    v->stream = c->stream;
    v->psi = c->psi;
    v->mid = c->mid;
    v->sc = c->sc;
    v->tabs_real = &c->tabs[1][0];
    v->tabs_adj = &c->tabs[2][0];
    v->geo = &c->geo;
    v->kp = c->kp;
    v->partials = c->partials;
    v->ready = c->psi != nullptr && c->have_params;
    return true;
}

sgpe_status ctx_fail(sgpe_ctx* c, sgpe_status st, const char* msg) { return fail(c, st, "%s", msg); }

cudaError_t ctx_flush(sgpe_ctx* c) { return flush_any(c); }
}  // namespace sgpe

// ---------------------------------------------------------------------------
// Measurement aid: the FP64 FMA rate of the current device.
// ---------------------------------------------------------------------------
namespace {

constexpr int kPeakChains = 16;
constexpr int kPeakIters = 1024;
__device__ double g_peak_sink[1];

// Every thread runs kPeakChains independent FMA chains of kPeakIters steps
// (x <- x * a + b with |a| < 1, so the values stay finite); the result is
// folded into one word so that the work is not optimised away.
__global__ void __launch_bounds__(256) k_fp64_fma(double a, double b, int rounds) {
    double x[kPeakChains];
#pragma unroll
    for (int c = 0; c < kPeakChains; c++) x[c] = (double)(threadIdx.x + c);
    for (int r = 0; r < rounds; r++) {
#pragma unroll 16
        for (int i = 0; i < kPeakIters; i++) {
#pragma unroll
            for (int c = 0; c < kPeakChains; c++) x[c] = fma(x[c], a, b);
        }
    }
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < kPeakChains; c++) s += x[c];
    if (s == 1.2345678e-300) g_peak_sink[0] = s;
}

}  // namespace

extern "C" sgpe_status sgpe_measure_fp64_rate(void* cuda_stream, double* tflops_out) {
    if (!tflops_out) return SGPE_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (!e) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    if (!e) e = cudaEventCreate(&t0);
    if (!e) e = cudaEventCreate(&t1);
    const int blocks = 8 * sms, threads = 256, rounds = 4;
    double best = 0.0;
    for (int rep = 0; rep < 4 && !e; rep++) {
        e = cudaEventRecord(t0, s);
        if (!e) {
            k_fp64_fma<<<blocks, threads, 0, s>>>(0.999999, 1e-7, rounds);
            e = cudaGetLastError();
        }
        if (!e) e = cudaEventRecord(t1, s);
        if (!e) e = cudaEventSynchronize(t1);
        float ms = 0.f;
        if (!e) e = cudaEventElapsedTime(&ms, t0, t1);
        const double flops = 2.0 * (double)blocks * threads * kPeakChains * kPeakIters * rounds;
        if (!e && rep > 0 && ms > 0.f) best = std::max(best, flops / (ms * 1e-3) / 1e12);
    }
    if (t0) cudaEventDestroy(t0);
    if (t1) cudaEventDestroy(t1);
    if (e) {
        set_thread_error(cudaGetErrorString(e));
        return SGPE_ECUDA;
    }
    *tflops_out = best;
    return SGPE_OK;
}

// ---------------------------------------------------------------------------
// Check aid: the FP32 exp(x) - 1 of the complex64 CALCNU substep on device data.
// ---------------------------------------------------------------------------
namespace {
__global__ void k_eval_expm1(const float* x, float* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = expm1_cw(x[i]);
}
}  // namespace

extern "C" sgpe_status sgpe_eval_expm1f(void* cuda_stream, const float* x_dev, float* y_dev, int n) {
    if (n < 0 || (n > 0 && (!x_dev || !y_dev))) return SGPE_EINVAL;
    if (n == 0) return SGPE_OK;
    k_eval_expm1<<<(n + 255) / 256, 256, 0, (cudaStream_t)cuda_stream>>>(x_dev, y_dev, n);
    const cudaError_t e = cudaGetLastError();
    if (e) {
        set_thread_error(cudaGetErrorString(e));
        return SGPE_ECUDA;
    }
    return SGPE_OK;
}
