// Host side of the C ABI declared in include/lbm.h: parameter validation, device
// buffers, kernel dispatch, checkpoint/resume and the adjoint driver.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_adjoint.h"
#include "lbm_internal.h"

using namespace lbm;

struct lbm_ctx {
    lbm_params p{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int device = 0;
    int sm_count = 0;
    size_t elem = 0;        // bytes per stored population
    size_t real = 0;        // bytes of the arithmetic type (psi field)
    int64_t pitch = 0;      // elements per row of a population plane
    int64_t plane = 0;      // elements per plane
    void *pops[2] = {nullptr, nullptr};
    float *refp[2] = {nullptr, nullptr};
    int cur = 0;
    void *psi = nullptr;    // psi field of the two-pass step; rows of sums of the diagnostics
    void *geometry = nullptr;  // one allocation, the arrays of lbm_set_geometry and what derives from them:
    uint8_t *solid = nullptr;
    double *wall_u = nullptr, *q = nullptr, *fext = nullptr;
    float *fext_f = nullptr;            // fext in FP32 (not for FP64 storage)
    float2 *link = nullptr;             // wall-link records of the tile kernel (KParams::link)
    uint16_t *links = nullptr;          // wall bits of every node (KParams::links)
    void *walls = nullptr;     // one allocation, the arrays of lbm_set_wall_density:
    double *wall_rho = nullptr, *wall_psi = nullptr;  // per solid node virtual density, its psi
    float *wall_psi_f = nullptr;        // wall_psi in FP32 (not for FP64 storage)
    double *dacc = nullptr;             // diagnostics: 9 sums, max |u|, count of non-finite nodes
    double *scratch = nullptr;          // host<->device staging for FP64 field copies
    size_t scratch_bytes = 0;
    int *derr = nullptr;
    bool initialised = false;
    bool fused_ok = false;
    cudaError_t (*one_pass)(const KParams &, cudaStream_t) = nullptr;  // the step's kernel; null: two-pass
    int64_t steps = 0;
    int64_t n_fluid = 0;                // nodes that are not solid
    Launchers L{};
    KParams kp{};
    std::string err;
    AdjointState *adj = nullptr;
};

static thread_local std::string g_create_error;

static lbm_status fail(lbm_ctx *c, lbm_status s, const std::string &msg)
{
    if (c) c->err = msg;
    else g_create_error = msg;
    return s;
}

static lbm_status cuda_fail(lbm_ctx *c, cudaError_t e, const char *what)
{
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    return fail(c, e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, m);
}

#define CK(call, what)                                   \
    do {                                                 \
        cudaError_t e_ = (call);                         \
        if (e_ != cudaSuccess) return cuda_fail(c, e_, what); \
    } while (0)

// ------------------------------------------------------------- params ------

static double host_p_eos(const lbm_params &p, double rho)
{
    if (p.eos == LBM_EOS_VDW) return p.K_eos * (rho * p.R * p.T / (1.0 - p.b * rho) - p.a * rho * rho);
    double eta = p.b * rho / 4.0;
    double num = 1.0 + eta + eta * eta - eta * eta * eta;
    double om = 1.0 - eta;
    return p.K_eos * (rho * p.R * p.T * num / (om * om * om) - p.a * rho * rho);
}

static double host_psi(const lbm_params &p, double rho) { return std::sqrt(2.0 * (host_p_eos(p, rho) - rho / 3.0) / p.G); }

extern "C" lbm_status lbm_params_default(lbm_params *p)
{
    if (!p) return LBM_EINVAL;
    std::memset(p, 0, sizeof(*p));
    p->struct_size = (int32_t)sizeof(lbm_params);
    p->nx = 4;
    p->ny = 128;
    p->periodic_x = 1;
    p->periodic_y = 0;
    p->precision = LBM_F64;
    p->scheme = LBM_SCHEME_IMPROVED;
    p->eos = LBM_EOS_CS;
    p->force_mode = LBM_FORCE_CONST;
    p->kernel = LBM_KERNEL_AUTO;
    p->storage_rounding = 1;
    p->a = 1.0;
    p->b = 4.0;
    p->R = 1.0;
    p->T = 0.7 * 0.3773 * 1.0 / (4.0 * 1.0);
    p->K_eos = 1.0;
    p->G = -1.0;
    p->k1 = p->k2 = -1.895 / 16.0;
    p->tau_l = p->tau_g = 0.8;
    p->rho_l = 0.3581443962580134;   // Maxwell densities of this EOS at 0.7 T_c
    p->rho_g = 0.009291723294794338;
    p->Lambda = 1.0 / 12.0;
    p->rho_s = p->rho_g;
    p->rho_ref = p->rho_g;
    p->rho_max = 0.0;
    return LBM_OK;
}

static lbm_status validate(lbm_ctx *c, const lbm_params &p)
{
    if (p.struct_size != (int32_t)sizeof(lbm_params)) return fail(c, LBM_EINVAL, "lbm_params.struct_size does not match this library");
    if (p.nx < 1 || p.ny < 1) return fail(c, LBM_EINVAL, "nx and ny must be >= 1");
    if ((int64_t)p.nx * p.ny > (int64_t)1 << 31) return fail(c, LBM_EINVAL, "lattice larger than 2^31 nodes");
    if (p.ny > 65535) return fail(c, LBM_EINVAL, "ny must be <= 65535 (one grid row of blocks per lattice row)");
    if (p.precision < LBM_F64 || p.precision > LBM_BF16DEV) return fail(c, LBM_EINVAL, "unknown precision");
    if (p.scheme != LBM_SCHEME_ORIGINAL && p.scheme != LBM_SCHEME_IMPROVED) return fail(c, LBM_EINVAL, "unknown scheme");
    if (p.eos != LBM_EOS_VDW && p.eos != LBM_EOS_CS) return fail(c, LBM_EINVAL, "unknown eos");
    if (p.force_mode < LBM_FORCE_CONST || p.force_mode > LBM_FORCE_FIELD) return fail(c, LBM_EINVAL, "unknown force_mode");
    if (p.kernel < LBM_KERNEL_AUTO || p.kernel > LBM_KERNEL_FUSED) return fail(c, LBM_EINVAL, "unknown kernel");
    if (!(p.tau_l > 0.5) || !(p.tau_g > 0.5)) return fail(c, LBM_EINVAL, "tau must be > 1/2");
    if (!(p.G < 0.0)) return fail(c, LBM_EINVAL, "G must be < 0");
    if (!(p.Lambda > 0.0)) return fail(c, LBM_EINVAL, "Lambda must be > 0");
    if (p.tau_l != p.tau_g && !(p.rho_l > p.rho_g)) return fail(c, LBM_EINVAL, "rho_l must exceed rho_g when tau_l != tau_g");
    if (p.storage_scale_log2 < -30 || p.storage_scale_log2 > 30) return fail(c, LBM_EINVAL, "storage_scale_log2 out of range");
    if (p.storage_rounding != 0 && p.storage_rounding != 1) return fail(c, LBM_EINVAL, "storage_rounding must be 0 or 1");
    if (p.diag_every < 0) return fail(c, LBM_EINVAL, "diag_every must be >= 0");
    if (p.precision == LBM_F16DEV && (p.storage_scale_log2 < -15 || p.storage_scale_log2 > 24))
        return fail(c, LBM_EINVAL, "FP16 storage needs storage_scale_log2 in [-15, 24] (2^-k must be an FP16 value)");
    double rmax = p.rho_max > 0 ? p.rho_max : 1.25 * std::fmax(std::fmax(p.rho_l, p.rho_g), p.rho_s);
    if (!(rmax > 0)) return fail(c, LBM_EINVAL, "rho_max must be > 0");
    for (int k = 1; k <= 4096; ++k) {
        double rho = rmax * k / 4096.0;
        double d = host_p_eos(p, rho) - rho / 3.0;
        if (!(d < 0.0)) {
            char buf[160];
            std::snprintf(buf, sizeof buf, "p_EOS - rho/3 >= 0 at rho = %.6g: psi is not real on (0, rho_max]", rho);
            return fail(c, LBM_EINVAL, buf);
        }
    }
    if (!(host_psi(p, p.rho_s) > 0)) return fail(c, LBM_EINVAL, "psi(rho_s) is not real");
    return LBM_OK;
}

// Derived kernel constants of the current parameters (Secs. 2-3).
static void fill_constants(lbm_ctx *c)
{
    const lbm_params &p = c->p;
    KParams &k = c->kp;
    k.nx = p.nx;
    k.ny = p.ny;
    k.device = c->device;
    k.sm_count = c->sm_count;
    k.pitch = c->pitch;
    k.plane = c->plane;
    k.periodic_x = p.periodic_x != 0;
    k.periodic_y = p.periodic_y != 0;
    k.improved = p.scheme == LBM_SCHEME_IMPROVED;
    k.eos = p.eos;
    k.force_mode = p.force_mode;
    k.var_tau = p.tau_l != p.tau_g;
    k.per_node_ref = (p.precision >= LBM_F16DEV) && p.per_node_ref;
    k.sr = (p.precision >= LBM_F16DEV) && p.storage_rounding;
    k.eos_a = p.a;
    k.eos_b = p.b;
    k.eos_RT = p.R * p.T;
    k.eos_K = p.K_eos;
    k.two_over_G = 2.0 / p.G;
    k.eos_R = p.R;
    k.eos_T = p.T;
    k.k1 = p.k1;
    k.k2 = p.k2;
    k.G = p.G;
    const double eps = -8.0 * (p.k1 + p.k2);
    k.q1c = 3.0 * (p.k1 + 2.0 * p.k2);
    k.q4a = (30.0 * eps - 15.0) / 16.0;
    k.q4b = 3.0 * eps / 8.0;
    k.two_inv_G = 2.0 / p.G;
    k.eos_b4 = p.b / 4.0;
    k.unit_R = p.R == 1.0;
    k.unit_K = p.K_eos == 1.0;
    int g_exp;
    k.G_pow2 = std::frexp(p.G, &g_exp) == -0.5 && std::abs(g_exp) < 500;
    k.kq1 = 3.0 * (p.k1 + 2.0 * p.k2) * p.G;
    k.kq7 = p.k1 * p.G;
    k.c1G = (30.0 * eps - 15.0) / 16.0 * p.G;
    k.c2G = 3.0 * eps / 8.0 * p.G;
    k.q2fac = (p.scheme == LBM_SCHEME_ORIGINAL || p.q2_original) ? -1.0 : -0.5;
    k.q2_full = k.q2fac == -1.0;
    const double tau = p.tau_l;
    k.sp = 1.0 / tau;
    k.sq = 1.0 / (0.5 + p.Lambda / (tau - 0.5));
    k.nu_l = (p.tau_l - 0.5) / 3.0;
    k.nu_g = (p.tau_g - 0.5) / 3.0;
    k.rho_l = p.rho_l;
    k.rho_g = p.rho_g;
    k.Lambda = p.Lambda;
    k.Fx = p.Fx;
    k.Fy = p.Fy;
    k.psi_s = host_psi(p, p.rho_s);
    k.rho_s = p.rho_s;
    k.rho_ref = p.rho_ref;
    k.scale = std::ldexp(1.0, p.storage_scale_log2);
    k.inv_scale = std::ldexp(1.0, -p.storage_scale_log2);
    // the same constants in each kernel arithmetic type
#define LBM_FILL(f) k.cd.f = k.f; k.cf.f = (float)k.f;
    LBM_FILL(eos_a) LBM_FILL(eos_b) LBM_FILL(eos_RT) LBM_FILL(eos_R) LBM_FILL(eos_K) LBM_FILL(two_over_G) LBM_FILL(G)
    LBM_FILL(kq1) LBM_FILL(kq7) LBM_FILL(c1G) LBM_FILL(c2G) LBM_FILL(q2fac) LBM_FILL(sp) LBM_FILL(sq)
    LBM_FILL(nu_l) LBM_FILL(nu_g) LBM_FILL(rho_l) LBM_FILL(rho_g) LBM_FILL(Lambda) LBM_FILL(Fx) LBM_FILL(Fy)
    LBM_FILL(psi_s) LBM_FILL(rho_s) LBM_FILL(rho_ref) LBM_FILL(scale) LBM_FILL(inv_scale)
#undef LBM_FILL
    k.cd.hsp = 1.0 - 0.5 * k.sp;
    k.cd.hsq = 1.0 - 0.5 * k.sq;
    k.cf.hsp = 1.0f - 0.5f * (float)k.sp;
    k.cf.hsq = 1.0f - 0.5f * (float)k.sq;
    {
        auto P = [](float v) { return make_float2(v, v); };
        PairConsts &q = k.c2;
        const Consts<float> &f = k.cf;
        q.m_G = P(-f.G), q.kq1 = P(f.kq1), q.q2fac = P(f.q2fac), q.kq7 = P(f.kq7), q.c1G = P(f.c1G), q.m_c2G = P(-f.c2G);
        q.sp = P(f.sp), q.sq = P(f.sq), q.hsp = P(f.hsp), q.six_hsp = P(6.f * f.hsp);
        q.m_six_hsp = P(-6.f * f.hsp), q.m_hsq = P(-f.hsq);
        q.Fx = P(f.Fx), q.Fy = P(f.Fy), q.rho_g = P(f.rho_g), q.inv_drho = P(1.0f / (f.rho_l - f.rho_g));
        q.dnu = P(f.nu_l - f.nu_g), q.nu_g = P(f.nu_g), q.Lambda = P(f.Lambda);
        q.m_b = P(-f.eos_b), q.b4 = P(f.eos_b * 0.25f), q.K = P(f.eos_K), q.RT = P(f.eos_RT), q.a = P(f.eos_a);
        q.two_over_G = P(f.two_over_G);
        q.scale = P(f.scale), q.m_scale = P(-f.scale);
        // 2^-k as FP16 (normal for k <= 14, subnormal down to 2^-24) or BF16 bits
        const int kk = p.storage_scale_log2;
        if (p.precision == LBM_BF16DEV) k.inv_scale_bits = (unsigned short)((127 - kk) << 7);
        else k.inv_scale_bits = kk <= 14 ? (unsigned short)((15 - kk) << 10) : (unsigned short)(1u << (24 - kk));
        for (int i = 0; i < 9; ++i) {
            const float w = i == 0 ? 4.0f / 9.0f : (i <= 4 ? 1.0f / 9.0f : 1.0f / 36.0f);
            const float wr = w * f.rho_ref;  // rounded like the kernels' w_i rho_ref
            q.w[i] = P(w);
            q.dec[i] = P(wr);
            q.enc[i] = P(-(wr * f.scale));
        }
    }
    k.psi = c->psi;
    k.solid = c->solid;
    k.wall_u = c->wall_u;
    k.q = c->q;
    k.fext = c->fext;
    k.wall_rho = c->wall_rho;
    k.wall_psi = c->wall_psi;
    k.fext_f = c->fext_f;
    k.wall_psi_f = c->wall_psi_f;
    k.link = c->link;
    k.links = c->links;
    k.skip_solid = c->n_fluid * 8 < (int64_t)p.nx * p.ny * 7;
    k.err = c->derr;
}

static void bind_buffers(lbm_ctx *c, int src)
{
    c->kp.src = c->pops[src];
    c->kp.dst = c->pops[src ^ 1];
    c->kp.ref_src = c->refp[src];
    c->kp.ref_dst = c->refp[src ^ 1];
}

static bool fused_possible(const lbm_ctx *c)
{
    const lbm_params &p = c->p;
    if ((c->solid || c->q || c->wall_u) && !c->L.fused_geometry) return false;
    if (c->L.fused_align <= 0 || p.nx % c->L.fused_align != 0) return false;
    // (the staged kernel's wrapped halo segment of the last strip must fit inside the lattice)
    if (p.nx < c->L.fused_tile_x + 16 || p.ny < 4) return false;
    return true;
}

// Which of the two requestable steps an LBM_KERNEL_AUTO context takes: LBM_KERNEL_FUSED's from these sizes on.  The
// tile kernel rounds accordingly (KParams::packed).
static bool auto_prefers_fused(const lbm_ctx *c)
{
    const int64_t n = (int64_t)c->p.nx * c->p.ny;
    if (c->q || c->wall_u) return n >= (int64_t(1) << 22);
    if (c->solid) return n >= (int64_t(1) << (c->p.precision == LBM_F32 ? 19 : 18));
    return (n >= (int64_t(1) << 18) && c->p.nx >= 512) || n >= (int64_t(1) << 21);
}

// Whether the context takes the step of LBM_KERNEL_FUSED (lbm_kernel_in_use).
static bool fused_step(const lbm_ctx *c)
{
    const int want = c->p.kernel;
    return want != LBM_KERNEL_TWO_PASS && fused_possible(c) &&
           (want == LBM_KERNEL_FUSED || c->p.precision == LBM_F64 || auto_prefers_fused(c));
}

// Which kernel steps the context: the two-pass kernels on request (LBM_KERNEL_TWO_PASS); else a
// one-pass kernel, the staged one (k_fused2) or the tile kernel (k_tile), which gives the two-pass
// step's results (where the context takes the step of LBM_KERNEL_FUSED: the staged one's).  The staged kernel
// reads each row once where the tile kernel re-reads its tiles' rings from L2, but a CTA walks its rows in
// series, and it has no walls; the tile kernel has thousands of short blocks.  Step times on a GB300 (us, tile /
// staged): FP32 periodic 512^2 5.0 / 10.2, 1024^2 13.0 / 22.8, 2048^2 48.7 / 56.4, 4096^2 183 / 195, 8192^2
// 744 / 746 (759 with exact products); FP16, whose ring costs instructions and not bytes, constant (buoyant) force, 1024^2 16.6 / 27.0
// (16.8 / 28.6), 1536 x 2048 46.4 / 53.6 (47.2 / 58.2), 2048^2 60.6 / 58.8 (61.1 / 63.8), 4096^2 226 / 194
// (226 / 213): the line at 3 2^20 is a little low.  (Two-pass kernels, FP32: 512^2 10.3, 1024^2 31, 2048^2
// 121; 256 x 2048 with walls 20.6 against the tile kernel's 8.9; banded 512^2 17.6 / 5.9; annulus 1024^2 44 / 16.)
static void choose_kernel(lbm_ctx *c)
{
    const int want = c->p.kernel;
    const bool possible = fused_possible(c);
    c->fused_ok = fused_step(c);
    const bool staged = possible && c->L.fused_pass && c->p.periodic_x && c->p.periodic_y && !c->solid && !c->q && !c->wall_u;
    const int64_t n = (int64_t)c->p.nx * c->p.ny;
    const bool large = n >= (c->p.precision == LBM_F32 ? (int64_t)1 << 25 : (int64_t)3 << 20);
    c->kp.packed = c->fused_ok && c->p.precision != LBM_F64;
    c->one_pass = nullptr;
    if (want == LBM_KERNEL_TWO_PASS || (want == LBM_KERNEL_FUSED && !possible)) return;
    c->one_pass = staged && (want == LBM_KERNEL_FUSED || large) ? c->L.fused_pass : c->L.tile_pass;
}

// ------------------------------------------------------------- lifetime ----

static void free_all(lbm_ctx *c)
{
    if (!c) return;
    if (c->stream) cudaStreamSynchronize(c->stream);
    void *bufs[] = {c->pops[0], c->pops[1], c->refp[0], c->refp[1], c->psi, c->geometry, c->walls, c->dacc, c->scratch, c->derr};
    for (void *b : bufs)
        if (b) cudaFree(b);
    adjoint_free(c->adj);
    c->adj = nullptr;
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

extern "C" lbm_status lbm_create(const lbm_params *p, void *cuda_stream, lbm_ctx **out)
{
    if (!p || !out) return fail(nullptr, LBM_EINVAL, "null argument");
    *out = nullptr;
    lbm_status s = validate(nullptr, *p);
    if (s != LBM_OK) return s;
    lbm_ctx *c = new (std::nothrow) lbm_ctx();
    if (!c) return fail(nullptr, LBM_ENOMEM, "host allocation failed");
    c->p = *p;
    cudaError_t e = cudaGetDevice(&c->device);
    if (e != cudaSuccess) {
        delete c;
        return fail(nullptr, LBM_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    }
    e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device);
    if (e != cudaSuccess) {
        delete c;
        return fail(nullptr, LBM_ECUDA, std::string("cudaDeviceGetAttribute: ") + cudaGetErrorString(e));
    }
    if (cuda_stream) {
        c->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            delete c;
            return fail(nullptr, LBM_ECUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
        }
        c->own_stream = true;
    }
    switch (p->precision) {
    case LBM_F64: c->L = launchers_f64(); c->elem = 8; c->real = 8; break;
    case LBM_F32: c->L = launchers_f32(); c->elem = 4; c->real = 4; break;
    case LBM_F16DEV: c->L = launchers_f16(); c->elem = 2; c->real = 4; break;
    default: c->L = launchers_bf16(); c->elem = 2; c->real = 4; break;
    }
    const int64_t per_line = 128 / (int64_t)c->elem;
    c->pitch = ((int64_t)p->nx + per_line - 1) / per_line * per_line;
    c->plane = c->pitch * p->ny;
    const int64_t n = (int64_t)p->nx * p->ny;
    const size_t pop_bytes = (size_t)9 * c->plane * c->elem;
    auto alloc = [&](void **ptr, size_t bytes) -> bool {
        cudaError_t ee = cudaMalloc(ptr, bytes);
        if (ee != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        return true;
    };
    // the psi field, and between steps the diagnostics' rows of sums
    c->kp.nx = p->nx, c->kp.ny = p->ny;
    const size_t psi_bytes = std::max((size_t)n * c->real, (size_t)c->L.diag_rows(c->kp) * 11 * sizeof(double));
    bool ok = alloc(&c->pops[0], pop_bytes) && alloc(&c->pops[1], pop_bytes) &&
              alloc(&c->psi, psi_bytes) && alloc((void **)&c->dacc, 16 * sizeof(double)) &&
              alloc((void **)&c->derr, sizeof(int));
    if (ok && p->precision >= LBM_F16DEV && p->per_node_ref)
        ok = alloc((void **)&c->refp[0], (size_t)c->plane * 4) && alloc((void **)&c->refp[1], (size_t)c->plane * 4);
    if (!ok) {
        free_all(c);
        delete c;
        return fail(nullptr, LBM_ENOMEM, "device allocation failed");
    }
    cudaMemsetAsync(c->pops[0], 0, pop_bytes, c->stream);
    cudaMemsetAsync(c->pops[1], 0, pop_bytes, c->stream);
    cudaMemsetAsync(c->derr, 0, sizeof(int), c->stream);
    c->n_fluid = n;
    fill_constants(c);
    choose_kernel(c);
    e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        free_all(c);
        delete c;
        return fail(nullptr, LBM_ECUDA, std::string("create: ") + cudaGetErrorString(e));
    }
    *out = c;
    return LBM_OK;
}

extern "C" lbm_status lbm_destroy(lbm_ctx *c)
{
    if (!c) return LBM_OK;
    free_all(c);
    delete c;
    return LBM_OK;
}

// scratch device buffer of at least `bytes`
static lbm_status need_scratch(lbm_ctx *c, size_t bytes)
{
    if (c->scratch_bytes >= bytes) return LBM_OK;
    if (c->scratch) {
        cudaStreamSynchronize(c->stream);
        cudaFree(c->scratch);
        c->scratch = nullptr;
        c->scratch_bytes = 0;
    }
    CK(cudaMalloc((void **)&c->scratch, bytes), "cudaMalloc(scratch)");
    c->scratch_bytes = bytes;
    return LBM_OK;
}

// Arrays one behind the other in an allocation: an array has its place before there is one.
struct Places {
    size_t used = 0;
    size_t take(size_t bytes)
    {
        const size_t at = used;
        used += (bytes + 255) / 256 * 256;
        return at;
    }
};
// An array at its place, or null where it is not wanted.
template <class T>
static void put_at(T **p, void *base, size_t at, bool wanted)
{
    *p = wanted ? reinterpret_cast<T *>(static_cast<char *>(base) + at) : nullptr;
}

template <class T>
static lbm_status upload(lbm_ctx *c, T *dst, const T *src, size_t count, const char *what)
{
    if (src) CK(cudaMemcpyAsync(dst, src, count * sizeof(T), cudaMemcpyHostToDevice, c->stream), what);
    return LBM_OK;
}

static __global__ void k_narrow(const double *in, float *out, int64_t n)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = float(in[k]);
}

// dst = src[count] in FP32, for the storage types whose arithmetic is FP32 (null dst: not wanted).
static lbm_status narrow(lbm_ctx *c, float *dst, const double *src, size_t count, const char *what)
{
    if (!dst) return LBM_OK;
    k_narrow<<<(unsigned)((count + 255) / 256), 256, 0, c->stream>>>(src, dst, (int64_t)count);
    CK(cudaGetLastError(), what);
    return LBM_OK;
}

// Wall-link records of the tile kernel (KParams::link), built on the host from the
// geometry as given: for each fluid node x and pulled population i whose source x - e_i is a
// wall (a solid node or beyond a non-periodic edge), the link fraction q of the outgoing
// population o = opp(i) (1/2 without link fractions, and 1/2 where q < 1/2 but the second
// node x + e_i is a wall too -- the same fallback as the two-pass step's bounce-back) and
// the velocity of the wall node along e_i, or the whole moving-wall coefficient
// 2 w_o (e_i . u_w) 3 for the packed step (0 beyond an edge).
static std::vector<float2> link_records(const lbm_ctx *c, const uint8_t *solid, const double *wall_u, const double *q)
{
    static const int EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    static const int OPP[9] = {0, 3, 4, 1, 2, 7, 8, 5, 6};
    static const double W[9] = {4.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};
    const bool packed = fused_step(c);
    const int nx = c->p.nx, ny = c->p.ny;
    const int64_t n = (int64_t)nx * ny, pitch = c->pitch, plane = c->plane;
    auto wall_at = [&](int x, int y, int64_t *node) -> bool {
        if (x < 0 || x >= nx) {
            if (!c->p.periodic_x) return true;
            x = x < 0 ? x + nx : x - nx;
        }
        if (y < 0 || y >= ny) {
            if (!c->p.periodic_y) return true;
            y = y < 0 ? y + ny : y - ny;
        }
        *node = (int64_t)y * nx + x;
        return solid && solid[*node] != 0;
    };
    std::vector<float2> h((size_t)(8 * plane), make_float2(0.5f, 0.0f));
    for (int y = 0; y < ny; ++y)
        for (int x = 0; x < nx; ++x) {
            const int64_t node = (int64_t)y * nx + x, k = (int64_t)y * pitch + x;
            if (solid && solid[node]) continue;
            for (int i = 1; i < 9; ++i) {
                int64_t wn = -1;
                if (!wall_at(x - EX[i], y - EY[i], &wn)) continue;
                const int o = OPP[i];
                double qq = q ? q[(int64_t)(o - 1) * n + node] : 0.5;
                int64_t bn;
                if (qq < 0.5 && wall_at(x + EX[i], y + EY[i], &bn)) qq = 0.5;
                float cw = 0.f;
                if (wall_u && wn >= 0)
                    cw = packed ? (float)(2.0 * W[o] * (EX[i] * wall_u[wn] + EY[i] * wall_u[n + wn]) * 3.0)
                                : (float)EX[i] * (float)wall_u[wn] + (float)EY[i] * (float)wall_u[n + wn];
                h[(size_t)((i - 1) * plane + k)] = make_float2((float)qq, cw);
            }
        }
    return h;
}

static void drop_geometry(lbm_ctx *c)
{
    if (c->geometry) {
        cudaStreamSynchronize(c->stream);
        cudaFree(c->geometry);
    }
    c->geometry = nullptr;
    c->solid = nullptr, c->wall_u = c->q = c->fext = nullptr, c->fext_f = nullptr, c->link = nullptr, c->links = nullptr;
    c->n_fluid = (int64_t)c->p.nx * c->p.ny;
}

static lbm_status build_geometry(lbm_ctx *c, const uint8_t *solid, const double *wall_u, const double *q,
                                 const double *force_field)
try {
    const size_t n = (size_t)c->p.nx * c->p.ny;
    const bool f32 = c->p.precision != LBM_F64, walls = solid || wall_u || q, records = f32 && (wall_u || q);
    Places at;
    const size_t at_solid = at.take(solid ? n : 0), at_wall_u = at.take(wall_u ? 2 * n * sizeof(double) : 0);
    const size_t at_q = at.take(q ? 8 * n * sizeof(double) : 0), at_fext = at.take(force_field ? 2 * n * sizeof(double) : 0);
    const size_t at_fext_f = at.take(force_field && f32 ? 2 * n * sizeof(float) : 0);
    const size_t at_link = at.take(records ? 8 * c->plane * sizeof(float2) : 0), at_links = at.take(walls ? n * sizeof(uint16_t) : 0);
    if (at.used == 0) return LBM_OK;
    CK(cudaMalloc(&c->geometry, at.used), "geometry");
    put_at(&c->solid, c->geometry, at_solid, solid != nullptr), put_at(&c->wall_u, c->geometry, at_wall_u, wall_u != nullptr);
    put_at(&c->q, c->geometry, at_q, q != nullptr), put_at(&c->fext, c->geometry, at_fext, force_field != nullptr);
    put_at(&c->fext_f, c->geometry, at_fext_f, force_field && f32), put_at(&c->link, c->geometry, at_link, records);
    put_at(&c->links, c->geometry, at_links, walls);
    if (solid)
        for (size_t k = 0; k < n; ++k) c->n_fluid -= solid[k] != 0;
    lbm_status s;
    if ((s = upload(c, c->solid, solid, n, "solid")) != LBM_OK) return s;
    if ((s = upload(c, c->wall_u, wall_u, 2 * n, "wall_u")) != LBM_OK) return s;
    if ((s = upload(c, c->q, q, 8 * n, "q")) != LBM_OK) return s;
    if ((s = upload(c, c->fext, force_field, 2 * n, "force_field")) != LBM_OK) return s;
    if ((s = narrow(c, c->fext_f, c->fext, 2 * n, "force_field")) != LBM_OK) return s;
    std::vector<float2> h;
    if (records) h = link_records(c, solid, wall_u, q);
    if (records && (s = upload(c, c->link, (const float2 *)h.data(), h.size(), "link records")) != LBM_OK) return s;
    if (walls) {
        fill_constants(c);
        CK(c->L.link_bits(c->kp, c->links, c->stream), "wall bits kernel");
    }
    CK(cudaStreamSynchronize(c->stream), "set_geometry");
    return LBM_OK;
} catch (const std::bad_alloc &) {
    return fail(c, LBM_ENOMEM, "host allocation failed");
}

extern "C" lbm_status lbm_set_geometry(lbm_ctx *c, const uint8_t *solid, const double *wall_u, const double *q,
                                       const double *force_field)
{
    if (!c) return LBM_EINVAL;
    const size_t n = (size_t)c->p.nx * c->p.ny;
    if (q) {
        for (size_t k = 0; k < 8 * n; ++k)
            if (!(q[k] > 0.0 && q[k] <= 1.0)) return fail(c, LBM_EINVAL, "q must lie in (0, 1]");
    }
    drop_geometry(c);
    const lbm_status s = build_geometry(c, solid, wall_u, q, force_field);
    if (s != LBM_OK) drop_geometry(c);  // (the old arrays gave way to the new ones, which are not all there)
    fill_constants(c);
    choose_kernel(c);
    return s;
}

static void drop_wall_density(lbm_ctx *c)
{
    if (c->walls) {
        cudaStreamSynchronize(c->stream);
        cudaFree(c->walls);
    }
    c->walls = nullptr;
    c->wall_rho = c->wall_psi = nullptr, c->wall_psi_f = nullptr;
}

static lbm_status build_wall_density(lbm_ctx *c, const double *wall_rho, const double *psi)
{
    const size_t n = (size_t)c->p.nx * c->p.ny;
    const bool f32 = c->p.precision != LBM_F64;
    Places at;
    const size_t at_rho = at.take(n * sizeof(double)), at_psi = at.take(n * sizeof(double)), at_psi_f = at.take(f32 ? n * sizeof(float) : 0);
    CK(cudaMalloc(&c->walls, at.used), "wall densities");
    put_at(&c->wall_rho, c->walls, at_rho, true), put_at(&c->wall_psi, c->walls, at_psi, true), put_at(&c->wall_psi_f, c->walls, at_psi_f, f32);
    lbm_status s;
    if ((s = upload(c, c->wall_rho, wall_rho, n, "wall_rho")) != LBM_OK) return s;
    if ((s = upload(c, c->wall_psi, psi, n, "wall_psi")) != LBM_OK) return s;
    if ((s = narrow(c, c->wall_psi_f, c->wall_psi, n, "wall_psi")) != LBM_OK) return s;
    CK(cudaStreamSynchronize(c->stream), "set_wall_density");
    return LBM_OK;
}

// psi of n wall densities under the parameters p: the same host evaluation as psi(rho_s), so a uniform field
// equals the scalar.  False where one is not real and positive.
static bool wall_psi_of(const lbm_params &p, const double *wall_rho, size_t n, std::vector<double> &psi)
{
    psi.resize(n);
    for (size_t k = 0; k < n; ++k) {
        psi[k] = host_psi(p, wall_rho[k]);
        if (!(wall_rho[k] > 0.0) || !(psi[k] > 0.0) || !std::isfinite(psi[k])) return false;
    }
    return true;
}

extern "C" lbm_status lbm_set_wall_density(lbm_ctx *c, const double *wall_rho)
try {
    if (!c) return LBM_EINVAL;
    const size_t n = (size_t)c->p.nx * c->p.ny;
    std::vector<double> psi;
    if (wall_rho && !wall_psi_of(c->p, wall_rho, n, psi))
        return fail(c, LBM_EINVAL, "psi of a wall density is not real and positive");
    drop_wall_density(c);
    const lbm_status s = wall_rho ? build_wall_density(c, wall_rho, psi.data()) : LBM_OK;
    if (s != LBM_OK) drop_wall_density(c);
    fill_constants(c);
    choose_kernel(c);
    return s;
} catch (const std::bad_alloc &) {
    return fail(c, LBM_ENOMEM, "host allocation failed");
}

// Bring `count` doubles from host or device into a device pointer (scratch slot `slot`).
static lbm_status device_input(lbm_ctx *c, const double *src, int on_device, size_t count, size_t slot,
                               const double **out)
{
    if (!src) {
        *out = nullptr;
        return LBM_OK;
    }
    if (on_device) {
        *out = src;
        return LBM_OK;
    }
    double *d = c->scratch + slot * count;
    CK(cudaMemcpyAsync(d, src, count * sizeof(double), cudaMemcpyHostToDevice, c->stream), "H2D");
    *out = d;
    return LBM_OK;
}

extern "C" lbm_status lbm_init_fields(lbm_ctx *c, const double *rho, const double *ux, const double *uy,
                                      int on_device)
{
    if (!c || !rho) return c ? fail(c, LBM_EINVAL, "rho is required") : LBM_EINVAL;
    const size_t n = (size_t)c->p.nx * c->p.ny;
    lbm_status s;
    if (!on_device && (s = need_scratch(c, 3 * n * sizeof(double))) != LBM_OK) return s;
    const double *dr, *du, *dv;
    if ((s = device_input(c, rho, on_device, n, 0, &dr)) != LBM_OK) return s;
    if ((s = device_input(c, ux, on_device, n, 1, &du)) != LBM_OK) return s;
    if ((s = device_input(c, uy, on_device, n, 2, &dv)) != LBM_OK) return s;
    c->cur = 0;
    bind_buffers(c, 1);  // init writes kp.dst = pops[0]
    CK(c->L.init(c->kp, dr, du, dv, c->stream), "init kernel");
    if (!on_device) CK(cudaStreamSynchronize(c->stream), "init");
    c->steps = 0;
    c->initialised = true;
    return LBM_OK;
}

// CTAs of the cluster that takes a call's steps in the small-lattice kernel; 0: one launch per step.  Asked when a
// call could use it: the first question in a process loads the kernel (12 ms), which a program that takes its
// steps one by one does not need.
static int small_ctas(const lbm_ctx *c, int64_t nsteps)
{
    return c->p.kernel == LBM_KERNEL_AUTO && nsteps >= 4 ? c->L.small_ctas(c->kp) : 0;
}

// How many of the next nsteps steps it takes in one launch (no more than 4096, so that no launch takes long); 0:
// none (fewer than four are as fast one by one).
static int64_t at_once(int ctas, int64_t nsteps) { return ctas > 0 && nsteps >= 4 ? std::min<int64_t>(nsteps, 4096) : 0; }

static lbm_status run_steps(lbm_ctx *c, int64_t nsteps)
{
    const int ctas = small_ctas(c, nsteps);
    while (const int64_t n = at_once(ctas, nsteps)) {
        bind_buffers(c, c->cur);
        CK(c->L.small_steps(c->kp, ctas, n, c->steps, c->stream), "small-lattice kernel");
        c->cur ^= (int)(n & 1);
        c->steps += n;
        c->kp.sr_seed = sr_seed_of(c->steps - 1);
        nsteps -= n;
    }
    for (int64_t t = 0; t < nsteps; ++t) {
        bind_buffers(c, c->cur);
        c->kp.sr_seed = sr_seed_of(c->steps);
        if (c->one_pass) {
            CK(c->one_pass(c->kp, c->stream), "one-pass step kernel");
        } else {
            CK(c->L.psi_pass(c->kp, c->stream), "psi kernel");
            CK(c->L.collide_pass(c->kp, c->stream), "collide kernel");
        }
        c->cur ^= 1;
        c->steps += 1;
    }
    return LBM_OK;
}

// Wait for the context stream and read the device error word (set by a bounded device-side
// wait that ran out, or a failed bounds check, in any step launched so far).  Every call
// that synchronises anyway reads it: lbm_sync, the host-side getters and lbm_save_state.
static lbm_status sync_and_check(lbm_ctx *c, const char *what)
{
    int h = 0;
    CK(cudaMemcpyAsync(&h, c->derr, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "error word");
    CK(cudaStreamSynchronize(c->stream), what);
    if (h & DERR_TIMEOUT) return fail(c, LBM_ETIMEOUT, "a device-side wait ran out of iterations");
    if (h & DERR_BOUNDS) return fail(c, LBM_EBOUNDS, "a device-side bounds check failed");
    return LBM_OK;
}

extern "C" lbm_status lbm_step(lbm_ctx *c, int64_t nsteps)
{
    if (!c) return LBM_EINVAL;
    if (!c->initialised) return fail(c, LBM_ESTATE, "fields not initialised");
    if (nsteps < 0) return fail(c, LBM_EINVAL, "nsteps < 0");
    const int64_t D = c->p.diag_every;
    if (D <= 0) return run_steps(c, nsteps);
    // launch up to the next multiple of D, then wait and check the state there
    while (nsteps > 0) {
        const int64_t n = std::min<int64_t>(nsteps, D - c->steps % D);
        lbm_status s = run_steps(c, n);
        if (s != LBM_OK) return s;
        nsteps -= n;
        if (c->steps % D == 0) {
            double d[LBM_NDIAG];
            if ((s = lbm_get_diagnostics(c, d)) != LBM_OK) return s;
        }
    }
    return LBM_OK;
}

extern "C" lbm_status lbm_get_moments(lbm_ctx *c, double *rho, double *ux, double *uy, int on_device)
{
    if (!c) return LBM_EINVAL;
    if (!c->initialised) return fail(c, LBM_ESTATE, "fields not initialised");
    const size_t n = (size_t)c->p.nx * c->p.ny;
    lbm_status s;
    bind_buffers(c, c->cur);
    if (on_device) {
        CK(c->L.moments(c->kp, rho, ux, uy, c->stream), "moments kernel");
        return LBM_OK;
    }
    if ((s = need_scratch(c, 3 * n * sizeof(double))) != LBM_OK) return s;
    double *d = c->scratch;
    CK(c->L.moments(c->kp, rho ? d : nullptr, ux ? d + n : nullptr, uy ? d + 2 * n : nullptr, c->stream), "moments kernel");
    if (rho) CK(cudaMemcpyAsync(rho, d, n * 8, cudaMemcpyDeviceToHost, c->stream), "D2H");
    if (ux) CK(cudaMemcpyAsync(ux, d + n, n * 8, cudaMemcpyDeviceToHost, c->stream), "D2H");
    if (uy) CK(cudaMemcpyAsync(uy, d + 2 * n, n * 8, cudaMemcpyDeviceToHost, c->stream), "D2H");
    return sync_and_check(c, "get_moments");
}

extern "C" lbm_status lbm_get_diagnostics(lbm_ctx *c, double out[LBM_NDIAG])
{
    if (!c || !out) return LBM_EINVAL;
    if (!c->initialised) return fail(c, LBM_ESTATE, "fields not initialised");
    lbm_status s;
    bind_buffers(c, c->cur);
    CK(c->L.diag(c->kp, static_cast<double *>(c->psi), c->dacc, c->stream), "diagnostics kernel");
    double h[11];
    CK(cudaMemcpyAsync(h, c->dacc, sizeof h, cudaMemcpyDeviceToHost, c->stream), "D2H");
    if ((s = sync_and_check(c, "diagnostics")) != LBM_OK) return s;
    for (int k = 0; k < 10; ++k) out[k] = h[k];
    if (h[10] > 0 || !std::isfinite(out[0])) return fail(c, LBM_ENAN, "non-finite density or velocity");
    return LBM_OK;
}

extern "C" lbm_status lbm_get_state(lbm_ctx *c, double *pops, int on_device)
{
    if (!c || !pops) return LBM_EINVAL;
    const size_t n = (size_t)c->p.nx * c->p.ny;
    bind_buffers(c, c->cur);
    if (on_device) {
        CK(c->L.get_state(c->kp, pops, c->stream), "get_state kernel");
        return LBM_OK;
    }
    lbm_status s;
    if ((s = need_scratch(c, 9 * n * sizeof(double))) != LBM_OK) return s;
    CK(c->L.get_state(c->kp, c->scratch, c->stream), "get_state kernel");
    CK(cudaMemcpyAsync(pops, c->scratch, 9 * n * 8, cudaMemcpyDeviceToHost, c->stream), "D2H");
    return sync_and_check(c, "get_state");
}

extern "C" lbm_status lbm_set_state(lbm_ctx *c, const double *pops, int on_device)
{
    if (!c || !pops) return LBM_EINVAL;
    const size_t n = (size_t)c->p.nx * c->p.ny;
    const double *src = pops;
    if (!on_device) {
        lbm_status s;
        if ((s = need_scratch(c, 9 * n * sizeof(double))) != LBM_OK) return s;
        CK(cudaMemcpyAsync(c->scratch, pops, 9 * n * 8, cudaMemcpyHostToDevice, c->stream), "H2D");
        src = c->scratch;
    }
    c->cur = 0;
    bind_buffers(c, 1);
    CK(c->L.set_state(c->kp, src, c->stream), "set_state kernel");
    if (!on_device) CK(cudaStreamSynchronize(c->stream), "set_state");
    c->steps = 0;
    c->initialised = true;
    return LBM_OK;
}

// --------------------------------------------------- checkpoint / resume ---

struct SnapHeader {
    char magic[8];
    int32_t precision, per_node_ref, nx, ny;
    int64_t pitch, steps;
};

extern "C" lbm_status lbm_save_state(lbm_ctx *c, void *host_buf, size_t *nbytes)
{
    if (!c || !nbytes) return LBM_EINVAL;
    const size_t pop_bytes = (size_t)9 * c->plane * c->elem;
    const size_t ref_bytes = c->refp[0] ? (size_t)c->plane * 4 : 0;
    const size_t need = sizeof(SnapHeader) + pop_bytes + ref_bytes;
    if (!host_buf) {
        *nbytes = need;
        return LBM_OK;
    }
    if (*nbytes < need) return fail(c, LBM_EINVAL, "buffer too small");
    SnapHeader h{};
    std::memcpy(h.magic, "LBMSNAP1", 8);
    h.precision = c->p.precision;
    h.per_node_ref = ref_bytes != 0;
    h.nx = c->p.nx;
    h.ny = c->p.ny;
    h.pitch = c->pitch;
    h.steps = c->steps;
    std::memcpy(host_buf, &h, sizeof h);
    char *dst = static_cast<char *>(host_buf) + sizeof h;
    CK(cudaMemcpyAsync(dst, c->pops[c->cur], pop_bytes, cudaMemcpyDeviceToHost, c->stream), "save");
    if (ref_bytes) CK(cudaMemcpyAsync(dst + pop_bytes, c->refp[c->cur], ref_bytes, cudaMemcpyDeviceToHost, c->stream), "save");
    lbm_status s = sync_and_check(c, "save");
    if (s != LBM_OK) return s;
    *nbytes = need;
    return LBM_OK;
}

extern "C" lbm_status lbm_load_state(lbm_ctx *c, const void *host_buf, size_t nbytes)
{
    if (!c || !host_buf) return LBM_EINVAL;
    const size_t pop_bytes = (size_t)9 * c->plane * c->elem;
    const size_t ref_bytes = c->refp[0] ? (size_t)c->plane * 4 : 0;
    SnapHeader h;
    if (nbytes < sizeof h) return fail(c, LBM_EINVAL, "snapshot too small");
    std::memcpy(&h, host_buf, sizeof h);
    if (std::memcmp(h.magic, "LBMSNAP1", 8) != 0 || h.precision != c->p.precision || h.nx != c->p.nx ||
        h.ny != c->p.ny || h.pitch != c->pitch || (h.per_node_ref != 0) != (ref_bytes != 0) ||
        nbytes != sizeof h + pop_bytes + ref_bytes)
        return fail(c, LBM_EINVAL, "snapshot does not match this context");
    const char *src = static_cast<const char *>(host_buf) + sizeof h;
    c->cur = 0;
    CK(cudaMemcpyAsync(c->pops[0], src, pop_bytes, cudaMemcpyHostToDevice, c->stream), "load");
    if (ref_bytes) CK(cudaMemcpyAsync(c->refp[0], src + pop_bytes, ref_bytes, cudaMemcpyHostToDevice, c->stream), "load");
    CK(cudaStreamSynchronize(c->stream), "load");
    c->steps = h.steps;
    c->initialised = true;
    return LBM_OK;
}

// psi of the wall densities under the parameters p, into the arrays that hold it.
static lbm_status refresh_wall_psi(lbm_ctx *c, const lbm_params &p)
{
    const size_t n = (size_t)c->p.nx * c->p.ny;
    std::vector<double> rho(n), psi;
    CK(cudaMemcpyAsync(rho.data(), c->wall_rho, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "wall_rho");
    CK(cudaStreamSynchronize(c->stream), "wall_rho");
    if (!wall_psi_of(p, rho.data(), n, psi)) return fail(c, LBM_EINVAL, "psi of a wall density is not real and positive");
    lbm_status s;
    if ((s = upload(c, c->wall_psi, (const double *)psi.data(), n, "wall_psi")) != LBM_OK) return s;
    if ((s = narrow(c, c->wall_psi_f, c->wall_psi, n, "wall_psi")) != LBM_OK) return s;
    CK(cudaStreamSynchronize(c->stream), "wall_psi");
    return LBM_OK;
}

extern "C" lbm_status lbm_set_param(lbm_ctx *c, int32_t which, double value)
try {
    if (!c) return LBM_EINVAL;
    lbm_params np = c->p;
    switch (which) {
    case LBM_PARAM_FX: np.Fx = value; break;
    case LBM_PARAM_FY: np.Fy = value; break;
    case LBM_PARAM_G: np.G = value; break;
    case LBM_PARAM_T: np.T = value; break;
    default: return fail(c, LBM_EINVAL, "unknown parameter id");
    }
    lbm_status s = validate(c, np);
    if (s != LBM_OK) return s;
    if (c->wall_rho && (which == LBM_PARAM_G || which == LBM_PARAM_T) && (s = refresh_wall_psi(c, np)) != LBM_OK) return s;
    c->p = np;
    fill_constants(c);
    return LBM_OK;
} catch (const std::bad_alloc &) {
    return fail(c, LBM_ENOMEM, "host allocation failed");
}

extern "C" lbm_status lbm_adjoint_step(lbm_ctx *c, int64_t nsteps, int32_t checkpoint_every, int32_t objective,
                                       double *J, double grad[4], double *lambda0)
{
    if (!c || !J) return LBM_EINVAL;
    if (!c->initialised) return fail(c, LBM_ESTATE, "fields not initialised");
    std::string msg;
    lbm_status s = adjoint_run(c, nsteps, checkpoint_every, objective, J, grad, lambda0, msg);
    if (s != LBM_OK) return fail(c, s, msg);
    return LBM_OK;
}

extern "C" lbm_status lbm_sync(lbm_ctx *c)
{
    if (!c) return LBM_EINVAL;
    return sync_and_check(c, "sync");
}

extern "C" int64_t lbm_step_count(const lbm_ctx *c) { return c ? c->steps : -1; }

extern "C" int32_t lbm_kernel_in_use(const lbm_ctx *c)
{
    if (!c) return -1;
    return c->fused_ok ? LBM_KERNEL_FUSED : LBM_KERNEL_TWO_PASS;
}

extern "C" int64_t lbm_step_launches(const lbm_ctx *c, int64_t nsteps, int32_t *kernel)
{
    if (!c || nsteps < 0) return -1;
    const int64_t D = c->p.diag_every;
    const int ctas = small_ctas(c, nsteps);
    const int64_t first = D > 0 ? std::min<int64_t>(nsteps, D - c->steps % D) : nsteps, rest = nsteps - first;
    auto launches = [&](int64_t n) {
        const int64_t most = at_once(ctas, n);
        if (most == 0) return c->one_pass ? n : 2 * n;
        const int64_t left = n % most;
        return n / most + (at_once(ctas, left) ? 1 : c->one_pass ? left : 2 * left);
    };
    if (kernel)
        *kernel = at_once(ctas, rest > 0 ? std::max(first, std::min(rest, D)) : first) ? LBM_STEP_SMALL
                  : !c->one_pass                                                    ? LBM_STEP_TWO_PASS
                  : c->one_pass == c->L.fused_pass                                  ? LBM_STEP_STAGED
                                                                                    : LBM_STEP_TILE;
    return launches(first) + (rest > 0 ? rest / D * launches(D) + launches(rest % D) : 0);
}

extern "C" const char *lbm_last_error(const lbm_ctx *c)
{
    if (!c) return g_create_error.c_str();
    return c->err.c_str();
}

// ---------------------------------------------- accessors for the adjoint ---

namespace lbm {
ContextView view_of(lbm_ctx *c)
{
    ContextView v;
    v.p = &c->p;
    v.kp = &c->kp;
    v.stream = c->stream;
    v.pops = c->pops;
    v.refp = c->refp;
    v.cur = &c->cur;
    v.steps = &c->steps;
    v.elem = c->elem;
    v.plane = c->plane;
    v.adj = &c->adj;
    v.run_steps = [](lbm_ctx *cc, int64_t n) { return run_steps(cc, n); };
    v.sr_seed = [](int64_t t) { return sr_seed_of(t); };
    v.bind = [](lbm_ctx *cc, int src) { bind_buffers(cc, src); };
    v.psi_pass = c->L.psi_pass;
    v.collide_pass = c->L.collide_pass;
    v.fused_pass = c->one_pass;
    v.L = &c->L;
    v.check_error = [](lbm_ctx *cc, std::string &m) {
        lbm_status s = sync_and_check(cc, "adjoint");
        if (s != LBM_OK) m = cc->err;
        return s;
    };
    v.n_fluid = c->n_fluid;
    v.ctx = c;
    return v;
}
}  // namespace lbm

// ------------------------------------------- helpers for lbm_noalloc.cu ----

namespace lbm {
// Kernel parameters for a lattice described by *p whose population planes have the given
// row pitch (elements); no geometry arrays.  Validates *p like lbm_create.
lbm_status kparams_for(const lbm_params *p, int64_t pitch, KParams *out)
{
    lbm_status s = validate(nullptr, *p);
    if (s != LBM_OK) return s;
    lbm_ctx tmp;
    tmp.p = *p;
    if (cudaGetDevice(&tmp.device) != cudaSuccess ||
        cudaDeviceGetAttribute(&tmp.sm_count, cudaDevAttrMultiProcessorCount, tmp.device) != cudaSuccess)
        return fail(nullptr, LBM_ECUDA, "cannot query the current device");
    tmp.pitch = pitch;
    tmp.plane = pitch * p->ny;
    fill_constants(&tmp);
    *out = tmp.kp;
    return LBM_OK;
}

// The driver's entry points are fetched through the runtime, so the library needs no link to the driver library.
unsigned long long current_context()
{
    struct Driver {
        CUresult (*get_current)(CUcontext *) = nullptr;
        CUresult (*get_id)(CUcontext, unsigned long long *) = nullptr;
        Driver()
        {
            void *a = nullptr, *b = nullptr;
            cudaDriverEntryPointQueryResult qa, qb;
            cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa);
            if (e == cudaSuccess) e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb);
            if (e != cudaSuccess || qa != cudaDriverEntryPointSuccess || qb != cudaDriverEntryPointSuccess) return;
            get_current = reinterpret_cast<CUresult (*)(CUcontext *)>(a);
            get_id = reinterpret_cast<CUresult (*)(CUcontext, unsigned long long *)>(b);
        }
    };
    static const Driver d;
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!d.get_current || !d.get_id || d.get_current(&ctx) != CUDA_SUCCESS || !ctx || d.get_id(ctx, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// A kernel's attributes belong to a context: what was set in one is not there after a reset of the device, nor in
// another context.  So what was set, and what the device answered, is kept with the context's ID.
cudaError_t ensure_smem_attribute_ptr(const void *kernel, int device, int bytes)
{
    struct Done {
        const void *kernel;
        int device;
        unsigned long long context;
    };
    static std::mutex mu;
    static std::vector<Done> done;
    const unsigned long long context = current_context();
    std::lock_guard<std::mutex> lock(mu);
    auto d = std::find_if(done.begin(), done.end(), [&](const Done &x) { return x.kernel == kernel && x.device == device; });
    if (d != done.end() && context != 0 && d->context == context) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    if (d == done.end()) done.push_back({kernel, device, context});
    else d->context = context;
    return e;
}

bool cluster_fits(const void *kernel, int device, int ctas, int threads, int smem_bytes)
{
    struct Asked {
        const void *kernel;
        int device, ctas;
        unsigned long long context;
        bool fits;
    };
    static std::mutex mu;
    static std::vector<Asked> done;
    const unsigned long long context = current_context();
    std::lock_guard<std::mutex> lock(mu);
    auto d = std::find_if(done.begin(), done.end(), [&](const Asked &x) { return x.kernel == kernel && x.device == device && x.ctas == ctas; });
    if (d != done.end() && context != 0 && d->context == context) return d->fits;
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem_bytes;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = ctas;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
    }
    if (e != cudaSuccess) cudaGetLastError();  // (not an error of the caller's: the lattice is stepped launch by launch)
    if (d == done.end()) d = done.insert(done.end(), Asked{kernel, device, ctas, context, false});
    d->context = context;
    d->fits = e == cudaSuccess && n > 0;
    return d->fits;
}

// psi of the EOS of *p at rho (the host evaluation create uses), for lbm_lbana.cu.
double eos_psi(const lbm_params &p, double rho) { return host_psi(p, rho); }

// Record a message for lbm_last_error(NULL).
lbm_status set_global_error(lbm_status s, const std::string &msg) { return fail(nullptr, s, msg); }
}  // namespace lbm
