// Internal types shared by the host API and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbm {

// Derived constants in the arithmetic type R of a kernel, computed on the host, so that
// no kernel converts between double and float per node (GB300's FP64 pipe is narrow).
template <class R>
struct Consts {
    R eos_a, eos_b, eos_RT, eos_R, eos_K, two_over_G, G, kq1, kq7, c1G, c2G, q2fac, sp, sq, nu_l, nu_g, rho_l, rho_g, Lambda, Fx, Fy, psi_s, rho_s, rho_ref, scale, inv_scale;
    R hsp, hsq;  // 1 - s_p/2 and 1 - s_q/2 of the constant relaxation rates
};

// Constant operands of the packed FP32x2 evaluation (lbm_f32.cuh), each splatted to a pair
// (c, c) on the host, so that the kernel never assembles a constant pair at run time.
struct PairConsts {
    float2 m_G, kq1, q2fac, kq7, c1G, m_c2G, sp, sq, hsp, six_hsp, m_six_hsp, m_hsq;
    float2 Fx, Fy, rho_g, inv_drho, dnu, nu_g, Lambda;
    float2 m_b, b4, K, RT, a, two_over_G;
    float2 scale, m_scale;
    float2 dec[9];  // w_i rho_ref (decode of deviations)
    float2 enc[9];  // -(w_i rho_ref) 2^k (encode of deviations)
    float2 w[9];    // w_i
};

// Everything a kernel needs, passed by value.  Physical constants are kept in double
// (host bookkeeping and the FP64 path) and, for kernels, in cd / cf by arithmetic type.
struct KParams {
    int nx, ny;
    int device;    // CUDA device of the context
    int sm_count;  // its multiprocessor count (queried once, at create)
    int64_t pitch;  // elements per row of a population plane (and of the rho_ref plane)
    int64_t plane;  // elements per population plane = pitch * ny
    int periodic_x, periodic_y;
    int improved;    // 1: improved Q4, Q6 (Eq. qm46.improved)
    int eos;         // 0 van der Waals, 1 Carnahan-Starling
    int force_mode;  // 0 constant, 1 (rho - rho_g) g, 2 field
    int var_tau;     // 1: tau(rho) from the linear nu(rho) interpolation
    int per_node_ref;
    int sr;            // FP16/BF16 storage: 1 stochastic rounding, 0 to nearest
    int packed;        // FP32 arithmetic: 1 the tile kernel rounds as the staged kernel does (k_tile.cuh)
    uint32_t sr_seed;  // random-bit seed of this step (a hash of the step count)
    // EOS: p = K (rho RT g(rho) - a rho^2); psi = sqrt(two_over_G (p - rho/3))
    double eos_a, eos_b, eos_RT, eos_K, two_over_G;
    double eos_R, eos_T;  // raw R and T (FP64 path evaluates (rho R) T like a plain formula)
    double G;
    double k1, k2;        // raw source coefficients (FP64 path)
    double q1c, q4a, q4b;  // 3 (k1 + 2 k2), (30 eps - 15)/16, 3 eps/8 (FP64 path, evaluated on the host)
    double two_inv_G;      // 2/G
    int G_pow2;            // 1: G is +- a power of two, so that 2 x/G = x two_inv_G exactly
    double eos_b4;         // b/4
    int unit_R, unit_K;    // R = 1, K = 1
    int q2_full;           // 1: Q_2 = -Q_1; 0: -Q_1/2
    // source term with G folded in (|F_int|^2/(G psi^2) = G |S|^2, S = F_int/(-G psi)):
    // Q1 = kq1 |S|^2, Q2 = q2fac Q1, Q7 = kq7 (Sx^2 - Sy^2), Q8 = kq7 Sx Sy,
    // Q4 = (c1G Sx^2 - c2G Sy^2) ux, Q6 = (c1G Sy^2 - c2G Sx^2) uy
    double kq1, kq7, c1G, c2G, q2fac;
    // relaxation: constant rates, or nu(rho) interpolation data
    double sp, sq;
    double nu_l, nu_g, rho_l, rho_g, Lambda;
    double Fx, Fy;
    double psi_s;  // psi(rho_s) of walls
    double rho_s;
    // FP16/BF16 storage codec
    double rho_ref, scale, inv_scale;
    // buffers
    const void *src;       // populations read (post-collision state of the last step)
    void *dst;             // populations written
    const float *ref_src;  // per-node reference density planes (FP16/BF16 with per_node_ref)
    float *ref_dst;
    void *psi;             // psi field [ny*nx] in the kernel's arithmetic type
    void *psi_out;         // one-pass kernels: also write psi of the state read here ([ny*nx] in
                           // the arithmetic type, as the psi pass does), or null
    const uint8_t *solid;  // [ny*nx] or null
    const double *wall_u;  // [2][ny*nx] or null
    const double *q;       // [8][ny*nx] or null
    const double *fext;    // [2][ny*nx] or null
    const double *wall_rho;  // [ny*nx] virtual density of each solid node, or null (rho_s)
    const double *wall_psi;  // [ny*nx] psi of wall_rho, or null (psi_s)
    const float *fext_f, *wall_psi_f;  // the same two in FP32 (kernels of FP32 arithmetic convert no FP64 value)
    // [8][ny][pitch] per fluid node and pulled population i = 1..8 whose source x - e_i is a
    // wall: (q, c) with q the link fraction after the fallback of a missing second node, and c the wall's
    // part of the moving-wall term: e_i . u_w as the two-pass step forms it (mw = 2 w_o rho_w c 3) or, in the
    // packed step, 6 w_o (e_i . u_w) (mw = c rho_w).  Null without interpolated or moving walls, and in FP64.
    // Read by the tile kernel's wall links.
    const float2 *link;
    // [ny*nx] per node: bit i (1..8) set when the source x - e_i is a wall, bit 0 when the node is
    // solid; null without solid nodes, link fractions and wall velocities.  Read by the tile kernel.
    const uint16_t *links;
    int skip_solid;        // 1: more than an eighth of the nodes are solid
    int64_t pull[9];       // bytes from a node to population i of the row it is pulled from, (i plane - e_iy pitch)
    int *err;              // device error word (0 = fine)
    Consts<double> cd;     // constants for FP64 arithmetic
    Consts<float> cf;      // constants for FP32 arithmetic
    PairConsts c2;         // the same as pairs, for the packed kernels
    unsigned short inv_scale_bits;  // 2^-k in the storage type (FP16 or BF16 bits)
};

// Per-block partial sums of the transposed steps: slots of one row (8 doubles).  dJ/dFx, dJ/dFy,
// dJ/dG (explicit and wall psi), dJ/dT (wall psi), <W, A_t>, and dJ/dG and dJ/dT through psi(rho).
constexpr int kAdjSlots = 8;
enum AdjSlot { SLOT_FX = 0, SLOT_FY = 1, SLOT_G1 = 2, SLOT_T1 = 3, SLOT_J = 4, SLOT_G2 = 5, SLOT_T2 = 6 };

// Buffers and scalars of one transposed step.  Planes use the population row pitch.  The _in planes
// are what the step after left (g, dJ/dS, the local part of dJ/dpsi, rho of its pulled populations
// and, in FP64, its psi); c, which completes lambda, is formed from them.
struct AdjArgs {
    const void *g_in;   // [9] planes (null: lambda_{t+1} = W_{t+1} only)
    const void *dS_in;  // [2] planes
    const void *dpsi_in, *rho_in, *psi_in;
    void *g_out, *dS_out, *dpsi_out, *rho_out, *psi_out;
    void *c_out;        // plane: c of the _in planes, written by the tail launch
    int tail;           // 1: form c and its parameter sums, no further step
    int ahead;          // rows between a tile and the one whose lines it prefetches into L2; 0: none
    int64_t push[9];    // bytes from a node to plane i of the row ahead, (i plane + e_iy pitch)
    double w_scale;     // weight of W in lambda_{t+1} (1/n for J = (1/n) sum_t <W, A_t>)
    int objective;      // 0: y momentum handed to the walls by the next streaming; 1: mean j_x
    double inv_nfluid;  // 1 / number of fluid nodes (objective 1)
    double *part;       // per-block FP64 partial sums [blocks][kAdjSlots]
    int sum_J;          // also sum <W, A_t> of the state
    float w_scale_f, inv_nfluid_f;  // the two scales rounded to FP32 on the host (FP32 arithmetic
                                    // converts no FP64 value per node)
};

// Seed of the stochastic-rounding bits of step t (MurmurHash3's 32-bit finaliser of the
// step count's two halves; any well-mixed function of t would do).
#ifdef __CUDACC__
__host__ __device__
#endif
inline uint32_t sr_seed_of(int64_t t)
{
    uint32_t h = (uint32_t)t * 0x9E3779B1u ^ (uint32_t)((uint64_t)t >> 32) * 0x85EBCA77u;
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

// Storage precisions (match lbm_precision)
enum Prec { P_F64 = 0, P_F32 = 1, P_F16 = 2, P_BF16 = 3 };

// Device error word bits
enum DevErr { DERR_TIMEOUT = 1, DERR_BOUNDS = 2 };

// ID of the calling thread's current context (0: none is current, or it cannot be had).  A device that is
// reset and another context made current get new ones; lbm_api.cu.
unsigned long long current_context();

// One-time set-up of a kernel's dynamic shared-memory limit, per kernel, device and context (an
// attribute set in one context does not apply to another); lbm_api.cu.
cudaError_t ensure_smem_attribute_ptr(const void *kernel, int device, int bytes);
template <class K>
inline cudaError_t ensure_smem_attribute(K kernel, int device, int bytes)
{
    return ensure_smem_attribute_ptr(reinterpret_cast<const void *>(kernel), device, bytes);
}

// Whether the device can hold a cluster of `ctas` blocks of the kernel with these limits (shared memory
// and cluster size are then allowed for it), asked once per kernel, device, context and size; lbm_api.cu.
bool cluster_fits(const void *kernel, int device, int ctas, int threads, int smem_bytes);

// Launchers, defined in the per-precision translation units (k_f64.cu, k_f32.cu,
// k_f16.cu).  All run on `st` and return the launch status.
struct Launchers {
    cudaError_t (*psi_pass)(const KParams &, cudaStream_t);
    cudaError_t (*collide_pass)(const KParams &, cudaStream_t);
    cudaError_t (*fused_pass)(const KParams &, cudaStream_t);  // staged one-pass step (periodic, FP32 arithmetic); null in FP64
    cudaError_t (*tile_pass)(const KParams &, cudaStream_t);   // one-pass step on tiles (k_tile.cuh)
    // many steps of a small lattice in one launch (k_small.cuh); small_ctas: 0 where it does not fit
    int (*small_ctas)(const KParams &);
    cudaError_t (*small_steps)(const KParams &, int ctas, int64_t nsteps, int64_t step0, cudaStream_t);
    cudaError_t (*link_bits)(const KParams &, uint16_t *out, cudaStream_t);  // KParams::links
    cudaError_t (*init)(const KParams &, const double *rho, const double *ux, const double *uy,
                        cudaStream_t);
    cudaError_t (*moments)(const KParams &, double *rho, double *ux, double *uy, cudaStream_t);
    int64_t (*diag_rows)(const KParams &);  // rows (of 11 doubles) of `part`
    // out[11]: the nine sums of lbm_get_diagnostics, max |u|, number of nodes that are not finite
    cudaError_t (*diag)(const KParams &, double *part, double *out, cudaStream_t);
    cudaError_t (*get_state)(const KParams &, double *out, cudaStream_t);
    cudaError_t (*set_state)(const KParams &, const double *in, cudaStream_t);
    // transposed step (FP64 arithmetic for FP64 storage, FP32 otherwise); AdjArgs in k_adjoint.cuh
    cudaError_t (*adj_step)(const KParams &, const AdjArgs &, cudaStream_t);
    cudaError_t (*adj_lambda)(const KParams &, const void *g, const void *c, double *out, cudaStream_t);
    cudaError_t (*objective)(const KParams &, int objective, double inv_nfluid, double *acc, cudaStream_t);
    int64_t (*adj_blocks)(const KParams &);  // rows of the per-block partial-sum array (8 doubles each)
    cudaError_t (*adj_reduce)(const KParams &, const double *part, double *out8, cudaStream_t);
    // lattices on which LBM_KERNEL_FUSED is granted (and lbm_kernel_in_use says so)
    int fused_tile_x;     // nx at least this and 16
    int fused_align;      // nx must be a multiple of this
    int fused_geometry;   // 1: also with solid nodes, moving and interpolated walls
};

Launchers launchers_f64();
Launchers launchers_f32();
Launchers launchers_f16();
Launchers launchers_bf16();

}  // namespace lbm
