// Two-pass step (psi pass + fused collide-and-pull-stream pass) and the per-node
// service kernels (init, state copy), for one storage type S.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

constexpr int kRowThreads = 128;

// Reads population k of node (x, y) of kp.src from global memory.
template <class S>
struct GlobalAt {
    static constexpr bool DEV = IsDev<S>::value;
    const KParams &kp;
    __device__ __forceinline__ typename Codec<S>::R operator()(int k, int x, int y) const { return load_pop<S>(kp, k, x, y); }
    __device__ __forceinline__ typename Codec<S>::R at_k(int k, int64_t kk) const { return load_pop_at<S>(kp, k, kk); }
};

// psi of the neighbour along e_i from the field written by the psi pass: inside the lattice (solid
// nodes hold psi of their virtual density there) the field, psi(rho_s) beyond a non-periodic edge.
template <class R>
struct AroundPsi {
    const KParams &kp;
    const R *psi;
    const Around &nb;
    __device__ __forceinline__ R operator()(int i) const { return nb.in(i) ? psi[nb.n(i)] : cst<R>(kp).psi_s; }
};

__device__ __forceinline__ bool node_is_solid(const KParams &kp, int64_t node)
{
    return kp.solid != nullptr && kp.solid[node] != 0;
}

// Pass 1: rho(x) = sum_i f_i(x) of the pulled populations, psi(rho) (Sec. 2).
template <class S>
__global__ void __launch_bounds__(kRowThreads) k_psi(KParams kp)
{
    typedef typename Codec<S>::R R;
    grid_dependency_wait();
    allow_dependent_launch();
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const int64_t node = (int64_t)y * kp.nx + x;
    R *psi = static_cast<R *>(kp.psi);
    if (node_is_solid(kp, node)) {
        psi[node] = kp.wall_psi ? R(kp.wall_psi[node]) : cst<R>(kp).psi_s;
        return;
    }
    R f[9];
    pull_node_nb<R>(kp, around(kp, x, y), x, y, GlobalAt<S>{kp}, f, (R *)nullptr);
    psi[node] = psi_of<R>(kp, density<R>(f));
}

// Pass 2: pull, force from the psi stencil, collision, store.
template <class S>
__global__ void __launch_bounds__(kRowThreads) k_collide(KParams kp)
{
    typedef typename Codec<S>::R R;
    grid_dependency_wait();
    allow_dependent_launch();
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const int64_t node = (int64_t)y * kp.nx + x;
    if (node_is_solid(kp, node)) return;
    const R *psi = static_cast<const R *>(kp.psi);
    R f[9], fb[9], Sx, Sy, Fex, Fey, ux, uy;
    const Around nb = around(kp, x, y);
    pull_node_nb<R>(kp, nb, x, y, GlobalAt<S>{kp}, f, (R *)nullptr);
    const R rho = density<R>(f);
    stencil_S<R>(AroundPsi<R>{kp, psi, nb}, Sx, Sy);
    external_force<R>(kp, node, rho, Fex, Fey);
    collide<R>(kp, f, rho, psi[node], Sx, Sy, Fex, Fey, fb, ux, uy);
    store_node<S>(kp, x, y, fb, rho);
}

// f_bar = M^-1 m_eq(rho, u) at every node (solid nodes too; they are never read).
template <class S>
__global__ void __launch_bounds__(kRowThreads) k_init(KParams kp, const double *rho0, const double *ux0, const double *uy0)
{
    typedef typename Codec<S>::R R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const int64_t node = (int64_t)y * kp.nx + x;
    const R rho = R(rho0[node]);
    const R ux = ux0 ? R(ux0[node]) : R(0), uy = uy0 ? R(uy0[node]) : R(0);
    R fb[9];
    equilibrium<R>(rho, ux, uy, fb);
    store_node<S>(kp, x, y, fb, rho);
}

template <class S>
__global__ void __launch_bounds__(kRowThreads) k_get_state(KParams kp, double *out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const int64_t n = (int64_t)kp.nx * kp.ny, node = (int64_t)y * kp.nx + x;
#pragma unroll
    for (int i = 0; i < 9; ++i) out[i * n + node] = double(load_pop<S>(kp, i, x, y));
}

template <class S>
__global__ void __launch_bounds__(kRowThreads) k_set_state(KParams kp, const double *in)
{
    typedef typename Codec<S>::R R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const int64_t n = (int64_t)kp.nx * kp.ny, node = (int64_t)y * kp.nx + x;
    R fb[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) fb[i] = R(in[i * n + node]);
    // the reference density of a node is the sum of its stored populations
    store_node<S>(kp, x, y, fb, density<R>(fb));
}

inline dim3 row_grid(const KParams &kp) { return dim3((kp.nx + kRowThreads - 1) / kRowThreads, kp.ny); }

template <class S>
struct TwoPass {
    static cudaError_t psi_pass(const KParams &kp, cudaStream_t st)
    {
        return launch_dependent(k_psi<S>, row_grid(kp), dim3(kRowThreads), 0, st, kp);
    }
    static cudaError_t collide_pass(const KParams &kp, cudaStream_t st)
    {
        return launch_dependent(k_collide<S>, row_grid(kp), dim3(kRowThreads), 0, st, kp);
    }
    static cudaError_t init(const KParams &kp, const double *r, const double *u, const double *v, cudaStream_t st)
    {
        k_init<S><<<row_grid(kp), kRowThreads, 0, st>>>(kp, r, u, v);
        return cudaGetLastError();
    }
    static cudaError_t get_state(const KParams &kp, double *out, cudaStream_t st)
    {
        k_get_state<S><<<row_grid(kp), kRowThreads, 0, st>>>(kp, out);
        return cudaGetLastError();
    }
    static cudaError_t set_state(const KParams &kp, const double *in, cudaStream_t st)
    {
        k_set_state<S><<<row_grid(kp), kRowThreads, 0, st>>>(kp, in);
        return cudaGetLastError();
    }
};

}  // namespace lbm
