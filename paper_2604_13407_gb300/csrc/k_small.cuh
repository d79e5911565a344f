// Many steps of a small lattice in one launch: the lattice lives in the shared memory of one thread-block
// cluster, a strip of rows per CTA.
//
// What bounds a small lattice is neither bytes nor instructions but the launch and the two trips through
// L2 that a step of its own kernel takes (2.9 us a step on 37 x 23 nodes, whatever is computed).  Here a step
// is two phases between cluster barriers: pull, rho and psi; then the psi stencil, collision and the
// write-back in place.  A thread owns one node for the whole launch (or, where a strip has more than 512,
// two; in FP64 four threads share one).  What a
// neighbouring strip needs -- psi of the edge rows, and the populations that leave them -- is pushed into
// its halo rows through distributed shared memory, so every load is a local one.
//
// Measured per step (us, one launch per step / here): 37 x 23 FP32 3.0 / 0.90, FP16 3.0 / 1.2; 64^2 FP32 3.0 / 1.06;
// 128^2 3.0 / 2.1 (16 SMs are busy there: the last size that gains); FP64 4 x 128 column 18 / 5.4, 4 x 181
// 18 / 7.9, 37 x 23 18 / 11.2.
//
// The functions, their order and the storage type's rounding are the tile kernel's (k_tile.cuh), so
// the state after n steps is, bit for bit, what n of its launches leave.
#pragma once

#include "k_tile.cuh"

namespace lbm {

constexpr int kSmallThreads = 512;  // most threads of a CTA

__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Shared-memory address of this CTA as the same variable's address in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to(const void *p, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void push(uint32_t a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void push(uint32_t a, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ void push(uint32_t a, __half v) { asm volatile("st.shared::cluster.b16 [%0], %1;" ::"r"(a), "h"(__half_as_ushort(v)) : "memory"); }
__device__ __forceinline__ void push(uint32_t a, __nv_bfloat16 v) { asm volatile("st.shared::cluster.b16 [%0], %1;" ::"r"(a), "h"(__bfloat16_as_ushort(v)) : "memory"); }

// Shared memory of a CTA: nine planes, the reference plane and psi, of `rows` own rows and a halo row
// above and below; a psi row ends with one entry that always holds psi(rho_s), the neighbour beyond a
// non-periodic x edge.
template <class S>
struct SmallLayout {
    typedef typename Codec<S>::R R;
    int nx, rows;
    __host__ __device__ size_t plane() const { return (size_t)(rows + 2) * nx; }
    __host__ __device__ size_t psi_at() const { return (9 * plane() * sizeof(S) + 15) / 16 * 16; }
    __host__ __device__ size_t ref_at() const { return psi_at() + ((size_t)(rows + 2) * (nx + 1) * sizeof(R) + 15) / 16 * 16; }
    __host__ __device__ size_t bytes(bool ref) const { return ref_at() + (ref ? plane() * sizeof(float) : 0); }
};

// A CTA's strip of the lattice in its shared memory.
template <class S>
struct Strip {
    typedef typename Codec<S>::R R;
    const KParams &kp;
    S *pop;
    R *psi;
    float *ref;
    int nx, C, rank, y0, m;  // own rows y0 .. y0 + m - 1: local rows 1 .. m
    uint32_t PS;             // elements per plane
    uint32_t up_pop, up_psi, up_ref, down_pop, down_psi, down_ref;  // halo rows of the strips above and below
    bool has_ref;

    __device__ __forceinline__ int first_row(int r) const { return (int)((int64_t)r * kp.ny / C); }
    // Reads the strip and its halo rows; every thread of the cluster is past its end when it returns.
    __device__ __forceinline__ void load(unsigned char *smem, int max_rows)
    {
        nx = kp.nx, C = (int)gridDim.x, rank = (int)cluster_rank();
        const SmallLayout<S> L{nx, max_rows};
        PS = (uint32_t)L.plane();
        pop = reinterpret_cast<S *>(smem);
        psi = reinterpret_cast<R *>(smem + L.psi_at());
        ref = reinterpret_cast<float *>(smem + L.ref_at());
        has_ref = IsDev<S>::value && kp.per_node_ref;
        y0 = first_row(rank), m = first_row(rank + 1) - y0;
        for (int lr = 0; lr < m + 2; ++lr) {
            int gy = y0 + lr - 1;
            const bool in = (gy >= 0 && gy < kp.ny) || kp.periodic_y;
            gy = gy < 0 ? gy + kp.ny : gy >= kp.ny ? gy - kp.ny : gy;
            for (int x = threadIdx.x; x < nx; x += blockDim.x) {
                if (in) {
                    const int64_t k = (int64_t)gy * kp.pitch + x;
#pragma unroll
                    for (int i = 0; i < 9; ++i) pop[i * PS + lr * nx + x] = static_cast<const S *>(kp.src)[i * kp.plane + k];
                    if (has_ref) ref[lr * nx + x] = kp.ref_src[k];
                } else {
                    psi[lr * (nx + 1) + x] = cst<R>(kp).psi_s;
                }
            }
            if (threadIdx.x == 0) psi[lr * (nx + 1) + nx] = cst<R>(kp).psi_s;
        }
        const int up = rank == C - 1 ? 0 : rank + 1, down = rank == 0 ? C - 1 : rank - 1;
        const uint32_t above_down = (uint32_t)(first_row(down + 1) - first_row(down) + 1);  // its halo row above its own
        up_pop = map_to(pop, up), up_psi = map_to(psi, up), up_ref = map_to(ref, up);
        down_pop = map_to(pop, down) + above_down * nx * (uint32_t)sizeof(S);
        down_psi = map_to(psi, down) + above_down * (nx + 1) * (uint32_t)sizeof(R);
        down_ref = map_to(ref, down) + above_down * nx * 4u;
        cluster_barrier();
    }
    __device__ __forceinline__ void barrier() const
    {
        if (C == 1) __syncthreads();
        else cluster_barrier();
    }
};

// A node of a strip: its places in shared memory and in the lattice.
template <class S>
struct StripNode {
    typedef typename Codec<S>::R R;
    bool live, fluid, top, bottom;        // a node; a fluid one; in a row that the strip above / below reads
    uint32_t row, cm, c0, cp, pm, pp;     // local row; columns x - 1, x, x + 1 of the populations, and of psi
    uint32_t node, kg;                    // lattice and plane index
    unsigned w;                           // wall bits
    StripNode() = default;
    __device__ __forceinline__ StripNode(const Strip<S> &s, int idx)
    {
        const KParams &kp = s.kp;
        live = idx < s.m * s.nx;
        const int ly = live ? idx / s.nx : 0, x = live ? idx - ly * s.nx : 0, y = s.y0 + ly;
        row = ly + 1;
        const Around nb = around(kp, x, y);
        cm = nb.xc[0], c0 = x, cp = nb.xc[2];
        pm = x > 0 || kp.periodic_x ? cm : s.nx;
        pp = x < s.nx - 1 || kp.periodic_x ? cp : s.nx;
        node = (uint32_t)y * s.nx + x;
        kg = (uint32_t)y * (uint32_t)kp.pitch + x;
        w = kp.links != nullptr ? kp.links[node] : edge_walls(nb.inside);
        fluid = live && !(w & 1u);
        top = live && ly == s.m - 1 && (y < kp.ny - 1 || kp.periodic_y);
        bottom = live && ly == 0 && (y > 0 || kp.periodic_y);
    }
    __device__ __forceinline__ uint32_t from(const Strip<S> &s, int i) const  // x - e_i
    {
        return (row - ey_(i)) * s.nx + (ex_(i) > 0 ? cm : ex_(i) < 0 ? cp : c0);
    }
    __device__ __forceinline__ uint32_t own(const Strip<S> &s) const { return row * s.nx + c0; }
    __device__ __forceinline__ uint32_t psi_at(const Strip<S> &s, int i) const  // x + e_i
    {
        return (row + ey_(i)) * (s.nx + 1) + (ex_(i) > 0 ? pp : ex_(i) < 0 ? pm : c0);
    }
    __device__ __forceinline__ R read(const Strip<S> &s, int i, uint32_t o) const
    {
        if constexpr (IsDev<S>::value)
            return Raw<S>::f(s.pop[i * s.PS + o], __fmul_rn(w_<float>(i), s.has_ref ? s.ref[o] : s.kp.cf.rho_ref), s.kp);
        else return s.pop[i * s.PS + o];
    }
    // Pull, Eq. (lbe.str); on wall links the population that left the node toward the wall comes back.
    __device__ __forceinline__ void pull(const Strip<S> &s, R (&f)[9]) const
    {
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = read(s, i, from(s, i));
        if ((w & 0x1feu) && fluid) {
#pragma unroll
            for (int i = 1; i < 9; ++i)
                if ((w >> i) & 1u) f[i] = read(s, opp_(i), own(s)) + R(0);
        }
    }
    __device__ __forceinline__ void put_psi(const Strip<S> &s, R v) const
    {
        if (!live) return;
        s.psi[row * (s.nx + 1) + c0] = v;
        if (top) push(s.up_psi + c0 * (uint32_t)sizeof(R), v);
        if (bottom) push(s.down_psi + c0 * (uint32_t)sizeof(R), v);
    }
    // Stores the populations of the node whose bits are set.
    __device__ __forceinline__ void put(const Strip<S> &s, const S (&v)[9], unsigned which = 0x1ffu) const
    {
        if (!fluid) return;
        S *p = s.pop + own(s);
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if ((which >> i) & 1u) p[i * s.PS] = v[i];
        if (top) {
#pragma unroll
            for (int i = 0; i < 9; ++i)
                if (ey_(i) > 0 && ((which >> i) & 1u)) push(s.up_pop + (i * s.PS + c0) * (uint32_t)sizeof(S), v[i]);
        }
        if (bottom) {
#pragma unroll
            for (int i = 0; i < 9; ++i)
                if (ey_(i) < 0 && ((which >> i) & 1u)) push(s.down_pop + (i * s.PS + c0) * (uint32_t)sizeof(S), v[i]);
        }
    }
    // The state after an odd number of steps goes to the other buffer, as step by step.
    __device__ __forceinline__ void write_back(const Strip<S> &s, bool odd) const
    {
        if (!fluid) return;
        S *dst = static_cast<S *>(odd ? s.kp.dst : const_cast<void *>(s.kp.src));
#pragma unroll
        for (int i = 0; i < 9; ++i)
            dst[i * s.kp.plane + kg] = s.pop[i * s.PS + own(s)];
        if (s.has_ref) (odd ? s.kp.ref_dst : const_cast<float *>(s.kp.ref_src))[kg] = s.ref[own(s)];
    }
};

// FP32 arithmetic: a thread owns one node of its strip (v1) or two (v2x), `units` apart, for the whole launch.
template <class T> struct Owned;
template <> struct Owned<v1> {
    static constexpr int N = 1;
    static __device__ __forceinline__ v1 of(const float *v, int) { return v1{v[0]}; }
    static __device__ __forceinline__ float get(v1 a, int) { return a.v; }
    static __device__ __forceinline__ void set(v1 &a, int, float v) { a.v = v; }
};
template <> struct Owned<v2x> {
    static constexpr int N = 2;
    static __device__ __forceinline__ v2x of(const float *v, int pitch) { return X2(v[0], v[pitch]); }
    static __device__ __forceinline__ float get(v2x a, int e) { return e ? a.v.y : a.v.x; }
    static __device__ __forceinline__ void set(v2x &a, int e, float v) { (e ? a.v.y : a.v.x) = v; }
};
template <class S, class T, int THREADS>
__global__ void __launch_bounds__(THREADS) k_small2(KParams kp, int64_t nsteps, int64_t step0, int max_rows)
{
    typedef Owned<T> Z;
    constexpr bool DEV = IsDev<S>::value;
    constexpr int N = Z::N;
    extern __shared__ __align__(128) unsigned char smem[];
    Strip<S> s{kp};
    s.load(smem, max_rows);
    const int nodes = s.m * s.nx, units = (nodes + N - 1) / N, t0 = (int)threadIdx.x;
    StripNode<S> n[N];
    float wall[N];       // psi of solid nodes
    unsigned pick = 0x5400u;  // which half of its row pair's random word each node takes: its column's parity
#pragma unroll
    for (int e = 0; e < N; ++e) {
        // (threads past the last unit, and the second node of an odd strip's last thread: not live)
        n[e] = StripNode<S>(s, t0 < units ? t0 + e * units : nodes);
        wall[e] = (n[e].w & 1u) && kp.wall_psi_f ? kp.wall_psi_f[n[e].node] : kp.cf.psi_s;
        pick = e == 0 ? (pick & 0xff00u) | (n[e].c0 & 1u ? 0x32u : 0x10u) : (pick & 0xffu) | (n[e].c0 & 1u ? 0x7600u : 0x5400u);
    }

    for (int64_t t = 0; t < nsteps; ++t) {
        float f_[N][9];
#pragma unroll
        for (int e = 0; e < N; ++e) n[e].pull(s, f_[e]);
        T d[9], rho, psi;
        {
            T f[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = Z::of(&f_[0][i], 9);
            to_dev(f, d);
        }
        rho = density_dev(d);
        psi = psi_v<T>(kp, rho);
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (n[e].w & 1u) Z::set(psi, e, wall[e]), Z::set(rho, e, 1.f);
            n[e].put_psi(s, Z::get(psi, e));
        }
        s.barrier();

        auto p = [&](int i) {
            float v[N];
#pragma unroll
            for (int e = 0; e < N; ++e) v[e] = s.psi[n[e].psi_at(s, i)];
            return Z::of(v, 1);
        };
        T Sx, Sy, Fex = ks<T>(0.f), Fey = Fex, o[9], ux, uy;
        stencil_v<T>(p(1), p(2), p(3), p(4), p(5), p(6), p(7), p(8), Sx, Sy);
        if (kp.force_mode == 0) {
            Fex = kc<T>(kp.c2.Fx), Fey = kc<T>(kp.c2.Fy);
        } else if (kp.force_mode == 1) {
            const T x = rho - kc<T>(kp.c2.rho_g);
            Fex = x * kc<T>(kp.c2.Fx), Fey = x * kc<T>(kp.c2.Fy);
        } else if (kp.fext_f) {
            const int64_t all = (int64_t)kp.nx * kp.ny;
#pragma unroll
            for (int e = 0; e < N; ++e) Z::set(Fex, e, kp.fext_f[n[e].node]), Z::set(Fey, e, kp.fext_f[all + n[e].node]);
        }
        collide_v<T, RuntimeOpts>(kp, d, rho, psi, Sx, Sy, Fex, Fey, o, ux, uy);
        S v[N][9];
        if constexpr (DEV) {
            const uint32_t seed = sr_seed_of(step0 + t);
            const uint32_t ha = sr_hash(n[0].kg >> 1, seed), hb = N == 2 ? sr_hash(n[N - 1].kg >> 1, seed) : 0u;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const T wr = s.has_ref ? kc<T>(kp.c2.w[i]) * rho : kc<T>(kp.c2.dec[i]);
                const T q = (o[i] - wr) * kc<T>(kp.c2.scale);
                const float qa = Z::get(q, 0), qb = N == 2 ? Z::get(q, N - 1) : 0.f;
                if (kp.sr) {
                    const uint32_t h = SRound<S>::pack(qa, qb, __byte_perm(sr_bits(ha, i), N == 2 ? sr_bits(hb, i) : 0u, pick));
                    v[0][i] = SRound<S>::from_bits((unsigned short)(h & 0xffffu));
                    if (N == 2) v[N - 1][i] = SRound<S>::from_bits((unsigned short)(h >> 16));
                } else {
                    v[0][i] = Codec<S>::enc(qa, 0.f, 1.f);
                    if (N == 2) v[N - 1][i] = Codec<S>::enc(qb, 0.f, 1.f);
                }
            }
            if (s.has_ref) {
#pragma unroll
                for (int e = 0; e < N; ++e) {
                    if (!n[e].fluid) continue;
                    s.ref[n[e].own(s)] = Z::get(rho, e);
                    if (n[e].top) push(s.up_ref + n[e].c0 * 4u, Z::get(rho, e));
                    if (n[e].bottom) push(s.down_ref + n[e].c0 * 4u, Z::get(rho, e));
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < N; ++e)
#pragma unroll
                for (int i = 0; i < 9; ++i) v[e][i] = Z::get(o[i], e);
        }
#pragma unroll
        for (int e = 0; e < N; ++e) n[e].put(s, v[e]);
        s.barrier();
    }
#pragma unroll
    for (int e = 0; e < N; ++e) n[e].write_back(s, nsteps & 1);
}

// FP64.  An FP64 instruction holds its scheduler's quarter of the SM for 64 cycles, whatever the
// number of active lanes and however independent its neighbours are, so a node's 328 of them in one
// warp take 11 us, and a small lattice leaves most schedulers idle.  Four warps therefore share a
// group of 32 nodes, one per scheduler, and hand each other the few values they need through
// shared memory, in six parts between barriers (a barrier costs no more than one FP64 instruction):
// density and the terms of p_EOS; psi, moments, 1/rho; the x and y force and velocity, 1/(G psi^2); the
// quotients by G psi^2; the relaxed moments; the populations, each warp those it stores.  (4 x 128 column:
// 18 us a step with one launch per step, 13.2 with one warp per 32 nodes, 7.5 in four parts, 6.5 in six, 5.4
// with 328 FP64 instructions a node instead of 395.)
struct Small64Shared {
    static constexpr int M = kSmallThreads / 4;
    double num[M], attraction[M], third[M];                      // of psi: p_EOS = K (num/den - attraction), rho/3
    double r[M];                                                 // 1/(G psi^2)
    double Fix[M], Fiy[M], Fx[M], Fy[M], ux[M], uy[M];
    double X[M], Y[M], Q7[M];
    double u[9][M];                                              // m_bar_k without |M_k|^2's odd factor
};
template <class S>
__global__ void __launch_bounds__(kSmallThreads) k_small1(KParams kp, int64_t nsteps, int64_t step0, int max_rows)
{
    using namespace f64;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ Small64Shared x;
    Strip<S> s{kp};
    s.load(smem, max_rows);
    const int role = (threadIdx.x >> 5) & 3, at = (threadIdx.x >> 7) * 32 + (threadIdx.x & 31);
    const StripNode<S> a(s, at);

    for (int64_t t = 0; t < nsteps; ++t) {
        double f[9], sp = kp.sp, sq = kp.sq, m_a = 0.0, m_b = 0.0;
        a.pull(s, f);
        const double rho = density(f);  // (each warp its own: shorter than handing it over)
        Divisor by{};
        if (role == 0) {
            by = divisor(eos_den(kp, rho));
        } else if (role == 2) {
            x.attraction[at] = eos_attraction(kp, rho), x.third[at] = div_const<3>(rho);
            m_a = f[1] - f[3] + f[5] - f[6] - f[7] + f[8];                                  // j_x
        } else if (role == 3) {
            x.num[at] = eos_num(kp, rho);
        }
        __syncthreads();

        if (role == 0) {
            a.put_psi(s, a.w & 1u ? (kp.wall_psi ? kp.wall_psi[a.node] : kp.psi_s) : psi_of(kp, by(x.num[at]), x.attraction[at], x.third[at]));
        } else if (role == 1) {
            moments_12(f, m_a, m_b);
        } else if (role == 2) {
            by = divisor(rho);
            m_b = fma_(2.0, f[3], -2.0 * f[1]) + f[5] - f[6] - f[7] + f[8];               // m_4
        } else {
            by = divisor(rho);
            m_a = f[2] - f[4] + f[5] + f[6] - f[7] - f[8];                                  // j_y
            m_b = fma_(2.0, f[4], -2.0 * f[2]) + f[5] + f[6] - f[7] - f[8];               // m_6
        }
        if (kp.var_tau && role != 0) relaxation(kp, rho, sp, sq);
        s.barrier();

        const double psi = s.psi[a.row * (s.nx + 1) + a.c0], Gpsi = kp.G * psi;
        if (role >= 2) {
            double S_ = 0.0, Fex, Fey;
            auto ps = [&](int i) { return s.psi[a.psi_at(s, i)]; };
            if (role == 2) S_ = stencil_x(ps);
            else S_ = stencil_y(ps);
            external_force<double>(kp, a.node, rho, Fex, Fey);
            const double Fi = -Gpsi * S_, F = Fi + (role == 2 ? Fex : Fey), u = by(fma_(0.5, F, m_a));
            if (role == 2) x.Fix[at] = Fi, x.Fx[at] = F, x.ux[at] = u;
            else x.Fiy[at] = Fi, x.Fy[at] = F, x.uy[at] = u;
        } else if (role == 1) {
            x.r[at] = __drcp_rn(Gpsi * psi);
        } else {
            m_a = f[1] - f[2] + f[3] - f[4], m_b = f[5] - f[6] + f[7] - f[8];               // m_7, m_8
            x.u[0][at] = div_const<9>(rho);
            if (kp.var_tau) relaxation(kp, rho, sp, sq);
        }
        __syncthreads();

        const double Fix = x.Fix[at], Fiy = x.Fiy[at], Fx = x.Fx[at], Fy = x.Fy[at], ux = x.ux[at], uy = x.uy[at];
        const double Gpsi2 = Gpsi * psi;
        const Divisor by_Gpsi2{Gpsi2, x.r[at], in_range(Gpsi2) && is_nonzero(Gpsi2)};
        Stress12 st{};
        double ru = 0.0;
        if (role == 0) {
            ru = rho * ux;
            x.u[8][at] = relaxed_8(ru, m_b, Fx, Fy, ux, uy, by_Gpsi2(kp.k1 * Fix * Fiy), sp);
        } else if (role == 1) {
            st = stress_12(rho, m_a, m_b, Fx, Fy, ux, uy);
        } else if (role == 2) {
            const double xx = Fix * Fix;
            x.X[at] = by_Gpsi2(xx);
            x.Q7[at] = by_Gpsi2(kp.k1 * (xx - Fiy * Fiy));
        } else {
            x.Y[at] = by_Gpsi2(Fiy * Fiy);
            ru = rho * uy;
            x.u[5][at] = div_const<3>(relaxed_j(m_a, Fy, ru));
        }
        __syncthreads();

        if (role == 0) {
            x.u[7][at] = relaxed_7(ru, rho * uy, m_a, Fx, Fy, ux, uy, x.Q7[at], sp);
        } else if (role == 1) {
            double a1, a2;
            relaxed_12(kp, st, m_a, m_b, x.X[at], x.Y[at], sp, a1, a2);
            x.u[1][at] = div_const<9>(a1), x.u[2][at] = div_const<9>(a2);
        } else if (role == 2) {
            ru = rho * ux;
            x.u[3][at] = div_const<3>(relaxed_j(m_a, Fx, ru));
            x.u[4][at] = div_const<3>(relaxed_q(kp, m_b, Fx, ru, ux, x.X[at], x.Y[at], sq));
        } else {
            x.u[6][at] = div_const<3>(relaxed_q(kp, m_b, Fy, ru, uy, x.Y[at], x.X[at], sq));
        }
        __syncthreads();

        double u[9], o[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) u[i] = x.u[i][at];
        if (role == 0) populations_013(u, o), a.put(s, o, 0x00bu);
        else if (role == 1) populations_24(u, o), a.put(s, o, 0x014u);
        else if (role == 2) populations_58(u, o), a.put(s, o, 0x120u);
        else populations_67(u, o), a.put(s, o, 0x0c0u);
        s.barrier();
    }
    if (role == 0) a.write_back(s, nsteps & 1);
}

template <class S>
struct Small {
    typedef typename Codec<S>::R R;
    static constexpr bool F64 = sizeof(R) == 8;
    static int rows(const KParams &kp, int ctas) { return (kp.ny + ctas - 1) / ctas; }
    typedef void (*Kernel)(KParams, int64_t, int64_t, int);
    // The launch for a strip: its kernel, the most threads that is compiled for, and the threads.  FP64: four
    // warps per 32 nodes.
    struct Form {
        Kernel kernel;
        int most, threads;
    };
    static Form form(const KParams &kp, int ctas)
    {
        const int nodes = rows(kp, ctas) * kp.nx;
        if constexpr (F64) {
            return Form{k_small1<S>, kSmallThreads, (nodes + 31) / 32 * 128};
        } else {
            const int one = (nodes + 31) / 32 * 32, two = (nodes + 63) / 64 * 32;
            // One node a thread as long as a strip's fit: a warp's instructions are a step's time, and a pair's
            // loads and stores are twice a node's (100 x 40 FP32 1.44 -> 1.21 us a step).  Up to 128 threads the
            // kernel may keep every address in registers (37 x 23 FP32 0.95 -> 0.89).
            if (one <= 128) return Form{k_small2<S, v1, 128>, 128, one};
            if (one <= kSmallThreads) return Form{k_small2<S, v1, kSmallThreads>, kSmallThreads, one};
            return Form{k_small2<S, v2x, kSmallThreads>, kSmallThreads, two};
        }
    }
    static size_t bytes(const KParams &kp, int ctas) { return SmallLayout<S>{kp.nx, rows(kp, ctas)}.bytes(IsDev<S>::value && kp.per_node_ref); }
    static constexpr int SMEM = 190 * 1024;
    static constexpr int64_t MAX_NODES = F64 ? 2048 : 16384;
    // CTAs of the cluster that steps this lattice; 0: it is too large (or has interpolated or moving
    // walls), or the device cannot hold the cluster.
    static int ctas(const KParams &kp)
    {
        if (kp.q || kp.wall_u) return 0;
        const int64_t n = (int64_t)kp.nx * kp.ny;
        if (n > MAX_NODES) return 0;
        int c = n > (F64 ? 128 : 1024) ? 16 : 8;
        while (c > kp.ny) c /= 2;
        if ((int64_t)rows(kp, c) * kp.nx > 2 * kSmallThreads || bytes(kp, c) > SMEM) return 0;
        const Form f = form(kp, c);
        return f.threads <= f.most && cluster_fits(reinterpret_cast<const void *>(f.kernel), kp.device, c, f.most, SMEM) ? c : 0;
    }
    static cudaError_t steps(const KParams &kp, int ctas, int64_t nsteps, int64_t step0, cudaStream_t st)
    {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctas);
        const Form f = form(kp, ctas);
        cfg.blockDim = dim3(f.threads);
        cfg.dynamicSmemBytes = bytes(kp, ctas);
        cfg.stream = st;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = ctas;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, f.kernel, kp, nsteps, step0, rows(kp, ctas));
    }
};

}  // namespace lbm
