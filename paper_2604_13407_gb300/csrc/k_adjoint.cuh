// Transposed (adjoint) step of the D2Q9 pseudopotential MRT update, for one storage type
// S with arithmetic type R (FP64 for FP64 storage, FP32 for FP32 and 16-bit storage).
//
// The step maps the stored populations A_t to A_{t+1} = Step(A_t; Fx, Fy, G, T) (Sec. 2:
// pull streaming, moments, psi(rho) from the EOS, F_int = -G psi S with
// S = sum w psi(x + e) e, velocity, m = M f, m_eq, F_m, Q_m, relaxation, M^-1).  Its
// adjoint maps lambda_{t+1} = dJ/dA_{t+1} to lambda_t = W_t + Step'(A_t)^T lambda_{t+1}
// and accumulates dJ/d(Fx, Fy, G, T).  The local chain rule runs backwards through the
// collision at each node; what couples nodes is (i) the psi stencil, which sends dJ/dS(x)
// to psi of the eight neighbours, and (ii) the pull, whose transpose is again a gather:
//
//   lambda_t[i](y) = W_t[i](y) + ( y + e_i is a wall ? g_o(y) + c(y)
//                                                     : g_i(y + e_i) + c(y + e_i) ),
//   o = opposite of i,
//
// where g_i(x) is the part of dJ/df_i(x) that does not pass through psi(rho(x)) and
// c(x) = psi'(rho(x)) dJ/dpsi(x) is the part that does (the same for all nine f_i since
// d rho/d f_i = 1).  So lambda_t is never stored: it is held as the pair (g, c) of the
// step after it, and the next transposed step assembles lambda at its own node.
//
// k_adj runs one transposed step on tiles (as k_tile: 32 columns, two rows a thread in packed FP32,
// one in FP64).  First c of the step after, on the tile and the ring of nodes around it, into shared
// memory: dJ/dpsi(x) = local part + sum_i w_i e_i . dJ/dS(x - e_i) over fluid x - e_i, then c(x) =
// psi'(rho) dJ/dpsi.  Then, per fluid node of the tile: assemble lambda_{t+1} from g and c, recompute
// the forward quantities from A_t and the psi field of A_t, and run the chain rule back to g(x),
// dJ/dS(x), the local part of dJ/dpsi(x) (through F_int = -G psi S) and rho(x).  The last launch of a
// call (AdjArgs::tail) does the first part alone, for the parameter sums and lambda_0.  Parameter
// derivatives are summed per block into per-block FP64 slots that one reduction sums at the end of
// the call.
//
// What bounds it: 148 B a node in FP32 (A_t and g 36 each, psi, dS, rho and the local part of dJ/dpsi,
// read; g, dS, rho and the local part written).  One thread per node in two passes (c in a pass of its
// own) issued 1231 + 390 instructions a node and was bound by them; the packed pair, the shared
// ring and one block-wide reduction (each warp sums one quantity of the block) cut that to 753 (2048^2:
// 322 us for the two passes, about 145 now, 0.64 of the copy rate; 57 % of the schedulers' cycles issue).
#pragma once

#include "k_tile.cuh"
#include "k_twopass.cuh"

namespace lbm {

__device__ __forceinline__ bool wall_link(const KParams &kp, int x, int y, int i, int64_t &kn)
{
    int xn = x + ex_(i), yn = y + ey_(i);
    if (!wrap_xy(kp, xn, yn)) return true;
    if (kp.solid != nullptr && kp.solid[(int64_t)yn * kp.nx + xn] != 0) return true;
    kn = (int64_t)yn * kp.pitch + xn;
    return false;
}

// Objective weights W_i(x) at a fluid node (before the 1/n of the time average);
// inv_nf = 1 / number of fluid nodes in the arithmetic type.
template <class R>
__device__ __forceinline__ R objective_weight(int objective, int i, bool wall_ahead, R inv_nf)
{
    if (objective == 0) return wall_ahead ? R(2 * ey_(i)) : R(0);
    return R(ex_(i)) * inv_nf;
}

// ------------------------------------------------------------ lanes --------------
// The transposed step is written once for a lane type: v2 (two nodes, packed FP32) or d1 (one node,
// FP64; multiply-adds written out, since the FP64 units are compiled without contraction).
struct d1 {
    double v;
};
__device__ __forceinline__ d1 operator+(d1 a, d1 b) { return d1{a.v + b.v}; }
__device__ __forceinline__ d1 operator-(d1 a, d1 b) { return d1{a.v - b.v}; }
__device__ __forceinline__ d1 operator*(d1 a, d1 b) { return d1{a.v * b.v}; }
__device__ __forceinline__ d1 vfma(d1 a, d1 b, d1 c) { return d1{__fma_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ d1 vrcp(d1 a) { return d1{1.0 / a.v}; }
__device__ __forceinline__ d1 vclamp01(d1 a) { return d1{fmin(fmax(a.v, 0.0), 1.0)}; }
__device__ __forceinline__ v2 operator-(v2 a) { return V(-a.v.x, -a.v.y); }
__device__ __forceinline__ d1 operator-(d1 a) { return d1{-a.v}; }

template <class R> struct Lanes;
template <> struct Lanes<float> {
    typedef v2 T;
    static constexpr int N = 2;
    static __device__ __forceinline__ T all(float a) { return S2(a); }
    static __device__ __forceinline__ float get(T a, int e) { return e ? a.v.y : a.v.x; }
    static __device__ __forceinline__ void set(T &a, int e, float v) { (e ? a.v.y : a.v.x) = v; }
};
template <> struct Lanes<double> {
    typedef d1 T;
    static constexpr int N = 1;
    static __device__ __forceinline__ T all(double a) { return d1{a}; }
    static __device__ __forceinline__ double get(T a, int) { return a.v; }
    static __device__ __forceinline__ void set(T &a, int, double v) { a.v = v; }
};

// dp/drho and dp/dT of the EOS.
template <class R, class T>
__device__ __forceinline__ void p_eos_derivs(const KParams &kp, T rho, T &p_rho, T &p_T)
{
    typedef Lanes<R> Z;
    const Consts<R> &c = cst<R>(kp);
    const T one = Z::all(R(1)), RT = Z::all(c.eos_RT), K = Z::all(c.eos_K), KR = Z::all(c.eos_K * c.eos_R), m2a = Z::all(R(-2) * c.eos_a);
    if (kp.eos == 0) {
        const T r = vrcp(vfma(Z::all(-c.eos_b), rho, one));
        p_rho = K * vfma(RT * r, r, m2a * rho);
        p_T = KR * rho * r;
        return;
    }
    const T eta = Z::all(c.eos_b * R(0.25)) * rho;
    const T om = one - eta;
    const T r = vrcp(om), r3 = r * r * r;
    const T g = vfma(eta, vfma(eta, om, one), one) * r3;                                                // (1 + eta + eta^2 - eta^3) / om^3
    const T dg = vfma(eta, vfma(Z::all(R(-2)), eta, Z::all(R(4))), Z::all(R(4))) * (r3 * r);           // dg / d eta
    p_rho = K * vfma(RT, vfma(eta, dg, g), m2a * rho);
    p_T = KR * rho * g;
}

// Block sum of one double added to *acc with one FP64 atomic per block.
__device__ __forceinline__ void block_atomic_add(double v, double *acc)
{
    __shared__ double red[kRowThreads / 32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) red[wid] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int q = 0; q < kRowThreads / 32; ++q) s += red[q];
        if (s != 0.0) atomicAdd(acc, s);
    }
}

// Row units of a block (pairs of rows, FP64: rows), one warp each, and the units of its ring, which the
// same warps take first.
template <class R, int U> struct AdjTile {
    static constexpr int UNITS = U;
    static constexpr int RING = sizeof(R) == 8 ? 3 : 2;
    static constexpr int ROWS = sizeof(R) == 8 ? UNITS : 2 * UNITS;
    static constexpr int THREADS = 32 * UNITS;
};
template <class R, int U>
struct AdjShared {
    typedef AdjTile<R, U> G;
    R c[G::ROWS + 2][kTilePitch];                     // c of the tile and its ring
    R red[7][Lanes<R>::N * 32 * G::UNITS];            // the parameter terms of every node of the tile
};

// One block of a transposed step.  INNER: no node of the tile or its ring reads across an edge of the
// lattice and there are no solid nodes, so every node is a live one and every address is the node's own
// plus a constant of the launch.  (The two instantiations
// share nothing, so the common one carries no tests and no merges of the other's values.)
template <class S, int U, bool INNER>
__device__ __forceinline__ void adj_block(const KParams &kp, const AdjArgs &aa, AdjShared<typename Codec<S>::R, U> &sh_)
{
    typedef typename Codec<S>::R R;
    typedef Lanes<R> Z;
    typedef typename Z::T T;
    typedef AdjTile<R, U> G;
    constexpr int N = Z::N, ROWS = G::ROWS, UNITS = G::UNITS;
    auto &cs = sh_.c;
    auto &red = sh_.red;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = blockIdx.x * kTileX, y0 = blockIdx.y * ROWS;
    // lane's nodes of unit u: their places in the tile (row and column 0 are the ring's) and the lattice
    struct Place {
        int x[N], y[N], r[N], c[N];
    };
    auto place = [&](int u) -> Place {
        Place q;
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (u < UNITS) q.r[e] = N * u + 1 + e, q.c[e] = lane + 1;
            else if (N == 2 && u == UNITS) q.r[e] = e ? ROWS + 1 : 0, q.c[e] = lane + 1;
            else if (N == 1 && u < UNITS + 2) q.r[e] = u == UNITS ? 0 : ROWS + 1, q.c[e] = lane + 1;
            else if (N == 2) q.r[e] = min(lane, ROWS + 1), q.c[e] = e ? kTileX + 1 : 0;
            else q.r[e] = min(lane >> 1, ROWS + 1), q.c[e] = (lane & 1) * (kTileX + 1);
            q.x[e] = x0 + q.c[e] - 1, q.y[e] = y0 + q.r[e] - 1;
        }
        return q;
    };
    // wall bits of a node of the lattice: bit i when x - e_i is a wall
    auto walls_of = [&](const Site &a) -> unsigned {
        if (kp.links != nullptr) return kp.links[(int64_t)a.y * kp.nx + a.x];
        return edge_walls(around(kp, a.x, a.y).inside);
    };
    const int64_t P = kp.plane;
    const Place me = place(warp);
    if (aa.ahead > 0 && lane < (aa.g_in ? 23 : 10)) {
        // the lines of the tile that a block of the next wave will read
        const int ya = me.y[0] + aa.ahead;
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (ya + e >= kp.ny) break;
            const int64_t at = (int64_t)(ya + e) * kp.pitch + x0;
            const void *q;
            if (lane < 9) q = static_cast<const S *>(kp.src) + (lane * P + at);
            else if (lane == 9) q = static_cast<const R *>(kp.psi) + ((int64_t)(ya + e) * kp.nx + x0);
            else if (lane < 19) q = static_cast<const R *>(aa.g_in) + ((lane - 10) * P + at);
            else if (lane < 21) q = static_cast<const R *>(aa.dS_in) + ((lane - 19) * P + at);
            else q = static_cast<const R *>(lane == 21 ? aa.dpsi_in : aa.rho_in) + at;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
        }
    }
    const Consts<R> &cc = cst<R>(kp);
    const T zero = Z::all(R(0));
    T gG2 = zero, gT2 = zero;
    Site at[N];        // this thread's nodes of the tile: in the lattice, wall bits, whether it updates them
    unsigned w[N], walls = 0;
    bool own[N], any = INNER;
#pragma unroll
    for (int e = 0; e < N; ++e) {
        at[e] = INNER ? Site{me.x[e], me.y[e], true} : site_of(kp, me.x[e], me.y[e]);
        w[e] = INNER ? 0u : walls_of(at[e]);
        own[e] = INNER || (at[e].in && !(w[e] & 1u) && me.x[e] < kp.nx && me.y[e] < kp.ny);
        walls |= w[e];
        any |= own[e];
    }

    // ---- c of the step after
    if (aa.g_in != nullptr)
#pragma unroll 1
    for (int u = warp + G::RING < UNITS ? warp : warp + G::RING; u >= 0; u = u >= UNITS ? u - G::RING : -1) {
        // (the last RING warps take a ring unit first, then their own)
        const Place q_ = place(u);
        const R *dSx = static_cast<const R *>(aa.dS_in), *dSy = dSx + P;
        const R *dp = static_cast<const R *>(aa.dpsi_in), *rp = static_cast<const R *>(aa.rho_in);
        T sx[9], sy[9], loc, rho, psi;
        Site a[N];
        bool live[N];
        // the node x - e_i has x in its stencil along e_i
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if constexpr (INNER) {
                a[e] = Site{q_.x[e], q_.y[e], true};
                live[e] = true;
                const int64_t k = (int64_t)a[e].y * kp.pitch + a[e].x;
                const R *px = dSx + k, *pn = px + kp.pitch, *ps_ = px - kp.pitch;
#pragma unroll
                for (int i = 1; i < 9; ++i) {
                    const R *r = ey_(i) > 0 ? ps_ : ey_(i) < 0 ? pn : px;
                    if (ex_(i)) Z::set(sx[i], e, r[-ex_(i)]);
                    if (ey_(i)) Z::set(sy[i], e, (r + P)[-ex_(i)]);
                }
                Z::set(loc, e, dp[k]);
                Z::set(rho, e, rp[k]);
                if constexpr (sizeof(R) == 8) Z::set(psi, e, static_cast<const R *>(aa.psi_in)[k]);
            } else {
                a[e] = site_of(kp, q_.x[e], q_.y[e]);
                const unsigned wq = walls_of(a[e]);
                live[e] = a[e].in && !(wq & 1u);
                unsigned in;
                const Nine nn = nine_of(kp, a[e], in);
#pragma unroll
                for (int i = 1; i < 9; ++i) {
                    const bool wall = (wq >> i) & 1u;
                    if (ex_(i)) Z::set(sx[i], e, wall ? R(0) : dSx[nn.from(i)]);
                    if (ey_(i)) Z::set(sy[i], e, wall ? R(0) : dSy[nn.from(i)]);
                }
                Z::set(loc, e, live[e] ? dp[nn.own()] : R(0));
                Z::set(rho, e, live[e] ? rp[nn.own()] : R(1.0 / 16.0));
                if constexpr (sizeof(R) == 8) Z::set(psi, e, live[e] ? static_cast<const R *>(aa.psi_in)[nn.own()] : R(1));
            }
        }
        if constexpr (sizeof(R) == 4) psi = psi_v<T>(kp, rho);
        const T ax = (sx[1] - sx[3]) + (sy[2] - sy[4]);
        const T dg = ((sx[5] - sx[7]) + (sy[5] - sy[7])) + ((sx[8] - sx[6]) + (sy[6] - sy[8]));
        const T dpsi = vfma(Z::all(R(1.0 / 3.0)), ax, vfma(Z::all(R(1.0 / 12.0)), dg, loc));
        T p_rho, p_T;
        p_eos_derivs<R>(kp, rho, p_rho, p_T);
        // psi^2 = 2 (p - rho/3)/G
        const T q = dpsi * vrcp(Z::all(cc.G) * psi);
        const T c = (p_rho - Z::all(R(1.0 / 3.0))) * q;
#pragma unroll
        for (int e = 0; e < N; ++e) cs[q_.r[e]][q_.c[e]] = live[e] ? Z::get(c, e) : R(0);
        if (u < UNITS) {
            gT2 = p_T * q;
            gG2 = psi * dpsi * Z::all(R(-0.5) / cc.G);
#pragma unroll
            for (int e = 0; e < N; ++e)
                if (aa.tail && own[e]) static_cast<R *>(aa.c_out)[(int64_t)at[e].y * kp.pitch + at[e].x] = Z::get(c, e);
        }
    }
    // ---- the state: the pull of Eq. (lbe.str) with half-way walls (the only walls the adjoint
    // accepts): f_i = A_o(x) + 0 when x - e_i is a wall, as the forward step evaluates it; what
    // lambda_{t+1} takes of g; psi of A_t around the node.  With FP32 storage loaded before the barrier:
    // nothing of the first part is live any more, and their latency passes while the ring's warps finish
    // (2048^2: 244 -> 235 us a step of the call).  Behind it in the others: a 16-bit population's
    // conversion would wait for the load (256 x 1024: 31.2 -> 32.1), and FP64 is bound by its pipe.
    const bool update = any && !aa.tail;
    constexpr bool DEV = IsDev<S>::value, EARLY = sizeof(S) == 4;
    const R *g = static_cast<const R *>(aa.g_in), *psif = static_cast<const R *>(kp.psi);
    T f[9], lam[9], ps[9];
    R pa[N + 2][3];  // psi of the rows y - 1 .. y + N of the thread's column and the columns beside it
    auto load_psi = [&] {
        const R *p = psif + ((int64_t)(me.y[0] - 1) * kp.nx + me.x[0]);
#pragma unroll
        for (int r = 0; r < N + 2; ++r, p += kp.nx)
#pragma unroll
            for (int d = 0; d < 3; ++d) pa[r][d] = p[d - 1];
    };
    auto load = [&](int e) {
        const S *src = static_cast<const S *>(kp.src);
        const int64_t k = (int64_t)at[e].y * kp.pitch + at[e].x;
        if constexpr (INNER) {
            const char *ps_ = reinterpret_cast<const char *>(src + k), *pg = reinterpret_cast<const char *>(g + k);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                R wref = R(0);
                if constexpr (DEV) wref = __fmul_rn(w_<R>(i), kp.per_node_ref ? (kp.ref_src + (k - ey_(i) * kp.pitch))[-ex_(i)] : cc.rho_ref);
                Z::set(f[i], e, Codec<S>::dec(reinterpret_cast<const S *>(ps_ + kp.pull[i])[-ex_(i)], wref, cc.inv_scale));
                Z::set(lam[i], e, g != nullptr ? reinterpret_cast<const R *>(pg + aa.push[i])[ex_(i)] : R(0));
                Z::set(ps[i], e, pa[e + 1 + ey_(i)][1 + ex_(i)]);
            }
        } else {
            unsigned in;
            const Nine nn = nine_of(kp, at[e], in);
            const Around nb = around(kp, at[e].x, at[e].y);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                Z::set(f[i], e, load_pop_at<S>(kp, i, nn.from(i)));
                Z::set(lam[i], e, g != nullptr ? g[i * P + nn.from(opp_(i))] : R(0));
                Z::set(ps[i], e, nb.in(i) ? psif[nb.n(i)] : cc.psi_s);
            }
        }
        if (!INNER && (w[e] & 0x1feu)) {
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                const int o = opp_(i);
                if ((w[e] >> i) & 1u) Z::set(f[i], e, load_pop_at<S>(kp, o, k) + R(0));
                if (((w[e] >> o) & 1u) && g != nullptr) Z::set(lam[i], e, g[o * P + k]);  // x + e_i is a wall
            }
        }
    };
    if (EARLY && update) {
        if (INNER) load_psi();
#pragma unroll
        for (int e = 0; e < N; ++e) load(e);
    }
    const bool walled = INNER ? (__syncthreads(), false) : __syncthreads_or(walls & 0x1feu) != 0;

    T gFx = zero, gFy = zero, gG = zero, gT = zero, Jt = zero;
    if (update) {
        const R wscale = sizeof(R) == 8 ? R(aa.w_scale) : R(aa.w_scale_f);
        const R inv_nf = sizeof(R) == 8 ? R(aa.inv_nfluid) : R(aa.inv_nfluid_f);
        // ---- lambda_{t+1} = W + g + c
        R ca[N + 2][3];  // c like pa
#pragma unroll
        for (int r = 0; r < N + 2; ++r)
#pragma unroll
            for (int d = 0; d < 3; ++d) ca[r][d] = g != nullptr ? cs[me.r[0] - 1 + r][me.c[0] - 1 + d] : R(0);
        const R wi = aa.objective == 0 ? R(0) : wscale * inv_nf;  // objective 1: W_i = e_ix / N_fluid
        if (!EARLY && INNER) load_psi();
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (!EARLY) load(e);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                R v = R(ex_(i)) * wi, c = ca[e + 1 + ey_(i)][1 + ex_(i)];
                if (!INNER && ((w[e] >> opp_(i)) & 1u) && i > 0) {  // x + e_i is a wall
                    v = wscale * objective_weight<R>(aa.objective, i, true, inv_nf);
                    c = ca[e + 1][1];
                }
                if (g != nullptr) v += Z::get(lam[i], e) + c;
                Z::set(lam[i], e, v);
            }
            // the pair's other node may be no fluid node (past the lattice, or solid): keep its arithmetic finite
            if (!INNER && !own[e]) {
#pragma unroll
                for (int i = 0; i < 9; ++i) Z::set(f[i], e, w_<R>(i)), Z::set(lam[i], e, R(0));
            }
        }
        T rho;
        if constexpr (sizeof(R) == 8) {
            rho = d1{((((f[0].v + f[1].v) + f[2].v) + f[3].v) + f[4].v) + f[5].v + f[6].v + f[7].v + f[8].v};
        } else {
            T d[9];
            to_dev(f, d);
            rho = density_dev(d);
        }
        const T p13 = f[1] + f[3], p24 = f[2] + f[4], a13 = f[1] - f[3], a24 = f[2] - f[4];
        const T p57 = f[5] + f[7], p68 = f[6] + f[8], a57 = f[5] - f[7], a68 = f[6] - f[8];
        const T tx = a57 - a68, ty = a57 + a68;
        const T jx = a13 + tx, jy = a24 + ty;
        if (aa.sum_J) {
            // <W, A_t> at this node from its pulled populations: a population stored at x that the next
            // streaming sends into a wall is pulled back by x itself as f_i with x - e_i a wall; every
            // other one is pulled by exactly one fluid node
            T wall_x = zero, wall_y = zero;
            if (!INNER && (walls & 0x1feu)) {
#pragma unroll
                for (int e = 0; e < N; ++e) {
                    R wx = R(0), wy = R(0);
#pragma unroll
                    for (int i = 1; i < 9; ++i)
                        if ((w[e] >> i) & 1u) wx += R(ex_(i)) * Z::get(f[i], e), wy += R(ey_(i)) * Z::get(f[i], e);
                    Z::set(wall_x, e, wx), Z::set(wall_y, e, wy);
                }
            }
            Jt = aa.objective == 0 ? Z::all(R(-2)) * wall_y : vfma(Z::all(R(-2)), wall_x, jx) * Z::all(inv_nf);
        }
        const T third = Z::all(R(1.0 / 3.0)), twelfth = Z::all(R(1.0 / 12.0));
        const T dd = ps[5] - ps[7], de = ps[8] - ps[6];
        const T Sx = vfma(third, ps[1] - ps[3], twelfth * (dd + de));
        const T Sy = vfma(third, ps[2] - ps[4], twelfth * (dd - de));
        const T psi = ps[0];
        const bool buoyant = kp.force_mode != 0;
        const T cFx = Z::all(cc.Fx), cFy = Z::all(cc.Fy), rexc = rho - Z::all(cc.rho_g);
        const T mG = Z::all(-cc.G), nGpsi = mG * psi;
        const T Fx = buoyant ? vfma(nGpsi, Sx, rexc * cFx) : vfma(nGpsi, Sx, cFx);
        const T Fy = buoyant ? vfma(nGpsi, Sy, rexc * cFy) : vfma(nGpsi, Sy, cFy);
        const T half = Z::all(R(0.5)), two = Z::all(R(2)), six = Z::all(R(6)), three = Z::all(R(3));
        const T inv = vrcp(rho);
        const T ux = vfma(half, Fx, jx) * inv, uy = vfma(half, Fy, jy) * inv;
        const T uxx = ux * ux, uyy = uy * uy, u2 = uxx + uyy, ud = uxx - uyy, uxy = ux * uy;
        const T Sx2 = Sx * Sx, Sy2 = Sy * Sy;
        const bool improved = kp.improved != 0;
        const T kq1 = Z::all(cc.kq1), kq7 = Z::all(cc.kq7), q2f = Z::all(cc.q2fac), c1G = Z::all(cc.c1G), mc2G = Z::all(-cc.c2G);
        const T Q1 = kq1 * (Sx2 + Sy2), Q7 = kq7 * (Sx2 - Sy2), Q8 = kq7 * (Sx * Sy);
        T A4 = zero, A6 = zero;
        if (improved) A4 = vfma(c1G, Sx2, mc2G * Sy2), A6 = vfma(c1G, Sy2, mc2G * Sx2);

        // ---- backward: lambda -> dJ/d m_bar (f_bar = M^T diag(1/|M_k|^2) m_bar)
        const T l13p = lam[1] + lam[3], l24p = lam[2] + lam[4], l13 = lam[1] - lam[3], l24 = lam[2] - lam[4];
        const T l57p = lam[5] + lam[7], l68p = lam[6] + lam[8], l57 = lam[5] - lam[7], l68 = lam[6] - lam[8];
        const T lt = l57 - l68, lv = l57 + l68, a14 = l13p + l24p, a58 = l57p + l68p;
        const T b0 = (lam[0] + a14 + a58) * Z::all(R(1.0 / 9.0));
        const T b1 = vfma(Z::all(R(4)), lam[0], vfma(Z::all(R(-2)), a58, a14)) * Z::all(R(-1.0 / 36.0));
        const T b2 = vfma(Z::all(R(4)), lam[0], vfma(Z::all(R(-2)), a14, a58)) * Z::all(R(1.0 / 36.0));
        const T b3 = (l13 + lt) * Z::all(R(1.0 / 6.0)), b4 = vfma(Z::all(R(-2)), l13, lt) * Z::all(R(1.0 / 12.0));
        const T b5 = (l24 + lv) * Z::all(R(1.0 / 6.0)), b6 = vfma(Z::all(R(-2)), l24, lv) * Z::all(R(1.0 / 12.0));
        const T b7 = (l13p - l24p) * Z::all(R(0.25)), b8 = (l57p - l68p) * Z::all(R(0.25));

        T sp = Z::all(cc.sp), sq = Z::all(cc.sq), drho = zero;
        if (kp.var_tau) {
            const T inv_d = Z::all(R(1) / (cc.rho_l - cc.rho_g)), dnu = Z::all(cc.nu_l - cc.nu_g);
            const T wraw = rexc * inv_d, tm = three * vfma(vclamp01(wraw), dnu, Z::all(cc.nu_g));  // tau - 1/2
            const T rtm = vrcp(tm);
            sp = vrcp(tm + half);
            sq = vrcp(vfma(Z::all(cc.Lambda), rtm, half));
            const T s14 = p13 + p24, s58 = p57 + p68;
            const T m1 = vfma(Z::all(R(-4)), f[0], vfma(two, s58, -s14)), m2 = vfma(Z::all(R(4)), f[0], vfma(Z::all(R(-2)), s14, s58));
            const T m4 = vfma(Z::all(R(-2)), a13, tx), m6 = vfma(Z::all(R(-2)), a24, ty), m7 = p13 - p24, m8 = p57 - p68;
            const T Fu = vfma(Fx, ux, Fy * uy), t3 = three * rho * u2;
            const T e1 = (vfma(Z::all(R(-2)), rho, t3) - m1) - three * Fu + Q1;
            const T e2 = ((rho - t3) - m2) + three * Fu + q2f * Q1;
            const T e7 = vfma(rho, ud, -m7) - vfma(Fx, ux, -(Fy * uy)) + Q7;
            const T e8 = vfma(rho, uxy, -m8) - half * vfma(Fx, uy, Fy * ux) + Q8;
            const T e4 = vfma(half, Fx, vfma(A4, ux, -vfma(rho, ux, m4)));
            const T e6 = vfma(half, Fy, vfma(A6, uy, -vfma(rho, uy, m6)));
            const T dsp = vfma(b1, e1, vfma(b2, e2, vfma(b7, e7, b8 * e8)));
            const T dsq = vfma(b4, e4, b6 * e6);
            const T dtau = vfma(dsq * sq * sq, Z::all(cc.Lambda) * rtm * rtm, -(dsp * sp * sp));
            const T dr = three * dtau * dnu * inv_d;
#pragma unroll
            for (int e = 0; e < N; ++e)
                if (Z::get(wraw, e) > R(0) && Z::get(wraw, e) < R(1)) Z::set(drho, e, Z::get(dr, e));
        }
        const T one = Z::all(R(1)), hsp = vfma(Z::all(R(-0.5)), sp, one), mhsq = vfma(half, sq, Z::all(R(-1)));  // 1 - s_p/2, -(1 - s_q/2)

        // m_bar_k = (1 - s_k) m_k + s_k m_eq_k + (1 - s_k/2) F_m_k + s_k Q_k (Eq. lbe.col);
        // s_0 = s_j = 1 (m_bar_0 = rho, m_bar_j = rho u + F/2).  d_k = s_k b_k = dJ/d m_eq_k = dJ/d Q_k
        const T d1_ = sp * b1, d2 = sp * b2, d4 = sq * b4, d6 = sq * b6, d7 = sp * b7, d8 = sp * b8;
        const T dm1 = b1 - d1_, dm2 = b2 - d2, dm4 = b4 - d4, dm6 = b6 - d6, dm7 = b7 - d7, dm8 = b8 - d8;
        const T d12 = d1_ - d2, d34 = b3 - d4, d56 = b5 - d6;
        // m_eq(rho, u)
        drho = drho + (vfma(Z::all(R(-2)), d1_, b0) + d2) + vfma(three * u2, d12, vfma(ux, d34, vfma(uy, d56, vfma(ud, d7, uxy * d8))));
        const T s12 = six * d12, t7 = two * d7;
        T dux = rho * vfma(ux, s12 + t7, vfma(uy, d8, d34));
        T duy = rho * vfma(uy, s12 - t7, vfma(ux, d8, d56));
        // F_m(F, u)
        const T dFu = six * hsp * (b1 - b2), g7 = two * hsp * b7, g8 = hsp * b8;
        T dFx = vfma(ux, dFu + g7, vfma(uy, g8, vfma(half, b3, mhsq * b4)));
        T dFy = vfma(uy, dFu - g7, vfma(ux, g8, vfma(half, b5, mhsq * b6)));
        dux = vfma(Fx, dFu + g7, vfma(Fy, g8, dux));
        duy = vfma(Fy, dFu - g7, vfma(Fx, g8, duy));
        // Q(S, u), with |F_int|^2/(G psi^2) = G |S|^2; the coefficients carry one factor G
        const T dQ1 = vfma(q2f, d2, d1_);
        const T k1 = kq1 * dQ1, k7 = kq7 * d7, k8 = kq7 * d8;
        T dSx = vfma(two * Sx, k1 + k7, Sy * k8);
        T dSy = vfma(two * Sy, k1 - k7, Sx * k8);
        T dG = vfma(Q1, dQ1, vfma(Q7, d7, Q8 * d8));
        if (improved) {
            const T x4 = ux * d4, y6 = uy * d6;
            dux = vfma(A4, d4, dux);
            duy = vfma(A6, d6, duy);
            dSx = vfma(two * Sx, vfma(c1G, x4, mc2G * y6), dSx);
            dSy = vfma(two * Sy, vfma(c1G, y6, mc2G * x4), dSy);
            dG = vfma(A4, x4, vfma(A6, y6, dG));
        }
        dG = dG * Z::all(R(1) / cc.G);
        // u = (j + F/2)/rho
        const T djx = dux * inv, djy = duy * inv;
        dFx = vfma(half, djx, dFx);
        dFy = vfma(half, djy, dFy);
        drho = drho - vfma(ux, djx, uy * djy);
        // F = -G psi S + F_ext
        if (buoyant) {
            gFx = rexc * dFx;
            gFy = rexc * dFy;
            drho = vfma(cFx, dFx, vfma(cFy, dFy, drho));
        } else {
            gFx = dFx;
            gFy = dFy;
        }
        const T SdF = vfma(Sx, dFx, Sy * dFy);
        const T dpsi_loc = mG * SdF;
        dG = dG - psi * SdF;
        dSx = vfma(nGpsi, dFx, dSx);
        dSy = vfma(nGpsi, dFy, dSy);
        // walls in the stencil carry psi(rho_s; T, G)
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (INNER || !own[e] || !(w[e] & 0x1feu)) continue;
            R dpsi_s = R(0);
#pragma unroll
            for (int i = 1; i < 9; ++i)
                if ((w[e] >> opp_(i)) & 1u) dpsi_s += omega_<R>(i) * (R(ex_(i)) * Z::get(dSx, e) + R(ey_(i)) * Z::get(dSy, e));
            if (dpsi_s != R(0)) {
                T prs, pTs;
                p_eos_derivs<R>(kp, Z::all(cc.rho_s), prs, pTs);
                Z::set(dG, e, Z::get(dG, e) - cc.psi_s / (R(2) * cc.G) * dpsi_s);
                Z::set(gT, e, Z::get(pTs, e) / (cc.G * cc.psi_s) * dpsi_s);
            }
        }
        gG = dG;

        // g_i = drho + e_i . dj + (M^T dm)_i
        const T ga = drho - vfma(two, dm2, dm1), gd = drho + vfma(two, dm1, dm2);
        const T hx = vfma(Z::all(R(-2)), dm4, djx), hy = vfma(Z::all(R(-2)), dm6, djy);
        const T ax7 = ga + dm7, ay7 = ga - dm7, ex = djx + dm4, ey = djy + dm6;
        const T dp = gd + dm8, dq = gd - dm8, es = ex + ey, ed = ey - ex;
        const T go[9] = {vfma(Z::all(R(4)), dm2 - dm1, drho), ax7 + hx, ay7 + hy, ax7 - hx, ay7 - hy, dp + es, dq + ed, dp - es, dq - ed};
#pragma unroll
        for (int e = 0; e < N; ++e) {
            if (!INNER && !own[e]) continue;
            const int64_t k = (int64_t)at[e].y * kp.pitch + at[e].x;
            R *out = static_cast<R *>(aa.g_out) + k, *dS = static_cast<R *>(aa.dS_out) + k;
#pragma unroll
            for (int i = 0; i < 9; ++i, out += P) *out = Z::get(go[i], e);
            dS[0] = Z::get(dSx, e);
            dS[P] = Z::get(dSy, e);
            static_cast<R *>(aa.dpsi_out)[k] = Z::get(dpsi_loc, e);
            static_cast<R *>(aa.rho_out)[k] = Z::get(rho, e);
            if constexpr (sizeof(R) == 8) static_cast<R *>(aa.psi_out)[k] = Z::get(psi, e);
        }
    }
    // ---- parameter sums, in the order of AdjSlot: one row of FP64 partial sums per block, accumulated over
    // all steps of a call and reduced once at its end (no other block adds to it: a fixed order).  Added in L2:
    // a load of the row's entry and an FP64 add were the last thing a block waited for (2048^2: 231 -> 226 us
    // a step of the call).
    {
        const T v[7] = {gFx, gFy, gG, gT, Jt, gG2, gT2};
#pragma unroll
        for (int q = 0; q < 7; ++q)
#pragma unroll
            for (int e = 0; e < N; ++e) red[q][threadIdx.x + e * 32 * UNITS] = own[e] ? Z::get(v[q], e) : R(0);
    }
    __syncthreads();
    // away from walls the wall terms (and objective 0, the force on them) are zero
    const unsigned skip = walled ? 0u : (1u << SLOT_T1) | (aa.objective == 0 ? 1u << SLOT_J : 0u);
    block_add<R>(&red[0][0], N * 32 * UNITS, 7, N * 32 * UNITS, UNITS, skip,
                 [&](int q, double t) { atomicAdd(&aa.part[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kAdjSlots + q], t); });
}

// One transposed step at A_t (kp.src) with the psi field of A_t (kp.psi).  U: units of a block, B: blocks
// per SM the registers must allow.
template <class S, int U, int B>
__global__ void __launch_bounds__(32 * U, B) k_adj(KParams kp, AdjArgs aa)
{
    typedef AdjTile<typename Codec<S>::R, U> G;
    __shared__ AdjShared<typename Codec<S>::R, U> sh;
    grid_dependency_wait();
    allow_dependent_launch();
    const int x0 = blockIdx.x * kTileX, y0 = blockIdx.y * G::ROWS;
    if (x0 >= 2 && x0 + kTileX + 2 <= kp.nx && y0 >= 2 && y0 + G::ROWS + 2 <= kp.ny && kp.links == nullptr)
        adj_block<S, U, true>(kp, aa, sh);
    else
        adj_block<S, U, false>(kp, aa, sh);
}

// lambda_0 = dJ/dA at the starting state (no objective weight at t = 0), FP64 [9][ny][nx], from g and c.
template <class S>
__global__ void __launch_bounds__(kRowThreads) k_adj_lambda(KParams kp, const typename Codec<S>::R *g,
                                                            const typename Codec<S>::R *c, double *out)
{
    typedef typename Codec<S>::R R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const int64_t n = (int64_t)kp.nx * kp.ny, node = (int64_t)y * kp.nx + x, k = (int64_t)y * kp.pitch + x;
    const bool solid = node_is_solid(kp, node);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        int64_t kn = k;
        R v = R(0);
        if (!solid) v = i != 0 && wall_link(kp, x, y, i, kn) ? g[opp_(i) * kp.plane + k] + c[k] : g[i * kp.plane + kn] + c[kn];
        out[i * n + node] = double(v);
    }
}

// FP64 sum over fluid nodes of sum_i W_i(x) A_i(x) for the state kp.src.
template <class S>
__global__ void __launch_bounds__(kRowThreads) k_objective(KParams kp, int objective, double inv_nfluid, double *acc)
{
    typedef typename Codec<S>::R R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    const int64_t node = (int64_t)y * kp.nx + x;
    double v = 0.0;
    if (x < kp.nx && !node_is_solid(kp, node)) {
        AdjArgs aa{};
        aa.objective = objective;
        aa.inv_nfluid = inv_nfluid;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            int64_t kn;
            const bool wall = (i != 0) && wall_link(kp, x, y, i, kn);
            const double w = double(objective_weight<R>(aa.objective, i, wall, R(aa.inv_nfluid)));
            if (w != 0.0) v += w * double(load_pop<S>(kp, i, x, y));
        }
    }
    block_atomic_add(v, acc);
}

// Sum of the per-block slots: out[k] = sum over blocks of part[b][k], one block per slot,
// in a fixed order (instantiated per storage type S, like the passes it sums).
template <class S>
__global__ void __launch_bounds__(256) k_adj_reduce(const double *part, int64_t blocks, double *out)
{
    __shared__ double red[8];
    const int k = blockIdx.x;
    double s = 0.0;
    for (int64_t b = threadIdx.x; b < blocks; b += blockDim.x) s += part[b * kAdjSlots + k];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < 8; ++q) t += red[q];
        out[k] = t;
    }
}

template <class S>
struct Adjoint {
    // FP32 arithmetic: tall tiles and 128 registers on small lattices, where a block's ring is a large
    // part of its work and there are few blocks to hide latency (256 x 1024: 27.0 us a step of the call
    // against 28.8; between them, six units by three blocks, 29.2); short ones and five blocks per SM from
    // 2^19 nodes (2048^2: 234 against 254; six by three 240).
    static constexpr bool F64 = sizeof(typename Codec<S>::R) == 8;
    static bool tall(const KParams &kp) { return F64 || (int64_t)kp.nx * kp.ny < (int64_t)1 << 19; }
    static int rows(const KParams &kp) { return F64 ? 8 : tall(kp) ? 16 : 8; }
    static dim3 grid(const KParams &kp) { return dim3((kp.nx + kTileX - 1) / kTileX, (kp.ny + rows(kp) - 1) / rows(kp)); }
    static cudaError_t step(const KParams &kp, const AdjArgs &args, cudaStream_t st)
    {
        typedef typename Codec<S>::R R;
        AdjArgs aa = args;
        KParams kq = kp;
        for (int i = 0; i < 9; ++i) {
            kq.pull[i] = (i * kp.plane - ey_(i) * kp.pitch) * (int64_t)sizeof(S);
            aa.push[i] = (i * kp.plane + ey_(i) * kp.pitch) * (int64_t)sizeof(R);
        }
        // rows between a tile and the one it prefetches: two blocks per SM further on, where the planes
        // read and written exceed the 129 MB L2
        const int sms = kp.sm_count > 0 ? kp.sm_count : 148;
        const double bytes = kp.plane * (9.0 * sizeof(S) + 27.0 * sizeof(R));
        aa.ahead = bytes > 120e6 && !aa.tail ? (int)(2u * sms / grid(kp).x + 1) * rows(kp) : 0;
        if constexpr (F64) {
            return launch_dependent(k_adj<S, 8, 1>, grid(kp), dim3(256), 0, st, kq, aa);
        } else {
            return tall(kp) ? launch_dependent(k_adj<S, 8, 2>, grid(kp), dim3(256), 0, st, kq, aa)
                            : launch_dependent(k_adj<S, 4, 5>, grid(kp), dim3(128), 0, st, kq, aa);
        }
    }
    // blocks of the transposed step (rows of the partial-sum array)
    static int64_t blocks(const KParams &kp) { return (int64_t)grid(kp).x * grid(kp).y; }
    static cudaError_t lambda(const KParams &kp, const void *g, const void *c, double *out, cudaStream_t st)
    {
        typedef typename Codec<S>::R R;
        k_adj_lambda<S><<<row_grid(kp), kRowThreads, 0, st>>>(kp, static_cast<const R *>(g), static_cast<const R *>(c), out);
        return cudaGetLastError();
    }
    static cudaError_t reduce(const KParams &kp, const double *part, double *out, cudaStream_t st)
    {
        k_adj_reduce<S><<<kAdjSlots, 256, 0, st>>>(part, blocks(kp), out);
        return cudaGetLastError();
    }
    static cudaError_t objective(const KParams &kp, int obj, double inv_nfluid, double *acc, cudaStream_t st)
    {
        k_objective<S><<<row_grid(kp), kRowThreads, 0, st>>>(kp, obj, inv_nfluid, acc);
        return cudaGetLastError();
    }
};

}  // namespace lbm
