// One-pass step on tiles of 32 columns: psi of the tile and of the ring of nodes around it goes
// through shared memory, so one launch does what the psi pass and the collide pass do in two.
//
// FP32 arithmetic (k_tile2; FP32, FP16 and BF16 storage): a thread owns two nodes of one column,
// rows y and y + 1, and evaluates them as one packed pair.  A vertical pair keeps every access of a
// warp 32 consecutive elements wide at any lattice width, alignment and storage type, and a pair
// needs no alignment of nx; the packed instructions halve the arithmetic instructions of the
// one-node passes.  The packed products are written as multiply-adds with -0 (v2x): the assembler
// fuses a packed product into a following packed sum, which rounds once where the one-node
// evaluation rounds twice; with them every node's result is the two-pass step's, bit for bit (the
// links of interpolated and moving walls to rounding: their coefficients come from the link
// records, formed in FP64).
// FP64 (k_tile1): one node per thread, the two-pass step's own functions, the same bits.
//
// A tile of n pairs (rows) has n warps for them; one more warp pulls the rows above and below the
// tile and one the columns beside it (FP64: two and one), for psi only.  The tile's height is
// chosen per launch (tile_height) so that the last wave of blocks is nearly full.
//
// What bounds it (FP32): small lattices the latency of one block's chain, mid-size ones instruction
// issue (578 a pair of rows and 32 columns, ring included; the two-pass kernels 1840), from 2048^2 on HBM:
// 4096^2 193 us, 94 % of the measured copy rate at 72 B a node. Four pairs and five blocks per SM (64
// registers) against two blocks of eight pairs: 512 x 4096 46 -> 36 us; the L2 prefetch 70 -> 59 at 2048^2;
// the instantiation without edge tests (INNER) 59 -> 52, FP16 81 -> 67.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// ------------------------------------------------------- exact packed pairs ------
// Packed FP32x2 with every operation rounded as written: a product is a multiply-add with -0 from
// constant memory, whose value the assembler does not know (RN(a b + -0) = RN(a b), signs of zero
// included), so it cannot be fused with the sum that follows.
struct v2x {
    float2 v;
};
static __constant__ float2 kNegZero = {-0.0f, -0.0f};
__device__ __forceinline__ v2x X2(float a, float b) { return v2x{make_float2(a, b)}; }
__device__ __forceinline__ v2x operator+(v2x a, v2x b) { return v2x{__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ v2x operator-(v2x a, v2x b) { return v2x{__fadd2_rn(a.v, make_float2(-b.v.x, -b.v.y))}; }
__device__ __forceinline__ v2x operator*(v2x a, v2x b) { return v2x{__ffma2_rn(a.v, b.v, kNegZero)}; }
__device__ __forceinline__ v2x vfma(v2x a, v2x b, v2x c) { return v2x{__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ v2x vrcp(v2x a) { return X2(rcp32(a.v.x), rcp32(a.v.y)); }
__device__ __forceinline__ v2x vsqrt(v2x a) { return X2(sqrt32(a.v.x), sqrt32(a.v.y)); }
__device__ __forceinline__ v2x vclamp01(v2x a) { return X2(fminf(fmaxf(a.v.x, 0.f), 1.f), fminf(fmaxf(a.v.y, 0.f), 1.f)); }
template <> __device__ __forceinline__ v2x ks<v2x>(float a) { return X2(a, a); }
template <> __device__ __forceinline__ v2x kc<v2x>(const float2 &c) { return v2x{c}; }

// ------------------------------------------------------------------ tiles --------
constexpr int kTileX = 32;        // columns of a tile
constexpr int kTilePairs = 4;     // most row pairs of a tile (FP32 arithmetic)
constexpr int kTileRows = 8;      // most rows of a tile (FP64)
constexpr int kTilePitch = kTileX + 2;

// Node (x, y) of a tile or of the ring around it: its place in the lattice after wrapping, or
// `in` = false beyond a non-periodic edge (psi(rho_s)) and for the part of a ragged tile that lies
// past the lattice and its ring (never used); x and y are then some node's, so loads stay inside.
struct Site {
    int x, y;
    bool in;
};
__device__ __forceinline__ Site site_of(const KParams &kp, int x, int y)
{
    Site s{x, y, true};
    if (x < 0 || x >= kp.nx) {
        s.in = kp.periodic_x && x >= -1 && x <= kp.nx;
        s.x = s.in ? (x < 0 ? x + kp.nx : x - kp.nx) : 0;
    }
    if (y < 0 || y >= kp.ny) {
        const bool ok = kp.periodic_y && y >= -1 && y <= kp.ny;
        s.in = s.in && ok;
        s.y = ok ? (y < 0 ? y + kp.ny : y - kp.ny) : 0;
    }
    return s;
}

// Wall bits of a node: bit i (1..8) when the source x - e_i of population i is a wall (a solid node
// or beyond a non-periodic edge), bit 0 when the node itself is solid.
__device__ __forceinline__ unsigned edge_walls(unsigned inside)
{
    unsigned w = 0;
#pragma unroll
    for (int i = 1; i < 9; ++i)
        if (!((inside >> opp_(i)) & 1u)) w |= 1u << i;
    return w;
}

// The same plane for every node, from the solid flags (KParams::links; built by set_geometry, read by
// the steps: one 2-byte load where the pull would test nine flags).
static __global__ void __launch_bounds__(128) k_link_bits(KParams kp, uint16_t *out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= kp.nx) return;
    const Around nb = around(kp, x, y);
    unsigned w = edge_walls(nb.inside);
#pragma unroll
    for (int i = 1; i < 9; ++i)
        if (nb.in(opp_(i)) && kp.solid && kp.solid[nb.n(opp_(i))] != 0) w |= 1u << i;
    if (kp.solid && kp.solid[nb.n(0)] != 0) w |= 1u;
    out[nb.n(0)] = (uint16_t)w;
}

// A stored population as FP32: converted and multiplied in one mixed-precision instruction (exact
// product, one rounding of the sum: Codec's value).
template <class S> struct Raw;
template <> struct Raw<float> {
    static __device__ __forceinline__ float f(float v, float, const KParams &) { return v; }
};
template <> struct Raw<__half> {
    static __device__ __forceinline__ float f(__half v, float wref, const KParams &kp)
    {
        float x;
        asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(x) : "h"(__half_as_ushort(v)), "h"(kp.inv_scale_bits), "f"(wref));
        return x;
    }
};
template <> struct Raw<__nv_bfloat16> {
    static __device__ __forceinline__ float f(__nv_bfloat16 v, float wref, const KParams &kp)
    {
        float x;
        asm("fma.rn.f32.bf16 %0, %1, %2, %3;" : "=f"(x) : "h"(__bfloat16_as_ushort(v)), "h"(kp.inv_scale_bits), "f"(wref));
        return x;
    }
};

// Offsets (elements; a plane of a lattice of 2^31 nodes still fits 32 bits) of the 3 x 3 neighbourhood
// of a node.
struct Nine {
    uint32_t r[3], c[3];
    __device__ __forceinline__ uint32_t from(int i) const { return r[1 - ey_(i)] + c[1 - ex_(i)]; }  // x - e_i
    __device__ __forceinline__ uint32_t own() const { return r[1] + c[1]; }
};
__device__ __forceinline__ Nine nine_of(const KParams &kp, const Site &s, unsigned &inside)
{
    const Around a = around(kp, s.x, s.y);
    Nine n;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        n.r[d] = (uint32_t)a.yr[d] * (uint32_t)kp.pitch;
        n.c[d] = (uint32_t)a.xc[d];
    }
    inside = a.inside;
    return n;
}
// One block of a step.  GEOM: 0 no solid nodes; 1 solid nodes with half-way links; 2 also interpolated
// or moving walls.  INNER: the tile lies inside the lattice and no node of it or its ring pulls across
// an edge, so every address is the node's own plus a constant of the launch (KParams::pull).
template <class S, int GEOM, class O, bool INNER>
__device__ __forceinline__ void tile2_block(const KParams &kp, int ahead, float (&sm)[2 * kTilePairs + 2][kTilePitch])
{
    constexpr bool DEV = IsDev<S>::value;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int np = (blockDim.x >> 5) - 2, rows = 2 * np;  // pairs and rows of this launch's tiles
    const int x0 = blockIdx.x * kTileX, y0 = blockIdx.y * rows;
    const bool has_ref = DEV && O::per_node_ref(kp);
    // the two nodes of this thread, and where their psi goes
    int ax, ay, bx, by, ra, rb, ca, cb;
    if (warp < np) {
        ax = bx = x0 + lane, ay = y0 + 2 * warp, by = ay + 1;
        ra = 2 * warp + 1, rb = ra + 1, ca = cb = lane + 1;
    } else if (warp == np) {
        ax = bx = x0 + lane, ay = y0 - 1, by = y0 + rows;
        ra = 0, rb = rows + 1, ca = cb = lane + 1;
    } else {
        const int r = min(lane, rows + 1);
        ax = x0 - 1, bx = x0 + kTileX, ay = by = y0 + r - 1;
        ra = rb = r, ca = 0, cb = kTileX + 1;
    }
    if (ahead > 0 && warp < np && lane < 18) {
        // the lines of the tile that a block of the next wave will pull (row y, columns x0 .. x0 + 31)
        const int i = lane < 9 ? lane : lane - 9, y = ay + (lane < 9 ? 0 : 1) + ahead;
        if (y < kp.ny) {
            const S *p = static_cast<const S *>(kp.src) + (i * kp.plane + (int64_t)y * kp.pitch + x0);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
        }
    }
    Site a{ax, ay, true}, b{bx, by, true};
    if constexpr (!INNER) a = site_of(kp, ax, ay), b = site_of(kp, bx, by);
    const uint32_t node_a = (uint32_t)a.y * (uint32_t)kp.nx + a.x, node_b = (uint32_t)b.y * (uint32_t)kp.nx + b.x;
    const uint32_t ka = (uint32_t)a.y * (uint32_t)kp.pitch + a.x, kb = (uint32_t)b.y * (uint32_t)kp.pitch + b.x;
    unsigned wa = 0, wb = 0;  // wall bits
    if (GEOM) wa = kp.links[node_a], wb = kp.links[node_b];

    // pull, Eq. (lbe.str)
    const S *src = static_cast<const S *>(kp.src);
    v2x f[9];
    S va[9], vb[9];
    float refa[9], refb[9];
    if constexpr (INNER) {
        const char *pa = reinterpret_cast<const char *>(src + ka), *pb = reinterpret_cast<const char *>(src + kb);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            va[i] = reinterpret_cast<const S *>(pa + kp.pull[i])[-ex_(i)];
            vb[i] = reinterpret_cast<const S *>(pb + kp.pull[i])[-ex_(i)];
        }
        if (has_ref) {
            const float *qa = kp.ref_src + ka, *qb = kp.ref_src + kb;
            const int64_t P = kp.pitch;
            if (warp < np) {  // rows y and y + 1: twelve references for both nodes
#pragma unroll
                for (int d = -1; d <= 1; ++d) {
                    const int up = d < 0 ? 5 : d > 0 ? 6 : 2, in = d < 0 ? 1 : d > 0 ? 3 : 0, dn = d < 0 ? 8 : d > 0 ? 7 : 4;
                    refa[up] = (qa - P)[d];
                    refa[in] = refb[up] = qa[d];
                    refa[dn] = refb[in] = qb[d];
                    refb[dn] = (qb + P)[d];
                }
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) refa[i] = (qa - ey_(i) * P)[-ex_(i)], refb[i] = (qb - ey_(i) * P)[-ex_(i)];
            }
        }
    } else {
        unsigned ia, ib;
        const Nine na = nine_of(kp, a, ia), nb = nine_of(kp, b, ib);
        if (GEOM == 0) wa = edge_walls(ia), wb = edge_walls(ib);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const S *p = src + i * kp.plane;
            va[i] = p[na.from(i)], vb[i] = p[nb.from(i)];
            if (has_ref) refa[i] = kp.ref_src[na.from(i)], refb[i] = kp.ref_src[nb.from(i)];
        }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        v2x wr = X2(0.f, 0.f);
        if (DEV) wr = has_ref ? v2x{kp.c2.w[i]} * X2(refa[i], refb[i]) : v2x{kp.c2.dec[i]};
        f[i] = X2(Raw<S>::f(va[i], wr.v.x, kp), Raw<S>::f(vb[i], wr.v.y, kp));
    }
    if ((!INNER || GEOM) && ((wa | wb) & 0x1feu)) {
        // wall links: the population that left the node toward the wall comes back
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const unsigned w = e ? wb : wa;
            if (!(w & 0x1feu) || (w & 1u)) continue;
            const uint32_t k = e ? kb : ka;
            auto own = [&](int i) -> float {
                float wr = 0.f;
                if (DEV) wr = __fmul_rn(w_<float>(i), has_ref ? (e ? refb[0] : refa[0]) : kp.cf.rho_ref);
                return Raw<S>::f((src + i * kp.plane)[k], wr, kp);
            };
            float rho_w = 0.f;
            bool summed = false;
#pragma unroll
            for (int i = 1; i < 9; ++i) {
                if (!((w >> i) & 1u)) continue;
                const int o = opp_(i);
                const float fo = own(o);
                float g = fo + 0.f;
                if constexpr (GEOM == 2) {
                    // interpolated or moving wall: link fraction and moving-wall coefficient
                    const float2 lk = kp.link[(int64_t)(i - 1) * kp.plane + k];
                    float mw = 0.f;
                    if (lk.y != 0.f) {
                        if (!summed) {
#pragma unroll
                            for (int n = 0; n < 9; ++n) rho_w += own(n);
                            summed = true;
                        }
                        mw = lk.y * rho_w;
                    }
                    const float q = lk.x;
                    if (q < 0.5f) {
                        // fbar_o of the second node x + e_i (fluid: the record's q is 1/2 otherwise), which
                        // is what the pull of population o brought here
                        const float f2 = e ? f[o].v.y : f[o].v.x;
                        g = 2.f * q * fo + (1.f - 2.f * q) * f2 + mw;
                    } else if (q == 0.5f) {
                        g = fo + mw;
                    } else {
                        g = fo / (2.f * q) + (2.f * q - 1.f) / (2.f * q) * own(i) + mw / (2.f * q);
                    }
                }
                if (e) f[i].v.y = g;
                else f[i].v.x = g;
            }
        }
    }
    v2x d[9];
    to_dev(f, d);
    v2x rho = density_dev(d);
    v2x psi = psi_v<v2x>(kp, rho);
    if (GEOM) {
        if (wa & 1u) psi.v.x = kp.wall_psi ? float(kp.wall_psi[node_a]) : kp.cf.psi_s, rho.v.x = 1.f;
        if (wb & 1u) psi.v.y = kp.wall_psi ? float(kp.wall_psi[node_b]) : kp.cf.psi_s, rho.v.y = 1.f;
    }
    if (!INNER && !a.in) psi.v.x = kp.cf.psi_s;
    if (!INNER && !b.in) psi.v.y = kp.cf.psi_s;
    sm[ra][ca] = psi.v.x;
    sm[rb][cb] = psi.v.y;
    __syncthreads();
    if (warp >= np) return;
    const bool la = INNER || (ax < kp.nx && ay < kp.ny), lb = INNER || (ax < kp.nx && by < kp.ny);
    if (!la) return;
    if (kp.psi_out != nullptr) {
        float *out = static_cast<float *>(kp.psi_out);
        out[node_a] = psi.v.x;
        if (lb) out[node_b] = psi.v.y;
    }
    const bool sa = !(GEOM && (wa & 1u)), sb = lb && !(GEOM && (wb & 1u));
    if (!sa && !sb) return;

    // S of Eq. (fint) from the four psi rows around the pair
    const float *q = &sm[2 * warp][lane];
    float c[4][3];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) c[r][k] = q[r * kTilePitch + k];
    v2x Sx, Sy, Fex, Fey, fb[9], ux, uy;
    stencil_v<v2x>(X2(c[1][2], c[2][2]), X2(c[2][1], c[3][1]), X2(c[1][0], c[2][0]), X2(c[0][1], c[1][1]),
                   X2(c[2][2], c[3][2]), X2(c[2][0], c[3][0]), X2(c[0][0], c[1][0]), X2(c[0][2], c[1][2]), Sx, Sy);
    const int mode = O::force_mode(kp);
    if (mode == 0) {
        Fex = v2x{kp.c2.Fx}, Fey = v2x{kp.c2.Fy};
    } else if (mode == 1) {  // Sec. 3.3: (rho - rho_g) g
        const v2x e = rho - v2x{kp.c2.rho_g};
        Fex = e * v2x{kp.c2.Fx}, Fey = e * v2x{kp.c2.Fy};
    } else if (kp.fext) {
        const int64_t n = (int64_t)kp.nx * kp.ny;
        Fex = X2(float(kp.fext[node_a]), float(kp.fext[node_b]));
        Fey = X2(float(kp.fext[n + node_a]), float(kp.fext[n + node_b]));
    } else {
        Fex = Fey = X2(0.f, 0.f);
    }
    collide_v<v2x, O>(kp, d, rho, psi, Sx, Sy, Fex, Fey, fb, ux, uy);

    // encode and store
    S *da = static_cast<S *>(kp.dst) + ka, *db = static_cast<S *>(kp.dst) + kb;
    if constexpr (!DEV) {
#pragma unroll
        for (int i = 0; i < 9; ++i, da += kp.plane, db += kp.plane) {
            if (sa) *da = fb[i].v.x;
            if (sb) *db = fb[i].v.y;
        }
    } else {
        if (has_ref) {
            if (sa) kp.ref_dst[ka] = rho.v.x;
            if (sb) kp.ref_dst[kb] = rho.v.y;
        }
        const uint32_t ha = sr_hash(ka >> 1, kp.sr_seed), hb = sr_hash(kb >> 1, kp.sr_seed);
        // a node's random bits are the half of its row pair's word that its column's parity names;
        // both columns are the same, so one conversion rounds the two rows
        const unsigned pick = (ka & 1u) ? 0x7632u : 0x5410u;
#pragma unroll
        for (int i = 0; i < 9; ++i, da += kp.plane, db += kp.plane) {
            const v2x wr = has_ref ? v2x{kp.c2.w[i]} * rho : v2x{kp.c2.dec[i]};
            const v2x s = (fb[i] - wr) * v2x{kp.c2.scale};
            uint32_t h;
            if (kp.sr) {
                h = SRound<S>::pack(s.v.x, s.v.y, __byte_perm(sr_bits(ha, i), sr_bits(hb, i), pick));
            } else {
                const S lo = Codec<S>::enc(s.v.x, 0.f, 1.f), hi = Codec<S>::enc(s.v.y, 0.f, 1.f);
                h = (uint32_t)*reinterpret_cast<const unsigned short *>(&lo) |
                    (uint32_t)*reinterpret_cast<const unsigned short *>(&hi) << 16;
            }
            if (sa) *da = SRound<S>::from_bits((unsigned short)(h & 0xffffu));
            if (sb) *db = SRound<S>::from_bits((unsigned short)(h >> 16));
        }
    }
}

template <class S, int GEOM, class O>
__global__ void __launch_bounds__(32 * (kTilePairs + 2), 5) k_tile2(KParams kp, int ahead)
{
    __shared__ float sm[2 * kTilePairs + 2][kTilePitch];
    grid_dependency_wait();
    allow_dependent_launch();
    const int rows = 2 * ((blockDim.x >> 5) - 2), x0 = blockIdx.x * kTileX, y0 = blockIdx.y * rows;
    if (x0 >= 2 && x0 + kTileX + 2 <= kp.nx && y0 >= 2 && y0 + rows + 2 <= kp.ny) tile2_block<S, GEOM, O, true>(kp, ahead, sm);
    else tile2_block<S, GEOM, O, false>(kp, ahead, sm);
}

// FP64: one node per thread.  Warps 0 .. n-1 own the tile's rows, two more the rows above and below
// it, one the columns beside it.
struct PlaneAt {
    const KParams &kp;
    __device__ __forceinline__ double operator()(int k, int x, int y) const { return load_pop<double>(kp, k, x, y); }
    __device__ __forceinline__ double at_k(int k, int64_t kk) const { return load_pop_at<double>(kp, k, kk); }
};
template <int GEOM>
__global__ void __launch_bounds__(32 * (kTileRows + 3), 2) k_tile1(KParams kp)
{
    __shared__ double sm[kTileRows + 2][kTilePitch];
    grid_dependency_wait();
    allow_dependent_launch();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = (blockDim.x >> 5) - 3;
    const int x0 = blockIdx.x * kTileX, y0 = blockIdx.y * rows;
    int x = x0 + lane, r = warp + 1, c = lane + 1;
    if (warp == rows) r = 0;
    else if (warp == rows + 1) r = rows + 1;
    else if (warp == rows + 2) {
        if (lane >= 2 * (rows + 2)) r = 0, c = 0, x = x0 - 1;  // more lanes than ring nodes: the first again
        else r = lane >> 1, c = (lane & 1) * (kTileX + 1), x = x0 - 1 + c;
    }
    const int y = y0 + r - 1;
    const Site s = site_of(kp, x, y);
    const int64_t node = (int64_t)s.y * kp.nx + s.x;
    const bool solid = GEOM && kp.solid != nullptr && kp.solid[node] != 0;
    const double psi_s = kp.cd.psi_s;
    double f[9], psi;
    if (!s.in) {
        psi = psi_s;
    } else if (solid) {
        psi = kp.wall_psi ? kp.wall_psi[node] : psi_s;
    } else {
        pull_node_nb<double>(kp, around(kp, s.x, s.y), s.x, s.y, PlaneAt{kp}, f, (double *)nullptr);
        psi = f64::psi_of(kp, f64::density(f));
    }
    sm[r][c] = psi;
    __syncthreads();
    if (warp >= rows || x >= kp.nx || y >= kp.ny) return;
    if (kp.psi_out != nullptr) static_cast<double *>(kp.psi_out)[node] = psi;
    if (solid) return;
    const double *q = &sm[r][c];
    double fb[9], Sx, Sy, Fex, Fey, ux, uy;
    f64::stencil_S([&](int i) { return q[ey_(i) * kTilePitch + ex_(i)]; }, Sx, Sy);
    external_force<double>(kp, node, f64::density(f), Fex, Fey);
    f64::collide(kp, f, psi, Sx, Sy, Fex, Fey, fb, ux, uy);
    store_node<double>(kp, x, y, fb, 0.0);
}

// Rows (units: pairs or rows) of a tile: of the heights from `most`/2 to `most`, the one whose fullest
// SM has the least to do, a block counting its units and its ring warps.
inline int tile_height(const KParams &kp, int most, int rows_per_unit, int ring_warps)
{
    const int64_t sms = kp.sm_count > 0 ? kp.sm_count : 148;
    const int64_t tx = (kp.nx + kTileX - 1) / kTileX;
    int best = most;
    int64_t least = 0;
    for (int h = most; 2 * h >= most; --h) {
        const int64_t blocks = tx * ((kp.ny + h * rows_per_unit - 1) / (h * rows_per_unit));
        const int64_t cost = (blocks + sms - 1) / sms * (h + ring_warps);
        if (h == most || cost < least) best = h, least = cost;
    }
    return best;
}

template <class S>
struct Tile {
    static cudaError_t link_bits(const KParams &kp, uint16_t *out, cudaStream_t st)
    {
        k_link_bits<<<dim3((kp.nx + 127) / 128, kp.ny), 128, 0, st>>>(kp, out);
        return cudaGetLastError();
    }
    static cudaError_t step(const KParams &kp, cudaStream_t st)
    {
        if constexpr (std::is_same<S, double>::value) {
            const int h = tile_height(kp, kTileRows, 1, 3);
            const dim3 grid((kp.nx + kTileX - 1) / kTileX, (kp.ny + h - 1) / h), block(32 * (h + 3));
            return kp.solid ? launch_dependent(k_tile1<1>, grid, block, 0, st, kp) : launch_dependent(k_tile1<0>, grid, block, 0, st, kp);
        } else {
            const int h = tile_height(kp, kTilePairs, 2, 2);
            const dim3 grid((kp.nx + kTileX - 1) / kTileX, (kp.ny + 2 * h - 1) / (2 * h)), block(32 * (h + 2));
            // rows between a tile and the one it prefetches: three blocks per SM further on, where the
            // two population buffers exceed the 129 MB L2 (below that the lines are in L2 anyway)
            const int sms = kp.sm_count > 0 ? kp.sm_count : 148;
            const int ahead = 2.0 * 9.0 * kp.plane * sizeof(S) > 120e6 ? (int)(3u * sms / grid.x + 1) * 2 * h : 0;
            KParams kq = kp;
            for (int i = 0; i < 9; ++i) kq.pull[i] = (i * kp.plane - ey_(i) * kp.pitch) * (int64_t)sizeof(S);
            if (kp.q || kp.wall_u) return launch_dependent(k_tile2<S, 2, RuntimeOpts>, grid, block, 0, st, kq, ahead);
            if (kp.solid) return launch_dependent(k_tile2<S, 1, RuntimeOpts>, grid, block, 0, st, kq, ahead);
            return launch_dependent(k_tile2<S, 0, RuntimeOpts>, grid, block, 0, st, kq, ahead);
        }
    }
};

}  // namespace lbm
