// One-pass step on tiles of 32 columns: psi of the tile and of the ring of nodes around it goes
// through shared memory, so one launch does what the psi pass and the collide pass do in two.
//
// FP32 arithmetic (k_tile2; FP32, FP16 and BF16 storage): a thread owns two nodes of one column,
// rows y and y + 1, and evaluates them as one packed pair.  A vertical pair keeps every access of a
// warp 32 consecutive elements wide at any lattice width, alignment and storage type, and a pair
// needs no alignment of nx; the packed instructions halve the arithmetic instructions of the
// one-node passes.  The packed products are written as multiply-adds with -0 (v2x): the assembler
// fuses a packed product into a following packed sum, which rounds once where the one-node
// evaluation rounds twice; with them every node's result is the two-pass step's, bit for bit.  Where the
// context takes the step of LBM_KERNEL_FUSED (KParams::packed) the products are plain packed ones and 16-bit
// storage encodes as the staged kernel does (v2): the state is then the staged kernel's, bit for bit,
// whichever of the two kernels a size gets.
// FP64 (k_tile1): one node per thread, the two-pass step's own functions, the same bits.
//
// A tile of n pairs (rows) has n warps for them; one more warp pulls the rows above and below the
// tile and one the columns beside it (FP64: two and one), for psi only.  The tile's height is
// chosen per launch (tile_height) so that the last wave of blocks is nearly full.
//
// What bounds it (FP32): small lattices the latency of one block's chain, mid-size ones instruction
// issue (546 a pair of rows and 32 columns, ring included, 557 with exact products, FP16 787; the two-pass kernels
// 1840), from 2048^2 on HBM: 4096^2 183 us, 99 % of the measured copy rate at 72 B a node. Four pairs and five blocks per SM (64
// registers) against two blocks of eight pairs: 512 x 4096 46 -> 36 us; the L2 prefetch 70 -> 59 at 2048^2;
// the instantiation without edge tests (INNER) 59 -> 52, FP16 81 -> 67.
//
// lbm_get_moments and lbm_get_diagnostics run the same tiles (k_read2, k_read1): one launch where a psi
// pass and a node pass read the populations twice (8192^2 moments 2.04 -> 0.71 ms, bound by its 60 B a
// node), and block sums into rows that one reduction adds where every block put ten atomics on the
// same addresses (256 x 2048 diagnostics 123 -> 23 us).
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
// two floats as a pair of either rounding (v2, v2x)
template <class V> __device__ __forceinline__ V pair_of(float a, float b) { return V{make_float2(a, b)}; }

// ------------------------------------------------------------- block sums --------
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Warp sum of one value per lane as a compensated FP32 pair (hi, lo) in lane 0: Knuth's TwoSum at
// every shuffle level, about 2^-48 relative.
__device__ __forceinline__ void two_sum(float &hi, float &lo, float x, float xlo)
{
    const float sum = hi + x, z = sum - hi;
    lo += xlo + ((hi - (sum - z)) + (x - z));
    hi = sum;
}
__device__ __forceinline__ void warp_sum_pair(float &hi, float &lo)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        two_sum(hi, lo, __shfl_down_sync(0xffffffffu, hi, o), __shfl_down_sync(0xffffffffu, lo, o));
}

// Sums of the `n` quantities v[k][0 .. count) in shared memory (all threads past a barrier) but those
// in `skip` (known to be zero), handed to put(k, sum) by one lane: a warp of `warps` sums one quantity at
// a time, each lane its share and then the lanes, compensated in FP32 arithmetic (FP64 work stays out
// of it: GB300's FP64 pipe is narrow).
template <class R, class Put>
__device__ __forceinline__ void block_add(const R *v, int pitch, int n, int count, int warps, unsigned skip, const Put &put)
{
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < n; k += warps) {
        if ((skip >> k) & 1u) continue;
        double t;
        if constexpr (sizeof(R) == 8) {
            double s = 0.0;
            for (int q = lane; q < count; q += 32) s += v[k * pitch + q];
            t = warp_sum(s);
        } else {
            float hi = 0.f, lo = 0.f;
            for (int q = lane; q < count; q += 32) two_sum(hi, lo, v[k * pitch + q], 0.f);
            warp_sum_pair(hi, lo);
            t = double(hi) + double(lo);
        }
        if (lane == 0) put(k, t);
    }
}

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
// What a tile's kernel leaves: the next state; rho and u of the state read (lbm_get_moments); or the
// block's sums for lbm_get_diagnostics, one row of kDiagSlots doubles (kDiagSums sums, the largest |u|,
// the number of nodes whose density or velocity is not finite).
enum TileMode { TILE_STEP = 0, TILE_MOMENTS = 1, TILE_DIAG = 2 };
constexpr int kDiagSums = 9, kDiagSlots = 11;
struct TileOut {
    double *rho, *ux, *uy;  // [ny*nx], each may be null
    double *part;           // [blocks][kDiagSlots]
};

// A float as a double without the conversion instruction, which runs on the narrow FP64 pipe.
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
    if (e - 0x00800000u >= 0x7f000000u) return double(x);  // zero, subnormal, infinite or NaN
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// One block of a step.  GEOM: 0 no solid nodes; 1 solid nodes with half-way links; 2 also interpolated
// or moving walls; 3 any of these, told apart at run time.  INNER: the tile lies inside the lattice and no node of it or its ring pulls across
// an edge, so every address is the node's own plus a constant of the launch (KParams::pull).
struct Tile2Shared {
    float psi[2 * kTilePairs + 2][kTilePitch];
};
struct Tile2SharedDiag : Tile2Shared {
    float v[kDiagSums][64 * kTilePairs];
    float umax[kTilePairs];
    int bad[kTilePairs];
};
template <class S, int GEOM, class O, int MODE, bool INNER, class V, class Shared>
__device__ __forceinline__ void tile2_block(const KParams &kp, int ahead, const TileOut &out, Shared &sh)
{
    auto &sm = sh.psi;
    constexpr bool DEV = IsDev<S>::value, PACKED = std::is_same<V, v2>::value;
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
    Site a{ax, ay, true}, b{bx, by, true};
    if constexpr (!INNER) a = site_of(kp, ax, ay), b = site_of(kp, bx, by);
    const uint32_t node_a = (uint32_t)a.y * (uint32_t)kp.nx + a.x, node_b = (uint32_t)b.y * (uint32_t)kp.nx + b.x;
    const uint32_t ka = (uint32_t)a.y * (uint32_t)kp.pitch + a.x, kb = (uint32_t)b.y * (uint32_t)kp.pitch + b.x;
    unsigned wa = 0, wb = 0;  // wall bits
    const bool masked = GEOM == 3 ? kp.links != nullptr : GEOM != 0;
    if (masked) wa = kp.links[node_a], wb = kp.links[node_b];

    // Up to here nothing that a step writes was read: the launch waits for the one before it now.
    if constexpr (MODE == TILE_STEP) {
        grid_dependency_wait();
        allow_dependent_launch();
    }
    // A warp whose nodes are all solid has nothing to pull: psi is the walls'.  Only where solid nodes are
    // many (KParams::skip_solid, an eighth), since the others' pulls then wait for the wall bits.  Step without
    // / with it at 1024^2 (us): a disc of 3, 9, 12.5 and 40 % of the nodes 15.8 / 15.6, 15.4 / 14.8, 15.2 /
    // 14.3 and 13.8 / 11.9 (FP16 18.0 / 17.9, 17.8 / 17.4, 17.7 / 17.0, 16.5 / 14.3); grains of 24^2 nodes
    // within 1 % either way at any share; solid bands (0.1 %) the same: the line is on the safe side, nothing
    // was slower with it.
    const bool still = masked && kp.skip_solid && __all_sync(0xffffffffu, (wa & 1u) && (wb & 1u));
    if (ahead > 0 && warp < np && lane < (masked ? 20 : 18)) {
        // the lines of the tile that a block of the next wave will read (rows y and y + 1, columns x0 ..
        // x0 + 31): the nine planes, and the wall bits
        const int i = lane >> 1, y = ay + (lane & 1) + ahead;
        if (y < kp.ny) {
            const void *p = i < 9 ? (const void *)(static_cast<const S *>(kp.src) + (i * kp.plane + (int64_t)y * kp.pitch + x0))
                                  : (const void *)(kp.links + ((int64_t)y * kp.nx + x0));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
        }
    }
    V f[9], d[9], rho = pair_of<V>(1.f, 1.f), psi = pair_of<V>(0.f, 0.f);
    V momx = pair_of<V>(0.f, 0.f), momy = momx;  // momentum handed to the walls (diagnostics)
    if (!still) {
        // pull, Eq. (lbe.str)
        const S *src = static_cast<const S *>(kp.src);
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
            if (!masked) wa = edge_walls(ia), wb = edge_walls(ib);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const S *p = src + i * kp.plane;
                va[i] = p[na.from(i)], vb[i] = p[nb.from(i)];
                if (has_ref) refa[i] = kp.ref_src[na.from(i)], refb[i] = kp.ref_src[nb.from(i)];
            }
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            V wr = pair_of<V>(0.f, 0.f);
            if (DEV) wr = has_ref ? V{kp.c2.w[i]} * pair_of<V>(refa[i], refb[i]) : V{kp.c2.dec[i]};
            f[i] = pair_of<V>(Raw<S>::f(va[i], wr.v.x, kp), Raw<S>::f(vb[i], wr.v.y, kp));
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
                    if constexpr (GEOM >= 2) if (GEOM == 2 || kp.link != nullptr) {
                        // interpolated or moving wall: link fraction and moving-wall coefficient
                        const float2 lk = kp.link[(int64_t)(i - 1) * kp.plane + k];
                        // the coefficient's form: KParams::link
                        const bool whole = MODE == TILE_STEP ? PACKED : kp.packed != 0;
                        float mw = 0.f;
                        if (lk.y != 0.f) {
                            if (!summed) {
#pragma unroll
                                for (int n = 0; n < 9; ++n) rho_w += own(n);
                                summed = true;
                            }
                            mw = whole ? lk.y * rho_w : 2.f * w_<float>(o) * rho_w * lk.y * 3.f;
                        }
                        const float q = lk.x;
                        if (q < 0.5f) {
                            // fbar_o of the second node x + e_i (fluid: the record's q is 1/2 otherwise), which
                            // is what the pull of population o brought here
                            const float f2 = e ? f[o].v.y : f[o].v.x;
                            g = near_link<DEV>(q, fo, f2, mw);
                        } else if (q == 0.5f) {
                            g = fo + mw;
                        } else {
                            g = fo / (2.f * q) + (2.f * q - 1.f) / (2.f * q) * own(i) + mw / (2.f * q);
                        }
                    }
                    if (e) f[i].v.y = g;
                    else f[i].v.x = g;
                    if constexpr (MODE == TILE_DIAG) {
                        float &mx = e ? momx.v.y : momx.v.x, &my = e ? momy.v.y : momy.v.x;
                        mx += -float(ex_(i)) * (fo + g), my += -float(ey_(i)) * (fo + g);
                    }
                }
            }
        }
        to_dev(f, d);
        rho = density_dev(d);
        psi = psi_v<V>(kp, rho);
    } else if constexpr (MODE == TILE_DIAG) {
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = pair_of<V>(0.f, 0.f);
    }
    if (GEOM) {
        if (wa & 1u) psi.v.x = kp.wall_psi_f ? kp.wall_psi_f[node_a] : kp.cf.psi_s, rho.v.x = 1.f;
        if (wb & 1u) psi.v.y = kp.wall_psi_f ? kp.wall_psi_f[node_b] : kp.cf.psi_s, rho.v.y = 1.f;
    }
    if (!INNER && !a.in) psi.v.x = kp.cf.psi_s;
    if (!INNER && !b.in) psi.v.y = kp.cf.psi_s;
    sm[ra][ca] = psi.v.x;
    sm[rb][cb] = psi.v.y;
    __syncthreads();
    if constexpr (MODE != TILE_DIAG)
        if (warp >= np) return;
    const bool la = INNER || (ax < kp.nx && ay < kp.ny), lb = INNER || (ax < kp.nx && by < kp.ny);
    if constexpr (MODE != TILE_DIAG)
        if (!la) return;
    if (MODE == TILE_STEP && kp.psi_out != nullptr) {
        float *out = static_cast<float *>(kp.psi_out);
        out[node_a] = psi.v.x;
        if (lb) out[node_b] = psi.v.y;
    }
    const bool sa = la && !(GEOM && (wa & 1u)), sb = lb && !(GEOM && (wb & 1u));
    if constexpr (MODE == TILE_STEP)
        if (!sa && !sb) return;

    // S of Eq. (fint) from the four psi rows around the pair
    const float *q = &sm[MODE == TILE_DIAG ? min(2 * warp, 2 * kTilePairs - 2) : 2 * warp][lane];
    float c[4][3];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) c[r][k] = q[r * kTilePitch + k];
    V Sx, Sy, Fex, Fey, fb[9], ux, uy;
    stencil_v<V>(pair_of<V>(c[1][2], c[2][2]), pair_of<V>(c[2][1], c[3][1]), pair_of<V>(c[1][0], c[2][0]), pair_of<V>(c[0][1], c[1][1]),
                   pair_of<V>(c[2][2], c[3][2]), pair_of<V>(c[2][0], c[3][0]), pair_of<V>(c[0][0], c[1][0]), pair_of<V>(c[0][2], c[1][2]), Sx, Sy);
    const int mode = O::force_mode(kp);
    if (mode == 0) {
        Fex = V{kp.c2.Fx}, Fey = V{kp.c2.Fy};
    } else if (mode == 1) {  // Sec. 3.3: (rho - rho_g) g
        const V e = rho - V{kp.c2.rho_g};
        Fex = e * V{kp.c2.Fx}, Fey = e * V{kp.c2.Fy};
    } else if (kp.fext_f) {
        const int64_t n = (int64_t)kp.nx * kp.ny;
        Fex = pair_of<V>(kp.fext_f[node_a], kp.fext_f[node_b]);
        Fey = pair_of<V>(kp.fext_f[n + node_a], kp.fext_f[n + node_b]);
    } else {
        Fex = Fey = pair_of<V>(0.f, 0.f);
    }
    collide_v<V, O>(kp, d, rho, psi, Sx, Sy, Fex, Fey, fb, ux, uy);

    if constexpr (MODE == TILE_MOMENTS) {
        // solid nodes report their virtual density at rest
        auto put = [&](bool fluid, uint32_t n, float r, float u, float v) {
            if (out.rho) out.rho[n] = fluid ? widen(r) : (kp.wall_rho ? kp.wall_rho[n] : kp.rho_s);
            if (out.ux) out.ux[n] = fluid ? widen(u) : 0.0;
            if (out.uy) out.uy[n] = fluid ? widen(v) : 0.0;
        };
        put(sa, node_a, rho.v.x, ux.v.x, uy.v.x);
        if (lb) put(sb, node_b, rho.v.y, ux.v.y, uy.v.y);
        return;
    }
    if constexpr (MODE == TILE_DIAG) {
        const V jx = ((f[1] - f[3]) + (f[5] - f[6])) + (f[8] - f[7]), jy = ((f[2] - f[4]) + (f[5] + f[6])) - (f[7] + f[8]);
        const V nGpsi = V{kp.c2.m_G} * psi, Fx = vfma(nGpsi, Sx, Fex), Fy = vfma(nGpsi, Sy, Fey);
        const float half_lg = float(0.5 * (kp.rho_l + kp.rho_g));
        float um = 0.f;
        int bad = 0;
        if (warp < np) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                auto get = [&](V a) { return e ? a.v.y : a.v.x; };
                const bool on = e ? sb : sa;
                const float r = get(rho), u = get(ux), v = get(uy);
                const bool liquid = on && r > half_lg;
                const float t[kDiagSums] = {r, get(jx), get(jy), get(Fx), get(Fy), get(momx), get(momy), r * v, r};
#pragma unroll
                for (int k = 0; k < kDiagSums; ++k) sh.v[k][threadIdx.x + 32 * kTilePairs * e] = (k < 7 ? on : liquid) ? t[k] : 0.f;
                if (on) {
                    const float w = sqrtf(u * u + v * v);
                    um = fmaxf(um, w);
                    if (!isfinite(r) || !isfinite(w)) bad += 1;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                um = fmaxf(um, __shfl_down_sync(0xffffffffu, um, o));
                bad += __shfl_down_sync(0xffffffffu, bad, o);
            }
            if (lane == 0) sh.umax[warp] = um, sh.bad[warp] = bad;
        }
        __syncthreads();
        double *row = out.part + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kDiagSlots;
        block_add<float>(&sh.v[0][0], 64 * kTilePairs, kDiagSums, 64 * kTilePairs, kTilePairs + 2, 0u,
                         [&](int k, double t) { row[k] = t; });
        if (threadIdx.x == 0) {
            for (int w = 1; w < kTilePairs; ++w) um = fmaxf(um, sh.umax[w]), bad += sh.bad[w];
            row[kDiagSums] = double(um);
            row[kDiagSums + 1] = double(bad);
        }
        return;
    }

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
            const V wr = has_ref ? V{kp.c2.w[i]} * rho : V{kp.c2.dec[i]};
            V s;
            if constexpr (PACKED) s = vfma(fb[i], V{kp.c2.scale}, has_ref ? V{kp.c2.m_scale} * wr : V{kp.c2.enc[i]});
            else s = (fb[i] - wr) * V{kp.c2.scale};
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

__device__ __forceinline__ bool tile_inner(const KParams &kp, int rows)
{
    const int x0 = blockIdx.x * kTileX, y0 = blockIdx.y * rows;
    return x0 >= 2 && x0 + kTileX + 2 <= kp.nx && y0 >= 2 && y0 + rows + 2 <= kp.ny;
}
template <class S, int GEOM, class O, class V>
__global__ void __launch_bounds__(32 * (kTilePairs + 2), 5) k_tile2(KParams kp, int ahead)
{
    __shared__ Tile2Shared sh;
    const TileOut none{};
    if (tile_inner(kp, 2 * ((blockDim.x >> 5) - 2))) tile2_block<S, GEOM, O, TILE_STEP, true, V>(kp, ahead, none, sh);
    else tile2_block<S, GEOM, O, TILE_STEP, false, V>(kp, ahead, none, sh);
}
// The readings of a state, on tiles of kTilePairs pairs (the whole block's sums want a full one).
template <class S, int MODE>
__global__ void __launch_bounds__(32 * (kTilePairs + 2), MODE == TILE_MOMENTS ? 5 : 4) k_read2(KParams kp, int ahead, TileOut out)
{
    __shared__ typename std::conditional<MODE == TILE_DIAG, Tile2SharedDiag, Tile2Shared>::type sh;
    if (tile_inner(kp, 2 * kTilePairs)) tile2_block<S, 3, RuntimeOpts, MODE, true, v2x>(kp, ahead, out, sh);
    else tile2_block<S, 3, RuntimeOpts, MODE, false, v2x>(kp, ahead, out, sh);
}

// Column sums of the blocks' rows (kDiagSlots columns; the largest |u| by maximum), one block per column
// in a fixed order.
template <class S>
__global__ void __launch_bounds__(256) k_diag_reduce(const double *part, int64_t blocks, double *out)
{
    __shared__ double red[8];
    const int k = blockIdx.x;
    const bool top = k == kDiagSums;
    double s = 0.0;
    for (int64_t b = threadIdx.x; b < blocks; b += blockDim.x) {
        const double x = part[b * kDiagSlots + k];
        s = top ? fmax(s, x) : s + x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double x = __shfl_down_sync(0xffffffffu, s, o);
        s = top ? fmax(s, x) : s + x;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) s = top ? fmax(s, red[q]) : s + red[q];
        out[k] = s;
    }
}

// FP64: one node per thread.  Warps 0 .. n-1 own the tile's rows, two more the rows above and below
// it, one the columns beside it.
struct PlaneAt {
    static constexpr bool DEV = false;
    const KParams &kp;
    __device__ __forceinline__ double operator()(int k, int x, int y) const { return load_pop<double>(kp, k, x, y); }
    __device__ __forceinline__ double at_k(int k, int64_t kk) const { return load_pop_at<double>(kp, k, kk); }
};
struct Tile1Shared {
    double psi[kTileRows + 2][kTilePitch];
};
struct Tile1SharedDiag : Tile1Shared {
    double v[kDiagSums][32 * kTileRows];
    double umax[kTileRows];
    int bad[kTileRows];
};
template <int MODE, class Shared>
__device__ __forceinline__ void tile1_block(const KParams &kp, const TileOut &out, Shared &sh)
{
    auto &sm = sh.psi;
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
    const bool solid = kp.solid != nullptr && kp.solid[node] != 0;
    const double psi_s = kp.cd.psi_s;
    double f[9], psi, mom[2] = {0.0, 0.0};
    if (!s.in) {
        psi = psi_s;
    } else if (solid) {
        psi = kp.wall_psi ? kp.wall_psi[node] : psi_s;
    } else {
        pull_node_nb<double>(kp, around(kp, s.x, s.y), s.x, s.y, PlaneAt{kp}, f, MODE == TILE_DIAG ? mom : (double *)nullptr);
        psi = f64::psi_of(kp, f64::density(f));
    }
    sm[r][c] = psi;
    __syncthreads();
    const bool mine = warp < rows && x < kp.nx && y < kp.ny;
    if constexpr (MODE != TILE_DIAG) {
        if (!mine) return;
        if (MODE == TILE_STEP && kp.psi_out != nullptr) static_cast<double *>(kp.psi_out)[node] = psi;
        if (solid) {
            if constexpr (MODE == TILE_MOMENTS) {
                if (out.rho) out.rho[node] = kp.wall_rho ? kp.wall_rho[node] : kp.rho_s;
                if (out.ux) out.ux[node] = 0.0;
                if (out.uy) out.uy[node] = 0.0;
            }
            return;
        }
    }
    double fb[9], Sx, Sy, Fex, Fey, ux = 0.0, uy = 0.0, rho = 0.0;
    if (mine && !solid) {
        const double *q = &sm[r][c];
        f64::stencil_S([&](int i) { return q[ey_(i) * kTilePitch + ex_(i)]; }, Sx, Sy);
        rho = f64::density(f);
        external_force<double>(kp, node, rho, Fex, Fey);
        f64::collide(kp, f, psi, Sx, Sy, Fex, Fey, fb, ux, uy);
    }
    if constexpr (MODE == TILE_STEP) {
        store_node<double>(kp, x, y, fb, 0.0);
    } else if constexpr (MODE == TILE_MOMENTS) {
        if (out.rho) out.rho[node] = rho;
        if (out.ux) out.ux[node] = ux;
        if (out.uy) out.uy[node] = uy;
    } else {
        double um = 0.0;
        int bad = 0;
        if (warp < rows) {
            const bool on = mine && !solid, liquid = on && rho > 0.5 * (kp.rho_l + kp.rho_g);
            if (on) {
                const double G = kp.cd.G;
                const double t[kDiagSums] = {rho,
                                             ((f[1] - f[3]) + (f[5] - f[6])) + (f[8] - f[7]),
                                             ((f[2] - f[4]) + (f[5] + f[6])) - (f[7] + f[8]),
                                             -G * psi * Sx + Fex,
                                             -G * psi * Sy + Fey,
                                             mom[0],
                                             mom[1],
                                             liquid ? rho * uy : 0.0,
                                             liquid ? rho : 0.0};
#pragma unroll
                for (int k = 0; k < kDiagSums; ++k) sh.v[k][threadIdx.x] = t[k];
                um = sqrt(ux * ux + uy * uy);
                bad = !isfinite(rho) || !isfinite(um);
                if (!(um > 0.0)) um = 0.0;  // (NaN counts as bad)
            } else {
#pragma unroll
                for (int k = 0; k < kDiagSums; ++k) sh.v[k][threadIdx.x] = 0.0;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                um = fmax(um, __shfl_down_sync(0xffffffffu, um, o));
                bad += __shfl_down_sync(0xffffffffu, bad, o);
            }
            if (lane == 0) sh.umax[warp] = um, sh.bad[warp] = bad;
        }
        __syncthreads();
        double *row = out.part + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kDiagSlots;
        block_add<double>(&sh.v[0][0], 32 * kTileRows, kDiagSums, 32 * kTileRows, kTileRows + 3, 0u,
                          [&](int k, double t) { row[k] = t; });
        if (threadIdx.x == 0) {
            for (int w = 1; w < kTileRows; ++w) um = fmax(um, sh.umax[w]), bad += sh.bad[w];
            row[kDiagSums] = um;
            row[kDiagSums + 1] = double(bad);
        }
    }
}
template <class S>
__global__ void __launch_bounds__(32 * (kTileRows + 3), 2) k_tile1(KParams kp)
{
    __shared__ Tile1Shared sh;
    grid_dependency_wait();
    allow_dependent_launch();
    tile1_block<TILE_STEP>(kp, TileOut{}, sh);
}
template <class S, int MODE>
__global__ void __launch_bounds__(32 * (kTileRows + 3), 1) k_read1(KParams kp, TileOut out)
{
    __shared__ typename std::conditional<MODE == TILE_DIAG, Tile1SharedDiag, Tile1Shared>::type sh;
    tile1_block<MODE>(kp, out, sh);
}

// Options fixed at compile time: the force law, one or two relaxation times and, for 16-bit storage, the
// reference plane.  Each costs a block a branch that the schedule does not cross and a value that is live
// through it, in a kernel that is short of registers (64): 1024^2 14.4 -> 13.7 us, 512 x 4096 30.1 -> 29.3,
// FP16 (exact products) 37.7 -> 35.4.  The EOS and the scheme stay run-time options (fixed as well: within 1 %).
template <int VT, int REF, class F>
inline cudaError_t with_force(const KParams &kp, const F &f)
{
    return kp.force_mode == 0 ? f(Opts<-1, VT, 0, REF>()) : kp.force_mode == 1 ? f(Opts<-1, VT, 1, REF>()) : f(Opts<-1, VT, 2, REF>());
}
template <bool DEV, class F>
inline cudaError_t with_options(const KParams &kp, const F &f)
{
    if (DEV && kp.per_node_ref) return kp.var_tau ? with_force<1, DEV ? 1 : 0>(kp, f) : with_force<0, DEV ? 1 : 0>(kp, f);
    return kp.var_tau ? with_force<1, 0>(kp, f) : with_force<0, 0>(kp, f);
}

// The packed rounding fixes fewer of them: the assembler fuses a packed product into a sum where both stand in one
// block of the code, so the relaxation and the scheme stay branches exactly where the staged kernel
// (Fused2::launch) has them.  512 x 4096 with walls, FP16: 36.6 us with all at run time, 34.7 here, 35.4 with
// exact products and the options above (FP32 29.3 / 28.8 with exact products / here); bands 2048^2, two
// relaxation times, FP16 72.6 / 70.6 / 80.3 (FP32 60.9 / 57.5); 4096^2 FP32 185.0 / 182.7.
template <bool DEV, class F>
inline cudaError_t with_packed_options(const KParams &kp, bool plain, const F &f)
{
    constexpr int ON = DEV ? 1 : 0;  // (the reference plane, where there can be one)
    const bool ref = DEV && kp.per_node_ref;
    if (plain && kp.force_mode == 0 && !kp.var_tau) {
        if (ref) return kp.improved ? f(Opts<1, 0, 0, ON>()) : f(Opts<0, 0, 0, ON>());
        return kp.improved ? f(Opts<1, 0, 0, 0>()) : f(Opts<0, 0, 0, 0>());
    }
    if (DEV && !ref) return f(Opts<-1, -1, -1, 0>());
    return kp.force_mode == 0 ? f(Opts<-1, -1, 0, ON>()) : kp.force_mode == 1 ? f(Opts<-1, -1, 1, ON>()) : f(Opts<-1, -1, 2, ON>());
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
    static constexpr bool F64 = std::is_same<S, double>::value;
    static constexpr int READ_ROWS = F64 ? kTileRows : 2 * kTilePairs;
    static KParams with_pull(const KParams &kp)
    {
        KParams kq = kp;
        for (int i = 0; i < 9; ++i) kq.pull[i] = (i * kp.plane - ey_(i) * kp.pitch) * (int64_t)sizeof(S);
        return kq;
    }
    // rows between a tile and the one it prefetches: three blocks per SM further on, where the two
    // population buffers exceed the 129 MB L2 (below that the lines are in L2 anyway)
    static int ahead_of(const KParams &kp, dim3 grid, int rows)
    {
        const unsigned sms = kp.sm_count > 0 ? kp.sm_count : 148;
        return 2.0 * 9.0 * kp.plane * sizeof(S) > 120e6 ? (int)(3u * sms / grid.x + 1) * rows : 0;
    }
    static dim3 read_grid(const KParams &kp) { return dim3((kp.nx + kTileX - 1) / kTileX, (kp.ny + READ_ROWS - 1) / READ_ROWS); }
    template <int MODE>
    static cudaError_t read(const KParams &kp, const TileOut &out, cudaStream_t st)
    {
        if constexpr (F64) k_read1<S, MODE><<<read_grid(kp), 32 * (kTileRows + 3), 0, st>>>(kp, out);
        else k_read2<S, MODE><<<read_grid(kp), 32 * (kTilePairs + 2), 0, st>>>(with_pull(kp), ahead_of(kp, read_grid(kp), READ_ROWS), out);
        return cudaGetLastError();
    }
    // rho and u = (j + F/2)/rho of the state kp.src, as the step computes them
    static cudaError_t moments(const KParams &kp, double *rho, double *ux, double *uy, cudaStream_t st)
    {
        return read<TILE_MOMENTS>(kp, TileOut{rho, ux, uy, nullptr}, st);
    }
    static int64_t diag_rows(const KParams &kp) { return (int64_t)read_grid(kp).x * read_grid(kp).y; }
    static cudaError_t diag(const KParams &kp, double *part, double *out, cudaStream_t st)
    {
        cudaError_t e = read<TILE_DIAG>(kp, TileOut{nullptr, nullptr, nullptr, part}, st);
        if (e != cudaSuccess) return e;
        k_diag_reduce<S><<<kDiagSlots, 256, 0, st>>>(part, diag_rows(kp), out);
        return cudaGetLastError();
    }
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
            return launch_dependent(k_tile1<S>, grid, block, 0, st, kp);
        } else {
            const int h = tile_height(kp, kTilePairs, 2, 2);
            const dim3 grid((kp.nx + kTileX - 1) / kTileX, (kp.ny + 2 * h - 1) / (2 * h)), block(32 * (h + 2));
            const int ahead = ahead_of(kp, grid, 2 * h);
            const KParams kq = with_pull(kp);
            auto go = [&](auto kernel) { return launch_dependent(kernel, grid, block, 0, st, kq, ahead); };
            const bool links = kp.q || kp.wall_u, solid = kp.solid != nullptr;
            constexpr bool DEV = IsDev<S>::value;
            if (kp.packed) {
                const bool plain = !links && !solid && kp.periodic_x && kp.periodic_y;
                return with_packed_options<DEV>(kp, plain, [&](auto o) {
                    typedef decltype(o) O;
                    return links ? go(k_tile2<S, 2, O, v2>) : solid ? go(k_tile2<S, 1, O, v2>) : go(k_tile2<S, 0, O, v2>);
                });
            }
            return with_options<DEV>(kp, [&](auto o) {
                typedef decltype(o) O;
                return links ? go(k_tile2<S, 2, O, v2x>) : solid ? go(k_tile2<S, 1, O, v2x>) : go(k_tile2<S, 0, O, v2x>);
            });
        }
    }
};

}  // namespace lbm
