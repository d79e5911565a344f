// Kernel instantiations for __half population storage.
#include "k_adjoint.cuh"
#include "k_fused2.cuh"
#include "k_small.cuh"
#include "k_tile.cuh"
#include "k_twopass.cuh"

// staged kernel (k_fused2.cuh): consumer warps of 60 columns and ring depth
#ifndef LBM_FUSED2_NW
#define LBM_FUSED2_NW 4
#endif
#ifndef LBM_FUSED2_RING
#define LBM_FUSED2_RING 8  // 16-bit rows are half as large: 8 staged rows fit 4 CTAs per SM
#endif

namespace lbm {

Launchers launchers_f16()
{
    Launchers L{};
    L.psi_pass = &TwoPass<__half>::psi_pass;
    L.collide_pass = &TwoPass<__half>::collide_pass;
    L.fused_pass = &Fused2<__half, LBM_FUSED2_NW, LBM_FUSED2_RING>::launch;
    L.fused_tile_x = FusedLayout2<__half, LBM_FUSED2_NW, LBM_FUSED2_RING>::TX;
    L.tile_pass = &Tile<__half>::step;
    L.small_ctas = &Small<__half>::ctas;
    L.small_steps = &Small<__half>::steps;
    L.link_bits = &Tile<__half>::link_bits;
    L.init = &TwoPass<__half>::init;
    L.moments = &Tile<__half>::moments;
    L.diag = &Tile<__half>::diag;
    L.diag_rows = &Tile<__half>::diag_rows;
    L.get_state = &TwoPass<__half>::get_state;
    L.set_state = &TwoPass<__half>::set_state;
    L.adj_step = &Adjoint<__half>::step;
    L.adj_lambda = &Adjoint<__half>::lambda;
    L.objective = &Adjoint<__half>::objective;
    L.adj_blocks = &Adjoint<__half>::blocks;
    L.adj_reduce = &Adjoint<__half>::reduce;
    L.fused_align = FusedGeom<__half>::HX;
    L.fused_geometry = 1;
    return L;
}

}  // namespace lbm
