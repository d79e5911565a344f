// Kernel instantiations for __nv_bfloat16 population storage.
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

Launchers launchers_bf16()
{
    Launchers L{};
    L.psi_pass = &TwoPass<__nv_bfloat16>::psi_pass;
    L.collide_pass = &TwoPass<__nv_bfloat16>::collide_pass;
    L.fused_pass = &Fused2<__nv_bfloat16, LBM_FUSED2_NW, LBM_FUSED2_RING>::launch;
    L.fused_tile_x = FusedLayout2<__nv_bfloat16, LBM_FUSED2_NW, LBM_FUSED2_RING>::TX;
    L.tile_pass = &Tile<__nv_bfloat16>::step;
    L.small_ctas = &Small<__nv_bfloat16>::ctas;
    L.small_steps = &Small<__nv_bfloat16>::steps;
    L.link_bits = &Tile<__nv_bfloat16>::link_bits;
    L.init = &TwoPass<__nv_bfloat16>::init;
    L.moments = &Tile<__nv_bfloat16>::moments;
    L.diag = &Tile<__nv_bfloat16>::diag;
    L.diag_rows = &Tile<__nv_bfloat16>::diag_rows;
    L.get_state = &TwoPass<__nv_bfloat16>::get_state;
    L.set_state = &TwoPass<__nv_bfloat16>::set_state;
    L.adj_step = &Adjoint<__nv_bfloat16>::step;
    L.adj_lambda = &Adjoint<__nv_bfloat16>::lambda;
    L.objective = &Adjoint<__nv_bfloat16>::objective;
    L.adj_blocks = &Adjoint<__nv_bfloat16>::blocks;
    L.adj_reduce = &Adjoint<__nv_bfloat16>::reduce;
    L.fused_align = FusedGeom<__nv_bfloat16>::HX;
    L.fused_geometry = 1;
    return L;
}

}  // namespace lbm
