// Kernel instantiations for float population storage.
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
#define LBM_FUSED2_RING 4
#endif

namespace lbm {

Launchers launchers_f32()
{
    Launchers L{};
    L.psi_pass = &TwoPass<float>::psi_pass;
    L.collide_pass = &TwoPass<float>::collide_pass;
    L.fused_pass = &Fused2<float, LBM_FUSED2_NW, LBM_FUSED2_RING>::launch;
    L.fused_tile_x = FusedLayout2<float, LBM_FUSED2_NW, LBM_FUSED2_RING>::TX;
    L.tile_pass = &Tile<float>::step;
    L.small_ctas = &Small<float>::ctas;
    L.small_steps = &Small<float>::steps;
    L.link_bits = &Tile<float>::link_bits;
    L.init = &TwoPass<float>::init;
    L.moments = &Tile<float>::moments;
    L.diag = &Tile<float>::diag;
    L.diag_rows = &Tile<float>::diag_rows;
    L.get_state = &TwoPass<float>::get_state;
    L.set_state = &TwoPass<float>::set_state;
    L.adj_step = &Adjoint<float>::step;
    L.adj_lambda = &Adjoint<float>::lambda;
    L.objective = &Adjoint<float>::objective;
    L.adj_blocks = &Adjoint<float>::blocks;
    L.adj_reduce = &Adjoint<float>::reduce;
    L.fused_align = FusedGeom<float>::HX;
    L.fused_geometry = 1;
    return L;
}

}  // namespace lbm
