// Kernel instantiations for double population storage.
#include "k_adjoint.cuh"
#include "k_small.cuh"
#include "k_tile.cuh"
#include "k_twopass.cuh"

namespace lbm {

Launchers launchers_f64()
{
    Launchers L{};
    L.psi_pass = &TwoPass<double>::psi_pass;
    L.collide_pass = &TwoPass<double>::collide_pass;
    L.tile_pass = &Tile<double>::step;
    L.small_ctas = &Small<double>::ctas;
    L.small_steps = &Small<double>::steps;
    L.link_bits = &Tile<double>::link_bits;
    L.init = &TwoPass<double>::init;
    L.moments = &Tile<double>::moments;
    L.diag = &Tile<double>::diag;
    L.diag_rows = &Tile<double>::diag_rows;
    L.get_state = &TwoPass<double>::get_state;
    L.set_state = &TwoPass<double>::set_state;
    L.adj_step = &Adjoint<double>::step;
    L.adj_lambda = &Adjoint<double>::lambda;
    L.objective = &Adjoint<double>::objective;
    L.adj_blocks = &Adjoint<double>::blocks;
    L.adj_reduce = &Adjoint<double>::reduce;
    L.fused_tile_x = 240;
    L.fused_align = 2;
    return L;
}

}  // namespace lbm
