// labs_walk8f.cu -- walk kernels with four walkers per warp for few walkers (every neighbour's HT slot
// looked up at a step's start): walk_lockstep in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, 1) walk_quad_few_kernel(KParams p, int chunk_index)
{
    walk_group<Quad, Tile<8>, RMAX, false, false, true>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn8f(int rmax)
{
    switch (rmax) {
        case 1: return walk_quad_few_kernel<1>;
        case 2: return walk_quad_few_kernel<2>;
        case 3: return walk_quad_few_kernel<3>;
        case 4: return walk_quad_few_kernel<4>;
        case 5: return walk_quad_few_kernel<5>;
        case 6: return walk_quad_few_kernel<6>;
        case 7: return walk_quad_few_kernel<7>;
        case 9: return walk_quad_few_kernel<9>;
        default: return walk_quad_few_kernel<10>;
    }
}

}  // namespace labsgpu
