// labs_walk8a.cu -- walk kernels with four walkers per warp, lane blocks 1-6:
// walk_lockstep in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, step_ctas(8, RMAX)) walk_quad_kernel(KParams p, int chunk_index)
{
    walk_group<Quad, Tile<8>, RMAX>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn8a(int rmax)
{
    switch (rmax) {
        case 1: return walk_quad_kernel<1>;
        case 2: return walk_quad_kernel<2>;
        case 3: return walk_quad_kernel<3>;
        case 4: return walk_quad_kernel<4>;
        case 5: return walk_quad_kernel<5>;
        default: return walk_quad_kernel<6>;
    }
}

}  // namespace labsgpu
