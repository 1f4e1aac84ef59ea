// labs_walk8b.cu -- walk kernels with four walkers per warp, lane blocks 7-10:
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

WalkFn walk_fn8b(int rmax)
{
    switch (rmax) {
        case 7: return walk_quad_kernel<7>;
        case 9: return walk_quad_kernel<9>;
        default: return walk_quad_kernel<10>;
    }
}

}  // namespace labsgpu
