// labs_walk32b.cu -- best-first search kernels, one walker per warp (lane blocks are odd):
// walk_bestfirst in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, step_ctas(32, RMAX)) walk_bestfirst_kernel(KParams p, int chunk_index)
{
    walk_group<Tile<32>, Tile<32>, RMAX, false, true>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn32b(int rmax)
{
    switch (rmax) {
        case 1: return walk_bestfirst_kernel<1>;
        case 3: return walk_bestfirst_kernel<3>;
        case 5: return walk_bestfirst_kernel<5>;
        case 7: return walk_bestfirst_kernel<7>;
        default: return walk_bestfirst_kernel<9>;
    }
}

}  // namespace labsgpu
