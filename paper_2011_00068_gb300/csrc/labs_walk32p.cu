// labs_walk32p.cu -- PSL walk kernels with one walker per warp (lane blocks are odd):
// walk_lockstep in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, step_ctas(32, RMAX, true)) walk_psl_chunk_kernel(KParams p, int chunk_index)
{
    walk_group<Tile<32>, Tile<32>, RMAX, true>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn32p(int rmax)
{
    switch (rmax) {
        case 1: return walk_psl_chunk_kernel<1>;
        case 3: return walk_psl_chunk_kernel<3>;
        case 5: return walk_psl_chunk_kernel<5>;
        case 7: return walk_psl_chunk_kernel<7>;
        default: return walk_psl_chunk_kernel<9>;
    }
}

}  // namespace labsgpu
