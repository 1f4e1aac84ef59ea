// labs_walk16q.cu -- PSL walk kernels with two walkers per warp, lane blocks 6-9:
// walk_lockstep in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, step_ctas(16, RMAX, true)) walk_psl_pair_kernel(KParams p, int chunk_index)
{
    walk_group<Pair, Tile<16>, RMAX, true>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn16q(int rmax)
{
    switch (rmax) {
        case 6: return walk_psl_pair_kernel<6>;
        case 7: return walk_psl_pair_kernel<7>;
        default: return walk_psl_pair_kernel<9>;
    }
}

}  // namespace labsgpu
