// labs_walk16b.cu -- walk kernels with two walkers per warp, lane blocks 6-10:
// walk_lockstep in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, step_ctas(16, RMAX)) walk_pair_kernel(KParams p, int chunk_index)
{
    walk_group<Pair, Tile<16>, RMAX>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn16b(int rmax)
{
    switch (rmax) {
        case 6: return walk_pair_kernel<6>;
        case 7: return walk_pair_kernel<7>;
        case 9: return walk_pair_kernel<9>;
        default: return walk_pair_kernel<10>;
    }
}

}  // namespace labsgpu
