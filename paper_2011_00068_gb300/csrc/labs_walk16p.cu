// labs_walk16p.cu -- PSL walk kernels with two walkers per warp, lane blocks 1-5:
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

WalkFn walk_fn16p(int rmax)
{
    switch (rmax) {
        case 1: return walk_psl_pair_kernel<1>;
        case 2: return walk_psl_pair_kernel<2>;
        case 3: return walk_psl_pair_kernel<3>;
        default: return walk_psl_pair_kernel<5>;
    }
}

}  // namespace labsgpu
