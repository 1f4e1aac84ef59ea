// labs_walk32f.cu -- walk kernels with one walker per warp for few walkers (every neighbour's HT slot
// looked up at a step's start): walk_lockstep in labs_step.cuh, compiled in their own unit.
#include "labs_step.cuh"

namespace labsgpu {

namespace {

template <int RMAX>
__global__ void __launch_bounds__(256, 1) walk_chunk_few_kernel(KParams p, int chunk_index)
{
    walk_group<Tile<32>, Tile<32>, RMAX, false, false, true>(p, chunk_index);
}

}  // namespace

WalkFn walk_fn32f(int rmax)
{
    switch (rmax) {
        case 1: return walk_chunk_few_kernel<1>;
        case 3: return walk_chunk_few_kernel<3>;
        case 5: return walk_chunk_few_kernel<5>;
        case 7: return walk_chunk_few_kernel<7>;
        default: return walk_chunk_few_kernel<9>;
    }
}

}  // namespace labsgpu
