// Prints the plain walk's shared-memory layout (labs_internal.cuh, compiled for the host),
// one line per (PSL objective, tile, n): the layout of the kernel a context of longest n takes, h0 hc ks r8 g gneg gpos z zneg x xp b bvec words R, and per
// (tile, lane block) its column groups and lag blocks.
#define __host__
#define __device__
#include <cstdio>

#include "labs_internal.cuh"

using namespace labsgpu;

int main()
{
    const int tiles[3] = {8, 16, 32}, top[3] = {80, 160, 256};
    for (int psl = 0; psl < 2; ++psl)
        for (int ti = psl; ti < 3; ++ti)
            for (int n = 2; n <= (psl && ti == 1 ? 128 : top[ti]); ++n) {
                const StepSmem w = step_smem(tiles[ti], step_R(n, tiles[ti]), psl != 0);
                std::printf("step %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d\n", psl, tiles[ti], n, w.h0, w.hc, w.ks,
                            w.r8, w.g, w.gneg, w.gpos, w.z, w.zneg, w.x, w.xp, w.b, w.bvec, w.words,
                            step_R(n, tiles[ti]));
            }
    for (int ti = 0; ti < 3; ++ti)
        for (int R = 1; R <= 10; ++R)
            std::printf("shape %d %d %d %d %d\n", tiles[ti], R, step_groups(tiles[ti], R), step_lag_blocks(tiles[ti], R),
                        step_n(tiles[ti], R));
    return 0;
}
