// Instantiations and dispatch of the small-lattice FP64 step, 2N+2 hierarchy.
#include "glbm_step2d_small.cuh"
#include "glbm_tiles_zv.h"

template <int N>
static cudaError_t small_zv(int zv, const SmallArgs &a, int n_inst, cudaStream_t s)
{
    if (zv == GLBM_ZV_Y)
        return launch_small<N, 1, 1, 0, TilesZv<N, double, GLBM_ZVK_X1>::shape[0].G>(a, n_inst, s);
    if constexpr (N <= GLBM_MAXN_2N1)
        return launch_small<N, N, 1, 1, TilesZv<N, double, GLBM_ZVK_XY>::shape[0].G>(a, n_inst, s);
    return cudaErrorInvalidValue;
}

cudaError_t glbm_launch_step2d_small_zv(int N, int zv, const SmallArgs &a, int n_inst, cudaStream_t s)
{
    switch (N) {
#define GLBM_CASE(NN) \
    case NN: return small_zv<NN>(zv, a, n_inst, s);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4) GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7)
        GLBM_CASE(8) GLBM_CASE(9) GLBM_CASE(10) GLBM_CASE(11) GLBM_CASE(12) GLBM_CASE(13)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}
