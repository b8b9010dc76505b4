// Instantiations and dispatch of the small-lattice FP64 step, 2N+1 hierarchy.
#include "glbm_step2d_small.cuh"

cudaError_t glbm_launch_step2d_small(int N, int NX, int zv, const SmallArgs &a, int n_inst,
                                     cudaStream_t s)
{
    if (zv != 0) return glbm_launch_step2d_small_zv(N, zv, a, n_inst, s);
    const bool x1 = NX != N;
    switch (N) {
#define GLBM_CASE(NN)                                                                     \
    case NN:                                                                              \
        return x1 ? launch_small<NN, 1, 0, 0, TilesX1<NN, double>::shape[0].G>(a, n_inst, s) \
                  : launch_small<NN, NN, 0, 0, Tiles<NN, double>::shape[0].G>(a, n_inst, s);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}
