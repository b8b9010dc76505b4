// Moment reducers of 2D lattices whose x axis is on the 2N+2 hierarchy.
#include "glbm_moments.cuh"

cudaError_t glbm_moments_2n2(int NX, const MomArgs &a, int prec, bool full, cudaStream_t s)
{
    switch (NX) {
#define GLBM_CASE(NN) \
    case NN: return launch_moments_kind<2, NN, 1>(a, prec, full, s);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}
