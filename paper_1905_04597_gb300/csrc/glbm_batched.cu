// Launch sequence of one heterogeneous-batch step: one launch per level present,
// dealt to the context's stream and two side streams (the kernels are in
// glbm_batched.cuh). One stream left the chip partly idle at the end of each of the
// up to eight launches of 10 to 85 us (GB300, 64 channels of levels 2..8 and 64 columns,
// 20 steps with states set and moments read: 8.41 -> 8.16 ms).
#include <algorithm>

#include "glbm_internal.h"

int glbm_batched_launches(const BatchArgs &a)
{
    int n = 0;
    for (int N = 1; N <= GLBM_MAXN; ++N) n += a.group[N + 1] > a.group[N] ? 1 : 0;
    return n;
}

cudaError_t glbm_launch_batched_level(int N, const BatchArgs &a, bool advance, cudaStream_t s)
{
    switch (N) {
    case 1: return glbm_batched_level<1>(a, advance, s);
    case 2: return glbm_batched_level<2>(a, advance, s);
    case 3: return glbm_batched_level<3>(a, advance, s);
    case 4: return glbm_batched_level<4>(a, advance, s);
    case 5: return glbm_batched_level<5>(a, advance, s);
    case 6: return glbm_batched_level<6>(a, advance, s);
    case 7: return glbm_batched_level<7>(a, advance, s);
    case 8: return glbm_batched_level<8>(a, advance, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t glbm_launch_batched_f32(const BatchArgs &a, cudaStream_t s, const SideStreams &side)
{
    // the levels in order of decreasing work (items times populations per node), each
    // to the stream with the least work so far
    struct Level {
        int N;
        long long work;
    } lv[GLBM_MAXN_2N1];
    int n = 0;
    for (int N = 1; N <= GLBM_MAXN_2N1; ++N) {
        const long long items = a.group[N + 1] - a.group[N];
        if (items > 0) lv[n++] = Level{N, items * (2 * N + 1) * (2 * N + 1)};
    }
    std::sort(lv, lv + n, [](const Level &x, const Level &y) { return x.work > y.work; });
    const int used = std::min(n, GLBM_SIDE_STREAMS + 1);
    cudaError_t e = cudaSuccess;
    if (used > 1) e = cudaEventRecord(side.fork, s);
    for (int k = 0; k + 1 < used && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(side.s[k], side.fork, 0);
    long long load[GLBM_SIDE_STREAMS + 1] = {0};
    for (int i = 0; i < n && e == cudaSuccess; ++i) {
        const int k = (int)(std::min_element(load, load + used) - load);
        load[k] += lv[i].work;
        e = glbm_launch_batched_level(lv[i].N, a, true, k == 0 ? s : side.s[k - 1]);
    }
    for (int k = 0; k + 1 < used; ++k) {  // (joined also after an error: a capture needs it)
        cudaError_t e2 = cudaEventRecord(side.join[k], side.s[k]);
        if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(s, side.join[k], 0);
        if (e == cudaSuccess) e = e2;
    }
    return e;
}
