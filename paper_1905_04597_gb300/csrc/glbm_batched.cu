// Launch sequence of one heterogeneous-batch step: one launch per level present,
// dealt to the context's stream and two side streams (the kernels are in
// glbm_batched.cuh). One stream left the chip partly idle at the end of each of the up
// to eight launches. Three are faster, but two where five or more levels together fill
// the chip (from 30 million populations a step): with three, the end of every chain
// meets fewer other CTAs to fill up with. GB300, us per step in calls of 8 steps, three
// and two (one in chunks of 64 in brackets): levels 2 to 8, 7 channels of 64 x 60 (4 M)
// 33.8 and 41.8 (50), 7 of 64 x 200 (13 M) 52.9 and 52.9 (69), 21 of 64 x 200 (38 M) 120
// and 110 (125), 63 (114 M) 261 and 227 (255), 21 of 512 x 128 (197 M) 409 and 373 (408);
// levels 2 to 4, 3 of 16 x 40 14.2 and 18.1 (17), 27 of 128 x 300 (55 M) 100 and 103 (103);
// 64 channels of levels 2 to 8, 64 columns and 32 to 512 rows (138 M) 284 and 262.
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
    // the levels in order of decreasing work (populations), each to the stream with the
    // least work so far
    struct Level {
        int N;
        long long work;
    } lv[GLBM_MAXN_2N1];
    int n = 0;
    for (int N = 1; N <= GLBM_MAXN_2N1; ++N) {
        if (a.pops[N] > 0) lv[n++] = Level{N, a.pops[N]};
    }
    std::sort(lv, lv + n, [](const Level &x, const Level &y) { return x.work > y.work; });
    long long total = 0;
    for (int i = 0; i < n; ++i) total += lv[i].work;
    const int used = std::min(n, n >= 5 && total > 30000000 ? 2 : GLBM_SIDE_STREAMS + 1);
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
