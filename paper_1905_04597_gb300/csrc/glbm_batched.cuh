// Heterogeneous batches: many independent channel instances of different
// level, size, relaxation time, walls and force advance one step together.
// The work list holds every (instance, x0, y0) tile, grouped by level; a step
// is one launch per level present, each CTA taking one tile of that level and
// running the fused stream-collide tile (one-node or packed pair) with the
// level's tile shape. The levels' instances are independent, so their launches go to
// three streams and overlap where one level's last wave leaves SMs idle; the CTAs of
// all of them count towards the step's end, and the last one advances the dither
// counter.
#pragma once
#include "glbm_step2d_pair.cuh"
#include "glbm_tiles.h"

// CTAs per SM asked of a one-node tile (0: the compiler's choice). At level 7 the
// compiler took 128 registers, three CTAs of (5, 1, 1); 96 hold its three rows of 15
// without spills, four CTAs (GB300, 64 channels of 64 columns, per step: 283 -> 277.6
// us).
template <int N, int G, int R>
constexpr int ITEMS_CTAS = N == 7 && R == 1 && G == 5 ? 4 : 0;

template <int N, int G, int R>
__global__ void __launch_bounds__(32 * G * R, ITEMS_CTAS<N, G, R>)
    k_step2d_items(const __grid_constant__ BatchLevelArgs a)
{
    using S = Step2D<N, float, G, R>;
    __shared__ typename S::Smem sm;
    const bool live = !step_halted(a.status);  // needed only at the stores
    const int4 it = a.items[blockIdx.x];  // (instance, x0, y0, N)
    const InstParams &ip = a.ip[it.x];
    const float *fin = static_cast<const float *>(a.fin) + ip.off;
    float *fout = static_cast<float *>(a.fout) + ip.off;
    const unsigned seed = hash32(__ldcg(a.step_ctr) * 0x632BE5ABu + (unsigned)it.x);
    S::run(a.tab, a.tab, ip, ip.Lx, ip.Ly, ip.pitch, (int)ip.plane, ip.bc, fin, fout,
           it.y, it.z, sm, a.status, seed, nullptr, live);
    if (a.total && live) finish_step(a.status, a.total);
}

template <int N, int G, int R>
__global__ void __launch_bounds__(32 * G * R)
    k_step2d_pair_items(const __grid_constant__ BatchLevelArgs a)
{
    using S = Step2DPair<N, G, R>;
    __shared__ __align__(16) typename S::Smem sm;
    const bool live = !step_halted(a.status);  // needed only at the stores
    const int4 it = a.items[blockIdx.x];  // (instance, x0, y0, N)
    const InstParams &ip = a.ip[it.x];
    const float *fin = static_cast<const float *>(a.fin) + ip.off;
    float *fout = static_cast<float *>(a.fout) + ip.off;
    const unsigned seed = hash32(__ldcg(a.step_ctr) * 0x632BE5ABu + (unsigned)it.x);
    S::run(a.tab, a.tab, ip, ip.Lx, ip.Ly, ip.pitch, (int)ip.plane, ip.bc, fin, fout,
           it.y, it.z, sm, a.status, seed, nullptr, live);
    if (a.total && live) finish_step(a.status, a.total);
}

template <int N, int I = 0>
cudaError_t launch_items_shape(int shape, const BatchLevelArgs &a, int count, cudaStream_t s)
{
    if constexpr (I < Tiles<N, float>::count) {
        if (shape == I) {
            constexpr TileShape t = Tiles<N, float>::shape[I];
            constexpr int G = t.G, R = t.R;
            if constexpr (t.V == 2)
                k_step2d_pair_items<N, G, R><<<count, 32 * G * R, 0, s>>>(a);
            else
                k_step2d_items<N, G, R><<<count, 32 * G * R, 0, s>>>(a);
            return cudaGetLastError();
        }
        return launch_items_shape<N, I + 1>(shape, a, count, s);
    } else {
        return cudaErrorInvalidValue;
    }
}

// The launch takes its own level's table only (the eight together are 18 KB of
// kernel parameters).
template <int N>
cudaError_t glbm_batched_level(const BatchArgs &b, bool advance, cudaStream_t s)
{
    const int first = b.group[N], count = b.group[N + 1] - b.group[N];
    if (count <= 0) return cudaSuccess;
    BatchLevelArgs a;
    a.tab = b.tab[N - 1];
    a.fin = b.fin;
    a.fout = b.fout;
    a.ip = b.ip;
    a.items = b.items + first;
    a.status = b.status;
    a.step_ctr = b.step_ctr;
    a.total = advance ? (unsigned)b.n_items : 0u;
    return launch_items_shape<N>(b.shape[N], a, count, s);
}
