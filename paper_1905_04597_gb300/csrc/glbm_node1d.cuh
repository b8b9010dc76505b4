// One node of the 1D step (Sec. 5.1): moments of the pulled populations,
// equilibrium, relaxation. pull(ix) gives the streamed population of velocity index
// ix, store(ix, v) takes its new value; returns false when the node has left the
// positivity domain.
#pragma once
#include "glbm_device.cuh"

template <int N, typename T, class Tab, class Pull, class Store>
__device__ __forceinline__ bool node1d(const Tab &tab, const InstParams &ip, Pull &&pull, Store &&store)
{
    constexpr int Q1 = 2 * N + 1;
    constexpr bool DEV = sizeof(T) == 4;
    using Acc = TabAcc<T>;
    T f[Q1];
#pragma unroll
    for (int ix = 0; ix < Q1; ++ix) f[ix] = pull(ix);
    const T umax = (T)(0.816496580927726 * N);
    if constexpr (DEV) {
        T s = T(0), c = T(0), sj = T(0), cj = T(0);
#pragma unroll
        for (int ix = 0; ix < Q1; ++ix) acc2(s, c, f[ix]);
#pragma unroll
        for (int n = 1; n <= N; ++n) acc2(sj, cj, T(n) * (f[N + n] - f[N - n]));
        const T drho = s + c;
        const T rho = T(1) + drho;
        const T j = sj + cj;
        T u = j / rho;
        // u = j / (1 + delta rho) from the unrounded density, by one correction with
        // the residual (j - u) - u delta rho (j - u is exact)
        u += fma(-u, drho, j - u) / rho;
        T d[Q1];
        eq_dev_all<N, T>(tab, u, d);
        const T om = (T)ip.omega_f;
#pragma unroll
        for (int ix = 0; ix < Q1; ++ix) {
            // delta f^eq = d + drho (W + d), the momentum-carrying d unscaled by a
            // rounded rho
            const T w = Acc::W(tab, ix);
            const T eq = fma(drho, w + d[ix], d[ix]);
            store(ix, fma(om, eq - f[ix], f[ix]));  // f + omega (f^eq - f)
        }
        return rho > T(0) && fabs(u) <= umax;
    } else {
        // FP64: as few instructions as the pipe's 64 cycles per warp ask for. W joins
        // the even part (E_{+-n} = (W + Ae) +- u Bo), f^eq - f is one fused rounding
        T rho = f[0], j = f[N + 1] - f[N - 1];
#pragma unroll
        for (int ix = 1; ix < Q1; ++ix) rho += f[ix];
#pragma unroll
        for (int n = 2; n <= N; ++n) j = fma(T(n), f[N + n] - f[N - n], j);
        const T u = j / rho, v = u * u, om = (T)ip.omega;
#pragma unroll
        for (int n = 0; n <= N; ++n) {
            T a = Acc::Ce(tab, n, N);
#pragma unroll
            for (int i = N - 1; i >= 1; --i) a = fma(a, v, Acc::Ce(tab, n, i));
            a = fma(a, v, Acc::W(tab, N + n));
            if (n == 0) {
                store(N, fma(om, fma(rho, a, -f[N]), f[N]));
            } else {
                T b = Acc::Co(tab, n, N - 1);
#pragma unroll
                for (int i = N - 2; i >= 0; --i) b = fma(b, v, Acc::Co(tab, n, i));
                store(N + n, fma(om, fma(rho, fma(u, b, a), -f[N + n]), f[N + n]));
                store(N - n, fma(om, fma(rho, fma(-u, b, a), -f[N - n]), f[N - n]));
            }
        }
        return rho > T(0) && fabs(u) <= umax;
    }
}

// The same in global or block-wide coordinates: populations fin[q][x] of a lattice of
// L nodes, halfway bounce-back or periodic ends.
template <int N, typename T>
__device__ __forceinline__ void node1d_at(const AuxArgs &a, const InstParams &ip, const T *fin,
                                          T *fout, int x, int L, long long plane, unsigned *status)
{
    const bool ok = node1d<N, T>(
        a.tab, ip,
        [&](int ix) {
            int xs = x - (ix - N), q = ix;
            if (a.bc == GLBM_BC_PERIODIC) {
                xs = wrap_index(xs, L);
            } else if (xs < 0) {
                xs = -1 - xs;
                q = 2 * N - ix;
            } else if (xs >= L) {
                xs = 2 * L - 1 - xs;
                q = 2 * N - ix;
            }
            return fin[(long long)q * plane + xs];
        },
        [&](int ix, T v) { fout[(long long)ix * plane + x] = v; });
    if (!ok) flag_unstable(status);
}
