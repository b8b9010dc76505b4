// Initial equilibrium of one instance (Eq. maineq02 with the product form of Sec. 4)
// from FP64 fields, 1D, 2D and 3D, on every lattice kind.
//
// A CTA covers 32 nodes of the flattened lattice with four warps: the values and
// mirror pairs of E - W of every axis are dealt to the warps and meet in shared
// memory, then the velocity rows. Per row A = rho E^y E^z and B = A - W^y W^z =
// (rho - 1) W^y W^z + rho (d^y E^z + W^y d^z) (no cancellation); a population is E^x A
// (FP64 storage) or W^x B + d^x A (FP32 deviations).
//
// What bounds it: FP64 needs two instructions and a conversion per population on a
// pipe that issues two per cycle and SM, fourteen times the time of the stores. FP32
// deviations are formed in float pairs (value = h + l, 48 bits) on the FP32 pipe
// instead. The value before the rounding to float is off by at most 2^-44.4 of the
// magnitudes of its terms (the largest of 2 x 10^8 populations per level and dimension
// against FP64, levels 1 to 8 and 13, velocities up to 1), the terms of B and of d taken
// before they cancel. Where the rounding could go either way within 2^-42 of them (one
// population in 2^14 to 2^15 at velocities of 0.03) it is formed in FP64, so every
// stored float is that of the FP64 formula. Fields outside 1e-18..1e18 in magnitude (or
// not finite) take FP64. The pairs' kernel is bound by its issue slots (92 instructions
// per population at D3Q125 and 65 at D2Q289 with run-time row lengths), so the x axis's
// velocities are a template parameter, populations too close to call are collected and
// formed after their row, and E^y, rho E^z and rho (E^z - W^z) are formed once per node.
// Measured on GB300, FP32, FP64 pipe -> pairs -> this: D2Q81 512 x 256 95 -> 39 -> 34 us,
// D2Q289 1024 x 128 311 -> 95 -> 84 us, D3Q125 250 x 61 x 45 815 -> 257 -> 194 us (3 to
// 6 % of it for the terms' magnitudes; tolerances of |W^x B| + |d^x A| alone left one
// population in 10^8 a float off, one in 10^4 where rows cancel); D1Q3 x D1Q28 200 nodes
// (FP64) 25 -> 10 us; large FP64 lattices stay on the FP64 pipe (D2Q81 54 us).
#include "glbm_device.cuh"

namespace {

struct df {  // h + l, |l| <= ulp(h) / 2
    float h, l;
};

__device__ __forceinline__ df df_norm(float h, float l)  // |h| >= |l|
{
    const float s = h + l;
    return df{s, l - (s - h)};
}
__device__ __forceinline__ df df_add(df a, df b)
{
    const float s = a.h + b.h, t = s - a.h;
    const float e = (a.h - (s - t)) + (b.h - t);
    return df_norm(s, e + (a.l + b.l));
}
__device__ __forceinline__ df df_mul(df a, df b)
{
    const float p = __fmul_rn(a.h, b.h);
    return df_norm(p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ df df_fma(df a, df b, df c)
{
    const float p = __fmul_rn(a.h, b.h);
    const float pe = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
    const float s = p + c.h, t = s - p;
    const float e = (p - (s - t)) + (c.h - t);
    return df_norm(s, e + (pe + c.l));
}
__device__ __forceinline__ df df_neg(df a) { return df{-a.h, -a.l}; }
__device__ __forceinline__ df to_df(double x)
{
    const float h = (float)x;
    return df{h, (float)(x - f2d(h))};
}

// Arithmetic of one precision: V holds a value, C reads the coefficients.
struct F64 {
    using V = double;
    static __device__ __forceinline__ V conv(double x) { return x; }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    static __device__ __forceinline__ V mul(V a, V b) { return mul_rn(a, b); }
    static __device__ __forceinline__ V fma_(V a, V b, V c) { return fma(a, b, c); }
    static __device__ __forceinline__ V neg(V a) { return -a; }
};
struct F32 {
    using V = df;
    static __device__ __forceinline__ V conv(double x) { return to_df(x); }
    static __device__ __forceinline__ V add(V a, V b) { return df_add(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return df_mul(a, b); }
    static __device__ __forceinline__ V fma_(V a, V b, V c) { return df_fma(a, b, c); }
    static __device__ __forceinline__ V neg(V a) { return df_neg(a); }
};

constexpr float EQ_V = 0x1p-6f;

// Table of one axis in the arithmetic's values: rest weights by velocity index, and
// the even and odd coefficients of every mirror pair (Ce[m][i], i = 0..N-1 for v^(i+1)).
// M: the highest level it holds (kernel parameters of 5 KB at 8, 12 KB at 13).
template <class V, int M>
struct EqAxis {
    int N, zv;
    V W[2 * M + 2];
    V Ce[M + 1][M], Co[M + 1][M];
    float me[M + 1], mo[M + 1];  // sums of |Ce| v^i and |Co| v^i at v = EQ_V
};
struct NoAxis {};
template <class V, int M>
struct EqArgs {
    EqAxis<V, M> y, x;  // 3D: y holds for z too
    // float pairs: the FP64 tables too
    std::conditional_t<std::is_same<V, df>::value, EqAxis<double, M>, NoAxis> y64, x64;
    // float pairs, 3D: W^y W^z
    std::conditional_t<std::is_same<V, df>::value, V, NoAxis> wyz[2 * GLBM_MAXN_3D + 1]
                                                                 [2 * GLBM_MAXN_3D + 1];
    const double *rho, *u[3];  // null: 1, 0
    void *f;
    unsigned *status;           // the status words a new state resets, or null
    int Lx, nodes, pitch, dims;
    long long plane;
};

// E - W of the mirror pair m of one axis (plus: the positive velocity). Float pairs:
// also the sum of its terms' magnitudes, which its error is a fraction of, with 2^-80
// for the words that underflow at tiny velocities (0 at u = 0, where both are exact):
// from its sums at v = 2^-6 up to there, term by term beyond.
template <class P, int M>
__device__ __forceinline__ void eq_pair(const EqAxis<typename P::V, M> &t, int m, typename P::V u,
                                        typename P::V &plus, typename P::V &minus, float &mag)
{
    using V = typename P::V;
    constexpr bool F = std::is_same<V, df>::value;
    const int N = t.N;
    const V v = P::mul(u, u);
    V e = t.Ce[m][N - 1], o = t.Co[m][N - 1];
    for (int i = N - 2; i >= 0; --i) {
        e = P::fma_(e, v, t.Ce[m][i]);
        o = P::fma_(o, v, t.Co[m][i]);
    }
    e = P::mul(e, v);
    if constexpr (F) {
        float me = t.me[m], mo = t.mo[m];
        if (v.h > EQ_V) {
            me = mo = 0.f;
            for (int i = N - 1; i >= 0; --i) {
                me = fmaf(me, v.h, fabsf(t.Ce[m][i].h));
                mo = fmaf(mo, v.h, fabsf(t.Co[m][i].h));
            }
        }
        mag = u.h != 0.f ? fmaf(fabsf(u.h), mo, fmaf(me, v.h, 0x1p-80f)) : 0.f;
    }
    if (m == 0 && !t.zv) {  // the zero velocity
        plus = minus = e;
        return;
    }
    plus = P::fma_(u, o, e);
    minus = P::fma_(P::neg(u), o, e);
}

// Population (iz, iy, ix) of node n in FP64.
template <int M>
__device__ __noinline__ float eq_exact(const EqArgs<df, M> &a, int n, int iz, int iy, int ix)
{
    const auto dev = [](const EqAxis<double, M> &t, double u, int i) {
        const int vel = t.zv ? 2 * i - (2 * t.N + 1) : i - t.N, av = vel < 0 ? -vel : vel;
        const int m = t.zv ? (av - 1) / 2 : av;
        const double v = u * u;
        double e = t.Ce[m][t.N - 1], o = t.Co[m][t.N - 1];
        for (int k = t.N - 2; k >= 0; --k) {
            e = fma(e, v, t.Ce[m][k]);
            o = fma(o, v, t.Co[m][k]);
        }
        e = mul_rn(e, v);
        return vel == 0 ? e : fma(vel > 0 ? u : -u, o, e);
    };
    const double r = a.rho ? a.rho[n] : 1.0;
    double A = r, B = r - 1.0;
    if (a.dims >= 2) {
        const double wy = a.y64.W[iy], dy = dev(a.y64, a.u[1] ? a.u[1][n] : 0.0, iy);
        if (a.dims == 2) {
            A = r * (wy + dy);
            B = fma(r - 1.0, wy, mul_rn(r, dy));
        } else {
            const double wz = a.y64.W[iz], dz = dev(a.y64, a.u[2] ? a.u[2][n] : 0.0, iz);
            A = r * mul_rn(wy + dy, wz + dz);
            B = fma(r - 1.0, mul_rn(wy, wz), mul_rn(r, fma(dy, wz + dz, mul_rn(wy, dz))));
        }
    }
    return (float)fma(dev(a.x64, a.u[0] ? a.u[0][n] : 0.0, ix), A, mul_rn(a.x64.W[ix], B));
}

// W^x B + d^x A rounded once to float; false where the rounding is too close to call
// for an error of up to `tol`.
__device__ __forceinline__ bool eq_dev(df w, df B, df d, df A, float tol, float &out)
{
    const float p = __fmul_rn(w.h, B.h), q = __fmul_rn(d.h, A.h);
    const float pe = fmaf(w.l, B.h, fmaf(w.h, B.l, fmaf(w.h, B.h, -p)));
    const float qe = fmaf(d.l, A.h, fmaf(d.h, A.l, fmaf(d.h, A.h, -q)));
    const float s = p + q, t = s - p;
    const float e = ((p - (s - t)) + (q - t)) + (pe + qe);
    out = s + (e - tol);
    return out == s + (e + tol);
}

constexpr int EQ_WARPS = 4;

// QX: the velocities of the x axis (float pairs), or 0: known at run time only.
template <class P, int M, int QX>
__global__ void __launch_bounds__(32 * EQ_WARPS)
    k_equilibrium(const __grid_constant__ EqArgs<typename P::V, M> a)
{
    using V = typename P::V;
    constexpr bool F = std::is_same<V, df>::value;  // float pairs
    __shared__ V in[5][32];                  // u_x, u_y, u_z, rho, rho - 1
    __shared__ V dx[2 * GLBM_MAXN_2N1 + 2][32];  // FP32: E^x - W^x; FP64: E^x
    __shared__ V dy[2 * M + 2][32];              // E^y - W^y
    // float pairs: E^y, the magnitudes of E^x - W^x's terms by mirror pair, and per row
    // the tolerances of W^x B and d^x A over the x axis's factors (3D: their factors)
    __shared__ V ey[F ? 2 * M + 2 : 1][32];
    __shared__ float magx[F ? GLBM_MAXN_2N1 + 1 : 1][32];
    __shared__ float2 ty[F ? 2 * M + 2 : 1][32];
    // 3D: E^z - W^z, and for float pairs rho E^z, rho (E^z - W^z) and the tolerances'
    // factors, in the rows that its levels leave free
    constexpr int QZ = 2 * GLBM_MAXN_3D + 1;
    static_assert(2 * M + 2 >= 2 * QZ, "room for the z axis");
    V(*const dz)[32] = dy + QZ, (*const pz)[32] = ey + QZ, (*const qz)[32] = dx + QZ;
    float2(*const tz)[32] = ty + QZ;
    if (a.status && blockIdx.x == 0 && threadIdx.x == 0) reset_status(a.status);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n = blockIdx.x * 32 + lane, nc = n < a.nodes ? n : a.nodes - 1;
    const int row = nc / a.Lx, x = nc - row * a.Lx;
    const long long base = (long long)row * a.pitch + x;
    bool ok = true;  // every field within the float pairs' range
    for (int k = w; k < 5; k += EQ_WARPS) {
        double v = 0.0;
        if (k < 3) {
            if (a.u[k]) v = a.u[k][nc];
        } else {
            v = a.rho ? a.rho[nc] : 1.0;
        }
        if (F && !(fabs(v) < 1e18 && (fabs(v) > 1e-18 || v == 0.0))) ok = false;
        if (k == 4) v -= 1.0;
        in[k][lane] = P::conv(v);
    }
    unsigned bad = 0u;  // lanes (nodes) out of range in any warp
    if (F) {
        __shared__ unsigned badw[EQ_WARPS];
        const unsigned b = __ballot_sync(0xFFFFFFFFu, !ok);
        if (lane == 0) badw[w] = b;
        __syncthreads();
        for (int k = 0; k < EQ_WARPS; ++k) bad |= badw[k];
    } else {
        __syncthreads();
    }
    // the mirror pairs of the axes, dealt to the warps
    const int nx = a.x.N + 1, ny = a.dims >= 2 ? a.y.N + 1 : 0, nz = a.dims == 3 ? a.y.N + 1 : 0;
    for (int t = w; t < nx + ny + nz; t += EQ_WARPS) {
        const int ax = t < nx ? 0 : t < nx + ny ? 1 : 2;
        const int m = ax == 0 ? t : ax == 1 ? t - nx : t - nx - ny;
        const EqAxis<V, M> &tab = ax == 0 ? a.x : a.y;
        V plus, minus;
        float mag;
        eq_pair<P>(tab, m, in[ax][lane], plus, minus, mag);
        const int ip = tab.zv ? tab.N + 1 + m : tab.N + m, im = tab.N - m;
        if (!F && ax == 0) {
            plus = P::add(tab.W[ip], plus);
            minus = P::add(tab.W[im], minus);
        }
        if constexpr (F) {
            const float w = tab.W[ip].h, ar = 0x1p-42f * fabsf(in[3][lane].h);
            const float ar1 = 0x1p-42f * fabsf(in[4][lane].h);
            if (ax == 0)
                magx[m][lane] = mag;
            else if (ax == 2)
                tz[im][lane] = tz[ip][lane] = make_float2(ar * (w + mag), ar * mag);
            else if (a.dims == 2)
                ty[im][lane] = ty[ip][lane] = make_float2(ar * (w + mag), fmaf(ar1, w, ar * mag));
            else
                ty[im][lane] = ty[ip][lane] = make_float2(w + mag, mag);
        }
        if (F && ax == 1) {
            ey[im][lane] = P::add(tab.W[im], minus);
            ey[ip][lane] = P::add(tab.W[ip], plus);
        }
        if (F && ax == 2) {
            const V r = in[3][lane];
            pz[im][lane] = P::mul(r, P::add(tab.W[im], minus));
            pz[ip][lane] = P::mul(r, P::add(tab.W[ip], plus));
            qz[im][lane] = P::mul(r, minus);
            qz[ip][lane] = P::mul(r, plus);
            continue;
        }
        V(*const d)[32] = ax == 0 ? dx : ax == 1 ? dy : dz;
        d[im][lane] = minus;
        d[ip][lane] = plus;
    }
    __syncthreads();
    const int Qx = QX ? QX : 2 * a.x.N + 1 + a.x.zv, Qy = a.dims >= 2 ? 2 * a.y.N + 1 + a.y.zv : 1;
    const int rows = a.dims == 3 ? Qy * Qy : Qy;
    const V r = in[3][lane], r1 = in[4][lane];
    const bool live = n < a.nodes, pairs = !((bad >> lane) & 1u);
    // float pairs: the tolerances of A's and B's terms (1D: of rho and rho - 1)
    float t0 = 0.f, t1 = 0.f;
    if constexpr (F) t0 = 0x1p-42f * fabsf(r.h), t1 = 0x1p-42f * fabsf(r1.h);
    int iz = 0, iy = w;
    for (int j = w; j < rows; j += EQ_WARPS, iy += EQ_WARPS) {
        V A = r, B = r1;
        float tA = t0, tB = t1;
        if (a.dims == 3) {
            for (; iy >= Qy; iy -= Qy) ++iz;
            if constexpr (F) {
                const V z = pz[iz][lane];
                A = P::mul(z, ey[iy][lane]);
                B = P::fma_(r1, a.wyz[iz][iy],
                            P::fma_(dy[iy][lane], z, P::mul(a.y.W[iy], qz[iz][lane])));
                const float2 fy = ty[iy][lane], fz = tz[iz][lane];
                tA = fz.x * fy.x;
                tB = fmaf(t1, a.wyz[iz][iy].h, fmaf(fy.y, fz.x, a.y.W[iy].h * fz.y));
            } else {
                A = P::mul(r, P::mul(P::add(a.y.W[iy], dy[iy][lane]), P::add(a.y.W[iz], dz[iz][lane])));
            }
        } else if (a.dims == 2) {
            if constexpr (F) {
                A = P::mul(r, ey[iy][lane]);
                B = P::fma_(r1, a.y.W[iy], P::mul(r, dy[iy][lane]));
                const float2 t = ty[iy][lane];
                tA = t.x;
                tB = t.y;
            } else {
                A = P::mul(r, P::add(a.y.W[iy], dy[iy][lane]));
            }
        }
        if (!live) continue;
        const long long o = base + (long long)(j * Qx) * a.plane;
        if constexpr (F) {
            float *out = static_cast<float *>(a.f) + o;
            unsigned open = 0u;  // columns to form in FP64
#pragma unroll
            for (int ix = 0; ix < QX; ++ix, out += a.plane) {
                constexpr int PX = QX / 2, MX = (QX - 1) / 2;  // columns of the pair number 0
                const float tol = fmaf(a.x.W[ix].h, tB, magx[ix >= PX ? ix - PX : MX - ix][lane] * tA);
                float v;
                if (!eq_dev(a.x.W[ix], B, dx[ix][lane], A, tol, v)) open |= 1u << ix;
                *out = v;
            }
            if (!pairs) open = (1u << QX) - 1u;
            for (; open; open &= open - 1u) {
                const int ix = __ffs(open) - 1;
                static_cast<float *>(a.f)[o + ix * a.plane] = eq_exact(a, nc, iz, iy, ix);
            }
        } else {
            double *out = static_cast<double *>(a.f) + o;
#pragma unroll 3
            for (int ix = 0; ix < Qx; ++ix, out += a.plane) *out = dx[ix][lane] * A;
        }
    }
}

double host_value(double x, double *) { return x; }
df host_value(double x, df *)
{
    df d;
    d.h = (float)x;
    d.l = (float)(x - (double)d.h);
    return d;
}

template <class V, int M>
void fill_axis(const AxisTableHi &t, EqAxis<V, M> &e)
{
    V *const tag = nullptr;
    e.N = t.N;
    e.zv = t.zv;
    for (int i = 0; i < ax_q(t); ++i) e.W[i] = host_value(t.W[i], tag);
    for (int m = 0; m <= t.N; ++m)
        for (int i = 0; i < t.N; ++i) {
            e.Ce[m][i] = host_value(t.Ce[m][i + 1], tag);
            e.Co[m][i] = host_value(m == 0 && !t.zv ? 0.0 : t.Co[m][i], tag);
        }
    for (int m = 0; m <= t.N; ++m) {
        double se = 0.0, so = 0.0;
        for (int i = t.N - 1; i >= 0; --i) {
            se = se * EQ_V + fabs(t.Ce[m][i + 1]);
            so = so * EQ_V + (m == 0 && !t.zv ? 0.0 : fabs(t.Co[m][i]));
        }
        e.me[m] = (float)se;
        e.mo[m] = (float)so;
    }
}

template <class P, int M>
cudaError_t launch_eq(const AuxArgs &a, void *f, const double *rho, const double *ux,
                      const double *uy, const double *uz, unsigned *status, cudaStream_t s)
{
    EqArgs<typename P::V, M> e = {};
    fill_axis(a.tab, e.y);
    fill_axis(a.dims == 2 ? a.tabx : a.tab, e.x);
    if constexpr (std::is_same<P, F32>::value) {
        fill_axis(a.tab, e.y64);
        fill_axis(a.dims == 2 ? a.tabx : a.tab, e.x64);
        df *const tag = nullptr;
        for (int i = 0; a.dims == 3 && i < ax_q(a.tab); ++i)
            for (int j = 0; j < ax_q(a.tab); ++j)
                e.wyz[i][j] = host_value(a.tab.W[i] * a.tab.W[j], tag);
    }
    e.rho = rho;
    e.u[0] = ux;
    e.u[1] = a.dims >= 2 ? uy : nullptr;
    e.u[2] = a.dims == 3 ? uz : nullptr;
    e.f = f;
    e.status = status;
    e.Lx = a.Lx;
    e.nodes = a.Lx * a.Ly * a.Lz;
    e.pitch = a.pitch;
    e.dims = a.dims;
    e.plane = a.plane;
    const int blocks = (e.nodes + 31) / 32, threads = 32 * EQ_WARPS;
    if constexpr (std::is_same<P, F64>::value) {
        k_equilibrium<P, M, 0><<<blocks, threads, 0, s>>>(e);
    } else {
        const int QX = 2 * e.x.N + 1 + e.x.zv;
        if constexpr (M > GLBM_MAXN_2N1) {  // these levels are compiled with D1Q3 along x
            if (QX != 3) return cudaErrorInvalidValue;
            k_equilibrium<P, M, 3><<<blocks, threads, 0, s>>>(e);
        } else {
            switch (QX) {
#define GLBM_CASE(QX) \
            case QX: k_equilibrium<P, M, QX><<<blocks, threads, 0, s>>>(e); break;
                GLBM_CASE(3) GLBM_CASE(4) GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
                GLBM_CASE(9) GLBM_CASE(10) GLBM_CASE(11) GLBM_CASE(12) GLBM_CASE(13) GLBM_CASE(14)
                GLBM_CASE(15) GLBM_CASE(16) GLBM_CASE(17) GLBM_CASE(18)
#undef GLBM_CASE
            default: return cudaErrorInvalidValue;
            }
        }
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t glbm_launch_set_equilibrium(const AuxArgs &a, void *f, const double *rho,
                                        const double *ux, const double *uy, const double *uz,
                                        unsigned *status, cudaStream_t s)
{
    const bool hi = a.N > GLBM_MAXN_2N1;
    if (a.prec == GLBM_FP64)
        return hi ? launch_eq<F64, GLBM_MAXN>(a, f, rho, ux, uy, uz, status, s)
                  : launch_eq<F64, GLBM_MAXN_2N1>(a, f, rho, ux, uy, uz, status, s);
    return hi ? launch_eq<F32, GLBM_MAXN>(a, f, rho, ux, uy, uz, status, s)
              : launch_eq<F32, GLBM_MAXN_2N1>(a, f, rho, ux, uy, uz, status, s);
}
