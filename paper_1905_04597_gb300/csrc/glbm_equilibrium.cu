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
// instead: the result is rounded to float once from a value exact to 2^-46 of its
// terms, which differs from the rounding of the FP64 value about once in 2^20
// populations, at a tie. Fields outside 1e-18..1e18 in magnitude (or not finite)
// take FP64 per node. Measured on GB300, FP32: D2Q81 512 x 256 95 -> 26 us, D2Q289
// 1024 x 128 311 -> 75 us, D3Q125 250 x 61 x 45 815 -> 227 us, D1Q3 x D1Q28 200 nodes
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

// Table of one axis in the arithmetic's values: rest weights by velocity index, and
// the even and odd coefficients of every mirror pair (Ce[m][i], i = 0..N-1 for v^(i+1)).
template <class V>
struct EqAxis {
    int N, zv;
    V W[GLBM_MAXQA];
    V Ce[GLBM_MAXN + 1][GLBM_MAXN], Co[GLBM_MAXN + 1][GLBM_MAXN];
};
template <class V>
struct EqArgs {
    EqAxis<V> y, x;  // 3D: y holds for z too
    const double *rho, *u[3];  // null: 1, 0
    void *f;
    int Lx, nodes, pitch, dims;
    long long plane;
};

// E - W of the mirror pair m of one axis (plus: the positive velocity).
template <class P>
__device__ __forceinline__ void eq_pair(const EqAxis<typename P::V> &t, int m, typename P::V u,
                                        typename P::V &plus, typename P::V &minus)
{
    using V = typename P::V;
    const int N = t.N;
    const V v = P::mul(u, u);
    V e = t.Ce[m][N - 1], o = t.Co[m][N - 1];
    for (int i = N - 2; i >= 0; --i) {
        e = P::fma_(e, v, t.Ce[m][i]);
        o = P::fma_(o, v, t.Co[m][i]);
    }
    e = P::mul(e, v);
    if (m == 0 && !t.zv) {  // the zero velocity
        plus = minus = e;
        return;
    }
    plus = P::fma_(u, o, e);
    minus = P::fma_(P::neg(u), o, e);
}

// W^x B + d^x A rounded once to float.
__device__ __forceinline__ float eq_dev(df w, df B, df d, df A)
{
    const float p = __fmul_rn(w.h, B.h), q = __fmul_rn(d.h, A.h);
    const float pe = fmaf(w.l, B.h, fmaf(w.h, B.l, fmaf(w.h, B.h, -p)));
    const float qe = fmaf(d.l, A.h, fmaf(d.h, A.l, fmaf(d.h, A.h, -q)));
    const float s = p + q, t = s - p;
    const float e = (p - (s - t)) + (q - t);
    return s + (e + (pe + qe));
}

constexpr int EQ_WARPS = 4;

// One node of FP32 storage entirely in FP64 (out-of-range fields).
__device__ __noinline__ void eq_node_f64(const EqArgs<df> &a, int n, long long base)
{
    const int Qx = 2 * a.x.N + 1 + a.x.zv, Qy = a.dims >= 2 ? 2 * a.y.N + 1 + a.y.zv : 1;
    const int Qz = a.dims == 3 ? Qy : 1;
    const auto val = [](df t) { return (double)t.h + (double)t.l; };
    const auto dev = [&](const EqAxis<df> &t, double u, int i) {
        const int vel = t.zv ? 2 * i - (2 * t.N + 1) : i - t.N, av = vel < 0 ? -vel : vel;
        const int m = t.zv ? (av - 1) / 2 : av;
        const double v = u * u;
        double e = 0.0, o = 0.0;
        for (int k = t.N - 1; k >= 0; --k) {
            e = fma(e, v, val(t.Ce[m][k]));
            o = fma(o, v, val(t.Co[m][k]));
        }
        e *= v;
        return vel == 0 ? e : fma(vel > 0 ? u : -u, o, e);
    };
    const double r = a.rho ? a.rho[n] : 1.0, ux = a.u[0] ? a.u[0][n] : 0.0;
    const double uy = a.u[1] ? a.u[1][n] : 0.0, uz = a.u[2] ? a.u[2][n] : 0.0;
    float *const out = static_cast<float *>(a.f) + base;
    for (int iz = 0; iz < Qz; ++iz) {
        const double wz = a.dims == 3 ? val(a.y.W[iz]) : 1.0;
        const double dz = a.dims == 3 ? dev(a.y, uz, iz) : 0.0;
        for (int iy = 0; iy < Qy; ++iy) {
            const double wy = a.dims >= 2 ? val(a.y.W[iy]) : 1.0;
            const double dy = a.dims >= 2 ? dev(a.y, uy, iy) : 0.0;
            const double A = r * ((wy + dy) * (wz + dz));
            const double B = fma(r - 1.0, wy * wz, r * fma(dy, wz + dz, wy * dz));
            for (int ix = 0; ix < Qx; ++ix)
                out[(long long)((iz * Qy + iy) * Qx + ix) * a.plane] =
                    (float)fma(dev(a.x, ux, ix), A, val(a.x.W[ix]) * B);
        }
    }
}

template <class P>
__global__ void __launch_bounds__(32 * EQ_WARPS) k_equilibrium(const __grid_constant__ EqArgs<typename P::V> a)
{
    using V = typename P::V;
    constexpr bool F = std::is_same<V, df>::value;  // float pairs
    __shared__ V in[5][32];                  // u_x, u_y, u_z, rho, rho - 1
    __shared__ V dx[GLBM_MAXQA][32];         // FP32: E^x - W^x; FP64: E^x
    __shared__ V dy[GLBM_MAXQA][32], dz[2 * GLBM_MAXN_3D + 1][32];
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
        const EqAxis<V> &tab = ax == 0 ? a.x : a.y;
        V plus, minus;
        eq_pair<P>(tab, m, in[ax][lane], plus, minus);
        const int ip = tab.zv ? tab.N + 1 + m : tab.N + m, im = tab.N - m;
        if (!F && ax == 0) {
            plus = P::add(tab.W[ip], plus);
            minus = P::add(tab.W[im], minus);
        }
        V(*const d)[32] = ax == 0 ? dx : ax == 1 ? dy : dz;
        d[im][lane] = minus;
        d[ip][lane] = plus;
    }
    __syncthreads();
    const int Qx = 2 * a.x.N + 1 + a.x.zv, Qy = a.dims >= 2 ? 2 * a.y.N + 1 + a.y.zv : 1;
    const int rows = a.dims == 3 ? Qy * Qy : Qy;
    const V r = in[3][lane], r1 = in[4][lane];
    const bool live = n < a.nodes && !((bad >> lane) & 1u);
    for (int j = w; j < rows; j += EQ_WARPS) {
        V A = r, B = r1;
        if (a.dims >= 2) {
            const int iz = a.dims == 3 ? j / Qy : 0, iy = j - iz * Qy;
            const V wy = a.y.W[iy], d = dy[iy][lane], E = P::add(wy, d);
            if (a.dims == 2) {
                A = P::mul(r, E);
                if (F) B = P::fma_(r1, wy, P::mul(r, d));
            } else {
                const V wz = a.y.W[iz], e = dz[iz][lane], Ez = P::add(wz, e);
                A = P::mul(r, P::mul(E, Ez));
                if (F) B = P::fma_(r1, P::mul(wy, wz), P::mul(r, P::fma_(d, Ez, P::mul(wy, e))));
            }
        }
        if (!live) continue;
        const long long o = base + (long long)(j * Qx) * a.plane;
        if constexpr (F) {
            float *out = static_cast<float *>(a.f) + o;
#pragma unroll 3
            for (int ix = 0; ix < Qx; ++ix, out += a.plane)
                *out = eq_dev(a.x.W[ix], B, dx[ix][lane], A);
        } else {
            double *out = static_cast<double *>(a.f) + o;
#pragma unroll 3
            for (int ix = 0; ix < Qx; ++ix, out += a.plane) *out = dx[ix][lane] * A;
        }
    }
    if constexpr (F) {
        if (w == 0 && n < a.nodes && ((bad >> lane) & 1u)) eq_node_f64(a, n, base);
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

template <class V>
void fill_axis(const AxisTableHi &t, EqAxis<V> &e)
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
}

template <class P>
cudaError_t launch_eq(const AuxArgs &a, void *f, const double *rho, const double *ux,
                      const double *uy, const double *uz, cudaStream_t s)
{
    EqArgs<typename P::V> e = {};
    fill_axis(a.tab, e.y);
    fill_axis(a.dims == 2 ? a.tabx : a.tab, e.x);
    e.rho = rho;
    e.u[0] = ux;
    e.u[1] = a.dims >= 2 ? uy : nullptr;
    e.u[2] = a.dims == 3 ? uz : nullptr;
    e.f = f;
    e.Lx = a.Lx;
    e.nodes = a.Lx * a.Ly * a.Lz;
    e.pitch = a.pitch;
    e.dims = a.dims;
    e.plane = a.plane;
    k_equilibrium<P><<<(e.nodes + 31) / 32, 32 * EQ_WARPS, 0, s>>>(e);
    return cudaGetLastError();
}

}  // namespace

cudaError_t glbm_launch_set_equilibrium(const AuxArgs &a, void *f, const double *rho,
                                        const double *ux, const double *uy, const double *uz,
                                        cudaStream_t s)
{
    return a.prec == GLBM_FP64 ? launch_eq<F64>(a, f, rho, ux, uy, uz, s)
                               : launch_eq<F32>(a, f, rho, ux, uy, uz, s);
}
