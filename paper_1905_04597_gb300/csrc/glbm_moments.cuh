// Moments of the streamed state S(X) of 2D and 3D lattices (Sec. 2 for rho and
// u; temperature, heat flux and shear stress as central moments), one pass over
// the pulled populations.
//
// Every field is a combination of raw moments sum xi_x^p xi_y^q xi_z^r f with
// p + q + r <= 3. A thread owns a node (nodes are flattened over the lattice, so
// a narrow lattice fills its warps too) and walks the velocity rows (iz, iy);
// each row gives R_p = sum_ix xi_x^p v, p = 0..3, from mirror column pairs
// (+c, -c): the even powers take the pair's sum, the odd ones its difference.
//
// What bounds it: GB300 issues 2 FP64 instructions per cycle and SM (one warp
// instruction in 64 cycles per sub-partition; a float <-> double conversion
// takes the same slot), so a D2Q81 node at 4.5 FP64 instructions per population
// costs ten times its HBM time. FP32 deviations are therefore summed as exact
// integers: v = d0 2^-u0 + d1 2^-u1 + r, with the two integer digits taken by
// adding a power of two (the low mantissa bits of v + 1.5 2^k are the digit) and
// an exact float remainder |r| <= 2^-(u1+1). The row sums and the sums over the
// rows of d0 and d1 are integer arithmetic without any rounding, the remainders'
// sums are plain floats whose rounding lies 2^-24 below 2^-u1: as close to the
// exact sums of the stored floats as FP64 accumulation. The integers become
// doubles once per node and moment. The FP64 pipe is left with about 60
// instructions per node. Measured on GB300 against one pass with FP64 accumulation
// and runtime levels, wall densities repeated by every node near a wall: D2Q81
// 512 x 256 FP32 173 -> 36 us, FP64 138 -> 102 us; D2Q289 1024 x 128 FP32
// 585 -> 92 us; D3Q125 250 x 61 x 45 FP32 1844 -> 214 us; the wall densities add 5
// to 19 us as a launch of their own, which the moments' launch overlaps: it starts
// once the first has waited for the state, and waits for the densities after its sums
// (64 channels of 64 columns, all moments of every instance: 1491 -> 910 us; D2Q81
// 512 x 256, three instances 137 -> 107 us; D2Q289 1024 x 128, eight 885 -> 910 us).
#pragma once
#include "glbm_device.cuh"

// The arguments of one instance's moments.
struct MomArgs {
    const void *f;          // populations of the instance
    const InstParams *ip;
    const double *rw;       // wall densities [2][columns] (k_moment_walls), or null: no walls
    double *out[9];         // rho, ux, uy, T, qx, qy, sxy, uz, qz; null: not wanted
    int Lx, Ly, Lz, pitch, bc;
    int N, zv;              // the y axis (its velocities may differ from the x axis's)
    int plane;              // elements per velocity plane
    double vy[GLBM_MAXQA];  // velocities of the y axis
    double mx[3], my[3];    // sums of W xi^p, p = 0, 2, of the x and the y (z) axis
    double rest[3];         // rho, Pxx and Pyy of the rest weights
    double sw[GLBM_MAXQA][4];  // sum of W^y xi_y^q over xi_y > d, q = 0..3
};

// Number of raw moments: rho, j, P_ab, M_a = sum xi_a |xi|^2 f.
template <int DIM>
__host__ __device__ constexpr int mom_count(bool full)
{
    return full ? (DIM == 3 ? 13 : 8) : (DIM == 3 ? 4 : 3);
}
// Their order: rho, jx, jy, [jz,] then Pxx, Pyy, Pxy, Mx, My (2D) or
// Pxx, Pyy, Pxy, Pzz, Pxz, Pyz, Mx, My, Mz (3D).

// The weights of a row's R_p in every raw moment it feeds: add(k, w, p) adds
// w R_p to moment k. W is int or double (the row's velocities as W).
template <int DIM, bool FULL, class W, class F>
__device__ __forceinline__ void mom_row_terms(W cy, W cz, F &&add)
{
    add(0, W(1), 0);
    add(1, W(1), 1);
    add(2, cy, 0);
    if constexpr (DIM == 3) add(3, cz, 0);
    if constexpr (FULL) {
        const W y2 = cy * cy;
        if constexpr (DIM == 2) {
            add(3, W(1), 2);
            add(4, y2, 0);
            add(5, cy, 1);
            add(6, W(1), 3);
            add(6, y2, 1);
            add(7, cy, 2);
            add(7, cy * y2, 0);
        } else {
            const W z2 = cz * cz, s2 = y2 + z2;
            add(4, W(1), 2);
            add(5, y2, 0);
            add(6, cy, 1);
            add(7, z2, 0);
            add(8, cz, 1);
            add(9, cy * cz, 0);
            add(10, W(1), 3);
            add(10, s2, 1);
            add(11, cy, 2);
            add(11, cy * s2, 0);
            add(12, cz, 2);
            add(12, cz * s2, 0);
        }
    }
}

// ---- accumulation in FP64 --------------------------------------------------
// FP64 populations, and FP32 deviations outside the digits' range.
template <int DIM, int NX, int ZX, bool FULL>
struct MomAccD {
    using AX = AxisVel<NX, ZX>;
    static constexpr int NM = mom_count<DIM>(FULL);
    static constexpr bool DIGITS = false;
    double m[NM];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int k = 0; k < NM; ++k) m[k] = 0.0;
    }
    template <typename T>
    __device__ __forceinline__ void row(const T (&v)[AX::Q], double cy, double cz)
    {
        double R[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int p = AX::M0; p <= NX; ++p) {
            const double vp = (double)v[AX::ipos(p)], vm = (double)v[AX::ineg(p)];
            const double c = AX::vmag(p);
            const double s = vp + vm, d = vp - vm;
            R[0] += s;
            R[1] = fma(c, d, R[1]);
            if (FULL) {
                R[2] = fma(c * c, s, R[2]);
                R[3] = fma(c * c * c, d, R[3]);
            }
        }
        if (!ZX) R[0] += (double)v[NX];
        mom_row_terms<DIM, FULL>(cy, cz, [&](int k, double w, int p) { m[k] = fma(w, R[p], m[k]); });
    }
};

// ---- accumulation of FP32 deviations in integer digits ---------------------
// Weight sums that bound the digits: 2 sum c^2 and 2 sum c^3 over the x speeds (a
// row), and the largest sum over the whole lattice of |xi_a| |xi|^2 when every
// axis has the x axis's velocities.
template <int DIM, int NX, int ZX>
__host__ __device__ constexpr double mom_weight(int what)
{
    using AX = AxisVel<NX, ZX>;
    double s1 = 0, s2 = 0, s3 = 0;
    for (int p = AX::M0; p <= NX; ++p) {
        const double c = AX::vmag(p);
        s1 += 2 * c;
        s2 += 2 * c * c;
        s3 += 2 * c * c * c;
    }
    const double q = AX::Q;
    return what == 2 ? s2 : DIM == 3 ? s3 * q * q + 2 * s1 * s2 * q : s3 * q + s1 * s2;
}
// Largest B with w 2^B < 2^31 (1 % to spare), at most 20.
__host__ __device__ constexpr int mom_bits(double w)
{
    int b = 20;
    while (1.01 * w * (double)(1u << b) >= 2147483648.0) --b;
    return b;
}

template <int DIM, int NX, int ZX, bool FULL>
struct MomAccI {
    using AX = AxisVel<NX, ZX>;
    static constexpr int NM = mom_count<DIM>(FULL);
    static constexpr bool DIGITS = true;
    // Digits of B bits: |d0|, |d1| <= 2^B for |v| < 2^(1-E). Low levels keep every
    // sum of the lattice in 32 bits; where that would leave fewer than 17 bits
    // (or the y level may be higher than the x level's: D1Q3 along x) the sums
    // over the rows are 64-bit, and sum c^3 is formed at the end from column sums
    // over the rows, so that a row's largest weight sum is that of c^2.
    static constexpr int B32 = mom_bits(mom_weight<DIM, NX, ZX>(3));
    static constexpr bool WIDE = DIM == 2 && (B32 < 17 || (NX == 1 && !ZX));
    static constexpr bool COLS = FULL && WIDE && NX > 1;
    static constexpr int B = WIDE ? mom_bits(mom_weight<DIM, NX, ZX>(2)) : B32;
    // |v| < 2 (rest weights up to 4/9) or, from level 3 on, 1/4 (below 1/12)
    static constexpr int E = NX >= 3 || ZX ? 3 : 0;
    static constexpr int U0 = B - 1 + E, U1 = U0 + B + 1;
    static constexpr int NC = COLS ? NX + ZX : 1;  // column pairs
    using I = std::conditional_t<WIDE, long long, int>;

    I a0[NM], a1[NM];
    float r[NM];
    int c0[NC], c1[NC];  // column sums of v(+c) - v(-c)
    float cr[NC];
    unsigned seen;  // or of d0 + 2^B: bits above B are set by values out of range

    __device__ __forceinline__ void init()
    {
        seen = 0u;
#pragma unroll
        for (int k = 0; k < NM; ++k) {
            a0[k] = 0;
            a1[k] = 0;
            r[k] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            c0[k] = 0;
            c1[k] = 0;
            cr[k] = 0.f;
        }
    }
    static __device__ __forceinline__ float M(int u) { return 1.5f * (float)(1 << 23) / (float)(1LL << u); }
    __device__ __forceinline__ void row(const float (&v)[AX::Q], int cy, int cz)
    {
        const float M0 = M(U0), M1 = M(U1);
        const unsigned b0 = __float_as_uint(M0), b1 = __float_as_uint(M1), lo = b0 - (1u << B);
        const f32x2 M02 = pk2(M0, M0), M12 = pk2(M1, M1);
        unsigned R[4][2] = {{0u, 0u}, {0u, 0u}, {0u, 0u}, {0u, 0u}};
        float q[4] = {0.f, 0.f, 0.f, 0.f};
        unsigned n0 = 0, n2 = 0;  // how often the bias entered R_0 and R_2
#pragma unroll
        for (int p = AX::M0; p <= NX; ++p) {
            const unsigned c = AX::vmag(p);
            // the digits of a pair, as the bits of v + M (biased by M's), and the
            // exact remainders
            const f32x2 vv = pk2(v[AX::ipos(p)], v[AX::ineg(p)]);
            const f32x2 t0 = add2(vv, M02);
            const f32x2 r0 = sub2(vv, sub2(t0, M02));
            const f32x2 t1 = add2(r0, M12);
            const f32x2 rem = sub2(r0, sub2(t1, M12));
            const unsigned p0 = __float_as_uint(lo2(t0)), m0 = __float_as_uint(hi2(t0));
            const unsigned p1 = __float_as_uint(lo2(t1)), m1 = __float_as_uint(hi2(t1));
            seen |= (p0 - lo) | (m0 - lo);
            const unsigned s0 = p0 + m0, d0 = p0 - m0, s1 = p1 + m1, d1 = p1 - m1;
            const float sr = lo2(rem) + hi2(rem), dr = lo2(rem) - hi2(rem);
            R[0][0] += s0;
            R[0][1] += s1;
            R[1][0] += c * d0;
            R[1][1] += c * d1;
            q[0] += sr;
            q[1] = fmaf((float)c, dr, q[1]);
            n0 += 2;
            if (FULL) {
                R[2][0] += c * c * s0;
                R[2][1] += c * c * s1;
                q[2] = fmaf((float)(c * c), sr, q[2]);
                n2 += 2 * c * c;
                if constexpr (COLS) {
                    c0[p - AX::M0] += (int)d0;
                    c1[p - AX::M0] += (int)d1;
                    cr[p - AX::M0] += dr;
                } else {
                    R[3][0] += c * c * c * d0;
                    R[3][1] += c * c * c * d1;
                    q[3] = fmaf((float)(c * c * c), dr, q[3]);
                }
            }
        }
        if (!ZX) {
            const float v0 = v[NX];
            const float t0 = v0 + M0, r0 = v0 - (t0 - M0), t1 = r0 + M1;
            seen |= __float_as_uint(t0) - lo;
            q[0] += r0 - (t1 - M1);
            R[0][0] += __float_as_uint(t0);
            R[0][1] += __float_as_uint(t1);
            n0 += 1;
        }
        // the biases leave (arithmetic modulo 2^32; the true sums fit)
        R[0][0] -= n0 * b0;
        R[0][1] -= n0 * b1;
        if (FULL) {
            R[2][0] -= n2 * b0;
            R[2][1] -= n2 * b1;
        }
        mom_row_terms<DIM, FULL>(cy, cz, [&](int k, int w, int p) {
            if (COLS && p == 3) return;
            a0[k] += (I)(int)R[p][0] * w;
            a1[k] += (I)(int)R[p][1] * w;
            r[k] = fmaf((float)w, q[p], r[k]);
        });
    }
    // sum c^3 of the column sums joins the moment M_x (number 6 in 2D)
    __device__ __forceinline__ void close()
    {
        if constexpr (COLS) {
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const int c = AX::vmag(k + AX::M0), c3 = c * c * c;
                a0[6] += (I)c0[k] * c3;
                a1[6] += (I)c1[k] * c3;
                r[6] = fmaf((float)c3, cr[k], r[6]);
            }
        }
    }
    __device__ __forceinline__ bool in_range() const { return seen < (2u << B); }
    __device__ __forceinline__ double total(int k) const
    {
        const long long a = ((long long)a0[k] << (U1 - U0)) + (long long)a1[k];
        return fma((double)a, 1.0 / (double)(1LL << U1), f2d(r[k]));
    }
};

// j / rho from inv, the rounded 1 / rho, by one correction with the exact residual
// (Markstein's scheme: with a correctly rounded reciprocal the result is the
// division's but for rare operands, with another one, as 3 rho's below, within an ulp);
// the division itself where the correction is not finite.
__device__ __forceinline__ double mom_div(double j, double rho, double inv)
{
    double q = j * inv;
    q = fma(fma(-rho, q, j), inv, q);
    if ((__double2hiint(q) & 0x7FF00000) == 0x7FF00000) q = j / rho;
    return q;
}

// Raw moments of one node over the pulled velocity rows row0, row0 + step, ...
// (rows emitted by a wall are left out).
template <class ACC, int DIM, int NX, int ZX, typename T>
__device__ __forceinline__ void mom_node(const MomArgs &a, int x, int y, int z, int row0, int step,
                                         ACC &acc)
{
    using AX = AxisVel<NX, ZX>;
    constexpr int QX = AX::Q;
    const T *const f = static_cast<const T *>(a.f);
    const bool walls = a.bc == GLBM_BC_WALLS;
    // the y axis (3D lattices: the x axis's level, known at compile time)
    const int N = DIM == 3 ? NX : a.N, zv = DIM == 3 ? 0 : a.zv;
    const int Qy = 2 * N + 1 + zv;
    const int vmax = zv ? 2 * N + 1 : N;
    const int rows = DIM == 3 ? Qy * Qy : Qy;
    int cofs[QX];
#pragma unroll
    for (int ix = 0; ix < QX; ++ix)
        cofs[ix] = ix * a.plane + wrap_shift(x - AX::vel(ix), a.Lx, a.Lx > AX::VMAX);
    auto place = [&](int j, int &cy, int &cz, bool &in) {
        const int iz = DIM == 3 ? j / Qy : 0, iy = DIM == 3 ? j - iz * Qy : j;
        cy = zv ? 2 * iy - (2 * N + 1) : iy - N;
        cz = DIM == 3 ? iz - N : 0;
        const int ys = y - cy;
        in = !walls || (ys >= 0 && ys < a.Ly);
        int src = walls ? min(max(ys, 0), a.Ly - 1) : wrap_shift(ys, a.Ly, a.Ly > vmax);
        if (DIM == 3) src += wrap_shift(z - cz, a.Lz, a.Lz > N) * a.Ly;
        return j * QX * a.plane + src * a.pitch;
    };
    T v[QX];
    int cy, cz;
    bool in;
    int base = place(row0 < rows ? row0 : 0, cy, cz, in);
#pragma unroll
    for (int ix = 0; ix < QX; ++ix) v[ix] = f[base + cofs[ix]];
#pragma unroll 1
    for (int j = row0; j < rows; j += step) {
        // the next row's loads are in flight while this row is summed
        T nv[QX];
        int ncy, ncz;
        bool nin;
        base = place(j + step < rows ? j + step : j, ncy, ncz, nin);
#pragma unroll
        for (int ix = 0; ix < QX; ++ix) nv[ix] = f[base + cofs[ix]];
        if (in) {
            if constexpr (ACC::DIGITS) {
                acc.row(v, cy, cz);
            } else {
                const int iz = DIM == 3 ? j / Qy : 0, iy = DIM == 3 ? j - iz * Qy : j;
                acc.row(v, a.vy[iy], DIM == 3 ? a.vy[iz] : 0.0);
            }
        }
        cy = ncy;
        cz = ncz;
        in = nin;
#pragma unroll
        for (int ix = 0; ix < QX; ++ix) v[ix] = nv[ix];
    }
}

// The same entirely in FP64, for a node with a deviation outside the digits'
// range: rare, so kept out of the kernel's own code.
template <int DIM, int NX, int ZX, typename T, bool FULL>
__device__ __noinline__ void mom_node_slow(const MomArgs &a, int x, int y, int z, int row0, int step,
                                           double (&m)[mom_count<DIM>(FULL)])
{
    MomAccD<DIM, NX, ZX, FULL> acc;
    acc.init();
    mom_node<MomAccD<DIM, NX, ZX, FULL>, DIM, NX, ZX, T>(a, x, y, z, row0, step, acc);
#pragma unroll
    for (int k = 0; k < mom_count<DIM>(FULL); ++k) m[k] = acc.m[k];
}

// The rows emitted by one wall at distance d from it (d = 0 the row next to it;
// sg = 1 the wall at y = -1/2, -1 the other): every velocity with sg xi_y > d.
// Their populations are rho_w E^x(u_w) W^y (W^z), so their raw moments are
// products of K_p = sum E^x xi_x^p, s_q = sum_{emitted} W^y xi_y^q and the z axis's
// rest moments; FP32 deviations take out the rest weights' m_p.
template <int DIM, bool DEV, bool FULL>
__device__ __forceinline__ void mom_emitted(const MomArgs &a, const double *K, double rw, int d,
                                            double sg, double (&m)[mom_count<DIM>(FULL)])
{
    double P[4], s[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        P[p] = rw * K[p];
        if (DEV && (p == 0 || p == 2)) P[p] -= a.mx[p];
        s[p] = (p & 1) ? sg * a.sw[d][p] : a.sw[d][p];
    }
    m[0] = fma(P[0], s[0], m[0]);
    m[1] = fma(P[1], s[0], m[1]);
    m[2] = fma(P[0], s[1], m[2]);
    if constexpr (FULL) {
        constexpr int k = DIM == 3 ? 4 : 3, kM = DIM == 3 ? 10 : 6;
        m[k] = fma(P[2], s[0], m[k]);
        m[k + 1] = fma(P[0], s[2], m[k + 1]);
        m[k + 2] = fma(P[1], s[1], m[k + 2]);
        m[kM] += fma(P[3], s[0], P[1] * s[2]);
        m[kM + 1] += fma(P[2], s[1], P[0] * s[3]);
        if constexpr (DIM == 3) {
            const double z2 = a.my[2];
            m[7] = fma(P[0] * s[0], z2, m[7]);
            m[kM] = fma(P[1] * s[0], z2, m[kM]);
            m[kM + 1] = fma(P[0] * s[1], z2, m[kM + 1]);
        }
    }
}

constexpr int MOM_WARPS = 4;  // warps per CTA

// S warps share the rows of 32 nodes (S = 1, 2, 4, by the number of rows); their
// sums meet in shared memory in slice order, the integer digits as they are.
template <int DIM, int NX, int ZX, typename T, bool FULL>
__global__ void __launch_bounds__(32 * MOM_WARPS)
    k_moments_nd(const __grid_constant__ MomArgs a, int S)
{
    constexpr int NM = mom_count<DIM>(FULL);
    constexpr bool DEV = sizeof(T) == 4;
    using ACC = std::conditional_t<DEV, MomAccI<DIM, NX, ZX, FULL>, MomAccD<DIM, NX, ZX, FULL>>;
    extern __shared__ __align__(16) unsigned char smem[];
    df_launch_next();  // the next instance's wall launch queues up (it waits)
    if (a.bc != GLBM_BC_WALLS) wait_prior_grid();  // else k_moment_walls has done so
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int s = w % S;
    const int nodes = a.Lx * a.Ly * a.Lz;
    const int n = (blockIdx.x * (MOM_WARPS / S) + w / S) * 32 + lane;
    const int nc = n < nodes ? n : nodes - 1;
    const int zy = nc / a.Lx, x = nc - zy * a.Lx;
    const int z = DIM == 3 ? zy / a.Ly : 0, y = DIM == 3 ? zy - z * a.Ly : zy;

    ACC acc;
    acc.init();
    mom_node<ACC, DIM, NX, ZX, T>(a, x, y, z, s, S, acc);
    if constexpr (DEV) acc.close();
    if (S > 1) {
        ACC *const part = reinterpret_cast<ACC *>(smem);
        if (s > 0) {
            ACC &o = part[threadIdx.x];
            if constexpr (DEV) {
#pragma unroll
                for (int k = 0; k < NM; ++k) {
                    o.a0[k] = acc.a0[k];
                    o.a1[k] = acc.a1[k];
                    o.r[k] = acc.r[k];
                }
                o.seen = acc.seen;
            } else {
                o = acc;
            }
        }
        __syncthreads();
        if (s > 0) return;
        for (int t = 1; t < S; ++t) {
            const ACC &o = part[threadIdx.x + 32 * t];
            if constexpr (DEV) {
#pragma unroll
                for (int k = 0; k < NM; ++k) {
                    acc.a0[k] += o.a0[k];
                    acc.a1[k] += o.a1[k];
                    acc.r[k] += o.r[k];
                }
                acc.seen |= o.seen;
            } else {
#pragma unroll
                for (int k = 0; k < NM; ++k) acc.m[k] += o.m[k];
            }
        }
    }
    double m[NM];
    if constexpr (DEV) {
        if (acc.in_range()) {
#pragma unroll
            for (int k = 0; k < NM; ++k) m[k] = acc.total(k);
        } else {
            mom_node_slow<DIM, NX, ZX, T, FULL>(a, x, y, z, 0, 1, m);
        }
        // the rest weights' moments of the whole lattice (odd ones vanish)
        m[0] += a.rest[0];
        if constexpr (FULL) {
            constexpr int P = DIM == 3 ? 4 : 3;
            m[P] += a.rest[1];
            m[P + 1] += a.rest[2];
            if constexpr (DIM == 3) m[P + 3] += a.rest[2];  // the z axis's level is y's
        }
    } else {
#pragma unroll
        for (int k = 0; k < NM; ++k) m[k] = acc.m[k];
    }
    if (a.bc == GLBM_BC_WALLS) {
        wait_prior_grid();  // the wall densities
        const int vmax = a.zv ? 2 * a.N + 1 : a.N, col = z * a.Lx + x;
        if (y < vmax) mom_emitted<DIM, DEV, FULL>(a, a.ip->kw_lo, __ldcg(a.rw + col), y, 1.0, m);
        if (a.Ly - 1 - y < vmax)
            mom_emitted<DIM, DEV, FULL>(a, a.ip->kw_hi, __ldcg(a.rw + (a.Lx * a.Lz + col)), a.Ly - 1 - y,
                                         -1.0, m);
    }
    if (n >= nodes) return;
    const double rho = m[0], jx = m[1], jy = m[2];
    // u_x = (j_x + g/2) / rho with Guo's force (gx = 0 otherwise), so that
    // rho u_x = j_x + gx in the central moments below
    const double gx = a.ip->g_half;
    const double inv = 1.0 / rho;
    const double ux = mom_div(jx + gx, rho, inv), uy = mom_div(jy, rho, inv);
    if (a.out[0]) a.out[0][n] = rho;
    if (a.out[1]) a.out[1][n] = ux;
    if (a.out[2]) a.out[2][n] = uy;
    if constexpr (DIM == 3) {
        const double jz = m[3], uz = mom_div(jz, rho, inv);
        if (a.out[7]) a.out[7][n] = uz;
        if constexpr (FULL) {
            const double Pxx = m[4], Pyy = m[5], Pxy = m[6], Pzz = m[7], Pxz = m[8], Pyz = m[9];
            const double trP = Pxx + Pyy + Pzz, uj = fma(ux, jx, fma(uy, jy, uz * jz));
            const double e2 = trP - uj, h = trP - 2.0 * uj;
            const double qx = m[10] - ux * (h + 2.0 * Pxx) - 2.0 * fma(uy, Pxy, uz * Pxz);
            const double qy = m[11] - uy * (h + 2.0 * Pyy) - 2.0 * fma(ux, Pxy, uz * Pyz);
            const double qz = m[12] - uz * (h + 2.0 * Pzz) - 2.0 * fma(ux, Pxz, uy * Pyz);
            if (a.out[3]) a.out[3][n] = mom_div(e2, 3.0 * rho, inv * (1.0 / 3.0));
            if (a.out[4]) a.out[4][n] = 0.5 * qx;
            if (a.out[5]) a.out[5][n] = 0.5 * qy;
            if (a.out[6]) a.out[6][n] = fma(-ux, jy, Pxy);
            if (a.out[8]) a.out[8][n] = 0.5 * qz;
        }
    } else if constexpr (FULL) {
        const double Pxx = m[3], Pyy = m[4], Pxy = m[5];
        // sum c_a c_b f = P_ab - u_a j_b + (Guo: u gx), sum c_a |c|^2 f =
        // M_a - u_a (tr P + 2 P_aa - 2 u.j) - 2 u_b P_ab (- |u|^2 gx), c = xi - u
        const double trP = Pxx + Pyy, uj = fma(ux, jx, uy * jy), h = trP - 2.0 * uj;
        const double e2 = fma(ux, gx, trP - uj);
        const double sxy = fma(gx, uy, fma(-ux, jy, Pxy));
        const double qx = fma(-fma(ux, ux, uy * uy), gx,
                              m[6] - ux * (h + 2.0 * Pxx) - 2.0 * (uy * Pxy));
        const double qy = m[7] - uy * (h + 2.0 * Pyy) - 2.0 * (ux * Pxy);
        if (a.out[3]) a.out[3][n] = mom_div(0.5 * e2, rho, inv);
        if (a.out[4]) a.out[4][n] = 0.5 * qx;
        if (a.out[5]) a.out[5][n] = 0.5 * qy;
        if (a.out[6]) a.out[6][n] = sxy;
    }
}

// Wall densities of every column (x, z) of one instance in FP64, rho_w =
// absorbed mass / sum_{v>0} v W_v: out[h * columns + column], h = 0 the wall at
// y = -1/2. FP32 deviations: 1 + (sum of the absorbed deviations) / den. CTA:
// WALL_TX columns x 32 slices of the (speed, row) pairs of wall blockIdx.y; the
// slices' partial sums are added in a fixed order. Once per column, where the
// nodes within reach of a wall used to repeat the sums each for itself. Eight
// columns per CTA (one 32-byte sector) spread the sums over the chip.
constexpr int WALL_TX = 8, WALL_SL = 32;

template <int DIM, typename T>
__global__ void __launch_bounds__(WALL_TX *WALL_SL)
    k_moment_walls(const __grid_constant__ MomArgs a, int QX, int vx0, int vxs, double *out)
{
    __shared__ double part[WALL_SL][WALL_TX];
    wait_prior_grid();
    df_launch_next();  // k_moments_nd: its pulls need nothing of this launch
    const int h = blockIdx.y;
    const int tx = threadIdx.x % WALL_TX, sl = threadIdx.x / WALL_TX;
    const int cols = a.Lx * a.Lz;
    const int c = blockIdx.x * WALL_TX + tx, cc = c < cols ? c : cols - 1;
    const int z = DIM == 3 ? cc / a.Lx : 0, x = cc - z * a.Lx;
    const T *const f = static_cast<const T *>(a.f);
    const int Qy = 2 * a.N + 1 + a.zv, nz = DIM == 3 ? Qy : 1;
    const int npair = a.zv ? (a.N + 1) * (a.N + 1) : a.N * (a.N + 1) / 2;
    double D = 0.0;
    for (int i = sl; i < npair * nz; i += WALL_SL) {
        const int iz = DIM == 3 ? i / npair : 0;
        int m = a.zv ? 0 : 1, k = i - iz * npair;
        for (int v; k >= (v = a.zv ? 2 * m + 1 : m); ++m) k -= v;
        const int iy = h == 0 ? a.N - m : (a.zv ? a.N + 1 + m : a.N + m);
        int row = h == 0 ? k : a.Ly - 1 - k;
        if (DIM == 3) row += wrap_index(z - (iz - a.N), a.Lz) * a.Ly;
        const T *const p = f + ((iz * Qy + iy) * QX * a.plane + row * a.pitch);
#pragma unroll 6
        for (int ix = 0; ix < QX; ++ix)
            D += (double)p[ix * a.plane + wrap_index(x - (vx0 + vxs * ix), a.Lx)];
    }
    part[sl][tx] = D;
    __syncthreads();
    for (int st = WALL_SL / 2; st > 0; st >>= 1) {
        if (sl < st) part[sl][tx] += part[sl + st][tx];
        __syncthreads();
    }
    if (sl == 0 && c < cols) {
        const double v = part[0][tx] * a.ip->inv_den;
        out[(long long)h * cols + c] = sizeof(T) == 4 ? 1.0 + v : v;
    }
}

// Launch of one lattice kind: x level NX (ZX: 2N+2 hierarchy), 2D or 3D.
template <int DIM, int NX, int ZX>
cudaError_t launch_moments_kind(const MomArgs &a, int prec, bool full, cudaStream_t s)
{
    // Warps per 32 nodes, by the number of rows alone (so that a node's sums do
    // not depend on the lattice's size): long nodes are split for occupancy and
    // for the latency of small lattices.
    const int groups = (a.Lx * a.Ly * a.Lz + 31) / 32;
    const int rows = 2 * a.N + 1 + a.zv;
    const int S = DIM == 3 || rows < 8 ? 1 : (rows < 16 ? 2 : 4);
    const int blocks = (groups + MOM_WARPS / S - 1) / (MOM_WARPS / S);
    const dim3 b(32 * MOM_WARPS);
    const auto smem = [&](size_t acc) { return S > 1 ? b.x * acc : (size_t)0; };
    if (prec == GLBM_FP64) {
        if (full)
            return launch_serialized_smem(k_moments_nd<DIM, NX, ZX, double, true>, dim3(blocks), b,
                                          smem(sizeof(MomAccD<DIM, NX, ZX, true>)), s, a, S);
        return launch_serialized_smem(k_moments_nd<DIM, NX, ZX, double, false>, dim3(blocks), b,
                                      smem(sizeof(MomAccD<DIM, NX, ZX, false>)), s, a, S);
    }
    if (full)
        return launch_serialized_smem(k_moments_nd<DIM, NX, ZX, float, true>, dim3(blocks), b,
                                      smem(sizeof(MomAccI<DIM, NX, ZX, true>)), s, a, S);
    return launch_serialized_smem(k_moments_nd<DIM, NX, ZX, float, false>, dim3(blocks), b,
                                  smem(sizeof(MomAccI<DIM, NX, ZX, false>)), s, a, S);
}
cudaError_t glbm_moments_2n1(int NX, const MomArgs &a, int prec, bool full, cudaStream_t s);
cudaError_t glbm_moments_2n2(int NX, const MomArgs &a, int prec, bool full, cudaStream_t s);
