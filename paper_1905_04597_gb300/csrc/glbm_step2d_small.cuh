// The fused FP64 2D step of small lattices (the same step as glbm_step2d.cuh, with
// the linearised force), spread over as many SMs as its work allows.
//
// An FP64 warp instruction takes its SM sub-partition's pipe for 64 cycles whatever
// its active lanes, so on a lattice too small to fill the chip the tiles' step time
// is the number of FP64 instructions of one warp: a warp of 32 columns x several
// velocity rows runs several hundred (16.5 us at D2Q81 40 x 24, 80 us for D1Q3 x
// D1Q28 at 1 x 200, where 31 of 32 lanes repeat one column). Here a thread holds
// one velocity row of one node: NB = 8 consecutive nodes of the flattened lattice
// (y Lx + x) x Q_y rows per CTA, about 80 FP64 instructions per thread, one to two
// warps per sub-partition. The coefficients a thread needs (one row of each axis's
// table) are loaded before the wait for the previous step. The wall densities of a
// node's column are summed by its own threads, with no launch of their own.
//
// Every sum is taken in the order of the tile with G0 warp groups (the level's
// default) and of k_wall_rho, so the results are those of the tiles bit for bit.
// Measured on GB300, us per step in 64-step graphs, against the tiles: D2Q81 40 x 24
// 20.4 -> 8.0, D1Q3 x D1Q28 5 x (1 x 200) 106.6 -> 12.7 (choose_small, glbm_api.cpp).
#pragma once
#include "glbm_step2d_launch.cuh"

constexpr int SMALL_NB = 8;  // nodes per CTA

template <int N, int NXL, int ZY, int ZX, int G0>
__global__ void __launch_bounds__((SMALL_NB * AxisVel<N, ZY>::Q + 31) / 32 * 32)
    k_step2d_small(const __grid_constant__ SmallArgs a)
{
    using AY = AxisVel<N, ZY>;
    using AX = AxisVel<NXL, ZX>;
    using S = Step2D<N, double, 1, 1, NXL, ZY, ZX>;
    constexpr int Q1 = AY::Q, QX = AX::Q, NB = SMALL_NB, NV = S::NV;
    __shared__ double rs[Q1][NB], jr[Q1][NB];      // row sums of f and of xi_x f
    __shared__ double part[3 * G0][NB], tot[3][NB];  // rho, j_x, j_y: per group, total
    __shared__ double ex[QX][NB];                  // E^x
    __shared__ double dsum[2 * NV][NB], rw[2][NB];  // wall fluxes (lower, upper), densities
    const int j = threadIdx.x % NB, i = threadIdx.x / NB;  // node of the CTA, velocity row
    const bool row = i < Q1;
    const int iy = row ? i : Q1 - 1;
    const int inst = blockIdx.y;
    const int nodes = a.Lx * a.Ly, n0 = blockIdx.x * NB;
    const int n = n0 + j < nodes ? n0 + j : nodes - 1;
    const int y = n / a.Lx, x = n - y * a.Lx;
    const int ny = AY::vel(iy), my = ZY ? ((ny < 0 ? -ny : ny) - 1) / 2 : (ny < 0 ? -ny : ny);
    const int mx = i <= NXL ? i : NXL;

    // this thread's coefficients: E^y of its row, E^x of the mirror pair number i
    double cey[N], coy[N], cex[NXL], cox[NXL];
    const AxisTableHi &ty = *a.ty, &tx = *a.tx;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        cey[k] = ty.Ce[my][k + 1];
        coy[k] = ty.Co[my][k];
    }
#pragma unroll
    for (int k = 0; k < NXL; ++k) {
        cex[k] = tx.Ce[mx][k + 1];
        cox[k] = tx.Co[mx][k];
    }
    const double wy = ty.W[iy], wx = tx.W[AX::ipos(mx)];
    const InstParams &ip = a.ip[inst];
    const double om = ip.omega, gto = ip.g_theta_om;

    wait_prior_grid();
    df_launch_next();  // the next step's CTAs load their coefficients meanwhile
    const bool live = !step_halted(a.status);
    const double *const fin = a.fin + (long long)inst * a.inst_stride;
    double *const fout = a.fout + (long long)inst * a.inst_stride;
    const bool walls = a.bc == GLBM_BC_WALLS;
    int cofs[QX];
#pragma unroll
    for (int ix = 0; ix < QX; ++ix)
        cofs[ix] = ix * a.plane + wrap_shift(x - AX::vel(ix), a.Lx, a.Lx > AX::VMAX);
    // the pull of this row (a row out of the walls loads the edge row)
    const int ys = y - ny;
    const int yc = walls ? min(max(ys, 0), a.Ly - 1) : wrap_shift(ys, a.Ly, a.Ly > AY::VMAX);
    double f[QX];
    {
        const double *const p = fin + (iy * QX * a.plane + yc * a.pitch);
#pragma unroll
        for (int ix = 0; ix < QX; ++ix) f[ix] = p[cofs[ix]];
    }
    // wall densities of the column: the NV accumulators of each wall dealt to the
    // node's threads (order of additions: Step2D::wall_densities)
    const bool need_lo = walls && y < AY::VMAX, need_hi = walls && y >= a.Ly - AY::VMAX;
    if (__syncthreads_or(need_lo || need_hi)) {
        constexpr int U = QX >= 24 ? 1 : 24 / QX;
        for (int acc = i; acc < 2 * NV && row; acc += Q1) {
            const int h = acc / NV, v = acc - h * NV;
            if (!(h == 0 ? need_lo : need_hi)) continue;
            double s = 0.0;
#pragma unroll 1
            for (int p0 = v; p0 < AY::NPAIR; p0 += U * NV) {
                double val[U][QX];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int p = p0 + u * NV;
                    if (p < AY::NPAIR) {
                        int m = AY::M0, k = p;
                        while (k >= AY::vmag(m)) k -= AY::vmag(m++);
                        const int wiy = h == 0 ? AY::ineg(m) : AY::ipos(m);
                        const double *const q =
                            fin + (wiy * QX * a.plane + (h == 0 ? k : a.Ly - 1 - k) * a.pitch);
#pragma unroll
                        for (int ix = 0; ix < QX; ++ix) val[u][ix] = q[cofs[ix]];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (p0 + u * NV < AY::NPAIR) {
#pragma unroll
                        for (int ix = 0; ix < QX; ++ix) s += val[u][ix];
                    }
                }
            }
            dsum[acc][j] = s;
        }
        __syncthreads();
        if (i < 2 && (i == 0 ? need_lo : need_hi)) {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < NV; ++k) s += dsum[i * NV + k][j];
            rw[i][j] = s * ip.inv_den;
        }
        __syncthreads();
        if (walls && (ys < 0 || ys >= a.Ly)) {  // emitted by a wall
            const double *const ew = ys < 0 ? ip.ew_lo : ip.ew_hi;
            const double r = rw[ys < 0 ? 0 : 1][j];
#pragma unroll
            for (int ix = 0; ix < QX; ++ix) f[ix] = mul_rn(r * ew[ix], wy);
        }
    }
    // moments: row sums, then the sums over the rows in the order of G0 warp groups
    if (row) {
        double r, jx;
        S::row_sums(f, r, jx);
        rs[i][j] = r;
        jr[i][j] = jx;
    }
    __syncthreads();
    for (int t = i; t < 3 * G0; t += Q1) {
        const int k = t / G0, g = t - k * G0;
        if (row) {
            double s = k == 0 ? rs[g][j] : k == 1 ? jr[g][j] : (double)AY::vel(g) * rs[g][j];
#pragma unroll 4
            for (int q = g + G0; q < Q1; q += G0) {
                if (k < 2)
                    s += k == 0 ? rs[q][j] : jr[q][j];
                else if (AY::vel(q) != 0)
                    s = fma(to_f64((float)AY::vel(q)), rs[q][j], s);
            }
            (G0 == 1 ? tot[k][j] : part[t][j]) = s;
        }
    }
    __syncthreads();
    if constexpr (G0 > 1) {
        if (i < 3) {
            double s = part[i * G0][j];
#pragma unroll
            for (int g = 1; g < G0; ++g) s += part[i * G0 + g][j];
            tot[i][j] = s;
        }
        __syncthreads();
    }
    const double rho = tot[0][j], inv_rho = 1.0 / rho;
    const double ux = tot[1][j] * inv_rho, uy = tot[2][j] * inv_rho;
    const bool active = n0 + j < nodes && live;
    if (i == 0 && active) {  // positivity bound (Sec. 3), see Step2D
        const double umax = 0.816496580927726 * (ZY ? 2 * N : N);
        const double umaxx = 0.816496580927726 * (ZX ? 2 * NXL : NXL);
        if (!(rho > 0.0) || !(fabs(ux) <= umaxx) || !(fabs(uy) <= umax)) flag_unstable(a.status);
    }
    if (i <= NXL) {  // E^x of the pair number i
        const double v = ux * ux;
        double e = cex[NXL - 1], o = cox[NXL - 1];
#pragma unroll
        for (int k = NXL - 1; k >= 1; --k) e = fma(e, v, cex[k - 1]);
#pragma unroll
        for (int k = NXL - 2; k >= 0; --k) o = fma(o, v, cox[k]);
        e = mul_rn(e, v);
        const bool single = i == 0 && !ZX;
        if (!single) ex[AX::ineg(i)][j] = wx + fma(-ux, o, e);
        ex[AX::ipos(i)][j] = wx + (single ? e : fma(ux, o, e));
    }
    // E^y - W^y of this row
    double dy;
    {
        const double v = uy * uy;
        double e = cey[N - 1], o = coy[N - 1];
#pragma unroll
        for (int k = N - 1; k >= 1; --k) e = fma(e, v, cey[k - 1]);
#pragma unroll
        for (int k = N - 2; k >= 0; --k) o = fma(o, v, coy[k]);
        e = mul_rn(e, v);
        dy = ny == 0 ? e : fma(ny > 0 ? uy : -uy, o, e);
    }
    __syncthreads();
    if (row && active) {
        const double rey = rho * (wy + dy), gr = mul_rn(gto, wy);
        double *const op = fout + (iy * QX * a.plane + y * a.pitch + x);
#pragma unroll
        for (int ix = 0; ix < QX; ++ix) {
            double d = fma(ex[ix][j], rey, -f[ix]);
            if (AX::vel(ix) != 0 && gto != 0.0) d = fma(tx.WN[ix], gr, d);
            op[ix * a.plane] = fma(om, d, f[ix]);
        }
    }
    if (live) finish_step(a.status);
}

template <int N, int NXL, int ZY, int ZX, int G0>
inline cudaError_t launch_small(const SmallArgs &a, int n_inst, cudaStream_t s)
{
    constexpr int threads = (SMALL_NB * AxisVel<N, ZY>::Q + 31) / 32 * 32;
    return launch_serialized(k_step2d_small<N, NXL, ZY, ZX, G0>,
                             dim3((a.Lx * a.Ly + SMALL_NB - 1) / SMALL_NB, n_inst), dim3(threads), s, a);
}
