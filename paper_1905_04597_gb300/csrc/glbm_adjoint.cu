// Discrete adjoint of the 2D stream-collide step, for the gradient of the flow
// rate J = (1/Lx) sum_nodes sum_i xi_x,i F_i(T) (F = S(X): the streamed
// populations, Sec. 5.4 volumetric flow) with respect to the relaxation time
// tau, the body force g and the two wall speeds (Sec. 5.3).
//
// Forward: X_{t+1} = C(F_t), F_t = S(X_t). With mu_t = dJ/dF_t:
//   mu_T = xi_x / Lx,
//   lambda_{t+1} = S^T mu_{t+1}         (reverse streaming, wall terms below),
//   mu_t = (dC/dF)^T lambda_{t+1}        (rank-3 collision Jacobian, Eq. maineq01),
//   dJ/dtau += lambda_{t+1} . dC/dtau = -omega^2 lambda . (f^eq - f),
//   dJ/dg   += lambda_{t+1} . dC/dg   = lambda . W xi_x / theta.
// The collision Jacobian of f* = f + omega (f^eq(rho, u) - f) + F is
//   df*_i/df_j = (1 - omega) delta_ij
//              + omega [E_i + sum_a dE_i/du_a (xi_j,a - u_a)],
// so its transpose maps lambda to
//   mu_j = (1 - omega) lambda_j + omega [a0 + ax (xi_x,j - u_x) + ay (xi_y,j - u_y)],
//   a0 = sum_i lambda_i E_i,  a_a = sum_i lambda_i dE_i/du_a.
// Wall transpose: a population absorbed into a wall changes the wall density
// rho_w of the column it would reach by 1/den, and rho_w scales every emitted
// ghost rho_w E^x_i(u_w) W^y_i; so lambda of an absorbed population is
//   G(x_d) / den,  G(x) = sum_{emitted (i, y) of that wall} mu_i(x, y) E^x_i(u_w) W^y_i.
// A wall speed enters F_t only through E^x(u_w) of its emitted ghosts (rho_w
// balances the absorbed mass), so
//   dJ/du_w = sum_t sum_{emitted (x, y, i) of that wall} mu_t,i(x, y) rho_w,t(x)
//             dE^x_i/du(u_w) W^y_i,
// with rho_w,t from X_t: the step of time t adds its term at the wall rows,
// k_adj_final_walls the term of F_T.
//
// What bounds the adjoint step: the FP64 pipe (two instructions per cycle and SM;
// mu is FP64, and a step's 79 MB at D2Q121 256 x 128 stay in L2). So the kernel
// pulls a node's lambda and F once (instead of three times and twice), deals its
// velocity rows to G warps, sums the forward moments of FP32
// states in integers (glbm_moments.cuh), evaluates each equilibrium slope once per
// node, and forms every contraction from row sums: with d = E - W per axis,
//   sum_i lambda E^x   = sum lambda d^x + sum lambda W^x   (per row),
//   lambda . (f^eq - f) = rho E^y sum lambda d^x + B sum lambda W^x - sum lambda delta,
//   B = rho E^y - W^y, delta = f - W (FP64 states, which may have any density: with
//   rho W^y and rho W in place of W^y and W),
// five FP64 instructions per population for all contractions and two for mu_t (12 in
// all with the polynomials, slopes and moments, D2Q121), no term larger than the
// deviations. The wall sums of mu and the wall densities of
// X_t have a launch of their own (once per column, spread over the chip). D2Q121
// 256 x 128, FP32 states, GB300, per step: 350 -> 103 us, the wall sums 65 -> 6 us.
#include "glbm_moments.cuh"

namespace {

// E_{+-n}(u) - W_n and dE_{+-n}/du of one |n| in FP64, from the even/odd table.
template <int N>
__device__ __forceinline__ void eq_and_slope(const AxisTable &t, int n, double u, double &dp,
                                             double &dm, double &sp, double &sm)
{
    const double v = u * u;
    // Ae(v) = sum_{i=1..N} Ce[n][i] v^i and its derivative in v
    double a = t.Ce[n][N], da = 0.0;
#pragma unroll
    for (int i = N - 1; i >= 1; --i) {
        da = fma(da, v, a);
        a = fma(a, v, t.Ce[n][i]);
    }
    // a now is sum_{i>=1} Ce v^(i-1); Ae = a v, Ae' = a + v da
    const double Ae = a * v, sa = 2.0 * u * fma(v, da, a);
    if (n == 0) {
        dp = dm = Ae;
        sp = sm = sa;
        return;
    }
    double b = t.Co[n][N - 1], db = 0.0;
#pragma unroll
    for (int i = N - 2; i >= 0; --i) {
        db = fma(db, v, b);
        b = fma(b, v, t.Co[n][i]);
    }
    // E_{+-n} - W = Ae(v) +- u Bo(v);  dE/du = 2u Ae'(v) +- (Bo + 2v Bo'(v))
    const double so = fma(2.0 * v, db, b);
    dp = fma(u, b, Ae);
    dm = fma(-u, b, Ae);
    sp = sa + so;
    sm = sa - so;
}

// Sums over the two walls' columns before an adjoint step, a CTA of ADJ_WX columns x
// ADJ_WS slices per wall and quantity (blockIdx.y): 0, 1 the densities rho_w of
// the forward state X_t (lower, upper wall), 2, 3 the wall sums G(x) of mu_{t+1}.
// The slices' partial sums are added in a fixed order.
constexpr int ADJ_WX = 8, ADJ_WS = 32;

template <int N, typename TF>
__global__ void __launch_bounds__(ADJ_WX *ADJ_WS) k_adj_walls(const __grid_constant__ AdjArgs a)
{
    constexpr int Q1 = 2 * N + 1;
    __shared__ double part[ADJ_WS][ADJ_WX];
    wait_prior_grid();
    const int tx = threadIdx.x % ADJ_WX, sl = threadIdx.x / ADJ_WX;
    const int x = blockIdx.x * ADJ_WX + tx, xc = x < a.Lx ? x : a.Lx - 1;
    const bool lower = !(blockIdx.y & 1), dens = blockIdx.y < 2;
    const InstParams &ip = *a.ip;
    double D = 0.0;
    for (int i = sl; i < N * (N + 1) / 2; i += ADJ_WS) {
        int m = 1, k = i;  // speed |xi_y| and row
        while (k >= m) k -= m++;
        const int row = lower ? k : a.Ly - 1 - k;
        if (dens) {  // absorbed by the wall
            const int iy = lower ? N - m : N + m;
            const TF *const p = static_cast<const TF *>(a.X) + (long long)iy * Q1 * a.plane +
                                (long long)row * a.pitch;
#pragma unroll
            for (int ix = 0; ix < Q1; ++ix)
                D += to_f64(p[(long long)ix * a.plane + wrap_shift(xc - (ix - N), a.Lx, a.Lx > N)]);
        } else {  // emitted by the wall: velocity away from it
            const int iy = lower ? N + m : N - m;
            const double *const p =
                a.mu_in + (long long)iy * Q1 * a.plane + (long long)row * a.pitch + xc;
            double r = 0.0;
#pragma unroll
            for (int ix = 0; ix < Q1; ++ix)
                r = fma(p[(long long)ix * a.plane], lower ? ip.ew_lo[ix] : ip.ew_hi[ix], r);
            D = fma(r, a.tab.W[iy], D);
        }
    }
    part[sl][tx] = D;
    __syncthreads();
    for (int st = ADJ_WS / 2; st > 0; st >>= 1) {
        if (sl < st) part[sl][tx] += part[sl + st][tx];
        __syncthreads();
    }
    if (sl == 0 && x < a.Lx) {
        double v = part[0][tx] * ip.inv_den;
        if (dens && sizeof(TF) == 4) v += 1.0;  // FP32 stores deviations
        // G is stored over den, as the pull of an absorbed lambda takes it
        a.walls[(long long)blockIdx.y * a.Lx + x] = v;
    }
}

// Warps a node's velocity rows are dealt to (three rows per warp) and CTAs per SM asked
// for, 15 or 16 warps where 8 left the FP64 pipe 61 % busy between the kernel's
// barriers (D2Q121 256 x 128: 128 us with 8 warps, 103 us with 16; two rows per warp ran
// no faster). That caps the registers at 128 (168 at level 8), where part of lambda
// and F spills from level 4 on (bytes stored and loaded per thread, FP32 and FP64
// states: level 4 136/216 and 232/336, 5 400/648 and 460/756, 6 572/1164 and 860/1288, 7
// 760/1512 and 1200/1800, 8 608/1300 and 968/1472), but the warps are worth more than
// the spills cost: us per step of forward and adjoint at 256 x 128 with a CTA per SM
// less (levels 5 and up: without spills or nearly) / as here / one more, FP32 states:
// level 3 69 / 67 / 68, 4 101 / 101 / 102, 5 136 / 127 / 128, 6 197 / 179 / 172, 7 256 /
// 234 / 221, 8 333 / 311 / 305; FP64: 3 109 / 106 / 107, 4 172 / 176 / 178, 5 232 / 229 /
// 230, 6 330 / 324 / 302, 7 425 / 421 / 395, 8 560 / 575 / 567. Every level is 1.8 to 4.2
// times as fast as with one thread per node.
template <int N>
constexpr int ADJ_G = N == 1 ? 1 : N == 2 ? 2 : N <= 4 ? 3 : N == 5 ? 4 : N <= 7 ? 5 : 6;
template <int N>
constexpr int ADJ_CTAS = N == 1 ? 12 : N == 2 ? 8 : N <= 4 ? 5 : N == 5 ? 4 : N <= 7 ? 3 : 2;

template <int N, typename TF>
__global__ void __launch_bounds__(32 * ADJ_G<N>, ADJ_CTAS<N>)
    k_adj_step(const __grid_constant__ AdjArgs a)
{
    constexpr int Q1 = 2 * N + 1, G = ADJ_G<N>, RPG = (Q1 + G - 1) / G;
    constexpr bool DEV = sizeof(TF) == 4;
    using ACC = std::conditional_t<DEV, MomAccI<2, N, 0, false>, MomAccD<2, N, 0, false>>;
    __shared__ double eq[4][Q1][32];   // d^x, dE^x, d^y, dE^y
    __shared__ double con[G][5][32];   // the groups' partial moments, then contractions
    __shared__ double rup[3][32];      // rho (FP32 states: rho - 1), u_x, u_y
    __shared__ double tot[5][32];      // the contractions' totals
    wait_prior_grid();
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + lane, y = blockIdx.y;
    const bool active = x < a.Lx;
    const int xc = active ? x : a.Lx - 1;
    const InstParams &ip = *a.ip;
    const bool walls = a.bc == GLBM_BC_WALLS;
    const int plane = (int)a.plane;  // Q plane < 2^31 (checked at creation)

    int xs[Q1];  // source column of velocity column ix; the mirror's is its target
#pragma unroll
    for (int ix = 0; ix < Q1; ++ix) xs[ix] = wrap_shift(xc - (ix - N), a.Lx, a.Lx > N);
    double rw_lo = 0.0, rw_hi = 0.0;
    if (walls && y < N) rw_lo = a.walls[xc];
    if (walls && y >= a.Ly - N) rw_hi = a.walls[a.Lx + xc];

    // F_t and lambda_{t+1} of this group's rows iy = g + k G: F pulled from the node
    // a population comes from, lambda from the node it streams to; a row out of
    // the walls loads the edge row's F (replaced by the emission below) and takes
    // the wall's G for lambda
    TF f[RPG][Q1];
    double lam[RPG][Q1];
    const TF *const X = static_cast<const TF *>(a.X);
#pragma unroll
    for (int k = 0; k < RPG; ++k) {
        const int iy = g + k * G;
        if (iy < Q1) {
            const int cy = iy - N;
            int ys = y - cy, yd = y + cy;
            const bool absorbed = walls && (yd < 0 || yd >= a.Ly);
            const double *lp = a.walls + (yd < 0 ? 2 : 3) * (long long)a.Lx;
            int lstep = 0;
            if (walls) {
                ys = min(max(ys, 0), a.Ly - 1);
            } else {
                ys = wrap_shift(ys, a.Ly, a.Ly > N);
                yd = wrap_shift(yd, a.Ly, a.Ly > N);
            }
            if (!absorbed) {
                lp = a.mu_in + (iy * Q1 * plane + yd * a.pitch);
                lstep = plane;
            }
            const TF *const p = X + (iy * Q1 * plane + ys * a.pitch);
#pragma unroll
            for (int ix = 0; ix < Q1; ++ix) f[k][ix] = p[ix * plane + xs[ix]];
#pragma unroll
            for (int ix = 0; ix < Q1; ++ix) lam[k][ix] = lp[ix * lstep + xs[Q1 - 1 - ix]];
        }
    }

    // forward moments (deviations of rho in FP32)
    ACC acc;
    acc.init();
    double em[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < RPG; ++k) {
        const int iy = g + k * G;
        if (iy < Q1) {
            const int cy = iy - N;
            if (walls && (y - cy < 0 || y - cy >= a.Ly)) {  // emitted by a wall
                const bool lo = y - cy < 0;
                const double wy = a.tab.W[iy], rw = lo ? rw_lo : rw_hi;
                const double R0 = wy * (rw * (lo ? ip.kw_lo[0] : ip.kw_hi[0]) - (DEV ? 1.0 : 0.0));
                em[0] += R0;
                em[1] = fma(wy * rw, lo ? ip.kw_lo[1] : ip.kw_hi[1], em[1]);
                em[2] = fma((double)cy, R0, em[2]);
            } else if constexpr (DEV) {
                acc.row(f[k], cy, 0);
            } else {
                acc.row(f[k], (double)cy, 0.0);
            }
        }
    }
    {
        double m[3];
        bool ok = true;
        if constexpr (DEV) {
            ok = acc.in_range();
#pragma unroll
            for (int k = 0; k < 3; ++k) m[k] = acc.total(k);
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) m[k] = acc.m[k];
        }
        if (!ok) {  // a deviation outside the digits' range: in FP64
            MomAccD<2, N, 0, false> slow;
            slow.init();
#pragma unroll 1
            for (int iy = g; iy < Q1; iy += G) {
                const int ys = y - (iy - N);
                if (walls && (ys < 0 || ys >= a.Ly)) continue;
                const TF *const p = X + (iy * Q1 * plane +
                                         (walls ? ys : wrap_shift(ys, a.Ly, a.Ly > N)) * a.pitch);
                TF v[Q1];
#pragma unroll
                for (int ix = 0; ix < Q1; ++ix) v[ix] = p[ix * plane + xs[ix]];
                slow.row(v, (double)(iy - N), 0.0);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) m[k] = slow.m[k];
        }
        if (walls && (y < N || y >= a.Ly - N)) {
#pragma unroll
            for (int k = 0; k < 3; ++k) m[k] += em[k];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) con[g][k][lane] = m[k];
    }
    __syncthreads();
    if (g == 0) {
        double m[3] = {con[0][0][lane], con[0][1][lane], con[0][2][lane]};
#pragma unroll
        for (int t = 1; t < G; ++t) {
#pragma unroll
            for (int k = 0; k < 3; ++k) m[k] += con[t][k][lane];
        }
        const double rho = DEV ? 1.0 + m[0] : m[0], inv = 1.0 / rho;
        rup[0][lane] = m[0];
        rup[1][lane] = mom_div(m[1], rho, inv);
        rup[2][lane] = mom_div(m[2], rho, inv);
    }
    __syncthreads();
    const double dens = rup[0][lane], rho = DEV ? 1.0 + dens : dens;
    const double ux = rup[1][lane], uy = rup[2][lane];
    // the equilibrium and its slopes: group g evaluates the (|n|, axis) pairs g,
    // g + G, ...
#pragma unroll
    for (int n = 0; n <= N; ++n) {
#pragma unroll
        for (int ax = 0; ax < 2; ++ax) {
            if ((2 * n + ax) % G != g) continue;
            double dp, dm, sp, sm;
            eq_and_slope<N>(a.tab, n, ax ? uy : ux, dp, dm, sp, sm);
            eq[2 * ax][N - n][lane] = dm;
            eq[2 * ax + 1][N - n][lane] = sm;
            eq[2 * ax][N + n][lane] = dp;
            eq[2 * ax + 1][N + n][lane] = sp;
        }
    }
    __syncthreads();
    // contractions of lambda_{t+1} with the equilibrium and its slopes
    double a0 = 0.0, ax = 0.0, ay = 0.0, gt = 0.0, gg = 0.0;
#pragma unroll
    for (int k = 0; k < RPG; ++k) {
        const int iy = g + k * G;
        if (iy < Q1) {
            double Ld = 0.0, Lw = 0.0, Ls = 0.0, Lg = 0.0, Lf = 0.0;
            const double wy = a.tab.W[iy], base = DEV ? wy : rho * wy;
            const int ys = y - (iy - N);
            const bool ghost = walls && (ys < 0 || ys >= a.Ly);
#pragma unroll
            for (int ix = 0; ix < Q1; ++ix) {
                const double l = lam[k][ix];
                Ld = fma(l, eq[0][ix][lane], Ld);
                Ls = fma(l, eq[1][ix][lane], Ls);
                Lw = fma(l, a.tab.W[ix], Lw);
                if (ix != N) Lg = fma(l, a.tab.WN[ix], Lg);
            }
            if (ghost) {
                const double *const ew = ys < 0 ? ip.ew_lo : ip.ew_hi;
#pragma unroll
                for (int ix = 0; ix < Q1; ++ix) Lf = fma(lam[k][ix], ew[ix], Lf);
                const double rw = ys < 0 ? rw_lo : rw_hi;
                Lf = DEV ? wy * fma(rw, Lf, -Lw) : fma(wy * rw, Lf, -(base * Lw));
            } else {
#pragma unroll
                for (int ix = 0; ix < Q1; ++ix) {
                    const double d = DEV ? to_f64(f[k][ix]) : fma(-base, a.tab.W[ix], to_f64(f[k][ix]));
                    Lf = fma(lam[k][ix], d, Lf);
                }
            }
            const double dy = eq[2][iy][lane], L0 = Ld + Lw;
            const double Ey = wy + dy;
            const double B = DEV ? fma(dens, wy, rho * dy) : fma(rho, dy, fma(rho, wy, -base));
            a0 = fma(Ey, L0, a0);
            ax = fma(Ey, Ls, ax);
            ay = fma(eq[3][iy][lane], L0, ay);
            gt += fma(base + B, Ld, fma(B, Lw, -Lf));
            gg = fma(wy, Lg, gg);
        }
    }
    if constexpr (G > 1) {
        con[g][0][lane] = a0;
        con[g][1][lane] = ax;
        con[g][2][lane] = ay;
        con[g][3][lane] = gt;
        con[g][4][lane] = gg;
        __syncthreads();
        // the five sums over the groups, each by one warp
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if (k % G != g) continue;
            double t = con[0][k][lane];
#pragma unroll
            for (int u = 1; u < G; ++u) t += con[u][k][lane];
            tot[k][lane] = t;
        }
        __syncthreads();
        a0 = tot[0][lane];
        ax = tot[1][lane];
        ay = tot[2][lane];
    }
    // mu_t = (dC/dF)^T lambda at this node (the density cancels: d f^eq_i / d f_j =
    // E_i + sum_a dE_i/du_a (xi_j,a - u_a)), and the wall speeds' term of F_t: mu_t
    // of every ghost this node pulls from a wall, times rho_w dE^x/du(u_w) W^y
    double glo = 0.0, ghi = 0.0;
    if (active) {
        const double om = ip.omega, keep = 1.0 - om, oax = om * ax, oay = om * ay;
        const double b0 = om * (a0 - fma(ax, ux, ay * uy));
#pragma unroll
        for (int k = 0; k < RPG; ++k) {
            const int iy = g + k * G;
            if (iy < Q1) {
                const double b = fma(oay, f2d((float)(iy - N)), b0);
                double *const op = a.mu_out + (iy * Q1 * plane + y * a.pitch + x);
                const int ys = y - (iy - N);
                const bool ghost = walls && (ys < 0 || ys >= a.Ly);
                double gw = 0.0;
#pragma unroll
                for (int ix = 0; ix < Q1; ++ix) {
                    const double m = fma(keep, lam[k][ix], ix == N ? b : fma(oax, (double)(ix - N), b));
                    op[ix * plane] = m;
                    if (ghost) gw = fma(m, ys < 0 ? ip.dew_lo[ix] : ip.dew_hi[ix], gw);
                }
                if (ghost) {
                    gw *= a.tab.W[iy];
                    if (ys < 0)
                        glo = fma(gw, rw_lo, glo);
                    else
                        ghi = fma(gw, rw_hi, ghi);
                }
            }
        }
    }
    // gradient partials of this block, summed in a fixed order: the groups, then
    // the lanes
    const bool near = walls && (y < N || y >= a.Ly - N);
    if constexpr (G > 1) {
        if (near) {  // (con is free: its totals are taken)
            con[g][0][lane] = glo;
            con[g][1][lane] = ghi;
            __syncthreads();
        }
    }
    if (g == 0) {
        double v[GLBM_ADJ_NG] = {gt, gg, glo, ghi};
        if constexpr (G > 1) {
            v[0] = tot[3][lane];
            v[1] = tot[4][lane];
            if (near) {
#pragma unroll
                for (int t = 1; t < G; ++t) {
                    v[2] += con[t][0][lane];
                    v[3] += con[t][1][lane];
                }
            }
        }
        v[0] *= active ? -ip.omega * ip.omega : 0.0;
        v[1] *= active ? 3.0 / N : 0.0;  // 1 / theta_x
#pragma unroll
        for (int k = 0; k < GLBM_ADJ_NG; ++k) {
            if (k >= 2 && !near) continue;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) v[k] += __shfl_down_sync(0xFFFFFFFFu, v[k], d);
        }
        if (lane == 0) {
            double *const p = a.gpart + GLBM_ADJ_NG * ((long long)blockIdx.y * gridDim.x + blockIdx.x);
            p[0] += v[0];
            p[1] += v[1];
            if (near) {
                p[2] += v[2];
                p[3] += v[3];
            }
        }
    }
}

// The wall speeds' term of F_T = S(X_T): mu_T = xi_x / Lx (the seed) at every
// ghost a wall emits, times rho_w(X_T) dE^x/du(u_w) W^y. The ghosts of a column
// have sum n W^y_n = den, so the term is den / Lx sum_i xi_x,i dE^x_i/du times the
// sum of rho_w over the columns (from k_adj_walls): one block, added to the first
// block's partials.
template <int N>
__global__ void __launch_bounds__(256) k_adj_final_walls(const __grid_constant__ AdjArgs a)
{
    __shared__ double red[2][256];
    double s[2] = {0.0, 0.0};
    for (int x = threadIdx.x; x < a.Lx; x += 256) {
        s[0] += a.walls[x];
        s[1] += a.walls[a.Lx + x];
    }
    red[0][threadIdx.x] = s[0];
    red[1][threadIdx.x] = s[1];
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st) {
            red[0][threadIdx.x] += red[0][threadIdx.x + st];
            red[1][threadIdx.x] += red[1][threadIdx.x + st];
        }
        __syncthreads();
    }
    if (threadIdx.x < 2) {
        const double *const dew = threadIdx.x ? a.ip->dew_hi : a.ip->dew_lo;
        double t = 0.0;
        for (int ix = 0; ix <= 2 * N; ++ix) t = fma((double)(ix - N), dew[ix], t);
        a.gpart[2 + threadIdx.x] += red[threadIdx.x][0] * t / (a.ip->inv_den * a.Lx);
    }
}

// mu_T = xi_x / Lx at every node, zero in the padding.
template <int N>
__global__ void k_adj_seed(const __grid_constant__ AdjArgs a)
{
    constexpr int Q1 = 2 * N + 1;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, iy = blockIdx.z;
    if (x >= a.pitch) return;
    double *const p = a.mu_out + (long long)iy * Q1 * a.plane + (long long)y * a.pitch + x;
#pragma unroll
    for (int ix = 0; ix < Q1; ++ix)
        p[(long long)ix * a.plane] = x < a.Lx ? (double)(ix - N) / a.Lx : 0.0;
}

// The blocks' partials summed in a fixed order, one block.
__global__ void __launch_bounds__(256) k_adj_sum(const double *gpart, long long nblocks, double *out)
{
    __shared__ double red[256];
    const int k = threadIdx.x % GLBM_ADJ_NG;
    double s = 0.0;
    for (long long b = threadIdx.x / GLBM_ADJ_NG; b < nblocks; b += 256 / GLBM_ADJ_NG)
        s += gpart[GLBM_ADJ_NG * b + k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = 128; st >= GLBM_ADJ_NG; st >>= 1) {
        if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x < GLBM_ADJ_NG) out[threadIdx.x] = red[threadIdx.x];
}

// The wall sums of a (a.mu_in, a.X).
template <int N>
cudaError_t adj_walls_n(const AdjArgs &a, int quantities, cudaStream_t s)
{
    const dim3 grid((a.Lx + ADJ_WX - 1) / ADJ_WX, quantities);
    return a.prec == GLBM_FP64
               ? launch_serialized(k_adj_walls<N, double>, grid, dim3(ADJ_WX * ADJ_WS), s, a)
               : launch_serialized(k_adj_walls<N, float>, grid, dim3(ADJ_WX * ADJ_WS), s, a);
}

template <int N>
cudaError_t adj_step_n(const AdjArgs &a, cudaStream_t s)
{
    if (a.bc == GLBM_BC_WALLS) {
        const cudaError_t e = adj_walls_n<N>(a, 4, s);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((a.Lx + 31) / 32, a.Ly);
    return a.prec == GLBM_FP64
               ? launch_serialized(k_adj_step<N, double>, grid, dim3(32 * ADJ_G<N>), s, a)
               : launch_serialized(k_adj_step<N, float>, grid, dim3(32 * ADJ_G<N>), s, a);
}

template <int N>
cudaError_t adj_final_walls_n(const AdjArgs &a, cudaStream_t s)
{
    if (a.bc != GLBM_BC_WALLS) return cudaSuccess;
    const cudaError_t e = adj_walls_n<N>(a, 2, s);
    if (e != cudaSuccess) return e;
    k_adj_final_walls<N><<<1, 256, 0, s>>>(a);
    return cudaGetLastError();
}

template <int N>
cudaError_t adj_seed_n(const AdjArgs &a, cudaStream_t s)
{
    dim3 grid((a.pitch + 127) / 128, a.Ly, 2 * N + 1);
    k_adj_seed<N><<<grid, 128, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

long long glbm_adj_blocks(int Lx, int Ly)
{
    return (long long)((Lx + 31) / 32) * Ly;
}

cudaError_t glbm_launch_adj_seed(const AdjArgs &a, cudaStream_t s)
{
    switch (a.N) {
#define GLBM_CASE(NN) \
    case NN: return adj_seed_n<NN>(a, s);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t glbm_launch_adj_final_walls(const AdjArgs &a, cudaStream_t s)
{
    switch (a.N) {
#define GLBM_CASE(NN) \
    case NN: return adj_final_walls_n<NN>(a, s);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t glbm_launch_adj_step(const AdjArgs &a, cudaStream_t s)
{
    switch (a.N) {
#define GLBM_CASE(NN) \
    case NN: return adj_step_n<NN>(a, s);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t glbm_launch_adj_sum(const double *gpart, long long nblocks, double *out, cudaStream_t s)
{
    k_adj_sum<<<1, 256, 0, s>>>(gpart, nblocks, out);
    return cudaGetLastError();
}
