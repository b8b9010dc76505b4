// Fused pull-stream + BGK collide for the 3D tensor-product lattices (Sec. 4:
// the product of 1D levels on three axes, D3Q(2N+1)^3), with the diffuse
// walls at y = -1/2 and y = Ly - 1/2 (periodic in x and z), the linearised
// body force along x (Sec. 5.4) and the FP32-deviation or FP64 storage of the
// 2D step.
//
// One CTA covers 32 columns x R rows of one z-slice of one instance. A node's
// (2N+1)^3 populations form (2N+1)^2 velocity rows (n_z, n_y) of 2N+1
// columns (n_x); the rows are dealt to G warps, so a thread keeps
// ceil((2N+1)^2 / G) (2N+1) values in registers. Phases as in the 2D tile:
//   phase 0 (CTAs touching a wall): the mass streaming into each wall per
//           (x, z) column, turned into the wall density rho_w(x, z);
//   phase 1: pull (periodic in x and z; sources inside a wall take the
//           wall's emission rho_w E^x(u_w) W^y W^z), partial moments;
//   phase 2: moments, E - W per axis, relaxation plus force, store.
// The equilibrium deviation is built row by row:
//   delta f^eq = d^x rho e^y e^z + W^x (rho e^y e^z - W^y W^z),
//   rho e^y e^z - W^y W^z = d^y rho e^z + W^y (drho W^z + rho d^z),
// with e = W + d per axis.
#pragma once
#include "glbm_step2d.cuh"

template <int N, typename T, int G, int R>
struct Step3D {
    static constexpr int Q1 = 2 * N + 1;
    static constexpr int NROW = Q1 * Q1;               // velocity rows (n_z, n_y)
    static constexpr int RPG = (NROW + G - 1) / G;     // rows per warp group
    static constexpr int NW = G * R;
    static constexpr int NV = 4;                       // wall-flux accumulators
    static constexpr bool DEV = sizeof(T) == 4;
    using A = TabAcc<T>;
    // With G == 2N+1 warp groups, group g holds the rows (n_z = k - N, n_y = g - N):
    // n_z is a compile-time index of the unrolled loop and n_y is fixed per thread.
    static constexpr bool ZROW = G == Q1;
    __device__ static int row_z(int row, int k) { return ZROW ? k : row / Q1; }
    __device__ static int row_y(int row, int g) { return ZROW ? g : row % Q1; }

    struct Smem {
        T part[R][G][8][32];  // (s, c) of delta rho, j_x, j_y, j_z per row and group
        T tot[R][8][32];      // and over the groups
        T dev[R][3][Q1][32];  // E - W of the nodes per axis (FP64: E^x on the x axis)
        T rw[2][32];          // wall density (FP64) or its deviation (FP32): lo, hi
        T dsum[NV][2][32];
    };

    __device__ static void run(const AxisTable &tab, const InstParams &ip, int Lx, int Ly, int Lz,
                               int pitch, int plane, int bc, const T *__restrict__ fin,
                               T *__restrict__ fout, int x0, int y0, int z, Smem &sm,
                               unsigned *status, unsigned seed, bool live = true)
    {
        const int lane = threadIdx.x & 31;
        const int w = threadIdx.x >> 5;
        const int g = w % G;
        const int r = w / G;
        const bool walls = bc == GLBM_BC_WALLS;
        const int x = x0 + lane, y = y0 + r;
        // live: no earlier step halted the run (else nothing is stored)
        const bool active = (x < Lx) && (y < Ly) && live;
        const int xc = x < Lx ? x : Lx - 1;
        const int yc = y < Ly ? y : Ly - 1;
        const int slab = Ly * pitch;  // elements per z-slice of a velocity plane

        int cofs[Q1];
#pragma unroll
        for (int ix = 0; ix < Q1; ++ix) cofs[ix] = ix * plane + wrap_shift(xc - (ix - N), Lx, Lx > N);

        // ---- phase 0: wall densities of this tile's (x, z) columns ----------
        const bool need_lo = walls && (y0 < N);
        const bool need_hi = walls && (y0 + R > Ly - N);
        if (need_lo || need_hi) {
            // (n_y, row) pairs with row < |n_y| in order of |n_y|, each over
            // every n_z, through NV fixed accumulators (order independent of
            // the tile shape)
#pragma unroll 1
            for (int v = w; v < NV; v += NW) {
                T slo = T(0), shi = T(0);
#pragma unroll 1
                for (int p = v; p < N * (N + 1) / 2 * Q1; p += NV) {
                    const int iz = p % Q1;
                    int aa = 1, k = p / Q1;
                    while (k >= aa) {
                        k -= aa;
                        ++aa;
                    }
                    const int zs = wrap_shift(z - (iz - N), Lz, Lz > N);
                    if (need_lo) {  // n_y = -aa leaving row k through y = -1/2
                        const T *pl = fin + ((iz * Q1 + N - aa) * Q1 * plane + zs * slab + k * pitch);
#pragma unroll
                        for (int ix = 0; ix < Q1; ++ix) slo += __ldg(pl + cofs[ix]);
                    }
                    if (need_hi) {  // n_y = +aa leaving row Ly-1-k through y = Ly-1/2
                        const T *ph =
                            fin + ((iz * Q1 + N + aa) * Q1 * plane + zs * slab + (Ly - 1 - k) * pitch);
#pragma unroll
                        for (int ix = 0; ix < Q1; ++ix) shi += __ldg(ph + cofs[ix]);
                    }
                }
                sm.dsum[v][0][lane] = slo;
                sm.dsum[v][1][lane] = shi;
            }
            __syncthreads();
            if (w == 0) {
                T s0 = T(0), s1 = T(0);
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    s0 += sm.dsum[j][0][lane];
                    s1 += sm.dsum[j][1][lane];
                }
                const T inv_den = DEV ? (T)ip.inv_den_f : (T)ip.inv_den;
                sm.rw[0][lane] = s0 * inv_den;
                sm.rw[1][lane] = s1 * inv_den;
            }
            __syncthreads();
        }

        // ---- phase 1: pull and partial moments -----------------------------
        T f[RPG][Q1];
        T s_r = T(0), c_r = T(0), s_x = T(0), c_x = T(0), s_y = T(0), c_y = T(0), s_z = T(0),
          c_z = T(0);
        f32x2 s_rx = 0ull, c_rx = 0ull, s_yz = 0ull, c_yz = 0ull;  // FP32: the same in pairs
#pragma unroll
        for (int k = 0; k < RPG; ++k) {
            const int row = g + k * G;
            if (row < NROW) {
                const int iz = row_z(row, k), iy = row_y(row, g);
                int ys = yc - (iy - N);
                ys = walls ? min(max(ys, 0), Ly - 1) : wrap_shift(ys, Ly, Ly > N);
                const int zs = wrap_shift(z - (iz - N), Lz, Lz > N);
                const T *rowp = fin + (row * Q1 * plane + zs * slab + ys * pitch);
#pragma unroll
                for (int ix = 0; ix < Q1; ++ix) f[k][ix] = __ldg(rowp + cofs[ix]);
            }
        }
#pragma unroll
        for (int k = 0; k < RPG; ++k) {
            const int row = g + k * G;
            if (row < NROW) {
                const int iz = row_z(row, k), iy = row_y(row, g);
                const int ny = iy - N, nz = iz - N;
                const int ys = yc - ny;
                if (walls && (ys < 0 || ys >= Ly)) {  // uniform across the warp
                    const bool lo = ys < 0;
                    const T wyz = mul_rn(A::W(tab, iy), A::W(tab, iz));
                    const T rw = sm.rw[lo ? 0 : 1][lane];
#pragma unroll
                    for (int ix = 0; ix < Q1; ++ix) {
                        if (DEV) {
                            const T dw = lo ? (T)ip.dw_lo_f[ix] : (T)ip.dw_hi_f[ix];
                            // no rounded 1 + drho_w scales the emitted momentum
                            f[k][ix] = mul_rn(wyz, fma(rw, A::W(tab, ix), fma(rw, dw, dw)));
                        } else {
                            const T ew = lo ? (T)ip.ew_lo[ix] : (T)ip.ew_hi[ix];
                            f[k][ix] = mul_rn(rw * ew, wyz);
                        }
                    }
                }
                T rs = T(0);
#pragma unroll
                for (int ix = 0; ix < Q1; ++ix) rs += f[k][ix];
                T jx = T(0);
#pragma unroll
                for (int n = 1; n <= N; ++n) jx = fma(T(n), f[k][N + n] - f[k][N - n], jx);
                if constexpr (DEV) {
                    // two sums per two-lane instruction (adding zero changes nothing):
                    // 14 instructions per row instead of 28 where the issue slots bound
                    // the kernel, D3Q125 250 x 61 x 45 146 -> 141.5 us (GB300)
                    acc2x2(s_rx, c_rx, pk2(rs, jx));
                    acc2x2(s_yz, c_yz, pk2(mul_rn(T(ny), rs), mul_rn(T(nz), rs)));
                } else {
                    acc2(s_r, c_r, rs);
                    acc2(s_x, c_x, jx);
                    if (ny != 0) acc2(s_y, c_y, mul_rn(T(ny), rs));
                    if (nz != 0) acc2(s_z, c_z, mul_rn(T(nz), rs));
                }
            }
        }
        if constexpr (DEV) {
            s_r = lo2(s_rx), s_x = hi2(s_rx), s_y = lo2(s_yz), s_z = hi2(s_yz);
            c_r = lo2(c_rx), c_x = hi2(c_rx), c_y = lo2(c_yz), c_z = hi2(c_yz);
        }
        // ---- phase 2: moments, equilibrium, relaxation, store --------------
        // The G warps of a node share this work: warp f sums functional f over the
        // groups, then warp a takes the velocity of axis a and its equilibrium
        // polynomials; the values meet in shared memory. Every warp for itself took
        // 250 of the 1370 instructions of a thread at D3Q125, where the issue slots
        // bound the kernel (IPC 3.1): 250 x 61 x 45 FP32 160 -> 143 us per step, 256 x
        // 64 x 32 FP64 1203 -> 933 us (GB300).
        T tS[4], tC[4];  // delta rho (FP64: rho), j_x, j_y, j_z: sums and compensations
        if constexpr (G == 1) {
            tS[0] = s_r, tS[1] = s_x, tS[2] = s_y, tS[3] = s_z;
            tC[0] = c_r, tC[1] = c_x, tC[2] = c_y, tC[3] = c_z;
        } else {
            T *const pp = &sm.part[r][g][0][lane];
            pp[0 * 32] = s_r;
            pp[1 * 32] = c_r;
            pp[2 * 32] = s_x;
            pp[3 * 32] = c_x;
            pp[4 * 32] = s_y;
            pp[5 * 32] = c_y;
            pp[6 * 32] = s_z;
            pp[7 * 32] = c_z;
            __syncthreads();
            for (int q = g; q < 4; q += G) {
                T S = T(0), C = T(0);
#pragma unroll
                for (int gi = 0; gi < G; ++gi) {
                    acc2(S, C, sm.part[r][gi][2 * q][lane]);
                    if (DEV) C += sm.part[r][gi][2 * q + 1][lane];
                }
                sm.tot[r][2 * q][lane] = S;
                if (DEV) sm.tot[r][2 * q + 1][lane] = C;
            }
            __syncthreads();
            tS[0] = sm.tot[r][0][lane];
            tC[0] = DEV ? sm.tot[r][1][lane] : T(0);
        }
        const T m0 = DEV ? tS[0] + tC[0] : tS[0];
        const T rho = DEV ? T(1) + m0 : m0;
        const T drho = DEV ? m0 : m0 - T(1);
        const unsigned hnode = DEV ? hash32((unsigned)((z * Ly + y) * Lx + x) ^ seed) : 0u;
        const T inv_rho = G == 1 || g < 3 ? T(1) / rho : T(0);
        for (int ax = G == 1 ? 0 : g; ax < 3; ax += G) {
            T S, C;
            if constexpr (G == 1) {
                S = ax == 0 ? tS[1] : ax == 1 ? tS[2] : tS[3];
                C = ax == 0 ? tC[1] : ax == 1 ? tC[2] : tC[3];
            } else {
                S = sm.tot[r][2 + 2 * ax][lane];
                C = DEV ? sm.tot[r][3 + 2 * ax][lane] : T(0);
            }
            T u = (DEV ? S + C : S) * inv_rho;
            float re = 0.0f;
            if constexpr (DEV) {
                // u = j / (1 + delta rho), rounded stochastically (as in the 2D tile):
                // j times the rounded reciprocal alone carries a fixed relative bias
                // of up to 2^-24 where rho lies just below 1; the polynomial values
                // are rounded stochastically too, one draw per node and axis
                const unsigned wu = ax == 0   ? dither_word_ux(hnode)
                                    : ax == 1 ? dither_word_uy(hnode)
                                              : dither_word_uz(hnode);
                const unsigned we = ax == 0   ? dither_word_ex(hnode)
                                    : ax == 1 ? dither_word_ey(hnode)
                                              : dither_word_ez(hnode);
                const T du = dither_ulp(u, dither_unit(wu));
                u = fma(fma(-u, drho, (S - u) + C) + du, inv_rho, u);
                re = dither_unit2(we);
            }
            if (active) {
                const T umax = (T)(0.816496580927726 * N);  // sqrt(2/3) N (Sec. 3)
                if (!(rho > T(0)) || !(fabs(u) <= umax)) flag_unstable(status);
            }
            T d[Q1];
            if constexpr (DEV)
                eq_dev_all_sr<N>(tab, u, re, d);
            else
                eq_dev_all<N, T>(tab, u, d);
#pragma unroll
            for (int i = 0; i < Q1; ++i) {
                if (!DEV && ax == 0) d[i] += A::W(tab, i);  // E^x, once per node
                sm.dev[r][ax][i][lane] = d[i];
            }
        }
        if constexpr (G > 1) __syncthreads();
        T dx[Q1];
#pragma unroll
        for (int ix = 0; ix < Q1; ++ix) dx[ix] = sm.dev[r][0][ix][lane];
        const T dy_g = ZROW ? sm.dev[r][1][g][lane] : T(0);  // ZROW: this thread's n_y
        const T om = DEV ? (T)ip.omega_f : (T)ip.omega;
        const T gto = DEV ? (T)ip.g_theta_om_f : (T)ip.g_theta_om;  // g / (theta omega)
        if (!live) return;  // an earlier step halted the run: store nothing
        // rows past Ly store into the plane's spare row after its Lz Ly rows,
        // columns past Lx into the row padding (pitch is a multiple of 64): no
        // store needs a per-node condition, and nothing reads those places
        T *const obase = fout + ((y < Ly ? z * slab + y * pitch : Lz * slab) + x);
        const float iom = DEV ? 1.0f / ip.omega_f : 0.0f;  // the dither enters f^eq over omega
#pragma unroll
        for (int k = 0; k < RPG; ++k) {
            const int row = g + k * G;
            if (row < NROW) {
                const int iz = row_z(row, k), iy = row_y(row, g);
                const T wy = A::W(tab, iy), wz = A::W(tab, iz);
                const T dyv = ZROW ? dy_g : sm.dev[r][1][iy][lane], dzv = sm.dev[r][2][iz][lane];
                const T rez = rho * (wz + dzv);       // rho e^z
                const T rez_y = rez * (wy + dyv);     // rho e^y e^z
                const T wyz = mul_rn(wy, wz);
                const T gr = mul_rn(gto, wyz);        // W^y W^z g / (theta omega)
                // FP32: B = rho e^y e^z - W^y W^z = d^y W^z + (W^y + d^y) Bz with
                // Bz = rho e^z - W^z = drho W^z + d^z + drho d^z: no momentum
                // carrier (d^y, d^z) is scaled by a rounded rho or e^y
                const T Bz = DEV ? fma(drho, wz, fma(drho, dzv, dzv)) : T(0);
                const T B = DEV ? fma(dyv, wz, fma(dyv, Bz, mul_rn(wy, Bz))) : T(0);
                T *const op = obase + row * Q1 * plane;
                const unsigned hrow = hnode + (unsigned)row * 0x85EBCA6Bu;
                // the row's dither draws, divided by omega
                const float ua = DEV ? mul_rn(dither_unit(hrow), iom) : 0.0f;
                const float ub = DEV ? mul_rn(dither_unit(dither_word_b(hrow)), iom) : 0.0f;
                if constexpr (DEV) {
                    // velocity columns in pairs (ix, ix + 1) on the two-lane FP32
                    // instructions, each lane doing exactly the scalar loop's
                    // operations in its order (bit-identical results); the last
                    // of the odd 2N+1 columns takes the scalar loop
                    const f32x2 B2 = pk2(B, B), gr2 = pk2(gr, gr), om2 = pk2(om, om),
                                nwy2 = pk2(-wy, -wy), wz2 = pk2(wz, wz);
#pragma unroll
                    for (int ix = 0; ix + 1 < Q1; ix += 2) {
                        const f32x2 f0 = pk2(f[k][ix], f[k][ix + 1]);
                        const f32x2 Bn = fma2(pk2(T(ix - N), T(ix + 1 - N)), gr2, B2);
                        const f32x2 dxv = pk2(dx[ix], dx[ix + 1]);
                        const float p0 = __int_as_float(__float_as_int(lo2(f0)) & 0x7F800000);
                        const float p1 = __int_as_float(__float_as_int(hi2(f0)) & 0x7F800000);
                        const f32x2 dith = mul2(pk2(dither_pick(ix, ua, ub, -ua, -ub),
                                                    dither_pick(ix + 1, ua, ub, -ua, -ub)),
                                                pk2(p0, p1));
                        const f32x2 t1 =
                            fma2(dxv, B2, fma2(pk2(A::W(tab, ix), A::W(tab, ix + 1)), Bn, dith));
                        const f32x2 rr = fma2(mul2(dxv, nwy2), wz2, f0);
                        const f32x2 v2 = fma2(om2, sub2(t1, rr), f0);
                        op[ix * plane] = lo2(v2);
                        op[(ix + 1) * plane] = hi2(v2);
                    }
                }
#pragma unroll
                for (int ix = (DEV ? Q1 - 1 : 0); ix < Q1; ++ix) {
                    const int nx = ix - N;
                    const T f0 = f[k][ix];
                    T v;
                    if (DEV) {
                        const T Bn = nx != 0 ? fma(T(nx), gr, B) : B;
                        // delta f^eq = d^x W^y W^z + E^x B + F/omega: the
                        // momentum-carrying d^x is rounded with W^y, then meets W^z
                        // in a fused rounding (no rounded rho or W^y W^z factor,
                        // whose fixed error would scale the momentum at every
                        // step); as in 2D, r = f0 - d^x W^y W^z, t1 holds the rest
                        // plus the dither (half an ulp of f0, over omega), and the
                        // store f0 + omega (t1 - r) is one rounding
                        const float u = dither_pick(ix, ua, ub, -ua, -ub);
                        const T dith = (T)dither_ulp((float)f0, u);
                        const T t1 = fma(dx[ix], B, fma(A::W(tab, ix), Bn, dith));
                        const T r = fma(-mul_rn(dx[ix], wy), wz, f0);  // f0 - d^x W^y W^z
                        v = fma(om, t1 - r, f0);
                    } else {
                        // dx holds E^x itself in FP64 mode; f^eq - f0 in one
                        // fused rounding, the force term, f0 + omega (...)
                        T d = fma(dx[ix], rez_y, -f0);
                        if (nx != 0 && gto != T(0)) d = fma(A::WN(tab, ix), gr, d);
                        v = fma(om, d, f0);
                    }
                    op[ix * plane] = v;
                }
            }
        }
    }
};

template <int N, typename T, int G, int R>
__global__ void __launch_bounds__(32 * G * R) k_step3d(const __grid_constant__ Step3DArgs a)
{
    using S = Step3D<N, T, G, R>;
    __shared__ typename S::Smem sm;
    wait_prior_grid();
    const bool live = !step_halted(a.status);  // needed only at the stores
    const int inst = blockIdx.z / a.Lz;
    const int z = blockIdx.z - inst * a.Lz;
    const T *fin = static_cast<const T *>(a.fin) + (long long)inst * a.inst_stride;
    T *fout = static_cast<T *>(a.fout) + (long long)inst * a.inst_stride;
    const unsigned seed = S::DEV ? hash32(__ldcg(a.step_ctr) * 0x632BE5ABu + inst) : 0u;
    S::run(a.tab, a.ip[inst], a.Lx, a.Ly, a.Lz, a.pitch, (int)a.plane, a.bc, fin, fout,
           blockIdx.x * 32, blockIdx.y * R, z, sm, a.status, seed, live);
    if (live) finish_step(a.status);
}
