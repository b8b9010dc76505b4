// Moments of one 2D or 3D instance: the wall densities of its columns, then the
// reducer of its lattice kind (glbm_moments.cuh); 3D kinds are instantiated here.
#include "glbm_moments.cuh"

cudaError_t glbm_launch_moments(const AuxArgs &a, const void *f, double *rw, const MomPtrs &out,
                                cudaStream_t s)
{
    MomArgs m = {};
    m.f = f;
    m.ip = a.ip;
    for (int k = 0; k < 9; ++k) m.out[k] = out.p[k];
    m.Lx = a.Lx;
    m.Ly = a.Ly;
    m.Lz = a.Lz;
    m.pitch = a.pitch;
    m.bc = a.bc;
    m.N = a.N;
    m.zv = a.tab.zv;
    m.plane = (int)a.plane;  // Q plane < 2^31 (checked at creation)
    // (odd moments of the rest weights vanish: mirror velocities, equal weights)
    for (int i = 0; i < ax_q(a.tab); ++i) {
        const double v = ax_vel(a.tab, i);
        m.vy[i] = v;
        m.my[0] += a.tab.W[i];
        m.my[2] += v * v * a.tab.W[i];
        // emitted by a wall at distance d: the velocities beyond d
        for (int d = 0; d < (int)v; ++d) {
            double w = a.tab.W[i];
            for (int q = 0; q < 4; ++q, w *= v) m.sw[d][q] += w;
        }
    }
    for (int i = 0; i < ax_q(a.tabx); ++i) {
        const double v = ax_vel(a.tabx, i);
        m.mx[0] += a.tabx.W[i];
        m.mx[2] += v * v * a.tabx.W[i];
    }
    const bool d3 = a.dims == 3;
    const double z0 = d3 ? m.my[0] : 1.0;
    m.rest[0] = m.mx[0] * m.my[0] * z0;
    m.rest[1] = m.mx[2] * m.my[0] * z0;
    m.rest[2] = m.mx[0] * m.my[2] * z0;
    if (a.bc == GLBM_BC_WALLS) {
        m.rw = rw;
        const int cols = a.Lx * a.Lz, QX = ax_q(a.tabx);
        const dim3 grid((cols + WALL_TX - 1) / WALL_TX, 2), blk(WALL_TX * WALL_SL);
        const int v0 = ax_vel(a.tabx, 0), vs = a.tabx.zv ? 2 : 1;
        auto *const kern = d3 ? (a.prec == GLBM_FP64 ? k_moment_walls<3, double> : k_moment_walls<3, float>)
                              : (a.prec == GLBM_FP64 ? k_moment_walls<2, double> : k_moment_walls<2, float>);
        const cudaError_t e = launch_serialized(kern, grid, blk, s, m, QX, v0, vs, rw);
        if (e != cudaSuccess) return e;
    }
    bool full = false;  // any field beyond the density and the velocities
    for (int k = 3; k < 9; ++k) full = full || (k != 7 && out.p[k]);
    if (d3) {
        switch (a.N) {
        case 1: return launch_moments_kind<3, 1, 0>(m, a.prec, full, s);
        case 2: return launch_moments_kind<3, 2, 0>(m, a.prec, full, s);
        case 3: return launch_moments_kind<3, 3, 0>(m, a.prec, full, s);
        default: return cudaErrorInvalidValue;
        }
    }
    return a.tabx.zv ? glbm_moments_2n2(a.NX, m, a.prec, full, s)
                     : glbm_moments_2n1(a.NX, m, a.prec, full, s);
}
