// Auxiliary kernels of libglbm: import/export of populations in the FP64 logical
// layout, the 1D moment reducer (2D and 3D: glbm_moments.cuh), deterministic global
// sums, and the 1D step (Sec. 5.1 shock tube, halfway bounce-back) both per launch
// and resident in one CTA for many steps.
#include <algorithm>
#include <mutex>

#include "glbm_node1d.cuh"

namespace {

__device__ __forceinline__ double load_full(const AuxArgs &a, const void *f, long long idx)
{
    if (a.prec == GLBM_FP64) return static_cast<const double *>(f)[idx];
    return (double)static_cast<const float *>(f)[idx];
}

// rest weight of flat velocity q (q = iy Qx + ix in 2D, (iz Q1 + iy) Q1 + ix in 3D)
__device__ __forceinline__ double rest_weight(const AuxArgs &a, int q)
{
    if (a.dims == 1) return a.tab.W[q];
    if (a.dims == 3) {
        const int Q1 = ax_q(a.tab);
        return a.tab.W[q / (Q1 * Q1)] * a.tab.W[(q / Q1) % Q1] * a.tab.W[q % Q1];
    }
    const int Qx = ax_q(a.tabx);
    return a.tab.W[q / Qx] * a.tabx.W[q % Qx];
}

// Import and export of populations in the FP64 logical layout. FP32 deviations: one
// FP64 addition per population (conversions and the velocity's rest weight, formed
// per population, took three slots of the FP64 pipe and bound the copies), COPY_ROWS
// rows per thread in flight. D2Q81 2048 x 256 (510 MB each), GB300, import plus
// export: 496 -> 203 us. Grid: columns, rows, velocities.
constexpr int COPY_ROWS = 8;

template <typename T, bool SET>
__global__ void __launch_bounds__(128)
    k_copy_populations(const __grid_constant__ AuxArgs a, T *f, double *p, unsigned *status)
{
    if (SET && blockIdx.x + blockIdx.y + blockIdx.z + threadIdx.x == 0) reset_status(status);
    const int x = blockIdx.x * 128 + threadIdx.x, q = blockIdx.z;
    if (x >= a.Lx) return;
    const int rows = a.Ly * a.Lz, y0 = blockIdx.y * COPY_ROWS;
    const double w = sizeof(T) == 4 ? rest_weight(a, q) : 0.0;
    f += (long long)q * a.plane + (long long)y0 * a.pitch + x;
    p += ((long long)q * rows + y0) * a.Lx + x;
    const int n = min(COPY_ROWS, rows - y0);
    if constexpr (SET) {
        double v[COPY_ROWS];
#pragma unroll
        for (int r = 0; r < COPY_ROWS; ++r)
            if (r < n) v[r] = __ldcs(p + (long long)r * a.Lx);
#pragma unroll
        for (int r = 0; r < COPY_ROWS; ++r) {
            if (r >= n) continue;
            if constexpr (sizeof(T) == 4)
                f[(long long)r * a.pitch] = d2f(v[r] - w);
            else
                f[(long long)r * a.pitch] = v[r];
        }
    } else {
        T v[COPY_ROWS];
#pragma unroll
        for (int r = 0; r < COPY_ROWS; ++r)
            if (r < n) v[r] = f[(long long)r * a.pitch];
#pragma unroll
        for (int r = 0; r < COPY_ROWS; ++r) {
            if (r >= n) continue;
            __stcs(p + (long long)r * a.Lx, sizeof(T) == 4 ? to_f64(v[r]) + w : to_f64(v[r]));
        }
    }
}

// Moments of S(X) of a 1D lattice: rho, u_x, T and q_x at every node. One thread
// per node takes the mirror pairs (+n, -n) (their sum for the even powers of xi,
// their difference for the odd ones) with halfway bounce-back or periodic ends;
// FP32 deviations are summed as stored and the rest weights' moments added once
// (a reflected population has its mirror's weight). FP64 throughout.
__global__ void k_moments1d(const __grid_constant__ AuxArgs a, const void *f, MomPtrs out)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= a.Lx) return;
    const int N = a.N;
    const auto pulled = [&](int n) {
        int xs = x - n;
        if (a.bc == GLBM_BC_PERIODIC) {
            xs = wrap_shift(xs, a.Lx, a.Lx > N);
        } else if (xs < 0) {
            xs = -1 - xs;
            n = -n;
        } else if (xs >= a.Lx) {
            xs = 2 * a.Lx - 1 - xs;
            n = -n;
        }
        return load_full(a, f, (long long)(N + n) * a.plane + xs);
    };
    double R0 = pulled(0), R1 = 0.0, R2 = 0.0, R3 = 0.0, c = 0.0;
    double w0 = a.tab.W[N], w2 = 0.0;
    for (int n = 1; n <= N; ++n) {
        const double vp = pulled(n), vm = pulled(-n);
        c += 1.0;
        const double c2 = c * c, s = vp + vm, d = c * (vp - vm), w = 2.0 * a.tab.W[N + n];
        R0 += s;
        R1 += d;
        R2 = fma(c2, s, R2);
        R3 = fma(c2, d, R3);
        w0 += w;
        w2 = fma(c2, w, w2);
    }
    if (a.prec != GLBM_FP64) {
        R0 += w0;
        R2 += w2;
    }
    const double u = R1 / R0;
    if (out.p[0]) out.p[0][x] = R0;
    if (out.p[1]) out.p[1][x] = u;
    // central moments about u from the raw ones (R1 = rho u)
    if (out.p[3]) out.p[3][x] = fma(-u, R1, R2) / R0;
    if (out.p[4]) out.p[4][x] = 0.5 * fma(-u, 3.0 * R2 - 2.0 * (u * R1), R3);
}

// Deterministic sums of rho, rho u_x, rho u_y over n nodes: every block sums a
// fixed contiguous range in a fixed tree order; a second launch adds the
// block partials in index order.
constexpr int SUM_THREADS = 256;

__global__ void k_field_partials(const double *__restrict__ fields, int nfields, long long n,
                                 double *__restrict__ partials)
{
    __shared__ double sh[3][SUM_THREADS];
    const long long per = (n + gridDim.x - 1) / gridDim.x;
    const long long lo = blockIdx.x * per;
    const long long hi = min(n, lo + per);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (long long i = lo + threadIdx.x; i < hi; i += SUM_THREADS) {
        const double r = fields[i];
        s0 += r;
        s1 += r * fields[n + i];
        if (nfields > 2) s2 += r * fields[2 * n + i];
    }
    sh[0][threadIdx.x] = s0;
    sh[1][threadIdx.x] = s1;
    sh[2][threadIdx.x] = s2;
    __syncthreads();
    for (int stride = SUM_THREADS / 2; stride > 0; stride >>= 1) {
        if ((int)threadIdx.x < stride)
            for (int m = 0; m < 3; ++m) sh[m][threadIdx.x] += sh[m][threadIdx.x + stride];
        __syncthreads();
    }
    if (threadIdx.x < 3) partials[blockIdx.x * 3 + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void k_field_final(const double *__restrict__ partials, int nblocks, double *out)
{
    if (threadIdx.x < 3) {
        double s = 0.0;
        for (int b = 0; b < nblocks; ++b) s += partials[b * 3 + threadIdx.x];
        out[threadIdx.x] = s;
    }
}

// ---------------------------------------------------------------------------
// Channel diagnostics (Sec. 5.3, 5.4) from the moment fields of one instance
// (rho at field 0, u_x at field 1, each [z][y][x]): the row means over x (and
// z) of u_x and rho u_x, then the flow rate, the volumetric flow and the slip
// ratios. FP64, every sum in a fixed order (deterministic).
// ---------------------------------------------------------------------------
constexpr int ROW_THREADS = 256;

// Fixed tree over ROW_THREADS shared values (two arrays at once).
__device__ __forceinline__ void tree2(double *a, double *b)
{
    __syncthreads();
    for (int stride = ROW_THREADS / 2; stride > 0; stride >>= 1) {
        if ((int)threadIdx.x < stride) {
            a[threadIdx.x] += a[threadIdx.x + stride];
            b[threadIdx.x] += b[threadIdx.x + stride];
        }
        __syncthreads();
    }
}

// Block y: prof[y] = mean over (z, x) of u_x, prof[Ly + y] = mean of rho u_x.
__global__ void k_row_means(const double *__restrict__ mom, int Lx, int Ly, int Lz,
                            double *__restrict__ prof)
{
    __shared__ double su[ROW_THREADS], sj[ROW_THREADS];
    const int y = blockIdx.x;
    const long long plane = (long long)Lx * Ly * Lz;
    double a = 0.0, b = 0.0;
    for (int z = 0; z < Lz; ++z)
        for (int x = threadIdx.x; x < Lx; x += ROW_THREADS) {
            const long long node = ((long long)z * Ly + y) * Lx + x;
            const double u = mom[plane + node];
            a += u;
            b += mom[node] * u;
        }
    su[threadIdx.x] = a;
    sj[threadIdx.x] = b;
    tree2(su, sj);
    if (threadIdx.x == 0) {
        const double n = (double)Lx * (double)Lz;
        prof[y] = su[0] / n;
        prof[Ly + y] = sj[0] / n;
    }
}

// One block: stats[GLBM_CH_*] from the row means (see glbm_channel_diagnostics).
__global__ void k_channel_stats(const double *__restrict__ prof, int Ly, ChannelParams p,
                                double *__restrict__ stats)
{
    __shared__ double su[ROW_THREADS], sj[ROW_THREADS];
    double a = 0.0, b = 0.0;
    for (int y = threadIdx.x; y < Ly; y += ROW_THREADS) {
        a += prof[y];
        b += prof[Ly + y];
    }
    su[threadIdx.x] = a;
    sj[threadIdx.x] = b;
    tree2(su, sj);
    if (threadIdx.x == 0) {
        const double nan = __longlong_as_double(0x7FF8000000000000LL);
        const double H = (double)Ly;
        // volumetric flow Q = (1/Kn) int_0^H u dy / (4 U0 H), U0 = g H^2 / (8 nu)
        const double nu = p.theta_y * p.tau;
        const double U0 = p.g * H * H / (8.0 * nu);
        const double kn = p.tau * sqrt(2.0 * p.theta_y) / H;  // Eq. (kn) with nu = theta tau
        stats[GLBM_CH_FLOW_RATE] = sj[0];
        stats[GLBM_CH_VOLUMETRIC] = p.g != 0.0 ? su[0] / (kn * 4.0 * U0 * H) : nan;
        // the row means extrapolated linearly to the wall planes y = -1/2, Ly - 1/2
        const double ulo = Ly > 1 ? 1.5 * prof[0] - 0.5 * prof[1] : prof[0];
        const double uhi = Ly > 1 ? 1.5 * prof[Ly - 1] - 0.5 * prof[Ly - 2] : prof[Ly - 1];
        const double du = p.u_hi - p.u_lo;
        stats[GLBM_CH_U_LO] = p.walls ? ulo : nan;
        stats[GLBM_CH_U_HI] = p.walls ? uhi : nan;
        stats[GLBM_CH_SLIP_LO] = p.walls && du != 0.0 ? (ulo - p.u_lo) / du : nan;
        stats[GLBM_CH_SLIP_HI] = p.walls && du != 0.0 ? (p.u_hi - uhi) / du : nan;
    }
}

// ---------------------------------------------------------------------------
// 1D step (glbm_node1d.cuh), one thread per node: a launch per step, or many steps
// of a small lattice in one CTA. Most calls take the cluster of glbm_run1d.cu; these
// serve the lattices it does not hold and the calls whose run fails inside it.
// ---------------------------------------------------------------------------
template <int N, typename T>
__global__ void k_step1d(const __grid_constant__ AuxArgs a, const T *__restrict__ fin,
                         T *__restrict__ fout, int inst, unsigned *status)
{
    if (step_halted(status)) return;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < a.Lx) node1d_at<N, T>(a, a.ip[inst], fin, fout, x, a.Lx, a.plane, status);
    finish_step(status);
}

// Many steps of one small 1D lattice inside one CTA: both population copies
// live in shared memory and a block barrier separates the steps, so the whole
// run is one launch (the shock tube is launch-latency bound, not HBM bound).
template <int N, typename T>
__global__ void k_run1d_resident(const __grid_constant__ AuxArgs a, T *__restrict__ f,
                                 int inst, long long steps, unsigned *status)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned bad;
    constexpr int Q1 = 2 * N + 1;
    if (step_halted(status)) return;  // an earlier step left the positivity domain
    const int L = a.Lx;
    T *A = reinterpret_cast<T *>(smem_raw);
    T *B = A + (long long)Q1 * L;
    for (int i = threadIdx.x; i < Q1 * L; i += blockDim.x) {
        const int q = i / L, x = i % L;
        A[i] = f[(long long)q * a.plane + x];
    }
    if (threadIdx.x == 0) bad = 0u;
    __syncthreads();
    long long done = 0;
    while (done < steps) {
        for (int x = threadIdx.x; x < L; x += blockDim.x)
            node1d_at<N, T>(a, a.ip[inst], A, B, x, L, L, status);
        __syncthreads();  // the step's flags (global atomics of this block) are visible
        T *tmp = A;
        A = B;
        B = tmp;
        ++done;
        // stop after a step that left the positivity domain: one read,
        // broadcast, so that every thread leaves the loop at the same step
        if (threadIdx.x == 0) bad = __ldcg(status + ST_FLAGS) & 1u;
        __syncthreads();
        if (bad) break;
    }
    for (int i = threadIdx.x; i < Q1 * L; i += blockDim.x) {
        const int q = i / L, x = i % L;
        f[(long long)q * a.plane + x] = A[i];
    }
    if (threadIdx.x == 0) {
        atomicAdd(status + ST_STEPS, (unsigned)done);
        if (bad) atomicExch(status + ST_HALT, 1u);
    }
}

template <typename T>
cudaError_t launch_step1d_t(const AuxArgs &a, const void *fin, void *fout, int inst,
                            unsigned *status, cudaStream_t s)
{
    const T *in = static_cast<const T *>(fin) + (long long)inst * a.inst_stride;
    T *out = static_cast<T *>(fout) + (long long)inst * a.inst_stride;
    const int threads = 128;
    const int blocks = (a.Lx + threads - 1) / threads;
    switch (a.N) {
#define GLBM_CASE(NN) \
    case NN: k_step1d<NN, T><<<blocks, threads, 0, s>>>(a, in, out, inst, status); break;
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

constexpr int RESIDENT_SMEM = 200 * 1024;

template <int N, typename T>
cudaError_t launch_resident_n(const AuxArgs &a, T *f, int inst, long long steps,
                              unsigned *status, cudaStream_t s, size_t smem)
{
    // (one limit for every launch: a smaller one set by another thread in between
    // would refuse this one)
    cudaError_t e = cudaFuncSetAttribute(k_run1d_resident<N, T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, RESIDENT_SMEM);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;  // FP64 of the higher levels: fewer threads than 1024 fit
    e = cudaFuncGetAttributes(&fa, k_run1d_resident<N, T>);
    if (e != cudaSuccess) return e;
    const int most = fa.maxThreadsPerBlock / 32 * 32;
    const int threads = std::min(most, ((a.Lx + 31) / 32) * 32);
    k_run1d_resident<N, T><<<1, threads, smem, s>>>(a, f, inst, steps, status);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_resident_t(const AuxArgs &a, void *fv, int inst, long long steps,
                              unsigned *status, cudaStream_t s, int *ok)
{
    const size_t smem = (size_t)2 * (2 * a.N + 1) * a.Lx * sizeof(T);
    *ok = 0;
    if (smem > RESIDENT_SMEM) return cudaSuccess;  // caller falls back to per-step launches
    *ok = 1;
    T *f = static_cast<T *>(fv) + (long long)inst * a.inst_stride;
    switch (a.N) {
#define GLBM_CASE(NN) \
    case NN: return launch_resident_n<NN, T>(a, f, inst, steps, status, s, smem);
        GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4)
        GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

static int velocities(const AuxArgs &a)
{
    const int q = ax_q(a.tab);
    return a.dims == 3 ? q * q * q : (a.dims == 2 ? q * ax_q(a.tabx) : q);
}

template <bool SET>
static cudaError_t copy_populations(const AuxArgs &a, void *f, double *p, unsigned *status,
                                    cudaStream_t s)
{
    const dim3 grid((a.Lx + 127) / 128, (a.Ly * a.Lz + COPY_ROWS - 1) / COPY_ROWS, velocities(a));
    if (a.prec == GLBM_FP64)
        k_copy_populations<double, SET><<<grid, 128, 0, s>>>(a, static_cast<double *>(f), p, status);
    else
        k_copy_populations<float, SET><<<grid, 128, 0, s>>>(a, static_cast<float *>(f), p, status);
    return cudaGetLastError();
}

cudaError_t glbm_launch_set_populations(const AuxArgs &a, void *f, const double *src,
                                        unsigned *status, cudaStream_t s)
{
    return copy_populations<true>(a, f, const_cast<double *>(src), status, s);
}

cudaError_t glbm_launch_get_populations(const AuxArgs &a, const void *f, double *dst, cudaStream_t s)
{
    return copy_populations<false>(a, const_cast<void *>(f), dst, nullptr, s);
}

cudaError_t glbm_launch_moments1d(const AuxArgs &a, const void *f, const MomPtrs &out,
                                  cudaStream_t s)
{
    k_moments1d<<<(a.Lx + 31) / 32, 32, 0, s>>>(a, f, out);
    return cudaGetLastError();
}

int glbm_field_sum_blocks(long long n)
{
    long long b = (n + 4095) / 4096;
    if (b < 1) b = 1;
    if (b > 1024) b = 1024;
    return (int)b;
}

cudaError_t glbm_launch_field_sums(const double *fields, int nfields, long long n, double *partials,
                                   int nblocks, double *out, cudaStream_t s)
{
    k_field_partials<<<nblocks, SUM_THREADS, 0, s>>>(fields, nfields, n, partials);
    k_field_final<<<1, 32, 0, s>>>(partials, nblocks, out);
    return cudaGetLastError();
}

cudaError_t glbm_launch_step1d(const AuxArgs &a, const void *fin, void *fout, int inst,
                               unsigned *status, cudaStream_t s)
{
    if (a.prec == GLBM_FP64) return launch_step1d_t<double>(a, fin, fout, inst, status, s);
    return launch_step1d_t<float>(a, fin, fout, inst, status, s);
}

cudaError_t glbm_launch_run1d_resident(const AuxArgs &a, void *f, int inst, long long steps,
                                       unsigned *status, cudaStream_t s, int *ok)
{
    if (a.prec == GLBM_FP64) return launch_resident_t<double>(a, f, inst, steps, status, s, ok);
    return launch_resident_t<float>(a, f, inst, steps, status, s, ok);
}

// ---------------------------------------------------------------------------
// Conservation sums without allocation (glbm_conservation_noalloc).
//
// The block partials of the deterministic sum live in this file-scope device
// array instead of context memory, for callers that may not allocate device
// memory. Every GPU that loads the library holds it (24 KiB) until the process
// exits, and every call shares it.
// ---------------------------------------------------------------------------
#define GLBM_NOALLOC_MAX_BLOCKS 1024
static __device__ __align__(256) double g_noalloc_partials[3 * GLBM_NOALLOC_MAX_BLOCKS];

static std::mutex g_noalloc_mu;
static void *g_noalloc_ptr[64];  // device address of g_noalloc_partials, per device

extern "C" glbm_status glbm_conservation_noalloc(const double *fields, int dims, int64_t nodes,
                                                 double *sums, void *stream)
{
    if (!fields || !sums) return glbm_set_error(GLBM_E_INVAL, "null fields or sums");
    if (dims != 1 && dims != 2) return glbm_set_error(GLBM_E_INVAL, "dims must be 1 or 2");
    if (nodes < 1 || nodes > GLBM_NOALLOC_MAX_NODES)
        return glbm_set_error(GLBM_E_INVAL,
                              "glbm_conservation_noalloc takes 1 to %lld nodes (got %lld): its "
                              "static scratch holds %d block partials of 4096 nodes",
                              (long long)GLBM_NOALLOC_MAX_NODES, (long long)nodes,
                              GLBM_NOALLOC_MAX_BLOCKS);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return glbm_set_error(GLBM_E_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= 64) return glbm_set_error(GLBM_E_UNSUPPORTED, "device index %d >= 64", dev);
    void *scratch = nullptr;
    {
        // set-up once per device, with that device current: in host code the
        // array's name is only a stand-in, its device address comes from here
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            e = cudaGetSymbolAddress(&g_noalloc_ptr[dev], g_noalloc_partials);
            if (e != cudaSuccess) {
                g_noalloc_ptr[dev] = nullptr;
                return glbm_set_error(GLBM_E_CUDA, "cudaGetSymbolAddress of the scratch: %s",
                                      cudaGetErrorString(e));
            }
        }
        scratch = g_noalloc_ptr[dev];
    }
    // every block writes all three of its partials before the final pass reads
    // them, so nothing has to be cleared between calls
    const int nblocks = glbm_field_sum_blocks(nodes);
    e = glbm_launch_field_sums(fields, dims == 2 ? 3 : 2, nodes, static_cast<double *>(scratch),
                               nblocks, sums, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return glbm_set_error(GLBM_E_CUDA, "launch: %s", cudaGetErrorString(e));
    return GLBM_OK;
}

cudaError_t glbm_launch_channel_diagnostics(const double *mom, int Lx, int Ly, int Lz,
                                            const ChannelParams &p, double *prof, double *stats,
                                            cudaStream_t s)
{
    k_row_means<<<Ly, ROW_THREADS, 0, s>>>(mom, Lx, Ly, Lz, prof);
    k_channel_stats<<<1, ROW_THREADS, 0, s>>>(prof, Ly, p, stats);
    return cudaGetLastError();
}

// FP64 FMA throughput probe (glbm_measure_fp64_rate): a measurement aid for the
// FP64 roofline, not part of the method. Every thread runs 8 independent FMA
// chains (enough independent work per warp to keep the FP64 pipe busy), and
// the sum goes to a sink only when it takes a value it never takes, so the
// chains are not removed.
namespace {
constexpr int PROBE_CHAINS = 8;

__global__ void k_fp64_rate(double *sink, int iters, double a, double b)
{
    double x[PROBE_CHAINS];
#pragma unroll
    for (int c = 0; c < PROBE_CHAINS; ++c) x[c] = 1e-3 * (threadIdx.x + c);
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int c = 0; c < PROBE_CHAINS; ++c) x[c] = fma(x[c], a, b);
    }
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < PROBE_CHAINS; ++c) s += x[c];
    if (s == -1.0) sink[threadIdx.x] = s;
}
}  // namespace

extern "C" glbm_status glbm_measure_fp64_rate(void *stream, double *fma_per_s)
{
    if (!fma_per_s) return glbm_set_error(GLBM_E_INVAL, "null argument");
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    double *sink = nullptr;
    if (e == cudaSuccess) e = cudaMalloc(&sink, 256 * sizeof(double));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    const int threads = 256, blocks = sms * 8, iters = 4096;
    double best = 0.0;
    for (int rep = 0; rep < 3 && e == cudaSuccess; ++rep) {
        cudaEventRecord(e0, s);
        k_fp64_rate<<<blocks, threads, 0, s>>>(sink, iters, 0.9999999, 1e-7);
        cudaEventRecord(e1, s);
        e = cudaEventSynchronize(e1);
        float ms = 0.0f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        const double rate = (double)blocks * threads * iters * PROBE_CHAINS / (ms * 1e-3);
        if (e == cudaSuccess && rep > 0 && rate > best) best = rate;  // the first run warms up
    }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (sink) cudaFree(sink);
    if (e != cudaSuccess) return glbm_set_error(GLBM_E_CUDA, "FP64 probe: %s", cudaGetErrorString(e));
    *fma_per_s = best;
    return GLBM_OK;
}

// Start of a dataflow chunk (glbm_internal.h): the band counts and the
// per-step CTA counts go back to zero, and ST_BASE takes the step clock that
// the chunk's first step starts from.
namespace {
__global__ void k_df_start(unsigned *status, unsigned *words, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        words[i] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) status[ST_BASE] = status[ST_CLOCK];
}
}  // namespace

cudaError_t glbm_launch_df_start(unsigned *status, unsigned *words, long long n, cudaStream_t s)
{
    const int blocks = (int)std::min<long long>((n + 255) / 256, 1024);
    k_df_start<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(status, words, n);
    return cudaGetLastError();
}
