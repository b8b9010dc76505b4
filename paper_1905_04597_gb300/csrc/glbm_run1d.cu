// Many steps of 1D lattices in one launch, each lattice spread over a thread-block
// cluster (the shock tube of Sec. 5.1 is a chain of dependent steps on a few hundred
// to a few thousand nodes).
//
// A step is bound by the latency of one node's arithmetic, and in FP64 by the SMs'
// FP64 pipes: one CTA on one SM left its 32 warps queueing for a pipe that takes 64
// cycles per warp instruction, and every step read the status word from L2. Here
// each CTA of the cluster keeps a chunk of nodes plus H = m N halo nodes per side in
// shared memory and takes m steps on a region that shrinks by N per side and step;
// then the chunk's edges go to the neighbours' halos through distributed shared
// memory, one cluster barrier per m steps (receive buffers alternate, so that one
// barrier orders both the writes and their reuse). The results equal the one-CTA and
// the per-launch steps': every node is computed by the same arithmetic from the same
// values. The input buffer is not written: if a node leaves the positivity domain
// the caller steps again from it one launch after another (or in one CTA), which
// stops at the failing step. Measured on GB300, us per step in calls of 500: D1Q5 x 1000
// FP32 1.70 -> 0.40, D1Q7 x 800 FP64 16.5 -> 2.5.
#include "glbm_node1d.cuh"

namespace {

constexpr int RUN1D_THREADS = 512;
constexpr int RUN1D_SMEM = 200 * 1024;

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned smem_of_rank(const void *p, unsigned rank)
{
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(unsigned addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

struct Run1DArgs {
    AuxArgs a;
    const void *f;     // instance 0 of the input, instances inst_stride elements apart
    void *out;
    long long steps;
    unsigned *status;
    int C, m, maxn;    // CTAs per lattice, steps per exchange, largest chunk
};

template <int N, typename T>
__global__ void __launch_bounds__(RUN1D_THREADS) k_run1d_cluster(const __grid_constant__ Run1DArgs r)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int Q1 = 2 * N + 1;
    const AuxArgs &a = r.a;
    const int L = a.Lx, C = r.C, H = N * r.m, P = r.maxn + 2 * H;
    const int c = blockIdx.x % C, inst = blockIdx.x / C;  // c: the rank in the cluster
    const int lo = (int)((long long)c * L / C), n = (int)((long long)(c + 1) * L / C) - lo;
    const bool periodic = a.bc == GLBM_BC_PERIODIC;
    T *A = reinterpret_cast<T *>(smem_raw), *B = A + Q1 * P;
    T *const inbox = B + Q1 * P;  // [parity][side 0: from the left, 1: from the right][q][H]
    InstParams ip;  // (only the relaxation rate is read)
    ip.omega = a.ip[inst].omega;
    ip.omega_f = a.ip[inst].omega_f;
    const T *const f = static_cast<const T *>(r.f) + (long long)inst * a.inst_stride;
    T *const out = static_cast<T *>(r.out) + (long long)inst * a.inst_stride;
    const int x0 = lo - H;  // lattice coordinate of local index 0
    for (int t = threadIdx.x; t < Q1 * (n + 2 * H); t += blockDim.x) {
        const int q = t / (n + 2 * H), i = t - q * (n + 2 * H);
        int x = x0 + i;
        if (periodic)
            x = wrap_index(x, L);
        else if (x < 0 || x >= L)
            continue;  // never read: bounce-back ends reflect into the lattice
        A[q * P + i] = f[(long long)q * a.plane + x];
    }
    cluster_sync_all();  // every CTA of the cluster has started before the first remote write
    bool bad = false;
    int parity = 0;
    // a chunk and its halos in one node per thread: the places a thread reads stay the
    // same in every step, and it takes part while its node lies in the region, that
    // is for the first `last` steps after an exchange
    const bool one = n + 2 * H <= (int)blockDim.x;
    int off[Q1], last = 0;
    if (one) {
        const int i = threadIdx.x, x = x0 + i;
        if (i < n + 2 * H && (periodic || (x >= 0 && x < L))) last = min(i, n + 2 * H - 1 - i) / N;
#pragma unroll
        for (int ix = 0; ix < Q1; ++ix) {
            int xs = x - (ix - N), q = ix;
            if (!periodic) {
                if (xs < 0) {
                    xs = -1 - xs;
                    q = 2 * N - ix;
                } else if (xs >= L) {
                    xs = 2 * L - 1 - xs;
                    q = 2 * N - ix;
                }
            }
            off[ix] = last > 0 ? q * P + (xs - x0) : 0;
        }
    }
    for (long long done = 0; done < r.steps;) {
        const int b = (int)min((long long)r.m, r.steps - done);
        if (one) {
            for (int s = 1; s <= b; ++s) {
                if (s <= last) {
                    T *const o = B + threadIdx.x;
                    const bool ok = node1d<N, T>(
                        a.tab, ip, [&](int ix) { return A[off[ix]]; },
                        [&](int ix, T v) { o[ix * P] = v; });
                    bad = bad || !ok;
                }
                __syncthreads();
                T *const t = A;
                A = B;
                B = t;
            }
        } else {
            for (int s = 1; s <= b; ++s) {
                int xa = x0 + s * N, xb = lo + n + H - s * N;
                if (!periodic) {
                    xa = max(xa, 0);
                    xb = min(xb, L);
                }
                for (int x = xa + threadIdx.x; x < xb; x += blockDim.x) {
                    const bool ok = node1d<N, T>(
                        a.tab, ip,
                        [&](int ix) {
                            int xs = x - (ix - N), q = ix;
                            if (!periodic) {
                                if (xs < 0) {
                                    xs = -1 - xs;
                                    q = 2 * N - ix;
                                } else if (xs >= L) {
                                    xs = 2 * L - 1 - xs;
                                    q = 2 * N - ix;
                                }
                            }
                            return A[q * P + (xs - x0)];
                        },
                        [&](int ix, T v) { B[ix * P + (x - x0)] = v; });
                    bad = bad || !ok;
                }
                __syncthreads();
                T *const t = A;
                A = B;
                B = t;
            }
        }
        done += b;
        if (done >= r.steps) break;
        // the first and last H owned nodes to the neighbours' inboxes
        T *const box = inbox + parity * 2 * Q1 * H;
        const bool left = periodic || c > 0, right = periodic || c < C - 1;
        const unsigned to_left = smem_of_rank(box + Q1 * H, (unsigned)((c + C - 1) % C));
        const unsigned to_right = smem_of_rank(box, (unsigned)((c + 1) % C));
        for (int t = threadIdx.x; t < Q1 * H; t += blockDim.x) {
            const int q = t / H, k = t - q * H;
            if (left) st_cluster(to_left + t * (unsigned)sizeof(T), A[q * P + H + k]);
            if (right) st_cluster(to_right + t * (unsigned)sizeof(T), A[q * P + n + k]);
        }
        cluster_sync_all();
        for (int t = threadIdx.x; t < Q1 * H; t += blockDim.x) {
            const int q = t / H, k = t - q * H;
            if (left) A[q * P + k] = box[t];
            if (right) A[q * P + H + n + k] = box[Q1 * H + t];
        }
        __syncthreads();
        parity ^= 1;
    }
    for (int t = threadIdx.x; t < Q1 * n; t += blockDim.x) {
        const int q = t / n, i = t - q * n;
        out[(long long)q * a.plane + lo + i] = A[q * P + H + i];
    }
    if (bad) flag_unstable(r.status);
}

void fill_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[1], int C, int ctas, int threads,
                 size_t smem, cudaStream_t s)
{
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// The plan of a kernel: chunks, steps per exchange and the launch's shape. C stays 0
// for lattices that a cluster does not hold.
template <int N, typename T>
void plan_n(int L, Run1DPlan &p)
{
    constexpr int Q1 = 2 * N + 1;
    auto *const kern = k_run1d_cluster<N, T>;
    // chunks of at least 32 nodes; clusters of 16 CTAs are opt-in
    int C = 16;
    while (C > 1 && L / C < 32) C /= 2;
    for (; C >= 1; C /= 2) {
        const int maxn = (L + C - 1) / C;
        // steps per exchange: as many as 16, with the halos inside four warps (one
        // per SM sub-partition) or one more warp than the chunk has, and within the
        // neighbour's chunk
        const int warps = maxn / 32 + 1 > 4 ? maxn / 32 + 1 : 4;
        int m = (32 * warps - maxn) / (2 * N);
        m = m > 16 ? 16 : m;
        if (m > L / C / N) m = L / C / N;
        m = m < 1 ? 1 : m;
        const int H = N * m;
        if (H > L / C) return;  // shorter than the reach: the caller's other paths
        const size_t smem = sizeof(T) * Q1 * (2 * (size_t)(maxn + 2 * H) + 4 * (size_t)H);
        if (smem > RUN1D_SMEM) return;
        // (one limit for every plan: the kernel is shared by contexts of other sizes)
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, RUN1D_SMEM);
        if (e == cudaSuccess && C > 8)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        int threads = (maxn + 2 * H + 31) / 32 * 32;
        threads = threads > RUN1D_THREADS ? RUN1D_THREADS : threads;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        fill_config(cfg, attr, C, C, threads, smem, nullptr);
        int clusters = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
        if (e == cudaSuccess && clusters >= 1) {
            p.C = C;
            p.m = m;
            p.maxn = maxn;
            p.threads = threads;
            p.smem = smem;
            return;
        }
        cudaGetLastError();
        if (C <= 8) return;  // (no GPC holds 16 CTAs: the portable size)
    }
}

template <int N, typename T>
cudaError_t launch_n(const Run1DPlan &p, const Run1DArgs &r, int n_inst, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    fill_config(cfg, attr, p.C, p.C * n_inst, p.threads, p.smem, s);
    return cudaLaunchKernelEx(&cfg, k_run1d_cluster<N, T>, r);
}

}  // namespace

#define GLBM_LEVELS_1D GLBM_CASE(1) GLBM_CASE(2) GLBM_CASE(3) GLBM_CASE(4) \
                       GLBM_CASE(5) GLBM_CASE(6) GLBM_CASE(7) GLBM_CASE(8)

Run1DPlan glbm_plan_run1d(int N, int prec, int L, int n_inst)
{
    Run1DPlan p = {};
    const int Q1 = 2 * N + 1;
    // A cluster has at most 16 of the chip's SMs. In FP64 beyond 3072 nodes it has more
    // warps per SM than pipes to hide them, and one launch per step over the whole
    // chip is as fast. One instance alone stops earlier: at D1Q17 from 2900 nodes
    // (per step, cluster against launches: 2900 13.4 and 14.6 us, 3000 15.5 and 14.5;
    // D1Q15 12.5 and 12.5 at 3072, D1Q3 to D1Q13 1.07 to 2.5 times as fast there), in
    // FP32 from Q L = 256000 (D1Q3 64000 4.8 and 6.3 us, 100000 7.4 and 6.3; D1Q5
    // 50000 6.1 and 6.3, 70000 7.8 and 6.3; D1Q11 24000 6.1 and 6.3, 30000 7.5 and
    // 6.3; D1Q17 15000 6.0 and 6.3, 17000 7.6 and 6.3). Several instances run side by
    // side in clusters but one after another in launches (two: 1.6 times as fast at
    // those sizes). Measured on GB300 in calls of 200 steps.
    if (prec == GLBM_FP64 && L > (N == 8 && n_inst == 1 ? 2900 : 3072)) return p;
    if (prec != GLBM_FP64 && n_inst == 1 && (long long)Q1 * L > 256000) return p;
    switch (N) {
#define GLBM_CASE(NN) \
    case NN: prec == GLBM_FP64 ? plan_n<NN, double>(L, p) : plan_n<NN, float>(L, p); break;
        GLBM_LEVELS_1D
#undef GLBM_CASE
    default: break;
    }
    return p;
}

cudaError_t glbm_launch_run1d_cluster(const Run1DPlan &p, const AuxArgs &a, const void *f, void *out,
                                      int n_inst, long long steps, unsigned *status, cudaStream_t s)
{
    Run1DArgs r;
    r.a = a;
    r.f = f;
    r.out = out;
    r.steps = steps;
    r.status = status;
    r.C = p.C;
    r.m = p.m;
    r.maxn = p.maxn;
    switch (a.N) {
#define GLBM_CASE(NN)                                                   \
    case NN:                                                            \
        return a.prec == GLBM_FP64 ? launch_n<NN, double>(p, r, n_inst, s) \
                                   : launch_n<NN, float>(p, r, n_inst, s);
        GLBM_LEVELS_1D
#undef GLBM_CASE
    default: return cudaErrorInvalidValue;
    }
}
