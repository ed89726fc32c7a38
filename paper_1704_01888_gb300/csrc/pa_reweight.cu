// pa_reweight.cu -- the reweighting of population annealing as a function of
// the temperature step, with derivatives (Barash, Weigel, Shchur & Janke,
// arXiv:1704.01888, Sec. 2 step 2), and the adaptive temperature step.
//
//   ln Q(dbeta) = ln( sum_j exp(-dbeta E_j) / R ),  tau_j = exp(-dbeta E_j) / Q,
//   d ln Q / d dbeta = -<E>_tau,   d <E>_tau / d dbeta = -var_tau(E),
//   d var_tau(E) / d dbeta = -k3_tau(E),
//   <O>_tau = sum_j O_j tau_j / R,  d <O>_tau / d dbeta = -cov_tau(O, E),
//   d <O>_tau / d O_j = tau_j / R.
// The sums are taken about the reference energy E_ref (lowest energy for
// dbeta >= 0, highest otherwise) in a fixed order, with explicitly rounded
// double operations.
//
// Adaptive step (the paper uses constant steps; this is a reading added here):
// with mean-one weights t_j = R w_j / S, the overlap of the populations at
// beta and beta + dbeta is alpha = (1/R) sum_j min(1, t_j), with derivative
// alpha' = (1/R) sum_{t_j < 1} t_j (<E>_tau - E_j).  The step solves
// alpha = target by bisection-safeguarded Newton iterations, stopping once
// |alpha - target| <= 1e-12, and is rounded down to a multiple of 2^-24.
#include <climits>
#include <mutex>

#include "../../include/pa.h"
#include "pa_cluster.cuh"

namespace pa {

namespace {

constexpr int kB = 1024;

// Fixed-order block sum; every thread receives the result.
__device__ double bsum(double v, double *sc)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xFFFFFFFFu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sc[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double r = (lane < (int)(blockDim.x >> 5)) ? sc[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r = __dadd_rn(r, __shfl_down_sync(0xFFFFFFFFu, r, o));
        if (lane == 0) sc[0] = r;
    }
    __syncthreads();
    return sc[0];
}

// Block-wide min (lowest = true) or max of ints; every thread receives it.
__device__ int bextreme(int v, bool lowest, int *sc)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const int w = __shfl_down_sync(0xFFFFFFFFu, v, o);
        v = lowest ? min(v, w) : max(v, w);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sc[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int r = (lane < (int)(blockDim.x >> 5)) ? sc[lane] : (lowest ? INT_MAX : INT_MIN);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int w = __shfl_down_sync(0xFFFFFFFFu, r, o);
            r = lowest ? min(r, w) : max(r, w);
        }
        if (lane == 0) sc[0] = r;
    }
    __syncthreads();
    return sc[0];
}

// ---- Block and cluster reductions ---------------------------------------
// The FP64 pipe runs about two lanes per clock and SM (a warp instruction
// occupies it for 16 cycles), so sums are taken with few warp instructions:
// every thread leaves its partial sums in shared memory and warp v alone adds
// up value v (blockDim / 32 values per lane, then five shuffle steps) instead
// of every warp running a shuffle tree.  Fixed order.

constexpr int kClusterMax = 16;

// Sums v[0..NV-1] over the block and, as a tree over the ranks, over the
// cluster; every thread of every block receives the totals.  (Sixteen blocks'
// sums added one after the other round at every sixteenth of the total: S is
// then off by 1.5e-16 in the mean square against 1.0e-16, and 1.1e-16 in one
// block.)  part: NV x blockDim doubles;
// mine[NV]: this block's sums, read by the other blocks.  NV <= blockDim / 32.
// The caller alternates two sets of mine between calls (a block may read the
// others' sums of one call while they write those of the next).  part and total
// need no barrier between calls: a thread writes them again only after a
// barrier that their readers have passed.
template <int NV>
__device__ __forceinline__ void cluster_sum(cg::cluster_group &cl, double (&v)[NV], double *part, double *mine,
                                            double *total)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = blockDim.x;
#pragma unroll
    for (int i = 0; i < NV; ++i) part[i * n + tid] = v[i];
    __syncthreads();
    if (warp < NV) {
        double r = 0.0;
        for (int k = lane; k < n; k += 32) r = __dadd_rn(r, part[warp * n + k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r = __dadd_rn(r, __shfl_down_sync(0xFFFFFFFFu, r, o));
        if (lane == 0) mine[warp] = r;
    }
    cl.sync();
    if (warp < NV) {
        const int C = (int)cl.num_blocks();
        double r = lane < C ? cl.map_shared_rank(mine, lane)[warp] : 0.0;
#pragma unroll
        for (int o = kClusterMax / 2; o > 0; o >>= 1) r = __dadd_rn(r, __shfl_down_sync(0xFFFFFFFFu, r, o));
        if (lane == 0) total[warp] = r;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = total[i];
}

// out[0..7] = ln Q, <E>_tau, var_tau(E), <O>_tau, cov_tau(O, E), E_ref, S, k3_tau(E).
//
// Bound by FP64: one exp and the moments take about 30 FP64 instructions, 16
// cycles per replica on one SM (1640 us for R = 2e5 in one block, 838 us for
// 1e5 with an observable).  One cluster therefore shares the replicas and,
// where the energies span at most kRwBins values and fewer than R, takes the
// moments over an energy histogram: each block counts its replicas in shared
// memory, block c adds up the counts of the c-th slice of the bins over the
// cluster and evaluates one exp per occupied bin.  The observable's sums read
// {w, w e} per replica from a table that the blocks fill in one another's
// shared memory, two fused multiply-adds each.  Otherwise (few replicas, or
// energies spread wider than the table) one exp per replica.
// One launch of one cluster: no workspace to allocate, share or clear.  Now
// 12.8 us for R = 2e5 (two readings of E and three cluster barriers) and 17.0 us
// for 1e5 with an observable (12 more bytes per replica through 16 SMs).
constexpr int kRwThreads = 512;
constexpr int kRwBins = 8192;
constexpr size_t kRwHistBytes = sizeof(int) * kRwBins;
constexpr size_t kRwTableBytes = sizeof(double2) * kRwBins;

__global__ void __launch_bounds__(kRwThreads) k_rw_forward(const int32_t *__restrict__ E, const double *__restrict__ O,
                                                           int R, const double *dbeta_p, double *out)
{
    extern __shared__ uint4 rw_smem[];
    double2 *tab = reinterpret_cast<double2 *>(rw_smem);  // with O only: {w, w e} per bin
    int *hist = reinterpret_cast<int *>(rw_smem) + (O ? kRwTableBytes / sizeof(int) : 0);
    __shared__ double part[6 * kRwThreads];
    __shared__ double mine[6], total[6];
    __shared__ int si[64], ext[2];
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), c = (int)cl.block_rank(), tid = threadIdx.x;
    const int j0 = (int)((long long)R * c / C), j1 = (int)((long long)R * (c + 1) / C);
    const double dbeta = *dbeta_p;
    const bool lowest = dbeta >= 0.0;
    int lo = INT_MAX, hi = INT_MIN;
#pragma unroll 8
    for (int j = j0 + tid; j < j1; j += kRwThreads) {
        const int e = E[j];
        lo = min(lo, e);
        hi = max(hi, e);
    }
    dev::cluster_extremes(cl, lo, hi, si, ext);
    const int ref = lowest ? lo : hi;
    const long long range = (long long)hi - lo + 1;
    double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};  // S, S1, S2, S3, SO, SOe
    if (range <= kRwBins && range < R) {
        const int nb = (int)range;
        for (int b = tid; b < nb; b += kRwThreads) hist[b] = 0;
        __syncthreads();
#pragma unroll 4
        for (int j = j0 + tid; j < j1; j += kRwThreads) atomicAdd(hist + (E[j] - lo), 1);
        cl.sync();
        const int b1 = (int)((long long)nb * (c + 1) / C);
        for (int b = (int)((long long)nb * c / C) + tid; b < b1; b += kRwThreads) {
            int h = 0;
            for (int r = 0; r < C; ++r) h += cl.map_shared_rank(hist, r)[b];
            if (h == 0) continue;
            const double e = (double)(b + lo - ref);
            const double w = exp(__dmul_rn(-dbeta, e));
            const double hw = __dmul_rn((double)h, w);
            const double hwe = __dmul_rn(hw, e);
            const double hwee = __dmul_rn(hwe, e);
            v[0] = __dadd_rn(v[0], hw);
            v[1] = __dadd_rn(v[1], hwe);
            v[2] = __dadd_rn(v[2], hwee);
            v[3] = __dadd_rn(v[3], __dmul_rn(hwee, e));
            if (O) {
                const double2 t = make_double2(w, __dmul_rn(w, e));
                for (int r = 0; r < C; ++r) cl.map_shared_rank(tab, r)[b] = t;
            }
        }
        if (O) {
            cl.sync();
#pragma unroll 4
            for (int j = j0 + tid; j < j1; j += kRwThreads) {
                const double2 t = tab[E[j] - lo];
                const double o = O[j];
                v[4] = __fma_rn(t.x, o, v[4]);
                v[5] = __fma_rn(t.y, o, v[5]);
            }
        }
    } else {
        for (int j = j0 + tid; j < j1; j += kRwThreads) {
            const double e = (double)E[j] - (double)ref;
            const double w = exp(__dmul_rn(-dbeta, e));
            const double we = __dmul_rn(w, e);
            const double wee = __dmul_rn(we, e);
            v[0] = __dadd_rn(v[0], w);
            v[1] = __dadd_rn(v[1], we);
            v[2] = __dadd_rn(v[2], wee);
            v[3] = __dadd_rn(v[3], __dmul_rn(wee, e));
            if (O) {
                const double wo = __dmul_rn(w, O[j]);
                v[4] = __dadd_rn(v[4], wo);
                v[5] = __dadd_rn(v[5], __dmul_rn(wo, e));
            }
        }
    }
    cluster_sum(cl, v, part, mine, total);
    if (c == 0 && tid == 0) {
        const double S = v[0];
        const double m1 = __ddiv_rn(v[1], S);
        const double m2 = __ddiv_rn(v[2], S);
        const double m3 = __ddiv_rn(v[3], S);
        out[0] = __dadd_rn(__dmul_rn(-dbeta, (double)ref), log(__ddiv_rn(S, (double)R)));
        out[1] = __dadd_rn((double)ref, m1);
        out[2] = __dsub_rn(m2, __dmul_rn(m1, m1));
        out[3] = out[4] = 0.0;
        if (O) {
            // cov = (SOe - (SO / S) S1) / S is a small difference of large
            // terms: the residuals of SO / S and of the product come along
            const double mO = __ddiv_rn(v[4], S);
            const double mO_lo = __ddiv_rn(__fma_rn(-mO, S, v[4]), S);
            const double p = __dmul_rn(mO, v[1]), p_lo = __fma_rn(mO, v[1], -p);
            const double cov = __ddiv_rn(__dsub_rn(__dsub_rn(__dsub_rn(v[5], p), p_lo), __dmul_rn(mO_lo, v[1])), S);
            out[3] = mO;
            // sums that overflow have no residuals
            out[4] = isfinite(cov) ? cov : __dsub_rn(__ddiv_rn(v[5], S), __dmul_rn(mO, m1));
        }
        out[5] = (double)ref;
        out[6] = S;
        out[7] = __dadd_rn(__dsub_rn(m3, __dmul_rn(__dmul_rn(3.0, m1), m2)),
                           __dmul_rn(__dmul_rn(__dmul_rn(2.0, m1), m1), m1));
    }
    cl.sync();  // the blocks' shared memory stays until every reader is done
}

// dst[0] = sign * g[0] * src[idx]: the dbeta-gradient of one forward output.
__global__ void k_rw_scale(const double *src, int idx, double sign, const double *g, double *dst)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) dst[0] = __dmul_rn(__dmul_rn(sign, g[0]), src[idx]);
}

// grad_O[j] = g tau_j / R = g exp(-dbeta (E_j - E_ref)) / S.
__global__ void k_rw_grad_O(const int32_t *E, int R, const double *dbeta_p, const double *fwd, const double *g,
                            double *grad_O)
{
    const double dbeta = *dbeta_p;
    // (g / S once per thread would round every gradient once more)
    const double ref = fwd[5], S = fwd[6], gg = g[0];
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < R; j += gridDim.x * blockDim.x) {
        const double w = exp(__dmul_rn(-dbeta, __dsub_rn((double)E[j], ref)));
        grad_O[j] = __dmul_rn(gg, __ddiv_rn(w, S));
    }
}

// Overlap and its derivative over the replicas: out[0..1] = alpha, alpha'.
__global__ void __launch_bounds__(kB) k_overlap(const int32_t *E, int R, const double *dbeta_p, double *out)
{
    __shared__ double sd[32];
    __shared__ int si[32];
    const double dbeta = *dbeta_p;
    const bool lowest = dbeta >= 0.0;
    int ref = lowest ? INT_MAX : INT_MIN;
    for (int j = threadIdx.x; j < R; j += blockDim.x) ref = lowest ? min(ref, E[j]) : max(ref, E[j]);
    ref = bextreme(ref, lowest, si);
    double S = 0.0, S1 = 0.0;
    for (int j = threadIdx.x; j < R; j += blockDim.x) {
        const double e = (double)(E[j] - ref);
        const double w = exp(__dmul_rn(-dbeta, e));
        S = __dadd_rn(S, w);
        S1 = __dadd_rn(S1, __dmul_rn(w, e));
    }
    S = bsum(S, sd);
    S1 = bsum(S1, sd);
    const double m1 = __ddiv_rn(S1, S);
    double a = 0.0, da = 0.0;
    for (int j = threadIdx.x; j < R; j += blockDim.x) {
        const double e = (double)(E[j] - ref);
        const double t = __ddiv_rn(__dmul_rn((double)R, exp(__dmul_rn(-dbeta, e))), S);
        if (t < 1.0) {
            a = __dadd_rn(a, t);
            da = __dadd_rn(da, __dmul_rn(t, __dsub_rn(m1, e)));
        } else {
            a = __dadd_rn(a, 1.0);
        }
    }
    a = bsum(a, sd);
    da = bsum(da, sd);
    if (threadIdx.x == 0) {
        out[0] = __ddiv_rn(a, (double)R);
        out[1] = __ddiv_rn(da, (double)R);
    }
}

// The Newton step on the current population's histogram.
//
// Every evaluation of the overlap takes an exp per occupied bin and two
// dependent sums over the bins.  In one block that is bound by the SM's FP64
// pipe and by two scans of all 2N + 1 bins (185 us at q = 8, L = 128 with 10^4
// replicas, about 2000 occupied bins; now 51 us, two cluster barriers and one
// exp per thread and evaluation).  One cluster shares the occupied range:
// block c keeps the c-th slice of it in shared memory, the weights of the
// first sum are kept for the second, and every block takes the same Newton
// decisions from the same cluster-wide sums.  Slices beyond the shared arrays
// (energies spread over more than C x kNewtonBins bins) read the histogram
// and evaluate exp again.
constexpr int kNewtonThreads = 256;
constexpr int kNewtonBins = 2048;

struct NewtonShared {
    int h[kNewtonBins];
    double w[kNewtonBins];
    double part[2 * kNewtonThreads];
    double mine[2][2], total[2];
    int si[64], ext[2];
};

__global__ void __launch_bounds__(kNewtonThreads) k_newton_hist(const int32_t *__restrict__ hist, int nbins,
                                                                const DevState *st, double target, double cap,
                                                                int iters, double *out)
{
    __shared__ NewtonShared sh;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), c = (int)cl.block_rank(), tid = threadIdx.x;
    int kmin = INT_MAX, kmax = INT_MIN;
    const int stride = C * kNewtonThreads;
#pragma unroll 8
    for (int k = c * kNewtonThreads + tid; k < nbins; k += stride)
        if (hist[k] > 0) {
            kmin = min(kmin, k);
            kmax = max(kmax, k);
        }
    dev::cluster_extremes(cl, kmin, kmax, sh.si, sh.ext);
    const long long range = kmin <= kmax ? (long long)kmax - kmin + 1 : 0;
    const int k0 = kmin + (int)(range * c / C);
    const int m = (int)(range * (c + 1) / C) - (int)(range * c / C);
    const bool kept = m <= kNewtonBins;
    if (kept)
        for (int i = tid; i < m; i += kNewtonThreads) sh.h[i] = hist[k0 + i];  // own entries only: no barrier needed
    const double R = (double)st->pop;
    int set = 0;
    auto overlap = [&](double x, double *a_out, double *da_out) {
        double v[2] = {0.0, 0.0};
        for (int i = tid; i < m; i += kNewtonThreads) {
            const int h = kept ? sh.h[i] : hist[k0 + i];
            if (h == 0) continue;
            const double e = (double)(k0 + i - kmin);
            const double w = exp(__dmul_rn(-x, e));
            if (kept) sh.w[i] = w;
            const double hw = __dmul_rn((double)h, w);
            v[0] = __dadd_rn(v[0], hw);
            v[1] = __dadd_rn(v[1], __dmul_rn(hw, e));
        }
        cluster_sum(cl, v, sh.part, sh.mine[set], sh.total);
        set ^= 1;
        const double S = v[0], m1 = __ddiv_rn(v[1], v[0]);
        v[0] = v[1] = 0.0;
        for (int i = tid; i < m; i += kNewtonThreads) {
            const int h = kept ? sh.h[i] : hist[k0 + i];
            if (h == 0) continue;
            const double e = (double)(k0 + i - kmin);
            const double w = kept ? sh.w[i] : exp(__dmul_rn(-x, e));
            const double t = __ddiv_rn(__dmul_rn(R, w), S);
            if (t < 1.0) {
                v[0] = __dadd_rn(v[0], __dmul_rn((double)h, t));
                v[1] = __dadd_rn(v[1], __dmul_rn((double)h, __dmul_rn(t, __dsub_rn(m1, e))));
            } else {
                v[0] = __dadd_rn(v[0], (double)h);
            }
        }
        cluster_sum(cl, v, sh.part, sh.mine[set], sh.total);
        set ^= 1;
        *a_out = __ddiv_rn(v[0], R);
        *da_out = __ddiv_rn(v[1], R);
    };
    double a, da;
    overlap(cap, &a, &da);
    double x;
    if (a >= target) {
        x = cap;
    } else {
        double lo = 0.0, hi = cap;
        x = __dmul_rn(0.5, __dadd_rn(lo, hi));
        for (int it = 0; it < iters; ++it) {
            overlap(x, &a, &da);
            const double f = __dsub_rn(a, target);
            if (fabs(f) <= 1e-12) break;  // converged: stop before rounding noise decides the bracket
            if (f > 0.0) lo = x; else hi = x;
            double nx = da != 0.0 ? __dsub_rn(x, __ddiv_rn(f, da)) : __dmul_rn(0.5, __dadd_rn(lo, hi));
            if (!(nx > lo && nx < hi)) nx = __dmul_rn(0.5, __dadd_rn(lo, hi));
            x = nx;
        }
        const double qx = floor(__dmul_rn(x, 16777216.0)) / 16777216.0;
        x = qx > 0.0 ? qx : 1.0 / 16777216.0;
    }
    if (c == 0 && tid == 0) {
        out[0] = x;
        out[1] = a;
        out[2] = (double)range;  // bins from the lowest to the highest occupied one
    }
    cl.sync();  // the blocks' shared memory stays until every reader is done
}

// Blocks of the largest cluster of `kernel` with `smem` bytes that this
// device runs: 16 (above the portable 8) where a GPU cluster has that many
// SMs free of other limits, else 8.
template <typename K>
int cluster_blocks(K kernel, int threads, size_t smem)
{
    cudaError_t e =
        launch_result(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (e != cudaSuccess) return 0;  // not kept: the next call asks again
    int n = 0;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kClusterMax;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(kClusterMax);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
    }
    if (e != cudaSuccess) (void)cudaGetLastError();  // a refused size is no error of the caller's
    return e == cudaSuccess && n > 0 ? kClusterMax : 8;
}

// The cluster size of a kernel, looked up once per device.
struct ClusterSize {
    std::mutex mu;
    int blocks[64] = {};
    template <typename K>
    int get(K kernel, int threads, size_t smem)
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
        std::lock_guard<std::mutex> lock(mu);
        if (!blocks[dev]) blocks[dev] = cluster_blocks(kernel, threads, smem);
        return blocks[dev];
    }
};

ClusterSize g_rw_cluster, g_newton_cluster;

}  // namespace

cudaError_t launch_newton(const int32_t *hist, int nbins, const DevState *st, double target, double cap, int iters,
                          double *out, cudaStream_t s)
{
    const int C = g_newton_cluster.get(k_newton_hist, kNewtonThreads, 0);
    bump_launch_count(1);
    return launch_clusters(k_newton_hist, C, C, kNewtonThreads, 0, s, hist, nbins, st, target, cap, iters, out);
}

}  // namespace pa

extern "C" {

pa_status pa_reweight_forward(const int32_t *E, const double *O, int32_t R, const double *dbeta, double *out,
                              void *stream)
{
    if (!E || !dbeta || !out || R < 1) return PA_ERR_INVALID;
    const size_t smem = pa::kRwHistBytes + (O ? pa::kRwTableBytes : 0);
    const int C = pa::g_rw_cluster.get(pa::k_rw_forward, pa::kRwThreads, pa::kRwHistBytes + pa::kRwTableBytes);
    pa::bump_launch_count(1);
    // a small population does not fill a cluster: one block per 1024 replicas
    int blocks = C;
    while (blocks > 1 && (long long)(blocks / 2) * 1024 >= R) blocks /= 2;
    const cudaError_t e = pa::launch_clusters(pa::k_rw_forward, blocks, blocks, pa::kRwThreads, smem,
                                              (cudaStream_t)stream, E, O, R, dbeta, out);
    return e == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}

pa_status pa_reweight_scale(const double *src, int32_t idx, double sign, const double *g, double *dst, void *stream)
{
    if (!src || !g || !dst || idx < 0 || idx > 7) return PA_ERR_INVALID;
    pa::k_rw_scale<<<1, 32, 0, (cudaStream_t)stream>>>(src, idx, sign, g, dst);
    pa::bump_launch_count(1);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}

pa_status pa_reweight_grad_O(const int32_t *E, int32_t R, const double *dbeta, const double *fwd, const double *g,
                             double *grad_O, void *stream)
{
    if (!E || !dbeta || !fwd || !g || !grad_O || R < 1) return PA_ERR_INVALID;
    int grid = (R + 255) / 256;
    if (grid > 4096) grid = 4096;
    pa::k_rw_grad_O<<<grid, 256, 0, (cudaStream_t)stream>>>(E, R, dbeta, fwd, g, grad_O);
    pa::bump_launch_count(1);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}

pa_status pa_overlap(const int32_t *E, int32_t R, const double *dbeta, double *out, void *stream)
{
    if (!E || !dbeta || !out || R < 1) return PA_ERR_INVALID;
    pa::k_overlap<<<1, pa::kB, 0, (cudaStream_t)stream>>>(E, R, dbeta, out);
    pa::bump_launch_count(1);
    return cudaGetLastError() == cudaSuccess ? PA_OK : PA_ERR_CUDA;
}

}  // extern "C"
