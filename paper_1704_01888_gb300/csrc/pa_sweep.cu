// pa_sweep.cu -- the Metropolis sweep kernel of population annealing
// (Barash, Weigel, Shchur & Janke, arXiv:1704.01888, Sec. 2 step 3 and Sec. 3),
// fused with the replica gather of the preceding resampling step (Sec. 2 step 2)
// and with the per-replica measurements of step 4 (Eq. 3 energy, Eq. 5
// largest-state occupation) and the energy histogram.
//
// One block keeps `rpb` whole lattices resident in shared memory and runs all
// theta sweeps on them, so HBM sees each lattice once in and once out per
// temperature step.  Blocks are persistent: they stride over groups of rpb
// replicas until the device-side population size is covered.
//
// Spins are multi-spin coded: the states of 32 same-colour sites of a row sit
// in B bit planes (B = ceil(log2 q)), and each thread updates such a site
// word with 32-bit logic: the proposal by ripple-carry additions over the
// planes, the energy change by bitwise equality tests and a carry-save count,
// the acceptance by a most-significant-bit-first comparison of random bits
// with the thresholds (the body is dev::sweep_group_bits).  One kernel is
// compiled per B and row geometry.
#include "pa_sweep_kernel.cuh"

namespace pa {

namespace {

// Allows each kernel the device's full opt-in shared memory (less its static
// shared memory), so that the per-launch request alone decides occupancy.
cudaError_t prepare(SweepFn kernel)
{
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    return e;
}

SweepFn pick_kernel(int q, int L, bool lat)
{
    if (lat) return sweep_lat_kernel(q, L);
    if (L == 64) return pick_q<0>(q);
    if (L % 64 == 0) return pick_q<1>(q);
    return sweep_rows_kernel(q, L);
}

}  // namespace

size_t sweep_smem_bytes(int q, int L, int rpb) { return (size_t)rpb * replica_bytes(q, L); }

int sweep_max_blocks_per_sm(int q, int L, int rpb, int threads, bool lat)
{
    SweepFn k = pick_kernel(q, L, lat);
    const size_t smem = sweep_smem_bytes(q, L, rpb);
    if (prepare(k) != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) return 0;
    return n;
}

cudaError_t launch_sweep(const SweepArgs &a, int threads, int grid, cudaStream_t s)
{
    SweepFn k = pick_kernel(a.q, a.L, a.lat != 0);
    const size_t smem = sweep_smem_bytes(a.q, a.L, a.rpb);
    const cudaError_t e = launch_after(k, 1, grid, threads, smem, s, a);
    bump_launch_count(1);
    return e;
}

}  // namespace pa
