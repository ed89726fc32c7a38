// pa_sweep_lat.cu -- the sweep kernels for launches whose threads have one site
// word each (pa_sweep_kernel.cuh): every acceptance call of a word is drawn by
// its own thread, three of them together with the proposal, so that a half
// sweep is one chain and one barrier; up to 128 registers per thread.  One
// kernel per bit count and row geometry (q from the arguments).
#include "pa_sweep_kernel.cuh"

namespace pa {

namespace {

template <int B, int MODE>
__global__ void __launch_bounds__(512) k_sweep_lat(const SweepArgs a)
{
    sweep_blocks<B, MODE, 0, true>(a);
}

template <int MODE>
SweepFn pick_lat(int q)
{
    switch (state_bits(q)) {
    case 1: return k_sweep_lat<1, MODE>;
    case 2: return k_sweep_lat<2, MODE>;
    case 3: return k_sweep_lat<3, MODE>;
    case 4: return k_sweep_lat<4, MODE>;
    case 5: return k_sweep_lat<5, MODE>;
    case 6: return k_sweep_lat<6, MODE>;
    default: return k_sweep_lat<7, MODE>;
    }
}

}  // namespace

SweepFn sweep_lat_kernel(int q, int L)
{
    if (L == 64) return pick_lat<0>(q);
    if (L % 64 == 0) return pick_lat<1>(q);
    if (rows_packed(L)) return pick_lat<3>(q);
    if (rows_banded(L)) return pick_lat<4>(q);
    return pick_lat<2>(q);
}

}  // namespace pa
