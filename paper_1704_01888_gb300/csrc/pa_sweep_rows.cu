// pa_sweep_rows.cu -- the throughput sweep kernels (pa_sweep_kernel.cuh) of
// lattices whose rows are not whole words: packed (L = 8, 16, 32), banded (L =
// 48, 80, 96, ...) and padded rows.
#include "pa_sweep_kernel.cuh"

namespace pa {

SweepFn sweep_rows_kernel(int q, int L)
{
    if (rows_packed(L)) return pick_q<3>(q);
    if (rows_banded(L)) return pick_q<4>(q);
    return pick_q<2>(q);
}

}  // namespace pa
