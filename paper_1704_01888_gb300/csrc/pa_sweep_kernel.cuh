// pa_sweep_kernel.cuh -- the persistent block loop of the single-run sweep
// kernels (Barash, Weigel, Shchur & Janke, arXiv:1704.01888, Sec. 2 step 3),
// compiled by three translation units in parallel: the throughput kernels of
// whole-word rows (pa_sweep.cu) and of the other row geometries
// (pa_sweep_rows.cu), and the latency kernels (pa_sweep_lat.cu).
#pragma once
#include "pa_kernels.cuh"

namespace pa {

using SweepFn = void (*)(const SweepArgs);
SweepFn sweep_rows_kernel(int q, int L);  // pa_sweep_rows.cu: packed, banded and padded rows
SweepFn sweep_lat_kernel(int q, int L);   // pa_sweep_lat.cu

namespace {

// Group of the local slots [first, first + nrep).  A population spread over
// several GPUs numbers its replicas by global slot (slot0 + local slot): the
// group carries global slot numbers, for the random keys, and array bases
// moved down by slot0, so that indexing by global slot lands on the local
// entries (slot0 = 0 on one GPU).
__device__ __forceinline__ dev::Group make_group(const SweepArgs &a, int parity, int first, int nrep)
{
    const size_t s0 = a.slot0;
    const size_t RW = (size_t)replica_words(a.q, a.L);
    // arrays indexed by slot move down by slot0; a gather's sources are indexed
    // by the parent map's values, which are local
    const size_t s_in = a.gather ? 0 : s0;
    dev::Group G;
    G.in = a.buf[parity] - s_in * RW;
    G.out = (a.gather ? a.buf[parity ^ 1] : a.buf[parity]) - s0 * RW;
    G.parent = a.parent ? a.parent - s0 : nullptr;
    G.anc_in = a.anc[parity] ? a.anc[parity] - s_in : nullptr;
    G.anc_out = a.gather ? a.anc[parity ^ 1] : a.anc[parity];
    if (G.anc_out) G.anc_out -= s0;
    G.fam = a.fam;
    G.E = a.E - s0;
    G.Mt = a.Mt - s0;
    G.hist = a.hist;
    G.first = (int)a.slot0 + first;
    G.nrep = nrep;
    G.q = a.q;
    G.theta = a.theta;
    G.step = a.step;
    G.stream_hi = a.stream_hi;
    G.gather = a.gather != 0;
    G.write_back = a.gather || a.theta > 0;
    G.err = &a.st->err;
    G.gave_up = nullptr;
#if PA_CHECKED
    G.src_limit = a.st->pop;  // the old population (received runs on a shard) until k_finalize
    G.give_up = a.give_up == first + 1;
#endif
    return G;
}

// Group of a ticket, when groups are handed out from a counter: whole groups
// of rpb replicas, and in launches of more than three rounds the last half
// round's worth in halves (whole passes each).  With whole groups to the end a
// block that took its last one late held the launch up by half a round: 2043 or
// 2178 us from step to step at q = 10, L = 64, R = 1e5 (6.86 rounds), 2015 with
// halves.  Returns the first replica (R or more: no group left) and the size.
__device__ __forceinline__ int2 ticket_range(int t, int R, int rpb, int quantum, int blocks)
{
    const long long round = (long long)blocks * rpb;
    const int n1 = R <= 3 * round ? INT_MAX / rpb : (int)((R - round / 2) / rpb);
    if (t < n1) return make_int2((int)min((long long)t * rpb, (long long)INT_MAX), rpb);
    const int h = max(quantum, rpb / 2 / quantum * quantum);
    return make_int2((int)min((long long)n1 * rpb + (long long)(t - n1) * h, (long long)INT_MAX), h);
}

// Persistent blocks over groups of at most rpb replicas of the current
// population (R_i is known only on the device).  With a.dynamic the blocks take
// groups from a counter (for launches of a few groups per block: 1915 against
// 1845 attempts/ns at q = 10, L = 64, R = 1e5); else each block takes an equal
// share, counted in quanta of blockDim / (site words per colour) replicas, the
// number that fills one pass of the block's threads over the site words, so
// that no block and no pass is left part-empty.
// B: bits per state; MODE: 0 for L = 64, 1 for L a multiple of 64, 3 for
// L = 8, 16, 32 (rows packed several to a word), 4 for L = 48, 80, 96, ...
// (banded 8-column segments), 2 otherwise (rows padded to whole words).
template <int B, int MODE, int Q, bool LAT>
__device__ __forceinline__ void sweep_blocks(const SweepArgs &a)
{
    extern __shared__ uint4 smem4[];
    __shared__ uint4 s_tab[dev::kThresholdEntries];
    constexpr int QCAP = LAT ? dev::kLatQueue : B <= 4 ? 384 : dev::kQueueCap;
    __shared__ __align__(16) uint32_t s_queue[dev::queue_words(B, QCAP)];
    dev::build_threshold_table(s_tab, a.thr);
    wait_prerequisites();
    DevState *st = a.st;
    const int parity = st->parity;
    // thread 0 hands out the groups from shared memory: nothing of it stays in
    // registers through the sweeps
    __shared__ int2 s_group;  // first replica and number of replicas
    __shared__ int s_R, s_next, s_end;
    const int quantum = max(1, min(a.rpb, (int)blockDim.x / colour_words(a.L)));
    if (threadIdx.x == 0) {
        const int R = a.gather ? st->pop_next : st->pop;
        const long long nq = (R + quantum - 1) / quantum;
        s_R = R;
        s_next = (int)(nq * blockIdx.x / gridDim.x) * quantum;
        s_end = min(R, (int)(nq * (blockIdx.x + 1) / gridDim.x) * quantum);
    }
    for (;;) {
        if (threadIdx.x == 0) {
            int2 g;
            if (a.dynamic) {
                g = ticket_range(atomicAdd(a.counters, 1), s_R, a.rpb, quantum, gridDim.x);
                g.y = min(g.y, s_R - g.x);
            } else {
                g = make_int2(s_next, min(a.rpb, s_end - s_next));
                s_next += a.rpb;
            }
            // the run has failed, before this launch or by a block that gave up
            // (PA_ERR_TIMEOUT; this one too): no group, and every block still counts
            // itself below
            if (*(volatile int32_t *)&st->err) g.y = 0;
            s_group = g;
        }
        __syncthreads();
        const int2 g = s_group;  // written again only after the barriers of a group
        if (g.y <= 0) break;
        const dev::Group G = make_group(a, parity, g.x, g.y);
        dev::sweep_group_bits<B, MODE, Q, QCAP, LAT>(G, a.L, reinterpret_cast<uint32_t *>(smem4), s_tab, s_queue,
                                                     a.rk0, a.rk1, a.acc);
    }
    launch_dependents();
    if (threadIdx.x == 0) dev::bulk_stores_done();
    // the last block to end clears the counters for the next launch and writes
    // the step's estimators (a launch of its own took 5.5 us and a gap)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(a.counters + 1, 1) == (int)gridDim.x - 1) {
        __threadfence();
        a.counters[0] = a.counters[1] = 0;
        if (a.obs && !*(volatile int32_t *)&st->err)
            dev::finalize_record(st, a.acc, a.obs, a.beta, a.q, a.L * a.L, a.gather, a.gather, 0, 0.0, 0);
    }
}

template <int B, int MODE, int Q>
__global__ void __launch_bounds__(1024) k_sweep(const SweepArgs a)
{
    sweep_blocks<B, MODE, Q, false>(a);
}

// Kernels for the common q with q fixed at compile time (the reduction mod q
// then uses constant masks), and one kernel per bit count for any other q.
template <int MODE>
SweepFn pick_q(int q)
{
    switch (q) {
    case 2: return k_sweep<state_bits(2), MODE, 2>;
    case 3: return k_sweep<state_bits(3), MODE, 3>;
    case 4: return k_sweep<state_bits(4), MODE, 4>;
    case 5: return k_sweep<state_bits(5), MODE, 5>;
    case 6: return k_sweep<state_bits(6), MODE, 6>;
    case 8: return k_sweep<state_bits(8), MODE, 8>;
    case 10: return k_sweep<state_bits(10), MODE, 10>;
    case 20: return k_sweep<state_bits(20), MODE, 20>;
    }
    switch (state_bits(q)) {
    case 1: return k_sweep<1, MODE, 0>;
    case 2: return k_sweep<2, MODE, 0>;
    case 3: return k_sweep<3, MODE, 0>;
    case 4: return k_sweep<4, MODE, 0>;
    case 5: return k_sweep<5, MODE, 0>;
    case 6: return k_sweep<6, MODE, 0>;
    default: return k_sweep<7, MODE, 0>;
    }
}

}  // namespace

}  // namespace pa
