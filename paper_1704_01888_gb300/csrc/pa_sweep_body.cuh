// pa_sweep_body.cuh -- device body of the Metropolis sweep of population
// annealing (Barash, Weigel, Shchur & Janke, arXiv:1704.01888, Sec. 2 step 3
// and Sec. 3), with the replica gather of step 2 fused into its load and the
// measurements of step 4 (Eq. 3 energy, Eq. 5 largest-state occupation, the
// energy histogram) in its epilogue.  Shared by the single-run sweep kernel
// (pa_sweep.cu) and the batched sweep kernels (pa_batch.cuh).
//
// One block holds a group of whole lattices in shared memory and runs theta
// checkerboard sweeps on them.  Spins are multi-spin coded (layout in
// pa_internal.cuh): every logic instruction of the update acts on the 32 sites
// of one site word.
#pragma once
#include <climits>
#include <type_traits>

#include "pa_internal.cuh"

namespace pa {
namespace dev {

// ===========================================================================
// Bit-plane helpers
// ===========================================================================

// BP consecutive words (the planes of one site word): one 16-byte access per
// four planes (BP = 4: the site word's planes start on a 16-byte boundary),
// 8-byte accesses for BP = 2 and 6, single words for BP = 1, 5 and 7 (a
// warp's loads of one plane then fall in distinct banks: the words of
// consecutive site words lie an odd number of words apart).
template <int BP>
__device__ __forceinline__ void load_planes(uint32_t (&v)[BP], const uint32_t *src)
{
    if constexpr (BP % 4 == 0) {
#pragma unroll
        for (int h = 0; h < BP / 4; ++h) {
            const uint4 a = reinterpret_cast<const uint4 *>(src)[h];
            v[4 * h + 0] = a.x;
            v[4 * h + 1] = a.y;
            v[4 * h + 2] = a.z;
            v[4 * h + 3] = a.w;
        }
    } else if constexpr (BP % 2 == 0) {
#pragma unroll
        for (int h = 0; h < BP / 2; ++h) {
            const uint2 a = reinterpret_cast<const uint2 *>(src)[h];
            v[2 * h + 0] = a.x;
            v[2 * h + 1] = a.y;
        }
    } else {
#pragma unroll
        for (int p = 0; p < BP; ++p) v[p] = src[p];
    }
}

template <int BP>
__device__ __forceinline__ void store_planes(uint32_t *dst, const uint32_t (&v)[BP])
{
    if constexpr (BP % 4 == 0) {
#pragma unroll
        for (int h = 0; h < BP / 4; ++h)
            reinterpret_cast<uint4 *>(dst)[h] = make_uint4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
    } else if constexpr (BP % 2 == 0) {
#pragma unroll
        for (int h = 0; h < BP / 2; ++h) reinterpret_cast<uint2 *>(dst)[h] = make_uint2(v[2 * h], v[2 * h + 1]);
    } else {
#pragma unroll
        for (int p = 0; p < BP; ++p) dst[p] = v[p];
    }
}

// Bit set where the B-bit states held in planes a and b differ.
template <int B, int BP>
__device__ __forceinline__ uint32_t differ(const uint32_t (&a)[BP], const uint32_t (&b)[BP])
{
    uint32_t d = a[0] ^ b[0];
#pragma unroll
    for (int p = 1; p < B; ++p) d |= a[p] ^ b[p];
    return d;
}

// Bit set where the B-bit state in planes a equals the constant state s.
template <int B, int BP>
__device__ __forceinline__ uint32_t equal_state(const uint32_t (&a)[BP], int s)
{
    uint32_t d = 0;
#pragma unroll
    for (int p = 0; p < B; ++p) d |= a[p] ^ (((s >> p) & 1) ? 0xFFFFFFFFu : 0u);
    return ~d;
}

__device__ __forceinline__ void accumulate_totals(unsigned long long *acc, long long sE, long long sE2, long long sM)
{
    atomicAdd(acc + 0, (unsigned long long)sE);
    atomicAdd(acc + 1, (unsigned long long)sE2);
    atomicAdd(acc + 2, (unsigned long long)sM);
}

// Division by a divisor d fixed for a replica group (d < 2^15) of x < 2^16,
// without a division instruction sequence per use: with inv = ceil(2^31 / d)
// = (2^31 + e) / d, 0 <= e < d, floor(x inv / 2^31) = floor(x / d) because
// x e < x d < 2^31.
__device__ __forceinline__ uint32_t div_inverse(uint32_t d) { return (uint32_t)((0x80000000ull + d - 1u) / d); }
__device__ __forceinline__ int div_by(int x, uint32_t inv) { return (int)__umulhi((uint32_t)x << 1, inv); }

__device__ __forceinline__ void full_add(uint32_t a, uint32_t b, uint32_t c, uint32_t &sum, uint32_t &carry)
{
    sum = a ^ b ^ c;
    carry = (a & b) | (c & (a ^ b));
}

// Valid-column mask of word t of a row with WPR words and nb_last valid bits
// in its last word.
__device__ __forceinline__ uint32_t valid_mask(int t, int WPR, int nb_last)
{
    return (t < WPR - 1 || nb_last == 32) ? 0xFFFFFFFFu : ((1u << nb_last) - 1u);
}

// The row word H (other colour, row y) shifted so that bit b holds the
// horizontal neighbour of column 32 t + b that is not at the same column:
// column m + 1 when par = 1, column m - 1 when par = 0 (par = (x & 1) of the
// row's sites).  E is the adjacent word of the row (t + 1 for par = 1, t - 1
// for par = 0, cyclically); MODE 0 is L = 64 (one full word per row), MODE 1
// rows of full words, MODE 2 rows whose last word holds nb_last < 32 columns.
template <int MODE>
__device__ __forceinline__ uint32_t shifted_row(uint32_t H, uint32_t E, int par, int nb, int nbe)
{
    if constexpr (MODE == 0) {
        return __funnelshift_l(H, H, par ? 31 : 1);
    } else if constexpr (MODE == 1) {
        return par ? __funnelshift_r(H, E, 1) : __funnelshift_r(E, H, 31);
    } else {
        // bits past a row's columns are zero in E and not looked at in the result
        return par ? ((H >> 1) | (E << (nb - 1))) : ((H << 1) | (E >> (nbe - 1)));
    }
}

// Packed rows (MODE 3, L = 8, 16, 32): the horizontal neighbour word of H.
// Each word holds 32 / S rows of S = L/2 columns; in a row whose sites sit at
// odd x (par = 1) the neighbour not at the same column is column m + 1, else
// m - 1, both cyclic within the row's S-bit segment.  Rows alternate par, and
// `odd` marks the segments with par = 1 (the same in every word of a colour).
// L = 8 (four-bit rows): masked shifts.
__device__ __forceinline__ uint32_t shifted_nibbles(uint32_t H, uint32_t odd)
{
    constexpr uint32_t bot = 0x11111111u, top = bot << 3;
    const uint32_t right = ((H >> 1) & ~top) | ((H << 3) & top);  // column m + 1
    const uint32_t left = ((H << 1) & ~bot) | ((H >> 3) & bot);   // column m - 1
    return (odd & right) | (~odd & left);
}

// L = 16 and 32 (rows of one or two bytes): the rows that take column m - 1
// are doubled side by side (byte selector l) and shifted left, the others (r)
// doubled and shifted right, so that each row's wrapped bit arrives from its
// copy; `out` picks the rows' bytes: five instructions per plane against
// eight with masks.
struct RowSelectors {
    uint32_t l, r, out;
};
__device__ __forceinline__ RowSelectors row_selectors(int L, int c)
{
    if (L == 32) return c ? RowSelectors{0x3232u, 0x1010u, 0x3254u} : RowSelectors{0x1010u, 0x3232u, 0x5432u};
    return c ? RowSelectors{0x3311u, 0x2200u, 0x3614u} : RowSelectors{0x2200u, 0x3311u, 0x6341u};
}
__device__ __forceinline__ uint32_t shifted_bytes(uint32_t H, const RowSelectors &sel)
{
    const uint32_t l = __byte_perm(H, 0u, sel.l) << 1, r = __byte_perm(H, 0u, sel.r) >> 1;
    return __byte_perm(l, r, sel.out);
}

// The four neighbour words of site word `it` (its index within its colour) of
// colour c: up, down and same-row words of the other colour (oth) and the
// same-row word shifted by one column.  Returns the mask of the word's valid
// columns.  MODE as for shifted_row, 3 for packed rows, 4 for banded rows;
// inv_row = div_inverse of the words per row (MODE 1, 2) or of the segments
// per row (MODE 4).
template <int B, int MODE, int BP>
__device__ __forceinline__ uint32_t neighbour_planes(const uint32_t *oth, int L, int IPC, int WPR, int nb_last,
                                                     uint32_t inv_row, int it, int c, uint32_t (&U)[BP],
                                                     uint32_t (&D)[BP], uint32_t (&H)[BP], uint32_t (&X)[BP])
{
    if constexpr (MODE == 4) {
        // word (k, j): segment j of rows k + a L/4 in byte a.  The rows above
        // and below are the same bytes of words (k -+ 1, j), except across the
        // band edges: above row 0 of a band lies the last row of the band
        // before (byte a - 1 of word (L/4 - 1, j), cyclically), below its last
        // row the first row of the next band (byte a + 1 of word (0, j)).
        const int segs = L >> 4, band_rows = L >> 2;
        const int k = div_by(it, inv_row), j = it - k * segs;
        const int ku = k == 0 ? band_rows - 1 : k - 1;
        const int kd = k == band_rows - 1 ? 0 : k + 1;
        const int par = (k + c) & 1;  // band heights are even: one parity per word
        const int je = par ? (j + 1 == segs ? 0 : j + 1) : (j == 0 ? segs - 1 : j - 1);
        uint32_t Uw[BP], Dw[BP], Eg[BP];
        load_planes<BP>(H, oth + it * BP);
        load_planes<BP>(Uw, oth + (ku * segs + j) * BP);
        load_planes<BP>(Dw, oth + (kd * segs + j) * BP);
        load_planes<BP>(Eg, oth + (k * segs + je) * BP);
        const uint32_t ru = k == 0 ? 8u : 0u, rd = k == band_rows - 1 ? 8u : 0u;
#pragma unroll
        for (int p = 0; p < B; ++p) {
            U[p] = __funnelshift_l(Uw[p], Uw[p], ru);
            D[p] = __funnelshift_r(Dw[p], Dw[p], rd);
            // column m + 1 (par = 1) or m - 1 (par = 0) within each 8-column
            // byte, the edge column from the adjacent segment Eg
            X[p] = par ? (((H[p] >> 1) & 0x7F7F7F7Fu) | ((Eg[p] << 7) & 0x80808080u))
                       : (((H[p] << 1) & 0xFEFEFEFEu) | ((Eg[p] >> 7) & 0x01010101u));
        }
        return 0xFFFFFFFFu;
    } else if constexpr (MODE == 3) {
        const int wu = it == 0 ? IPC - 1 : it - 1;
        const int wd = it == IPC - 1 ? 0 : it + 1;
        uint32_t Hu[BP], Hd[BP];
        load_planes<BP>(H, oth + it * BP);
        load_planes<BP>(Hu, oth + wu * BP);
        load_planes<BP>(Hd, oth + wd * BP);
        const int S = L >> 1;
#pragma unroll
        for (int p = 0; p < B; ++p) {
            U[p] = __funnelshift_l(Hu[p], H[p], S);
            D[p] = __funnelshift_r(H[p], Hd[p], S);
        }
        if (L == 8) {
            const uint32_t seg = c ? 0x0F0F0F0Fu : 0xF0F0F0F0u;
#pragma unroll
            for (int p = 0; p < B; ++p) X[p] = shifted_nibbles(H[p], seg);
        } else {
            const RowSelectors sel = row_selectors(L, c);
#pragma unroll
            for (int p = 0; p < B; ++p) X[p] = shifted_bytes(H[p], sel);
        }
        return 0xFFFFFFFFu;
    } else {
        const int y = MODE == 0 ? it : div_by(it, inv_row);
        const int t = MODE == 0 ? 0 : it - y * WPR;
        const int yu = (y == 0) ? L - 1 : y - 1;
        const int yd = (y == L - 1) ? 0 : y + 1;
        const int par = (y + c) & 1;
        load_planes<BP>(U, oth + (yu * WPR + t) * BP);
        load_planes<BP>(D, oth + (yd * WPR + t) * BP);
        load_planes<BP>(H, oth + (y * WPR + t) * BP);
        if constexpr (MODE == 0) {
#pragma unroll
            for (int p = 0; p < B; ++p) X[p] = shifted_row<0>(H[p], 0u, par, 32, 32);
            return 0xFFFFFFFFu;
        } else {
            const int te = par ? (t + 1 == WPR ? 0 : t + 1) : (t == 0 ? WPR - 1 : t - 1);
            uint32_t Eg[BP];
            load_planes<BP>(Eg, oth + (y * WPR + te) * BP);
            const int nb = t == WPR - 1 ? nb_last : 32;
            const int nbe = te == WPR - 1 ? nb_last : 32;
#pragma unroll
            for (int p = 0; p < B; ++p) X[p] = shifted_row<MODE>(H[p], Eg[p], par, nb, nbe);
            return valid_mask(t, WPR, nb_last);
        }
    }
}

// ===========================================================================
// One group of resident replicas
// ===========================================================================
struct Group {
    const uint32_t *in;      // buffer holding the parents (or the replicas themselves)
    uint32_t *out;           // buffer receiving the swept replicas
    const int32_t *parent;   // parent map of a pending resample (used when gather)
    const int32_t *anc_in;   // family ids (null: no families)
    int32_t *anc_out;
    int32_t *fam;            // family counts (null: no families)
    int32_t *E, *Mt, *hist;  // per-replica energies and occupations, energy histogram
    int first, nrep;         // slots [first, first + nrep): global slots (random keys); the
                             // arrays above are indexed by them
    int q, theta, step;
    uint32_t stream_hi;      // stream number << 24, or'ed into the slot counter word
    bool gather, write_back;
    int32_t *err;            // the run's error flag
    int *gave_up;            // shared, set where the block may take no further group (null: it reads err)
#if PA_CHECKED
    int src_limit;           // a gather's parent slots lie in [0, src_limit)
    bool give_up;            // a test: count the wait for the bulk copies as run out
#endif
};

// ---- Bulk copies of whole replicas (cp.async.bulk: 16-byte aligned, sizes
// multiples of 16 bytes, as replicas are) -----------------------------------
__device__ __forceinline__ uint32_t shared_address(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Orders this thread's accesses to shared memory before bulk copies that touch
// the same bytes after the next barrier.
__device__ __forceinline__ void fence_bulk() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void bulk_barrier_init(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(bar)
                 : "memory");
}

// Waits for the barrier's bytes, at most about a second (kBulkClocks); false if
// they did not come.  Whoever gives up takes no further group: the barrier and
// the shared memory may still be written by the copies that are late.
constexpr long long kBulkClocks = 2000000000ll;
__device__ __forceinline__ bool bulk_wait(uint32_t bar)
{
    const long long start = clock64();
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar)
            : "memory");
        if (done) return true;
        if (clock64() - start > kBulkClocks) return false;
    }
}

__device__ __forceinline__ void bulk_store(void *dst, uint32_t src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(__cvta_generic_to_global(dst)),
                 "r"(src), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// The issuing thread: until its bulk stores have read shared memory / are done.
__device__ __forceinline__ void bulk_stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_stores_done() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Smallest replica that a gather copies in bulk, one copy each; smaller ones
// are gathered by the threads.
constexpr uint32_t kBulkReplica = 512;

__device__ __forceinline__ void record_replica(const Group &G, int slot, int E, int Mt, int N, long long &sE,
                                               long long &sE2, long long &sM)
{
    G.E[slot] = E;
    G.Mt[slot] = Mt;
#if PA_CHECKED
    if (E < -2 * N || E > 0) {
        atomicExch(G.err, 1);  // PA_ERR_INVALID
        return;
    }
#endif
    atomicAdd(G.hist + (E + 2 * N), 1);
    sE += E;
    sE2 += (long long)E * (long long)E;
    sM += Mt;
}

__device__ __forceinline__ void group_families(const Group &G)
{
    if (!G.fam) return;
    for (int r = threadIdx.x; r < G.nrep; r += blockDim.x) {
        const int slot = G.first + r;
        const int f = G.anc_in[G.gather ? G.parent[slot] : slot];
        if (G.gather) G.anc_out[slot] = f;
        atomicAdd(G.fam + f, 1);
    }
}

// Shared-memory table of the acceptance thresholds for the bitwise
// comparison v < T[dE]: entry j (0..31) holds, for d = 1..4, all ones where
// bit 31 - j of T[d] is set; entries 32..39 are zero (planes past the last bit
// of v, which the loop may draw when it takes acceptance words four at a time:
// a zero threshold bit never accepts); entry 40 marks T[d] = 2^32.  The
// block's threads share the 41 entries (blocks may have as few as 32 threads).
constexpr int kThresholdEntries = 41;
constexpr int kThresholdFull = 40;

// Two-pass acceptance.  In the first pass every site word draws exactly
// kFirstPassCalls Philox calls of acceptance words; a word with sites still
// undecided after that (about 8 % of words at low temperature) goes to a
// block-wide queue, and in the second pass whole warps serve only queued
// words, so a warp does not wait for the slowest of its ~700 sites.  (No vote
// before the first-pass calls: a call is skipped only if all 1024 sites of a
// warp are decided, which half of the open sites per plane all but rules
// out.)  The word itself is written with its decided sites in the first
// pass; the queue entry keeps what the second pass needs for the others:
// {word index, undecided, class bits c0, e1, B proposal planes}, padded to
// whole 16-byte vectors, after two counters.  A full queue is not an error:
// the word's own thread finishes it.  The single-run kernel with up to four
// planes takes 384 entries (its 48 lattices give up to ~250 queued words at
// low temperature, so 256 entries overflowed: 1846 against 1837 attempts/ns
// over the at-scale schedule; two blocks per SM still fit); the batched kernel
// keeps 256: more gave 3104 against 3124 PA steps/s in blocks of 96 KB of
// lattices, and its default blocks hold a third of those.
constexpr int kFirstPassCalls = 2;
constexpr int kLatCalls = 3;
constexpr int kLatQueue = 90;
constexpr int kQueueCap = 256;
__host__ __device__ constexpr int queue_entry_words(int B) { return (4 + B + 3) & ~3; }
__host__ __device__ constexpr int queue_words(int B, int cap = kQueueCap) { return 4 + queue_entry_words(B) * cap; }
// Entry j holds, for the threshold bits t_1..t_4 of plane j (bit 31 - j of
// T[1..4]), the coefficients of two multiply-adds: c0 * (t_1 - t_2) - t_2
// gives the threshold bits of the dE = 1, 2 sites (c0: dE odd) and
// c0 * (t_3 - t_4) - t_4 those of the dE = 3, 4 sites, bit for bit: the four
// results 0, c0, ~c0 = -c0 - 1 and ~0 are the four two-way selections.  The
// selections thus run on the multiply-add pipe; only the choice by e1 is a
// logic operation.
__device__ __forceinline__ void build_threshold_table(uint4 *tab, const Thresholds &th)
{
    auto coef = [](uint32_t ta, uint32_t tb) { return make_uint2(ta - tb, 0u - tb); };
    for (int j = threadIdx.x; j < kThresholdEntries; j += blockDim.x) {
        uint32_t t[4] = {0u, 0u, 0u, 0u};
        if (j < 32) {
            for (int d = 0; d < 4; ++d) t[d] = (th.T[d] >> (31 - j)) & 1u;
        } else if (j == kThresholdFull) {
            for (int d = 0; d < 4; ++d) t[d] = (th.full >> d) & 1u;
        }
        const uint2 lo = coef(t[0], t[1]), hi = coef(t[2], t[3]);
        tab[j] = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
}

// Threshold bit of plane entry tb for each site: the site's dE class is
// given by c0 (dE odd) and e1 (dE >= 3).
__device__ __forceinline__ uint32_t threshold_bits(const uint4 &tb, uint32_t c0, uint32_t e1)
{
    const uint32_t lo = c0 * tb.x + tb.y;  // dE = 1 where c0, dE = 2 elsewhere
    const uint32_t hi = c0 * tb.z + tb.w;  // dE = 3 where c0, dE = 4 elsewhere
    return (e1 & hi) | (~e1 & lo);
}

// One bit plane j of the acceptance numbers v (bits of the word v_bits).  A
// site still undecided takes T's bit into acc -- the outcome of v < T if v's
// bit differs from it -- and stays undecided where the two bits agree.  So
// once the planes are done a site is accepted where acc is set and und is
// clear (a site whose v equals T in every plane is rejected).
__device__ __forceinline__ void acceptance_plane(uint32_t v_bits, int j, const uint4 *s_tab, uint32_t c0, uint32_t e1,
                                                 uint32_t &acc, uint32_t &und)
{
    const uint32_t tj = threshold_bits(s_tab[j], c0, e1);
    acc = (und & tj) | (~und & acc);
    und &= ~(v_bits ^ tj);
}

// ---- Philox calls of the sweep, the first rounds shared ------------------
// The sweep's counters (w, ctr, step, slot) differ between the calls of a word
// only in ctr (sweep, colour, call number), between the replicas only in
// slot.  Followed through the rounds: round 0's products depend on w and on
// step, round 1's on ctr and on (w, slot), round 2's on (w, slot) and on
// (w, ctr).  So of a call's twenty products only the fourteen of rounds 3..9
// belong to the call alone; two are made once per word (PhiloxWord) and one
// once per word index and counter (PhiloxCtr), which a thread that keeps one
// word index through its replicas makes once per half sweep.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;

struct PhiloxWord {
    uint32_t y, z, w;  // state words after round 2, less the parts that follow ctr (z: without w2)
};
struct PhiloxCtr {
    uint32_t x, y, w2;  // x: without PhiloxWord::y
};

__device__ __forceinline__ PhiloxWord philox_word(uint32_t w, uint32_t step, uint32_t slot, const uint32_t *rk0,
                                                  const uint32_t *rk1)
{
    const uint32_t z1 = __umulhi(kPhiloxM0, w) ^ slot ^ rk1[0];
    const uint64_t p1 = (uint64_t)kPhiloxM1 * z1;
    const uint32_t x2 = (uint32_t)(p1 >> 32) ^ (kPhiloxM1 * step) ^ rk0[1];
    const uint64_t p0 = (uint64_t)kPhiloxM0 * x2;
    return {(uint32_t)p1, (uint32_t)(p0 >> 32) ^ rk1[2], (uint32_t)p0};
}

__device__ __forceinline__ PhiloxCtr philox_ctr(uint32_t w, uint32_t ctr, uint32_t step, const uint32_t *rk0,
                                                const uint32_t *rk1)
{
    const uint32_t x1 = __umulhi(kPhiloxM1, step) ^ ctr ^ rk0[0];
    const uint64_t p0 = (uint64_t)kPhiloxM0 * x1;
    const uint32_t z2 = (uint32_t)(p0 >> 32) ^ (kPhiloxM0 * w) ^ rk1[1];
    const uint64_t p1 = (uint64_t)kPhiloxM1 * z2;
    return {(uint32_t)(p1 >> 32) ^ rk0[2], (uint32_t)p1, (uint32_t)p0};
}

// The call's four words: philox10_rk of (w, ctr, step, slot).
__device__ __forceinline__ uint4 philox_finish(const PhiloxWord &a, const PhiloxCtr &b, const uint32_t *rk0,
                                               const uint32_t *rk1)
{
    uint4 c = make_uint4(b.x ^ a.y, b.y, a.z ^ b.w2, a.w);
#pragma unroll
    for (int round = 3; round < 10; ++round) {
        const uint64_t p0 = (uint64_t)kPhiloxM0 * c.x;
        const uint64_t p1 = (uint64_t)kPhiloxM1 * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ rk0[round], (uint32_t)p1,
                       (uint32_t)(p0 >> 32) ^ c.w ^ rk1[round], (uint32_t)p0);
    }
    return c;
}

// The four acceptance planes of Philox call n of a site word's stream (words
// 4n .. 4n + 3, i.e. planes j = 4n - B ..).
template <int B>
__device__ __forceinline__ void acceptance_call(const uint4 &z, int n, const uint4 *s_tab, uint32_t c0, uint32_t e1,
                                                uint32_t &acc, uint32_t &und)
{
    const int j0 = 4 * n - B;
    acceptance_plane(z.x, j0, s_tab, c0, e1, acc, und);
    acceptance_plane(z.y, j0 + 1, s_tab, c0, e1, acc, und);
    acceptance_plane(z.z, j0 + 2, s_tab, c0, e1, acc, und);
    acceptance_plane(z.w, j0 + 3, s_tab, c0, e1, acc, und);
}

// Acceptance words of Philox calls n = ch_begin .. ch_end - 1 of a site word's
// stream, drawn while a site is undecided: in the whole warp (WARP_VOTE, all
// lanes must take part) or in this thread's word alone.
template <int B, bool WARP_VOTE>
__device__ __forceinline__ void acceptance_calls(int ch_begin, int ch_end, const PhiloxWord &pw, uint32_t w,
                                                 uint32_t ctr1, uint32_t step, const uint32_t *rk0,
                                                 const uint32_t *rk1, const uint4 *s_tab, uint32_t c0, uint32_t e1,
                                                 uint32_t &acc, uint32_t &und)
{
#pragma unroll 1
    for (int ch = ch_begin; ch < ch_end; ++ch) {
        if (WARP_VOTE ? !__any_sync(0xFFFFFFFFu, und) : !und) break;
        const uint4 z = philox_finish(pw, philox_ctr(w, ctr1 | (uint32_t)ch, step, rk0, rk1), rk0, rk1);
        acceptance_call<B>(z, ch, s_tab, c0, e1, acc, und);
    }
}

// Proposal planes P = (s + t) mod q of the states in planes W, with t = 1 + u
// for direction sigma = 0 and q - (1 + u) for sigma = 1 (planes sg, u_p =
// Z[p + 1], p < B - 1): t = (u ^ sigma) + (q - 1 where sigma) + 1 over B planes,
// S = s + t, q taken off where S >= q (compared from the lowest plane up).
// qb / q1b: the bits of q and q - 1 as plane masks.  With q fixed at compile
// time the masks fold into the three-input logic: 21 operations for q = 10
// against 28 for s +- (1 + u) with a conditional q added or taken off.
template <int B, int BP>
__device__ __forceinline__ void propose(const uint32_t (&W)[BP], const uint32_t *Z, const uint32_t (&qb)[B + 1],
                                        const uint32_t (&q1b)[B + 1], uint32_t (&P)[BP])
{
    const uint32_t sg = Z[0];
    uint32_t S[B + 1];
    uint32_t ct = 0xFFFFFFFFu, cs = 0u;
#pragma unroll
    for (int p = 0; p < B; ++p) {
        const uint32_t y = p < B - 1 ? (Z[p + 1] ^ sg) : sg;
        const uint32_t k = sg & q1b[p];
        uint32_t t;
        full_add(y, k, ct, t, ct);
        full_add(W[p], t, cs, S[p], cs);
    }
    S[B] = cs;
    uint32_t ge = 0xFFFFFFFFu;
#pragma unroll
    for (int p = 0; p <= B; ++p) ge = (S[p] & ~qb[p]) | (~(S[p] ^ qb[p]) & ge);
    uint32_t bw = 0u;
#pragma unroll
    for (int p = 0; p < BP; ++p) {
        if (p < B) {
            const uint32_t d = ge & qb[p];
            P[p] = S[p] ^ d ^ bw;
            bw = (~S[p] & (d | bw)) | (d & bw);
        } else {
            P[p] = 0u;
        }
    }
}

// Multi-spin-coded sweep body.  B = bits per state (compile time), MODE as
// for neighbour_planes, Q = q when fixed at compile time (0: q from G).  Each
// loop step of a thread updates one site word: 32 same-colour sites.  The
// random numbers follow this rule: in sweep k, colour c, the site word with
// index w = y WPR + t draws the stream Z_0, Z_1, ... (Z_{4n+i} = word i of the
// Philox call with counter
// (w, SWEEP | (2k + c) << 8 | n, step, slot | stream)); the site at bit b takes
// bit b of each: direction sigma from Z_0, offset u from Z_1..Z_{B-1}, and
// acceptance bits v_j from Z_{B+j}, most significant first.  Proposal
// s' = s + (1 + u) mod q (sigma = 0) or s - (1 + u) mod q (sigma = 1) by
// ripple-carry additions over the planes; dE + 4 is the count of eight
// indicator bits (neighbours equal to s, neighbours different from s'), summed
// by a carry-save tree; moves with dE > 0 compare v with T[dE] bit by bit.
//
// Bound by the ALU pipe (half a warp instruction per clock and scheduler; 65 %
// busy at q = 10, L = 64, R = 65536) and beside it the FMA-heavy one (a quarter),
// which takes the Philox products.  What is made once per word, per word index
// or per half sweep is therefore kept out of the 362 instructions per word (409
// before the shared Philox rounds, the shorter proposal and the smaller queue
// entries).  Launches of theta = 10 next to beta_t, with 409 instructions and the
// launch shapes of then against now: 2138 -> 1979 us at q = 10, L = 64, R = 1e5;
// 9721 -> 8097 at q = 20, L = 256, R = 2e4; 4359 -> 3820 at q = 8, L = 128, R = 5e4; 743
// -> 525 at q = 6, L = 32, R = 1e5; 774 -> 595 at q = 8, L = 48, R = 5e4; 3782 -> 3041
// at q = 3, L = 100, R = 5e4.
//
// Where the copies into shared memory do not come, G.err becomes PA_ERR_TIMEOUT
// and the block must leave its loop over the groups.
template <int B, int MODE, int Q = 0, int QCAP = kQueueCap, bool LAT = false>
__device__ __forceinline__ void sweep_group_bits(const Group &G, int Lrt, uint32_t *sw, const uint4 *s_tab,
                                                 uint32_t *qbuf, const uint32_t *rk0, const uint32_t *rk1,
                                                 unsigned long long *totals)
{
    constexpr int BP = plane_stride(B);
    // the measurement's per-replica counts reuse the queue (at most 16 replicas x (q + 1))
    static_assert((LAT ? 8 : 16) * ((1 << B) + 1) <= queue_words(B, QCAP), "queue too small for the counts");
    const int L = MODE == 0 ? 64 : Lrt;
    const int N = L * L;
    const int WPR = MODE == 0 ? 1 : row_words(L);
    const int nb_last = L / 2 - 32 * (WPR - 1);
    const int IPC = colour_words(L);  // site words per colour per replica
    const int RW = replica_words_of(B, L);  // words per replica
    const int UPR = RW / 4;       // uint4 per replica
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;
    const int q = Q > 0 ? Q : G.q;  // Q > 0: q fixed at compile time, the mod-q masks fold
    const int first = G.first, nrep = G.nrep;
    uint4 *smem4 = reinterpret_cast<uint4 *>(sw);

    // Load: replica first + r comes from its parent's lattice.  All copies of
    // the group are in flight at once; a loop of dependent loads (parent, then
    // lattice) per 16 bytes took about 15 us per group of 48 lattices of 2 KB.
    __shared__ __align__(8) unsigned long long s_bar;
    const uint32_t bar = shared_address(&s_bar), RB = (uint32_t)RW * 4u;
    auto source = [&](int r) {
        const int slot = first + r;
        int src = G.gather ? G.parent[slot] : slot;
#if PA_CHECKED
        if (G.gather && (src < 0 || src >= G.src_limit)) {
            atomicExch(G.err, 1);  // PA_ERR_INVALID
            src = 0;
        }
#endif
        return G.in + (size_t)src * RW;
    };
    // (the latency kernel's few pieces per thread are quicker by hand)
    const bool bulk = !LAT && (!G.gather || RB >= kBulkReplica);
    if (bulk) {
        if (tid == 0) bulk_barrier_init(bar, RB * (uint32_t)nrep);
        __syncthreads();
        if (!G.gather) {
            if (tid == 0) bulk_load(shared_address(sw), source(0), RB * (uint32_t)nrep, bar);
        } else {
            for (int r = tid; r < nrep; r += blockDim.x) bulk_load(shared_address(sw + r * RW), source(r), RB, bar);
        }
        bool here = bulk_wait(bar);
#if PA_CHECKED
        here = here && !G.give_up;
#endif
        if (__syncthreads_or(!here)) {
            // not expected to happen: report it, give the copies once more the
            // time to land, and leave the group
            if (tid == 0) {
                atomicExch(G.err, 4);  // PA_ERR_TIMEOUT
                if (G.gave_up) *G.gave_up = 1;
                bulk_wait(bar);
            }
            __syncthreads();
            return;
        }
        if (tid == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
    } else {
        constexpr int U4 = 4;  // 16-byte pieces in flight per thread
        const uint32_t inv_upr = div_inverse(UPR);
        const int pieces = nrep * UPR, step = (int)blockDim.x;
        for (int i0 = tid; i0 < pieces; i0 += U4 * step) {
            uint4 v[U4];
#pragma unroll
            for (int u = 0; u < U4; ++u) {
                const int i = min(i0 + u * step, pieces - 1), r = div_by(i, inv_upr);
                v[u] = reinterpret_cast<const uint4 *>(source(r))[i - r * UPR];
            }
#pragma unroll
            for (int u = 0; u < U4; ++u)
                if (i0 + u * step < pieces) smem4[i0 + u * step] = v[u];
        }
        __syncthreads();
    }

    // q and q - 1 as plane masks, for the proposal
    uint32_t qm[B + 1], q1m[B + 1];
#pragma unroll
    for (int p = 0; p <= B; ++p) {
        qm[p] = ((q >> p) & 1) ? 0xFFFFFFFFu : 0u;
        q1m[p] = (((q - 1) >> p) & 1) ? 0xFFFFFFFFu : 0u;
    }
    const bool any_full = s_tab[kThresholdFull].x | s_tab[kThresholdFull].y | s_tab[kThresholdFull].z |
                          s_tab[kThresholdFull].w;

    // site words still undecided after the first pass wait in qbuf for the second
    constexpr int EW = queue_entry_words(B) / 4;  // 16-byte vectors per entry
    int *q_count = reinterpret_cast<int *>(qbuf);
    uint4 *q_entry = reinterpret_cast<uint4 *>(qbuf + 4);
    if (tid < 2) q_count[tid] = 0;
    __syncthreads();
    int half = 0;
    // A thread keeps one site word index through its replicas (several in turn
    // where a colour has more words than the block threads), so that its row,
    // neighbour offsets, counter word and the Philox products that follow them
    // are made once per half sweep.  Threads beyond the last whole replica's
    // words idle; the launch shapes keep them few.
    const int threads = (int)blockDim.x;
    const bool wide = IPC > threads;
    const int per_pass = wide ? 1 : threads / IPC;
    const int r_first = wide ? 0 : tid / IPC;
    const int it_first = r_first < per_pass ? tid - r_first * IPC : IPC;
    const int it_step = wide ? threads : IPC;
    // replica of a block-wide word index, and row (segment row) of a word
    const uint32_t inv_ipc = div_inverse(IPC);
    const uint32_t inv_row = div_inverse(MODE == 4 ? L >> 4 : WPR);
    auto replica_of = [&](int x) { return MODE == 0 ? x / IPC : div_by(x, inv_ipc); };

    for (int k = 0; k < G.theta; ++k) {
        for (int c = 0; c < 2; ++c, ++half) {
            const uint32_t ctr1 = DOM_SWEEP | ((uint32_t)(2 * k + c) << 8);
            if (tid == 0) q_count[(half + 1) & 1] = 0;
            int *qc = q_count + (half & 1);
            constexpr int fc = (B + 3) / 4;  // proposal calls; acceptance calls follow
            constexpr int kCalls = fc + (LAT ? kLatCalls : kFirstPassCalls);
            // one site word: replica r, word it within the colour (its counter
            // word w); pc: the calls' shared Philox products
            auto site_word = [&](const int r, const int it, const PhiloxCtr (&pc)[kCalls]) {
                const int ii = r * IPC + it;
                uint32_t *rep = sw + r * RW;
                uint32_t *own = rep + (c * IPC + it) * BP;
                const uint32_t *oth = rep + (c ^ 1) * IPC * BP;
                uint32_t W[BP], U[BP], D[BP], H[BP], X[BP];
                load_planes<BP>(W, own);
                const uint32_t vmask =
                    neighbour_planes<B, MODE, BP>(oth, L, IPC, WPR, nb_last, inv_row, it, c, U, D, H, X);

                const uint32_t slot = (uint32_t)(first + r) | G.stream_hi;
                const uint32_t w = (uint32_t)it;
                const PhiloxWord pw = philox_word(w, (uint32_t)G.step, slot, rk0, rk1);
                auto call = [&](int n) { return philox_finish(pw, pc[n], rk0, rk1); };
                // proposal: direction sigma = Z_0, offset bits u = Z_1..Z_{B-1}
                uint32_t Z[4 * fc];
#pragma unroll
                for (int n = 0; n < fc; ++n) {
                    const uint4 z = call(n);
                    Z[4 * n + 0] = z.x;
                    Z[4 * n + 1] = z.y;
                    Z[4 * n + 2] = z.z;
                    Z[4 * n + 3] = z.w;
                }
                uint32_t P[BP];
                propose<B, BP>(W, Z, qm, q1m, P);

                // dE + 4 = #(neighbours equal to s) + #(neighbours different from s')
                const uint32_t a1 = ~differ<B, BP>(W, U), a2 = ~differ<B, BP>(W, D);
                const uint32_t a3 = ~differ<B, BP>(W, H), a4 = ~differ<B, BP>(W, X);
                const uint32_t b1 = differ<B, BP>(P, U), b2 = differ<B, BP>(P, D);
                const uint32_t b3 = differ<B, BP>(P, H), b4 = differ<B, BP>(P, X);
                uint32_t s1, k1, s2, k2, s3, k3, s5, k5;
                full_add(a1, a2, a3, s1, k1);
                full_add(a4, b1, b2, s2, k2);
                full_add(b3, b4, s1, s3, k3);
                const uint32_t c0 = s2 ^ s3, k4 = s2 & s3;
                full_add(k1, k2, k3, s5, k5);
                const uint32_t c1 = s5 ^ k4, k6 = s5 & k4;
                const uint32_t c2 = k5 ^ k6, c3 = k5 & k6;
                const uint32_t pos = vmask & (c3 | (c2 & (c1 | c0)));  // dE > 0
                const uint32_t e1 = c3 | (c1 & c0);                     // dE >= 3

                // acceptance: dE <= 0 always; otherwise v < T[dE], bit by bit
                uint32_t acc = vmask & ~pos;
                uint32_t und = pos;
                if (any_full) {
                    const uint32_t tj = threshold_bits(s_tab[kThresholdFull], c0, e1);
                    acc |= und & tj;
                    und &= ~tj;
                }
                // acceptance bit j is word B + j: the rest of the last proposal call first
#pragma unroll
                for (int wi = B; wi < 4 * fc; ++wi) acceptance_plane(Z[wi], wi - B, s_tab, c0, e1, acc, und);
#pragma unroll
                for (int n = fc; n < kCalls; ++n) acceptance_call<B>(call(n), n, s_tab, c0, e1, acc, und);
                if constexpr (LAT) {
                    acceptance_calls<B, false>(kCalls, fc + 8, pw, w, ctr1, (uint32_t)G.step, rk0, rk1, s_tab, c0, e1,
                                               acc, und);
                } else
                if (und) {
                    const int e = atomicAdd(qc, 1);
                    if (e < QCAP) {
                        uint4 *dst = q_entry + e * EW;
                        dst[0] = make_uint4((uint32_t)ii, und, c0, e1);
                        uint32_t pv[4 * (EW - 1)];
#pragma unroll
                        for (int p = 0; p < 4 * (EW - 1); ++p) pv[p] = p < B ? P[p < BP ? p : 0] : 0u;
#pragma unroll
                        for (int h = 0; h < EW - 1; ++h)
                            dst[1 + h] = make_uint4(pv[4 * h], pv[4 * h + 1], pv[4 * h + 2], pv[4 * h + 3]);
                    } else {
                        // queue full: this thread finishes its word alone (no warp votes)
                        acceptance_calls<B, false>(kCalls, fc + 8, pw, w, ctr1, (uint32_t)G.step, rk0, rk1, s_tab, c0,
                                                   e1, acc, und);
                    }
                }
                const uint32_t a = acc & ~und;
#pragma unroll
                for (int p = 0; p < B; ++p) W[p] = (a & P[p]) | (~a & W[p]);
                store_planes<BP>(own, W);
            };
            for (int it = it_first; it < IPC; it += it_step) {
                PhiloxCtr pc[kCalls];
#pragma unroll
                for (int n = 0; n < kCalls; ++n)
                    pc[n] = philox_ctr((uint32_t)it, ctr1 | (uint32_t)n, (uint32_t)G.step, rk0, rk1);
                for (int r = r_first; r < nrep; r += per_pass) {
                    // keeps the row and neighbour arithmetic in the loop: carried
                    // through it, its registers spill at 64 per thread
                    int iw = it;
                    asm volatile("" : "+r"(iw));
                    site_word(r, iw, pc);
                }
            }
            __syncthreads();
            if constexpr (LAT) continue;
            // second pass: the queued site words, 32 to a warp
            const int nq = min(*qc, QCAP);
            for (int base = warp * 32; base < nq; base += nwarps * 32) {
                const int e = base + lane;
                const bool live = e < nq;
                const int ee = live ? e : nq - 1;
                const uint4 head = q_entry[ee * EW];
                const int ii = (int)head.x;
                const int r = replica_of(ii);
                const int it = ii - r * IPC;
                uint32_t acc = 0u;
                uint32_t und = live ? head.y : 0u;
                const uint32_t c0 = head.z, e1 = head.w;
                const uint32_t slot = (uint32_t)(first + r) | G.stream_hi;
                const uint32_t w = (uint32_t)it;
                const PhiloxWord pw = philox_word(w, (uint32_t)G.step, slot, rk0, rk1);
                acceptance_calls<B, true>(kCalls, fc + 8, pw, w, ctr1, (uint32_t)G.step, rk0, rk1, s_tab, c0, e1, acc,
                                          und);
                if (live) {
                    uint32_t *own = sw + r * RW + (c * IPC + it) * BP;
                    uint32_t W[BP], pv[4 * (EW - 1)];
                    load_planes<BP>(W, own);
#pragma unroll
                    for (int h = 0; h < EW - 1; ++h) {
                        const uint4 a = q_entry[ee * EW + 1 + h];
                        pv[4 * h + 0] = a.x;
                        pv[4 * h + 1] = a.y;
                        pv[4 * h + 2] = a.z;
                        pv[4 * h + 3] = a.w;
                    }
                    const uint32_t a = acc & ~und;
#pragma unroll
                    for (int p = 0; p < B; ++p) W[p] = (a & pv[p]) | (~a & W[p]);
                    store_planes<BP>(own, W);
                }
            }
            __syncthreads();
        }
    }

    // Write back: the group's replicas lie one after the other on both sides, one
    // bulk copy that runs beside the measurements (which only read)
    if (G.write_back && LAT) {
        uint4 *out4 = reinterpret_cast<uint4 *>(G.out + (size_t)first * RW);
        for (int i = tid; i < nrep * UPR; i += blockDim.x) out4[i] = smem4[i];
    } else if (G.write_back) {
        fence_bulk();
        __syncthreads();
        if (tid == 0) bulk_store(G.out + (size_t)first * RW, shared_address(sw), RB * (uint32_t)nrep);
    }

    // sums of the replicas this warp records (lane 0), added up per group: kept
    // over the groups they would take six registers through the sweeps
    long long sE = 0, sE2 = 0, sM = 0;
    // Measurements.  A warp's lanes count their words' agreeing neighbours and
    // states; a chunk of states is counted per reading of the words and its
    // warp sums follow one another (one state per reading, each waiting for
    // its own sum, took 1.7 us per replica and warp at L = 16).
    auto agreeing = [&](const uint32_t *rep, int me, int stride) {
        int n = 0;
        // each bond has one colour-0 end: count equal neighbours of colour-0 sites
        for (int it = me; it < IPC; it += stride) {
            uint32_t W[BP], U[BP], D[BP], H[BP], X[BP];
            load_planes<BP>(W, rep + it * BP);
            const uint32_t vmask =
                neighbour_planes<B, MODE, BP>(rep + IPC * BP, L, IPC, WPR, nb_last, inv_row, it, 0, U, D, H, X);
            n += __popc(vmask & ~differ<B, BP>(W, U)) + __popc(vmask & ~differ<B, BP>(W, D)) +
                 __popc(vmask & ~differ<B, BP>(W, H)) + __popc(vmask & ~differ<B, BP>(W, X));
        }
        return __reduce_add_sync(0xFFFFFFFFu, n);
    };
    // emit(s, number of sites in state s) for every state, in every lane
    auto count_states = [&](const uint32_t *rep, int me, int stride, auto emit) {
        constexpr int CH = Q == 0 ? 4 : Q % 5 == 0 ? 5 : Q <= 8 ? Q : 8;
#pragma unroll(Q > 0 ? 32 : 1)
        for (int s0 = 0; s0 < q; s0 += CH) {
            int cnt[CH];
#pragma unroll
            for (int i = 0; i < CH; ++i) cnt[i] = 0;
            for (int it = me; it < 2 * IPC; it += stride) {
                uint32_t W[BP];
                load_planes<BP>(W, rep + it * BP);
                const uint32_t vmask = (MODE == 0 || MODE == 3 || MODE == 4)
                                           ? 0xFFFFFFFFu
                                           : valid_mask(it - div_by(it, inv_row) * WPR, WPR, nb_last);
#pragma unroll
                for (int i = 0; i < CH; ++i) cnt[i] += __popc(vmask & equal_state<B, BP>(W, s0 + i));
            }
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                const int c = __reduce_add_sync(0xFFFFFFFFu, cnt[i]);
                if (s0 + i < q) emit(s0 + i, c);
            }
        }
    };
    if (2 * nrep <= nwarps) {
        // fewer replicas than half the warps: several warps share each
        // replica's words and add their counts in shared memory (the queue's,
        // idle now; nrep <= nwarps / 2 replicas x (q + 1) counts fit it)
        int *s_cnt = reinterpret_cast<int *>(qbuf);
        for (int i = tid; i < nrep * (q + 1); i += blockDim.x) s_cnt[i] = 0;
        __syncthreads();
        const int share = nwarps / nrep;  // warps per replica
        const int r = warp / share;
        if (r < nrep) {
            const uint32_t *rep = sw + r * RW;
            int *cnt_r = s_cnt + r * (q + 1);
            const int me = (warp - r * share) * 32 + lane, stride = share * 32;
            const int agree = agreeing(rep, me, stride);
            if (lane == 0) atomicAdd(cnt_r + q, agree);
            count_states(rep, me, stride, [&](int s, int c) {
                if (lane == 0) atomicAdd(cnt_r + s, c);
            });
        }
        __syncthreads();
        // lane 0 of warp r records replica r (lane 0 of each warp carries the sums)
        if (lane == 0 && warp < nrep) {
            const int *cnt_r = s_cnt + warp * (q + 1);
            int best = 0;
            for (int s = 0; s < q; ++s) best = max(best, cnt_r[s]);
            record_replica(G, first + warp, -cnt_r[q], best, N, sE, sE2, sM);
        }
    } else {
        // one warp per replica
        for (int r = warp; r < nrep; r += nwarps) {
            const uint32_t *rep = sw + r * RW;
            const int agree = agreeing(rep, lane, 32);
            int best = 0;
            count_states(rep, lane, 32, [&](int, int c) { best = max(best, c); });
            if (lane == 0) record_replica(G, first + r, -agree, best, N, sE, sE2, sM);
        }
    }
    if (lane == 0 && (sE | sE2 | sM)) accumulate_totals(totals, sE, sE2, sM);
    group_families(G);
    if constexpr (!LAT) {
        fence_bulk();  // the next group's copies overwrite what was read here
        if (tid == 0) bulk_stores_read();
    }
    __syncthreads();
}

}  // namespace dev
}  // namespace pa
