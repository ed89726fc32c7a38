// pa_kernels.cuh -- device bodies of the population-annealing kernels
// (Barash, Weigel, Shchur & Janke, arXiv:1704.01888), shared by the
// single-run kernels (pa_resample.cu) and the batched kernels (pa_batch.cu)
// so that both run the same arithmetic.  The sweep body is in
// pa_sweep_body.cuh (included here).
//
// Initial populations and layout conversions; resampling bodies (Sec. 2
// step 2, Eq. 2): weights and ln Q, copy numbers and their scan, parent map;
// estimators (Sec. 2 step 4, Eqs. 4-5).
#pragma once
#include <climits>
#include <type_traits>

#include "pa_cluster.cuh"
#include "pa_sweep_body.cuh"

namespace pa {
namespace dev {

// ===========================================================================
// Block reductions (fixed order)
// ===========================================================================
template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Fixed-order block sum of doubles; result valid in thread 0.
__device__ __forceinline__ double block_sum_fixed(double v, double *scratch32)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xFFFFFFFFu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) scratch32[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (warp == 0) {
        r = (lane < (int)(blockDim.x >> 5)) ? scratch32[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r = __dadd_rn(r, __shfl_down_sync(0xFFFFFFFFu, r, o));
    }
    __syncthreads();
    return r;
}

// Block sum of int64; every thread receives the result.
__device__ __forceinline__ long long block_sum_ll(long long v, long long *scratch32)
{
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) scratch32[warp] = v;
    __syncthreads();
    long long r = 0;
    if (warp == 0) {
        r = (lane < (int)(blockDim.x >> 5)) ? scratch32[lane] : 0;
        r = warp_sum(r);
        if (lane == 0) scratch32[0] = r;
    }
    __syncthreads();
    r = scratch32[0];
    __syncthreads();
    return r;
}

// Block-wide exclusive scan of one int per thread; returns the exclusive
// prefix, writes the block total to *total.
__device__ __forceinline__ int block_exclusive_scan(int v, int *scratch32, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) scratch32[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int s = (lane < (int)(blockDim.x >> 5)) ? scratch32[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, s, o);
            if (lane >= o) s += y;
        }
        scratch32[lane] = s;  // inclusive prefix over warps
    }
    __syncthreads();
    const int before = (warp > 0 ? scratch32[warp - 1] : 0) + x - v;
    *total = scratch32[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before;
}

// ===========================================================================
// Initial populations (Sec. 2 step 1; Sec. 5 Eq. 6)
// ===========================================================================

// One site word (32 columns of one colour and row) of one replica; i indexes
// (slot, colour, row, word).  Random start: canonical site i_s = y L + x takes
// floor(Z q / 2^32), Z = word (i_s & 3) of the Philox call with counter
// (i_s >> 2, INIT, 0, slot | stream).  Ground start: every site of the replica
// in the state floor(Z q / 2^32), Z = word (slot & 3) of counter
// (slot >> 2, GROUND, 0, stream).
__device__ __forceinline__ void init_item(uint32_t *spins, int32_t *anc, int q, int L, long long i, uint32_t k0,
                                          uint32_t k1, uint32_t stream_hi, int ground, uint32_t slot0 = 0u)
{
    const int B = state_bits(q);
    const int BP = plane_stride(B);
    const int WPR = row_words(L);
    const int nb_last = L / 2 - 32 * (WPR - 1);
    const int IPC = colour_words(L);
    const int IPR = 2 * IPC;  // site words per replica
    const int slot = (int)(i / IPR);
    const int rem = (int)(i - (long long)slot * IPR);
    const int c = rem / IPC;
    const int it = rem - c * IPC;
    const bool packed = rows_packed(L), banded = rows_banded(L);
    const int nb = (packed || banded) ? 32 : ((it % WPR) == WPR - 1 ? nb_last : 32);
    uint32_t planes[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    const uint32_t key_slot = slot0 + (uint32_t)slot;  // the random numbers follow the global slot
    if (ground) {
        const uint4 w = philox10(make_uint4(key_slot >> 2, DOM_GROUND, 0u, stream_hi), k0, k1);
        const uint32_t alpha = __umulhi(pick_word(w, key_slot & 3), (uint32_t)q);
        const uint32_t vm = nb == 32 ? 0xFFFFFFFFu : ((1u << nb) - 1u);
        for (int p = 0; p < B; ++p) planes[p] = ((alpha >> p) & 1u) ? vm : 0u;
    } else {
        int last = -1;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        for (int b = 0; b < nb; ++b) {
            int y, m;
            if (packed) {
                const int h = 32 * it + b;
                y = h / (L / 2);
                m = h - y * (L / 2);
            } else if (banded) {
                const int k = it / (L / 16);
                y = k + (b >> 3) * (L / 4);
                m = 8 * (it - k * (L / 16)) + (b & 7);
            } else {
                y = it / WPR;
                m = 32 * (it - y * WPR) + b;
            }
            const int x = 2 * m + ((y + c) & 1);
            const int site = y * L + x;
            if ((site >> 2) != last) {
                last = site >> 2;
                w = philox10(make_uint4((uint32_t)last, DOM_INIT, 0u, key_slot | stream_hi), k0, k1);
            }
            const uint32_t s = __umulhi(pick_word(w, site & 3), (uint32_t)q);
            for (int p = 0; p < B; ++p) planes[p] |= ((s >> p) & 1u) << b;
        }
    }
    uint32_t *dst = spins + (size_t)slot * replica_words_of(B, L) + (size_t)rem * BP;
    for (int p = 0; p < BP; ++p) dst[p] = planes[p];
    if (rem == 0 && anc) anc[slot] = (int32_t)key_slot;
}

// Rows of whole words (L a multiple of 64) and packed rows: words w of the two
// colours together hold the 64 canonical sites 64 w .. 64 w + 63, in order:
// bit b the sites 64 w + 2 b and 64 w + 2 b + 1, the even one of colour 0 in
// even rows and of colour 1 in odd rows.
__host__ __device__ constexpr bool words_in_order(int L) { return L % 64 == 0 || rows_packed(L); }

// Bits of word w whose site lies in an odd row.
__device__ __forceinline__ uint32_t odd_row_bits(int L, int w)
{
    if (L >= 64) return (64 * w / L) & 1 ? 0xFFFFFFFFu : 0u;
    return L == 32 ? 0xFFFF0000u : L == 16 ? 0xFF00FF00u : 0xF0F0F0F0u;
}

// Random start of words w of both colours of one replica (words_in_order; i =
// slot IPC + w): 16 Philox calls of four sites, each made once (init_item makes
// them for either colour), the states' bits shifted into the planes site by
// site.  566 -> 149 us for q = 8, L = 128, R = 1e4.
template <int B>
__device__ __forceinline__ void init_words(uint32_t *spins, int32_t *anc, int q, int L, long long i, uint32_t k0,
                                           uint32_t k1, uint32_t stream_hi, uint32_t slot0)
{
    constexpr int BP = plane_stride(B);
    const int IPC = colour_words(L);
    const int slot = (int)(i / IPC);
    const int w = (int)(i - (long long)slot * IPC);
    const uint32_t key_slot = slot0 + (uint32_t)slot;
    uint32_t even[B], odd[B];
#pragma unroll
    for (int p = 0; p < B; ++p) even[p] = odd[p] = 0u;
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
        const uint4 z = philox10(make_uint4((uint32_t)(16 * w + c), DOM_INIT, 0u, key_slot | stream_hi), k0, k1);
        uint32_t s[4] = {__umulhi(z.x, (uint32_t)q), __umulhi(z.y, (uint32_t)q), __umulhi(z.z, (uint32_t)q),
                         __umulhi(z.w, (uint32_t)q)};
#pragma unroll
        for (int p = 0; p < B; ++p) {
            even[p] = __funnelshift_r(even[p], s[0] >> p, 1);
            even[p] = __funnelshift_r(even[p], s[2] >> p, 1);
            odd[p] = __funnelshift_r(odd[p], s[1] >> p, 1);
            odd[p] = __funnelshift_r(odd[p], s[3] >> p, 1);
        }
    }
    const uint32_t m = odd_row_bits(L, w);
    uint32_t c0[BP], c1[BP];
#pragma unroll
    for (int p = 0; p < BP; ++p) {
        c0[p] = p < B ? (even[p < B ? p : 0] & ~m) | (odd[p < B ? p : 0] & m) : 0u;
        c1[p] = p < B ? (odd[p < B ? p : 0] & ~m) | (even[p < B ? p : 0] & m) : 0u;
    }
    uint32_t *dst = spins + (size_t)slot * replica_words_of(B, L) + (size_t)w * BP;
    store_planes<BP>(dst, c0);
    store_planes<BP>(dst + (size_t)IPC * BP, c1);
    if (w == 0 && anc) anc[slot] = (int32_t)key_slot;
}

__device__ __forceinline__ void init_words_any(uint32_t *spins, int32_t *anc, int q, int L, long long i, uint32_t k0,
                                               uint32_t k1, uint32_t stream_hi, uint32_t slot0 = 0u)
{
    switch (state_bits(q)) {
    case 1: init_words<1>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    case 2: init_words<2>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    case 3: init_words<3>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    case 4: init_words<4>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    case 5: init_words<5>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    case 6: init_words<6>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    default: init_words<7>(spins, anc, q, L, i, k0, k1, stream_hi, slot0); break;
    }
}

// The 64 canonical sites of words w of both colours (words_in_order; i = slot
// IPC + w) as bytes: four sites at a time, each plane's bits spread over four
// bytes by a multiplication.  One site per thread, with divisions, took 136 us
// for 4000 replicas of 64 x 64 (16 MB); now 11 us.
__device__ __forceinline__ void canonical_words(const uint32_t *spins, uint8_t *out, int q, int L, long long i)
{
    const int B = state_bits(q), BP = plane_stride(B);
    const int IPC = colour_words(L);
    const long long r = i / IPC;
    const int w = (int)(i - r * IPC);
    const uint32_t *src = spins + (size_t)r * replica_words_of(B, L) + (size_t)w * BP;
    const uint32_t m = odd_row_bits(L, w);
    uint32_t v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = 0u;
    for (int p = 0; p < B; ++p) {
        const uint32_t c0 = src[p], c1 = src[(size_t)IPC * BP + p];
        const uint32_t even = (c0 & ~m) | (c1 & m), odd = (c1 & ~m) | (c0 & m);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const uint32_t e = (((even >> (2 * j)) & 3u) * 0x8001u) & 0x00010001u;
            const uint32_t o = (((odd >> (2 * j)) & 3u) * 0x800100u) & 0x01000100u;
            v[j] |= (e | o) << p;
        }
    }
    uint4 *dst = reinterpret_cast<uint4 *>(out + 64 * i);
#pragma unroll
    for (int j = 0; j < 4; ++j) dst[j] = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}

// One site word (i indexes (slot, colour, word) as in init_item) of the
// multi-spin-coded layout from a population in the canonical layout
// [slot][y][x], one byte per spin (the inverse of canonical_state).
__device__ __forceinline__ void from_canonical_item(uint32_t *spins, const uint8_t *canon, int q, int L, long long i)
{
    const int B = state_bits(q);
    const int BP = plane_stride(B);
    const int WPR = row_words(L);
    const int nb_last = L / 2 - 32 * (WPR - 1);
    const int IPC = colour_words(L);
    const int IPR = 2 * IPC;
    const long long slot = i / IPR;
    const int rem = (int)(i - slot * IPR);
    const int c = rem / IPC;
    const int it = rem - c * IPC;
    const bool packed = rows_packed(L), banded = rows_banded(L);
    const int nb = (packed || banded) ? 32 : ((it % WPR) == WPR - 1 ? nb_last : 32);
    const uint8_t *rep = canon + slot * (long long)L * L;
    uint32_t planes[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    for (int b = 0; b < nb; ++b) {
        int y, m;
        if (packed) {
            const int h = 32 * it + b;
            y = h / (L / 2);
            m = h - y * (L / 2);
        } else if (banded) {
            const int k = it / (L / 16);
            y = k + (b >> 3) * (L / 4);
            m = 8 * (it - k * (L / 16)) + (b & 7);
        } else {
            y = it / WPR;
            m = 32 * (it - y * WPR) + b;
        }
        const uint32_t s = rep[y * L + 2 * m + ((y + c) & 1)];
        for (int p = 0; p < B; ++p) planes[p] |= ((s >> p) & 1u) << b;
    }
    uint32_t *dst = spins + (size_t)slot * replica_words_of(B, L) + (size_t)rem * BP;
    for (int p = 0; p < BP; ++p) dst[p] = planes[p];
}

// State of canonical site i (= r N + y L + x) of a multi-spin-coded population.
__device__ __forceinline__ uint8_t canonical_state(const uint32_t *spins, int q, int L, long long i)
{
    const int N = L * L;
    const int B = state_bits(q);
    const int BP = plane_stride(B);
    const int IPC = colour_words(L);
    const long long r = i / N;
    const int site = (int)(i - r * N);
    const int y = site / L, x = site - y * L;
    const int c = (x + y) & 1;
    const int m = x >> 1;
    int it, b;
    if (rows_packed(L)) {
        const int h = y * (L / 2) + m;
        it = h >> 5;
        b = h & 31;
    } else if (rows_banded(L)) {
        const int a = y / (L / 4), k = y - a * (L / 4);
        it = k * (L / 16) + (m >> 3);
        b = 8 * a + (m & 7);
    } else {
        it = y * row_words(L) + (m >> 5);
        b = m & 31;
    }
    const uint32_t *w = spins + (size_t)r * replica_words_of(B, L) + (size_t)((c * IPC + it) * BP);
    uint32_t s = 0;
    for (int p = 0; p < B; ++p) s |= ((w[p] >> b) & 1u) << p;
    return (uint8_t)s;
}

// ===========================================================================
// Resampling bodies (Sec. 2 step 2, Eq. 2)
// ===========================================================================

// Exact sum of the weights.  S = sum_k h_k w_k over the occupied energy bins
// (h_k < 2^24 replicas, w_k a double in [0, 1]) is accumulated exactly and
// rounded once to the nearest double, ties to even, so that S -- and with it
// every rho_j -- does not depend on which lane, warp or block adds which term.
// The accumulator counts units of 2^-1074 (the smallest positive double): a
// term h m 2^(pos - 1074) (m the 53-bit significand) is the integer h m < 2^77
// placed at bit pos <= 1022.  Limb i of the shared array collects bits
// 32 i .. 32 i + 31 in a 64-bit counter, so the carries of up to 2^32
// additions fit and are propagated once, at the end.  The sum is below
// R_cap < 2^24, i.e. below bit 1098: 36 limbs.
constexpr int kSumLimbs = 36;

// The term h w (w > 0) as four 32-bit chunks c[0..3] of limbs li .. li + 3.
__device__ __forceinline__ int exact_term(uint32_t h, double w, uint32_t (&c)[4])
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(w);
    const int ef = (int)(bits >> 52) & 0x7FF;
    const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | (ef ? (1ull << 52) : 0ull);
    const int pos = ef ? ef - 1 : 0;
    const unsigned long long lo = m * (unsigned long long)h;
    const unsigned long long hi = __umul64hi(m, (unsigned long long)h);
    const int sh = pos & 31;
    const unsigned long long lo_s = lo << sh;
    const unsigned long long hi_s = (hi << sh) | (sh ? lo >> (64 - sh) : 0ull);
    c[0] = (uint32_t)lo_s;
    c[1] = (uint32_t)(lo_s >> 32);
    c[2] = (uint32_t)hi_s;
    c[3] = (uint32_t)(hi_s >> 32);
    return pos >> 5;
}

// Adds the terms of the occupied bins among k_begin .. k_end - 1 to the
// shared limbs.  Consecutive bins have weights within a few binades of one
// another, so a thread sums its terms in five register limbs (li - 1 .. li +
// 3 of the first term) and adds them to the shared array itself only when a
// term falls outside them; at the end the lanes of a warp whose limbs start at
// the same place add theirs up by shuffles and one lane adds the sums (64-bit
// shared atomics on the same few limbs are compare-and-swap loops).  Every
// thread of the block takes part.
__device__ __forceinline__ void exact_add_range(unsigned long long *acc, const int32_t *hist, const double *wtab,
                                                int kref, int k_begin, int k_end)
{
    unsigned long long w[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
    int base = -2;
    // four bins at a time: their loads issue together
    for (int k0 = k_begin; k0 < k_end; k0 += 4) {
        int h[4];
        double wk[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = k0 + i < k_end ? hist[k0 + i] : 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int k = k0 + i;
            wk[i] = h[i] > 0 ? wtab[k >= kref ? k - kref : kref - k] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (h[i] <= 0 || wk[i] == 0.0) continue;
            uint32_t c[4];
            const int li = exact_term((uint32_t)h[i], wk[i], c);
            if (li < base || li > base + 1) {
                if (base >= 0) {
#pragma unroll
                    for (int l = 0; l < 5; ++l) {
                        if (w[l]) atomicAdd(acc + base + l, w[l]);
                        w[l] = 0ull;
                    }
                }
                base = li > 0 ? li - 1 : 0;
            }
            const bool up = li != base;
            w[0] += up ? 0u : c[0];
            w[1] += up ? c[0] : c[1];
            w[2] += up ? c[1] : c[2];
            w[3] += up ? c[2] : c[3];
            w[4] += up ? c[3] : 0u;
        }
    }
    const int lane = threadIdx.x & 31;
    unsigned pending = __ballot_sync(0xFFFFFFFFu, base >= 0);
    while (pending) {
        const int at = __shfl_sync(0xFFFFFFFFu, base, __ffs(pending) - 1);
        const bool mine = base == at;
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            const unsigned long long sum = warp_sum(mine ? w[l] : 0ull);
            if (lane == 0 && sum) atomicAdd(acc + at + l, sum);
        }
        pending &= ~__ballot_sync(0xFFFFFFFFu, mine);
    }
}

// Bits lowpos .. lowpos + 63 of normalised 32-bit limbs (lowpos >= 0).
__device__ __forceinline__ unsigned long long limb_bits64(const unsigned long long *acc, int lowpos)
{
    const int li = lowpos >> 5, sh = lowpos & 31;
    auto limb = [&](int i) -> unsigned long long { return i < kSumLimbs ? acc[i] : 0ull; };
    const unsigned long long lo64 = limb(li) | (limb(li + 1) << 32);
    return sh ? (lo64 >> sh) | (limb(li + 2) << (64 - sh)) : lo64;
}

// Propagates the carries and rounds the accumulated value to the nearest
// double (one thread; the value must be at least 1, i.e. bit 1074 or above).
__device__ __forceinline__ double exact_round(unsigned long long *acc)
{
    unsigned long long carry = 0ull, nonzero = 0ull;  // bit i: limb i is not zero
#pragma unroll
    for (int i = 0; i < kSumLimbs; ++i) {
        const unsigned long long v = acc[i] + carry;
        acc[i] = v & 0xFFFFFFFFull;
        carry = v >> 32;
        nonzero |= (unsigned long long)((uint32_t)v != 0u) << i;
    }
    if (!nonzero) return 0.0;
    const int t = 63 - __clzll((long long)nonzero);
    int p = 32 * t + 31 - __clz((uint32_t)acc[t]);  // top bit
    const unsigned long long x = limb_bits64(acc, p - 63);  // bit 63 = top bit
    unsigned long long mant = x >> 11;
    const bool round = (x >> 10) & 1ull;
    const int low = p - 63;  // bits below it
    bool sticky = (x & 0x3FFull) != 0ull || (nonzero & ((1ull << (low >> 5)) - 1ull)) != 0ull;
    if (!sticky && (low & 31)) sticky = (acc[low >> 5] & ((1ull << (low & 31)) - 1ull)) != 0ull;
    if (round && (sticky || (mant & 1ull))) mant += 1ull;
    if (mant >> 53) {
        mant >>= 1;
        p += 1;
    }
    // value = mant 2^(p - 52 - 1074): biased exponent p - 1074 + 1023
    return __longlong_as_double((long long)(((unsigned long long)(p - 51) << 52) | (mant & 0xFFFFFFFFFFFFFull)));
}

// One cluster: reference bin, S (exact sum of h_k w_k, weights from the host
// table wtab by distance |k - k_ref|) and ln Q of the pending resample.
// Latency bound: a reading of the histogram for its occupied range, one of
// that range with its weights, and a serial rounding.  The blocks share the
// bins and the first adds up their limbs (in one block: 10, 25 and 97 us with
// 2049, 32769 and 131073 bins).
// R_prev_all: the population size R_{i-1} when the histogram covers several
// GPUs' replicas (0: this GPU's own, st->pop).
struct WeightsShared {
    unsigned long long acc[kSumLimbs], sum[kSumLimbs];
    int sc[64], ext[2];
};
constexpr int kWeightsThreads = 512;
__device__ __forceinline__ void weights_body(const int32_t *hist, int nbins, double dbeta, const double *wtab,
                                             DevState *st, WeightsShared &sh, int R_prev_all = 0)
{
    if (st->err) return;  // the same in every block
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), c = (int)cl.block_rank(), tid = threadIdx.x, n = blockDim.x;
    for (int i = tid; i < kSumLimbs; i += n) sh.acc[i] = 0ull;
    int lo = INT_MAX, hi = -1;
#pragma unroll 8
    for (int k = c * n + tid; k < nbins; k += C * n) {
        if (hist[k] > 0) {
            lo = min(lo, k);
            hi = max(hi, k);
        }
    }
    cluster_extremes(cl, lo, hi, sh.sc, sh.ext);
    // reference bin: lowest occupied for dbeta >= 0, highest for dbeta < 0
    const int kref = dbeta >= 0.0 ? lo : hi;
    const long long range = lo <= hi ? (long long)hi - lo + 1 : 0;
    const int k0 = lo + (int)(range * c / C), k1 = lo + (int)(range * (c + 1) / C);
    const int per = (k1 - k0 + n - 1) / n;  // a contiguous range of bins per thread
    exact_add_range(sh.acc, hist, wtab, kref, min(k1, k0 + tid * per), min(k1, k0 + (tid + 1) * per));
    cl.sync();
    if (c == 0) {
        if (tid < kSumLimbs) {
            unsigned long long s = 0ull;
            for (int r = 0; r < C; ++r) s += cl.map_shared_rank(sh.acc, r)[tid];
            sh.sum[tid] = s;
        }
        __syncthreads();
        if (tid == 0) {
            const double S = exact_round(sh.sum);
            const int E_ref = kref - (nbins - 1);
            st->S = S;
            st->E_ref = E_ref;
            st->ties = 0;
            const int R_prev = R_prev_all > 0 ? R_prev_all : st->pop;
            st->lnQ = __dadd_rn(__dmul_rn(-dbeta, (double)E_ref), log(S / (double)R_prev));
        }
    }
    cl.sync();  // the blocks' limbs stay until the first has read them
}

// Cumulative probabilities F_n of a full piece (mean 64) of a Poisson draw, by
// the recursion of poisson_draw; one thread, once.
constexpr double kPoissonPiece = 64.0;
constexpr int kPoissonTable = kPoissonTableEntries;
__device__ __forceinline__ void poisson_table(double *F_out)
{
    double p = exp(-kPoissonPiece), F = p;
    F_out[0] = F;
    for (int n = 1; n < kPoissonTable; ++n) {
        p = __ddiv_rn(__dmul_rn(p, kPoissonPiece), (double)n);
        F = __dadd_rn(F, p);
        F_out[n] = F;
    }
}

// inv[n] = 1 / n for n = 1 .. kPoissonTable - 1, by the whole block.
__device__ __forceinline__ void reciprocals(double *inv)
{
    for (int n = threadIdx.x; n < kPoissonTable; n += blockDim.x) inv[n] = n ? __ddiv_rn(1.0, (double)n) : 0.0;
}

// A Poisson draw with mean rho for replica j (Sec. 2, Eq. 1): inversion of
// the cumulative distribution with the mean split into pieces of at most 64;
// the k-th uniform (U_k + 1/2) / 2^32 is word k & 3 of counter
// (j, RESAMPLE | (1 + k / 4), step, stream).
//
// Bound by the serial chain of the replicas with the largest means (a population
// with a few families has copy numbers of hundreds: 149 us per launch for 5003
// replicas).  Full pieces share one cumulative table (full, null: none), in
// which the result is found by bisection -- the recursion visits F_0 .. F_n in
// rising order, so of the near-tie tests only those of F_{n-1} and F_n can
// differ from the rest.  The others divide by n < 256 through inv[n] = 1 / n and
// one residual (Markstein, IBM J. Res. Dev. 34, 1990): q = x inv is within two
// units in the last place of x / n, x - q n is exact in a fused operation, and
// q + (x - q n) inv misses x / n by less than 2^-50 units before it is rounded,
// while x / n stays 1 / (2 n) units away from every midpoint: the result is the
// quotient correctly rounded, and every F_n the double that the division gives.
__device__ __forceinline__ int poisson_draw(double rho, int j, int step, uint32_t stream_hi, uint32_t k0, uint32_t k1,
                                            const double *inv, const double *full, bool &tie)
{
    int r = 0;
    tie = false;
    double remaining = rho;
    uint32_t k = 0;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    while (remaining > 0.0) {
        const double mu = remaining < kPoissonPiece ? remaining : kPoissonPiece;
        remaining = __dsub_rn(remaining, mu);
        if ((k & 3) == 0)
            w = philox10(make_uint4((uint32_t)j, DOM_RESAMPLE | (1u + (k >> 2)), (uint32_t)step, stream_hi), k0, k1);
        const double u = __dmul_rn(__dadd_rn((double)pick_word(w, k & 3), 0.5), 0x1p-32);
        k += 1;
        if (full && mu == kPoissonPiece && u <= full[kPoissonTable - 1]) {
            int lo = 0, hi = kPoissonTable - 1;  // the first n with u <= F_n
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (u > full[mid]) lo = mid + 1; else hi = mid;
            }
            if (fabs(__dsub_rn(u, full[lo])) < 0x1p-40) tie = true;
            if (lo > 0 && fabs(__dsub_rn(u, full[lo - 1])) < 0x1p-40) tie = true;
            r += lo;
            continue;
        }
        double p = exp(-mu);
        double F = p;
        int n = 0;
        for (;;) {
            if (fabs(__dsub_rn(u, F)) < 0x1p-40) tie = true;
            if (!(u > F && n < 1000)) break;
            n += 1;
            const double x = __dmul_rn(p, mu);
            if (n < kPoissonTable) {
                const double q = __dmul_rn(x, inv[n]);
                p = __fma_rn(__fma_rn(-q, (double)n, x), inv[n], q);
            } else {
                p = __ddiv_rn(x, (double)n);
            }
            F = __dadd_rn(F, p);
        }
        r += n;
    }
    return r;
}

// Near-tie flag of a rounded copy number: frac(rho) within 2^-48 max(1, rho)
// of the rule's boundary (u / 2^32 for nearest-integer copy numbers, 1/2 for
// ROUND), where a last-place change of rho could change the outcome.
__device__ __forceinline__ bool round_tie(double rho, double frac, double boundary)
{
    return fabs(__dsub_rn(frac, boundary)) < __dmul_rn(0x1p-48, fmax(1.0, rho));
}

// One block of old replicas (chunk of blockDim): copy numbers and their block
// scan.  About 25 FP64 instructions per replica (many more for Poisson draws)
// at two lanes per clock and SM: small chunks spread them over the SMs.
// w(E_j) comes from the host table wtab by distance |E_j - E_ref|.
// j0: global index of local replica 0 (a population shared by several GPUs):
// the random numbers of replica j follow j0 + j.
__device__ __forceinline__ void counts_body(int chunk, const int32_t *E, int twoN, int R_target, int mode, int step,
                                            uint32_t stream_hi, uint32_t k0, uint32_t k1, const double *wtab,
                                            int32_t *counts, int32_t *local_off, int32_t *blocksum, DevState *st,
                                            int *s_i, double *s_inv, const double *poisson_full, int j0 = 0)
{
    if (st->err) return;
    const int R_prev = st->pop;
    if (chunk * (int)blockDim.x >= R_prev) return;
    if (mode == 2) {
        reciprocals(s_inv);
        __syncthreads();
    }
    const int j = chunk * blockDim.x + threadIdx.x;
    int r = 0;
    bool tie = false;
    if (j < R_prev) {
        const int d = E[j] - st->E_ref;
        const double w = wtab[d >= 0 ? d : -d];
        const double rho = __ddiv_rn(__dmul_rn((double)R_target, w), st->S);
        const double n = floor(rho);
        const double frac = __dsub_rn(rho, n);
        const int jg = j0 + j;
        if (mode == 2) {
            r = poisson_draw(rho, jg, step, stream_hi, k0, k1, s_inv, poisson_full, tie);
        } else if (mode == 3) {
            r = 1;
        } else if (mode == 1) {
            r = (int)n + (frac >= 0.5);
            tie = round_tie(rho, frac, 0.5);
        } else {
            const uint4 u = philox10(make_uint4((uint32_t)jg >> 2, DOM_RESAMPLE, (uint32_t)step, stream_hi), k0, k1);
            const uint32_t uj = pick_word(u, jg & 3);
            r = (int)n + ((double)uj < __dmul_rn(frac, 4294967296.0));
            tie = round_tie(rho, frac, __dmul_rn((double)uj, 0x1p-32));
        }
        counts[j] = r;
    }
    const unsigned nt = __popc(__ballot_sync(0xFFFFFFFFu, tie));
    if ((threadIdx.x & 31) == 0 && nt) atomicAdd(&st->ties, (int)nt);
    int total;
    const int before = block_exclusive_scan(r, s_i, &total);
    if (j < R_prev) local_off[j] = before;
    if (threadIdx.x == 0) blocksum[chunk] = total;
}

// One block (chunk of nchunks): block offsets, new size (capacity check),
// parent map; the chunks also clear the histogram for the next sweep.
// min_total: smallest valid number of children (1; 0 for one GPU's share of
// a population spread over several, which may receive all its replicas from
// the others).
//
// Every block takes the capacity decision from its own sum over the chunks.
// Chunk 0's block records a refusal in st->err while others may still be
// reading the flag here: threads that each went by their own reading could
// leave some of the block's barriers to the rest, which would use the stale
// sums of the chunk before as offsets into parent.  So thread 0 alone reads it,
// and what it saw reaches the others as part of the sum.
__device__ __forceinline__ void scatter_body(int chunk, int nchunks, const int32_t *counts, const int32_t *local_off,
                                             const int32_t *blocksum, int32_t *parent, int R_cap, int32_t *hist_zero,
                                             int nbins, DevState *st, long long *s_l, int min_total = 1)
{
    const bool failed = threadIdx.x == 0 && *(volatile int32_t *)&st->err;
    const int R_prev = st->pop;
    const int nb = (R_prev + blockDim.x - 1) / blockDim.x;
    long long off = 0, tot = failed ? 1ll << 60 : 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        const long long v = blocksum[b];
        tot += v;
        if (b < chunk) off += v;
    }
    tot = block_sum_ll(tot, s_l);
    off = block_sum_ll(off, s_l);
    if (tot > R_cap || tot < min_total) {
        if (chunk == 0 && threadIdx.x == 0 && !failed) st->err = 2;  // PA_ERR_CAPACITY
        return;
    }
    if (chunk == 0 && threadIdx.x == 0) st->pop_next = (int)tot;
    for (int k = chunk * blockDim.x + threadIdx.x; k < nbins; k += nchunks * blockDim.x) hist_zero[k] = 0;
    if (chunk >= nb) return;
    const int j = chunk * blockDim.x + threadIdx.x;
    if (j < R_prev) {
        const int o = (int)off + local_off[j];
        const int r = counts[j];
        for (int c = 0; c < r; ++c) parent[o + c] = j;
    }
}

// One thread: estimators of the step (Sec. 2 step 4, Eqs. 4-5), ln Z of Eq. 2,
// buffer parity flip.  S_f, nf: family entropy and count (0 without families).
// R_all: the population size when the sums and family counts cover several
// GPUs' replicas (0: this GPU's own).
__device__ __forceinline__ void finalize_record(DevState *st, unsigned long long *acc, DevObs *obs, double beta, int q,
                                                int N, int gathered, int resampled, int R_all, double S_f,
                                                long long nf)
{
    const int R_local = gathered ? st->pop_next : st->pop;
    const int R = R_all > 0 ? R_all : R_local;
    const long long sE = (long long)acc[0], sE2 = (long long)acc[1], sM = (long long)acc[2];
    acc[0] = acc[1] = acc[2] = 0ull;
    const double meanE = (double)sE / (double)R;
    const double meanE2 = (double)sE2 / (double)R;
    const double C =
        __ddiv_rn(__dmul_rn(__dmul_rn(beta, beta), __dsub_rn(meanE2, __dmul_rn(meanE, meanE))), (double)N);
    const double meanM = (double)((long long)q * sM - (long long)N * R) / __dmul_rn((double)(q - 1), (double)R);
    double lnQ = 0.0;
    if (resampled) {
        lnQ = st->lnQ;
        st->lnZ = __dadd_rn(st->lnZ, lnQ);
    }
    if (gathered) {
        st->pop = R_local;
        st->parity ^= 1;
    }
    DevObs o;
    o.beta = beta;
    o.lnQ = lnQ;
    o.lnZ = st->lnZ;
    o.meanE = meanE;
    o.meanE2 = meanE2;
    o.C = C;
    o.meanM = meanM;
    o.S_f = S_f;
    o.R = R;
    o.n_families = nf;
    // several GPUs: acc[3] holds the near ties summed over them
    o.n_near_ties = resampled ? (R_all > 0 ? (long long)acc[3] : (long long)st->ties) : 0;
    if (R_all > 0) acc[3] = 0ull;
    o.sumE = sE;
    o.sumE2 = sE2;
    o.sumMt = sM;
    *obs = o;
}

// One block: family entropy, then the estimators.
__device__ __forceinline__ void finalize_body(DevState *st, unsigned long long *acc, int32_t *fam, int R0, DevObs *obs,
                                              double beta, int q, int N, int gathered, int resampled, double *s_d,
                                              long long *s_l, int R_all = 0)
{
    if (st->err) return;
    const int R = R_all > 0 ? R_all : gathered ? st->pop_next : st->pop;
    double Sf = 0.0;
    long long nf = 0;
    if (fam) {
        double part = 0.0;
        for (int f = threadIdx.x; f < R0; f += blockDim.x) {
            const int c = fam[f];
            if (c > 0) {
                const double nu = (double)c / (double)R;
                part = __dsub_rn(part, __dmul_rn(nu, log(nu)));
                nf += 1;
                fam[f] = 0;
            }
        }
        Sf = block_sum_fixed(part, s_d);
        nf = block_sum_ll(nf, s_l);
    }
    if (threadIdx.x == 0) finalize_record(st, acc, obs, beta, q, N, gathered, resampled, R_all, Sf, nf);
}

}  // namespace dev
}  // namespace pa
