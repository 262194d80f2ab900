// Exhaustive seed search on the device (Section 5.2): for every slice of every plane the seed with the fewest
// wrong care bits among all 2^n_in is found (the smallest seed among equals).
//
// The seeds are not tried one by one.  Column c of M, restricted to the slice's care positions, is a bit vector v_c; a
// seed is a choice of columns and its error vector is (wanted bits) ^ xor of the chosen v_c.  Column operations bring
// the v_c into reduced form: in ascending order, a column that is not zero by then takes its lowest bit as its pivot, which is
// removed from all other columns and from the wanted bits, and t_c keeps the seed that belongs to v_c.  What is
// left of the wanted bits, E, is the error vector of the seed that gets every pivot bit right, and a set e of wrong pivots has
//
//     key(e) = popcount(E ^ xor of v_c, c in e) << 20 | seed(E) ^ xor of t_c, c in e,      at least |e| errors.
//
// The search is the minimum of the keys, taken in the order of |e|: once the best count is B, sizes above B cannot
// matter.  (Ties go to the smallest seed.  Pivot columns are the lowest possible ones, so the seed with all other bits 0, which
// the keys hold, is the smallest of those with the same errors.)  Sizes 0 and 1 are done by a thread per slice and decide
// 92 % of them; of the rest the warp finishes one slice after the other, the lanes sharing the pairs and, for one slice in a
// hundred, sets of three to five columns; what remains tries all 2^rank sets in Gray-code order.
// Columns that the elimination leaves zero are only sorted out for what the pairs have not decided: a test of all columns in every slice's
// own thread costs the LSTM gates 4 %.
//
// The care positions of a slice are squeezed together first: up to 32 of them make one word per column, up to 64 two, whatever
// n_out is.  A step takes each lane's next care position; its row of M, with the bits of four columns in the four
// bytes of a word, is added to the columns' bytes shifted by the step's number, so that eight steps fill a byte of every column with
// three additions each, for 12 columns.  Slices with more care bits than that try all seeds.
//
// Bound: integer instructions.  600 000 slices of 60 x 12 (20 % care bits, two planes of 6000 x 3000) take 53 us: 31.7 M warp
// instructions with 30.6 of 32 lanes active, 19.7 M of them on the integer pipe, which starts one every other cycle and is
// busy 70 % of the time.  (Elimination of rows in a loop over the care bits: 126 us, 79 M instructions with 18.5 lanes active.)
#include "sqnn_launch.h"

#include <cuda_runtime.h>

namespace sqnn {

namespace {

struct SearchArgs {
    uint32_t rows[SQNN_MAX_N_OUT];   // rows of M (the library holds no device memory: passed by value)
    uint32_t n_out, n_in, n_q;
    uint64_t mn, words64, slices;
    const uint64_t *planes, *mask;
    uint32_t *wc;
    uint16_t *np;
};

// NW words of a packed vector (`words` 32-bit words long) from bit p on; words past its end read 0.
template <int NW>
SQNN_DEV void load_bits(const uint64_t *__restrict__ vec, uint64_t words, uint64_t p, uint32_t (&out)[NW])
{
    const uint64_t w = p >> 5;
    const uint32_t *from = reinterpret_cast<const uint32_t *>(vec) + w;
    const uint32_t left = words - w < NW + 1 ? (uint32_t)(words - w) : NW + 1;
    uint32_t raw[NW + 1];
#pragma unroll
    for (uint32_t k = 0; k < NW + 1; ++k) raw[k] = k < left ? __ldg(from + k) : 0u;
#pragma unroll
    for (int k = 0; k < NW; ++k) out[k] = __funnelshift_r(raw[k], raw[k + 1], (uint32_t)p & 31u);
}

// Row j of M, another j in every lane: by a generic load, since the lanes of a constant load take turns.
SQNN_DEV uint32_t row_of(const SearchArgs &S, uint32_t j)
{
    uint32_t row;
    asm("ld.u32 %0, [%1];" : "=r"(row) : "l"(S.rows + j));
    return row;
}

constexpr uint32_t SEARCH_THREADS = 128;
constexpr uint32_t MAX_CARE = 64;                         // care bits the vectors have room for

SQNN_DEV uint32_t warp_min(uint32_t v)
{
    return __reduce_min_sync(0xffffffffu, v);
}

// The whole warp tries all seeds of one slice: the lanes split them by their top bits and walk the rest in
// Gray-code order, one XOR with a column of M per seed.
template <int NW>
SQNN_DEV uint32_t try_all_seeds(const uint32_t (*cols)[NW], uint32_t n_in, const uint32_t (&want)[NW], const uint32_t (&care)[NW], uint32_t lane)
{
    const uint32_t low_bits = n_in > 5 ? n_in - 5 : 0, lanes_used = n_in >= 5 ? 32u : (1u << n_in);
    uint32_t best = 0xffffffffu;
    if (lane < lanes_used) {
        const uint32_t top = lane << low_bits;
        uint32_t out[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) out[k] = 0;
        for (uint32_t t = low_bits; t < n_in; ++t)
            if ((top >> t) & 1u) {
#pragma unroll
                for (int k = 0; k < NW; ++k) out[k] ^= cols[t][k];
            }
        const uint32_t count = 1u << low_bits;
        for (uint32_t i = 0; i < count; ++i) {
            if (i != 0) {
                const uint32_t t = (uint32_t)__ffs((int)i) - 1u;          // bit that changes in the Gray code
#pragma unroll
                for (int k = 0; k < NW; ++k) out[k] ^= cols[t][k];
            }
            uint32_t wrong = 0;
#pragma unroll
            for (int k = 0; k < NW; ++k) wrong += (uint32_t)__popc((out[k] ^ want[k]) & care[k]);
            best = min(best, (wrong << 20) | top | (i ^ (i >> 1)));       // n_in <= 20, wrong <= 256
        }
    }
    return warp_min(best);
}

// How v_c and t_c are held: KW = 1 or 2 words of care bits and a word of t_c; KW = 0 for both in one word, t_c in its low NI bits,
// where the care bits fit above them (for the LSTM gates 20 are enough for seven warps of eight: a third of the
// elimination's instructions less).
template <int KW, int NI>
struct Candidate {                                                        // an error vector and its seed
    uint32_t e[KW], seed;
    SQNN_DEV uint32_t key() const
    {
        uint32_t wrong = 0;
#pragma unroll
        for (int k = 0; k < KW; ++k) wrong += (uint32_t)__popc(e[k]);
        return (wrong << 20) + seed;
    }
    SQNN_DEV bool none() const
    {
        uint32_t any = 0;
#pragma unroll
        for (int k = 0; k < KW; ++k) any |= e[k];
        return any == 0;
    }
    SQNN_DEV void add(const Candidate &o)
    {
#pragma unroll
        for (int k = 0; k < KW; ++k) e[k] ^= o.e[k];
        seed ^= o.seed;
    }
    SQNN_DEV Candidate lowest() const                                     // its lowest care bit, if any
    {
        Candidate p{};
        p.e[0] = e[0] & (0u - e[0]);
        if constexpr (KW == 2) p.e[KW - 1] = e[0] ? 0u : e[KW - 1] & (0u - e[KW - 1]);
        return p;
    }
    SQNN_DEV bool has(const Candidate &p) const
    {
        uint32_t any = 0;
#pragma unroll
        for (int k = 0; k < KW; ++k) any |= e[k] & p.e[k];
        return any != 0;
    }
    SQNN_DEV Candidate from(uint32_t src) const
    {
        Candidate x;
#pragma unroll
        for (int k = 0; k < KW; ++k) x.e[k] = __shfl_sync(0xffffffffu, e[k], src);
        x.seed = __shfl_sync(0xffffffffu, seed, src);
        return x;
    }
};
template <int NI>
struct Candidate<0, NI> {
    static constexpr uint32_t CARE = ~((1u << NI) - 1u);
    uint32_t w;
    SQNN_DEV uint32_t key() const { return ((uint32_t)__popc(w & CARE) << 20) + (w & ~CARE); }
    SQNN_DEV bool none() const { return (w & CARE) == 0; }
    SQNN_DEV void add(const Candidate &o) { w ^= o.w; }
    SQNN_DEV Candidate lowest() const { return Candidate{(w & CARE) & (0u - (w & CARE))}; }
    SQNN_DEV bool has(const Candidate &p) const { return (w & p.w) != 0; }
    SQNN_DEV Candidate from(uint32_t src) const { return Candidate{__shfl_sync(0xffffffffu, w, src)}; }
};

// The reduced columns of one slice per thread, for the slices the whole warp finishes.
template <int NI>
struct Columns {
    uint32_t word[3][NI][SEARCH_THREADS + 1];                            // + 1: the columns of a slice in different banks
    template <int KW>
    SQNN_DEV void put(uint32_t c, uint32_t slot, const Candidate<KW, NI> &x)
    {
        if constexpr (KW == 0) {
            word[0][c][slot] = x.w;
        } else {
#pragma unroll
            for (int k = 0; k < KW; ++k) word[k][c][slot] = x.e[k];
            word[2][c][slot] = x.seed;
        }
    }
    template <int KW>
    SQNN_DEV Candidate<KW, NI> get(uint32_t c, uint32_t slot) const
    {
        Candidate<KW, NI> x;
        if constexpr (KW == 0) {
            x.w = word[0][c][slot];
        } else {
#pragma unroll
            for (int k = 0; k < KW; ++k) x.e[k] = word[k][c][slot];
            x.seed = word[2][c][slot];
        }
        return x;
    }
};

// Columns that are zero after the elimination (sums of others, or empty at the care positions) add nothing to a set: one slice's go behind its
// other columns, whose number, the rank, is returned.  A network of rank 10 with 20 columns has 2^10 sets to try for a
// slice, not 2^20 (300 x 300, 64 x 20, us: 7745 with the zero columns among the others).
template <int KW, int NI>
SQNN_DEV uint32_t gather_columns(Columns<NI> &col, uint32_t slot, uint32_t lane)
{
    Candidate<KW, NI> own{};
    if (lane < NI) own = col.template get<KW>(lane, slot);
    const uint32_t some = __ballot_sync(0xffffffffu, !own.none()), rank = (uint32_t)__popc(some);
    if (some & (some + 1u)) {
        const uint32_t before = (uint32_t)__popc(some & ((1u << lane) - 1u));
        __syncwarp();
        if (lane < NI) col.put((some >> lane) & 1u ? before : rank + lane - before, slot, own);
        __syncwarp();
    }
    return rank;
}

// The whole warp tries all 2^rank sets of columns of one slice: the lanes split them by the top bits.
template <int KW, int NI>
SQNN_DEV uint32_t try_all_sets(const Columns<NI> &col, uint32_t slot, Candidate<KW, NI> x, uint32_t rank, uint32_t lane)
{
    const uint32_t low_bits = rank > 5 ? rank - 5 : 0, lanes_used = rank >= 5 ? 32u : (1u << rank);
    uint32_t best = 0xffffffffu;
    if (lane < lanes_used) {
        for (uint32_t c = low_bits; c < rank; ++c)
            if ((lane >> (c - low_bits)) & 1u) x.add(col.template get<KW>(c, slot));
        const uint32_t count = 1u << low_bits;
        for (uint32_t i = 0; i < count; ++i) {
            if (i != 0) x.add(col.template get<KW>((uint32_t)__ffs((int)i) - 1u, slot));
            best = min(best, x.key());
        }
    }
    return warp_min(best);
}

// The pairs of columns, numbered (1,0), (2,0), (2,1), (3,0), ..: those below column c are the first c (c - 1) / 2.  Lane l looks
// after pairs l, l + 32, ..; `lanes_pairs` holds the larger column of each with the smaller one in its upper half.
template <int NI>
constexpr int PAIRS_PER_LANE = (NI * (NI - 1) / 2 + 31) / 32;
template <int NI>
SQNN_DEV void number_pairs(uint32_t lane, uint32_t (&lanes_pairs)[PAIRS_PER_LANE<NI>])
{
    uint32_t high = 1, before = 0;                                        // pairs before those of `high`
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)PAIRS_PER_LANE<NI>; ++k) {
        while (before + high <= 32 * k + lane) before += high++;
        lanes_pairs[k] = high < NI ? high | (32 * k + lane - before) << 16 : 1u;
    }
}

// The best of all sets of MORE columns below `top` and a pair below those, added to x (`pair`: this lane's pair sums, v: all columns,
// the same in every lane).  The warp walks the columns together, the lanes share the pairs.  The innermost columns are walked
// in straight-line code: a slice that gets here holds up its warp, and a loop over them is all latency.
template <int MORE, int KW, int NI>
SQNN_DEV uint32_t walk_sets(const Columns<NI> &col, uint32_t slot, const Candidate<KW, NI> (&v)[NI], const Candidate<KW, NI> (&pair)[PAIRS_PER_LANE<NI>],
                            const Candidate<KW, NI> &x, uint32_t top, uint32_t lane, uint32_t best)
{
    if constexpr (MORE == 1) {
#pragma unroll
        for (uint32_t c = 2; c < NI; ++c) {
            if (c >= top) break;
            Candidate<KW, NI> y = x;
            y.add(v[c]);
            const uint32_t count = c * (c - 1) / 2;
#pragma unroll
            for (uint32_t k = 0; 32 * k < count; ++k) {
                Candidate<KW, NI> z = y;
                z.add(pair[k]);
                if (32 * k + 32 <= count || 32 * k + lane < count) best = min(best, z.key());
            }
        }
    } else {
#pragma unroll 1
        for (uint32_t c = MORE + 1; c < top; ++c) {
            Candidate<KW, NI> y = x;
            y.add(col.template get<KW>(c, slot));
            best = walk_sets<MORE - 1>(col, slot, v, pair, y, c, lane, best);
        }
    }
    return best;
}

// The whole warp finishes one slice whose best set of at most one column has two errors or more: pairs, then larger sets as
// long as the best count exceeds the sets' size, up to five columns; then all sets.  (Slices far from being consistent, with
// many care bits for their seed bits, go there at once: the next sizes would not decide them.)
template <int KW, int NI>
SQNN_DEV uint32_t try_larger_sets(Columns<NI> &col, uint32_t slot, const uint32_t (&lanes_pairs)[PAIRS_PER_LANE<NI>], const Candidate<KW, NI> &x,
                                  uint32_t best, uint32_t n_in, uint32_t lane)
{
    Candidate<KW, NI> pair[PAIRS_PER_LANE<NI>];
    auto load_pairs = [&] {
#pragma unroll
        for (uint32_t k = 0; k < (uint32_t)PAIRS_PER_LANE<NI>; ++k) {
            pair[k] = col.template get<KW>(lanes_pairs[k] & 0xffffu, slot);
            pair[k].add(col.template get<KW>(lanes_pairs[k] >> 16, slot));
        }
    };
    load_pairs();
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)PAIRS_PER_LANE<NI>; ++k) {
        Candidate<KW, NI> y = x;
        y.add(pair[k]);
        if (32 * k + lane < n_in * (n_in - 1) / 2) best = min(best, y.key());
    }
    best = warp_min(best);
    if ((best >> 20) <= 2u) return best;
    const uint32_t rank = gather_columns<KW>(col, slot, lane);
    if (rank < n_in) load_pairs();
    Candidate<KW, NI> v[NI];
#pragma unroll
    for (int c = 0; c < NI; ++c) v[c] = col.template get<KW>(c, slot);
    best = warp_min(walk_sets<1>(col, slot, v, pair, x, rank, lane, best));
    if ((best >> 20) <= 3u) return best;
    if ((best >> 20) <= 6u) {
        best = warp_min(walk_sets<2>(col, slot, v, pair, x, rank, lane, best));
        if ((best >> 20) <= 4u) return best;
        best = warp_min(walk_sets<3>(col, slot, v, pair, x, rank, lane, best));
        if ((best >> 20) <= 5u) return best;
    }
    return min(best, try_all_sets<KW>(col, slot, x, rank, lane));
}

// A lane's care positions in ascending order.  Up to two words sit in registers, more in the lane's slots of shared memory.
template <int NW>
struct CareBits {
    uint32_t care, want, base, care1, want1;
    const uint32_t *rest;                                                 // care and want of word k: 2 k, 2 k + 1
    // Position of the next care bit, 32 * NW if there is none, and its wanted bit.
    SQNN_DEV uint32_t next(uint32_t &bit)
    {
        if constexpr (NW <= 2) {
            if (care == 0) { care = care1; want = want1; care1 = 0; base = 32 * (NW - 1); }
        } else {
            while (care == 0 && base < 32 * (NW - 1)) {
                base += 32;
                care = rest[(base / 16) * SEARCH_THREADS];
                want = rest[(base / 16 + 1) * SEARCH_THREADS];
            }
        }
        const uint32_t j = (uint32_t)__clz((int)__brev(care));            // 32 for no bit
        bit = __funnelshift_rc(want, 0u, j) & 1u;                        // 0 for no bit
        care &= care - 1u;
        return base + j;
    }
};

// The search over one slice per lane; care bits of a slice fit KW words.  rows_s: byte b of word [w][j] is bit 4 w + b
// of row j of M.  Lanes without a slice have no care bits.
template <int KW, int NI, int NW>
SQNN_DEV uint32_t search_slices(const uint32_t (&rows_s)[(NI + 3) / 4][32 * NW + 1], Columns<NI> &col, const uint32_t (&lanes_pairs)[PAIRS_PER_LANE<NI>],
                                CareBits<NW> bits, uint32_t most, uint32_t n_in, uint32_t lane)
{
    constexpr int NB = (NI + 3) / 4, VW = KW == 0 ? 1 : KW;
    Candidate<KW, NI> v[NI], x{};
#pragma unroll
    for (int c = 0; c < NI; ++c) v[c] = Candidate<KW, NI>{};
#pragma unroll
    for (int k = 0; k < VW; ++k) {
        uint32_t squeezed[NI], wants = 0;
#pragma unroll
        for (int c = 0; c < NI; ++c) squeezed[c] = 0;
#pragma unroll 1
        for (uint32_t byte = 0; byte < 4 && 32 * k + 8 * byte < most; ++byte) {
            uint32_t acc[NB], wanted = 0;
#pragma unroll
            for (int w = 0; w < NB; ++w) acc[w] = 0;
#pragma unroll
            for (uint32_t half = 0; half < 2; ++half) {
                if (half == 1 && 32 * k + 8 * byte + 4 >= most) break;
#pragma unroll
                for (uint32_t i = 4 * half; i < 4 * half + 4; ++i) {
                    uint32_t bit;
                    const uint32_t j = bits.next(bit);
#pragma unroll
                    for (int w = 0; w < NB; ++w) acc[w] += rows_s[w][j] << i;
                    wanted += bit << i;
                }
            }
            wants |= wanted << (8 * byte);
            // byte c % 4 of acc[c / 4] becomes this byte of column c
            const uint32_t keep = 0x3210u & ~(0xfu << (4 * byte));
#pragma unroll
            for (int c = 0; c < NI; ++c) squeezed[c] = __byte_perm(squeezed[c], acc[c / 4], keep | ((4u + c % 4) << (4 * byte)));
        }
        if constexpr (KW == 0) {
            x.w = wants << NI;
#pragma unroll
            for (int c = 0; c < NI; ++c) v[c].w = squeezed[c] << NI;
        } else {
            x.e[k] = wants;
#pragma unroll
            for (int c = 0; c < NI; ++c) v[c].e[k] = squeezed[c];
        }
    }
#pragma unroll
    for (int c = 0; c < NI; ++c) {
        const uint32_t t = (uint32_t)c < n_in ? 1u << c : 0u;
        if constexpr (KW == 0) v[c].w += t;
        else v[c].seed = t;
    }
#pragma unroll
    for (int c = 0; c < NI; ++c) {
        const Candidate<KW, NI> p = v[c].lowest();
        if (x.has(p)) x.add(v[c]);
#pragma unroll
        for (int d = 0; d < NI; ++d)
            if (d != c && v[d].has(p)) v[d].add(v[c]);
    }
    uint32_t best = x.key();
    if (!x.none()) {                                                      // sets of one
#pragma unroll
        for (int c = 0; c < NI; ++c) {
            Candidate<KW, NI> y = x;
            y.add(v[c]);
            best = min(best, y.key());
        }
    }
    const bool open = (best >> 20) >= 2u;
    if (open) {
#pragma unroll
        for (int c = 0; c < NI; ++c) col.put(c, threadIdx.x, v[c]);
    }
    __syncwarp();
    for (uint32_t more = __ballot_sync(0xffffffffu, open); more; more &= more - 1u) {
        const uint32_t src = (uint32_t)__ffs((int)more) - 1u;
        const uint32_t found = try_larger_sets<KW>(col, (threadIdx.x & ~31u) + src, lanes_pairs, x.from(src), __shfl_sync(0xffffffffu, best, src),
                                                   n_in, lane);
        if (lane == src) best = found;
    }
    return best;
}

// NI >= n_in, 32 NW >= n_out.  The loops over columns have a fixed length; a column past n_in is a zero that changes nothing.
// Blocks per SM: what the elimination's 64, 80, 96 or 128 registers allow.  Left to itself the compiler takes 15 more for some and a block
// less is resident (LSTM gates, with five blocks instead of six, 55.6 -> 58.5 us), and 168 to 220 for 20 columns of eight words.
template <int NI, int NW>
__global__ void __launch_bounds__(SEARCH_THREADS, NI <= 8 ? 8 : NI <= 12 ? (NW <= 2 ? 6 : 5) : NI <= 16 && NW <= 2 ? 5 : 4)
k_search_seeds(const __grid_constant__ SearchArgs S)
{
    __shared__ uint32_t rows_s[(NI + 3) / 4][32 * NW + 1];                // rows past n_out are zero
    __shared__ uint32_t cols[SQNN_MAX_N_IN][NW];                          // column t of M as an n_out-bit word
    __shared__ uint32_t rest_s[NW > 2 ? 2 * NW : 1][SEARCH_THREADS];
    __shared__ Columns<NI> col_s;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lanes_pairs[PAIRS_PER_LANE<NI>];
    number_pairs<NI>(lane, lanes_pairs);
    for (uint32_t j = threadIdx.x; j < 32 * NW + 1; j += SEARCH_THREADS) {
        const uint32_t row = j < S.n_out ? row_of(S, j) & (uint32_t)((1ull << S.n_in) - 1ull) : 0u;
#pragma unroll
        for (uint32_t w = 0; w < (NI + 3) / 4; ++w) rows_s[w][j] = (((row >> (4 * w)) & 0xfu) * 0x00204081u) & 0x01010101u;
    }
    for (uint32_t k = threadIdx.x >> 5; k < NW; k += SEARCH_THREADS / 32) {
        const uint32_t row = 32 * k + lane < S.n_out ? row_of(S, 32 * k + lane) : 0u;
        for (uint32_t t = 0; t < S.n_in; ++t) {
            const uint32_t word = __ballot_sync(0xffffffffu, (row >> t) & 1u);
            if (lane == 0) cols[t][k] = word;
        }
    }
    __syncthreads();
    wait_prior_grid();
    launch_dependents();
    const uint64_t total = S.slices * S.n_q;
    const uint64_t step = (uint64_t)gridDim.x * SEARCH_THREADS;
    for (uint64_t job0 = (uint64_t)blockIdx.x * SEARCH_THREADS + (threadIdx.x & ~31u); job0 < total; job0 += step) {
        const uint64_t job = job0 + lane;
        const bool live = job < total;
        uint32_t want[NW], care[NW], count = 0;
#pragma unroll
        for (int k = 0; k < NW; ++k) want[k] = care[k] = 0;
        if (live) {
            uint64_t slice = job;
            const uint64_t *plane = S.planes;
            while (slice >= S.slices) { slice -= S.slices; plane += S.words64; }
            const uint64_t p0 = slice * S.n_out;
            load_bits<NW>(S.mask, 2 * S.words64, p0, care);
            load_bits<NW>(plane, 2 * S.words64, p0, want);
            const uint32_t bits = S.mn - p0 < S.n_out ? (uint32_t)(S.mn - p0) : S.n_out;        // the last slice may be shorter
#pragma unroll
            for (uint32_t k = 0; k < NW; ++k)
                if (bits < 32 * k + 32) care[k] &= bits > 32 * k ? (1u << (bits - 32 * k)) - 1u : 0u;
        }
#pragma unroll
        for (int k = 0; k < NW; ++k) count += (uint32_t)__popc(care[k]);
        const bool wide = count > MAX_CARE;
        CareBits<NW> bits{wide ? 0u : care[0], want[0], 0u, 0u, 0u, nullptr};
        if constexpr (NW == 2) { bits.care1 = wide ? 0u : care[1]; bits.want1 = want[1]; }
        if constexpr (NW > 2) {
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                rest_s[2 * k][threadIdx.x] = wide ? 0u : care[k];
                rest_s[2 * k + 1][threadIdx.x] = want[k];
            }
            bits.rest = &rest_s[0][threadIdx.x];
        }
        const uint32_t most = __reduce_max_sync(0xffffffffu, wide ? 0u : count);
        uint32_t best = most + NI <= 32 ? search_slices<0, NI, NW>(rows_s, col_s, lanes_pairs, bits, most, S.n_in, lane)
                        : most <= 32    ? search_slices<1, NI, NW>(rows_s, col_s, lanes_pairs, bits, most, S.n_in, lane)
                                        : search_slices<2, NI, NW>(rows_s, col_s, lanes_pairs, bits, most, S.n_in, lane);
        for (uint32_t more = __ballot_sync(0xffffffffu, wide); more; more &= more - 1u) {
            const uint32_t src = (uint32_t)__ffs((int)more) - 1u;
            uint32_t w_s[NW], c_s[NW];
#pragma unroll
            for (int k = 0; k < NW; ++k) { w_s[k] = __shfl_sync(0xffffffffu, want[k], src); c_s[k] = __shfl_sync(0xffffffffu, care[k], src); }
            const uint32_t found = try_all_seeds<NW>(cols, S.n_in, w_s, c_s, lane);
            if (lane == src) best = found;
        }
        if (live) {
            S.wc[job] = best & 0xfffffu;
            S.np[job] = (uint16_t)(best >> 20);
        }
        __syncwarp();
    }
}

template <int NI>
int launch_search(const SearchArgs &S, uint32_t blocks, cudaStream_t st)
{
    const uint32_t nw = (S.n_out + 31) / 32;
    auto k = nw <= 1 ? k_search_seeds<NI, 1> : nw <= 2 ? k_search_seeds<NI, 2> : nw <= 4 ? k_search_seeds<NI, 4> : k_search_seeds<NI, 8>;
    return launch_kernel(k, blocks, SEARCH_THREADS, 0, st, S);
}

}  // namespace

}  // namespace sqnn

static int search_seeds_queue(const sqnn_xornet *net, uint64_t m, uint64_t n, uint32_t n_q,
                              const uint64_t *d_planes, const uint64_t *d_mask, uint32_t *d_wc,
                              uint16_t *d_np, void *cuda_stream)
{
    using namespace sqnn;
    if (!net || !net->rows || !d_planes || !d_mask || !d_wc || !d_np) return SQNN_E_INVALID_ARG;
    if (net->n_out < 1 || net->n_out > SQNN_MAX_N_OUT || net->n_in < 1 || net->n_in > SQNN_MAX_N_IN ||
        n_q < 1 || n_q > SQNN_MAX_PLANES || m == 0 || n == 0 || m > ((uint64_t)1 << 40) / n)
        return SQNN_E_INVALID_ARG;
    if (net->n_in > 20) return SQNN_E_UNSUPPORTED;          // 2^n_in seeds per slice
    SearchArgs S;
    for (uint32_t j = 0; j < SQNN_MAX_N_OUT; ++j) S.rows[j] = j < net->n_out ? net->rows[j] : 0u;
    S.n_out = net->n_out; S.n_in = net->n_in; S.n_q = n_q;
    S.mn = m * n;
    S.words64 = (S.mn + 63) / 64;
    S.slices = (S.mn + net->n_out - 1) / net->n_out;
    S.planes = d_planes; S.mask = d_mask; S.wc = d_wc; S.np = d_np;
    const uint64_t jobs = S.slices * n_q;
    uint64_t blocks = (jobs + SEARCH_THREADS - 1) / SEARCH_THREADS;
    const uint64_t cap = (uint64_t)sm_count() * 16;         // about twice what is resident: few tables, an even end
    if (blocks > cap) blocks = cap;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    return net->n_in <= 8    ? launch_search<8>(S, (uint32_t)blocks, st)
           : net->n_in <= 12 ? launch_search<12>(S, (uint32_t)blocks, st)
           : net->n_in <= 16 ? launch_search<16>(S, (uint32_t)blocks, st)
                             : launch_search<20>(S, (uint32_t)blocks, st);
}

extern "C" int sqnn_search_seeds(const sqnn_xornet *net, uint64_t m, uint64_t n, uint32_t n_q,
                                 const uint64_t *d_planes, const uint64_t *d_mask, uint32_t *d_wc,
                                 uint16_t *d_np, void *cuda_stream)
{
    sqnn::ApiScope scope("sqnn_search_seeds");
    return scope.finish(search_seeds_queue(net, m, n, n_q, d_planes, d_mask, d_wc, d_np, cuda_stream), nullptr,
                        (cudaStream_t)cuda_stream);
}
