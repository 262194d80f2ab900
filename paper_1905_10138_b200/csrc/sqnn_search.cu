// Exhaustive seed search on the device (Section 5.2): for every slice of every plane the seed with the fewest
// wrong care bits among all 2^n_in is found (the smallest seed among equals).
//
// The seeds are not tried one by one.  Let r_j be the rows of M at the slice's care positions and b_j the
// wanted bits.  Elimination in ascending position makes some rows pivots (r of them, r = the rank); every
// other row is the sum of pivot rows in a known subset.  A seed is then a choice of the set e of pivots it
// gets wrong: which dependent rows are wrong follows (their syndrome s plus the columns C_i of the pivots in
// e), and so does the smallest seed with exactly these errors: the one with all free variables 0 when every
// pivot column is the lowest possible one, which is linear in the pivots' bits (columns Q_i).  So with
// V_i = C_i << 20 | Q_i the search is
//
//     min over e of  (|e| + |C part|) << 20 | Q part,   V(e) = V_0 ^ xor of V_i, i in e,
//
// and e can be taken in the order of its size: once the best count is B, sizes above B cannot matter.  Almost
// all slices are done after sizes 0 (consistent: no wrong bit), 1 and 2: about 80 candidates for r = 12
// instead of 4096.  One thread per slice does that much; slices that need larger sets are finished by the whole
// warp: sets of three (which decide nearly all of them), then all 2^r sets in Gray-code order; slices with more
// dependent rows than C has bits for by trying all seeds.
//
// Bound: integer instructions.  600 000 slices of 60 x 12 (20 % care bits, two planes of 6000 x 3000) take 127 us, 79 M
// warp instructions with 18.5 of 32 lanes active: the loop over a slice's care bits takes as many turns as the lane with
// the most of them needs.  (Trying all 2^12 seeds of every slice took 2540 us.)
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

// 32 bits of a packed vector starting at position p; positions >= limit (<= vector length) read 0
SQNN_DEV uint32_t bits32_at(const uint64_t *__restrict__ v, uint64_t p, uint64_t limit)
{
    if (p >= limit) return 0u;
    const uint64_t w = p >> 6;
    const uint32_t sh = (uint32_t)(p & 63);
    uint64_t x = __ldg(v + w) >> sh;
    if (sh > 32 && limit > ((w + 1) << 6)) x |= __ldg(v + w + 1) << (64 - sh);   // next word holds wanted positions
    uint32_t r = (uint32_t)x;
    if (p + 32 > limit) r &= (1u << (uint32_t)(limit - p)) - 1u;
    return r;
}

constexpr uint32_t SEARCH_THREADS = 128;
constexpr uint32_t MAX_DEP = 32;                          // dependent rows a word C has room for

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

// A candidate's key: number of wrong care bits, then the seed.
SQNN_DEV uint32_t set_key(uint32_t size, uint32_t c, uint32_t q) { return ((size + (uint32_t)__popc(c)) << 20) + q; }

// The whole warp tries all 2^r sets of wrong pivots of one slice (v: its (C_i, Q_i), one every SEARCH_THREADS).
SQNN_DEV uint32_t try_all_sets(const uint2 *v, uint2 v0, uint32_t r, uint32_t lane)
{
    const uint32_t low_bits = r > 5 ? r - 5 : 0, lanes_used = r >= 5 ? 32u : (1u << r);
    uint32_t best = 0xffffffffu;
    if (lane < lanes_used) {
        const uint32_t top = lane << low_bits, size0 = (uint32_t)__popc(lane);
        uint32_t c = v0.x, q = v0.y;
        for (uint32_t t = low_bits; t < r; ++t)
            if ((top >> t) & 1u) { c ^= v[t * SEARCH_THREADS].x; q ^= v[t * SEARCH_THREADS].y; }
        const uint32_t count = 1u << low_bits;
        for (uint32_t i = 0; i < count; ++i) {
            if (i != 0) {
                const uint2 w = v[((uint32_t)__ffs((int)i) - 1u) * SEARCH_THREADS];
                c ^= w.x;
                q ^= w.y;
            }
            best = min(best, set_key(size0 + (uint32_t)__popc(i ^ (i >> 1)), c, q));
        }
    }
    return warp_min(best);
}

// The whole warp tries all sets of three wrong pivots: the lanes split the pairs, each walks the third.
SQNN_DEV uint32_t try_triples(const uint2 *v, uint2 v0, uint32_t r, uint32_t lane)
{
    uint32_t best = 0xffffffffu;
    for (uint32_t p = lane; p < r * (r - 1) / 2; p += 32) {
        const uint32_t i = (uint32_t)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f), h = p - i * (i - 1) / 2;     // h < i
        const uint2 a = v[i * SEARCH_THREADS], b = v[h * SEARCH_THREADS];
        const uint32_t c = v0.x ^ a.x ^ b.x, q = v0.y ^ a.y ^ b.y;
        for (uint32_t g = 0; g < h; ++g) {
            const uint2 w = v[g * SEARCH_THREADS];
            best = min(best, set_key(3u, c ^ w.x, q ^ w.y));
        }
    }
    return warp_min(best);
}

// NI >= n_in.  Rows and bookkeeping of the elimination sit in registers; every loop over columns or pivots has a
// fixed length, and a column without a pivot row or a pivot that does not exist is a zero that changes nothing
// (a set with such a pivot only counts one error more than the set without it), so that the lanes of a warp,
// which have different numbers of care bits and pivots, stay together.
template <int NI, int NW>
__global__ void __launch_bounds__(SEARCH_THREADS)
k_search_seeds(const __grid_constant__ SearchArgs S)
{
    __shared__ uint32_t rows_s[SQNN_MAX_N_OUT];
    __shared__ uint32_t cols[SQNN_MAX_N_IN][NW];                          // column t of M as an n_out-bit word
    __shared__ uint2 v_s[NI][SEARCH_THREADS];
    wait_prior_grid();
    launch_dependents();
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t j = threadIdx.x; j < SQNN_MAX_N_OUT; j += SEARCH_THREADS) rows_s[j] = S.rows[j] & (uint32_t)((1ull << S.n_in) - 1ull);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < S.n_in * NW; i += SEARCH_THREADS) {
        const uint32_t t = i / NW, k = i % NW;
        uint32_t w = 0;
        for (uint32_t j = 32 * k; j < S.n_out && j < 32 * k + 32; ++j) w |= ((rows_s[j] >> t) & 1u) << (j - 32 * k);
        cols[t][k] = w;
    }
    __syncthreads();
    const uint64_t total = S.slices * S.n_q;
    const uint64_t step = (uint64_t)gridDim.x * SEARCH_THREADS;
    for (uint64_t job0 = (uint64_t)blockIdx.x * SEARCH_THREADS + (threadIdx.x & ~31u); job0 < total; job0 += step) {
        const uint64_t job = job0 + lane;
        const bool live = job < total;
        uint32_t want[NW], care[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) want[k] = care[k] = 0;
        if (live) {
            const uint32_t plane = (uint32_t)(job / S.slices);
            const uint64_t p0 = (job - (uint64_t)plane * S.slices) * S.n_out;
            const uint64_t limit = p0 + S.n_out < S.mn ? p0 + S.n_out : S.mn;   // slice end (ragged tail)
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                if (32u * k >= S.n_out) break;
                care[k] = bits32_at(S.mask, p0 + 32 * k, limit);
                want[k] = bits32_at(S.planes + (uint64_t)plane * S.words64, p0 + 32 * k, limit);
            }
        }
        // elimination: row[c] = the pivot row whose lowest set column is c, sub[c] = the original pivots it is the
        // sum of (numbered as they come), bits = the original pivots' wanted bits, dc[i] = C_i
        uint32_t row[NI], sub[NI], dc[NI], bits = 0, r = 0, dep = 0, syn = 0;
#pragma unroll
        for (int c = 0; c < NI; ++c) row[c] = sub[c] = dc[c] = 0;
#pragma unroll
        for (int k = 0; k < NW; k += 2) {
            unsigned long long left = care[k], wanted = want[k];
            if (k + 1 < NW) {
                left |= (unsigned long long)care[k + 1 < NW ? k + 1 : k] << 32;
                wanted |= (unsigned long long)want[k + 1 < NW ? k + 1 : k] << 32;
            }
            while (left) {
                const uint32_t j = (uint32_t)__ffsll((long long)left) - 1u;
                left &= left - 1ull;
                uint32_t a = rows_s[32 * k + j], of = 0;
                const uint32_t b = (uint32_t)(wanted >> j) & 1u;
#pragma unroll
                for (int c = 0; c < NI; ++c)
                    if ((a >> c) & 1u) { a ^= row[c]; of ^= sub[c]; }
                if (a) {                                                  // a new pivot
                    const uint32_t low = a & (0u - a);
                    of |= 1u << r;
#pragma unroll
                    for (int c = 0; c < NI; ++c)
                        if (low == (1u << c)) { row[c] = a; sub[c] = of; }
                    bits |= b << r;
                    ++r;
                } else {                                                  // the sum of the pivots in `of`
                    const uint32_t bit = dep < MAX_DEP ? 1u << dep : 0u;
                    if ((b ^ (uint32_t)__popc(bits & of)) & 1u) syn |= bit;
#pragma unroll
                    for (int i = 0; i < NI; ++i)
                        if ((of >> i) & 1u) dc[i] |= bit;
                    ++dep;
                }
            }
        }
        // reduced form: no pivot row contains another pivot's column
#pragma unroll
        for (int c = NI - 2; c >= 0; --c) {
#pragma unroll
            for (int d = c + 1; d < NI; ++d)
                if ((row[c] >> d) & 1u) { row[c] ^= row[d]; sub[c] ^= sub[d]; }
        }
        uint32_t seed = 0;
#pragma unroll
        for (int c = 0; c < NI; ++c) seed |= ((uint32_t)__popc(bits & sub[c]) & 1u) << c;
        uint32_t best = set_key(0u, syn, seed);
        const bool wide = live && dep > MAX_DEP;
        if (syn != 0 && !wide) {
            uint32_t dq[NI];                                              // Q_i
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                dq[i] = 0;
#pragma unroll
                for (int c = 0; c < NI; ++c) dq[i] |= ((sub[c] >> i) & 1u) << c;
                best = min(best, set_key(1u, syn ^ dc[i], seed ^ dq[i])); // one wrong pivot
            }
            if ((best >> 20) >= 2) {
#pragma unroll
                for (int i = 1; i < NI; ++i) {                            // two
                    const uint32_t c = syn ^ dc[i], q = seed ^ dq[i];
#pragma unroll
                    for (int h = 0; h < i; ++h) best = min(best, set_key(2u, c ^ dc[h], q ^ dq[h]));
                }
            }
            if ((best >> 20) > 2u) {
#pragma unroll
                for (int i = 0; i < NI; ++i) v_s[i][threadIdx.x] = make_uint2(dc[i], dq[i]);
            }
        }
        __syncwarp();
        // what is left for the whole warp: larger sets could still win or tie, or C has no room
        uint32_t more = __ballot_sync(0xffffffffu, wide || (live && syn != 0 && (best >> 20) > 2u));
        while (more) {
            const uint32_t src = (uint32_t)__ffs((int)more) - 1u;
            more &= more - 1u;
            uint32_t found;
            if (__shfl_sync(0xffffffffu, wide ? 1u : 0u, src)) {
                uint32_t w_s[NW], c_s[NW];
#pragma unroll
                for (int k = 0; k < NW; ++k) { w_s[k] = __shfl_sync(0xffffffffu, want[k], src); c_s[k] = __shfl_sync(0xffffffffu, care[k], src); }
                found = try_all_seeds<NW>(cols, S.n_in, w_s, c_s, lane);
            } else {
                const uint2 *v = &v_s[0][(threadIdx.x & ~31u) + src];
                const uint2 v0 = make_uint2(__shfl_sync(0xffffffffu, syn, src), __shfl_sync(0xffffffffu, seed, src));
                const uint32_t r_src = __shfl_sync(0xffffffffu, r, src);
                found = min(__shfl_sync(0xffffffffu, best, src), try_triples(v, v0, r_src, lane));
                if ((found >> 20) > 3u) found = try_all_sets(v, v0, r_src, lane);
            }
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
    const uint64_t cap = (uint64_t)sm_count() * 64;
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
