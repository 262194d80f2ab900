// Host side of the library: encryption of slices (Algorithm 1 / exhaustive search), the
// packed blob format, its validation and size accounting.  No CUDA in this file.
#include "sqnn.h"
#include "sqnn_blob.h"
#include "sqnn_layout.h"

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

namespace {

inline int popc64(uint64_t v) { return __builtin_popcountll(v); }
inline int ctz32(uint32_t v) { return __builtin_ctz(v); }

// `count` (<= 64) bits of a packed vector starting at flat position p; positions >= limit read 0.
inline uint64_t window(const uint64_t *words, uint64_t p, uint32_t count, uint64_t limit)
{
    if (p >= limit) return 0;
    if (p + count > limit) count = (uint32_t)(limit - p);
    const uint64_t w = p >> 6;
    const uint32_t sh = (uint32_t)(p & 63);
    uint64_t v = words[w] >> sh;
    if (sh && sh + count > 64) v |= words[w + 1] << (64 - sh);
    if (count < 64) v &= ((uint64_t)1 << count) - 1;
    return v;
}

inline uint32_t ceil_lg_u64(uint64_t v)   // smallest e with 2^e >= v (0 for v <= 1)
{
    uint32_t e = 0;
    while (((uint64_t)1 << e) < v) ++e;
    return e;
}

struct SliceBits {            // wanted bits and care flags of one slice, n_out <= 256
    uint64_t want[4];
    uint64_t care[4];
};

inline void load_slice(const uint64_t *plane, const uint64_t *mask, uint64_t mn, uint32_t n_out,
                       uint64_t s, SliceBits &sb)
{
    const uint64_t p0 = s * (uint64_t)n_out;
    for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t lo = k * 64;
        if (lo >= n_out) { sb.want[k] = sb.care[k] = 0; continue; }
        const uint32_t cnt = std::min<uint32_t>(64, n_out - lo);
        sb.care[k] = window(mask, p0 + lo, cnt, mn);
        sb.want[k] = window(plane, p0 + lo, cnt, mn);
    }
}

// w~ = M . w^c over GF(2) by table: the seed is cut into bytes, an entry is the XOR of the columns of M its byte
// selects.  (Taking the parity of every row with the seed was four fifths of the encoder's time.)
struct Expander {
    uint32_t words, bytes;
    std::vector<uint64_t> tab;                            // [byte][value][words]
    Expander(const uint32_t *rows, uint32_t n_out, uint32_t n_in)
        : words((n_out + 63) / 64), bytes((n_in + 7) / 8), tab((size_t)bytes * 256 * words, 0)
    {
        for (uint32_t t = 0; t < n_in; ++t) {             // the columns first: entries with one bit
            uint64_t *e = &tab[((size_t)(t >> 3) * 256 + (1u << (t & 7))) * words];
            for (uint32_t j = 0; j < n_out; ++j) e[j >> 6] |= (uint64_t)((rows[j] >> t) & 1) << (j & 63);
        }
        for (uint32_t b = 0; b < bytes; ++b)
            for (uint32_t v = 1; v < 256; ++v)
                if (v & (v - 1)) {
                    uint64_t *e = &tab[((size_t)b * 256 + v) * words];
                    const uint64_t *x = &tab[((size_t)b * 256 + (v & (v - 1))) * words], *y = &tab[((size_t)b * 256 + (v & (0u - v))) * words];
                    for (uint32_t k = 0; k < words; ++k) e[k] = x[k] ^ y[k];
                }
    }
    void operator()(uint32_t seed, uint64_t out[4]) const
    {
        out[0] = out[1] = out[2] = out[3] = 0;
        for (uint32_t b = 0; b < bytes; ++b, seed >>= 8) {
            const uint64_t *e = &tab[((size_t)b * 256 + (seed & 255u)) * words];
            for (uint32_t k = 0; k < words; ++k) out[k] ^= e[k];
        }
    }
};

// Algorithm 1 on eight slices at once, one per vector lane.  Care rows are appended in ascending position to a
// system kept in echelon form (a row's pivot is its lowest set column): a new row is reduced by the pivot row of
// every column in turn (zero where there is none) and what is left is kept at its lowest column; a row that
// reduces to 0 = 1 is the unsolvable case and is dropped (it will show up as a patch), one that reduces to 0 = 0 is
// redundant.  Free variables are 0, so the pivot variables follow from the highest column down.  (One slice at a
// time, with a branch for every reduction, spent most of its time on mispredicted branches: encoding 378 000 slices of
// 100 x 10 took 4.6 ms on 16 cores, and takes 2.5 ms this way.)
constexpr uint32_t LANES = 8;
typedef uint32_t Vec __attribute__((vector_size(4 * LANES)));
typedef int32_t SignedVec __attribute__((vector_size(4 * LANES)));

#if defined(__x86_64__) && defined(__GNUC__) && !defined(__clang__) && !defined(__SANITIZE_ADDRESS__) && !defined(__SANITIZE_THREAD__)
__attribute__((target_clones("avx2", "default")))
#endif
void encode_alg1_block(const uint32_t *rows, uint32_t n_out, uint32_t n_in, const SliceBits *sb, uint32_t *seeds)
{
    Vec piv[SQNN_MAX_N_IN], rhs[SQNN_MAX_N_IN];           // pivot rows by column; right-hand sides: all ones or zero
    for (uint32_t c = 0; c < n_in; ++c) piv[c] = rhs[c] = Vec{};
    for (uint32_t k = 0; k * 64 < n_out; ++k) {
        uint64_t left[LANES], any = 0;
        for (uint32_t e = 0; e < LANES; ++e) any |= left[e] = sb[e].care[k];
        while (any) {
            Vec a, b;
            any = 0;
            for (uint32_t e = 0; e < LANES; ++e) {
                const uint32_t j = left[e] ? (uint32_t)__builtin_ctzll(left[e]) : 0u;
                a[e] = left[e] ? rows[k * 64 + j] : 0u;
                b[e] = 0u - (uint32_t)((sb[e].want[k] >> j) & 1);
                any |= left[e] &= left[e] - (left[e] != 0);
            }
            for (uint32_t c = 0; c < n_in; ++c) {
                const Vec set = (Vec)((SignedVec)(a << (31 - c)) >> 31);      // all ones where column c is set
                a ^= piv[c] & set;
                b ^= rhs[c] & set;
            }
            const Vec low = a & -a;
            for (uint32_t c = 0; c < n_in; ++c) {
                const Vec here = (Vec)((SignedVec)(low << (31 - c)) >> 31);
                piv[c] |= a & here;
                rhs[c] |= b & here;
            }
        }
    }
    Vec seed = Vec{};
    for (uint32_t c = n_in; c-- > 0;) {
        Vec x = piv[c] & seed;                            // (columns above c)
        x ^= x >> 16; x ^= x >> 8; x ^= x >> 4; x ^= x >> 2; x ^= x >> 1;
        seed |= (((x ^ rhs[c]) & (piv[c] >> c)) & 1u) << c;
    }
    for (uint32_t e = 0; e < LANES; ++e) seeds[e] = seed[e];
}

// All 2^n_in outputs of the network, 4 words each.
void build_outputs(const uint32_t *rows, uint32_t n_out, uint32_t n_in, std::vector<uint64_t> &tab)
{
    const uint64_t cnt = (uint64_t)1 << n_in;
    const Expander expand(rows, n_out, n_in);
    tab.assign(cnt * 4, 0);
    for (uint64_t v = 0; v < cnt; ++v) expand((uint32_t)v, &tab[v * 4]);
}

inline uint32_t encode_exhaustive(const std::vector<uint64_t> &tab, uint32_t n_in, const SliceBits &sb)
{
    const uint64_t cnt = (uint64_t)1 << n_in;
    uint32_t best = 0;
    int best_wrong = 1 << 30;
    for (uint64_t v = 0; v < cnt; ++v) {
        const uint64_t *o = &tab[v * 4];
        int wrong = 0;
        for (int k = 0; k < 4; ++k) wrong += popc64((o[k] ^ sb.want[k]) & sb.care[k]);
        if (wrong < best_wrong) { best_wrong = wrong; best = (uint32_t)v; }
    }
    return best;
}

struct PlaneArrays {
    std::vector<uint32_t> wc;
    std::vector<uint16_t> np;
};

uint64_t round_up(uint64_t v, uint64_t a) { return (v + a - 1) / a * a; }

// Packs bit fields of `width` bits (value i at bits [i*width, (i+1)*width)) into uint32 words.
// Groups of 32 values fill whole words, so groups can be written independently.
template <typename T>
void pack_fields(const T *vals, uint64_t count, uint32_t width, uint32_t *dst)
{
    if (width == 0) return;
    const int64_t groups = (int64_t)((count + 31) / 32);
#pragma omp parallel for schedule(static) if (count >= 8192)
    for (int64_t g = 0; g < groups; ++g) {
        uint32_t *w = dst + (uint64_t)g * width;
        uint64_t acc = 0;
        uint32_t have = 0, wi = 0;
        const uint64_t lo = (uint64_t)g * 32, hi = std::min<uint64_t>(count, lo + 32);
        for (uint64_t i = lo; i < hi; ++i) {
            acc |= (uint64_t)vals[i] << have;
            have += width;
            while (have >= 32) { w[wi++] = (uint32_t)acc; acc >>= 32; have -= 32; }
        }
        if (have) w[wi] = (uint32_t)acc;
    }
}

inline uint32_t read_field(const uint32_t *src, uint64_t index, uint32_t width)
{
    if (width == 0) return 0;
    const uint64_t bit = index * width;
    const uint64_t w = bit >> 5;
    const uint32_t sh = (uint32_t)(bit & 31);
    uint64_t v = (uint64_t)src[w] | ((uint64_t)src[w + 1] << 32);   // sections end with slack
    return (uint32_t)((v >> sh) & (((uint64_t)1 << width) - 1));
}

// The lookup tables of the network in the layout the kernels index (sqnn_layout.h).
void build_tables(const uint32_t *rows, uint32_t n_out, uint32_t n_in, uint32_t *tab)
{
    const uint32_t nwp = sqnn::entry_words_padded(n_out);
    const uint32_t nch = sqnn::table_chunks(n_in, nwp), cb = sqnn::chunk_bits(n_in, nwp);
    std::memset(tab, 0, (size_t)sqnn::table_words(n_out, n_in) * 4);
    for (uint32_t ch = 0; ch < nch; ++ch)
        for (uint32_t v = 1; v < (1u << cb); ++v) {
            uint32_t *e = tab + (size_t)(((ch << cb) | v)) * nwp;
            if (v & (v - 1)) {                            // the sum of two entries made before it
                const uint32_t *x = tab + (size_t)((ch << cb) | (v & (v - 1))) * nwp, *y = tab + (size_t)((ch << cb) | (v & (0u - v))) * nwp;
                for (uint32_t k = 0; k < nwp; ++k) e[k] = x[k] ^ y[k];
                continue;
            }
            const uint32_t t = ch * cb + (uint32_t)ctz32(v);           // one column of M; bits past n_in select none
            if (t < n_in)
                for (uint32_t j = 0; j < n_out; ++j) e[j >> 5] |= ((rows[j] >> t) & 1u) << (j & 31);
        }
}

// Section offsets of a device blob for the given patch totals.
void plan_blob(uint64_t m, uint64_t n, uint32_t n_q, uint32_t n_out, uint32_t n_in, const uint64_t *n_pp, sqnn_desc *out)
{
    sqnn_desc d;
    std::memset(&d, 0, sizeof d);
    const uint64_t mn = m * n;
    const uint64_t l = (mn + n_out - 1) / n_out;
    const uint64_t lp = round_up(l, SQNN_PAD_SLICES);
    d.m = m; d.n = n; d.slices = l; d.slices_padded = lp;
    d.n_q = n_q; d.n_out = n_out; d.n_in = n_in; d.tile_slices = SQNN_TILE_SLICES;
    d.tab_entry_words = sqnn::entry_words_padded(n_out);
    d.tab_chunks = sqnn::table_chunks(n_in, d.tab_entry_words);
    d.tab_chunk_bits = sqnn::chunk_bits(n_in, d.tab_entry_words);
    uint64_t off = SQNN_BLOB_HEADER_BYTES;
    d.off_xornet = off;
    off += round_up((uint64_t)n_out * 4, 16) + 16;
    d.off_tables = off;
    d.tables_bytes = (uint64_t)sqnn::table_words(n_out, n_in) * 4;
    off += round_up(d.tables_bytes, 16) + 16;
    for (uint32_t i = 0; i < n_q; ++i) {
        d.n_pp[i] = n_pp[i];
        d.off_wc[i] = off;  off += round_up(lp * n_in / 8, 16) + 16;
        d.off_idx[i] = off; off += round_up((lp / SQNN_TILE_SLICES + 1) * 4, 16) + 16;
        d.off_pp[i] = off;  off += round_up(n_pp[i] * 2, 16) + 16;
    }
    d.total_bytes = off;
    *out = d;
}

// Host loops over slices or tiles run in parallel from this many slices on (below it a thread team costs more
// than it saves).
constexpr uint64_t PARALLEL_FROM = 8192;

// Allocates a blob for the given patch totals: header, rows of M and tables in place, streams zero.
uint8_t *start_blob(const sqnn_xornet *net, uint64_t m, uint64_t n, uint32_t n_q, const uint64_t *n_pp, sqnn_desc *d)
{
    plan_blob(m, n, n_q, net->n_out, net->n_in, n_pp, d);
    uint8_t *b = (uint8_t *)std::calloc(d->total_bytes, 1);
    if (!b) return nullptr;
    sqnn_blob_header *h = (sqnn_blob_header *)b;
    std::memcpy(h->magic, SQNN_BLOB_MAGIC, 8);
    h->version = SQNN_BLOB_VERSION;
    h->header_bytes = SQNN_BLOB_HEADER_BYTES;
    h->desc = *d;
    std::memcpy(b + d->off_xornet, net->rows, (size_t)net->n_out * 4);
    build_tables(net->rows, net->n_out, net->n_in, (uint32_t *)(b + d->off_tables));
    return b;
}

int build_blob(const sqnn_xornet *net, uint64_t m, uint64_t n, uint32_t n_q,
               const uint32_t *const *wc, const uint16_t *const *np, const uint16_t *const *dp, void **blob, size_t *blob_bytes)
{
    const uint64_t mn = m * n;
    const uint32_t n_out = net->n_out, n_in = net->n_in;
    const uint64_t l = (mn + n_out - 1) / n_out;
    const int64_t tiles = (int64_t)((l + SQNN_TILE_SLICES - 1) / SQNN_TILE_SLICES);
    const bool par = l >= PARALLEL_FROM;
    uint64_t n_pp[SQNN_MAX_PLANES] = {0};
    std::vector<std::vector<uint64_t>> first(n_q, std::vector<uint64_t>((size_t)tiles + 1));   // entries before each tile
    int bad = 0;
    for (uint32_t i = 0; i < n_q; ++i) {
#pragma omp parallel for schedule(static) if (par) reduction(| : bad)
        for (int64_t t = 0; t < tiles; ++t) {
            const uint64_t lo = (uint64_t)t * SQNN_TILE_SLICES, hi = std::min<uint64_t>(l, lo + SQNN_TILE_SLICES);
            uint64_t sum = 0;
            for (uint64_t s = lo; s < hi; ++s) {
                bad |= np[i][s] > n_out;
                bad |= n_in < 32 && (wc[i][s] >> n_in) != 0;
                sum += np[i][s];
            }
            first[i][(size_t)t + 1] = sum;
        }
        if (bad) return SQNN_E_INVALID_ARG;
        for (int64_t t = 0; t < tiles; ++t) first[i][(size_t)t + 1] += first[i][(size_t)t];
        n_pp[i] = first[i][(size_t)tiles];
        if (n_pp[i] > 0xffffffffull) return SQNN_E_INVALID_ARG;
    }
    sqnn_desc d;
    uint8_t *b = start_blob(net, m, n, n_q, n_pp, &d);
    if (!b) return SQNN_E_NOMEM;
    for (uint32_t i = 0; i < n_q; ++i) {
        pack_fields(wc[i], l, n_in, (uint32_t *)(b + d.off_wc[i]));
        uint32_t *idx = (uint32_t *)(b + d.off_idx[i]);
        uint16_t *dst = (uint16_t *)(b + d.off_pp[i]);
        for (uint64_t t = 0; t <= d.slices_padded / SQNN_TILE_SLICES; ++t) idx[t] = (uint32_t)first[i][std::min<uint64_t>(t, (uint64_t)tiles)];
#pragma omp parallel for schedule(static) if (par) reduction(| : bad)
        for (int64_t t = 0; t < tiles; ++t) {
            const uint64_t lo = (uint64_t)t * SQNN_TILE_SLICES, hi = std::min<uint64_t>(l, lo + SQNN_TILE_SLICES);
            uint64_t run = first[i][(size_t)t];
            for (uint64_t s = lo; s < hi; ++s) {
                int64_t prev = -1;
                for (uint32_t k = 0; k < np[i][s]; ++k, ++run) {
                    const uint32_t pos = dp[i][run];
                    // positions inside a slice ascend strictly; the last slice holds real positions only
                    bad |= pos >= n_out || (int64_t)pos <= prev || s * n_out + pos >= mn;
                    prev = pos;
                    dst[run] = (uint16_t)((s - lo) * n_out + pos);
                }
            }
        }
        if (bad) { std::free(b); return SQNN_E_INVALID_ARG; }
    }
    *blob = b;
    *blob_bytes = d.total_bytes;
    return SQNN_OK;
}

bool net_ok(const sqnn_xornet *net)
{
    return net && net->rows && net->n_out >= 1 && net->n_out <= SQNN_MAX_N_OUT &&
           net->n_in >= 1 && net->n_in <= SQNN_MAX_N_IN;
}

}  // namespace

extern "C" {

void sqnn_free(void *p) { std::free(p); }

const char *sqnn_status_string(int status)
{
    switch (status) {
        case SQNN_OK: return "ok";
        case SQNN_E_INVALID_ARG: return "invalid argument";
        case SQNN_E_BAD_BLOB: return "malformed blob";
        case SQNN_E_UNSUPPORTED: return "unsupported";
        case SQNN_E_NOMEM: return "out of host memory";
        case SQNN_E_CUDA: return "CUDA runtime error";
        case SQNN_E_TIMEOUT: return "device-side wait timed out";
        case SQNN_E_WORKSPACE: return "workspace missing or too small";
        default: return "unknown status";
    }
}

// Size accounting from the totals of a layer: hist over all planes, sum and max of n_patch per plane.
static void fill_stats(const sqnn_desc &d, const uint64_t *sum, const uint32_t *maxp, const uint64_t *hist, sqnn_stats *stats)
{
    std::memset(stats, 0, sizeof *stats);
    const uint64_t mn = d.m * d.n, l = d.slices, lp = d.slices_padded;
    stats->slices = l;
    std::memcpy(stats->patch_hist, hist, sizeof stats->patch_hist);
    double eq1_bits = 0.0;
    for (uint32_t i = 0; i < d.n_q; ++i) {
        stats->patches[i] = sum[i];
        stats->max_patch[i] = maxp[i];
        // Eq. 1, literally: n_in/n_out * mn + l * ceil(lg max p) + sum p * ceil(lg n_out)
        eq1_bits += (double)d.n_in / (double)d.n_out * (double)mn +
                    (double)l * ceil_lg_u64(maxp[i]) + (double)sum[i] * ceil_lg_u64(d.n_out);
        stats->bits_wc += (round_up(lp * d.n_in / 8, 16) + 16) * 8;
        stats->bits_index += (round_up((lp / SQNN_TILE_SLICES + 1) * 4, 16) + 16) * 8;
        stats->bits_dpatch += (round_up(sum[i] * 2, 16) + 16) * 8;
    }
    stats->bits_tables = (round_up(d.tables_bytes, 16) + 16) * 8;
    stats->bits_index += stats->bits_tables;
    stats->bpw_eq1 = eq1_bits / (double)mn;
    stats->bpw_actual = (double)(stats->bits_wc + stats->bits_npatch + stats->bits_index + stats->bits_dpatch) / (double)mn;
}

// Shared by sqnn_encode_host and sqnn_encode_seeds_host: seeds come from Algorithm 1, from the
// exhaustive search, or from the caller (given != NULL); patch counts and positions follow by
// expanding each seed and comparing on the care bits.  One parallel pass over the format tiles makes seeds,
// patch entries (kept in a buffer of the thread) and statistics; a second one, once the totals are known,
// packs the streams straight into the blob.
static int encode_impl(const sqnn_xornet *net, const sqnn_planes *layer, bool exhaustive,
                       const uint32_t *const *given, void **blob, size_t *blob_bytes, sqnn_stats *stats)
{
    try {
        const uint64_t mn = layer->m * layer->n;
        const uint32_t n_out = net->n_out, n_in = net->n_in, n_q = layer->n_q;
        const uint64_t l = (mn + n_out - 1) / n_out;
        const uint64_t words = (mn + 63) / 64;
        const int64_t tiles = (int64_t)((l + SQNN_TILE_SLICES - 1) / SQNN_TILE_SLICES), items = tiles * n_q;
        for (uint32_t j = 0; n_in < 32 && j < n_out; ++j)
            if (net->rows[j] >> n_in) return stats ? SQNN_E_BAD_BLOB : SQNN_E_INVALID_ARG;     // no blob can hold such rows
        const Expander expand(net->rows, n_out, n_in);
        std::vector<uint64_t> tab;
        if (exhaustive && !given) build_outputs(net->rows, n_out, n_in, tab);
        struct TileOut { const uint16_t *pp; uint32_t count; };
        std::vector<TileOut> made((size_t)items);
        std::unique_ptr<uint32_t[]> seeds(new uint32_t[(size_t)(l * n_q)]);
        // entries of a thread's tiles in blocks that never move (a tile has at most 256 * n_out entries)
        std::vector<std::unique_ptr<uint16_t[]>> blocks;
        uint64_t sum[SQNN_MAX_PLANES] = {0}, hist[SQNN_PATCH_HIST_BINS] = {0};
        uint32_t maxp[SQNN_MAX_PLANES] = {0};
        int bad_seed = 0, no_memory = 0;
        const uint32_t tile_bits = SQNN_TILE_SLICES * n_out;
#pragma omp parallel if (l * n_q >= PARALLEL_FROM)
        {
            uint64_t t_sum[SQNN_MAX_PLANES] = {0}, t_hist[SQNN_PATCH_HIST_BINS] = {0};
            uint32_t t_max[SQNN_MAX_PLANES] = {0};
            std::vector<std::unique_ptr<uint16_t[]>> t_blocks;
            SliceBits block[LANES];
            uint32_t block_seeds[LANES];
            uint32_t room = 0;
            uint16_t *at = nullptr;
            int t_bad = 0, t_nomem = 0;
#pragma omp for schedule(dynamic, 4)
            for (int64_t it = 0; it < items; ++it) {
                if (t_nomem) continue;
                const uint32_t i = (uint32_t)(it / tiles);
                const uint64_t lo = (uint64_t)(it - (int64_t)i * tiles) * SQNN_TILE_SLICES, hi = std::min<uint64_t>(l, lo + SQNN_TILE_SLICES);
                const uint64_t *plane = layer->planes + (uint64_t)i * words;
                if (room < tile_bits) {
                    room = std::max<uint32_t>(tile_bits, 1u << 17);
                    uint16_t *fresh = new (std::nothrow) uint16_t[room];
                    if (!fresh) { t_nomem = 1; continue; }
                    try { t_blocks.emplace_back(fresh); } catch (const std::bad_alloc &) { delete[] fresh; t_nomem = 1; continue; }
                    at = fresh;
                }
                uint16_t *const begin = at;
                for (uint64_t s = lo; s < hi; ++s) {
                    const uint32_t e = (uint32_t)(s - lo) % LANES;
                    if (e == 0) {                         // the next eight slices
                        for (uint32_t f = 0; f < LANES; ++f) {
                            if (s + f < hi) load_slice(plane, layer->mask, mn, n_out, s + f, block[f]);
                            else block[f] = SliceBits{};
                        }
                        if (!given && !exhaustive) encode_alg1_block(net->rows, n_out, n_in, block, block_seeds);
                    }
                    const SliceBits &sb = block[e];
                    uint32_t seed = given ? given[i][s] : exhaustive ? encode_exhaustive(tab, n_in, sb) : block_seeds[e];
                    if (n_in < 32 && (seed >> n_in)) { t_bad = 1; seed = 0; }
                    seeds[(size_t)(i * l + s)] = seed;
                    uint64_t out[4];
                    expand(seed, out);
                    const uint16_t *const before = at;
                    const uint32_t base = (uint32_t)(s - lo) * n_out;
                    for (uint32_t k = 0; k * 64 < n_out; ++k) {
                        uint64_t bad = (out[k] ^ sb.want[k]) & sb.care[k];
                        while (bad) {
                            *at++ = (uint16_t)(base + k * 64 + (uint32_t)__builtin_ctzll(bad));
                            bad &= bad - 1;
                        }
                    }
                    const uint32_t p = (uint32_t)(at - before);
                    t_max[i] = std::max(t_max[i], p);
                    ++t_hist[p < SQNN_PATCH_HIST_BINS - 1 ? p : SQNN_PATCH_HIST_BINS - 1];
                }
                const uint32_t count = (uint32_t)(at - begin);
                made[(size_t)it] = TileOut{begin, count};
                t_sum[i] += count;
                room -= count;
            }
#pragma omp critical
            {
                for (uint32_t i = 0; i < n_q; ++i) { sum[i] += t_sum[i]; maxp[i] = std::max(maxp[i], t_max[i]); }
                for (uint32_t k = 0; k < SQNN_PATCH_HIST_BINS; ++k) hist[k] += t_hist[k];
                bad_seed |= t_bad;
                no_memory |= t_nomem;
                try {
                    for (auto &b : t_blocks) blocks.push_back(std::move(b));
                } catch (const std::bad_alloc &) { no_memory = 1; }
            }
        }
        if (no_memory) return SQNN_E_NOMEM;
        if (bad_seed) return SQNN_E_INVALID_ARG;
        for (uint32_t i = 0; i < n_q; ++i)
            if (sum[i] > 0xffffffffull) return SQNN_E_INVALID_ARG;
        sqnn_desc d;
        uint8_t *b = start_blob(net, layer->m, layer->n, n_q, sum, &d);
        if (!b) return SQNN_E_NOMEM;
        for (uint32_t i = 0; i < n_q; ++i) {
            uint32_t *idx = (uint32_t *)(b + d.off_idx[i]);
            uint32_t run = 0;
            for (uint64_t t = 0; t <= d.slices_padded / SQNN_TILE_SLICES; ++t) {
                idx[t] = run;
                if ((int64_t)t < tiles) run += made[(size_t)(i * tiles + (int64_t)t)].count;
            }
            pack_fields(&seeds[(size_t)(i * l)], l, n_in, (uint32_t *)(b + d.off_wc[i]));
        }
#pragma omp parallel for schedule(static) if (l * n_q >= PARALLEL_FROM)
        for (int64_t it = 0; it < items; ++it) {
            const uint32_t i = (uint32_t)(it / tiles);
            const uint32_t *idx = (const uint32_t *)(b + d.off_idx[i]);
            std::memcpy(b + d.off_pp[i] + (size_t)idx[it - (int64_t)i * tiles] * 2, made[(size_t)it].pp, (size_t)made[(size_t)it].count * 2);
        }
        if (stats) fill_stats(d, sum, maxp, hist, stats);
        *blob = b;
        *blob_bytes = d.total_bytes;
        return SQNN_OK;
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
}

static bool layer_ok(const sqnn_planes *layer)
{
    return layer && layer->planes && layer->mask && layer->n_q >= 1 && layer->n_q <= SQNN_MAX_PLANES &&
           layer->m != 0 && layer->n != 0 && layer->m <= ((uint64_t)1 << 40) / layer->n;
}

int sqnn_encode_host(const sqnn_xornet *net, const sqnn_planes *layer, uint32_t flags,
                     void **blob, size_t *blob_bytes, sqnn_stats *stats)
{
    if (!net_ok(net) || !layer_ok(layer) || !blob || !blob_bytes) return SQNN_E_INVALID_ARG;
    const bool exhaustive = (flags & SQNN_ENCODE_EXHAUSTIVE) != 0;
    if (exhaustive && net->n_in > 20) return SQNN_E_INVALID_ARG;
    return encode_impl(net, layer, exhaustive, nullptr, blob, blob_bytes, stats);
}

int sqnn_encode_seeds_host(const sqnn_xornet *net, const sqnn_planes *layer, const uint32_t *const *wc,
                           void **blob, size_t *blob_bytes, sqnn_stats *stats)
{
    if (!net_ok(net) || !layer_ok(layer) || !wc || !blob || !blob_bytes) return SQNN_E_INVALID_ARG;
    for (uint32_t i = 0; i < layer->n_q; ++i)
        if (!wc[i]) return SQNN_E_INVALID_ARG;
    return encode_impl(net, layer, false, wc, blob, blob_bytes, stats);
}

int sqnn_pack_host(const sqnn_xornet *net, uint64_t m, uint64_t n, uint32_t n_q,
                   const uint32_t *const *wc, const uint16_t *const *np, const uint16_t *const *dp,
                   void **blob, size_t *blob_bytes)
{
    if (!net_ok(net) || !wc || !np || !dp || !blob || !blob_bytes) return SQNN_E_INVALID_ARG;
    if (n_q < 1 || n_q > SQNN_MAX_PLANES || m == 0 || n == 0 || m > ((uint64_t)1 << 40) / n)
        return SQNN_E_INVALID_ARG;
    for (uint32_t i = 0; i < n_q; ++i)
        if (!wc[i] || !np[i] || !dp[i]) return SQNN_E_INVALID_ARG;
    try {
        return build_blob(net, m, n, n_q, wc, np, dp, blob, blob_bytes);
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
}

int sqnn_describe_host(const void *blob, size_t blob_bytes, sqnn_desc *desc)
{
    if (!blob || !desc) return SQNN_E_INVALID_ARG;
    if (blob_bytes < SQNN_BLOB_HEADER_BYTES) return SQNN_E_BAD_BLOB;
    const uint8_t *b = (const uint8_t *)blob;
    sqnn_blob_header h;
    std::memcpy(&h, b, sizeof h);
    if (std::memcmp(h.magic, SQNN_BLOB_MAGIC, 8) != 0 || h.version != SQNN_BLOB_VERSION ||
        h.header_bytes != SQNN_BLOB_HEADER_BYTES)
        return SQNN_E_BAD_BLOB;
    const sqnn_desc &d = h.desc;
    if (d.n_out < 1 || d.n_out > SQNN_MAX_N_OUT || d.n_in < 1 || d.n_in > SQNN_MAX_N_IN ||
        d.n_q < 1 || d.n_q > SQNN_MAX_PLANES || d.tile_slices != SQNN_TILE_SLICES)
        return SQNN_E_BAD_BLOB;
    if (d.m == 0 || d.n == 0 || d.m > ((uint64_t)1 << 40) / d.n) return SQNN_E_BAD_BLOB;
    for (uint32_t i = 0; i < d.n_q; ++i)
        if (d.n_pp[i] > 0xffffffffull) return SQNN_E_BAD_BLOB;
    // every offset and size is a fixed function of the shape and the patch totals
    sqnn_desc want;
    plan_blob(d.m, d.n, d.n_q, d.n_out, d.n_in, d.n_pp, &want);
    if (std::memcmp(&want, &d, sizeof d) != 0 || d.total_bytes != blob_bytes) return SQNN_E_BAD_BLOB;
    const uint64_t mn = d.m * d.n, l = d.slices, lp = d.slices_padded;
    const uint32_t *rows = (const uint32_t *)(b + d.off_xornet);
    if (d.n_in < 32)
        for (uint32_t j = 0; j < d.n_out; ++j)
            if (rows[j] >> d.n_in) return SQNN_E_BAD_BLOB;
    try {
        std::vector<uint32_t> tab(sqnn::table_words(d.n_out, d.n_in));
        build_tables(rows, d.n_out, d.n_in, tab.data());
        if (std::memcmp(tab.data(), b + d.off_tables, (size_t)d.tables_bytes) != 0) return SQNN_E_BAD_BLOB;
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
    const uint64_t tiles = lp / SQNN_TILE_SLICES;
    const uint64_t tile_bits = (uint64_t)SQNN_TILE_SLICES * d.n_out;
    for (uint32_t i = 0; i < d.n_q; ++i) {
        const uint32_t *wcs = (const uint32_t *)(b + d.off_wc[i]);
        const uint32_t *idx = (const uint32_t *)(b + d.off_idx[i]);
        const uint16_t *pp = (const uint16_t *)(b + d.off_pp[i]);
        for (uint64_t s = l; s < lp; ++s)
            if (read_field(wcs, s, d.n_in) != 0) return SQNN_E_BAD_BLOB;
        if (idx[0] != 0 || idx[tiles] != d.n_pp[i]) return SQNN_E_BAD_BLOB;
        for (uint64_t t = 0; t < tiles; ++t) {
            if (idx[t + 1] < idx[t] || idx[t + 1] > d.n_pp[i]) return SQNN_E_BAD_BLOB;
            int64_t prev = -1;
            for (uint64_t k = idx[t]; k < idx[t + 1]; ++k) {
                const uint64_t pos = pp[k];
                if (pos >= tile_bits || (int64_t)pos <= prev || t * tile_bits + pos >= mn) return SQNN_E_BAD_BLOB;
                prev = (int64_t)pos;
            }
        }
    }
    *desc = d;
    return SQNN_OK;
}

// n_patch of every slice of one plane, from the patch positions of a validated blob.
static void count_patches(const uint8_t *b, const sqnn_desc &d, uint32_t plane, uint16_t *np)
{
    const uint32_t *idx = (const uint32_t *)(b + d.off_idx[plane]);
    const uint16_t *pp = (const uint16_t *)(b + d.off_pp[plane]);
    std::memset(np, 0, sizeof(uint16_t) * (size_t)d.slices);
    const uint64_t tiles = d.slices_padded / SQNN_TILE_SLICES;
    for (uint64_t t = 0; t < tiles; ++t)
        for (uint64_t k = idx[t]; k < idx[t + 1]; ++k)
            ++np[t * SQNN_TILE_SLICES + pp[k] / d.n_out];
}

int sqnn_unpack_host(const void *blob, size_t blob_bytes, uint32_t plane,
                     uint32_t **wc, uint16_t **np, uint16_t **dp, uint64_t *n_dp)
{
    if (!wc || !np || !dp || !n_dp) return SQNN_E_INVALID_ARG;
    sqnn_desc d;
    int rc = sqnn_describe_host(blob, blob_bytes, &d);
    if (rc != SQNN_OK) return rc;
    if (plane >= d.n_q) return SQNN_E_INVALID_ARG;
    const uint8_t *b = (const uint8_t *)blob;
    const uint64_t l = d.slices;
    uint32_t *w = (uint32_t *)std::malloc(sizeof(uint32_t) * (l ? l : 1));
    uint16_t *p = (uint16_t *)std::malloc(sizeof(uint16_t) * (l ? l : 1));
    uint16_t *q = (uint16_t *)std::malloc(sizeof(uint16_t) * (d.n_pp[plane] ? d.n_pp[plane] : 1));
    if (!w || !p || !q) { std::free(w); std::free(p); std::free(q); return SQNN_E_NOMEM; }
    const uint32_t *wcs = (const uint32_t *)(b + d.off_wc[plane]);
    for (uint64_t s = 0; s < l; ++s) w[s] = read_field(wcs, s, d.n_in);
    count_patches(b, d, plane, p);
    // positions ascend inside a tile, so they already stand in slice order, ascending inside a slice
    const uint16_t *pp = (const uint16_t *)(b + d.off_pp[plane]);
    for (uint64_t k = 0; k < d.n_pp[plane]; ++k) q[k] = (uint16_t)(pp[k] % d.n_out);
    *wc = w; *np = p; *dp = q; *n_dp = d.n_pp[plane];
    return SQNN_OK;
}

int sqnn_stats_host(const void *blob, size_t blob_bytes, sqnn_stats *stats)
{
    if (!stats) return SQNN_E_INVALID_ARG;
    sqnn_desc d;
    int rc = sqnn_describe_host(blob, blob_bytes, &d);
    if (rc != SQNN_OK) return rc;
    const uint8_t *b = (const uint8_t *)blob;
    uint64_t sum[SQNN_MAX_PLANES] = {0}, hist[SQNN_PATCH_HIST_BINS] = {0};
    uint32_t maxp[SQNN_MAX_PLANES] = {0};
    try {
        std::vector<uint16_t> np(d.slices ? d.slices : 1);
        for (uint32_t i = 0; i < d.n_q; ++i) {
            count_patches(b, d, i, np.data());
            for (uint64_t s = 0; s < d.slices; ++s) {
                const uint32_t p = np[s];
                maxp[i] = std::max(maxp[i], p);
                sum[i] += p;
                ++hist[p < SQNN_PATCH_HIST_BINS - 1 ? p : SQNN_PATCH_HIST_BINS - 1];
            }
        }
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
    fill_stats(d, sum, maxp, hist, stats);
    return SQNN_OK;
}

int sqnn_stats_blocked_host(const void *blob, size_t blob_bytes, uint64_t block_slices,
                            double *bpw_eq1, uint64_t *bits_npatch)
{
    if (block_slices == 0) return SQNN_E_INVALID_ARG;
    sqnn_desc d;
    int rc = sqnn_describe_host(blob, blob_bytes, &d);
    if (rc != SQNN_OK) return rc;
    const uint8_t *b = (const uint8_t *)blob;
    const uint64_t mn = d.m * d.n, l = d.slices;
    uint64_t np_bits = 0, dp_entries = 0;
    try {
        std::vector<uint16_t> np(l ? l : 1);
        for (uint32_t i = 0; i < d.n_q; ++i) {
            count_patches(b, d, i, np.data());
            for (uint64_t s0 = 0; s0 < l; s0 += block_slices) {
                const uint64_t s1 = std::min(l, s0 + block_slices);
                uint32_t maxp = 0;
                for (uint64_t s = s0; s < s1; ++s) maxp = std::max<uint32_t>(maxp, np[s]);
                np_bits += (s1 - s0) * ceil_lg_u64(maxp);
            }
            dp_entries += d.n_pp[i];
        }
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
    if (bits_npatch) *bits_npatch = np_bits;
    if (bpw_eq1)
        *bpw_eq1 = ((double)d.n_q * (double)d.n_in / (double)d.n_out * (double)mn + (double)np_bits +
                    (double)dp_entries * ceil_lg_u64(d.n_out)) / (double)mn;
    return SQNN_OK;
}

// ---------------------------------------------------------------------------------------------
// Algorithm 1 with 64-bit rows of M (host only)
// ---------------------------------------------------------------------------------------------
namespace {

inline uint32_t bit_at(const uint64_t *words, uint64_t p) { return (uint32_t)((words[p >> 6] >> (p & 63)) & 1); }

// Seed of one slice (positions [p0, p1) of the plane) by the same incremental elimination as
// encode_alg1, and the list of care positions the seed does not reproduce.
inline uint64_t encode_alg1_wide(const uint64_t *rows, const uint64_t *plane, const uint64_t *mask,
                                 uint64_t p0, uint64_t p1, std::vector<uint16_t> &wrong)
{
    uint64_t prow[64];
    uint32_t pcol[64];
    uint8_t prhs[64];
    uint32_t npiv = 0;
    for (uint64_t p = p0; p < p1; ++p) {
        if (!bit_at(mask, p)) continue;
        uint64_t a = rows[p - p0];
        uint8_t b = (uint8_t)bit_at(plane, p);
        for (uint32_t q = 0; q < npiv; ++q)
            if ((a >> pcol[q]) & 1) { a ^= prow[q]; b ^= prhs[q]; }
        if (a == 0) continue;
        const uint32_t col = (uint32_t)__builtin_ctzll(a);
        for (uint32_t q = 0; q < npiv; ++q)
            if ((prow[q] >> col) & 1) { prow[q] ^= a; prhs[q] ^= b; }
        prow[npiv] = a; prhs[npiv] = b; pcol[npiv] = col;
        ++npiv;
    }
    uint64_t seed = 0;
    for (uint32_t q = 0; q < npiv; ++q)
        if (prhs[q]) seed |= (uint64_t)1 << pcol[q];
    wrong.clear();
    for (uint64_t p = p0; p < p1; ++p)
        if (bit_at(mask, p) && (uint32_t)(__builtin_popcountll(rows[p - p0] & seed) & 1) != bit_at(plane, p))
            wrong.push_back((uint16_t)(p - p0));
    return seed;
}

}  // namespace

int sqnn_encode_wide_host(uint32_t n_out, uint32_t n_in, const uint64_t *rows, uint64_t mn,
                          const uint64_t *plane, const uint64_t *mask,
                          uint64_t **wc, uint16_t **np, uint16_t **dp, uint64_t *n_dp, double *bpw_eq1)
{
    if (!rows || !plane || !mask || !wc || !np || !dp || !n_dp || n_out < 1 || n_out > 4096 || n_in < 1 || n_in > 64 ||
        mn == 0 || mn > ((uint64_t)1 << 40))
        return SQNN_E_INVALID_ARG;
    if (n_in < 64)
        for (uint32_t j = 0; j < n_out; ++j)
            if (rows[j] >> n_in) return SQNN_E_INVALID_ARG;
    try {
        const uint64_t l = (mn + n_out - 1) / n_out;
        std::vector<uint64_t> seeds(l);
        std::vector<std::vector<uint16_t>> lists(l);
#pragma omp parallel
        {
            std::vector<uint16_t> wrong;
#pragma omp for schedule(dynamic, 256)
            for (int64_t s = 0; s < (int64_t)l; ++s) {
                const uint64_t p0 = (uint64_t)s * n_out, p1 = std::min(mn, p0 + n_out);
                seeds[s] = encode_alg1_wide(rows, plane, mask, p0, p1, wrong);
                lists[s] = wrong;
            }
        }
        uint64_t total = 0, maxp = 0;
        for (uint64_t s = 0; s < l; ++s) { total += lists[s].size(); maxp = std::max<uint64_t>(maxp, lists[s].size()); }
        uint64_t *w = (uint64_t *)std::malloc(sizeof(uint64_t) * l);
        uint16_t *c = (uint16_t *)std::malloc(sizeof(uint16_t) * l);
        uint16_t *q = (uint16_t *)std::malloc(sizeof(uint16_t) * (total ? total : 1));
        if (!w || !c || !q) { std::free(w); std::free(c); std::free(q); return SQNN_E_NOMEM; }
        uint64_t at = 0;
        for (uint64_t s = 0; s < l; ++s) {
            w[s] = seeds[s];
            c[s] = (uint16_t)lists[s].size();
            for (uint16_t v : lists[s]) q[at++] = v;
        }
        *wc = w; *np = c; *dp = q; *n_dp = total;
        if (bpw_eq1)
            *bpw_eq1 = ((double)n_in / (double)n_out * (double)mn + (double)l * ceil_lg_u64(maxp) +
                        (double)total * ceil_lg_u64(n_out)) / (double)mn;
        return SQNN_OK;
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
}

// ---------------------------------------------------------------------------------------------
// storage form
// ---------------------------------------------------------------------------------------------
namespace {

const char STORE_MAGIC[8] = {'S', 'Q', 'N', 'N', 'S', 'T', 'R', '1'};

struct StoreHeader {
    char magic[8];
    uint64_t m, n, block_slices, total_bytes;
    uint32_t n_q, n_out, n_in, reserved;
    uint64_t n_dp[SQNN_MAX_PLANES];
    uint64_t reserved2;
};
static_assert(sizeof(StoreHeader) == 128, "storage header is 128 bytes");

struct BitWriter {
    std::vector<uint8_t> &buf;
    uint64_t acc = 0;
    uint32_t have = 0;
    explicit BitWriter(std::vector<uint8_t> &b) : buf(b) {}
    void put(uint32_t v, uint32_t width)
    {
        if (width == 0) return;
        acc |= (uint64_t)v << have;
        have += width;
        while (have >= 8) { buf.push_back((uint8_t)acc); acc >>= 8; have -= 8; }
    }
    void flush() { if (have) { buf.push_back((uint8_t)acc); acc = 0; have = 0; } }     // streams start on a byte
};

struct BitReader {
    const uint8_t *p, *end;
    uint64_t acc = 0;
    uint32_t have = 0;
    bool ok = true;
    BitReader(const uint8_t *b, const uint8_t *e) : p(b), end(e) {}
    uint32_t get(uint32_t width)
    {
        if (width == 0) return 0;
        while (have < width) {
            if (p >= end) { ok = false; return 0; }
            acc |= (uint64_t)*p++ << have;
            have += 8;
        }
        const uint32_t v = (uint32_t)(acc & (((uint64_t)1 << width) - 1));
        acc >>= width;
        have -= width;
        return v;
    }
    void align() { acc = 0; have = 0; }
};

}  // namespace

int sqnn_store_host(const void *blob, size_t blob_bytes, uint64_t block_slices,
                    void **stored, size_t *stored_bytes, sqnn_store_info *info)
{
    if (!stored || !stored_bytes || block_slices == 0) return SQNN_E_INVALID_ARG;
    sqnn_desc d;
    int rc = sqnn_describe_host(blob, blob_bytes, &d);
    if (rc != SQNN_OK) return rc;
    try {
        const uint8_t *b = (const uint8_t *)blob;
        const uint64_t l = d.slices;
        const uint32_t w_dp = ceil_lg_u64(d.n_out);
        StoreHeader h;
        std::memset(&h, 0, sizeof h);
        std::memcpy(h.magic, STORE_MAGIC, 8);
        h.m = d.m; h.n = d.n; h.block_slices = block_slices;
        h.n_q = d.n_q; h.n_out = d.n_out; h.n_in = d.n_in;
        std::vector<uint8_t> out(sizeof h, 0);
        out.insert(out.end(), b + d.off_xornet, b + d.off_xornet + (size_t)d.n_out * 4);
        sqnn_store_info si;
        std::memset(&si, 0, sizeof si);
        std::vector<uint16_t> np(l ? l : 1);
        for (uint32_t i = 0; i < d.n_q; ++i) {
            h.n_dp[i] = d.n_pp[i];
            const uint32_t *wcs = (const uint32_t *)(b + d.off_wc[i]);
            const uint16_t *pp = (const uint16_t *)(b + d.off_pp[i]);
            count_patches(b, d, i, np.data());
            BitWriter bw(out);
            for (uint64_t s = 0; s < l; ++s) bw.put(read_field(wcs, s, d.n_in), d.n_in);
            bw.flush();
            si.bits_wc += l * d.n_in;
            const uint64_t blocks = (l + block_slices - 1) / block_slices;
            std::vector<uint8_t> widths(blocks);
            for (uint64_t k = 0; k < blocks; ++k) {
                uint32_t maxp = 0;
                for (uint64_t s = k * block_slices; s < std::min(l, (k + 1) * block_slices); ++s) maxp = std::max<uint32_t>(maxp, np[s]);
                widths[k] = (uint8_t)ceil_lg_u64((uint64_t)maxp + 1);
            }
            out.insert(out.end(), widths.begin(), widths.end());
            si.bits_widths += blocks * 8;
            for (uint64_t s = 0; s < l; ++s) {
                bw.put(np[s], widths[s / block_slices]);
                si.bits_npatch += widths[s / block_slices];
            }
            bw.flush();
            for (uint64_t k = 0; k < d.n_pp[i]; ++k) bw.put(pp[k] % d.n_out, w_dp);
            bw.flush();
            si.bits_dpatch += d.n_pp[i] * w_dp;
        }
        h.total_bytes = out.size();
        std::memcpy(out.data(), &h, sizeof h);
        uint8_t *res = (uint8_t *)std::malloc(out.size());
        if (!res) return SQNN_E_NOMEM;
        std::memcpy(res, out.data(), out.size());
        *stored = res;
        *stored_bytes = out.size();
        si.total_bytes = out.size();
        si.bpw = (double)(si.bits_wc + si.bits_widths + si.bits_npatch + si.bits_dpatch) / (double)(d.m * d.n);
        if (info) *info = si;
        return SQNN_OK;
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
}

int sqnn_load_host(const void *stored, size_t stored_bytes, void **blob, size_t *blob_bytes)
{
    if (!stored || !blob || !blob_bytes) return SQNN_E_INVALID_ARG;
    if (stored_bytes < sizeof(StoreHeader)) return SQNN_E_BAD_BLOB;
    const uint8_t *b = (const uint8_t *)stored, *end = b + stored_bytes;
    StoreHeader h;
    std::memcpy(&h, b, sizeof h);
    if (std::memcmp(h.magic, STORE_MAGIC, 8) != 0 || h.total_bytes != stored_bytes) return SQNN_E_BAD_BLOB;
    if (h.n_out < 1 || h.n_out > SQNN_MAX_N_OUT || h.n_in < 1 || h.n_in > SQNN_MAX_N_IN || h.n_q < 1 ||
        h.n_q > SQNN_MAX_PLANES || h.m == 0 || h.n == 0 || h.m > ((uint64_t)1 << 40) / h.n || h.block_slices == 0)
        return SQNN_E_BAD_BLOB;
    try {
        const uint64_t mn = h.m * h.n, l = (mn + h.n_out - 1) / h.n_out;
        const uint32_t w_dp = ceil_lg_u64(h.n_out);
        const uint8_t *p = b + sizeof h;
        if ((uint64_t)(end - p) < (uint64_t)h.n_out * 4) return SQNN_E_BAD_BLOB;
        std::vector<uint32_t> rows(h.n_out);
        std::memcpy(rows.data(), p, (size_t)h.n_out * 4);
        p += (size_t)h.n_out * 4;
        std::vector<PlaneArrays> pa(h.n_q);
        std::vector<std::vector<uint16_t>> dp16(h.n_q);
        for (uint32_t i = 0; i < h.n_q; ++i) {
            if (h.n_dp[i] > 0xffffffffull) return SQNN_E_BAD_BLOB;
            // nothing is allocated for more slices than the rest of the buffer could hold seeds for
            if (l > (uint64_t)(end - p) * 8 / h.n_in) return SQNN_E_BAD_BLOB;
            BitReader br(p, end);
            pa[i].wc.resize(l);
            pa[i].np.resize(l);
            for (uint64_t s = 0; s < l; ++s) pa[i].wc[s] = br.get(h.n_in);
            if (!br.ok) return SQNN_E_BAD_BLOB;
            br.align();
            const uint64_t blocks = (l + h.block_slices - 1) / h.block_slices;
            if ((uint64_t)(end - br.p) < blocks) return SQNN_E_BAD_BLOB;
            const uint8_t *widths = br.p;
            br.p += blocks;
            uint64_t sum = 0;
            for (uint64_t s = 0; s < l; ++s) {
                const uint32_t w = widths[s / h.block_slices];
                if (w > 9) return SQNN_E_BAD_BLOB;
                const uint32_t v = br.get(w);
                if (v > h.n_out) return SQNN_E_BAD_BLOB;
                pa[i].np[s] = (uint16_t)v;
                sum += v;
            }
            if (!br.ok || sum != h.n_dp[i]) return SQNN_E_BAD_BLOB;
            br.align();
            if (w_dp && sum > (uint64_t)(end - br.p) * 8 / w_dp) return SQNN_E_BAD_BLOB;
            dp16[i].resize(sum ? sum : 1);
            for (uint64_t k = 0; k < sum; ++k) dp16[i][k] = (uint16_t)br.get(w_dp);
            if (!br.ok) return SQNN_E_BAD_BLOB;
            br.align();
            p = br.p;
        }
        if (p != end) return SQNN_E_BAD_BLOB;
        sqnn_xornet net{h.n_out, h.n_in, rows.data()};
        if (h.n_in < 32)
            for (uint32_t j = 0; j < h.n_out; ++j)
                if (rows[j] >> h.n_in) return SQNN_E_BAD_BLOB;
        std::vector<const uint32_t *> wcp(h.n_q);
        std::vector<const uint16_t *> npp(h.n_q), dpp(h.n_q);
        for (uint32_t i = 0; i < h.n_q; ++i) { wcp[i] = pa[i].wc.data(); npp[i] = pa[i].np.data(); dpp[i] = dp16[i].data(); }
        const int rc = build_blob(&net, h.m, h.n, h.n_q, wcp.data(), npp.data(), dpp.data(), blob, blob_bytes);
        return rc == SQNN_E_INVALID_ARG ? SQNN_E_BAD_BLOB : rc;     // bad contents, not a bad call
    } catch (const std::bad_alloc &) {
        return SQNN_E_NOMEM;
    }
}

int sqnn_fifo_model_host(const uint16_t *np, uint64_t l, uint32_t n_fifo, uint32_t rate, uint32_t depth,
                         sqnn_fifo_result *result)
{
    if (!result || (!np && l) || n_fifo == 0 || rate == 0 || depth == 0) return SQNN_E_INVALID_ARG;
    std::memset(result, 0, sizeof *result);
    uint64_t left = 0;                                   // entries the stream has not delivered yet
    for (uint64_t s = 0; s < l; ++s) left += np[s];
    uint64_t held = 0;                                   // entries in the FIFO
    for (uint64_t s = 0; s < l; ++s) {
        uint64_t due = np[s];
        for (;;) {                                       // one pass = one cycle spent on slice s
            ++result->cycles;
            uint64_t in = std::min<uint64_t>(rate, left);
            if (in > depth - held) { in = depth - held; ++result->stall_full; }
            held += in;
            left -= in;
            result->peak = std::max(result->peak, held);
            const uint64_t out = std::min(std::min<uint64_t>(due, n_fifo), held);
            held -= out;
            due -= out;
            if (due == 0) break;
            if (out == n_fifo) ++result->stall_bandwidth; else ++result->stall_empty;
        }
    }
    return SQNN_OK;
}

}  // extern "C"
