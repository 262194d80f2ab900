// How the small-batch product (batch <= 15) is cut up, and which of its two forms takes a call.  Host code, no CUDA:
// shared by the launchers, and compiled by itself in a CPU test.
//
// Both forms give a block a run of whole rows of W and decode the bits of those rows into shared memory, in
// chunks of rows where they do not fit at once; they differ in the product:
//   expanding (sqnn_gemv_tc.cuh)  all weights to bf16, tensor cores; the same work at any density, once per pass of
//                                 activation vectors
//   walk (sqnn_gemv.cuh)          one care bit after the other on the plain ALUs; the work is the care bits'
//
// Which form.  The expanding one takes every call whose rows fit, with one exception: of layers with one plane and bf16
// activations the walk takes those it is estimated to do at least 10 % faster (`us` of the two plans).  That is the
// small and the sparse layer with few vectors, where the expanding form's longer chain of phases and its units of
// 16 rows x 1024 columns cost more than the care bits do.  Expanding / walk, one vector:
//   2048 x 1024, 7 % kept 5.7 / 4.4 us     1024 x 3072, 7 % kept 6.1 / 4.8     4096 x 9216, 9 % kept 9.8 / 11.5
// Over 1048 random calls of that kind (2^16 to 2^26 weights, 2 to 50 % kept, 1 to 15 vectors), all in whole format tiles, the rule takes 172 to the
// walk; none loses more than 5 %, and all 1048 together gain 3 % (geometric mean), where always choosing right
// would gain 4 %.  Layers of run-time shapes that have room for parts: plan_run_time_shape.
// The walk is also faster on sparse or wide layers with fp32 activations or several planes (2048 x 1024, 3.5 % kept, 8
// fp32 vectors: 10.2 / 7.5 us; 4096 x 12288, 10 % kept, 4 fp32 vectors, where the expanding form runs out of shared
// memory: 67 / 36).  It does not get those calls: its sums lie further from the 64-bit product.  Relative errors over
// 3984 random calls, expanding / walk, median (the walk's is the larger one in 96 % and more of the calls of each of the
// last three kinds, and in none of the first):
//   bf16, one plane 5.9e-8 / 2.7e-8        bf16, more planes 6.9e-8 / 1.0e-7
//   fp32, one plane 6.9e-8 / 9.2e-8        fp32, more planes 8.0e-8 / 1.0e-7
#ifndef SQNN_GEMV_PLAN_H_
#define SQNN_GEMV_PLAN_H_
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include "sqnn_layout.h"

namespace sqnn {

constexpr uint32_t TC_GROUPS = 4;                         // expander groups
constexpr uint32_t TC_TILE_ROWS = 16, TC_RANGES = 8;
constexpr uint32_t TC_MAX_Q = 12;                         // activation columns (vectors x pieces) per pass: N <= 96
constexpr uint32_t TC_WARPS = TC_GROUPS * 5;
constexpr size_t GEMV_SMEM_LIMIT = 220 * 1024;
constexpr double WALK_MARGIN = 0.9;

struct GemvLayer {
    uint64_t m, n;
    uint32_t batch, n_q;
    uint32_t W, tab_words;        // words per lane of a kernel tile (a tile is 32 W words of a plane), words of the tables
    uint32_t x_bytes;             // of an activation: 2 (bf16) or 4 (fp32)
    uint32_t sms;
    double density;               // share of unpruned weights, estimated (care_density); read for one plane and bf16 only
    double tile_us = 0.0;         // estimated time a warp takes to decode a tile; 0: by W, the constants of whole tiles
};

// The mask's density is on the device.  What the blob says of it: a slice with k care bits of rank r needs about
// (k - r) / 2 patches and r <= n_in, so k <= n_in + 2 x (patches per slice).  Equal to it when the network was chosen
// for the layer (as many care bits as seed bits, or more), too high otherwise, which favours the expanding form.
inline double care_density(uint32_t n_out, uint32_t n_in, double patches_per_slice)
{
    const double d = (n_in + 2.0 * patches_per_slice) / n_out;
    return d < 1.0 ? d : 1.0;
}

// Tiles of 32 W words that can cover `rows` rows, whatever bit the first one starts at.
inline uint64_t covering_tiles(const GemvLayer &L, uint64_t rows)
{
    const uint64_t tile_bits = 1024ull * L.W;
    return (rows * L.n + tile_bits - 1) / tile_bits + 1;
}
inline uint64_t up4(uint64_t v) { return (v + 3) & ~3ull; }

struct TcPlan {
    bool ok;
    uint32_t rows_per_block, rows_per_chunk, grid;
    uint32_t units;               // 128-column units per range
    uint32_t bt, N, slots;        // activation vectors per pass, MMA N, A slots per group
    uint32_t region_words, alpha_words, part_words;
    size_t smem;
    double us;
};

// Estimates for bf16 activations and one plane, with constants fitted to the calls above (standard deviation of the
// logarithm: 16 %).  Fixed costs, decode (per word of a lane's tile and warp, or GemvLayer::tile_us), and per pass of a chunk its staging, set-up and
// expansion: e us per 128 columns of 16 rows x 8 ranges and group, more with N (above 64 there is one A slot per
// group, and expansion and MMA take turns).
inline double tc_estimate_us(const GemvLayer &L, const TcPlan &p, uint32_t passes)
{
    const double e = p.N <= 64 ? 0.87 + 0.011 * (p.N - 16) : 1.4 + 0.0044 * p.N;
    double us = 3.5;
    uint64_t chunks = 0;
    for (uint64_t left = p.rows_per_block; left != 0;) {
        const uint64_t rows = left < p.rows_per_chunk ? left : p.rows_per_chunk, times = left / rows;
        const uint64_t list = (rows + TC_TILE_ROWS - 1) / TC_TILE_ROWS * L.n_q * p.units;
        us += times * (0.4 + passes * (1.1 + (double)((list + TC_GROUPS - 1) / TC_GROUPS) * e));
        chunks += times;
        left -= times * rows;
    }
    us += chunks * (L.tile_us > 0 ? L.tile_us : 0.056 * L.W) * (double)((covering_tiles(L, p.rows_per_chunk) * L.n_q + TC_WARPS - 1) / TC_WARPS);
    return us + (passes > 1 ? passes * chunks : 1) * 0.016 * p.bt * p.units;
}

inline TcPlan plan_gemv_tc(const GemvLayer &L)
{
    TcPlan p = {};
    const uint32_t pieces = L.x_bytes == 4 ? 3 : 1;       // fp32 activations enter as three bf16
    const uint64_t R = (L.m + L.sms - 1) / L.sms;
    if (R > 0xffffffffull || L.n > (1u << 24)) return p;
    p.rows_per_block = (uint32_t)R;
    p.grid = (uint32_t)((L.m + R - 1) / R);
    p.units = (uint32_t)((L.n + 128 * TC_RANGES - 1) / (128 * TC_RANGES));
    if (p.units % 8 == 0) ++p.units;                      // banks: see sqnn_gemv_tc.cuh
    const uint32_t kq = p.units * 128;
    // bits a lane may read past the end of the last row: its range's padding and the second vector
    const uint64_t slack = (TC_RANGES * (uint64_t)kq - L.n) / 32 + 12;
    // Activation vectors per pass: as many as the accumulators allow, fewer where they would leave too little
    // shared memory for a chunk of rows (every pass expands the weights again, every chunk decodes its boundary
    // tiles again and may leave a tile of 16 rows half empty).
    const uint32_t bt_max = TC_MAX_Q / pieces;
    for (uint32_t passes = (L.batch + bt_max - 1) / bt_max; passes <= L.batch; ++passes) {
        p.bt = (L.batch + passes - 1) / passes;
        p.N = (8 * p.bt * pieces + 15) / 16 * 16;
        p.slots = p.N <= 64 ? 2u : 1u;
        const size_t x_bytes = (size_t)(kq / 64) * p.N * 128 + 1024;
        for (uint64_t RC = R;; RC = (RC + 1) / 2) {
            const uint64_t region_words = up4(covering_tiles(L, RC) * 32 * L.W + slack);
            p.alpha_words = (uint32_t)up4(RC * L.n_q);
            p.part_words = (uint32_t)up4(TC_GROUPS * RC * p.bt);
            const uint64_t need = 4ull * L.tab_words + (uint64_t)(L.n_q + 1) * region_words * 4 + 4ull * (p.alpha_words + p.part_words) + x_bytes;
            if (need <= GEMV_SMEM_LIMIT) {
                p.ok = true;
                p.region_words = (uint32_t)region_words;
                p.rows_per_chunk = (uint32_t)RC;
                p.smem = (size_t)need;
                p.us = tc_estimate_us(L, p, passes);
                return p;
            }
            if (RC <= 8) break;
        }
    }
    return p;                                             // rows too long
}

struct WalkPlan {
    bool ok;
    uint32_t rows_per_block, rows_per_chunk, grid, warps;
    uint32_t bt, parts;           // activation vectors at a time, warps sharing a row
    bool xs;                      // activations staged in shared memory
    uint32_t region_words, alpha_words, part_words, xs_words;
    size_t smem;
    double us;
};

// As above.  Fixed costs, decode, and per chunk and group of vectors the walk: a step (one word of mask for every lane) takes as
// many turns as the fullest of 32 words has care bits.  Turns are bound by what the whole SM issues and loads, or by
// their latency where a block has few items (rows, or parts of rows) for its warps.
inline double walk_estimate_us(const GemvLayer &L, const WalkPlan &p)
{
    const double d = L.density, most = 32 * d + 2.0 * sqrt(32 * d * (1.0 - d)) + 0.3, turns = most < 32 ? most : 32;
    const uint64_t words = (L.n + 31) / 32 + 1, steps = ((words + p.parts - 1) / p.parts + 31) / 32;
    double us = 3.3;
    uint64_t chunks = 0;
    for (uint64_t left = p.rows_per_block; left != 0;) {
        const uint64_t rows = left < p.rows_per_chunk ? left : p.rows_per_chunk, times = left / rows;
        const uint64_t items = rows * p.parts, rounds = (items + p.warps - 1) / p.warps;
        const double issue = items * (0.0016 + 0.0030 * p.bt), latency = rounds * (0.0175 + 0.055 * p.bt);
        us += times * ((L.batch + p.bt - 1) / p.bt) * steps * turns * (issue > latency ? issue : latency);
        chunks += times;
        left -= times * rows;
    }
    return us + chunks * (L.tile_us > 0 ? L.tile_us : 0.07 * L.W) * (double)((covering_tiles(L, p.rows_per_chunk) * L.n_q + p.warps - 1) / p.warps);
}

inline WalkPlan plan_walk(const GemvLayer &L)
{
    WalkPlan p = {};
    const uint64_t R = (L.m + L.sms - 1) / L.sms;
    if (R > 0xffffffffull) return p;
    p.rows_per_block = (uint32_t)R;
    p.grid = (uint32_t)((L.m + R - 1) / R);
    p.bt = L.batch <= 2 ? L.batch : L.batch <= 4 ? 4 : 8;
    // a block with a few rows and a few tiles to decode gets a few warps: a thread block is cheaper to start
    // and to synchronise the smaller it is (tiny layers are all launch and latency)
    const uint64_t items = covering_tiles(L, R) * L.n_q, want = R > items ? R : items;
    p.warps = want <= 4 ? 4u : want <= 8 ? 8u : want <= 16 ? 16u : 32u;
    const size_t xbytes = ((size_t)L.n * p.bt * L.x_bytes + 15) & ~(size_t)15;
    bool xs = p.bt == 1 && xbytes <= 128 * 1024;          // several long vectors never fit
    // Warps sharing a row.  A warp walks its run of a row's words 32 at a time, and every item (a row, or one
    // of `parts` runs of it) costs about one such step more for its set-up and reduction, so the walk of a chunk
    // takes (rounds of items over the warps) x (steps per item + 1); the cheapest split wins, the smaller one on
    // a tie.  (Measured on 41 rows of 94 words, two planes: 1 part 13.5 us, 2 parts 15.2, 3 parts 13.8, 4 parts 16.5.)
    const uint64_t row_words = (L.n + 31) / 32 + 1;
    auto pick_parts = [&](uint64_t rows) {
        uint32_t best = 1;
        uint64_t best_cost = ~0ull;
        for (uint32_t c = 1; c <= 32 && c <= row_words; ++c) {
            const uint64_t per = (row_words + c - 1) / c;
            const uint64_t cost = ((rows * c + p.warps - 1) / p.warps) * ((per + 31) / 32 + 1);
            if (cost < best_cost) { best = c; best_cost = cost; }
        }
        return best;
    };
    for (uint64_t RC = R;;) {
        p.parts = pick_parts(RC);
        const uint64_t region_words = covering_tiles(L, RC) * 32 * L.W;
        p.alpha_words = (uint32_t)up4(RC * L.n_q);
        p.part_words = (uint32_t)up4(RC * p.parts * p.bt);
        p.xs_words = xs ? (uint32_t)(xbytes / 4) : 0u;
        const uint64_t need = 4ull * L.tab_words + (uint64_t)(L.n_q + 1) * region_words * 4 + 4ull * (p.alpha_words + p.part_words + p.xs_words);
        if (need <= GEMV_SMEM_LIMIT) {
            p.ok = true;
            p.xs = xs;
            p.region_words = (uint32_t)region_words;
            p.rows_per_chunk = (uint32_t)RC;
            p.smem = (size_t)need;
            p.us = walk_estimate_us(L, p);
            return p;
        }
        if (RC > 1) { RC = (RC + 1) / 2; continue; }
        if (!xs) return p;                                // one row of bits does not fit
        xs = false;                                       // leave the activations in global memory
        RC = R;
    }
}

// Run-time shapes: the tiles of a layer that has room for parts of format tiles (L.W: words of whole ones), for each of the two forms.  KT = 0:
// parts.  Whole tiles of slices with a single lookup are cheap (see most_parts_per_sm): where kernel tiles are single format tiles,
// the walk never cuts them (parts / whole, us: 960 x 576, 8 x 2 5.7 / 4.9; 8000 x 1984, 256 x 4 7.9 / 6.9; 512 x 576, 96 x 3 4.6 / 4.4) and the
// expanding form cuts them to one turn or not at all (96 x 7, one turn 6.6 / 7.0; 112 x 3, two turns 9.0 / 8.6); of
// two format tiles, to two turns at most (56 x 10, two of 16 7.3 / 7.8; 50 x 5, four 10.9 / 10.7).
// Estimates: a part costs its turns; whole tiles against parts of the other form their words, at less than where both are whole.
// 273 one-plane bf16 calls with room for parts (2^16 to 2^25 weights, 1 to 15 vectors, any network): 0.76 of the time of whole tiles for both forms,
// 0.9 % over always choosing right; 3 of them are more than 3 % slower than with whole tiles (by 4 % at most), 15 (by 20 %) where both
// forms cut all they can.
struct GemvTiles {
    uint32_t KT, W;
};
// Cuts the tiles of one form to at most `most` turns; L gets their words and, at turn_us a turn, the estimate of a part.
inline GemvTiles cut_gemv_tiles(uint32_t n_out, uint32_t most, double turn_us, GemvLayer *L)
{
    GemvTiles t{format_tiles_per_kernel_tile(n_out), L->W};
    const uint32_t turns = cut_tiles(n_out, most, &t.KT, &t.W, [&](uint32_t words) {
        GemvLayer M = *L;
        M.W = words;
        return covering_tiles(M, (L->m + L->sms - 1) / L->sms) * L->n_q <= TC_WARPS;
    });
    L->W = t.W;
    L->tile_us = turns * turn_us;
    return t;
}
struct GemvForms {
    TcPlan tc;
    WalkPlan walk;
    GemvTiles tc_tiles, walk_tiles;
};
inline GemvForms plan_run_time_shape(uint32_t n_out, uint32_t n_in, const GemvLayer &whole)
{
    const uint32_t KT = format_tiles_per_kernel_tile(n_out), most = most_turns(n_out);
    const bool cheap = table_chunks(n_in, entry_words_padded(n_out)) == 1 && KT < 4;
    const uint32_t few = cheap && KT < most ? KT : most;
    GemvForms f;
    GemvLayer L = whole, Lw = whole;
    f.tc_tiles = cut_gemv_tiles(n_out, most, 0.8, &L);
    f.tc = plan_gemv_tc(L);
    f.walk_tiles = cut_gemv_tiles(n_out, most, 0.7, &Lw);
    f.walk = plan_walk(Lw);
    if (!cheap) return f;
    // ... as long as the larger tiles take nothing else away: eight planes of them may leave less room for rows, vectors or activations, or none
    L = Lw = whole;
    const GemvTiles t = cut_gemv_tiles(n_out, few, 0.8, &L), w = cut_gemv_tiles(n_out, KT == 1 ? 0 : few, 0.7, &Lw);
    if (t.KT == 0 && w.KT != 0) Lw.tile_us = 0.02 * Lw.W;
    const TcPlan tc = plan_gemv_tc(L);
    const WalkPlan walk = plan_walk(Lw);
    if (tc.ok && tc.rows_per_chunk == f.tc.rows_per_chunk && tc.bt == f.tc.bt) { f.tc = tc; f.tc_tiles = t; }
    if (walk.ok && walk.rows_per_chunk == f.walk.rows_per_chunk && walk.xs == f.walk.xs) { f.walk = walk; f.walk_tiles = w; }
    return f;
}

inline bool take_walk(const GemvLayer &L, const TcPlan &t, const WalkPlan &w)
{
    if (!t.ok || !w.ok) return w.ok;
    return L.n_q == 1 && L.x_bytes == 2 && w.us < WALK_MARGIN * t.us;
}

}  // namespace sqnn
#endif
