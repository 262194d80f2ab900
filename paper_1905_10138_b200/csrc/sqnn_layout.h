// Geometry of the device blob that the host packer and the kernels must agree on: how the
// XOR-gate network's lookup tables are cut into chunks and how slices are grouped into tiles.
// Plain functions, usable from host C++ and from device code.
#ifndef SQNN_LAYOUT_H_
#define SQNN_LAYOUT_H_
#include <stdint.h>

#if defined(__CUDACC__)
#define SQNN_HD __host__ __device__
#else
#define SQNN_HD
#endif

namespace sqnn {

// The network (Section 3.1, w~ = M . w^c) is evaluated with tables: the seed is cut into chunks
// of cb bits and table[chunk][value] holds the XOR of the columns of M selected by the value, as
// an n_out-bit word padded to nwp 32-bit words (bits >= n_out are 0).  Entry (chunk, value)
// starts at word ((chunk << cb) | value) * nwp.
SQNN_HD constexpr uint32_t entry_words(uint32_t n_out) { return (n_out + 31) / 32; }
SQNN_HD constexpr uint32_t entry_words_padded(uint32_t n_out)
{
    return entry_words(n_out) <= 1 ? 1 : entry_words(n_out) <= 2 ? 2 : entry_words(n_out) <= 4 ? 4 : 8;
}
// A kernel may keep several copies of the tables in shared memory, copy j holding all its entries
// in the banks that lane j of a load wavefront owns, so that lookups at unrelated indices never
// collide: 32 / nwp lanes share a wavefront for entries of up to 16 bytes (8 lanes for 32-byte
// entries, read as two halves).  One replicated entry therefore takes 128 bytes (256 for 32-byte
// entries).  The chunking is the coarsest whose replicated tables stay within 128 KB, i.e. at
// most 1024 entries (512 of 32 bytes) over all chunks.
SQNN_HD constexpr uint32_t table_copies(uint32_t nwp) { return nwp >= 4 ? 8 : 32 / nwp; }
SQNN_HD constexpr uint32_t table_chunks(uint32_t n_in, uint32_t nwp)
{
    for (uint32_t c = 1; c <= 8; ++c) {
        uint32_t cb = (n_in + c - 1) / c;
        if (cb <= 10 && c * (1u << cb) <= (nwp == 8 ? 512u : 1024u)) return c;
    }
    return 8;
}
SQNN_HD constexpr uint32_t chunk_bits(uint32_t n_in, uint32_t nwp)
{
    return (n_in + table_chunks(n_in, nwp) - 1) / table_chunks(n_in, nwp);
}
// Words of all tables, rounded to a multiple of 4 (16 bytes).
SQNN_HD constexpr uint32_t table_words(uint32_t n_out, uint32_t n_in)
{
    return (table_chunks(n_in, entry_words_padded(n_out)) * (1u << chunk_bits(n_in, entry_words_padded(n_out))) *
            entry_words_padded(n_out) + 3u) & ~3u;
}

// A format tile is SQNN_TILE_SLICES = 256 consecutive slices: 32 * n_in bytes of seeds, 32 * n_out
// bytes of output, so every tile starts on a 32-byte boundary in both.  Kernels work on kernel
// tiles of 32 lanes x G slices with G * n_out a multiple of 32 bits: G = 8 * kt format tiles,
// kt = 1 when n_out is a multiple of 4, 2 when it is even, 4 otherwise.
SQNN_HD constexpr uint32_t format_tiles_per_kernel_tile(uint32_t n_out)
{
    return (n_out % 4 == 0) ? 1u : (n_out % 2 == 0) ? 2u : 4u;
}

// Run-time shapes: words per lane of a kernel tile that is a part of a format tile, `turns` turns of 32 slices.  Where n_out is no
// multiple of 32 the tile may start inside a slice and overlap one slice more than its length tells, which should not
// cost another turn.
SQNN_HD constexpr uint32_t range_words(uint32_t n_out, uint32_t turns)
{
    return n_out % 32 == 0 ? turns * n_out / 32 : (turns * 32 - 1) * n_out / 1024 ? (turns * 32 - 1) * n_out / 1024 : 1u;
}
// The most turns a part may have.  Large parts are not worth it: their slices wait for one another from turn to turn, where a whole tile's
// are expanded side by side.  The line is a third of the whole (part / whole, us: 3648 x 3072, 33 x 20, three planes, 10 turns of
// 32: 8.6 / 10.6; 5055 x 8957, 50 x 20, 10 of 16: 9.5 / 8.4; 5003 x 7001, 200 x 20, two planes, 4 of 8: 10.1 / 8.7), and a single turn where a
// slice is whole words, which takes no shifting in a whole tile (64 x 16, three planes, product of 1152 x 1664, 2 of 8: 9.9 / 9.5).
// Where n_out is odd that is up to 10 turns, more than a format tile (8).
SQNN_HD constexpr uint32_t most_turns(uint32_t n_out) { return n_out % 32 == 0 ? 1 : 8 * format_tiles_per_kernel_tile(n_out) / 3; }
// Cuts the kernel tiles (W words per lane, KT format tiles each) of a run-time shape smaller if there are idle warps:
// the smallest parts of at most `most` turns with which `fits(words per lane)` still finds a warp for every tile.  Returns the turns, 0 for
// whole tiles.
template <typename F>
inline uint32_t cut_tiles(uint32_t n_out, uint32_t most, uint32_t *KT, uint32_t *W, F fits)
{
    for (uint32_t turns = 1; turns <= most; ++turns) {
        const uint32_t words = range_words(n_out, turns);
        if (words < *W && fits(words)) {
            *KT = 0;
            *W = words;
            return turns;
        }
    }
    return 0;
}

// The decode kernels' tiles.  How many parts an SM may get (0: none): each warp can take one, but every part also costs some hundred
// instructions, which shows where whole tiles keep the schedulers busy already and take little time.  Slices of a
// single lookup do (n_in up to 9 or 10), in tiles of one format tile (n_out a multiple of 4).  Us, whole tiles / as cut / parts for every warp:
//   planes, 1728 x 640, 24 x 7, three planes    3.0 / 3.0 / 3.8      3008 x 2048, 44 x 3     2.9 / 2.9 / 3.9
//           3840 x 3008, 112 x 20               4.9 / 4.9 / 5.6      3390 x 870, 50 x 9      4.2 / 3.6 / 4.4
//           3.3 M weights, 20 x 12              3.5 / 2.9 / 2.9      240 x 16, two planes    5.5 / 4.8 / 5.3
// As the first half of a product with a batch, parts are worth more: 72 x 3, batch 59 13.6 / 11.2 / 11.2; 64 x 8, three planes, batch 94 9.0 / 8.9 / 10.4;
// 112 x 10, two planes, batch 41 7.9 / 7.9 / 10.5; bf16 weights always gain by them (their warps make weights out of what they decode).
// Over 117 random calls for planes and 132 for products, on the line and near it, the rule takes 0.75 and 0.82 of the time of whole tiles; 4 of each are
// more than 3 % slower than with those (by 15 % at most), with parts for every warp 24 and 9 (by 34 and 32 %).
enum class DecodeFor { PLANES, PRODUCT, BF16 };
inline uint32_t most_parts_per_sm(DecodeFor what, uint32_t n_out, uint32_t n_in, uint64_t whole_tiles, uint32_t sms, uint32_t warps)
{
    const uint32_t nwp = entry_words_padded(n_out);
    const bool single = table_chunks(n_in, nwp) == 1, one_tile = format_tiles_per_kernel_tile(n_out) == 1;
    if (what == DecodeFor::BF16) return warps;
    if (what == DecodeFor::PLANES) {
        if (one_tile && whole_tiles >= sms && (single || (whole_tiles >= 2ull * sms && nwp < 8))) return 0;
        return 2 * warps / 3;
    }
    if (one_tile && single && nwp < 8 && whole_tiles >= sms && whole_tiles < 2ull * sms) return 0;
    return single && nwp <= 2 ? 2 * warps / 3 : warps;
}
// words64: 64-bit words of a plane; planes: that are decoded by tiles of their own.
inline uint32_t cut_decode_tiles(DecodeFor what, uint32_t n_out, uint32_t n_in, uint64_t words64, uint32_t planes, uint32_t sms, uint32_t warps,
                                 uint32_t *KT, uint32_t *W)
{
    auto tiles = [&](uint32_t words) { return (words64 + 16ull * words - 1) / (16ull * words) * planes; };
    auto cut = [&](uint32_t per_sm) {
        return cut_tiles(n_out, most_turns(n_out), KT, W, [&](uint32_t words) { return tiles(words) <= (uint64_t)per_sm * sms; });
    };
    const uint32_t turns = cut(most_parts_per_sm(what, n_out, n_in, tiles(*W), sms, warps));
    // whole tiles of several format tiles and lookups are the slowest of all (3648 x 3072, 33 x 20, three planes: 22 parts per SM 8.6, whole 10.6)
    if (turns == 0 && what == DecodeFor::PLANES && format_tiles_per_kernel_tile(n_out) > 1 && table_chunks(n_in, entry_words_padded(n_out)) > 1)
        return cut(warps);
    return turns;
}

// Words of the replicated tables in shared memory.
SQNN_HD constexpr uint32_t table_words_replicated(uint32_t n_out, uint32_t n_in)
{
    return table_chunks(n_in, entry_words_padded(n_out)) * (1u << chunk_bits(n_in, entry_words_padded(n_out))) *
           entry_words_padded(n_out) * table_copies(entry_words_padded(n_out));
}

}  // namespace sqnn
#endif
