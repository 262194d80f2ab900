// Decode kernels (packed bits, bf16 weights, checksum sink) as templates over the network
// shape, with their launchers.
#pragma once
#include "sqnn.h"
#include "sqnn_decode.cuh"
#include "sqnn_launch.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

namespace sqnn {

// ------------------------------------------------------------------------------------------
// shared-memory layout of the warp-tile kernels:  [tables][warp 0: regions][warp 1: ...]...
// a region is a run of 32 * W words (one kernel tile of one plane)
// ------------------------------------------------------------------------------------------
SQNN_DEV uint64_t tile_word64(const uint32_t *region, uint32_t q)
{
    const uint2 v = *reinterpret_cast<const uint2 *>(region + 2 * q);
    return (uint64_t)v.x | ((uint64_t)v.y << 32);
}

template <int N_OUT>
SQNN_DEV uint32_t words_per_lane(const DecodeArgs &A)
{
    if constexpr (N_OUT != 0) return N_OUT / 4;
    else return A.W;
}

// Position of a warp in the list of (plane, tile) items, advanced without division.
struct TilePos {
    uint32_t plane, tile;
};
SQNN_DEV TilePos advance(TilePos p, uint32_t by, uint32_t live, uint32_t n_q)
{
    p.tile += by;
    while (p.plane < n_q && p.tile >= live) { p.tile -= live; ++p.plane; }
    return p;
}

// K1: decoded planes as packed bits.  One kernel tile = 16 * W consecutive uint64 of one plane,
// built in the warp's shared-memory region and written out by a bulk copy while the warp already
// works on its next tile (it waits for the copy only when it is about to overwrite the region).
// Global loads run two tiles ahead: while tile t is expanded, the seeds and the patch offsets of
// tile t + 2 and the patch entries of tile t + 1 (whose offsets arrived an iteration ago) are in
// flight.  REP: the lookup tables sit in shared memory in replicated form (every lane of a load
// wavefront reads its own copy in its own banks); filling them takes a few microseconds, which pays
// once a warp has several tiles to decode.  One block per SM.
// SINK = true: XOR of all those words instead of storing them.  Run-time shapes: REP says that kernel tiles are parts of
// format tiles (KT = 0); two kernels, since the code of both in one costs large layers 1 %.
constexpr uint32_t DECODE_BITS_THREADS = 768;
template <int N_OUT, int N_IN>
inline uint32_t decode_bits_table_words(const DecodeArgs &A, bool rep)
{
    if constexpr (N_OUT != 0) return rep ? table_words_replicated(N_OUT, N_IN) : A.tab_words;
    else return A.tab_words;
}
// ONE_PLANE: the layer has a single plane (its stream pointers are then kernel constants instead of
// being looked up by a plane index in every step).
//
// A small layer (the first half of a product with a batch, a tile or two per warp) is all latency.  What depends on
// the arguments alone is worked out before the wait for the grid ahead or comes from the launcher; the first fetches go out
// before tables and clearing; and a warp without a next tile does not take delivery of its patch entries
// before it expands.
struct BitsArgs {
    uint32_t live;         // tiles that hold at least one real word, per plane
    uint32_t full_tiles;   // tiles before this one lie wholly inside the plane and end on a whole word
};
// Networks with two lookups a slice in tables of four words and more (80 x 16, 200 x 10) need more registers than a thread has.  On large layers they
// spill in worse places with the counts that the launcher hands over and a branch around the deliveries (2^30 weights, us, with / without:
// 200 x 10, S = 0.95 39.4 / 36.3, 0.90 56.4 / 52.6, 0.80 83.9 / 80.2; 80 x 16, S = 0.90 34.0 / 32.1, 0.95 30.1 / 30.5), so there they keep
// the plain form; the others gain 1 % from it (100 x 10, S = 0.95 28.4 / 28.7).
SQNN_HD constexpr bool short_of_registers(uint32_t n_out, uint32_t n_in)
{
    return entry_words_padded(n_out) >= 4 && table_chunks(n_in, entry_words_padded(n_out)) > 1;
}
template <int N_OUT, int N_IN, bool SINK, bool ONE_PLANE, bool REP>
__global__ void __launch_bounds__(DECODE_BITS_THREADS, 1)
k_decode_bits(DecodeArgs A, uint64_t *__restrict__ out, const ClearArgs clear, const BitsArgs B)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const uint32_t W = words_per_lane<N_OUT>(A);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // the tables: replicated ones are filled below, after the first fetches are out
    const uint32_t tab_words_s = N_OUT != 0 && REP ? table_words_replicated(N_OUT, N_IN) : A.tab_words;
    uint32_t *region = smem + tab_words_s + warp * 32 * W;
    const uint64_t tail_bits = A.mn & 63;
    constexpr bool IN_KERNEL = N_OUT != 0 && REP && short_of_registers(N_OUT, N_IN);
    uint32_t live = B.live, full_tiles = B.full_tiles;
    if constexpr (IN_KERNEL) {
        wait_prior_grid();
        launch_dependents();
        live = (uint32_t)((A.words64 + 16 * W - 1) / (16 * W));
        full_tiles = (uint32_t)(A.words64 / (16 * W)) - ((tail_bits != 0 && A.words64 % (16 * W) == 0) ? 1u : 0u);
    }
    const uint32_t stride = gridDim.x * nwarps;
    TilePos p_first = advance(TilePos{0u, 0u}, blockIdx.x * nwarps + warp, live, A.n_q);
    const uint64_t clear_lo = blockIdx.x * clear.per_block;
    uint64_t sink = 0;
    if constexpr (!IN_KERNEL) {
        p_first.plane = settle(p_first.plane);
        p_first.tile = settle(p_first.tile);
        wait_prior_grid();
        launch_dependents();
    }

    auto write_out = [&](TilePos p) {
        uint64_t *pbase = out + (uint64_t)p.plane * A.words64;
        const uint64_t q0 = (uint64_t)p.tile * (16 * W);     // first uint64 of the tile inside the plane
        uint64_t *dst = pbase + q0;
        if (!SINK && p.tile < full_tiles && (reinterpret_cast<uintptr_t>(pbase) & 15) == 0) {
            fence_async_smem();
            __syncwarp();
            if (lane == 0) bulk_store(dst, region, 128 * W);
        } else {
            for (uint32_t q = lane; q < 16 * W; q += 32) {
                if (q0 + q >= A.words64) break;
                uint64_t v = tile_word64(region, q);
                if (q0 + q == A.words64 - 1 && tail_bits) v &= (1ull << tail_bits) - 1ull;
                if constexpr (SINK) sink ^= v; else dst[q] = v;
            }
            __syncwarp();
        }
    };

    // every block clears a run of Y's elements
    auto clear_y = [&] {
        const uint64_t total = clear.m * clear.batch;
        if (clear_lo >= total) return;
        const uint32_t count = (uint32_t)min(clear.per_block, total - clear_lo);
        if (clear.ldy == (int64_t)clear.m) {
            float *y = clear.y + clear_lo;
            uint32_t done = 0;
            if ((reinterpret_cast<uintptr_t>(y) & 15) == 0) {
                done = count & ~3u;
                for (uint32_t i = 4 * threadIdx.x; i < done; i += 4 * blockDim.x) *reinterpret_cast<float4 *>(y + i) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            for (uint32_t i = done + threadIdx.x; i < count; i += blockDim.x) y[i] = 0.0f;
        } else {
            for (uint64_t i = clear_lo + threadIdx.x; i < clear_lo + count; i += blockDim.x) {
                const uint64_t b = i / clear.m;
                clear.y[(int64_t)b * clear.ldy + (int64_t)(i - b * clear.m)] = 0.0f;
            }
        }
    };
    auto plane_of = [&](const TilePos &p) -> const PlanePtrs & { return ONE_PLANE ? A.pl[0] : A.pl[p.plane]; };
    if constexpr (N_OUT != 0) {
        using S = Shape<N_OUT, N_IN>;
        // Three sets of registers take turns as "current", "next" and "the one after": a step works on
        // the current tile while it requests the patch entries of the next (its offsets arrived a step
        // ago) and the seeds and offsets of the one after.  Nothing in flight is ever copied.
        TilePos pa = p_first, pb = advance(pa, stride, live, A.n_q), pc{A.n_q, 0u};
        TileSeeds<N_OUT, N_IN> sa, sb, sc;
        TileRun ra{0u, 0u}, rb{0u, 0u}, rc{0u, 0u};
        uint32_t wa[PATCH_AHEAD], wb[PATCH_AHEAD], wc[PATCH_AHEAD];
        if (pa.plane < A.n_q) { fetch_seeds<N_OUT, N_IN>(plane_of(pa), pa.tile, lane, sa); ra = fetch_run(plane_of(pa), pa.tile); }
        if (pb.plane < A.n_q) { fetch_seeds<N_OUT, N_IN>(plane_of(pb), pb.tile, lane, sb); rb = fetch_run(plane_of(pb), pb.tile); }
        if constexpr (REP) tables_replicate<entry_words_padded(N_OUT)>(A, smem);
        else tables_request(A, smem);
        if (clear.batch) clear_y();
        if (pa.plane < A.n_q) fetch_patches(A, plane_of(pa), ra, lane, wa);
        if constexpr (!REP) cp_async_wait_all();
        __syncthreads();                                 // the tables are in place
        auto step = [&](TilePos &p0, TileSeeds<N_OUT, N_IN> &s0, TileRun &r0, uint32_t (&w0)[PATCH_AHEAD],
                        TilePos &p1, TileRun &r1, uint32_t (&w1)[PATCH_AHEAD],
                        TilePos &p2, TileSeeds<N_OUT, N_IN> &s2, TileRun &r2) {
            if (IN_KERNEL || p1.plane < A.n_q) {
                // everything this step consumes was requested at least a step ago: take delivery of it now,
                // before the loads of this step are issued
#pragma unroll
                for (uint32_t k = 0; k < S::NRAW; ++k) s0.raw[k] = settle(s0.raw[k]);
#pragma unroll
                for (uint32_t k = 0; k < PATCH_AHEAD; ++k) w0[k] = settle(w0[k]);
                r0.base = settle(r0.base); r0.end = settle(r0.end);
                r1.base = settle(r1.base); r1.end = settle(r1.end);
            }
            p2 = advance(p1, stride, live, A.n_q);
            if (p1.plane < A.n_q) fetch_patches(A, plane_of(p1), r1, lane, w1);
            if (p2.plane < A.n_q) { fetch_seeds<N_OUT, N_IN>(plane_of(p2), p2.tile, lane, s2); r2 = fetch_run(plane_of(p2), p2.tile); }
            tile_expand<N_OUT, N_IN, !SINK, REP>(s0, region, smem, lane);
            __syncwarp();
            tile_patch(A, plane_of(p0), r0, w0, region, S::TILE_BITS, lane);
            __syncwarp();
            write_out(p0);
            return p1.plane < A.n_q;
        };
        if (pa.plane < A.n_q) {
            for (;;) {
                if (!step(pa, sa, ra, wa, pb, rb, wb, pc, sc, rc)) break;
                if (!step(pb, sb, rb, wb, pc, rc, wc, pa, sa, ra)) break;
                if (!step(pc, sc, rc, wc, pa, ra, wa, pb, sb, rb)) break;
            }
        }
    } else {
        tables_request(A, smem);
        if (clear.batch) clear_y();
        cp_async_wait_all();
        __syncthreads();
        for (TilePos p = p_first; p.plane < A.n_q; p = advance(p, stride, live, A.n_q)) {
            if (!SINK && lane == 0) bulk_wait_read<0>();         // the copy out of the region is over
            __syncwarp();
            if constexpr (REP) decode_range(A, p.plane, p.tile, region, smem, lane);
            else decode_whole_tiles(A, p.plane, p.tile, region, smem, lane);
            write_out(p);
        }
    }
    if constexpr (SINK) {
#pragma unroll
        for (uint32_t d = 16; d >= 1; d >>= 1) sink ^= __shfl_xor_sync(0xffffffffu, sink, d);
        if (lane == 0 && sink) atomicXor(reinterpret_cast<unsigned long long *>(out), (unsigned long long)sink);
    } else {
        if (lane == 0) bulk_wait_read<0>();              // shared memory must outlive the copies
    }
}

// Starts the copy of `words` mask words (first word gw0) into shared memory: 16-byte
// asynchronous copies where a whole vector is in range, plain loads (zero past the end) otherwise.
// `words` is a multiple of 4 and gw0 a multiple of 4.  The calling threads are `nthreads` threads
// numbered `t`.  Finish with a cp.async wait and a barrier over those threads.
SQNN_DEV void stage_mask(uint32_t *mask_s, const uint32_t *__restrict__ mask32, uint64_t gw0, uint64_t mask_words,
                         uint32_t words, uint32_t t, uint32_t nthreads, bool vec_ok)
{
    for (uint32_t v = t; v < words / 4; v += nthreads) {
        if (vec_ok && gw0 + 4 * v + 4 <= mask_words) {
            cp_async16(mask_s + 4 * v, mask32 + gw0 + 4 * v);
        } else {
#pragma unroll
            for (uint32_t e = 0; e < 4; ++e)
                mask_s[4 * v + e] = gw0 + 4 * v + e < mask_words ? __ldg(mask32 + gw0 + 4 * v + e) : 0u;
        }
    }
}

// K2: decoded, masked, rescaled weights as bf16.  A lane takes 32 weights (one word of every plane and of the mask)
// at a time and writes them as 64 bytes of a 2 KB buffer of its warp, which leaves by a bulk copy while the
// next one is filled.
//
// With up to three planes a weight is 0 or +-V[a], where the sign is plane 0's bit and a says which of the other
// planes disagree with it: at most four bf16 values per row, eight bytes, from which one byte permutation picks
// two weights.  Mask and sign bits, moved to the top of a half word, are the bf16 numbers 0, 2 and -2, so a
// multiply-add with V / 2 does the rest.  Selectors and those numbers come out of words in which even and odd
// columns have been separated, by a shift and an AND each: 3 instructions per weight with three planes.  What surrounds
// that -- words, separation, staging, copies, row bookkeeping -- takes nearly four more: 2^26 weights of three planes
// take 37 us and 21.8 M warp instructions, of which 7.3 M are the decode.  (Sums of the scales per weight took about 20
// instructions, and 64 us.)  Negating all terms of a sum
// negates it exactly, except when it is zero or not finite, and halving is exact except for the tiniest
// numbers; rows with such a value take the plain loop, as do rows of less than 32 weights and layers of four and
// more planes.  A lane whose 32 weights straddle two rows makes them for both and keeps the second row's from its first column on
// (with the straddling chunk weight by weight 5516 x 1166, three planes, 60 x 12 takes 15.9 us, 13.1 so).
// One block per SM, as many warps as shared memory holds, fewer where a lane's entries need the registers.
SQNN_HD constexpr uint32_t bf16_threads(uint32_t n_out) { return n_out > 128 ? 512 : 768; }
constexpr uint32_t BF16_STAGE_WORDS = 2 * 512;           // two buffers of 2 KB per warp

// Half the bf16 values of a row: V[0] | V[1] << 16, V[2] | V[3] << 16; plain: see above.
template <typename IT>
struct RowValues {
    IT row;
    uint32_t v0, v1;
    bool plain;
};
template <int NQ, typename IT>
SQNN_DEV RowValues<IT> row_values(const float *__restrict__ alpha, IT r)
{
    static_assert(NQ >= 1 && NQ <= 3, "up to four values");
    RowValues<IT> t{r, 0u, 0u, false};
    float a[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < NQ; ++i) a[i] = __ldg(alpha + (uint64_t)r * NQ + i);
    uint32_t h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        float s = a[0];
        if constexpr (NQ >= 2) s = __fadd_rn(s, (e & 1) ? -a[1] : a[1]);
        if constexpr (NQ >= 3) s = __fadd_rn(s, (e & 2) ? -a[2] : a[2]);
        if (!(fabsf(s) > 1e-36f && fabsf(s) < 1e38f)) t.plain = true;
        h[e] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(s)) - 0x0080u;       // exponent less one
    }
    t.v0 = __byte_perm(h[0], h[1], 0x5410);
    t.v1 = __byte_perm(h[2], h[3], 0x5410);
    return t;
}

// a * b + 0 on two bf16 numbers (the + 0 turns -0 into 0)
SQNN_DEV uint32_t bf16x2_mul0(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(0u));
    return r;
}

// 16 columns as eight words of two bf16.  zm: even columns' (mask, minus) bit pairs in the low half, odd ones'
// in the high half; qe: bytes even 0-7, odd 0-7, even 8-15, odd 8-15 of (e1, e2) pairs, e_i = plane i differs
// from plane 0.
template <int NQ, typename IT>
SQNN_DEV void weights16(uint32_t zm, uint32_t qe, const RowValues<IT> &t, uint32_t (&out)[8])
{
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        uint32_t lo, hi;
        if constexpr (NQ >= 2) {
            const uint32_t sel = ((qe >> (2 * j)) & 0x03030303u) * 0x22u + 0x10101010u;
            lo = __byte_perm(t.v0, t.v1, sel);
            hi = __byte_perm(t.v0, t.v1, sel >> 16);
        } else {
            lo = hi = t.v0;                                      // V[0] = V[1]
        }
        out[j] = bf16x2_mul0(lo, (zm << (14 - 2 * j)) & 0xc000c000u);                  // columns 2 j, 2 j + 1
        out[j + 4] = bf16x2_mul0(hi, (zm << (6 - 2 * j)) & 0xc000c000u);               // columns 8 + 2 j, 9 + 2 j
    }
}

// Run-time shapes: N_IN = 1 says that kernel tiles are parts of format tiles (KT = 0).
// ENDS: rows may end inside a lane's 32 weights (n no multiple of 32; kernels of their own, since it costs the others 5 to 15 %).  1: such a lane
// makes them twice; 2: it goes through them in chunks of 8 and weight by weight, for long rows, where few lanes do and the
// registers of the other way cost more (LONG_ROWS).
template <int N_OUT, int N_IN, int NQ, int ENDS>
__global__ void __launch_bounds__(bf16_threads(N_OUT), 1)
k_decode_bf16(DecodeArgs A, const uint32_t *__restrict__ mask32, const float *__restrict__ alpha,
              uint64_t n64, __nv_bfloat16 *__restrict__ out)
{
    using IT = typename std::conditional<NQ != 0, uint32_t, uint64_t>::type;       // rows and columns
    extern __shared__ __align__(16) uint32_t smem[];
    wait_prior_grid();
    launch_dependents();
    tables_request(A, smem);
    const IT n = (IT)n64;
    const uint32_t W = words_per_lane<N_OUT>(A);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint32_t ktiles = (uint32_t)((A.mn + (uint64_t)W * 1024 - 1) / ((uint64_t)W * 1024)), stride = gridDim.x * nwarps;
    // All planes' seeds and patch runs of a tile are requested together, the first tile's ahead of the tables and
    // every other tile's before the weights of the one before it are made; then all its patch entries.
    constexpr bool AHEAD = N_OUT != 0 && NQ != 0;
    constexpr int NF = AHEAD ? NQ : 1;
    TileSeeds<AHEAD ? N_OUT : 40, AHEAD ? N_IN : 12> seeds[NF];
    TileRun run[NF];
    auto request = [&](uint32_t tile) {
        if constexpr (AHEAD) {
            if (tile < ktiles) {
#pragma unroll
                for (int i = 0; i < NQ; ++i) {
                    run[i] = fetch_run(A.pl[i], tile);
                    fetch_seeds<N_OUT, N_IN>(A.pl[i], tile, lane, seeds[i]);
                }
            }
        }
    };
    const uint32_t first = blockIdx.x * nwarps + warp;
    request(first);
    cp_async_wait_all();
    __syncthreads();
    const uint32_t n_q = NQ ? NQ : A.n_q;
    uint32_t *region = smem + A.tab_words + warp * (n_q * 32 * W + BF16_STAGE_WORDS);
    uint32_t *stage = region + n_q * 32 * W;
    // A lane's four chunks of 8 weights are produced in an order that starts at `turn`, so that the 16-byte stores
    // of eight neighbouring lanes fall into different banks.
    const uint32_t turn = (lane >> 1) & 3u;
    uint32_t buf = 0;
    RowValues<IT> t{(IT)~0ull, 0u, 0u, true};
    for (uint32_t tile = first; tile < ktiles; tile += stride) {
        const uint64_t p_tile = tile * (uint64_t)W * 1024;
        const uint32_t here = A.mn - p_tile < (uint64_t)W * 1024 ? (uint32_t)(A.mn - p_tile) : W * 1024;   // weights of this tile
        const uint64_t p_lane = p_tile + 32ull * lane, r64 = p_lane / n64;
        IT r = (IT)r64, c = (IT)(p_lane - r64 * n64);            // row and column of the lane's first weight
        const uint32_t *mp = mask32 + (uint64_t)tile * 32 * W + lane;      // this lane's mask words: those below `here`
        uint32_t m_next = 32 * lane < here ? __ldg(mp) : 0u;
        if constexpr (AHEAD) {
            using S = Shape<N_OUT, N_IN>;
            uint32_t pw[NQ][PATCH_AHEAD];
#pragma unroll
            for (int i = 0; i < NQ; ++i) fetch_patches(A, A.pl[i], run[i], lane, pw[i]);
#pragma unroll
            for (int i = 0; i < NQ; ++i) tile_expand<N_OUT, N_IN>(seeds[i], region + i * 32 * W, smem, lane);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NQ; ++i) tile_patch(A, A.pl[i], run[i], pw[i], region + i * 32 * W, S::TILE_BITS, lane);
            __syncwarp();
            request(tile + stride);
        } else {
            for (uint32_t i = 0; i < n_q; ++i)
                decode_warp_tile<N_OUT, N_IN>(A, i, tile, region + i * 32 * W, smem, lane);
        }
        __nv_bfloat16 *to_g = out + p_tile;
        const uint32_t *bits = region + lane;
        for (uint32_t at = 0; at < here; at += 1024, bits += 32, to_g += 1024) {
            const uint32_t m = m_next;
            mp += 32;
            if (at + 1024 + 32 * lane < here) m_next = __ldg(mp); else m_next = 0u;
            uint32_t *to = stage + buf * 512 + lane * 16;
            if (lane == 0) bulk_wait_read<1>();                  // the copy out of this buffer is over
            __syncwarp();
            bool fast = false;
            if constexpr (NQ != 0) {
                // the next row begins inside the lane's 32 weights
                const bool next = ENDS == 1 && n - c < 32 && at + 32 * lane + (uint32_t)(n - c) < here;
                RowValues<IT> t2 = t;
                if ((ENDS == 0 || (ENDS == 1 ? n : n - c) >= 32) && at + 32 * lane < here) {
                    if (r != t.row) t = row_values<NQ, IT>(alpha, r);
                    fast = !t.plain;
                    if (next) {
                        t2 = row_values<NQ, IT>(alpha, r + 1);
                        fast = fast && !t2.plain;
                    }
                }
                if (fast) {
                    const uint32_t b0 = bits[0], sgn = ~b0;
                    // rotated so that chunk `turn` comes first
                    const uint32_t mr = __funnelshift_r(m, m, 8 * turn), sr = __funnelshift_r(sgn, sgn, 8 * turn);
                    const uint32_t me = (mr & 0x55555555u) | ((sr << 1) & 0xaaaaaaaau), mo = ((mr >> 1) & 0x55555555u) | (sr & 0xaaaaaaaau);
                    uint32_t qe = 0, qo = 0;
                    if constexpr (NQ >= 2) {
                        uint32_t e1 = b0 ^ bits[32 * W], e2 = 0;
                        if constexpr (NQ >= 3) e2 = b0 ^ bits[64 * W];
                        e1 = __funnelshift_r(e1, e1, 8 * turn);
                        e2 = __funnelshift_r(e2, e2, 8 * turn);
                        qe = (e1 & 0x55555555u) | ((e2 << 1) & 0xaaaaaaaau);
                        qo = ((e1 >> 1) & 0x55555555u) | (e2 & 0xaaaaaaaau);
                    }
#pragma unroll
                    for (uint32_t h = 0; h < 2; ++h) {           // 16 weights: chunks 2 h and 2 h + 1 of the rotated word
                        uint32_t o[8];
                        weights16<NQ, IT>(__byte_perm(me, mo, h ? 0x7632 : 0x5410), __byte_perm(qe, qo, h ? 0x7362 : 0x5140), t, o);
                        *reinterpret_cast<uint4 *>(to + 4 * ((2 * h + turn) & 3u)) = make_uint4(o[0], o[1], o[2], o[3]);
                        *reinterpret_cast<uint4 *>(to + 4 * ((2 * h + 1 + turn) & 3u)) = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                    if (next) {                                  // once more with the next row's values, from its first column on
                        const uint32_t k = (uint32_t)(n - c);
#pragma unroll
                        for (uint32_t h = 0; h < 2; ++h) {
                            uint32_t o[8];
                            weights16<NQ, IT>(__byte_perm(me, mo, h ? 0x7632 : 0x5410), __byte_perm(qe, qo, h ? 0x7362 : 0x5140), t2, o);
#pragma unroll
                            for (uint32_t j = 0; j < 8; ++j) {
                                const uint32_t word = 4 * ((2 * h + j / 4 + turn) & 3u) + j % 4;
                                if (2 * word >= k) to[word] = o[j];
                                else if (2 * word + 1 == k) to[word] = __byte_perm(to[word], o[j], 0x7610);
                            }
                        }
                        t = t2;
                    }
                }
            }
            if (!fast) {
                IT rr = r, cc = c;
#pragma unroll 1
                for (uint32_t ch = 0; ch < 4 && at + 32 * lane + 8 * ch < here; ++ch) {      // chunks of 8 weights
                    while (cc >= n) { cc -= n; ++rr; }
                    const uint32_t mk = (m >> (8 * ch)) & 0xffu;
                    if constexpr (NQ != 0) {
                        if (n - cc >= 8) {                       // one row
                            if (rr != t.row) t = row_values<NQ, IT>(alpha, rr);
                            if (!t.plain) {
                                const uint32_t b0 = bits[0] >> (8 * ch), sr = ~b0;
                                uint32_t e1 = 0, e2 = 0;
                                if constexpr (NQ >= 2) e1 = b0 ^ (bits[32 * W] >> (8 * ch));
                                if constexpr (NQ >= 3) e2 = b0 ^ (bits[64 * W] >> (8 * ch));
                                const uint32_t me = (mk & 0x55u) | ((sr << 1) & 0xaau), mo = ((mk >> 1) & 0x55u) | (sr & 0xaau);
                                const uint32_t qe = (e1 & 0x55u) | ((e2 << 1) & 0xaau), qo = ((e1 >> 1) & 0x55u) | (e2 & 0xaau);
                                uint32_t o[8];
                                weights16<NQ, IT>(me | (mo << 16), qe | (qo << 8), t, o);
                                *reinterpret_cast<uint4 *>(to + 4 * ch) = make_uint4(o[0], o[1], o[2], o[3]);
                                cc += 8;
                                continue;
                            }
                        }
                    }
#pragma unroll 1
                    for (uint32_t k = 0; k < 8 && at + 32 * lane + 8 * ch + k < here; ++k) {
                        while (cc >= n) { cc -= n; ++rr; }
                        float sum = 0.0f;
                        if ((mk >> k) & 1u)
                            for (uint32_t i = 0; i < n_q; ++i) {
                                const float a = __ldg(alpha + (uint64_t)rr * n_q + i);
                                const float term = ((bits[i * 32 * W] >> (8 * ch + k)) & 1u) ? a : -a;
                                sum = i == 0 ? term : __fadd_rn(sum, term);
                            }
                        reinterpret_cast<__nv_bfloat16 *>(to)[8 * ch + k] = __float2bfloat16_rn(sum);
                        ++cc;
                    }
                }
            }
            if (at + 1024 <= here) {
                fence_async_smem();
                __syncwarp();
                if (lane == 0) bulk_store(to_g, stage + buf * 512, 2048);
            } else {                                             // the last weights, one by one
                __syncwarp();
                const __nv_bfloat16 *from = reinterpret_cast<const __nv_bfloat16 *>(stage + buf * 512);
                for (uint32_t k = lane; at + k < here; k += 32) to_g[k] = from[k];
                __syncwarp();
            }
            buf ^= 1u;
            c += 1024;
            if (c >= n) {
                if (n > 1024) { c -= n; ++r; }
                else { const uint32_t q = (uint32_t)c / (uint32_t)n; c -= (IT)(q * (uint32_t)n); r += q; }
            }
        }
        __syncwarp();
    }
    if (lane == 0) bulk_wait_read<0>();                          // shared memory must outlive the copies
}

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------
// Columns from which on the compile-time shapes up to 128 bits with two or three planes take the plain way through lanes that straddle rows (twice
// / plain, us: 100 x 10, two, 4115 x 7228 22.2 / 19.9, 7026 x 13601 64.5 / 61.8; 40 x 12, three, 1419 x 6628 12.5 / 11.7; 40 x 16, two, 1121 x 6499
// 11.9 / 11.1; 80 x 8, two, 21341 x 5172 61.4 / 64.6; 60 x 12, two, 6052 x 4843 18.5 / 19.8).  With one plane the registers suffice: 40 x 12,
// 1855 x 6535 8.7 / 9.5; 100 x 10, 4465 x 4259 16.7 / 20.3.
constexpr uint64_t LONG_ROWS = 6144;
constexpr uint64_t CLEAR_PER_BLOCK = 4096;               // elements of Y that are worth a block

// A layer with fewer tiles than all SMs have warps: as many blocks as SMs with as few warps as that takes.
inline uint32_t spread_warps(uint64_t tiles, uint32_t most)
{
    const uint64_t share = (tiles + sm_count() - 1) / sm_count();
    const uint32_t want = share > 4 ? (share < most ? (uint32_t)share : most) : 4u;
    return want < most ? want : most;
}

inline uint32_t grid_for(uint64_t warp_tiles, uint32_t warps, uint32_t blocks_per_sm)
{
    uint64_t need = (warp_tiles + warps - 1) / warps;
    uint64_t cap = (uint64_t)sm_count() * blocks_per_sm;
    if (need < 1) need = 1;
    return (uint32_t)(need < cap ? need : cap);
}

template <int N_OUT, int N_IN>
inline int launch_decode(const DecodeArgs &A0, sqnn_out_mode mode, const uint64_t *d_mask,
                         const float *d_alpha, uint64_t n, void *d_out, const ClearArgs &clear,
                         cudaStream_t st)
{
    size_t smem = 0;
    DecodeArgs A = A0;
    if constexpr (N_OUT == 0) {
        const DecodeFor what = mode == SQNN_OUT_BF16 ? DecodeFor::BF16 : clear.batch ? DecodeFor::PRODUCT : DecodeFor::PLANES;
        const uint32_t planes = mode == SQNN_OUT_BF16 ? 1 : A.n_q;       // a warp takes a tile of one plane or of all
        cut_decode_tiles(what, A.n_out, A.n_in, A.words64, planes, (uint32_t)sm_count(), DECODE_BITS_THREADS / 32, &A.KT, &A.W);
    }
    if (mode == SQNN_OUT_BITS || mode == SQNN_OUT_SINK) {
        // one block per SM: the tables and one region per warp.  The replicated tables are worth their
        // fill only when a warp gets several tiles.
        const uint64_t live = (A.words64 + 16ull * A.W - 1) / (16ull * A.W);
        if (live * A.n_q >= (1ull << 31)) return SQNN_E_UNSUPPORTED;
        const bool rep = N_OUT == 0 ? A.KT == 0 : live * A.n_q >= 3ull * (DECODE_BITS_THREADS / 32) * (uint64_t)sm_count();
        const size_t tab = (size_t)decode_bits_table_words<N_OUT, N_IN>(A, rep) * 4, per_warp = (size_t)32 * A.W * 4;
        const size_t limit = 224 * 1024;
        if (tab + per_warp > limit) return SQNN_E_UNSUPPORTED;
        uint32_t warps = (uint32_t)((limit - tab) / per_warp);
        if (warps > DECODE_BITS_THREADS / 32) warps = DECODE_BITS_THREADS / 32;
        warps = spread_warps(live * A.n_q, warps);
        smem = tab + warps * per_warp;
        uint32_t grid = grid_for(live * A.n_q, warps, 1);
        // Blocks without a tile clear their share of Y: a small layer with a large batch has few tiles and a large Y (2240 x 896,
        // 80 x 8, batch 388: 25 blocks for 3.5 MB, 28.4 us; 13.6 with 148).
        const uint64_t clear_blocks = (clear.m * clear.batch + CLEAR_PER_BLOCK - 1) / CLEAR_PER_BLOCK;
        if (clear_blocks > grid) grid = clear_blocks < (uint64_t)sm_count() ? (uint32_t)clear_blocks : (uint32_t)sm_count();
        const uint64_t whole = A.words64 / (16ull * A.W);
        const BitsArgs B{(uint32_t)live, (uint32_t)(whole - (A.mn % 64 != 0 && whole * 16 * A.W == A.words64 ? 1 : 0))};
        ClearArgs c = clear;
        c.per_block = ((clear.m * clear.batch + grid - 1) / grid + 3) & ~3ull;             // on 16-byte boundaries
#define SQNN_BITS_LAUNCH2(SINKV, ONEV, REPV)                                                             \
    do {                                                                                                 \
        auto k = k_decode_bits<N_OUT, N_IN, SINKV, ONEV, REPV>;                                          \
        return launch_kernel(k, grid, warps * 32, smem, st, A, (uint64_t *)d_out, c, B);                 \
    } while (0)
#define SQNN_BITS_LAUNCH(SINKV, ONEV)                                                                    \
    do {                                                                                                 \
        if (rep) SQNN_BITS_LAUNCH2(SINKV, ONEV, true); else SQNN_BITS_LAUNCH2(SINKV, ONEV, false);       \
    } while (0)
        if (mode == SQNN_OUT_BITS) {
            if (A.n_q == 1) SQNN_BITS_LAUNCH(false, true); else SQNN_BITS_LAUNCH(false, false);
        } else {
            if (cudaMemsetAsync(d_out, 0, 8, st) != cudaSuccess) return SQNN_E_CUDA;
            if (A.n_q == 1) SQNN_BITS_LAUNCH(true, true); else SQNN_BITS_LAUNCH(true, false);
        }
#undef SQNN_BITS_LAUNCH2
#undef SQNN_BITS_LAUNCH
    } else {
        const size_t limit = 224 * 1024, tab = (size_t)A.tab_words * 4, per_warp = (size_t)(A.n_q * 32 * A.W + BF16_STAGE_WORDS) * 4;
        if (tab + per_warp > limit) return SQNN_E_UNSUPPORTED;
        const uint64_t live = (A.words64 * 2 + 32ull * A.W - 1) / (32ull * A.W);
        if (live >= (1ull << 31)) return SQNN_E_UNSUPPORTED;
        const uint32_t warps = spread_warps(live, (uint32_t)std::min<size_t>((limit - tab) / per_warp, bf16_threads(N_OUT) / 32));
        smem = tab + warps * per_warp;
        const uint32_t grid = grid_for(live, warps, 1);
        const bool ends = n % 32 != 0;
        constexpr bool LONG = N_OUT != 0 && N_OUT <= 128;
#define SQNN_BF16_LAUNCH2(NQV, PARTSV)                                                                   \
    do {                                                                                                 \
        auto k = ends ? k_decode_bf16<N_OUT, N_OUT ? N_IN : PARTSV, NQV, NQV != 0>                       \
                      : k_decode_bf16<N_OUT, N_OUT ? N_IN : PARTSV, NQV, 0>;                             \
        if constexpr (LONG && NQV >= 2) if (ends && n >= LONG_ROWS) k = k_decode_bf16<N_OUT, N_IN, NQV, 2>; \
        return launch_kernel(k, grid, warps * 32, smem, st, A, (const uint32_t *)d_mask, d_alpha, n, (__nv_bfloat16 *)d_out); \
    } while (0)
#define SQNN_BF16_LAUNCH(NQV)                                                                            \
    do {                                                                                                 \
        if (N_OUT == 0 && A.KT == 0) SQNN_BF16_LAUNCH2(NQV, 1); else SQNN_BF16_LAUNCH2(NQV, 0);          \
    } while (0)
        if (n >= (1ull << 31) || A.mn / n >= (1ull << 31)) SQNN_BF16_LAUNCH(0);       // 64-bit rows and columns
        else if (A.n_q == 1) SQNN_BF16_LAUNCH(1);
        else if (A.n_q == 2) SQNN_BF16_LAUNCH(2);
        else if (A.n_q == 3) SQNN_BF16_LAUNCH(3);
        else SQNN_BF16_LAUNCH(0);
#undef SQNN_BF16_LAUNCH
#undef SQNN_BF16_LAUNCH2
    }
    return cudaGetLastError() == cudaSuccess ? SQNN_OK : SQNN_E_CUDA;
}

// One network shape = one translation unit (sqnn_shape.cu compiled with -DSQNN_NO / -DSQNN_NI).
template <int N_OUT, int N_IN>
int decode_shape(const DecodeArgs &A, sqnn_out_mode mode, const uint64_t *d_mask, const float *d_alpha,
                 uint64_t n, void *d_out, const ClearArgs &clear, cudaStream_t st);
template <int N_OUT, int N_IN>
int gemv_shape(const DecodeArgs &A, const uint64_t *d_mask, const float *d_alpha, const void *d_x, int x_dtype,
               int64_t ldx, uint32_t batch, float *d_y, int64_t ldy, uint64_t m, uint64_t n, cudaStream_t st);

}  // namespace sqnn
