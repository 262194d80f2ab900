// Device-side decryption of one warp tile: seeds -> XOR-gate network (table lookup) ->
// patch flips, producing a run of consecutive output words in shared memory.
//
// Work split.  A kernel tile is 32 * W consecutive 32-bit words of the flattened plane, decoded by a warp.
// As a rule it is KT format tiles (256 slices), KT chosen so that 8 * KT * n_out is a multiple of 32 bits: a lane owns 8 * KT
// consecutive slices, whose W output words are private to it while it expands; in the seed stream a lane's 8 slices of
// one format tile are n_in consecutive bytes.  (Shapes with compile-time kernels have KT = 1.)  In small layers of other
// shapes it is a run of a few turns of 32 slices, wherever it starts, so that more warps have something to decode: see decode_range.
//
// The network (Section 3.1, w~ = M . w^c) is evaluated with the lookup tables stored in the
// blob (geometry in sqnn_layout.h), copied to shared memory once per block.
//
// Patches (Section 3.2) come per format tile as 16-bit bit positions inside the tile; the warp
// flips them in the shared-memory copy of the tile with one shared-memory reduction each, lanes
// taking entries in turn -- no counts, no prefix sum.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "sqnn.h"
#include "sqnn_layout.h"

#define SQNN_DEV __device__ __forceinline__

namespace sqnn {

struct PlanePtrs {
    const uint32_t *wc;    // seed stream
    const uint32_t *idx;   // patch entries before each format tile (+ closing entry)
    const uint16_t *pp;    // patch entries: bit position inside the format tile
    uint32_t n_pp;
};

struct DecodeArgs {
    uint64_t mn;           // weights per plane
    uint64_t words64;      // ceil(mn / 64)
    uint64_t slices;       // slices per plane that hold weights
    uint64_t inv_n_out;    // floor(2^64 / n_out) + 1: the upper half of its product with a bit position (< 2^40) is the slice (n_out > 1)
    uint32_t n_out, n_in, n_q;
    uint32_t KT;           // format tiles per kernel tile; 0: a kernel tile is a part of one (run-time shapes, small layers)
    uint32_t W;            // words of a kernel tile per lane
    uint32_t nw, nwp;      // words per table entry: used, padded (1, 2, 4, 8)
    uint32_t nchunks, cb;  // table chunks, bits per chunk
    uint32_t tab_words;    // words of all tables (multiple of 4)
    const uint32_t *tab;   // tables in the blob
    uint32_t *status;      // sticky error word or NULL
    PlanePtrs pl[8];
};

// Rows of Y the decode kernel clears for the product kernel that follows it (batch 0: nothing).
struct ClearArgs {
    float *y;
    uint64_t m;
    int64_t ldy;
    uint32_t batch;
    uint64_t per_block;    // elements a block clears, counted without the gaps between rows (set by the launcher)
};

// Programmatic dependent launch.  A kernel of this library may be scheduled before the kernel queued ahead of
// it has finished; wait_prior_grid() returns once that one is complete and its results are visible.  Nothing in
// global memory is read or written before it, with one exception: k_decode_mma reads activations and mask ahead of its
// wait.  The decode kernel queued just before it lets it in after its own wait, so whatever was queued before the
// two is complete by then.  launch_dependents() lets the next kernel in, which waits in turn for all of this one.
SQNN_DEV void wait_prior_grid() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
SQNN_DEV void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

SQNN_DEV void flag(uint32_t *status, uint32_t code)
{
    if (status) atomicMax(status, code);
}

SQNN_DEV uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Asynchronous copy shared -> global by the bulk-copy engine; 16-byte aligned, size % 16 == 0.
SQNN_DEV void bulk_store(void *gdst, const void *ssrc, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n"
                 :: "l"(gdst), "r"(smem_addr(ssrc)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
// Waits until at most PENDING of this thread's bulk copies still read their shared source.
template <int PENDING>
SQNN_DEV void bulk_wait_read()
{
    asm volatile("cp.async.bulk.wait_group.read %0;\n" :: "n"(PENDING) : "memory");
}
SQNN_DEV void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

SQNN_DEV void cp_async16(void *sdst, const void *gsrc)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" :: "r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
SQNN_DEV void cp_async4(void *sdst, const void *gsrc)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" :: "r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}
SQNN_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int PENDING>
SQNN_DEV void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;\n" :: "n"(PENDING) : "memory"); }
SQNN_DEV void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Read-only global loads that stay where they are written: the compiler may not move a volatile asm
// statement past another one, so a load issued ahead of time is not sunk down to its first use.
SQNN_DEV uint32_t ldg_ahead(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
SQNN_DEV uint2 ldg_ahead(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
SQNN_DEV uint4 ldg_ahead(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// Makes the warp wait here for a value loaded earlier (a volatile register move reads it).  Used before
// new loads are issued: the few scoreboards a warp has are shared between loads, so a register whose
// load finished long ago can otherwise end up waiting for loads issued just before its first use.
SQNN_DEV uint32_t settle(uint32_t v)
{
    uint32_t r;
    asm volatile("mov.u32 %0, %1;" : "=r"(r) : "r"(v));
    return r;
}

// Starts the copy of the lookup tables from the blob into shared memory (all threads of the
// block; one commit group).  Wait for the group and pass a block barrier before the first lookup.
SQNN_DEV void tables_request(const DecodeArgs &A, uint32_t *tab_s)
{
    for (uint32_t v = threadIdx.x; v < A.tab_words / 4; v += blockDim.x) cp_async16(tab_s + 4 * v, A.tab + 4 * v);
    cp_async_commit();
}

// The same tables, replicated for conflict-free lookups (sqnn_layout.h): element (entry e, copy j)
// -- for 32-byte entries (entry e, half h, copy j) -- is stored at consecutive 16-byte (or smaller)
// slots in the order of its linear index, so the fill is a coalesced copy in which 32 / NWP
// consecutive threads store the same entry.  All threads of the block; ends without a barrier.
template <int NWP>
SQNN_DEV void tables_replicate(const DecodeArgs &A, uint32_t *tab_s)
{
    constexpr uint32_t R = table_copies(NWP);
    constexpr uint32_t VW = NWP >= 4 ? 4 : NWP;                  // words per stored element (16, 8 or 4 bytes)
    constexpr uint32_t PER = 32 / R;                             // source elements one warp store covers
    const uint32_t elems = (A.nchunks << A.cb) * (NWP / VW);     // source elements (halves count separately)
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // a warp takes 32 source elements at a time: one coalesced load, then R stores of 32 consecutive
    // replicated elements each, the values handed round by shuffles
    for (uint32_t e0 = warp * 32; e0 < elems; e0 += nwarps * 32) {
        uint32_t v[VW];
#pragma unroll
        for (uint32_t k = 0; k < VW; ++k) v[k] = 0;
        if (e0 + lane < elems) {
            if constexpr (VW == 4) {
                const uint4 t = __ldg(reinterpret_cast<const uint4 *>(A.tab + 4 * (e0 + lane)));
                v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
            } else if constexpr (VW == 2) {
                const uint2 t = __ldg(reinterpret_cast<const uint2 *>(A.tab + 2 * (e0 + lane)));
                v[0] = t.x; v[1] = t.y;
            } else {
                v[0] = __ldg(A.tab + e0 + lane);
            }
        }
#pragma unroll
        for (uint32_t j = 0; j < R; ++j) {
            const uint32_t src = j * PER + lane / R;             // source element (within the 32) of this lane's store
            uint32_t o[VW];
#pragma unroll
            for (uint32_t k = 0; k < VW; ++k) o[k] = __shfl_sync(0xffffffffu, v[k], src);
            const uint32_t i = (e0 + j * PER) * R + lane;        // replicated element index
            if (e0 + src < elems) {
                if constexpr (VW == 4) *reinterpret_cast<uint4 *>(tab_s + 4 * i) = make_uint4(o[0], o[1], o[2], o[3]);
                else if constexpr (VW == 2) *reinterpret_cast<uint2 *>(tab_s + 2 * i) = make_uint2(o[0], o[1]);
                else tab_s[i] = o[0];
            }
        }
    }
}

// Entry e of the tables in shared memory.  REP: from the replicated tables, through the copy of this lane.
template <int NWP, bool REP>
SQNN_DEV void load_entry(const uint32_t *tab, uint32_t e, uint32_t lane, uint32_t (&x)[NWP])
{
    constexpr uint32_t R = table_copies(NWP);
    if constexpr (NWP == 1) {
        x[0] = REP ? tab[e * R + lane] : tab[e];
    } else if constexpr (NWP == 2) {
        const uint2 v = *reinterpret_cast<const uint2 *>(tab + 2 * (REP ? e * R + (lane & (R - 1)) : e));
        x[0] = v.x; x[1] = v.y;
    } else if constexpr (NWP == 4) {
        const uint4 v = *reinterpret_cast<const uint4 *>(tab + 4 * (REP ? e * R + (lane & (R - 1)) : e));
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    } else {
        const uint32_t i0 = REP ? (2 * e) * R + (lane & (R - 1)) : 2 * e;
        const uint32_t i1 = REP ? (2 * e + 1) * R + (lane & (R - 1)) : 2 * e + 1;
        const uint4 v = *reinterpret_cast<const uint4 *>(tab + 4 * i0);
        const uint4 u = *reinterpret_cast<const uint4 *>(tab + 4 * i1);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
        x[4] = u.x; x[5] = u.y; x[6] = u.z; x[7] = u.w;
    }
}

// Compile-time facts of a network shape (n_out a multiple of 4: one format tile per kernel tile).
template <int N_OUT, int N_IN>
struct Shape {
    static_assert(N_OUT % 4 == 0, "compile-time shapes have n_out a multiple of 4");
    static constexpr uint32_t n_out = N_OUT, n_in = N_IN;
    static constexpr uint32_t G = 8, W = N_OUT / 4;
    static constexpr uint32_t NW = entry_words(N_OUT), NWP = entry_words_padded(N_OUT);
    static constexpr uint32_t NCH = table_chunks(N_IN, NWP), CB = chunk_bits(N_IN, NWP);
    static constexpr uint32_t SPAN = 8 * N_IN;                       // seed bits of one lane
    static constexpr bool ALIGNED = SPAN % 32 == 0;                   // a lane's seeds start on a word
    static constexpr uint32_t NSW = (SPAN + 31) / 32;                 // words holding them
    static constexpr uint32_t NRAW = ALIGNED ? NSW : NSW + 1;
    static constexpr uint32_t TILE_BITS = SQNN_TILE_SLICES * N_OUT;
};

// The words holding a lane's 8 seeds of one tile.
template <int N_OUT, int N_IN>
struct TileSeeds {
    uint32_t raw[Shape<N_OUT, N_IN>::NRAW];
};
// A tile's run of patch entries [base, end) and the first words of it, fetched ahead of time:
// lane l holds 32-bit words (base >> 1) + l + 32 k, k < 4, of the entry array (two entries each).
struct TileRun {
    uint32_t base, end;
};
constexpr uint32_t PATCH_AHEAD = 4;

template <int N_OUT, int N_IN>
SQNN_DEV void fetch_seeds(const PlanePtrs &P, uint64_t tile, uint32_t lane, TileSeeds<N_OUT, N_IN> &s)
{
    using S = Shape<N_OUT, N_IN>;
    const uint32_t *w = P.wc + tile * (8 * S::n_in) + ((lane * S::SPAN) >> 5);
    if constexpr (S::ALIGNED && S::NSW == 4) {
        const uint4 v = ldg_ahead(reinterpret_cast<const uint4 *>(w));
        s.raw[0] = v.x; s.raw[1] = v.y; s.raw[2] = v.z; s.raw[3] = v.w;
    } else if constexpr (S::ALIGNED && S::NSW == 2) {
        const uint2 v = ldg_ahead(reinterpret_cast<const uint2 *>(w));
        s.raw[0] = v.x; s.raw[1] = v.y;
    } else {
#pragma unroll
        for (uint32_t k = 0; k < S::NRAW; ++k) s.raw[k] = ldg_ahead(w + k);     // sections end with slack
    }
}

SQNN_DEV TileRun fetch_run(const PlanePtrs &P, uint64_t tile)
{
    TileRun r;
    r.base = ldg_ahead(P.idx + tile);
    r.end = ldg_ahead(P.idx + tile + 1);
    return r;
}

// Checks the run against the section and requests its first words.
SQNN_DEV void fetch_patches(const DecodeArgs &A, const PlanePtrs &P, TileRun &run, uint32_t lane,
                            uint32_t (&pw)[PATCH_AHEAD])
{
    if (run.end < run.base || run.end > P.n_pp) {                // offsets point outside the section
        flag(A.status, 2u);
        run.end = run.base = 0;
    }
    const uint32_t *pp32 = reinterpret_cast<const uint32_t *>(P.pp);
    const uint32_t w0 = run.base >> 1, wend = (run.end + 1) >> 1;
#pragma unroll
    for (uint32_t k = 0; k < PATCH_AHEAD; ++k) {
        const uint32_t aw = w0 + lane + 32 * k;
        pw[k] = 0u;
        if (aw < wend) pw[k] = ldg_ahead(pp32 + aw);
    }
}

// One patch entry: flips the bit at pos of the format tile if the entry belongs to the run (t < total, t = its index minus
// the run's base, as unsigned) and pos lies inside the tile.  Branch-free: the reduction is predicated.  The region
// holds the tile or, PART, `bits` bits from bit -offset of it on (the others are passed over).  Returns pos if the entry
// belongs to the run, else 0 (for the range check).
template <bool PART>
SQNN_DEV uint32_t flip_entry(uint32_t region_sa, uint32_t offset, uint32_t bits, uint32_t tile_bits, uint32_t pos, uint32_t t, uint32_t total)
{
    uint32_t seen;
    if constexpr (PART) {
        asm volatile("{\n .reg .pred p, q;\n .reg .b32 a, v, s, b;\n"
                     " setp.lt.u32 q, %3, %4;\n"
                     " setp.lt.and.u32 p, %2, %5, q;\n"
                     " selp.u32 %0, %2, 0, q;\n"
                     " add.u32 b, %2, %6;\n"
                     " setp.lt.and.u32 p, b, %7, p;\n"
                     " shr.u32 a, b, 5;\n shl.b32 a, a, 2;\n add.u32 a, a, %1;\n"
                     " and.b32 s, b, 31;\n shl.b32 v, 1, s;\n"
                     " @p red.shared.xor.b32 [a], v;\n}"
                     : "=r"(seen) : "r"(region_sa), "r"(pos), "r"(t), "r"(total), "r"(tile_bits), "r"(offset), "r"(bits) : "memory");
    } else {
        asm volatile("{\n .reg .pred p, q;\n .reg .b32 a, v, s;\n"
                     " setp.lt.u32 q, %3, %4;\n"                    // the entry belongs to the run
                     " setp.lt.and.u32 p, %2, %5, q;\n"             // ... and its position lies inside the tile
                     " selp.u32 %0, %2, 0, q;\n"
                     " shr.u32 a, %2, 5;\n shl.b32 a, a, 2;\n add.u32 a, a, %1;\n"
                     " and.b32 s, %2, 31;\n shl.b32 v, 1, s;\n"
                     " @p red.shared.xor.b32 [a], v;\n}"
                     : "=r"(seen) : "r"(region_sa), "r"(pos), "r"(t), "r"(total), "r"(tile_bits) : "memory");
    }
    return seen;
}

// Flips the patched positions of one format tile (Section 3.2) in the region (PART, offset, bits: see flip_entry).
// Every lane's words of the tile must be in place (warp barrier before), and the
// region is complete after the warp barrier that follows.  `pw`: words fetched by fetch_patches.
template <bool PART = false>
SQNN_DEV void tile_patch(const DecodeArgs &A, const PlanePtrs &P, const TileRun &run, const uint32_t (&pw)[PATCH_AHEAD],
                         uint32_t *region, uint32_t tile_bits, uint32_t lane, uint32_t offset = 0, uint32_t bits = 0)
{
    if (run.end == run.base) return;                             // the same in every lane
    const uint32_t region_sa = smem_addr(region);
    const uint32_t total = run.end - run.base;
    const uint32_t w0 = run.base >> 1, wend = (run.end + 1) >> 1;
    // index, relative to the run, of the low entry of this lane's first word: -1 when the run starts
    // in the high half of its first word (the unsigned compare in flip_entry then rejects it)
    const uint32_t t0 = 2 * (w0 + lane) - run.base;
    uint32_t top = 0;                                            // largest position seen
#pragma unroll
    for (uint32_t k = 0; k < PATCH_AHEAD; ++k) {
        top = max(top, flip_entry<PART>(region_sa, offset, bits, tile_bits, pw[k] & 0xffffu, t0 + 64 * k, total));
        top = max(top, flip_entry<PART>(region_sa, offset, bits, tile_bits, pw[k] >> 16, t0 + 64 * k + 1, total));
    }
    // longer runs: eight words (sixteen entries) per lane and round; the words of the next round are
    // requested before this round's are used
    constexpr uint32_t RB = 8;
    const uint32_t *pp32 = reinterpret_cast<const uint32_t *>(P.pp);
    uint32_t a0 = w0 + 32 * PATCH_AHEAD;
    if (a0 < wend) {
        uint32_t cur[RB], nxt[RB];
        auto request = [&](uint32_t at, uint32_t (&w)[RB]) {
#pragma unroll
            for (uint32_t k = 0; k < RB; ++k) {
                const uint32_t aw = at + lane + 32 * k;
                w[k] = 0u;
                if (aw < wend) w[k] = ldg_ahead(pp32 + aw);
            }
        };
        request(a0, cur);
        for (; a0 < wend; a0 += 32 * RB) {
            request(a0 + 32 * RB, nxt);
            const uint32_t t = 2 * (a0 + lane) - run.base;
#pragma unroll
            for (uint32_t k = 0; k < RB; ++k) {
                top = max(top, flip_entry<PART>(region_sa, offset, bits, tile_bits, cur[k] & 0xffffu, t + 64 * k, total));
                top = max(top, flip_entry<PART>(region_sa, offset, bits, tile_bits, cur[k] >> 16, t + 64 * k + 1, total));
            }
#pragma unroll
            for (uint32_t k = 0; k < RB; ++k) cur[k] = nxt[k];
        }
    }
    if (top >= tile_bits) flag(A.status, 1u);
}

// Expands the lane's 8 slices of one tile into region[lane * W .. lane * W + W).  WAIT_BULK: lane 0
// first waits for its pending bulk copy out of `region`, just before the region is overwritten.
// REP: `tab` holds the replicated tables.
template <int N_OUT, int N_IN, bool WAIT_BULK = false, bool REP = false>
SQNN_DEV void tile_expand(const TileSeeds<N_OUT, N_IN> &in, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    using S = Shape<N_OUT, N_IN>;
    constexpr uint32_t G = S::G, W = S::W, NW = S::NW, NWP = S::NWP, NCH = S::NCH, CB = S::CB;
    constexpr uint32_t n_out = S::n_out, n_in = S::n_in, NSW = S::NSW;
    uint32_t *mine = region + lane * W;

    // seeds -> table entries
    uint32_t al[NSW];
    if constexpr (S::ALIGNED) {
#pragma unroll
        for (uint32_t k = 0; k < NSW; ++k) al[k] = in.raw[k];
    } else {
        const uint32_t sh0 = (lane * S::SPAN) & 31u;
#pragma unroll
        for (uint32_t k = 0; k < NSW; ++k) al[k] = __funnelshift_r(in.raw[k], in.raw[k + 1], sh0);
    }
    uint32_t x[G][NWP];
#pragma unroll
    for (uint32_t i = 0; i < G; ++i) {
        constexpr uint32_t smask = n_in >= 32 ? 0xffffffffu : ((1u << n_in) - 1u);
        const uint32_t o = i * n_in, w = o >> 5, s = o & 31;
        uint32_t seed;
        if (s + n_in <= 32) seed = (al[w] >> s) & smask;
        else seed = __funnelshift_r(al[w], al[w + 1 < NSW ? w + 1 : w], s) & smask;
        load_entry<NWP, REP>(tab, seed & ((1u << CB) - 1u), lane, x[i]);
#pragma unroll
        for (uint32_t ch = 1; ch < NCH; ++ch) {
            uint32_t y[NWP];
            load_entry<NWP, REP>(tab, (ch << CB) | ((seed >> (ch * CB)) & ((1u << CB) - 1u)), lane, y);
#pragma unroll
            for (uint32_t k = 0; k < NW; ++k) x[i][k] ^= y[k];
        }
    }
    // output word k = bits [32k, 32k + 32) of the concatenated entries (entry bits >= n_out are 0)
    uint32_t out[W];
#pragma unroll
    for (uint32_t k = 0; k < W; ++k) {
        const uint32_t i0 = (32 * k) / n_out, o = 32 * k - i0 * n_out;
        const uint32_t lo = x[i0][o >> 5];
        const uint32_t hi = ((o >> 5) + 1 < NW) ? x[i0][((o >> 5) + 1 < NW) ? (o >> 5) + 1 : 0] : 0u;
        uint32_t word = (o & 31) ? __funnelshift_r(lo, hi, o & 31) : lo;
        uint32_t filled = n_out - o;
#pragma unroll
        for (uint32_t i = i0 + 1; i < G; ++i) {
            if (filled < 32) { word |= x[i][0] << filled; filled += n_out; }
        }
        out[k] = word;
    }
    if constexpr (WAIT_BULK) {                       // the bulk copy of the previous tile still reads `region`
        if (lane == 0) bulk_wait_read<0>();
        __syncwarp();
    }
    // the widest stores the lane's base allows (lane stride W words): conflict-free for every W
    if constexpr (W % 4 == 0) {
#pragma unroll
        for (uint32_t k = 0; k < W; k += 4)
            *reinterpret_cast<uint4 *>(mine + k) = make_uint4(out[k], out[k + 1], out[k + 2], out[k + 3]);
    } else if constexpr (W % 2 == 0) {
#pragma unroll
        for (uint32_t k = 0; k < W; k += 2) *reinterpret_cast<uint2 *>(mine + k) = make_uint2(out[k], out[k + 1]);
    } else {
#pragma unroll
        for (uint32_t k = 0; k < W; ++k) mine[k] = out[k];
    }
}

// Entry e of the tables in shared memory is the XOR of one entry per chunk of the seed (run-time shapes).
template <int NWP>
SQNN_DEV void lookup(const DecodeArgs &A, const uint32_t *tab, uint32_t seed, uint32_t (&x)[NWP])
{
    const uint32_t cb = A.cb, cmask = (1u << cb) - 1u;
    load_entry<NWP, false>(tab, seed & cmask, 0, x);
    for (uint32_t ch = 1; ch < A.nchunks; ++ch) {
        uint32_t y[NWP];
        seed >>= cb;
        load_entry<NWP, false>(tab, (ch << cb) | (seed & cmask), 0, y);
#pragma unroll
        for (int k = 0; k < NWP; ++k) x[k] ^= y[k];
    }
}

// Run-time shape with n_out a multiple of 32: every slice is NW whole output words, so the lanes take slices in
// turn (lane l: slices l, l + 32, ...) and nothing has to be shifted into place; the stores of a warp are
// consecutive.  (With eight consecutive slices per lane all lanes would store to the same bank.)
template <int NW>
SQNN_DEV void expand_whole_words(const DecodeArgs &A, const PlanePtrs &P, uint64_t tile, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    constexpr int NWP = (int)(NW <= 2 ? NW : NW <= 4 ? 4 : 8);
    const uint32_t n_in = A.n_in, smask = n_in >= 32 ? 0xffffffffu : (1u << n_in) - 1u;
    uint32_t seed[8];
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) {
        const uint64_t bit = (tile * SQNN_TILE_SLICES + 32 * i + lane) * n_in;
        const uint32_t *w = P.wc + (bit >> 5);
        seed[i] = __funnelshift_r(__ldg(w), __ldg(w + 1), (uint32_t)bit & 31u) & smask;     // sections end with slack
    }
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) {
        uint32_t x[NWP];
        lookup<NWP>(A, tab, seed[i], x);
        uint32_t *out = region + (32 * i + lane) * NW;
        if constexpr (NW % 4 == 0) {
#pragma unroll
            for (int k = 0; k < NW; k += 4) *reinterpret_cast<uint4 *>(out + k) = make_uint4(x[k], x[k + 1], x[k + 2], x[k + 3]);
        } else if constexpr (NW % 2 == 0) {
#pragma unroll
            for (int k = 0; k < NW; k += 2) *reinterpret_cast<uint2 *>(out + k) = make_uint2(x[k], x[k + 1]);
        } else {
#pragma unroll
            for (int k = 0; k < NW; ++k) out[k] = x[k];
        }
    }
}

// Any other run-time shape: a lane owns 8 * KT consecutive slices and shifts their entries together.  The seeds of
// eight slices (n_in bytes) are fetched at once and move through registers.
template <int NWP>
SQNN_DEV void expand_shifted(const DecodeArgs &A, const PlanePtrs &P, uint64_t ktile, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    const uint32_t n_in = A.n_in, nw = A.nw, smask = n_in >= 32 ? 0xffffffffu : (1u << n_in) - 1u;
    const uint32_t last = A.n_out - 32 * (nw - 1);              // bits of an entry's last word, 1 .. 32
    uint32_t *out = region + lane * A.W;
    uint32_t have = 0, top = 0;                                  // pending bits: the upper `have` bits of `top`
    for (uint32_t f = 0; f < A.KT; ++f) {
        const uint64_t byte = ((ktile * 32 + lane) * A.KT + f) * n_in;
        const uint32_t *w = P.wc + (byte >> 2);
        const uint32_t sh = ((uint32_t)byte & 3u) * 8, bits = 8 * n_in + sh;
        uint32_t al[9];
#pragma unroll
        for (uint32_t k = 0; k < 9; ++k) al[k] = 32 * k < bits ? __ldg(w + k) : 0u;
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) al[k] = __funnelshift_r(al[k], al[k + 1], sh);
#pragma unroll
        for (uint32_t i = 0; i < 8; ++i) {
            uint32_t x[NWP];
            lookup<NWP>(A, tab, al[0] & smask, x);
#pragma unroll
            for (uint32_t k = 0; k < 7; ++k) al[k] = __funnelshift_rc(al[k], al[k + 1], n_in);
            al[7] = n_in >= 32 ? 0u : al[7] >> n_in;
            uint32_t prev = top, end = x[0];
#pragma unroll
            for (uint32_t k = 0; k < NWP; ++k) {
                if (k + 1 < nw) {                                // whole words
                    *out++ = __funnelshift_l(prev, x[k], have);
                    prev = x[k];
                    if (k + 1 < NWP) end = x[k + 1];
                }
            }
            const uint32_t word = __funnelshift_l(prev, end, have);          // bits past the pending ones are 0
            if (have + last >= 32) {
                *out++ = word;
                have = have + last - 32;
                top = last >= 32 ? end : end << (32 - last);
            } else {
                have += last;
                top = word << (32 - have);
            }
        }
    }
}

// Run-time shape, whole format tiles.  Ends with the warp synchronised.
SQNN_DEV void decode_whole_tiles(const DecodeArgs &A, uint32_t plane, uint64_t ktile, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    const PlanePtrs &P = A.pl[plane];
    const uint32_t tile_bits = SQNN_TILE_SLICES * A.n_out;
    uint32_t pw[PATCH_AHEAD];
    TileRun run = fetch_run(P, ktile * A.KT);
    if (A.n_out % 32 == 0) {
        switch (A.nw) {
            case 1: expand_whole_words<1>(A, P, ktile, region, tab, lane); break;
            case 2: expand_whole_words<2>(A, P, ktile, region, tab, lane); break;
            case 3: expand_whole_words<3>(A, P, ktile, region, tab, lane); break;
            case 4: expand_whole_words<4>(A, P, ktile, region, tab, lane); break;
            case 5: expand_whole_words<5>(A, P, ktile, region, tab, lane); break;
            case 6: expand_whole_words<6>(A, P, ktile, region, tab, lane); break;
            case 7: expand_whole_words<7>(A, P, ktile, region, tab, lane); break;
            default: expand_whole_words<8>(A, P, ktile, region, tab, lane); break;
        }
    } else {
        switch (A.nwp) {
            case 1: expand_shifted<1>(A, P, ktile, region, tab, lane); break;
            case 2: expand_shifted<2>(A, P, ktile, region, tab, lane); break;
            case 4: expand_shifted<4>(A, P, ktile, region, tab, lane); break;
            default: expand_shifted<8>(A, P, ktile, region, tab, lane); break;
        }
    }
    fetch_patches(A, P, run, lane, pw);
    __syncwarp();
    for (uint32_t f = 0; f < A.KT; ++f) {                        // one format tile after the other
        tile_patch(A, P, run, pw, region + f * (tile_bits / 32), tile_bits, lane);
        if (f + 1 < A.KT) {
            run = fetch_run(P, ktile * A.KT + f + 1);
            fetch_patches(A, P, run, lane, pw);
        }
    }
    __syncwarp();
}

// A kernel tile that is a part of a format tile: `words` words; the slices that overlap it, the first one starting at bit pos0 <= 0 of
// it and at bit `bit` of the words at wc, are taken by the lanes in turn.
struct RangeTile {
    const uint32_t *wc;
    uint32_t bit, slices, words;         // slices: those left in the plane
    int32_t pos0;
};
constexpr uint32_t SEEDS_AHEAD = 4;      // turns whose seeds are requested together
struct RangeSeeds {
    uint32_t lo[SEEDS_AHEAD], hi[SEEDS_AHEAD];
};
SQNN_DEV void request_seeds(const DecodeArgs &A, const RangeTile &T, uint32_t turn, uint32_t lane, RangeSeeds &s)
{
#pragma unroll
    for (uint32_t k = 0; k < SEEDS_AHEAD; ++k) {
        const uint32_t i = 32 * (turn + k) + lane;
        const uint32_t *w = T.wc + ((T.bit + i * A.n_in) >> 5);
        s.lo[k] = s.hi[k] = 0u;
        if (T.pos0 + (int32_t)(i * A.n_out) < (int32_t)(32 * T.words) && i < T.slices) { s.lo[k] = ldg_ahead(w); s.hi[k] = ldg_ahead(w + 1); }   // sections end with slack
    }
}

// Expands the tile's slices.  Slices of 33 bits and more share a word with one neighbour at most: its part is handed up
// the lanes, and from one turn to the next, to the slice the word ends in, which stores it.  Shorter ones are
// added to zeros by reductions.
template <int NWP>
SQNN_DEV void expand_range(const DecodeArgs &A, const RangeTile &T, RangeSeeds &s, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    const uint32_t n_out = A.n_out, n_in = A.n_in, smask = n_in >= 32 ? 0xffffffffu : (1u << n_in) - 1u, words = T.words;
    const uint32_t region_sa = smem_addr(region);
    if constexpr (NWP == 1) {
        for (uint32_t w = 4 * lane; w < words; w += 128) *reinterpret_cast<uint4 *>(region + w) = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
    }
    uint32_t carry = 0;                                          // part of the first slice's first word from the turn before
    int32_t first = T.pos0;                                      // where lane 0's slice starts
    for (uint32_t turn = 0;; turn += SEEDS_AHEAD) {
        RangeSeeds ahead;
        request_seeds(A, T, turn + SEEDS_AHEAD, lane, ahead);
#pragma unroll
        for (uint32_t j = 0; j < SEEDS_AHEAD; ++j, first += (int32_t)(32 * n_out)) {
            const uint32_t i = 32 * (turn + j) + lane;
            if (first >= (int32_t)(32 * words) || 32 * (turn + j) >= T.slices) return;
            const int32_t pos = first + (int32_t)(lane * n_out);
            const bool live = i < T.slices && pos < (int32_t)(32 * words);
            uint32_t x[NWP];
            lookup<NWP>(A, tab, __funnelshift_r(s.lo[j], s.hi[j], (T.bit + i * n_in) & 31u) & smask, x);
            const uint32_t sh = (uint32_t)pos & 31u, full = (sh + n_out) >> 5;                   // words that end in it
            const int32_t w = pos >> 5;
            uint32_t prev = 0;
            if constexpr (NWP == 1) {
#pragma unroll
                for (int k = 0; k <= 1; ++k) {
                    const uint32_t word = k == 0 ? x[0] << sh : __funnelshift_l(x[0], 0u, sh);
                    if (live && (uint32_t)(w + k) < words && word)
                        asm volatile("red.shared.xor.b32 [%0], %1;" :: "r"(region_sa + 4 * (uint32_t)(w + k)), "r"(word) : "memory");
                }
            } else {
                uint32_t out[NWP + 1], tail = 0;
#pragma unroll
                for (int k = 0; k <= NWP; ++k) {
                    const uint32_t cur = k < NWP ? x[k < NWP ? k : 0] : 0u;
                    out[k] = __funnelshift_l(prev, cur, sh);
                    prev = cur;
                    if (k > 0 && (uint32_t)k == full) tail = out[k];                             // (0 where no word is shared)
                }
                const uint32_t up = __shfl_up_sync(0xffffffffu, tail, 1);
                out[0] |= lane ? up : carry;
                carry = __shfl_sync(0xffffffffu, tail, 31);
                const uint32_t store = i + 1 == T.slices ? full + 1 : full;                      // the plane's last word may not end
#pragma unroll
                for (int k = 0; k <= NWP; ++k)
                    if (live && (uint32_t)k < store && (uint32_t)(w + k) < words)
                        asm volatile("st.shared.u32 [%0], %1;" :: "r"(region_sa + 4 * (uint32_t)(w + k)), "r"(out[k]) : "memory");
            }
        }
        s = ahead;
    }
}

// Run-time shape, part of a format tile, as the parts are called: up to 10 turns of 32 slices that start anywhere, so that one may overlap three
// format tiles (of 8 turns) and take from three patch runs.  A whole format tile per warp leaves most warps of a small layer idle
// while one walks its lanes' chains of 8, 16 or 32 slices.
// Before / with parts, us: planes of 223 x 673 with 33 x 20 11.4 / 4.3; bf16 of 1024 x 2560, three planes, 64 x 16 15.7 / 9.9; products
// of 4864 x 1152 with 128 x 24, batch 129 21.7 / 14.8, of 960 x 1984, two planes, 33 x 20, batch 1 15.5 / 9.8, of 512 x 192 with
// 200 x 20, batch 35 14.9 / 8.1.  Which layers: most_parts_per_sm, plan_run_time_shape.  Ends with the warp synchronised.
SQNN_DEV void decode_range(const DecodeArgs &A, uint32_t plane, uint64_t ktile, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    const PlanePtrs &P = A.pl[plane];
    const uint32_t n_out = A.n_out, words = 32 * A.W, tile_bits = SQNN_TILE_SLICES * n_out;
    const uint64_t bit0 = ktile * (32ull * words), s0 = n_out > 1 ? __umul64hi(bit0, A.inv_n_out) : bit0;
    uint64_t ftile = s0 / SQNN_TILE_SLICES;
    uint32_t offset = (uint32_t)(ftile * tile_bits - bit0);      // of the format tile inside the kernel tile, as a signed number
    auto goes_on = [&] { return (int32_t)(offset + tile_bits) < (int32_t)(32 * words) && (ftile + 1) * SQNN_TILE_SLICES < A.slices; };
    // the patch runs of the first two format tiles it overlaps, and the first seeds
    TileRun run = fetch_run(P, ftile), run2{0u, 0u};
    if (goes_on()) run2 = fetch_run(P, ftile + 1);
    const uint64_t sbit = s0 * A.n_in, left = A.slices - s0;
    const RangeTile T{P.wc + (sbit >> 5), (uint32_t)sbit & 31u, left < 0x7fffffffu ? (uint32_t)left : 0x7fffffffu, words, -(int32_t)(uint32_t)(bit0 - s0 * n_out)};
    RangeSeeds seeds;
    request_seeds(A, T, 0, lane, seeds);
    uint32_t pw[PATCH_AHEAD], pw2[PATCH_AHEAD];
    fetch_patches(A, P, run, lane, pw);
    fetch_patches(A, P, run2, lane, pw2);
    switch (A.nwp) {
        case 1: expand_range<1>(A, T, seeds, region, tab, lane); break;
        case 2: expand_range<2>(A, T, seeds, region, tab, lane); break;
        case 4: expand_range<4>(A, T, seeds, region, tab, lane); break;
        default: expand_range<8>(A, T, seeds, region, tab, lane); break;
    }
    __syncwarp();
    for (;;) {                                                   // one format tile after the other
        tile_patch<true>(A, P, run, pw, region, tile_bits, lane, offset, 32 * words);
        if (!goes_on()) break;
        offset += tile_bits;
        ++ftile;
        run = run2;
#pragma unroll
        for (uint32_t k = 0; k < PATCH_AHEAD; ++k) pw[k] = pw2[k];
        if (goes_on()) { run2 = fetch_run(P, ftile + 1); fetch_patches(A, P, run2, lane, pw2); }
    }
    __syncwarp();
}

// Run-time shape: one kernel tile.
SQNN_DEV void decode_ktile_generic(const DecodeArgs &A, uint32_t plane, uint64_t ktile, uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    if (A.KT) decode_whole_tiles(A, plane, ktile, region, tab, lane);
    else decode_range(A, plane, ktile, region, tab, lane);
}

// Fetch + expand + patch of one kernel tile without overlap (for the kernels that do more work per
// tile).  Run-time shapes: N_IN = 1 for parts of format tiles, else whole ones.  `tab`: the tables in shared memory.  Ends with the warp synchronised.
template <int N_OUT, int N_IN>
SQNN_DEV void decode_warp_tile(const DecodeArgs &A, uint32_t plane, uint64_t tile,
                               uint32_t *region, const uint32_t *tab, uint32_t lane)
{
    if constexpr (N_OUT != 0) {
        using S = Shape<N_OUT, N_IN>;
        const PlanePtrs &P = A.pl[plane];
        TileSeeds<N_OUT, N_IN> in;
        uint32_t pw[PATCH_AHEAD];
        fetch_seeds<N_OUT, N_IN>(P, tile, lane, in);
        TileRun run = fetch_run(P, tile);
        fetch_patches(A, P, run, lane, pw);
        tile_expand<N_OUT, N_IN>(in, region, tab, lane);
        __syncwarp();
        tile_patch(A, P, run, pw, region, S::TILE_BITS, lane);
        __syncwarp();
    } else if constexpr (N_IN == 1) {
        decode_range(A, plane, tile, region, tab, lane);
    } else {
        decode_whole_tiles(A, plane, tile, region, tab, lane);
    }
}

}  // namespace sqnn
