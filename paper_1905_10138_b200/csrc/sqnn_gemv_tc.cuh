// K3: decryption fused with Y[b][r] = sum_c W[r][c] X[b][c] for small batch (<= 15) on the tensor cores, as a
// template over the network shape, with its launcher.
//
// Work split.  As in sqnn_gemv.cuh a block owns a run of whole rows of W and decodes the kernel tiles that cover
// them into shared memory, next to the same range of the pruning mask.  The product then runs on tcgen05.mma
// with the expanded weights as the A operand in tensor memory:
//
//   - a tile is 16 rows; its columns are cut into 8 equal ranges (kq) of Kq columns, and TMEM lane
//     32 w + 8 i + kq holds row 4 w + i, range kq: the M = 128 lanes are all in use whatever the number of rows;
//   - B row 8 q + kq holds the activations of range kq, vector q (Kq columns, K-major), so lane (row, kq) of the
//     accumulator finds its own product in columns 8 q + kq (one column in eight; the others are the price of
//     sharing B, and cost nothing at these N);
//   - four expander groups of four warps each take an equal run of the list (tile, plane, 128 columns), with
//     an accumulator and A slots of their own, each fed to the tensor cores by a warp of its own; the scale of
//     a row and plane is applied to the accumulator, so weights are exact.  fp32 activations enter as three bf16
//     pieces that add up to them exactly (8 + 8 + 8 bits).
//
// Kq is a multiple of 128 columns (`units` of them): the 8 lanes of a row read 16-byte vectors of mask and plane bits
// that lie 16 x units bytes apart.  With a multiple of 8 units they would all read the same four banks, and one more
// unit is cheaper (LSTM-like layer 4096 x 8192, two planes, batch 1: 14.5 us against 15.4; 2048 x 16384: 14.5 against
// 15.6).  An even number that is none costs two or four passes of the same banks, less than another unit of
// expansion would: 16384 x 2048, two planes, batch 8 21.9 us with three units and 18.7 with two, 32736 x 1025
// 35.9 and 30.0, 8192 x 4096 19.6 (five) and 17.8 (four), 2730 x 12288 32.8 (13) and 31.4 (12).  Sums over the 8
// ranges (shuffles) and the four groups (shared memory) have a fixed order: results are bit-identical from run to run.
//
// Every wait on an mbarrier is bounded.  An expander warp whose wait gives up sets SQNN_E_TIMEOUT in the status word,
// makes the arrivals its MMA warp still counts on and leaves its loop; the MMA warp reaches the end of its list, and
// the block returns without storing this pass of Y, after a bounded wait for the MMAs it issued.  The barriers
// between the two only count: an arrival for a slot's next use while another warp had not yet arrived for the one
// before would complete the wrong one, and the MMA warp would wait for good; so the late arrivals follow the number
// of slots the MMA warp has taken.  (mbarriers with bounded waits between the two would need no such care, but FC6
// batch 1 takes 9.8 us with them against 9.5, 3001 x 4099 with four fp32 vectors 16.9 against 16.2.)
//
// Bound: integer instructions of the expansion (1.4 per weight and plane, against 42 per unpruned weight of the
// walk over care bits in sqnn_gemv.cuh, 3.8 per weight at 9 % density) and the latency of the block's phases
// (launch, staging, decode, product, reduction).  Which of the two takes a call: sqnn_gemv_plan.h.
#pragma once
#include "sqnn_gemv.cuh"
#include "sqnn_tc.cuh"

namespace sqnn {

constexpr uint32_t TC_THREADS = TC_WARPS * 32;             // per group four expander warps, and an MMA warp
constexpr uint64_t TC_WAIT_LIMIT = 2000000000ull;         // cycles a bounded wait may take: about a second

struct TcArgs {
    DecodeArgs A;
    const uint32_t *mask32;
    uint64_t mask_words;
    const float *alpha;
    const void *x;
    int64_t ldx;
    float *y;
    int64_t ldy;
    uint64_t m;
    uint32_t n, batch;
    uint32_t rows_per_block, rows_per_chunk;
    uint32_t region_words;        // words of one bit vector of a chunk in shared memory (with slack for the last row's ranges)
    uint32_t kq, units;           // columns per range, kq / 128
    uint32_t bt;                  // activation vectors per pass
    uint32_t N;                   // MMA N: 8 x bt x pieces, rounded up to 16
    uint32_t slots;               // A slots (64 columns) per group: 1 or 2
    uint32_t alpha_words, part_words;
    uint32_t x_vec;               // rows of X start on 16-byte boundaries
    uint32_t unheard;             // test only: completions are reported to barriers this far past the real ones (else 0)
    uint64_t wait_limit;          // cycles a bounded wait may take
};

SQNN_DEV void named_arrive(uint32_t id) { asm volatile("bar.arrive %0, 160;\n" :: "r"(id) : "memory"); }
SQNN_DEV void named_sync(uint32_t id) { asm volatile("bar.sync %0, 160;\n" :: "r"(id) : "memory"); }
// The arrivals of a warp that has given up, for slots [from, to) of its group: each once the MMA warp has taken the
// use before it of the same barrier (it waits for nothing but these arrivals; bounded all the same).
static __device__ __noinline__ void arrive_for_the_rest(const volatile uint32_t *taken, uint32_t barrier, uint32_t slot_mask, uint32_t from, uint32_t to, uint64_t limit)
{
    const long long t0 = clock64();
    for (; from != to; ++from) {
        while ((int32_t)(*taken - (from - slot_mask)) < 0 && (uint64_t)(clock64() - t0) <= limit) {}
        __syncwarp();
        named_arrive(barrier + (from & slot_mask));
    }
}

// 128 columns of one row from bit `o` of a packed vector in shared memory (address sa, 16-byte aligned).
template <bool ALIGNED>
SQNN_DEV void lds_bits128(uint32_t sa, uint32_t o, uint32_t (&out)[4])
{
    const uint32_t at = sa + ((o >> 7) << 4);
    uint32_t q[8];
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]) : "r"(at));
    if constexpr (ALIGNED) {
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] = q[k];
    } else {
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]) : "r"(at + 16));
        const bool two = (o & 64u) != 0, one = (o & 32u) != 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) q[k] = two ? q[k + 2] : q[k];
#pragma unroll
        for (int k = 0; k < 5; ++k) q[k] = one ? q[k + 1] : q[k];
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k] = __funnelshift_r(q[k], q[k + 1], o & 31u);
    }
}

SQNN_DEV void sts128(uint32_t at, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" :: "r"(at), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Stages activation vectors [bc, bc + bt) as B rows: vector q, range kq, piece p -> row 8 (q * PIECES + p) + kq of
// every 64-column step's box ([N rows][128 bytes], 128-byte swizzle).  Columns past n and vectors past the batch
// are zero.  A warp takes 32 chunks (of 8 columns) of one B row at a time.  bf16 rows on 16-byte boundaries go
// straight to shared memory (cp.async, the caller commits and waits); everything else passes through registers.
template <typename XT>
SQNN_DEV void tc_stage_x(const TcArgs &g, uint32_t x_sa, uint32_t bc)
{
    constexpr uint32_t PIECES = sizeof(XT) == 4 ? 3 : 1;
    const XT *x = reinterpret_cast<const XT *>(g.x);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t chunks = g.kq / 8, blocks = (chunks + 31) / 32, items = TC_RANGES * g.bt * blocks;
    for (uint32_t it = warp; it < items; it += TC_THREADS / 32) {
        const uint32_t row = it / blocks, ch = (it - row * blocks) * 32 + lane;                // row = 8 q + kq
        if (ch >= chunks) continue;
        const uint32_t q = row >> 3, kq = row & 7u, c = kq * g.kq + ch * 8;
        const uint32_t valid = bc + q < g.batch && c < g.n ? min(g.n - c, 8u) : 0u;
        const XT *src = x + (int64_t)(bc + q) * g.ldx + c;
        const uint32_t box = x_sa + (ch >> 3) * g.N * 128;
        if constexpr (PIECES == 1) {
            const uint32_t at = box + row * 128 + (((ch & 7u) ^ kq) << 4);
            if (g.x_vec) {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" :: "r"(at), "l"(valid ? src : x), "r"(2 * valid) : "memory");
            } else {
                const unsigned short *h = reinterpret_cast<const unsigned short *>(src);
                uint32_t w[4];
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    w[k] = (2 * k < valid ? (uint32_t)__ldg(h + 2 * k) : 0u) | (2 * k + 1 < valid ? (uint32_t)__ldg(h + 2 * k + 1) << 16 : 0u);
                sts128(at, w[0], w[1], w[2], w[3]);
            }
        } else {
            float v[8];
            if (g.x_vec && valid == 8) {
                const float4 t = __ldg(reinterpret_cast<const float4 *>(src)), u = __ldg(reinterpret_cast<const float4 *>(src) + 1);
                v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; v[4] = u.x; v[5] = u.y; v[6] = u.z; v[7] = u.w;
            } else {
#pragma unroll
                for (uint32_t k = 0; k < 8; ++k) v[k] = k < valid ? __ldg(reinterpret_cast<const float *>(src) + k) : 0.0f;
            }
            // the upper half of an fp32 word is a bf16 with its first 8 significant bits; what is left after
            // subtracting it has 16, and so on: three pieces, exactly
#pragma unroll
            for (uint32_t p = 0; p < PIECES; ++p) {
                const uint32_t r = 8 * (q * PIECES + p) + kq;
                uint32_t w[4];
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k) w[k] = __byte_perm(__float_as_uint(v[2 * k]), __float_as_uint(v[2 * k + 1]), 0x7632);
                sts128(box + r * 128 + (((ch & 7u) ^ kq) << 4), w[0], w[1], w[2], w[3]);
#pragma unroll
                for (uint32_t k = 0; k < 8; ++k) v[k] -= __uint_as_float(__float_as_uint(v[k]) & 0xffff0000u);
            }
        }
    }
}

// One output by a plain walk over the care bits: for sums that came out as no finite number.  A pruned weight must
// not meet an activation that is infinite or not a number, and in the matrix product it does (as zero).
template <typename XT>
SQNN_DEV float tc_walk(const TcArgs &g, const XT *x, const uint32_t *mask_s, const uint32_t *bits_s, const float *al, uint32_t o)
{
    float sum = 0.0f;
#pragma unroll 1
    for (uint32_t c = 0; c < g.n; ++c) {
        if (!((mask_s[(o + c) >> 5] >> ((o + c) & 31u)) & 1u)) continue;
        float w = 0.0f;
#pragma unroll 1
        for (uint32_t pl = 0; pl < g.A.n_q; ++pl)
            w += ((bits_s[pl * g.region_words + ((o + c) >> 5)] >> ((o + c) & 31u)) & 1u) ? al[pl] : -al[pl];
        sum = fmaf(w, to_float(x[c]), sum);
    }
    return sum;
}

template <int N_OUT, int N_IN, typename XT, bool ALIGNED>
__global__ void __launch_bounds__(TC_THREADS, 1)
k_gemv_tc(const TcArgs g)
{
    extern __shared__ __align__(16) uint32_t smem[];
    // per group: two A slots free, accumulator complete; then per group: all MMAs over (after a timeout); then for tests
    // the first three again, where nobody waits
    __shared__ uint64_t bars[7 * TC_GROUPS];
    __shared__ volatile uint32_t taken_s[TC_GROUPS];      // A slots the group's MMA warp has taken
    __shared__ uint32_t tmem_slot, abort_word;
    constexpr uint32_t PIECES = sizeof(XT) == 4 ? 3 : 1;
    const DecodeArgs &A = g.A;
    volatile uint32_t *abort_flag = &abort_word;
    const uint32_t W = words_per_lane<N_OUT>(A);
    const uint32_t TW = 32 * W;                                  // words per kernel tile
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr uint32_t nwarps = TC_THREADS / 32;
    const uint32_t n = g.n, n_q = A.n_q;
    uint32_t *tab_s = smem;
    uint32_t *bits_s = tab_s + A.tab_words;                      // [plane][region_words]
    uint32_t *mask_s = bits_s + n_q * g.region_words;
    float *alpha_s = reinterpret_cast<float *>(mask_s + g.region_words);
    float *part_s = alpha_s + g.alpha_words;                     // [group][row][bt]
    const uint32_t x_sa = (smem_addr(part_s + g.part_words) + 1023u) & ~1023u;
    const uint32_t bars_sa = smem_addr(bars);
    const bool mask_vec = (reinterpret_cast<uintptr_t>(g.mask32) & 15) == 0;
    const uint64_t row0 = (uint64_t)blockIdx.x * g.rows_per_block;
    const uint64_t row_end = row0 + g.rows_per_block < g.m ? row0 + g.rows_per_block : g.m;

    // The block takes all tensor memory of its SM.  A block of the next grid does so too, and may become resident here
    // as soon as this grid has let it in; if it got the columns first, it would hold them while it waits for this
    // grid, which could then never end.  So the next grid is let in (a block counts as soon as one of its threads
    // has) by the warp that allocates, after its allocation: then every block of this grid has its columns, and
    // a later one's allocation waits until they are given back.
    const bool holder = warp == nwarps - 1;
    if (holder) tmem_alloc(&tmem_slot, 512);
    if (warp == nwarps - 2) {
        if (lane < 7 * TC_GROUPS) mbar_init(bars_sa + 8 * lane, 1);
        if (lane < TC_GROUPS) taken_s[lane] = 0;
        if (lane == 0) abort_word = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    wait_prior_grid();
    if (holder) launch_dependents();
    uint32_t slot_seq = 0, parts_done = 0;                       // per group: A slots filled, accumulators read
    uint32_t gave_up = 0;                                        // a wait of this warp
    bool first = true;

    for (uint64_t ra = row0; ra < row_end; ra += g.rows_per_chunk) {
        const uint64_t rb = ra + g.rows_per_chunk < row_end ? ra + g.rows_per_chunk : row_end;
        const uint32_t nrows = (uint32_t)(rb - ra);
        // kernel tiles that cover the bits [ra * n, rb * n)
        const uint64_t tile_bits = 32ull * TW;
        const uint64_t kt0 = (ra * n) / tile_bits, kt1 = (rb * n + tile_bits - 1) / tile_bits;
        const uint32_t nt = (uint32_t)(kt1 - kt0);
        const uint64_t gw0 = kt0 * TW;                           // first word of the chunk's regions
        if (!first) __syncthreads();                             // the product of the previous chunk is over
        // decode: item = (tile, plane), dealt out over the warps.  A warp's first item is requested before
        // everything else, its patch entries (whose place the first answer tells) after the requests for tables,
        // activations, mask and scales.
        const uint32_t items = nt * n_q;
        uint32_t item = warp;
        auto stage_all = [&] {
            if (first) {
                tables_request(A, tab_s);                        // commit group: tables
                tc_stage_x<XT>(g, x_sa, 0);
            }
            stage_mask(mask_s, g.mask32, gw0, g.mask_words, nt * TW, threadIdx.x, TC_THREADS, mask_vec);
            for (uint32_t i = threadIdx.x; i < nrows * n_q; i += TC_THREADS) cp_async4(alpha_s + i, g.alpha + ra * n_q + i);
            cp_async_commit();                                   // commit group: activations, mask and scales
            for (uint32_t i = threadIdx.x; i < TC_GROUPS * nrows * g.bt; i += TC_THREADS) part_s[i] = 0.0f;
        };
        auto tables_ready = [&] {
            if (first) {
                cp_async_wait_group<1>();                        // (the younger group may be pending)
                __syncthreads();
            }
        };
        if constexpr (N_OUT != 0) {
            using S = Shape<N_OUT, N_IN>;
            TileSeeds<N_OUT, N_IN> s;
            TileRun run{0u, 0u};
            uint32_t pw[PATCH_AHEAD];
            auto fetch = [&](uint32_t it) {
                const uint32_t t = it / n_q, pl = it - t * n_q;
                run = fetch_run(A.pl[pl], kt0 + t);
                fetch_seeds<N_OUT, N_IN>(A.pl[pl], kt0 + t, lane, s);
            };
            if (item < items) fetch(item);
            stage_all();
            if (item < items) fetch_patches(A, A.pl[item % n_q], run, lane, pw);
            tables_ready();
            while (item < items) {
                const uint32_t t = item / n_q, pl = item - t * n_q;
                uint32_t *region = bits_s + pl * g.region_words + t * TW;
                tile_expand<N_OUT, N_IN>(s, region, tab_s, lane);
                __syncwarp();
                tile_patch(A, A.pl[pl], run, pw, region, S::TILE_BITS, lane);
                item += nwarps;
                if (item < items) { fetch(item); fetch_patches(A, A.pl[item % n_q], run, lane, pw); }
            }
        } else {
            stage_all();
            tables_ready();
            for (; item < items; item += nwarps) {
                const uint32_t t = item / n_q, pl = item - t * n_q;
                decode_ktile_generic(A, pl, kt0 + t, bits_s + pl * g.region_words + t * TW, tab_s, lane);
            }
        }
        first = false;
        cp_async_wait_all();
        fence_async_smem();                                      // staged activations -> visible to the tensor cores
        tc_fence_before();
        __syncthreads();                                         // bits, mask, scales, activations in place
        tc_fence_after();

        // a group's run of the list (tile, plane, 128 columns)
        const uint32_t tiles = (nrows + TC_TILE_ROWS - 1) / TC_TILE_ROWS, list = tiles * n_q * g.units;
        const uint32_t grp = warp < 4 * TC_GROUPS ? warp >> 2 : warp - 4 * TC_GROUPS;
        const uint32_t u_begin = list * grp / TC_GROUPS, u_end = list * (grp + 1) / TC_GROUPS;
        const uint32_t d_tmem = tmem_slot + grp * g.N, a_tmem = tmem_slot + TC_GROUPS * g.N + grp * g.slots * 32;
        const uint32_t free_a = bars_sa + 24 * grp, done = free_a + 16;
        const uint32_t slot_mask = g.slots - 1, slot_shift = g.slots - 1;      // 1 slot: 0, 2 slots: 1
        for (uint32_t bc = 0; bc < g.batch; bc += g.bt) {
            if (bc != 0 || (ra != row0 && g.bt < g.batch)) {     // another pass: its activations replace the last one's
                __syncthreads();
                tc_stage_x<XT>(g, x_sa, bc);
                cp_async_commit();
                cp_async_wait_all();
                for (uint32_t i = threadIdx.x; i < TC_GROUPS * nrows * g.bt; i += TC_THREADS) part_s[i] = 0.0f;
                fence_async_smem();
                __syncthreads();
            }
            if (warp < 4 * TC_GROUPS) {
                const uint32_t quad = warp & 3, kq = lane & 7, lane_sel = (quad * 32) << 16;
                const uint32_t mask_sa = smem_addr(mask_s), bits_sa = smem_addr(bits_s);
                const uint32_t seq_end = slot_seq + 2 * (u_end - u_begin);
                float acc[TC_MAX_Q];
#pragma unroll
                for (uint32_t q = 0; q < TC_MAX_Q; ++q) acc[q] = 0.0f;
                for (uint32_t u = u_begin; u < u_end;) {
                    const uint32_t it = u / g.units, t0 = u - it * g.units, tile = it / n_q, pl = it - tile * n_q;
                    const uint32_t len = min(g.units - t0, u_end - u);
                    const uint32_t rl = min(tile * TC_TILE_ROWS + quad * 4 + (lane >> 3), nrows - 1);
                    uint32_t o = (uint32_t)((ra + rl) * n - gw0 * 32) + kq * g.kq + t0 * 128;
                    const uint32_t plane_sa = bits_sa + pl * g.region_words * 4;
                    for (uint32_t k = 0; k < len; ++k, o += 128) {
                        uint32_t mw[4], bw[4];
                        lds_bits128<ALIGNED>(mask_sa, o, mw);
                        lds_bits128<ALIGNED>(plane_sa, o, bw);
#pragma unroll
                        for (uint32_t h = 0; h < 2; ++h, ++slot_seq) {
                            uint32_t v[32];
                            expand32(mw[2 * h], bw[2 * h], v);
                            expand32(mw[2 * h + 1], bw[2 * h + 1], v + 16);
                            const uint32_t slot = slot_seq & slot_mask, use = slot_seq >> slot_shift;
                            if (use > 0) {
                                if (!mbar_wait_warp(free_a + 8 * slot, (use - 1) & 1u, abort_flag, A.status, g.wait_limit)) goto late;
                                tc_fence_after();
                            }
                            tmem_st16(a_tmem + lane_sel + slot * 32, v);
                            tmem_st16(a_tmem + lane_sel + slot * 32 + 16, v + 16);
                            tmem_st_wait();
                            tc_fence_before();
                            named_arrive(1 + 2 * grp + slot);
                        }
                    }
                    u += len;
                    // the part's accumulator: this lane's range, scaled
                    const float al = 0.5f * alpha_s[rl * n_q + pl];
                    if (!mbar_wait_warp(done, parts_done & 1u, abort_flag, A.status, g.wait_limit)) goto late;
                    ++parts_done;
                    tc_fence_after();
#pragma unroll
                    for (uint32_t q4 = 0; q4 < TC_MAX_Q / 4; ++q4) {
                        if (32 * q4 >= g.N) break;
                        uint32_t d[32];
                        tmem_ld32(d_tmem + lane_sel + 32 * q4, d);           // (N = 16, 48, ..: the second half is not used)
#pragma unroll
                        for (uint32_t e = 0; e < 4; ++e) {
                            uint32_t a4[4], a2[2];
#pragma unroll
                            for (uint32_t k = 0; k < 4; ++k) a4[k] = (kq & 4u) ? d[8 * e + k + 4] : d[8 * e + k];
#pragma unroll
                            for (uint32_t k = 0; k < 2; ++k) a2[k] = (kq & 2u) ? a4[k + 2] : a4[k];
                            const float mine = __uint_as_float((kq & 1u) ? a2[1] : a2[0]);
                            const uint32_t q = 4 * q4 + e;
                            acc[q / PIECES] = fmaf(al, mine, acc[q / PIECES]);
                        }
                    }
                    tc_fence_before();
                    // the tile is complete for this group: sum over the ranges, hand over
                    if (u == u_end || u / g.units / n_q != tile) {
#pragma unroll
                        for (uint32_t q = 0; q < TC_MAX_Q / PIECES; ++q) {
                            if (q >= g.bt) break;
                            float sum = acc[q];
                            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                            sum += __shfl_xor_sync(0xffffffffu, sum, 4);
                            if (kq == 0 && tile * TC_TILE_ROWS + quad * 4 + (lane >> 3) < nrows) part_s[(grp * nrows + rl) * g.bt + q] = sum;
                            acc[q] = 0.0f;
                        }
                    }
                }
                goto pass_over;
            late:
                gave_up = 1;
                arrive_for_the_rest(taken_s + grp, 1 + 2 * grp, slot_mask, slot_seq, seq_end, g.wait_limit);
            } else {
                // the group's MMA warp: one slot at a time, in the order they are filled
                const uint32_t idesc = instr_desc_bf16(g.N);
                const uint64_t x_desc0 = smem_desc_sw128(x_sa);
                const uint32_t box_step = g.N * 128 >> 4;
                for (uint32_t u = u_begin; u < u_end;) {
                    const uint32_t it = u / g.units, t0 = u - it * g.units;
                    const uint32_t len = min(g.units - t0, u_end - u);
                    for (uint32_t k = 0; k < 2 * len; ++k, ++slot_seq) {
                        const uint32_t slot = slot_seq & slot_mask;
                        named_sync(1 + 2 * grp + slot);
                        if (lane == 0) taken_s[grp] = slot_seq + 1;
                        tc_fence_after();
                        mma_slot<4>(d_tmem, a_tmem + slot * 32, x_desc0 + (2 * t0 + k) * box_step, idesc, k, free_a + g.unheard + 8 * slot, 0);
                    }
                    mma_commit(done + g.unheard);
                    u += len;
                }
            }
        pass_over:
            if (__syncthreads_or(gave_up)) goto quit;
            for (uint32_t q = warp; q < g.bt && bc + q < g.batch; q += nwarps)
                for (uint32_t rl = lane; rl < nrows; rl += 32) {
                    float sum = 0.0f;
#pragma unroll
                    for (uint32_t p = 0; p < TC_GROUPS; ++p) sum += part_s[(p * nrows + rl) * g.bt + q];
                    if ((__float_as_uint(sum) & 0x7f800000u) == 0x7f800000u)
                        sum = tc_walk<XT>(g, reinterpret_cast<const XT *>(g.x) + (int64_t)(bc + q) * g.ldx, mask_s, bits_s,
                                          alpha_s + rl * n_q, (uint32_t)((ra + rl) * n - gw0 * 32));
                    g.y[(int64_t)(bc + q) * g.ldy + (int64_t)(ra + rl)] = sum;
                }
        }
    }
    goto leave;
quit:
    if (warp >= 4 * TC_GROUPS) {                                 // tensor and shared memory must outlive the MMAs
        const uint32_t over = bars_sa + 8 * (3 * TC_GROUPS + warp - 4 * TC_GROUPS);
        mma_commit(over);
        mbar_drain(over, 0, g.wait_limit);
    }
leave:
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (holder) tmem_dealloc(tmem_slot, 512);
}

// ------------------------------------------------------------------------------------------
// launcher
// ------------------------------------------------------------------------------------------
template <int N_OUT, int N_IN, typename XT>
inline int launch_gemv_tc(const DecodeArgs &A, const TcPlan &plan, const uint64_t *d_mask, const float *d_alpha, const void *d_x,
                          int64_t ldx, uint32_t batch, float *d_y, int64_t ldy, uint64_t m, uint64_t n, cudaStream_t st)
{
    TcArgs g;
    g.A = A;
    g.mask32 = (const uint32_t *)d_mask;
    g.mask_words = A.words64 * 2;
    g.alpha = d_alpha;
    g.x = d_x; g.ldx = ldx; g.y = d_y; g.ldy = ldy;
    g.m = m; g.n = (uint32_t)n; g.batch = batch;
    g.rows_per_block = plan.rows_per_block;
    g.rows_per_chunk = plan.rows_per_chunk;
    g.units = plan.units;
    g.kq = plan.units * 128;
    g.bt = plan.bt; g.N = plan.N; g.slots = plan.slots;
    g.region_words = plan.region_words; g.alpha_words = plan.alpha_words; g.part_words = plan.part_words;
    const DebugKnobs dbg = debug_knobs();
    g.unheard = (dbg.flags & 2u) ? 8 * 4 * TC_GROUPS : 0u;
    g.wait_limit = dbg.wait_cycles ? dbg.wait_cycles : TC_WAIT_LIMIT;
    g.x_vec = (((uintptr_t)d_x & 15) == 0 && (ldx * (int64_t)sizeof(XT)) % 16 == 0) ? 1u : 0u;
    return n % 128 == 0 ? launch_kernel(k_gemv_tc<N_OUT, N_IN, XT, true>, plan.grid, TC_THREADS, plan.smem, st, g)
                        : launch_kernel(k_gemv_tc<N_OUT, N_IN, XT, false>, plan.grid, TC_THREADS, plan.smem, st, g);
}

}  // namespace sqnn
