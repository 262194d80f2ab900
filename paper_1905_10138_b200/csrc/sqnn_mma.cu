// K4: decryption fused with the product for batch >= 16 on the 5th-generation tensor cores.
//
//   Y[b][r] = sum_i alpha[r][i] * sum_c s_i[r][c] X[b][c],      s_i = mask * (2 b_i - 1) in {-1, 0, +1}
//
//   D_u (TMEM, fp32) [128 weight rows x N batch rows] += A (TMEM, bf16) [128 x 64] . B (shared, bf16, K-major) [N x 64]^T
//
// The planes have been decoded to packed bits in the workspace by the tiled decode kernel (queued just before
// this one) and sit in L2.  A tile of work is a group of 128 rows, a group of planes and a chunk of N batch rows;
// its units u, one per plane, have an accumulator each and share the activation tile.  Per 64-column step and unit
//   - one thread fetches the activations with TMA (once for all units; rows past the batch and columns past n
//     are filled with zeros by the copy engine);
//   - the four warps of an expander group turn 64 bits of mask and plane per row into bf16 in registers and
//     store them to a slot of tensor memory (lane = weight row), so the expanded weights never touch shared
//     memory: its bandwidth is left to the activation operand;
//   - the unit's own MMA warp issues four tcgen05.mma (M = 128, K = 16, A from tensor memory) and commits the
//     slot.  (One warp for all units could not keep up: with its instruction stream evicted by the expanders'
//     between steps, a step of 256 tensor-core cycles took it 340.)
// The scale alpha[r][i] is applied to the accumulator in the epilogue, so the weights stay exact (one tile of
// rescaled weights rounded to bf16 would not meet the tolerance: a row has only 2^n_q distinct values and
// their rounding errors add up coherently).
//
// Expansion.  A weight is 0, +2 or -2 in bf16 (0x0000, 0x4000, 0xc000; the factor 2 is taken out of alpha):
// only the two top bits of a half word carry information, so once mask and sign bits are interleaved (mask bit
// 2f, sign bit 2f + 1 of a half word, even columns in the low, odd ones in the high half) two weights cost one
// shift and one AND.
//
// Split of the work.  All tiles x 256-column macros form one line that is cut into equal runs, one per CTA and
// at most one CTA per SM, whatever the shape; a CTA's run covers one or more tiles in part, and each part is
// added to Y (cleared by the decode kernel) with coalesced fp32 reductions.  Within a part the expander groups
// take units and column ranges in turn, so that consecutive slots come from different groups.
//
// Every wait on an mbarrier is bounded; a wait that gives up sets SQNN_E_TIMEOUT in the status word and
// makes all roles leave their loops; after a bounded wait for the copies and MMAs in flight the kernel frees its tensor
// memory and returns.
#include "sqnn_launch.h"
#include "sqnn_tc.cuh"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace sqnn {

namespace {

constexpr uint32_t MROWS = 128;           // weight rows per unit = MMA M = TMEM lanes
constexpr uint32_t KX = 128;              // columns per X stage (two TMA boxes of 64)
constexpr uint32_t MACRO = 2 * KX;        // columns whose bits an expander thread takes at a time
constexpr uint32_t MAX_SLOTS = 8;         // A slots per unit
constexpr uint32_t MAX_XSTAGES = 8;
constexpr uint32_t MAX_UNITS = 4;
constexpr uint32_t MAX_ACC_COLS = 384;    // TMEM columns of all accumulators; the other 128 and more are A slots
constexpr uint32_t XSTAGE_BUDGET = 192 * 1024;
constexpr uint64_t WAIT_LIMIT_CYCLES = 4000000000ull;   // about 2 s at 2 GHz

// Set by sqnn_set_debug_flags (for the library's own tests).
std::atomic<uint32_t> g_debug_flags{0};
std::atomic<uint64_t> g_debug_wait_cycles{0};

struct MmaArgs {
    const uint32_t *bits32;       // decoded planes in the workspace
    uint64_t plane_words32;       // 32-bit words per plane in the workspace
    const uint32_t *mask32;
    const float *alpha;
    float *y;
    int64_t ldy;
    uint64_t m, n;
    uint32_t n_q;
    uint32_t batch;
    uint32_t N;                   // batch rows per tile = MMA N (multiple of 16)
    uint32_t chunks;              // batch chunks
    uint32_t plane_groups;
    uint32_t macros;              // 256-column macros per row
    uint32_t total;               // tiles x macros
    uint32_t slots, xstages;      // A slots per unit (a power of two), X stages
    uint32_t acc_cols;            // first TMEM column of the A slots
    uint32_t skip_loads;          // test only: the TMA role issues no loads
    uint64_t wait_limit;          // cycles a bounded wait may take
    uint32_t *status;
};

// A row's packed bits as a stream of 256-column macros, eight words each.  ALIGNED: rows start on 16-byte
// boundaries; otherwise the three 16-byte vectors that cover a macro are fetched and shifted into place when
// the bits are used.
template <bool ALIGNED>
struct BitStream {
    static constexpr uint32_t RAW = ALIGNED ? 8 : 12;
    uint32_t t[RAW];
    const uint32_t *at, *first, *last;   // next macro; the vector's first word and the end of its last one
    uint32_t shift;
    bool inside;                         // all macros of this stream lie inside the vector with their slack
    // vec: 8-byte aligned, `words` long; from bit `pos` of it, `count` macros
    SQNN_DEV void open(const uint32_t *__restrict__ vec, uint64_t words, uint64_t pos, uint32_t count)
    {
        const uint32_t lead = (uint32_t)(reinterpret_cast<uintptr_t>(vec) >> 2) & 3u;     // words past a 16-byte boundary
        const uint64_t p = pos + 32 * lead;
        first = vec;
        last = vec + words;
        at = vec - lead + ((p >> 7) << 2);
        shift = (uint32_t)p & 127u;
        inside = at >= first && at + (uint64_t)count * 8 + (RAW - 8) <= last;
    }
    SQNN_DEV void fetch()
    {
        if (inside) {
#pragma unroll
            for (uint32_t k = 0; k < RAW; k += 4)
                asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(t[k]), "=r"(t[k + 1]), "=r"(t[k + 2]), "=r"(t[k + 3]) : "l"(at + k));
        } else {
#pragma unroll
            for (uint32_t k = 0; k < RAW; ++k) {
                t[k] = 0u;
                if (at + k >= first && at + k < last) t[k] = at[k];
            }
        }
        at += 8;
    }
    SQNN_DEV void take(uint32_t (&out)[8])
    {
        uint32_t q[RAW];
#pragma unroll
        for (uint32_t k = 0; k < RAW; ++k) q[k] = settle(t[k]);
        if constexpr (!ALIGNED) {
            const bool two = (shift & 64u) != 0, one = (shift & 32u) != 0;
#pragma unroll
            for (uint32_t k = 0; k < 10; ++k) q[k] = two ? q[k + 2] : q[k];
#pragma unroll
            for (uint32_t k = 0; k < 9; ++k) q[k] = one ? q[k + 1] : q[k];
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k) out[k] = __funnelshift_r(q[k], q[k + 1], shift & 31u);
        } else {
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k) out[k] = q[k];
        }
    }
};

// One part of the work of a CTA: macros [m0, m0 + len) of a tile, and how the phases share them.
template <uint32_t PHASES>
struct Part {
    uint32_t chunk, pg, group;    // batch chunk, plane group, row group
    uint32_t m0, len, base, rem;  // phase p takes base + (p < rem) macros from first(p) on
    SQNN_DEV Part(const MmaArgs &M, uint32_t pos, uint32_t end)
    {
        const uint32_t tile = pos / M.macros;
        m0 = pos - tile * M.macros;
        len = min(M.macros - m0, end - pos);
        const uint32_t rest = tile / M.chunks;
        chunk = tile - rest * M.chunks;
        group = rest / M.plane_groups;
        pg = rest - group * M.plane_groups;
        base = len / PHASES;
        rem = len - base * PHASES;
    }
    SQNN_DEV uint32_t first(uint32_t p) const { return m0 + p * base + min(p, rem); }
    SQNN_DEV uint32_t count(uint32_t p) const { return base + (p < rem ? 1u : 0u); }
    SQNN_DEV uint32_t rounds() const { return base + (rem ? 1u : 0u); }
    SQNN_DEV uint32_t active(uint32_t i) const { return i < base ? PHASES : rem; }
};

// Expander groups (four warps each) of the unit counts: every unit has as many (its phases), four in all where
// that divides.
SQNN_HD constexpr uint32_t phases_of(uint32_t units) { return units == 1 ? 4 : units == 2 ? 2 : 1; }
SQNN_HD constexpr uint32_t threads_of(uint32_t units) { return units * phases_of(units) * 128 + 32 + units * 32; }

// Order of the X stages inside a part, the same for all roles: round i (one macro of every active phase), half
// c of the macro, phase p.  Every unit has its own ring of A slots; within (i, c) the slots of the phases
// alternate.  A slot holds SLOT_COLS TMEM columns (two bf16 each): the 128 columns of an X stage or half of them.
template <uint32_t UNITS, bool ALIGNED, uint32_t SLOT_COLS>
__global__ void __launch_bounds__(threads_of(UNITS), 1)
k_decode_mma(const __grid_constant__ CUtensorMap xmap, const MmaArgs M)
{
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ uint64_t bars[2 * MAX_UNITS * MAX_SLOTS + 2 * MAX_XSTAGES + 2 + MAX_UNITS];
    __shared__ uint32_t tmem_slot, abort_word;
    volatile uint32_t *abort_flag = &abort_word;
    // barriers by shared address: barrier i of a kind is 8 i bytes further on
    const uint32_t full_a = smem_addr(bars), empty_a = full_a + 8 * MAX_UNITS * MAX_SLOTS, full_x = empty_a + 8 * MAX_UNITS * MAX_SLOTS;
    const uint32_t empty_x = full_x + 8 * MAX_XSTAGES, accum = empty_x + 8 * MAX_XSTAGES, acc_free = accum + 8;
    const uint32_t mma_over = acc_free + 8;                      // per unit, after a timeout: its MMAs are over
    const uint32_t x_sa = (smem_addr(smem_raw) + 1023u) & ~1023u;
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t units = UNITS, PHASES = phases_of(UNITS), groups = units * PHASES;
    const uint32_t box_bytes = M.N * 128, x_bytes = 2 * box_bytes;
    const uint32_t begin = (uint32_t)((uint64_t)M.total * blockIdx.x / gridDim.x);
    const uint32_t end = (uint32_t)((uint64_t)M.total * (blockIdx.x + 1) / gridDim.x);
    constexpr uint32_t PER_X = KX / 2 / SLOT_COLS;                           // slots per X stage and unit
    const uint32_t slot_mask = M.slots - 1, slot_shift = 31 - __clz((int)M.slots);

    if (warp == 4 * groups + 1) tmem_alloc(&tmem_slot, 512);
    if (warp == 4 * groups) {
        for (uint32_t s = lane; s < M.slots * units; s += 32) { mbar_init(full_a + 8 * s, 4); mbar_init(empty_a + 8 * s, 1); }
        if (lane < M.xstages) { mbar_init(full_x + 8 * lane, 1); mbar_init(empty_x + 8 * lane, units); }
        if (lane == 31) {
            mbar_init(accum, units);
            mbar_init(acc_free, 4 * groups);
            for (uint32_t u = 0; u < units; ++u) mbar_init(mma_over + 8 * u, 1);
            abort_word = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    launch_dependents();                                     // after the allocation: see k_gemv_tc

    if (warp < 4 * groups) {
        // ------------------------------ expander groups ------------------------------
        const uint32_t g = warp >> 2, quad = warp & 3;
        const uint32_t p = g / units, u = g - p * units;
        const uint32_t lane_sel = (quad * 32) << 16;
        uint32_t seq0 = 0, part_no = 0;
        for (uint32_t pos = begin; pos < end;) {
            const Part<PHASES> P(M, pos, end);
            const uint32_t row_in = P.group * MROWS + quad * 32 + lane;
            const uint64_t row = row_in < M.m ? row_in : M.m - 1;           // rows past the end repeat the last one
            uint32_t plane = P.pg * units + u;
            if (plane >= M.n_q) plane = M.n_q - 1;                          // weighted with zero in the epilogue
            const uint64_t c0 = row * M.n + (uint64_t)P.first(p) * MACRO;
            const uint32_t count = P.count(p);
            BitStream<ALIGNED> sm, sb;
            sm.open(M.mask32, M.plane_words32, c0, count);
            sb.open(M.bits32 + plane * M.plane_words32, M.plane_words32, c0, count);
            if (count) sm.fetch();
            // decoded planes and cleared Y are in place; mask and activations are inputs and were before (sqnn_decode.cuh)
            if (part_no == 0) wait_prior_grid();
            if (count) sb.fetch();
            uint32_t seq = seq0;
            for (uint32_t i = 0; i < count; ++i) {
                uint32_t mw[8], bw[8];
                sm.take(mw);
                sb.take(bw);
                if (i + 1 < count) { sm.fetch(); sb.fetch(); }
                const uint32_t act = P.active(i);
                constexpr uint32_t WORDS = SLOT_COLS / 16;                  // 2 or 4: 32 columns each
#pragma unroll
                for (uint32_t k = 0; k < 2 * PER_X; ++k) {                  // slots of the macro
                    const uint32_t s = seq + k * act + p, use = s >> slot_shift, slot = u * M.slots + (s & slot_mask);
                    const uint32_t at = tmem_base + lane_sel + M.acc_cols + slot * SLOT_COLS;
                    uint32_t v[32];
                    expand32(mw[k * WORDS], bw[k * WORDS], v);
                    expand32(mw[k * WORDS + 1], bw[k * WORDS + 1], v + 16);
                    if (use > 0) {
                        if (!mbar_wait_warp(empty_a + 8 * slot, (use - 1) & 1u, abort_flag, M.status, M.wait_limit)) goto leave;
                        tc_fence_after();
                    }
                    tmem_st16(at, v);
                    tmem_st16(at + 16, v + 16);
                    if constexpr (WORDS == 4) {
                        expand32(mw[k * WORDS + 2], bw[k * WORDS + 2], v);
                        expand32(mw[k * WORDS + 3], bw[k * WORDS + 3], v + 16);
                        tmem_st16(at + 32, v);
                        tmem_st16(at + 48, v + 16);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full_a + 8 * slot);
                }
                seq += 2 * PER_X * act;
            }
            seq0 += 2 * PER_X * P.len;
            // ------------------------------ epilogue of the part ------------------------------
            const uint32_t b0 = P.chunk * M.N;
            const uint32_t r = row_in;
            float al[units];
#pragma unroll
            for (uint32_t k = 0; k < units; ++k) {
                const uint32_t pl = P.pg * units + k;
                al[k] = pl < M.n_q && r < M.m ? 0.5f * __ldg(M.alpha + (uint64_t)r * M.n_q + pl) : 0.0f;
            }
            if (!mbar_wait_warp(accum, part_no & 1u, abort_flag, M.status, M.wait_limit)) goto leave;
            tc_fence_after();
            float *dst = M.y + (int64_t)(b0 + g * 16) * M.ldy + (int64_t)r;
            for (uint32_t j = g; j < M.N / 16; j += groups, dst += (int64_t)groups * 16 * M.ldy) {
                if (b0 + j * 16 >= M.batch) break;
                float sum[16];
#pragma unroll
                for (uint32_t e = 0; e < 16; ++e) sum[e] = 0.0f;
#pragma unroll
                for (uint32_t k = 0; k < units; ++k) {
                    uint32_t d[16];
                    tmem_ld16(tmem_base + lane_sel + k * M.N + j * 16, d);
#pragma unroll
                    for (uint32_t e = 0; e < 16; ++e) sum[e] = fmaf(al[k], __uint_as_float(d[e]), sum[e]);
                }
                if (r < M.m) {
                    float *q = dst;
#pragma unroll
                    for (uint32_t e = 0; e < 16; ++e, q += M.ldy)
                        if (b0 + j * 16 + e < M.batch) atomicAdd(q, sum[e]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free);
            ++part_no;
            pos += P.len;
        }
    } else if (warp == 4 * groups) {
        // ------------------------------ activations by TMA ------------------------------
        if (lane == 0 && !M.skip_loads) {
            uint32_t stage = 0, use = 0;
            bool ok = true;
            for (uint32_t pos = begin; pos < end && ok;) {
                const Part<PHASES> P(M, pos, end);
                const int32_t b0 = (int32_t)(P.chunk * M.N);
                for (uint32_t i = 0; i < P.rounds() && ok; ++i) {
                    const uint32_t act = P.active(i);
                    for (uint32_t cp = 0; cp < 2 * act && ok; ++cp) {
                        const uint32_t c = cp >= act ? 1u : 0u, p = cp - c * act;
                        if (use > 0) ok = mbar_wait(empty_x + 8 * stage, (use - 1) & 1u, abort_flag, M.status, M.wait_limit);
                        if (!ok) break;
                        const int32_t col = (int32_t)((P.first(p) + i) * MACRO + c * KX);
                        mbar_expect_tx(full_x + 8 * stage, x_bytes);
                        tma_load_2d(x_sa + stage * x_bytes, &xmap, full_x + 8 * stage, col, b0);
                        tma_load_2d(x_sa + stage * x_bytes + box_bytes, &xmap, full_x + 8 * stage, col + 64, b0);
                        if (++stage == M.xstages) { stage = 0; ++use; }
                    }
                }
                pos += P.len;
            }
            // after a wait that gave up: copies in flight must land before the block's shared memory goes away
            if (!ok)
                for (uint32_t s = 0; s < M.xstages; ++s) {
                    const uint32_t issued = use + (s < stage ? 1u : 0u);
                    if (issued) mbar_drain(full_x + 8 * s, (issued - 1) & 1u, M.wait_limit);
                }
        }
    } else {
        // ------------------------------ MMA issuers (one converged warp per unit) ------------------------------
        const uint32_t u = warp - (4 * groups + 1);
        const uint32_t idesc = instr_desc_bf16(M.N), d_tmem = tmem_base + u * M.N, a_tmem = tmem_base + M.acc_cols + u * M.slots * SLOT_COLS;
        // descriptors differ only in the start-address field (units of 16 bytes)
        const uint64_t x_desc0 = smem_desc_sw128(x_sa);
        const uint32_t x_step = x_bytes >> 4, box_step = box_bytes >> 4;
        const uint32_t my_full = full_a + 8 * u * M.slots, my_empty = empty_a + 8 * u * M.slots;
        uint32_t xs = 0, x_parity = 0, seq = 0, part_no = 0;      // first X stage of the round and its parity
        for (uint32_t pos = begin; pos < end;) {
            const Part<PHASES> P(M, pos, end);
            if (part_no && !mbar_wait_warp(acc_free, (part_no - 1) & 1u, abort_flag, M.status, M.wait_limit)) goto leave;
            uint32_t accumulate = 0;                              // the first slot of a part overwrites the accumulator
            for (uint32_t i2 = 0; i2 < 2 * P.rounds(); ++i2) {
                const uint32_t act = P.active(i2 >> 1);
#pragma unroll
                for (uint32_t j = 0; j < PER_X; ++j) {
                    uint32_t stage = xs, parity = x_parity;
                    for (uint32_t p = 0; p < act; ++p, ++seq) {
                        const uint32_t slot = seq & slot_mask;
                        if (j == 0 && !mbar_wait_warp(full_x + 8 * stage, parity, abort_flag, M.status, M.wait_limit)) goto leave;
                        if (!mbar_wait_warp(my_full + 8 * slot, (seq >> slot_shift) & 1u, abort_flag, M.status, M.wait_limit)) goto leave;
                        tc_fence_after();
                        mma_slot<SLOT_COLS / 8>(d_tmem, a_tmem + slot * SLOT_COLS, x_desc0 + stage * x_step + j * box_step, idesc,
                                                accumulate, my_empty + 8 * slot, box_step);
                        accumulate = 1;
                        if (j == PER_X - 1) mma_commit(empty_x + 8 * stage);
                        if (++stage == M.xstages) { stage = 0; parity ^= 1u; }
                    }
                    if (j == PER_X - 1) { xs = stage; x_parity = parity; }
                }
            }
            mma_commit(accum);
            ++part_no;
            pos += P.len;
        }
    }
leave:
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*abort_flag) {                                           // (the same for all: nobody waits any more)
        // tensor and shared memory must outlive the MMAs that were issued
        if (warp > 4 * groups) {
            const uint32_t over = mma_over + 8 * (warp - (4 * groups + 1));
            mma_commit(over);
            mbar_drain(over, 0, M.wait_limit);
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    if (warp == 4 * groups + 1) tmem_dealloc(tmem_base, 512);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static std::atomic<EncodeTiledFn> known{nullptr};         // several threads may ask at once
    EncodeTiledFn fn = known.load();
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            known.store(fn = (EncodeTiledFn)p);
    }
    return fn;
}

}  // namespace

DebugKnobs debug_knobs() { return DebugKnobs{g_debug_flags.load(), g_debug_wait_cycles.load()}; }

// Workspace of the two-stage form: the decoded planes as packed bits (1 bit per weight and plane).
size_t mma_workspace_bytes(const sqnn_desc *desc, uint32_t)
{
    const uint64_t words64 = (desc->m * desc->n + 63) / 64;
    return (size_t)((desc->n_q * words64 * 8 + 255) / 256 * 256);
}

int mma_dispatch(const sqnn_desc *desc, const DecodeArgs &A0, const uint64_t *d_mask, const float *d_alpha,
                 const void *d_x, int64_t ldx, uint32_t batch, float *d_y, int64_t ldy, void *d_workspace,
                 cudaStream_t st)
{
    if (((uintptr_t)d_x & 15) != 0 || (ldx % 8) != 0) return SQNN_E_UNSUPPORTED;   // TMA: 16-byte base and pitch
    if (desc->n > 0x7fffffffull || batch > 0x7fffffffu) return SQNN_E_UNSUPPORTED;
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return SQNN_E_CUDA;

    MmaArgs M;
    M.bits32 = (const uint32_t *)d_workspace;
    M.plane_words32 = A0.words64 * 2;
    M.mask32 = (const uint32_t *)d_mask;
    M.alpha = d_alpha;
    M.y = d_y;
    M.ldy = ldy;
    M.m = desc->m;
    M.n = desc->n;
    M.n_q = desc->n_q;
    M.batch = batch;
    M.status = A0.status;
    const DebugKnobs dbg = debug_knobs();
    M.skip_loads = (dbg.flags & 1u) ? 1u : 0u;
    M.wait_limit = dbg.wait_cycles ? dbg.wait_cycles : WAIT_LIMIT_CYCLES;

    // Units of a tile: all planes of 128 rows share the activation tile, up to four; more planes are taken in equal
    // groups.  (One plane with 256 rows per tile uses an activation tile twice but cuts the columns into twice as
    // many parts to add up: 5 to 25 % slower but for batch 16 and 32 of a 4096 x 9216 layer, where it is 1 to 2 %
    // faster.)
    const uint32_t units = M.n_q <= 4 ? M.n_q : M.n_q <= 6 ? 3u : 4u;
    M.plane_groups = (M.n_q + units - 1) / units;
    // Batch rows per tile: what the accumulators leave room for, in equal chunks.
    const uint32_t n_max = units == 1 ? 256u : MAX_ACC_COLS / units / 16 * 16;
    M.chunks = (batch + n_max - 1) / n_max;
    M.N = ((batch + M.chunks - 1) / M.chunks + 15) / 16 * 16;
    M.acc_cols = (units * M.N + 31) / 32 * 32;
    // A slots of 64 TMEM columns if every unit gets two of them, else of 32; one slot of 32 per unit is enough
    // where three or four units take turns on the tensor cores
    const uint32_t per_unit = (512 - M.acc_cols) / units, slot_cols = per_unit >= 128 ? 64u : 32u;
    M.slots = per_unit / slot_cols >= 8 ? 8u : per_unit / slot_cols >= 4 ? 4u : per_unit / slot_cols >= 2 ? 2u : 1u;
    const size_t x_bytes = (size_t)M.N * KX * 2;
    M.xstages = (uint32_t)(XSTAGE_BUDGET / x_bytes < MAX_XSTAGES ? XSTAGE_BUDGET / x_bytes : MAX_XSTAGES);
    const size_t smem = M.xstages * x_bytes + 1024;
    M.macros = (uint32_t)((desc->n + MACRO - 1) / MACRO);
    const uint64_t total = (M.m + MROWS - 1) / MROWS * M.plane_groups * M.chunks * M.macros;
    if (total > 0x7fffffffull || M.m > 0x7fffff00ull) return SQNN_E_UNSUPPORTED;
    M.total = (uint32_t)total;
    const uint32_t grid = M.total < (uint32_t)sm_count() ? M.total : (uint32_t)sm_count();
    // rows of mask and planes start on 16-byte boundaries
    const bool aligned = desc->n % 128 == 0 && ((uintptr_t)d_mask & 15) == 0 && (M.plane_words32 % 4 == 0 || M.n_q == 1);

    CUtensorMap xmap;
    const cuuint64_t gdim[2] = {(cuuint64_t)desc->n, (cuuint64_t)batch};
    const cuuint64_t gstride[1] = {(cuuint64_t)ldx * 2};
    const cuuint32_t box[2] = {KX / 2, M.N};
    const cuuint32_t estride[2] = {1, 1};
    if (encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(d_x), gdim, gstride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return SQNN_E_CUDA;

    // stage 1: the decode kernel writes the planes as packed bits into the workspace and clears Y
    const int rc = decode_bits_dispatch(A0, d_workspace, ClearArgs{d_y, desc->m, ldy, batch, 0}, st);
    if (rc != SQNN_OK) return rc;
#define SQNN_MMA_PICK(U, COLS) (aligned ? k_decode_mma<U, true, COLS> : k_decode_mma<U, false, COLS>)
    auto k = units == 1   ? SQNN_MMA_PICK(1, 64)
             : units == 2 ? (slot_cols == 64 ? SQNN_MMA_PICK(2, 64) : SQNN_MMA_PICK(2, 32))
             : units == 3 ? (slot_cols == 64 ? SQNN_MMA_PICK(3, 64) : SQNN_MMA_PICK(3, 32))
                          : SQNN_MMA_PICK(4, 32);
#undef SQNN_MMA_PICK
    return launch_kernel(k, grid, threads_of(units), smem, st, xmap, M);
}

}  // namespace sqnn

// For the library's own tests: bit 0 of `flags` makes the large-batch kernel's loader issue no loads, bit 1 the
// small-batch kernel's MMA warps report no completion, bit 2 the walk no bulk copies, so that the bounded waits of the roles behind them run out;
// wait_limit_cycles (0 = the kernel's default, one or two seconds) is the number of clock cycles such a wait may take.  Affects calls made after it; not meant for applications.
extern "C" void sqnn_set_debug_flags(uint32_t flags, uint64_t wait_limit_cycles)
{
    sqnn::g_debug_flags.store(flags);
    sqnn::g_debug_wait_cycles.store(wait_limit_cycles);
}

// ---------------------------------------------------------------------------------------------
// Tensor-core product for callers that must not allocate device memory.
//
// Some hosts of this library run where cudaMalloc is off limits: inside a stream capture, inside
// a framework that owns the whole device heap through its own pool, or in a serving loop whose
// memory plan is frozen at start-up.  For them the scratch that sqnn_decode_matmul takes from
// the caller (the decoded planes as packed bits) lives in the array below, which is part of the
// loaded library image on every GPU that loads it, for as long as the process lives.
// ---------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char sqnn_static_scratch[SQNN_STATIC_SCRATCH_BYTES];

namespace {

// In host code `sqnn_static_scratch` is only a handle for the runtime, not a device address, so
// the address is asked for once per device (with that device current) and remembered.
int static_scratch_address(void **out)
{
    static std::mutex mu;
    static void *addr[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SQNN_E_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, sqnn_static_scratch) != cudaSuccess || !p) return SQNN_E_CUDA;
        addr[dev] = p;
    }
    *out = addr[dev];
    return SQNN_OK;
}

}  // namespace

static int decode_matmul_static_queue(const sqnn_desc *desc, const void *d_blob, const uint64_t *d_mask,
                                      const float *d_alpha, const void *d_x, int x_dtype, uint32_t batch,
                                      int64_t ldx, float *d_y, int64_t ldy, uint32_t *d_status,
                                      void *cuda_stream)
{
    sqnn::DecodeArgs A;
    int rc = sqnn::fill_decode_args(desc, d_blob, d_status, &A);
    if (rc != SQNN_OK) return rc;
    if (!d_mask || !d_alpha || !d_x || !d_y || batch == 0) return SQNN_E_INVALID_ARG;
    if (ldx < (int64_t)desc->n || ldy < (int64_t)desc->m) return SQNN_E_INVALID_ARG;
    if (((uintptr_t)d_mask & 7) || ((uintptr_t)d_alpha & 3) || ((uintptr_t)d_y & 3)) return SQNN_E_INVALID_ARG;
    if (x_dtype != SQNN_X_F32 && x_dtype != SQNN_X_BF16) return SQNN_E_INVALID_ARG;
    if (x_dtype != SQNN_X_BF16 || batch < 16 || batch > SQNN_MAX_BATCH || desc->n > (1ull << 30))
        return SQNN_E_UNSUPPORTED;
    if (sqnn::mma_workspace_bytes(desc, batch) > SQNN_STATIC_SCRATCH_BYTES) return SQNN_E_WORKSPACE;
    void *scratch = nullptr;
    rc = static_scratch_address(&scratch);
    if (rc != SQNN_OK) return rc;
    // Nothing in the scratch has to start at zero: the decode stage overwrites every word the
    // product stage reads.  Y is cleared by the product path itself.
    return sqnn::mma_dispatch(desc, A, d_mask, d_alpha, d_x, ldx, batch, d_y, ldy, scratch,
                              (cudaStream_t)cuda_stream);
}

extern "C" int sqnn_decode_matmul_static(const sqnn_desc *desc, const void *d_blob, const uint64_t *d_mask,
                                         const float *d_alpha, const void *d_x, int x_dtype, uint32_t batch,
                                         int64_t ldx, float *d_y, int64_t ldy, uint32_t *d_status,
                                         void *cuda_stream)
{
    sqnn::ApiScope scope("sqnn_decode_matmul_static");
    return scope.finish(decode_matmul_static_queue(desc, d_blob, d_mask, d_alpha, d_x, x_dtype, batch, ldx, d_y, ldy,
                                                   d_status, cuda_stream),
                        d_status, (cudaStream_t)cuda_stream);
}
