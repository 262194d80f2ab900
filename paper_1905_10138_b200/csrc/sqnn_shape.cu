// Instantiates the kernels of one network shape (N_OUT x N_IN given by -DSQNN_NO / -DSQNN_NI; 0 x 0 is the
// run-time-shape fallback).  -DSQNN_PART compiles one part of them, so that the parts of a shape build side by side:
// 0 the decode, 1 the small-batch tensor-core product, 2 the walk over care bits and the choice between the two.
#include "sqnn_gemv_tc.cuh"

#ifndef SQNN_NO
#error "compile with -DSQNN_NO=<n_out> -DSQNN_NI=<n_in>"
#endif

#ifndef SQNN_PART
#error "compile with -DSQNN_PART=<0, 1 or 2>"
#endif

namespace sqnn {

#if SQNN_PART == 0
template <>
int decode_shape<SQNN_NO, SQNN_NI>(const DecodeArgs &A, sqnn_out_mode mode, const uint64_t *d_mask,
                                   const float *d_alpha, uint64_t n, void *d_out, const ClearArgs &clear,
                                   cudaStream_t st)
{
    return launch_decode<SQNN_NO, SQNN_NI>(A, mode, d_mask, d_alpha, n, d_out, clear, st);
}

#else
template <int N_OUT, int N_IN>
int gemv_tc_shape(const DecodeArgs &A, const TcPlan &plan, const uint64_t *d_mask, const float *d_alpha, const void *d_x, int x_dtype,
                  int64_t ldx, uint32_t batch, float *d_y, int64_t ldy, uint64_t m, uint64_t n, cudaStream_t st);
#if SQNN_PART == 1
template <>
int gemv_tc_shape<SQNN_NO, SQNN_NI>(const DecodeArgs &A, const TcPlan &plan, const uint64_t *d_mask, const float *d_alpha,
                                    const void *d_x, int x_dtype, int64_t ldx, uint32_t batch, float *d_y,
                                    int64_t ldy, uint64_t m, uint64_t n, cudaStream_t st)
{
    return x_dtype == SQNN_X_BF16
        ? launch_gemv_tc<SQNN_NO, SQNN_NI, __nv_bfloat16>(A, plan, d_mask, d_alpha, d_x, ldx, batch, d_y, ldy, m, n, st)
        : launch_gemv_tc<SQNN_NO, SQNN_NI, float>(A, plan, d_mask, d_alpha, d_x, ldx, batch, d_y, ldy, m, n, st);
}
#else
template <>
int gemv_tc_shape<SQNN_NO, SQNN_NI>(const DecodeArgs &, const TcPlan &, const uint64_t *, const float *, const void *, int, int64_t,
                                    uint32_t, float *, int64_t, uint64_t, uint64_t, cudaStream_t);

template <>
int gemv_shape<SQNN_NO, SQNN_NI>(const DecodeArgs &A0, const uint64_t *d_mask, const float *d_alpha,
                                 const void *d_x, int x_dtype, int64_t ldx, uint32_t batch, float *d_y,
                                 int64_t ldy, uint64_t m, uint64_t n, cudaStream_t st)
{
    DecodeArgs A = A0;
    uint64_t patches = 0;
    for (uint32_t i = 0; i < A.n_q; ++i) patches += A.pl[i].n_pp;
    const double slices = (double)A.n_q * (double)((A.mn + A.n_out - 1) / A.n_out);
    GemvLayer L;
    L.m = m; L.n = n; L.batch = batch; L.n_q = A.n_q;
    L.tab_words = A.tab_words;
    L.x_bytes = x_dtype == SQNN_X_BF16 ? 2 : 4;
    L.sms = (uint32_t)sm_count();
    L.W = A.W;
    L.density = care_density(A.n_out, A.n_in, (double)patches / slices);
    const GemvTiles own{A.KT, A.W};
    const GemvForms f = SQNN_NO == 0 ? plan_run_time_shape(A.n_out, A.n_in, L) : GemvForms{plan_gemv_tc(L), plan_walk(L), own, own};
    const bool expanding = !take_walk(L, f.tc, f.walk);
    A.KT = expanding ? f.tc_tiles.KT : f.walk_tiles.KT;
    A.W = expanding ? f.tc_tiles.W : f.walk_tiles.W;
    if (expanding)
        return f.tc.ok ? gemv_tc_shape<SQNN_NO, SQNN_NI>(A, f.tc, d_mask, d_alpha, d_x, x_dtype, ldx, batch, d_y, ldy, m, n, st)
                       : SQNN_E_UNSUPPORTED;                       // one row of bits does not fit
    return x_dtype == SQNN_X_BF16
        ? launch_gemv<SQNN_NO, SQNN_NI, __nv_bfloat16>(A, f.walk, d_mask, d_alpha, d_x, ldx, batch, d_y, ldy, m, n, st)
        : launch_gemv<SQNN_NO, SQNN_NI, float>(A, f.walk, d_mask, d_alpha, d_x, ldx, batch, d_y, ldy, m, n, st);
}
#endif
#endif

}  // namespace sqnn
