// Internal: launch helpers shared by the kernel translation units.
#pragma once
#include "sqnn.h"
#include "sqnn_decode.cuh"

namespace sqnn {
int fill_decode_args(const sqnn_desc *d, const void *d_blob, uint32_t *d_status, DecodeArgs *A);
int sm_count();
// Raises a kernel's dynamic shared-memory limit when `smem` needs it; remembered per kernel and
// device so that repeated launches cost nothing on the host.
int ensure_dynamic_smem(const void *kernel, size_t smem);
// Queues the packed-bits decode of every plane into `d_out` (n_q * ceil(mn/64) uint64); the same kernel clears
// what `clear` describes.
int decode_bits_dispatch(const DecodeArgs &A, void *d_out, const ClearArgs &clear, cudaStream_t st);

// Launches a kernel that begins with wait_prior_grid() (sqnn_decode.cuh): it may be scheduled while the
// kernel queued before it on the stream is finishing, so that consecutive launches do not each pay the launch
// latency.
template <typename... P, typename... Q>
inline int launch_kernel(void (*kernel)(P...), uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st, const Q &...args)
{
    if (ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), smem) != SQNN_OK) return SQNN_E_CUDA;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess ? SQNN_OK : SQNN_E_CUDA;
}
// What sqnn_set_debug_flags was given last (zeros in normal use).
struct DebugKnobs {
    uint32_t flags;
    uint64_t wait_cycles;
};
DebugKnobs debug_knobs();

size_t mma_workspace_bytes(const sqnn_desc *desc, uint32_t batch);
int mma_dispatch(const sqnn_desc *desc, const DecodeArgs &A, const uint64_t *d_mask, const float *d_alpha,
                 const void *d_x, int64_t ldx, uint32_t batch, float *d_y, int64_t ldy, void *d_workspace,
                 cudaStream_t st);

// A device entry point: an NVTX range for its duration on the host, and in checked mode
// (SQNN_DEBUG_CHECKS=1) the wait for the stream and the translation of what it left behind.
class ApiScope {
  public:
    explicit ApiScope(const char *name);
    ~ApiScope();
    ApiScope(const ApiScope &) = delete;
    ApiScope &operator=(const ApiScope &) = delete;
    // rc of the queueing code -> what the entry point returns
    int finish(int rc, const uint32_t *d_status, cudaStream_t st) const;
};
}  // namespace sqnn
