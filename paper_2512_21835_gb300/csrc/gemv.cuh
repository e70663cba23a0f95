// gemv.cuh -- what the decode projections' translation units share: the
// parameters of a matrix-vector product with its fused epilogue, small device
// helpers, and the launch with programmatic stream serialisation.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "internal.h"

namespace loip {

enum { EPI_QKV = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_LOGITS = 3 };

struct GemvParams {
    const float* in;     // [B, K] fp32 activations
    const uint16_t* g;   // [K] gain: input is RMSNorm(in) * g when non-null
    const uint16_t* w0;  // [N, K]
    const uint16_t* w1;  // [N, K] (SwiGLU up projection)
    int B, K, N, n_units;
    float eps;
    float* out;
    float* z;
    uint64_t* keys;
    // QKV epilogue
    int Hq, Hkv, d;
    const int32_t* positions;
    const int32_t* row_req;
    KvView kv;
    RopeFreqs rope;
    int w_host;  // weights are read in place from mapped host memory: no L2 prefetch of them
    float* qk_raw;  // QK-norm models: query/key rows leave unrotated here ([B][(Hq + 2 Hkv) d])
};

cudaError_t launch_gemv_batch(int epi, const GemvParams& p, cudaStream_t st, bool pdl, int* nblocks_out);
cudaError_t launch_gemv_ring(int epi, const GemvParams& p, cudaStream_t st, bool pdl);

namespace {

__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ float bf2f(uint16_t h) { return __uint_as_float((uint32_t)h << 16); }
__device__ __forceinline__ uint16_t f2bf(float f) { return __bfloat16_as_ushort(__float2bfloat16_rn(f)); }

// Programmatic dependent launch: let the next kernel of the stream start its
// independent prologue, and wait for the previous kernel's results.  Both are
// no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Orderable 64-bit argmax key: larger value wins; on equal values the lower
// index wins (the low word stores ~index).
__device__ __forceinline__ uint64_t argmax_key(float v, uint32_t idx) {
    uint32_t u = __float_as_uint(v);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((uint64_t)u << 32) | (uint64_t)(0xffffffffu - idx);
}

__device__ __forceinline__ char* kv_row(const KvView& kv, int req, int pos, int kv_or_v, int head, int Hkv, int d) {
    int page = pos / kv.page_tokens, t = pos - page * kv.page_tokens;
    char* p = kv.base + kv.page_offsets[(int64_t)req * kv.max_pages + page] + (uint64_t)kv.layer * kv.layer_page_bytes;
    p += ((uint64_t)(kv_or_v * Hkv + head) * kv.page_tokens + t) * (uint64_t)d * 2u;
    return p;
}

// Launch with programmatic stream serialisation when `pdl` (the previous
// operation on the stream is a kernel of the same chain).
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                     Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl ? at : nullptr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace
}  // namespace loip
