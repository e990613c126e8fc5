// Launch interface of the linear layers of fp32 models (linear_f32.cu) and of the plain fp32 attention.
#pragma once
#include "seq.cuh"

namespace scd {

// y = x W^T with the operation around it: F32_STORE y = .; F32_ADD y += .; F32_SWIGLU y = silu(gate) * up;
// F32_QKV rotates Q and K: Q goes to y, K and V of the rows to their cache slots.
enum { F32_STORE = 0, F32_ADD = 1, F32_SWIGLU = 2, F32_QKV = 3 };

struct LinearF32 {
    const float *x;            // [rows][K]
    const float *gain;         // RMSNorm of the x rows with this gain (NULL: x as it is)
    float eps;
    const float *w[3];         // [N][K]; SwiGLU: gate, up; QKV: Wq, Wk, Wv
    float *y;                  // [rows][ldy]
    int rows, N, K, ldy;       // N: output columns (QKV: (H + 2 Hkv) dh)
    const int *skip;           // optional device flag: set = nothing to do
    // F32_QKV
    SeqState seq;
    KvLayout kv;
    const float2 *rope;
    int n_heads;
};

int linear_f32(int epi, const LinearF32 &p, cudaStream_t st);

// Causal window attention over the paged KV cache, any head_dim that is a multiple of 32 (attention_simt.cu): fp32
// models, and bf16 models whose head_dim or page size the tensor-core kernels do not take. qkv: fp32 rows of
// (H + 2 Hkv) dh, Q rotated. lo_plane > 0: the output as two planes (out[lo_plane + .] = T(o - T(o))).
template <class T>
int attention_simt(const SeqState &seq, const float *qkv, const KvLayout &kv, T *out, int Q, int n_heads, float scale,
                   long long lo_plane, cudaStream_t st);

// A launch that may start while the kernel in front of it runs (the kernel calls pdl_wait()).
template <class... P, class... A>
int launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    SCD_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
    count_launches(1);
    return SCD_OK;
}

}  // namespace scd
