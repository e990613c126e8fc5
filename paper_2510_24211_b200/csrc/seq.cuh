// What the kernels of a forward share: the state of the sequences it works on and the layout of the KV cache.
#pragma once
#include "common.cuh"

namespace scd {

template <class T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <class T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

struct SeqState {             // where window inputs and positions come from
    const int *ids;           // explicit [Q][Mq] or NULL
    const int *n_known;       // [B]
    const int *tokens;        // [B][token_stride] conditional stream record
    const int *tokens_u;      // [B][prompt_cap] unconditional prompt
    const int *drafts;        // [B][L]
    int token_stride, prompt_cap, prompt_len, L, B, Mq, pos_override, vocab_in;
    const int *skip;          // all sequences finished: nothing to do
};

__device__ __forceinline__ int base_position(const SeqState &s, int q)
{
    return s.pos_override >= 0 ? s.pos_override : s.n_known[q % s.B] - 1;
}

struct KvLayout {
    void *k_pool, *v_pool;        // this layer's pools
    const int *page_table;        // [Q][pages_per_seq]
    int pages_per_seq, page_tokens, page_shift, n_kv_heads, head_dim, max_seq;
};

template <class T>
__device__ __forceinline__ size_t kv_offset(const KvLayout &kv, int q, int pos, int kvh)
{
    const int page = kv.page_table[(size_t)q * kv.pages_per_seq + (pos >> kv.page_shift)];
    return (((size_t)page * kv.n_kv_heads + kvh) * kv.page_tokens + (pos & (kv.page_tokens - 1))) * kv.head_dim;
}

}  // namespace scd
