// Linear layers of fp32 models, fused with what surrounds them: RMSNorm in front; residual add, SwiGLU, or RoPE and
// the KV-cache write behind. Five launches per decoder layer.
//
// With the few rows of a window these products are bound by latency, not by arithmetic or bytes (the four layers
// of a small decoder are 13 MB that stay in L2), so the split is over output columns: a warp owns NC columns of W
// (for QKV and SwiGLU the NC / 2 pairs whose halves meet in the output operation) and 16 rows of x, its lanes
// split K. W is read once per 16 rows with 16-byte loads, the first of them - like the rotation and the cache slots -
// before the kernel in front is waited for; the x rows go to shared memory once per CTA, two rows of a warp with all
// their loads in flight, and their norms are taken on the way. The 32 partial sums per output are folded with a
// butterfly that halves the rows a lane holds at every step (16 shuffles for 16 rows).
// Whole generation of 256 tokens, four layers of d 256, 16 rows: 173 ms with 32 x 32-tile products that loaded K 32 at
// a time behind barriers, norms and RoPE in launches of their own (51 per step); 65 ms with this split and x staged by
// single loads; 42 ms with the loads in flight together.
#include <algorithm>

#include "linear_f32.cuh"
#include "model.cuh"

namespace scd {

namespace {

constexpr int MT = 16;               // rows per CTA
constexpr int WARPS = 4;
constexpr int KC = 1024;             // K values of the rows in shared memory at a time
constexpr int PRE = 4;               // W loads per column in flight ahead of the wait

template <int VEC> struct Vec;
template <> struct Vec<4> {
    float4 v;
    __device__ static Vec load(const float *p) { return {__ldg((const float4 *)p)}; }
    __device__ static Vec lds(const float *p) { return {*(const float4 *)p}; }
    __device__ static Vec load_cg(const float *p) { return {__ldcg((const float4 *)p)}; }
    __device__ static Vec zero() { return {make_float4(0.f, 0.f, 0.f, 0.f)}; }
    __device__ void sts(float *p) const { *(float4 *)p = v; }
    __device__ void mul(const Vec &g) { v.x *= g.v.x; v.y *= g.v.y; v.z *= g.v.z; v.w *= g.v.w; }
};
template <> struct Vec<1> {
    float v;
    __device__ static Vec load(const float *p) { return {__ldg(p)}; }
    __device__ static Vec lds(const float *p) { return {*p}; }
    __device__ static Vec load_cg(const float *p) { return {__ldcg(p)}; }
    __device__ static Vec zero() { return {0.f}; }
    __device__ void sts(float *p) const { *p = v; }
    __device__ void mul(const Vec &g) { v *= g.v; }
};
__device__ __forceinline__ float dot(const Vec<4> &a, const Vec<4> &b, float s)
{
    return fmaf(a.v.w, b.v.w, fmaf(a.v.z, b.v.z, fmaf(a.v.y, b.v.y, fmaf(a.v.x, b.v.x, s))));
}
__device__ __forceinline__ float dot(const Vec<1> &a, const Vec<1> &b, float s) { return fmaf(a.v, b.v, s); }

// Sums of 16 values over the warp: lane l ends with the sum of value l >> 1.
__device__ __forceinline__ float fold16(const float (&a)[MT], int lane)
{
    float b[8], c[4], d[2];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool up = lane & 16;
        b[i] = (up ? a[i + 8] : a[i]) + __shfl_xor_sync(0xffffffffu, up ? a[i] : a[i + 8], 16);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = lane & 8;
        c[i] = (up ? b[i + 4] : b[i]) + __shfl_xor_sync(0xffffffffu, up ? b[i] : b[i + 4], 8);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool up = lane & 4;
        d[i] = (up ? c[i + 2] : c[i]) + __shfl_xor_sync(0xffffffffu, up ? c[i] : c[i + 2], 4);
    }
    const bool up = lane & 2;
    const float e = (up ? d[1] : d[0]) + __shfl_xor_sync(0xffffffffu, up ? d[0] : d[1], 2);
    return e + __shfl_xor_sync(0xffffffffu, e, 1);
}

template <int EPI, int NC, int VEC>
__global__ void __launch_bounds__(WARPS * 32) linear_f32_kernel(const __grid_constant__ LinearF32 p)
{
    extern __shared__ float xs[];                      // [MT][pitch]
    __shared__ float inv_s[MT];
    pdl_trigger();
    if (p.skip && *p.skip) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.y * MT, K = p.K;
    const int live = min(MT, p.rows - m0);
    const int dh = p.kv.head_dim, half = dh >> 1;
    // the warp's columns: c0 .. c0 + NC - 1 as they come, or pairs (QKV: j and j + dh / 2 of a head; SwiGLU: gate and up)
    const int c0 = (blockIdx.x * WARPS + warp) * NC;
    auto column = [&](int i) -> int {                  // output column (QKV) or row of W
        if (EPI == F32_QKV) { const int e = (c0 + i) >> 1; return (e / half) * dh + e % half + (i & 1) * half; }
        if (EPI == F32_SWIGLU) return (c0 + i) >> 1;
        return c0 + i;
    };
    const float *wrow[NC];
    bool have[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        const int n = column(i);
        have[i] = c0 + i < (EPI == F32_SWIGLU ? 2 * p.N : p.N);
        const float *w = p.w[0];
        int wr = n;
        if (EPI == F32_SWIGLU) w = p.w[i & 1];
        if (EPI == F32_QKV) {
            const int dq = p.n_heads * dh, dkv = p.kv.n_kv_heads * dh;
            if (n >= dq + dkv) { w = p.w[2]; wr = n - dq - dkv; }
            else if (n >= dq) { w = p.w[1]; wr = n - dq; }
        }
        wrow[i] = w + (size_t)(have[i] ? wr : 0) * K;
    }
    const int k_lane = lane * VEC;
    constexpr int STEP = 32 * VEC;
    Vec<VEC> pre[NC][PRE];
#pragma unroll
    for (int i = 0; i < NC; ++i)
#pragma unroll
        for (int t = 0; t < PRE; ++t)
            pre[i][t] = k_lane + t * STEP < K ? Vec<VEC>::load(wrow[i] + k_lane + t * STEP) : Vec<VEC>::zero();

    // QKV: this lane's row sits at `pos`; its rotation and its cache slot (older than the kernel in front)
    const int r = lane >> 1, m = m0 + r, odd = lane & 1;
    bool in_range = false;
    size_t slot = 0;
    float2 cs[NC / 2];
    if (EPI == F32_QKV && r < live) {
        const int q = m / p.seq.Mq, pos = base_position(p.seq, q) + m % p.seq.Mq;
        in_range = pos >= 0 && pos < p.kv.max_seq;
        const int pc = min(max(pos, 0), p.kv.max_seq - 1);
        slot = kv_offset<float>(p.kv, q, pc, 0);
#pragma unroll
        for (int i = 0; i < NC / 2; ++i) cs[i] = p.rope[(size_t)pc * half + ((c0 >> 1) + i) % half];
    }
    pdl_wait();                                        // x comes from the kernel in front
    const float *x = p.x + (size_t)m0 * K;
    float acc[NC][MT];
#pragma unroll
    for (int i = 0; i < NC; ++i)
#pragma unroll
        for (int j = 0; j < MT; ++j) acc[i][j] = 0.f;
    constexpr int RW = MT / WARPS;                     // rows a warp stages
    constexpr int LV = KC / STEP / (VEC == 4 ? 1 : 4); // loads per lane and row in flight together
    if (p.gain && K > KC) {                            // long rows: their norm first
#pragma unroll
        for (int j = 0; j < RW; ++j) {
            const int xr = warp * RW + j;
            float ss = 0.f;
            if (xr < live) for (int k = lane; k < K; k += 32) { const float v = __ldcg(x + (size_t)xr * K + k); ss = fmaf(v, v, ss); }
            ss = warp_sum_f(ss);
            if (lane == 0) inv_s[xr] = 1.0f / sqrtf(ss / (float)K + p.eps);
        }
        __syncwarp();
    }
    for (int k0 = 0; k0 < K; k0 += KC) {
        const int kc = min(KC, K - k0), pitch = min(KC, (K + 3) & ~3) + 4;
        if (k0 > 0) __syncthreads();
#pragma unroll 1
        for (int j = 0; j < RW; j += 2) {
            const int r0 = warp * RW + j;
            float ss[2] = {0.f, 0.f};
#pragma unroll 1
            for (int kb = k_lane; kb < kc; kb += LV * STEP) {
                Vec<VEC> v[2][LV];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int t = 0; t < LV; ++t)
                        v[h][t] = r0 + h < live && kb + t * STEP < kc ? Vec<VEC>::load_cg(x + (size_t)(r0 + h) * K + k0 + kb + t * STEP)
                                                                      : Vec<VEC>::zero();
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int t = 0; t < LV; ++t) {
                        ss[h] = dot(v[h][t], v[h][t], ss[h]);
                        if (kb + t * STEP < kc) v[h][t].sts(xs + (r0 + h) * pitch + kb + t * STEP);
                    }
            }
            if (p.gain) {
#pragma unroll
                for (int h = 0; h < 2; ++h) ss[h] = warp_sum_f(ss[h]);
                if (lane < 2 && K <= KC) inv_s[r0 + lane] = 1.0f / sqrtf((lane ? ss[1] : ss[0]) / (float)K + p.eps);
            }
        }
        __syncthreads();
        // (the gain goes into the weights, the rows' 1 / rms into the sums at the end)
        auto step = [&](int k, Vec<VEC> (&w)[NC]) {
            if (p.gain) {
                const Vec<VEC> g = Vec<VEC>::load(p.gain + k0 + k);
#pragma unroll
                for (int i = 0; i < NC; ++i) w[i].mul(g);
            }
#pragma unroll
            for (int j = 0; j < MT; ++j) {
                const Vec<VEC> xv = Vec<VEC>::lds(xs + j * pitch + k);
#pragma unroll
                for (int i = 0; i < NC; ++i) acc[i][j] = dot(xv, w[i], acc[i][j]);
            }
        };
        int k = k_lane;
        if (k0 == 0) {
#pragma unroll
            for (int t = 0; t < PRE; ++t, k += STEP) {
                Vec<VEC> w[NC];
#pragma unroll
                for (int i = 0; i < NC; ++i) w[i] = pre[i][t];
                if (k < kc) step(k, w);
            }
        }
#pragma unroll 4
        for (; k < kc; k += STEP) {
            Vec<VEC> w[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) w[i] = Vec<VEC>::load(wrow[i] + k0 + k);
            step(k, w);
        }
    }
    // lane l: row l >> 1 of every column; even lanes store the first of a pair (or column), odd lanes the second
    float out[NC];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        out[i] = fold16(acc[i], lane);
        if (p.gain) out[i] *= inv_s[r];
    }
    if (r >= live) return;
    if (EPI == F32_STORE || EPI == F32_ADD) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            if ((i & 1) != odd || !have[i]) continue;
            float *y = p.y + (size_t)m * p.ldy + c0 + i;
            *y = EPI == F32_ADD ? __ldcg(y) + out[i] : out[i];
        }
    } else if (EPI == F32_SWIGLU) {
#pragma unroll
        for (int i = 0; i < NC; i += 2) {
            if (!have[i] || odd) continue;
            p.y[(size_t)m * p.ldy + ((c0 + i) >> 1)] = out[i] / (1.0f + expf(-out[i])) * out[i + 1];
        }
    } else {
        const int dq = p.n_heads * dh, dkv = p.kv.n_kv_heads * dh;
#pragma unroll
        for (int i = 0; i < NC; i += 2) {
            if (!have[i]) continue;
            const int n = column(i);
            float a = out[i], b = out[i + 1];
            if (n < dq + dkv) {
                const float2 t = cs[i / 2];
                const float ra = a * t.x - b * t.y, rb = b * t.x + a * t.y;
                a = ra; b = rb;
            }
            const float v = odd ? b : a;
            if (n < dq) p.y[(size_t)m * p.ldy + n + odd * half] = v;
            else if (in_range) {
                const int e = n < dq + dkv ? n - dq : n - dq - dkv;
                float *pool = (float *)(n < dq + dkv ? p.kv.k_pool : p.kv.v_pool);
                pool[slot + (size_t)(e / dh) * p.kv.page_tokens * dh + e % dh + odd * half] = v;
            }
        }
    }
}

template <int EPI, int NC>
int launch(const LinearF32 &p, cudaStream_t st)
{
    const int cols = EPI == F32_SWIGLU ? 2 * p.N : p.N;
    const dim3 grid((unsigned)((cols + WARPS * NC - 1) / (WARPS * NC)), (unsigned)((p.rows + MT - 1) / MT));
    const size_t smem = (size_t)MT * (std::min(KC, (p.K + 3) & ~3) + 4) * sizeof(float);
    const bool vec = p.K % 4 == 0;
    void (*kernel)(const LinearF32) = vec ? linear_f32_kernel<EPI, NC, 4> : linear_f32_kernel<EPI, NC, 1>;
    if (smem > 48 * 1024) SCD_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return launch_dependent(kernel, grid, dim3(WARPS * 32), smem, st, p);
}

}  // namespace

// Two columns per warp leave the most warps; four halve the shared-memory reads of x per product and pay once
// there are eight warps per SM all the same (148 x 8).
int linear_f32(int epi, const LinearF32 &p, cudaStream_t st)
{
    const long long cols = epi == F32_SWIGLU ? 2ll * p.N : p.N;
    const bool wide = cols / 4 * ((p.rows + MT - 1) / MT) >= 148 * 8;
    switch (epi) {
    case F32_STORE: return wide ? launch<F32_STORE, 4>(p, st) : launch<F32_STORE, 2>(p, st);
    case F32_ADD: return wide ? launch<F32_ADD, 4>(p, st) : launch<F32_ADD, 2>(p, st);
    case F32_SWIGLU: return wide ? launch<F32_SWIGLU, 4>(p, st) : launch<F32_SWIGLU, 2>(p, st);
    default: return wide ? launch<F32_QKV, 4>(p, st) : launch<F32_QKV, 2>(p, st);
    }
}

}  // namespace scd
