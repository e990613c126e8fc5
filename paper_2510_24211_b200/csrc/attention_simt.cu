// Causal window attention over the paged KV cache in fp32 arithmetic, any head_dim that is a multiple of 32.
//
// Query i of a stream-sequence sits at position base + i and attends to cache entries 0 .. base + i (its own K/V are
// in the cache). A CTA takes one head and QT queries; its eight warps deal the tiles of 32 keys among
// themselves, so that the chain of a window over a few hundred keys is one or two tiles long: lane = key for the
// scores (a lane reads its whole K row, the queries come from shared memory), lane = dimension for P V. The
// warps' (max, sum, output) are merged at the end in warp order. Bound by the latency of its loads: 16 us per launch
// at 16 rows and 130 keys with one warp per four queries and all keys in sequence through shared memory, 5 us now.
#include "linear_f32.cuh"
#include "model.cuh"

namespace scd {

namespace {

constexpr int QT = 4;            // queries per CTA
constexpr int AW = 8;            // warps

__device__ __forceinline__ float4 load4(const float *p) { return __ldcg((const float4 *)p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p)
{
    const uint2 u = __ldcg((const uint2 *)p);
    const float2 a = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x), b = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
    return make_float4(a.x, a.y, b.x, b.y);
}

template <class T, int DH>
__global__ void __launch_bounds__(AW * 32) attention_simt_kernel(SeqState s, const float *__restrict__ qkv, KvLayout kv,
                                                                 T *__restrict__ out, int n_heads, float scale, long long lo_plane)
{
    constexpr int DPL = DH / 32;
    __shared__ __align__(16) float qs[QT][DH];
    __shared__ float4 ps[AW][32];                      // probabilities of a tile: [key] -> the four queries
    __shared__ float ms[AW][QT], ls[AW][QT];
    __shared__ float os[AW][QT][DH];
    pdl_trigger();
    if (s.skip && *s.skip) return;
    const int q = blockIdx.x / n_heads, hh = blockIdx.x % n_heads, i0 = blockIdx.y * QT;
    const int kvh = hh / (n_heads / kv.n_kv_heads);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nq = min(QT, s.Mq - i0);
    const size_t qstride = (size_t)(n_heads + 2 * kv.n_kv_heads) * DH;
    const int base = base_position(s, q);              // (older than the kernel in front)
    pdl_wait();
    for (int e = tid; e < QT * DH; e += AW * 32) {
        const int qi = e / DH, j = e % DH;
        qs[qi][j] = qi < nq ? __ldcg(qkv + ((size_t)q * s.Mq + i0 + qi) * qstride + (size_t)hh * DH + j) * scale : 0.f;
    }
    __syncthreads();
    const int n_keys = min(base + i0 + nq, kv.max_seq);
    float m[QT], l[QT], acc[QT][DPL];
#pragma unroll
    for (int a = 0; a < QT; ++a) {
        m[a] = -INFINITY; l[a] = 0.f;
#pragma unroll
        for (int c = 0; c < DPL; ++c) acc[a][c] = 0.f;
    }
    for (int k0 = warp * 32; k0 < n_keys; k0 += AW * 32) {
        const int kpos = k0 + lane;
        // pages hold a multiple of 16 tokens: the tile's values are two runs of 16 consecutive rows. The first run is
        // requested before the scores.
        const T *vrow[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) vrow[h] = (const T *)kv.v_pool + kv_offset<T>(kv, q, min(k0 + 16 * h, n_keys - 1) & ~15, kvh) + lane;
        T v0[16][DPL];
#pragma unroll
        for (int j = 0; j < 16; ++j)
#pragma unroll
            for (int c = 0; c < DPL; ++c) v0[j][c] = k0 + j < n_keys ? vrow[0][(size_t)j * DH + 32 * c] : from_f<T>(0.f);
        float sc[QT] = {0.f, 0.f, 0.f, 0.f};
        if (kpos < n_keys) {
            const T *kr = (const T *)kv.k_pool + kv_offset<T>(kv, q, kpos, kvh);
#pragma unroll 16
            for (int j = 0; j < DH; j += 4) {
                const float4 kk = load4(kr + j);
#pragma unroll
                for (int a = 0; a < QT; ++a) {
                    const float4 qv = *(const float4 *)&qs[a][j];
                    sc[a] = fmaf(qv.w, kk.w, fmaf(qv.z, kk.z, fmaf(qv.y, kk.y, fmaf(qv.x, kk.x, sc[a]))));
                }
            }
        }
        float pj[QT];
#pragma unroll
        for (int a = 0; a < QT; ++a) {
            const float v = kpos < n_keys && kpos <= base + i0 + a ? sc[a] : -INFINITY;
            const float m_new = fmaxf(m[a], warp_max(v));
            const float ref = m_new == -INFINITY ? 0.f : m_new;
            const float corr = expf(m[a] - ref);       // (-inf: nothing accumulated yet, 0)
            pj[a] = expf(v - ref);
            l[a] = l[a] * corr + warp_sum_f(pj[a]);
            m[a] = m_new;
#pragma unroll
            for (int c = 0; c < DPL; ++c) acc[a][c] *= corr;
        }
        __syncwarp();
        ps[warp][lane] = make_float4(pj[0], pj[1], pj[2], pj[3]);
        __syncwarp();
        auto add = [&](float4 pb, const T *v, int c) {
            const float x = to_f<T>(v[c]);
            acc[0][c] = fmaf(pb.x, x, acc[0][c]);
            acc[1][c] = fmaf(pb.y, x, acc[1][c]);
            acc[2][c] = fmaf(pb.z, x, acc[2][c]);
            acc[3][c] = fmaf(pb.w, x, acc[3][c]);
        };
#pragma unroll
        for (int j = 0; j < 16; ++j)
#pragma unroll
            for (int c = 0; c < DPL; ++c) add(ps[warp][j], v0[j], c);
        if (k0 + 16 < n_keys) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
#pragma unroll
                for (int c = 0; c < DPL; ++c) v0[j][c] = k0 + 16 + j < n_keys ? vrow[1][(size_t)j * DH + 32 * c] : from_f<T>(0.f);
#pragma unroll
            for (int j = 0; j < 16; ++j)
#pragma unroll
                for (int c = 0; c < DPL; ++c) add(ps[warp][16 + j], v0[j], c);
        }
    }
#pragma unroll
    for (int a = 0; a < QT; ++a) {
        if (lane == 0) { ms[warp][a] = m[a]; ls[warp][a] = l[a]; }
#pragma unroll
        for (int c = 0; c < DPL; ++c) os[warp][a][lane + 32 * c] = acc[a][c];
    }
    __syncthreads();
    for (int e = tid; e < nq * DH; e += AW * 32) {
        const int a = e / DH, j = e % DH;
        float M = -INFINITY, L = 0.f, o = 0.f;
#pragma unroll
        for (int w = 0; w < AW; ++w) M = fmaxf(M, ms[w][a]);
#pragma unroll
        for (int w = 0; w < AW; ++w) {
            const float f = ms[w][a] == -INFINITY ? 0.f : expf(ms[w][a] - M);
            L = fmaf(f, ls[w][a], L);
            o = fmaf(f, os[w][a][j], o);
        }
        const float r = L > 0.f ? o / L : 0.f;
        T *dst = out + ((size_t)q * s.Mq + i0 + a) * (size_t)n_heads * DH + (size_t)hh * DH + j;
        const T hi = from_f<T>(r);
        dst[0] = hi;
        if (lo_plane > 0) dst[lo_plane] = from_f<T>(r - to_f<T>(hi));
    }
}

}  // namespace

template <class T>
int attention_simt(const SeqState &seq, const float *qkv, const KvLayout &kv, T *out, int Q, int n_heads, float scale,
                   long long lo_plane, cudaStream_t st)
{
    const dim3 grid((unsigned)(Q * n_heads), (unsigned)((seq.Mq + QT - 1) / QT));
    auto kernel = kv.head_dim == 32 ? attention_simt_kernel<T, 32> : kv.head_dim == 64 ? attention_simt_kernel<T, 64>
                : kv.head_dim == 96 ? attention_simt_kernel<T, 96> : attention_simt_kernel<T, 128>;
    return launch_dependent(kernel, grid, dim3(AW * 32), 0, st, seq, qkv, kv, out, n_heads, scale, lo_plane);
}
template int attention_simt<float>(const SeqState &, const float *, const KvLayout &, float *, int, int, float, long long, cudaStream_t);
template int attention_simt<__nv_bfloat16>(const SeqState &, const float *, const KvLayout &, __nv_bfloat16 *, int, int, float, long long,
                                           cudaStream_t);

}  // namespace scd
