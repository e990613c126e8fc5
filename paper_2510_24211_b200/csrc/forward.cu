// Window-parallel forward of the Llama-style decoder p_theta (the parallel forward of Algorithm 6: all window
// positions are evaluated in one pass, causal attention over the KV cache plus the window).
//
// Pre-norm blocks: h += Wo Attn(RoPE(Wq n1), RoPE(Wk n1), Wv n1); h += Wdown(silu(Wgate n2) * Wup n2);
// logits = Wlm RMSNorm(h). The residual stream h and the logits are fp32; GEMM inputs, the KV
// cache and the attention output have the model dtype T (float or bf16).
#include <type_traits>
#include <algorithm>
#include <vector>

#include "model.cuh"
#include "gemm.cuh"
#include "linear_f32.cuh"
#include "seq.cuh"

namespace scd {

namespace {

// ---- window input assembly + embedding gather ---------------------------------------------
// Inputs of a stream-sequence are [x_{n-1}, D_0 .. D_{L-2}]: the last committed token, then the
// drafts; the unconditional stream sees its own (masked) prompt but the same generated tokens.
// With `gain` (bf16 sessions) the kernel also prepares the first RMSNorm for the GEMM that follows:
// xg = bf16(h * gain) and the row's sum of squares (one "partial").
constexpr int EMBED_THREADS = 512;      // a row of the table is one latency-bound read: many loads in flight
// `lo_plane` > 0: xg is kept as two planes, xg[lo_plane + .] = T(x - T(x)).
template <class T>
__global__ void __launch_bounds__(EMBED_THREADS) embed_kernel(SeqState s, const T *__restrict__ emb, float *__restrict__ h, int d,
                             const T *__restrict__ gain, T *__restrict__ xg, float *__restrict__ ss_out, long long lo_plane)
{
    __shared__ float red[EMBED_THREADS / 32];
    pdl_trigger();
    if (s.skip && *s.skip) return;
    const int r = blockIdx.x, q = r / s.Mq, i = r % s.Mq;
    int id;
    if (s.ids) {
        id = s.ids[r];
    } else if (s.pos_override >= 0) {
        // prefill: the prompt as recorded on the device (the unconditional stream has its own prompt)
        const int b = q % s.B, stream = q / s.B, pos = s.pos_override + i;
        id = stream == 1 ? s.tokens_u[(size_t)b * s.prompt_cap + pos] : s.tokens[(size_t)b * s.token_stride + pos];
    } else {
        const int b = q % s.B, stream = q / s.B;
        if (i == 0) {
            const int last = s.n_known[b] - 1;
            id = (stream == 1 && last < s.prompt_len) ? s.tokens_u[(size_t)b * s.prompt_cap + last]
                                                      : s.tokens[(size_t)b * s.token_stride + last];
        } else {
            id = (i - 1 < s.L) ? s.drafts[(size_t)b * s.L + i - 1] : 0;
        }
    }
    id = min(max(id, 0), s.vocab_in - 1);
    const T *src = emb + (size_t)id * d;
    float *dst = h + (size_t)r * d;
    float ss = 0.f;
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        const float v = to_f<T>(src[j]);
        dst[j] = v;
        if (gain) {
            const float x = v * to_f<T>(gain[j]);
            const T hi = from_f<T>(x);
            xg[(size_t)r * d + j] = hi;
            if (lo_plane > 0) xg[lo_plane + (size_t)r * d + j] = from_f<T>(x - to_f<T>(hi));
            ss += v * v;
        }
    }
    if (gain) {
        ss = warp_sum_f(ss);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;                       // fixed order: the sum does not depend on scheduling
#pragma unroll
            for (int w = 0; w < EMBED_THREADS / 32; ++w) t += red[w];
            ss_out[r] = t;
        }
    }
}

// ---- RoPE on Q and K, KV-cache write --------------------------------------------------------
// Pairs (i, i + dh/2), angle = pos * base^(-2i/dh); K is cached after rotation. The window's K/V
// land in cache slots [kv_len, kv_len + Mq): committing a prefix is then only a counter update.
// (bf16 models whose head_dim or page size the tensor-core attention does not take: projections in fp32 from the GEMM)
template <class T>
__global__ void rope_kv_kernel(SeqState s, float *__restrict__ qkv, KvLayout kv, const float2 *__restrict__ rope,
                               int n_heads)
{
    pdl_trigger();
    const int r = blockIdx.x, q = r / s.Mq, i = r % s.Mq;
    const int dh = kv.head_dim, half = dh >> 1, Hkv = kv.n_kv_heads;
    const int pos = base_position(s, q) + i;
    const bool in_range = pos >= 0 && pos < kv.max_seq;
    const int pc = min(max(pos, 0), kv.max_seq - 1);
    const float2 *cs = rope + (size_t)pc * half;
    float *row = qkv + (size_t)r * (n_heads + 2 * Hkv) * dh;
    // Q heads: rotate in place
    for (int e = threadIdx.x; e < n_heads * half; e += blockDim.x) {
        const int hh = e / half, j = e % half;
        float *v = row + (size_t)hh * dh;
        const float a = v[j], b = v[j + half];
        const float2 t = cs[j];
        v[j] = a * t.x - b * t.y;
        v[j + half] = b * t.x + a * t.y;
    }
    if (!in_range) return;
    // K heads: rotate into the cache; V heads: copy into the cache
    const float *krow = row + (size_t)n_heads * dh, *vrow = krow + (size_t)Hkv * dh;
    for (int e = threadIdx.x; e < Hkv * half; e += blockDim.x) {
        const int hh = e / half, j = e % half;
        const float a = krow[hh * dh + j], b = krow[hh * dh + j + half];
        const float2 t = cs[j];
        const size_t o = kv_offset<T>(kv, q, pos, hh);
        ((T *)kv.k_pool)[o + j] = from_f<T>(a * t.x - b * t.y);
        ((T *)kv.k_pool)[o + j + half] = from_f<T>(b * t.x + a * t.y);
        ((T *)kv.v_pool)[o + j] = from_f<T>(vrow[hh * dh + j]);
        ((T *)kv.v_pool)[o + j + half] = from_f<T>(vrow[hh * dh + j + half]);
    }
}

__global__ void rope_table_kernel(float2 *table, int max_seq, int half, int dh, double base)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)max_seq * half) return;
    const int pos = (int)(i / half), j = (int)(i % half);
    const double theta = pow(base, -2.0 * (double)j / (double)dh);
    double sn, cs;
    sincos((double)pos * theta, &sn, &cs);
    table[i] = make_float2((float)cs, (float)sn);
}

template <class T>
int forward_impl(scd_session *s, const ForwardArgs &a, cudaStream_t st)
{
    scd_model *m = s->model;
    const scd_model_config_t &c = m->cfg;
    const int d = c.d_model, H = c.n_heads, Hkv = c.n_kv_heads, dh = c.head_dim, F = c.d_ffn;
    const int dq = H * dh, dkv = Hkv * dh, dqkv = dq + 2 * dkv;
    const int rows = s->Q * a.Mq;
    const bool tc = std::is_same<T, __nv_bfloat16>::value && m->gemm_plan != nullptr;

    SeqState ss;
    ss.ids = a.ids; ss.n_known = s->n_known; ss.tokens = s->tokens; ss.tokens_u = s->tokens_u;
    ss.drafts = s->drafts; ss.token_stride = c.max_seq; ss.prompt_cap = c.max_seq;
    ss.prompt_len = s->prompt_len; ss.L = s->L; ss.B = s->B; ss.Mq = a.Mq;
    ss.pos_override = a.pos_override; ss.vocab_in = c.vocab_in; ss.skip = a.skip;

    StepProfiler *prof = a.prof;
    int rc = SCD_OK;
#define MARK(c) do { if (prof) prof->mark(c); } while (0)
#define TRY(expr) do { rc = (expr); if (rc != SCD_OK) return rc; } while (0)
    MARK(PROF_EMBED);
    // tensor-core path: the norms are folded into the GEMMs (see gemm.cuh); `parts` = partial sums
    // of squares the producer of xn left per row
    int parts = 1;
    embed_kernel<T><<<rows, EMBED_THREADS, 0, st>>>(ss, (const T *)m->tok_emb, s->h, d, tc ? (const T *)m->attn_norm[0] : nullptr,
                                                    (T *)s->xn, s->ss, tc ? (long long)s->rows_cap * d : 0ll);
    count_launches(1);

    KvLayout kv;
    kv.page_table = s->page_table; kv.pages_per_seq = s->pages_per_seq;
    kv.page_tokens = c.kv_page_tokens; kv.page_shift = __builtin_ctz((unsigned)c.kv_page_tokens);
    kv.n_kv_heads = Hkv; kv.head_dim = dh; kv.max_seq = c.max_seq;
    const float scale = 1.0f / sqrtf((float)dh);

    // fp32 models: x [rows][K] times W [N][K], with what goes in front and behind in the same launch
    LinearF32 lin;
    lin.eps = c.rms_eps; lin.rows = rows; lin.skip = a.skip; lin.seq = ss; lin.rope = m->rope_table; lin.n_heads = H;
    auto linear = [&](int epi, const float *x, const void *gain, const void *w0, const void *w1, const void *w2, int N, int K, float *y,
                      int ldy) -> int {
        lin.x = x; lin.gain = (const float *)gain; lin.w[0] = (const float *)w0; lin.w[1] = (const float *)w1; lin.w[2] = (const float *)w2;
        lin.N = N; lin.K = K; lin.y = y; lin.ldy = ldy; lin.kv = kv;
        return linear_f32(epi, lin, st);
    };

    for (int l = 0; l < c.n_layers; ++l) {
        kv.k_pool = (T *)s->kv_pool + (size_t)l * s->kv_layer_stride;
        kv.v_pool = (T *)kv.k_pool + s->kv_kind_stride;
        MARK(PROF_GEMM_QKV);
        if (tc) TRY(gemm_tc_qkv(s, l, rows, parts, st));
        else TRY(linear(F32_QKV, s->h, m->attn_norm[l], m->wq[l], m->wk[l], m->wv[l], dqkv, d, (float *)s->qkv, dqkv));
        if (tc && attention_tc_supported(s, a.Mq)) {
            MARK(PROF_ATTENTION);
            TRY(attention_tc(s, l, a.Mq, a.pos_override, st));
        } else {
            if (tc) {
                MARK(PROF_ROPE_KV);
                rope_kv_kernel<T><<<rows, 128, 0, st>>>(ss, (float *)s->qkv, kv, m->rope_table, H);
                count_launches(1);
            }
            MARK(PROF_ATTENTION);
            // (bf16 models: the output in two planes for the next GEMM)
            TRY(attention_simt<T>(ss, (const float *)s->qkv, kv, (T *)s->att, s->Q, H, scale, tc ? (long long)s->rows_cap * dq : 0ll, st));
        }
        MARK(PROF_GEMM_O);
        if (tc) TRY(gemm_tc_residual(s, l, /*which=*/0, rows, m->ffn_norm[l], &parts, st));
        else TRY(linear(F32_ADD, (const float *)s->att, nullptr, m->wo[l], nullptr, nullptr, d, dq, s->h, d));
        MARK(PROF_GEMM_GATE_UP);
        if (tc) TRY(gemm_tc_gate_up(s, l, rows, parts, st));
        else TRY(linear(F32_SWIGLU, s->h, m->ffn_norm[l], m->w_gate[l], m->w_up[l], nullptr, F, d, (float *)s->act, F));
        MARK(PROF_GEMM_DOWN);
        if (tc) TRY(gemm_tc_residual(s, l, /*which=*/1, rows, l + 1 < c.n_layers ? m->attn_norm[l + 1] : m->final_norm, &parts, st));
        else TRY(linear(F32_ADD, (const float *)s->act, nullptr, m->w_down[l], nullptr, nullptr, d, F, s->h, d));
    }
    MARK(PROF_OTHER);
    if (a.hidden)
        SCD_CUDA_TRY(cudaMemcpyAsync(a.hidden, s->h, (size_t)rows * d * sizeof(float),
                                     cudaMemcpyDeviceToDevice, st));
    if (a.want_logits) {
        MARK(PROF_GEMM_LM_HEAD);
        if (tc) {
            const bool all = a.lm_hi <= 0;
            TRY(gemm_tc_lm_head(s, rows, a.logits, all ? 0 : a.lm_lo, all ? c.vocab_out : a.lm_hi, all ? -1 : a.lm_eol, parts, st));
        } else {
            TRY(linear(F32_STORE, s->h, m->final_norm, m->lm_head, nullptr, nullptr, c.vocab_out, d, a.logits, c.vocab_out));
        }
    }
    MARK(PROF_OTHER);
#undef TRY
#undef MARK
    SCD_CUDA_TRY(cudaGetLastError());
    return SCD_OK;
}

}  // namespace

// ---- per-kernel event marks --------------------------------------------------------------------
namespace { thread_local unsigned long long *g_stamp_slot = nullptr; }

unsigned long long *take_stamp_slot()
{
    unsigned long long *p = g_stamp_slot;
    g_stamp_slot = nullptr;
    return p;
}

void StepProfiler::mark(int c)
{
    if (failed) return;
    if (stamps) {
        if (used == cls.size()) cls.push_back(PROF_OTHER);
        cls[used] = c;
        g_stamp_slot = used < stamp_launches ? stamps + used * 2 * STAMP_CTAS : nullptr;
        ++used;
        return;
    }
    if (used == events.size()) {
        cudaEvent_t e;
        if (cudaEventCreate(&e) != cudaSuccess) { failed = true; return; }
        events.push_back(e);
        cls.push_back(PROF_OTHER);
    }
    cls[used] = c;
    if (cudaEventRecord(events[used], st) != cudaSuccess) { failed = true; return; }
    ++used;
}

int StepProfiler::finish(float *ms_by_class, int *launches_by_class)
{
    if (stamps) {
        g_stamp_slot = nullptr;
        SCD_CUDA_TRY(cudaStreamSynchronize(st));
        const size_t n = std::min(used, stamp_launches);
        std::vector<unsigned long long> h(n * 2 * STAMP_CTAS);
        SCD_CUDA_TRY(cudaMemcpy(h.data(), stamps, h.size() * sizeof(unsigned long long), cudaMemcpyDeviceToHost));
        unsigned long long prev_end = 0;
        for (size_t i = 0; i < n; ++i) {
            unsigned long long first = ~0ull, last = 0;
            for (int c = 0; c < STAMP_CTAS; ++c) {
                const unsigned long long a = h[(i * 2) * STAMP_CTAS + c], b = h[(i * 2 + 1) * STAMP_CTAS + c];
                if (a) first = std::min(first, a);
                last = std::max(last, b);
            }
            if (last == 0) continue;                   // a kernel that leaves no stamps: charged to the next one
            if (prev_end == 0) prev_end = first;       // the first stamped kernel starts the clock
            if (last > prev_end) ms_by_class[cls[i]] += (float)((double)(last - prev_end) * 1e-6);
            launches_by_class[cls[i]] += 1;
            prev_end = std::max(prev_end, last);
        }
        used = 0;
        return SCD_OK;
    }
    mark(PROF_OTHER);
    SCD_REQUIRE(!failed, SCD_ERR_CUDA, "step profiler: event creation or record failed");
    SCD_CUDA_TRY(cudaEventSynchronize(events[used - 1]));
    for (size_t i = 0; i + 1 < used; ++i) {
        float ms = 0.f;
        SCD_CUDA_TRY(cudaEventElapsedTime(&ms, events[i], events[i + 1]));
        ms_by_class[cls[i]] += ms;
        launches_by_class[cls[i]] += 1;
    }
    used = 0;
    return SCD_OK;
}

StepProfiler::~StepProfiler()
{
    for (cudaEvent_t e : events) cudaEventDestroy(e);
}

int run_forward(scd_session *s, const ForwardArgs &a, cudaStream_t st)
{
    s->skip_now = a.skip;
    if (s->model->cfg.dtype == SCD_F32) return forward_impl<float>(s, a, st);
    return forward_impl<__nv_bfloat16>(s, a, st);
}

int build_rope_table(scd_model *m)
{
    const int half = m->cfg.head_dim / 2;
    const long long n = (long long)m->cfg.max_seq * half;
    SCD_CUDA_TRY(cudaMalloc(&m->rope_table, (size_t)n * sizeof(float2)));
    rope_table_kernel<<<(unsigned)((n + 255) / 256), 256>>>(m->rope_table, m->cfg.max_seq, half,
                                                            m->cfg.head_dim, (double)m->cfg.rope_base);
    SCD_CUDA_TRY(cudaGetLastError());
    SCD_CUDA_TRY(cudaDeviceSynchronize());
    return SCD_OK;
}

}  // namespace scd
