// Fused verify-and-redraft kernel for rows of more than 131072 ids (shorter ones: verify_rows.cu): logits -> CFG
// mix -> temperature -> top-k -> integer weights -> accept / reject -> residual sample -> redraft.
//
// One CTA per window row (Algorithm 6 evaluates ALL rows, with no break; Algorithm 1 per row). The kernel behind
// finds the first rejection (the Accept step of Algorithm 6), commits the accepted prefix and builds the next
// window: a row that survives keeps its MRS output as draft and its target distribution as draft distribution,
// which is the maximal coupling of Algorithm 3 at no extra cost (Sec. 4.3).
//
// Redraft rules besides the maximal coupling: the independent redraw of Algorithm 2 (SJD), its
// alpha-mixture with the coupling (Algorithm 5), and the Gumbel-sharing coupling (Algorithms 4
// and 7) as an integer exponential race with noise keyed by position and id only. Top-p after
// top-k as a threshold on the integer weights.
//
// Data flow of a row: logits -> x, in the row's cells (its row of xbuf, global memory) -> radix selection of the top-k
// threshold -> integer weights W, in the same cells; every later pass (sum, accept test, residual search, race) reads
// integers. A session keeps W there as the next iteration's draft distribution.
//
// Exactness: a distribution is the integer vector W_v = trunc(scd_exp(x_v - max x) * 2^30) over
// the ids whose post-processed logit x_v reaches the top-k threshold; every decision is an
// inequality between exact 128-bit integer expressions, so the result does not depend on the
// order in which threads sum.
#include "verify.cuh"

namespace scd {

namespace {

constexpr int VT = 1024;       // threads per CTA
constexpr int NW = VT / 32;    // warps per CTA
constexpr unsigned FULL = 0xffffffffu;

struct Smem {
    float red_f[NW];
    unsigned long long red_lo[NW], red_hi[NW];
    unsigned long long base_lo[NW], base_hi[NW], tot_lo, tot_hi;   // block_search: prefix of the warp sums
    unsigned int hist[256];
    unsigned long long mass[256];
    unsigned int sel_bin, sel_k;
    int result;
    int flag;
};

// Post-processed logit of id v of a stored row; raw draft logits still need the temperature.
struct XRow {
    const float *row;
    float T;
    bool div;
    __device__ __forceinline__ float operator()(int v) const
    {
        const float x = row[v];
        return div ? __fdiv_rn(x, T) : x;
    }
};

__device__ __forceinline__ float block_max(float v, Smem &sm)
{
    v = warp_max(v);
    if ((threadIdx.x & 31) == 0) sm.red_f[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = sm.red_f[0];
#pragma unroll
    for (int i = 1; i < NW; ++i) r = fmaxf(r, sm.red_f[i]);
    __syncthreads();
    return r;
}

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, Smem &sm)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if ((threadIdx.x & 31) == 0) sm.red_lo[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long r = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) r += sm.red_lo[i];
    __syncthreads();
    return r;
}

// After a histogram pass: the bin (from the top) in which the kk-th largest element falls, and its
// rank inside that bin. Warp 0 scans the 256 counters; the caller synchronises afterwards.
__device__ __forceinline__ void select_bin(Smem &sm, unsigned kk)
{
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 32) {
        unsigned c[8], s = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { c[j] = sm.hist[8 * lane + j]; s += c[j]; }
        unsigned incl = s;                       // suffix sum over lanes >= lane
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_down_sync(FULL, incl, o);
            if (lane + o < 32) incl += t;
        }
        const unsigned above = incl - s;
        if (above < kk && kk <= above + s) {
            unsigned acc = above;
#pragma unroll
            for (int j = 7; j >= 0; --j) {
                if (acc + c[j] >= kk) { sm.sel_bin = 8u * lane + j; sm.sel_k = kk - acc; break; }
                acc += c[j];
            }
        }
    }
}

// k-th largest post-processed logit of ids [lo, hi) by radix selection on order-preserving
// keys, 8 bits per pass. Exact; ties are resolved by the caller's ">= tau" test.
__device__ float kth_largest(const XRow &x, int lo, int hi, int k, Smem &sm)
{
    const int tid = threadIdx.x, lane = tid & 31;
    unsigned prefix = 0, mask = 0;
    unsigned kk = (unsigned)k;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = tid; i < 256; i += VT) sm.hist[i] = 0;
        __syncthreads();
        for (int base = lo; base < hi; base += 4 * VT) {     // (uniform trip count: warp-wide votes inside)
            float xv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) xv[j] = base + j * VT + tid < hi ? x(base + j * VT + tid) : 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int v = base + j * VT + tid;
                unsigned key = 0;
                bool match = false;
                if (v < hi) {
                    key = float_key(xv[j]);
                    match = (key & mask) == prefix;
                }
                const unsigned bin = (key >> shift) & 255u;
                if (shift == 24) {
                    // sign and high exponent bits: a handful of distinct bins per warp, so count the
                    // lanes of each bin once (match.any costs one round per distinct value)
                    const unsigned active = __ballot_sync(FULL, match);
                    if (match) {
                        const unsigned peers = __match_any_sync(active, bin);
                        if (lane == __ffs(peers) - 1) atomicAdd(&sm.hist[bin], (unsigned)__popc(peers));
                    }
                } else if (match) {
                    atomicAdd(&sm.hist[bin], 1u);          // lower bytes are spread out: few collisions
                }
            }
        }
        __syncthreads();
        select_bin(sm, kk);
        __syncthreads();
        prefix |= sm.sel_bin << shift;
        mask |= 0xFFu << shift;
        kk = sm.sel_k;
    }
    __syncthreads();
    return key_float(prefix);
}

// Nucleus (top-p) threshold on the integer weights of ids [lo, hi): the largest weight value theta
// for which the ids with W_v >= theta hold at least P24 / 2^24 of the mass Z (integer test
// mass * 2^24 >= P24 * Z). Radix descent over the weight value, 8 bits per pass, with per-bin MASS
// instead of counts. Returns theta; *kept = mass of {W_v >= theta}.
template <class F>
__device__ unsigned nucleus_threshold(const F &weight, int lo, int hi, unsigned long long Z, unsigned P24,
                                      Smem &sm, unsigned long long *kept)
{
    const int tid = threadIdx.x;
    unsigned prefix = 0, mask = 0;
    unsigned long long above = 0;                 // mass of the weights above the current prefix range
    const u128 need = (u128)P24 * Z;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = tid; i < 256; i += VT) sm.mass[i] = 0ull;
        __syncthreads();
        unsigned long long mine0 = 0;             // bin 0 of the top byte holds almost every id: keep it in a register
        for (int v = lo + tid; v < hi; v += VT) {
            const unsigned w = weight(v);
            if (w == 0u || (w & mask) != prefix) continue;
            const unsigned bin = (w >> shift) & 255u;
            if (shift == 24 && bin == 0u) mine0 += w;
            else atomicAdd(&sm.mass[bin], (unsigned long long)w);
        }
        if (shift == 24) {
            const unsigned long long all0 = block_sum_u64(mine0, sm);
            if (tid == 0) sm.mass[0] = all0;
        }
        __syncthreads();
        if (tid == 0) {
            unsigned long long cum = above;
            int sel = 0;
            for (int bin = 255; bin >= 0; --bin) {
                const unsigned long long mb = sm.mass[bin];
                if (mb == 0ull) continue;
                sel = bin;
                if (((u128)(cum + mb) << 24) >= need) break;
                cum += mb;
            }
            sm.sel_bin = (unsigned)sel;
            sm.red_lo[0] = cum;
            sm.red_hi[0] = cum + sm.mass[sel];
        }
        __syncthreads();
        prefix |= sm.sel_bin << shift;
        mask |= 0xFFu << shift;
        above = sm.red_lo[0];
        *kept = sm.red_hi[0];
        __syncthreads();
    }
    return prefix;
}

// Inverse-CDF search: smallest id v in [lo, hi) with sum_{v' <= v} f(v') > (U * total) >> 24,
// ids in increasing order. Warps own contiguous id ranges; the warp whose range holds the
// target walks it 32 ids at a time. Returns -1 when the total is zero.
template <class F>
__device__ int block_search(const F &f, int lo, int hi, unsigned U, Smem &sm)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = hi - lo;
    const int chunk = (((n + NW - 1) / NW) + 31) & ~31;
    const int w_lo = min(hi, lo + warp * chunk);
    const int w_hi = min(hi, w_lo + chunk);
    Limbs s = {0ull, 0ull};
#pragma unroll 4
    for (int v = w_lo + lane; v < w_hi; v += 32) s.add(f(v));
    s = warp_sum(s);
    if (lane == 0) { sm.red_lo[warp] = s.lo; sm.red_hi[warp] = s.hi; }
    if (tid == 0) sm.result = -1;
    __syncthreads();
    if (warp == 0) {
        // exclusive prefix of the warp sums, in warp (= id) order, and their total
        const Limbs t = {sm.red_lo[lane], sm.red_hi[lane]};
        const Limbs inc = warp_scan_inclusive(t, lane);
        sm.base_lo[lane] = inc.lo - t.lo;
        sm.base_hi[lane] = inc.hi - t.hi;
        if (lane == 31) { sm.tot_lo = inc.lo; sm.tot_hi = inc.hi; }
    }
    __syncthreads();
    const u128 base = ((u128)sm.base_hi[warp] << 40) + sm.base_lo[warp];
    const u128 total = ((u128)sm.tot_hi << 40) + sm.tot_lo;
    const u128 mine = s.value();
    const u128 target = ((u128)U * total) >> 24;
    if (total != 0 && base <= target && target < base + mine) {
        u128 run = base;
        for (int i = w_lo; i < w_hi; i += 32) {
            const int v = i + lane;
            Limbs r = {0ull, 0ull};
            if (v < w_hi) r.add(f(v));
            const Limbs inc = warp_scan_inclusive(r, lane);
            const unsigned hit = __ballot_sync(FULL, run + inc.value() > target);
            if (hit) {
                if (lane == 0) sm.result = i + __ffs(hit) - 1;
                break;
            }
            Limbs tot;
            tot.lo = __shfl_sync(FULL, inc.lo, 31);
            tot.hi = __shfl_sync(FULL, inc.hi, 31);
            run += tot.value();
        }
    }
    __syncthreads();
    const int res = sm.result;
    __syncthreads();
    return res;
}

// argmin over ids [lo, hi) with weight(v) > 0; the noise of id v at a position is the same in
// every iteration (the coupling shares it between the draft and the target distribution).
template <class F>
__device__ int block_race(const F &weight, int lo, int hi, const VerifyParams &p, int b, long long pos, Smem &sm)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Racer best = {0ull, 0u, -1};
    for (int v = lo + (int)threadIdx.x; v < hi; v += VT) {
        const unsigned W = weight(v);
        if (W == 0u) continue;
        const Racer c = {neglog2_q40(noise_u24(p.seed, NOISE_GUMBEL, (unsigned)b, pos, 0u, (unsigned)v)), W, v};
        if (race_before(c, best)) best = c;
    }
    best = warp_racer(best);
    if (lane == 0) { sm.red_lo[warp] = best.T; sm.red_hi[warp] = ((unsigned long long)best.W << 32) | (unsigned)best.v; }
    __syncthreads();
    Racer r = {0ull, 0u, -1};
    for (int i = 0; i < NW; ++i) {
        const Racer c = {sm.red_lo[i], (unsigned)(sm.red_hi[i] >> 32), (int)(unsigned)sm.red_hi[i]};
        if (race_before(c, r)) r = c;
    }
    __syncthreads();
    return r.v;
}

// argmin under equal weights
__device__ int block_fresh_race(int lo, int hi, const VerifyParams &p, int b, long long pos, Smem &sm)
{
    unsigned long long best = 0;
    for (int v = lo + (int)threadIdx.x; v < hi; v += VT) best = max(best, fresh_key(p, b, pos, v));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(FULL, best, o));
    if ((threadIdx.x & 31) == 0) sm.red_lo[threadIdx.x >> 5] = best;
    __syncthreads();
    best = sm.red_lo[0];
#pragma unroll
    for (int i = 1; i < NW; ++i) best = max(best, sm.red_lo[i]);
    __syncthreads();
    return fresh_key_id(best);
}

__global__ void __launch_bounds__(VT, 1) verify_kernel(const VerifyParams p)
{
    __shared__ Smem sm;
    const int tid = threadIdx.x;
    const int k = blockIdx.x, b = blockIdx.y;
    const WindowState w = load_state(p, b);
    const int L = p.L, V = p.V;

    if (k < w.Lw) {
        const long long pos = w.pos0 + k;
        int lo, hi;
        allowed_range(p, pos, lo, hi);
        const size_t row = (size_t)b * L + k;

        // ---- target distribution p = post-process(logits) ------------------------------------
        // The row's cells first hold the post-processed logits x and then, in place, the integer weights W: the exponential
        // is evaluated once per id and every later pass reads integers. In a session they are the next iteration's draft
        // distribution.
        float *const xp = p.xbuf[w.parity] + row * V;
        unsigned *const wp = (unsigned *)xp;
        const float *c = p.p_logits + row * V;
        const float *u = p.S == 2 ? p.p_logits + ((size_t)(p.B + b) * L + k) * V : nullptr;
        const bool mix = (p.S == 2);
        const bool div = (p.temperature != 1.0f);
        const bool use_topk = p.top_k > 0 && p.top_k < hi - lo;
        float m_p, tau_p;
        unsigned long long Zp;
        {
            // loads go out four at a time
            float mx = -INFINITY;
            for (int v0 = lo + tid; v0 < hi; v0 += 4 * VT) {
                float xc[4], xu[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int v = v0 + j * VT;
                    xc[j] = v < hi ? c[v] : 0.f;
                    xu[j] = (mix && v < hi) ? u[v] : 0.f;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int v = v0 + j * VT;
                    if (v < hi) {
                        float x = xc[j];
                        if (mix) x = __fsub_rn(__fmul_rn(p.one_plus_lam, x), __fmul_rn(p.lam, xu[j]));
                        if (div) x = __fdiv_rn(x, p.temperature);
                        xp[v] = x;
                        mx = fmaxf(mx, x);
                    }
                }
            }
            m_p = block_max(mx, sm);       // barrier inside: the row is visible to the CTA
            tau_p = use_topk ? kth_largest(XRow{xp, 1.0f, false}, lo, hi, p.top_k, sm) : -INFINITY;
            unsigned long long zp = 0;
            for (int v0 = lo + tid; v0 < hi; v0 += 4 * VT) {     // x -> W, each thread on its own cells
                float xv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) xv[j] = v0 + j * VT < hi ? xp[v0 + j * VT] : -INFINITY;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int v = v0 + j * VT;
                    if (v < hi) {
                        const unsigned wv = weight_of(xv[j], m_p, tau_p);
                        wp[v] = wv;
                        zp += wv;
                    }
                }
            }
            Zp = block_sum_u64(zp, sm);                          // (barriers inside: the weights are visible)
        }
        unsigned theta_p = 0u;
        if (p.top_p24) {
            auto fw = [&](int v) -> unsigned { return wp[v]; };
            unsigned long long kept;
            theta_p = nucleus_threshold(fw, lo, hi, Zp, p.top_p24, sm, &kept);
            Zp = kept;
            for (int v = lo + tid; v < hi; v += VT)
                if (wp[v] < theta_p) wp[v] = 0u;
            __syncthreads();
        }
        if (tid == 0) {
            RowStats st; st.m = m_p; st.tau = tau_p; st.Z = Zp; st.theta = theta_p; st.pad_ = 0u;
            p.stats[w.parity][row] = st;
        }
        auto WP = [&](int v) -> unsigned { return wp[v]; };

        // ---- draft distribution q: the previous iteration's p of the same position -----------
        // session: its integer weights, as stored by that iteration; stand-alone: raw logits that
        // go through the same steps here (recomputed per visit); fresh rows: uniform weights 1 on the allowed ids.
        const int qk = k + w.shift;
        const bool fresh = !(qk < w.prev_lw);
        unsigned long long Zq = (unsigned long long)(hi - lo);
        const unsigned *q_weights = nullptr;                  // the stored weights
        XRow XQ = {nullptr, p.temperature, false};            // the raw logits
        float m_q = 0.f, tau_q = -INFINITY;
        unsigned theta_q = 0u;
        if (!fresh) {
            const size_t qrow = (size_t)b * L + qk;
            if (p.q_is_raw) {
                XQ.row = p.xbuf[w.parity ^ 1] + qrow * V;
                XQ.div = div;
                float mq = -INFINITY;
                for (int v = lo + tid; v < hi; v += VT) mq = fmaxf(mq, XQ(v));
                m_q = block_max(mq, sm);
                tau_q = use_topk ? kth_largest(XQ, lo, hi, p.top_k, sm) : -INFINITY;
                unsigned long long zq = 0;
                for (int v = lo + tid; v < hi; v += VT) zq += weight_of(XQ(v), m_q, tau_q);
                Zq = block_sum_u64(zq, sm);
                if (p.top_p24) {
                    auto fq = [&](int v) -> unsigned { return weight_of(XQ(v), m_q, tau_q); };
                    unsigned long long kept;
                    theta_q = nucleus_threshold(fq, lo, hi, Zq, p.top_p24, sm, &kept);
                    Zq = kept;
                }
            } else {
                Zq = p.stats[w.parity ^ 1][qrow].Z;
                q_weights = (const unsigned *)(p.xbuf[w.parity ^ 1] + qrow * V);
            }
        }
        auto WQ = [&](int v) -> unsigned {
            if (fresh) return 1u;
            if (q_weights) return q_weights[v];
            return weight_of(XQ(v), m_q, tau_q, theta_q);
        };

        // ---- Algorithm 1 on (p, q, X) ----------------------------------------------------------
        const int X = p.draft_in[row];
        int Y = X, Yi = X, Yf = X;
        int accept = 1;
        if (p.mode == SCD_MODE_AR) {
            // vanilla AR: x ~ p by inverse CDF (Sec. 2.1)
            const unsigned U = noise_u24(p.seed, NOISE_INDEP, (unsigned)b, pos, 0u, 0);
            auto fw = [&](int v) -> u128 { return (u128)WP(v); };
            Y = block_search(fw, lo, hi, U, sm);
            if (Y < 0) Y = lo;
        } else {
            if (tid == 0) {
                unsigned WpX = 0, WqX = 0;
                if (X >= lo && X < hi) {
                    WpX = WP(X);
                    WqX = WQ(X);
                }
                const unsigned Ua = noise_u24(p.seed, NOISE_ACCEPT, (unsigned)b, pos, w.t, 0);
                // u <= min(1, p(X)/q(X)) with u = (Ua+1)/2^24  <=>  (Ua+1) Wq[X] Zp <= Wp[X] Zq 2^24
                // (a draft without mass under p - possible only when X was not drawn from q - is rejected)
                const u128 lhs = (u128)(Ua + 1u) * WqX * Zp;
                const u128 rhs = ((u128)WpX * Zq) << 24;
                sm.flag = (WpX != 0u && lhs <= rhs) ? 1 : 0;
            }
            __syncthreads();
            accept = sm.flag;
            __syncthreads();
            if (!accept) {
                // Y ~ norm(max(0, p - q)): R_v = max(0, Wp_v Zq - Wq_v Zp)
                const unsigned Ur = noise_u24(p.seed, NOISE_RESIDUAL, (unsigned)b, pos, w.t, 0);
                auto fr = [&](int v) -> u128 {
                    const u128 a = mul_32x64(WP(v), Zq);
                    const u128 bq = mul_32x64(WQ(v), Zp);
                    return a > bq ? a - bq : (u128)0;
                };
                Y = block_search(fr, lo, hi, Ur, sm);
                if (Y < 0) Y = X;
            }
            bool indep = p.mode == SCD_MODE_SJD;
            Yi = Y;
            if (p.mode == SCD_MODE_ALPHA) {
                // Algorithm 5: keep the coupled redraft with probability alpha, b = (Ub + 1) / 2^24
                const unsigned Ub = noise_u24(p.seed, NOISE_ALPHA, (unsigned)b, pos, w.t, 0);
                indep = !((double)(Ub + 1u) <= (double)p.alpha * 16777216.0);
            }
            if (p.mode == SCD_MODE_SCD_GS) {
                // Algorithm 7: beyond the committed prefix the next draft is the Gumbel-max sample
                // of p under this position's shared noise ...
                auto fw = [&](int v) -> unsigned { return WP(v); };
                Yi = block_race(fw, lo, hi, p, b, pos, sm);
                if (Yi < 0) Yi = lo;
                // ... and the row that may enter the window at position pos0 + L + k starts from the
                // same race under the uniform draft distribution of its allowed ids
                const long long posf = w.pos0 + L + k;
                int flo, fhi;
                allowed_range(p, posf, flo, fhi);
                Yf = block_fresh_race(flo, fhi, p, b, posf, sm);
            }
            if (indep) {
                // Algorithm 2 (its redraw step): the next draft is an independent draw from p
                const unsigned Ui = noise_u24(p.seed, NOISE_INDEP, (unsigned)b, pos, w.t, 0);
                auto fw = [&](int v) -> u128 { return (u128)WP(v); };
                Yi = block_search(fw, lo, hi, Ui, sm);
                if (Yi < 0) Yi = lo;
            }
        }
        if (tid == 0) {
            p.accept_flags[row] = (unsigned char)accept;
            p.row_y[row] = Y;
            p.row_y_indep[row] = Yi;
            if (p.mode == SCD_MODE_SCD_GS) p.row_y_indep[(size_t)p.B * L + row] = Yf;
        }
    }
}

// Window initialisation after prefill: every row fresh. Gumbel: a CTA per row.
__global__ void __launch_bounds__(VT) init_window_kernel(const VerifyParams p)
{
    __shared__ Smem sm;
    const int b = blockIdx.y;
    const long long pos0 = p.n_known[b];
    if (p.mode == SCD_MODE_SCD_GS) {
        const int k = blockIdx.x;
        int lo, hi;
        allowed_range(p, pos0 + k, lo, hi);
        const int d = block_fresh_race(lo, hi, p, b, pos0 + k, sm);
        if (threadIdx.x == 0) p.draft_out[(size_t)b * p.L + k] = d;
    } else {
        for (int k = threadIdx.x; k < p.L; k += blockDim.x)
            p.draft_out[(size_t)b * p.L + k] = fresh_draft(p, b, pos0 + k, 0u);
    }
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        p.iter[b] = 0u;
        p.shift[b] = 0;
        p.prev_lw[b] = 0;
        p.n_commit[b] = 0;
    }
}

}  // namespace

int launch_verify(const VerifyParams &p, cudaStream_t stream)
{
    count_launches(2);
    // a cluster per row; this kernel keeps the rows that are too long for one
    if (verify_rows_supported(p)) {
        const int rc = launch_verify_rows(p, stream);
        return rc == SCD_OK ? launch_commit(p, stream) : rc;
    }
    verify_kernel<<<dim3((unsigned)p.L, (unsigned)p.B), VT, 0, stream>>>(p);
    SCD_CUDA_TRY(cudaGetLastError());
    return launch_commit(p, stream);
}

int launch_init_window(const VerifyParams &p, cudaStream_t stream)
{
    init_window_kernel<<<dim3(p.mode == SCD_MODE_SCD_GS ? p.L : 1, p.B), VT, 0, stream>>>(p);
    SCD_CUDA_TRY(cudaGetLastError());
    return SCD_OK;
}

}  // namespace scd
