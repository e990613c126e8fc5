// Fused verify-and-redraft, one thread-block cluster of C CTAs per window row (Algorithm 6 evaluates all rows,
// Algorithm 1 per row). The row's ids are dealt to CTAs and warps in contiguous ranges.
//
// By bytes a row is nothing; a kernel over a few rows is bound by its chain of row-wide exchanges, one over many
// rows by issue slots. So the passes over ALL ids do as little as possible per id, and everything dear - the
// exponential, 128-bit products, noise - runs on the ids that survive the truncation (2000 of 16384 with the image
// settings), packed densely:
//   1. x = post-processed logit (guidance mix, temperature), of a sample of 1024 ids per CTA first: a bound that some
//      more ids than top_k should exceed
//   2. one sweep over the ids: row maximum m, and the ids at or above the bound go to a list per warp, in id order,
//      with their x                                                                                   -> exchange
//   3. on the lists: histogram over NB equal steps of m - x (live ids: x >= m - 22, only they have a weight
//      W = trunc(scd_exp(x - m) 2^30)); the step that holds the k-th largest. If the bound of any CTA lies in that
//      step or above it, the lists are built once more without one                                    -> exchange
//   4. mass above the step; the candidates OF the step, over the cluster, and by counting the exact k-th largest
//                                                                                                     -> exchange
//      Nucleus without top-k: maximum and weights take a sweep each; the bound is one on W, from a sample as well, the
//      mass below it is only summed. The step (logarithmic, of W) in which the mass from the top reaches top_p of the
//      row is divided again, NB ways, until it is one value of W or holds few ids, which are selected by counting.
//   5. accept test in 128-bit integers; on rejection the residual masses max(0, Wp_v Zq - Wq_v Zp)   -> exchange
//      and the inverse-CDF walk in the one warp that holds the target
// Rows of up to 256 ids per warp stay in registers (REG): there the histogram counts every id and the lists come after
// it, without a sample (28.9 us against 30.7 for 32 rows of 16384 ids). Longer ones are read again from L2 where a sweep
// repeats (three sweeps, one for the histogram: 63.7 us against 53.8 for 256 rows of 16384 ids).
// A warp whose list would overflow (a row that hardly is truncated) works on its whole range instead, reading x
// again (the nucleus leaves its weights in the list's place): entry e is then simply its e-th id. commit_kernel, one CTA per sequence behind this grid, does the
// only serial part: first rejection, commit, next window.
//
// us per scd_verify call on a B200, before (an exponential per id, four byte-wise passes over the cluster for the nucleus,
// tickets for the commit, the race on one CTA per row) and now: 1 x 32 rows of 16384 ids, top-k 2000: 32.8, 21.9;
// 8 x 32 with guidance: 107, 45.0; 64 rows of 64000 ids, top-p 0.8: 280, 66.2; 2 x 32 of 16384, Gumbel: 235, 34.2.
//
// Gumbel race (Algorithm 4): the winner is the smallest E_v / W_v of integers that take 40 squarings each. An fp32
// estimate of every ratio first, the integers only for ids within RACE_SLACK of the smallest estimate. A row that
// may enter the window races under equal weights, which is the largest variate (see fresh_key).
//
// Exactness: sums are integers, thresholds are exact selections, every decision is an integer inequality: nothing
// depends on how ids are dealt to threads or CTAs. No thread spins: the only waits are hardware barriers that
// every CTA of a cluster reaches the same number of times (branches that hold one are taken on values that all
// CTAs of the cluster compute from the same data).
#include <algorithm>
#include <type_traits>

#include "verify.cuh"

namespace scd {

namespace {

constexpr int CT = 512;
constexpr int NWARP = CT / 32;
constexpr int NB = 1024;           // steps of a histogram
constexpr int MAXC = 8;
constexpr int MAXG = 4;            // groups of 256 ids per warp: a CTA takes up to 16384 ids
constexpr int CAND_CAP = 1024;     // candidates of a row that are selected by counting
constexpr int NUC_CAP = 256;       // ... and weights of the nucleus' last step
constexpr int WCAP_LONG = 384;     // list entries of a warp of up to 1024 ids (two CTAs share an SM's memory)
constexpr float LIVE_SPAN = 22.0f; // scd_exp(x) = 0 below -22
constexpr unsigned W_TAIL = 1u << 14;   // nucleus: lighter ids are only summed at first
constexpr float LIST_SHARE = 0.28f;     // ... and so are those beyond this share of the ids (a list takes 384 of 1024)
constexpr float TAIL_WIDE = 0.6f, TAIL_TIGHT = 0.85f, LIST_FILL = 0.8f, FAR = 1.6f;   // (where the lists are built)
constexpr float RACE_SLACK = 2e-4f;
constexpr unsigned FULLM = 0xffffffffu;

// Code that runs on the target row and, when the draft row arrives as raw logits, on the draft row too: the
// index is a compile-time constant inside, so that per-thread values stay in registers.
template <int A> struct RowIndex { static constexpr int value = A; };
#define EACH_ROW(...) do { auto fn_ = __VA_ARGS__; fn_(RowIndex<0>{}); if (NA > 1) fn_(RowIndex<1>{}); } while (0)

struct Xchg {                                  // read by the peers through distributed shared memory
    unsigned hist[2][2][NB];                   // [row]: counts, or masses in two parts (low 15 bits of the weights, the rest);
                                               // once the peers have read them: the row's candidates
    uint2 cand[2][CAND_CAP];                   // (order-preserving key of x, W) of the ids in the selected step ...
    unsigned long long u64[8];
    unsigned long long racer[2], fresh;        // (T, W : id) of this CTA's best racer; its largest fresh key
    float f32[4];                              // maxima, bounds
    unsigned cand_n[2];
};

struct Local {
    unsigned short cand_at[2][CAND_CAP];       // ... and where they are in this CTA's lists
    float red_f[2][NWARP];
    unsigned long long red_a[NWARP], red_b[NWARP];   // per-warp values of a block reduction
    unsigned long long scan[2][NWARP / 2];
    unsigned long long peer[4][MAXC];
    unsigned peer_n[2][MAXC];
    int sel[2];
    float bound[2], cuts[2][5];
    bool give_up[2];
    unsigned sel_k[2], tau_key[2];
    unsigned long long above[2], kept[2], total[2];
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ unsigned ld_peer_u32(const void *local, uint32_t rank)
{
    unsigned v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(peer_addr(smem_addr(local), rank)) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_peer_u64(const void *local, uint32_t rank)
{
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(peer_addr(smem_addr(local), rank)) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_peer_u32x4(const void *local, uint32_t rank)
{
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(peer_addr(smem_addr(local), rank)) : "memory");
    return v;
}

// order-preserving key of a logit for the selection of the threshold. -0 takes the key of +0: the ids at the threshold are
// those that compare equal to it as floats (with a key of its own -0 lost its weight here and kept it in the accept test)
__device__ __forceinline__ unsigned logit_key(float x) { return float_key(__fadd_rn(x, 0.0f)); }

// step of the live range an id falls into: 0 at the maximum, NB - 1 at m - 22; -1: not live
__device__ __forceinline__ int live_step(float x, float m)
{
    const float dlt = __fsub_rn(m, x);                 // = -(x - m) exactly
    if (!(dlt <= LIVE_SPAN)) return -1;
    return min(max(__float2int_rd(__fmul_rn(dlt, (float)NB / 22.5f)), 0), NB - 1);
}
// logarithmic step of a weight, heaviest first: exponent and five more bits (W >= 1, monotone)
__device__ __forceinline__ int weight_step(unsigned w)
{
    const int e = 31 - __clz(w);
    return NB - 1 - ((e << 5) | (int)(((w << (31 - e)) >> 26) & 31u));
}
__device__ __forceinline__ unsigned weight_step_lo(int step)         // smallest weight of a step
{
    const int s = NB - 1 - step, e = s >> 5;
    const unsigned long long f = (32ull | (unsigned)(s & 31)) << e;  // in units of 2^-5, rounded up
    return (unsigned)((f + 31) >> 5);
}

// residual mass of one id: max(0, Wp Zq - Wq Zp)
__device__ __forceinline__ u128 residual_of(unsigned wp, unsigned wq, unsigned long long Zp, unsigned long long Zq)
{
    if (wp == 0u) return (u128)0;
    const u128 a = mul_32x64(wp, Zq), b = mul_32x64(wq, Zp);
    return a > b ? a - b : (u128)0;
}

// Whether row (b, pos) of iteration t is redrawn independently (Algorithm 2 always, Algorithm 5 by its coin).
__device__ __forceinline__ bool redraw_independent(const VerifyParams &p, int b, long long pos, unsigned t)
{
    if (p.mode == SCD_MODE_SJD) return true;
    if (p.mode != SCD_MODE_ALPHA) return false;
    const unsigned Ub = noise_u24(p.seed, NOISE_ALPHA, (unsigned)b, pos, t, 0);
    return !((double)(Ub + 1u) <= (double)p.alpha * 16777216.0);
}

// fp32 estimate of -log2((U + 1/2) / 2^24). Both arguments are exact (below 1/2 and above, 24 bits each), log2f and
// log1pf err by an ulp or two.
__device__ __forceinline__ float neglog2_estimate(unsigned U)
{
    if (U < (1u << 23)) return -log2f((float)(2u * U + 1u) * 0x1p-25f);
    return -log1pf(-((float)(2u * (0xFFFFFFu - U) + 1u) * 0x1p-25f)) * 0x1.715476p+0f;
}

// post-processed logit of one id (u: unconditional row or null), off the main path
__device__ __noinline__ float post_logit(const float *c, const float *u, int v, float one_plus_lam, float lam, float T)
{
    float x = __ldcg(c + v);
    if (u) x = __fsub_rn(__fmul_rn(one_plus_lam, x), __fmul_rn(lam, __ldcg(u + v)));
    return T != 1.0f ? __fdiv_rn(x, T) : x;
}

// Nucleus: the candidates of every CTA (up to NUC_CAP weights of each row's last step) to this one, and among them the largest
// weight whose ids, with the mass above the step, hold top_p of the mass Z: into lc.tau_key, the mass into lc.kept. Half the
// threads per row, a candidate each. (Off the main path: inlined it cost every call registers)
__device__ __noinline__ void nucleus_among(Xchg &xc, Local &lc, int C, unsigned p24, unsigned long long Z0, unsigned long long Z1,
                                           unsigned long long above0, unsigned long long above1)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, a = tid >> 8;
    const unsigned t = tid & 255;
    if (warp < 2 && lane < MAXC) lc.peer_n[warp][lane] = lane < C ? ld_peer_u32(&xc.cand_n[warp], (uint32_t)lane) : 0u;
    __syncthreads();
    unsigned n = 0;
#pragma unroll
    for (int r = 0; r < MAXC; ++r) n += lc.peer_n[a][r];
    unsigned *const all = &xc.hist[a][0][0];           // (the tables are done with)
    if (t < n) {
        unsigned off = 0;
        int rr = 0;
#pragma unroll
        for (int r = 0; r < MAXC - 1; ++r) {
            const unsigned end = off + lc.peer_n[a][r];
            if (rr == r && t >= end) { off = end; rr = r + 1; }
        }
        all[t] = ld_peer_u32(&xc.cand[a][t - off].x, (uint32_t)rr);
    }
    __syncthreads();
    if (t < n) {
        const unsigned wv = all[t];
        unsigned long long gt = a ? above1 : above0, ge = gt;
        for (unsigned i = 0; i < n; ++i) {
            const unsigned o = all[i];
            gt += o > wv ? o : 0u;
            ge += o >= wv ? o : 0u;
        }
        const u128 need = (u128)p24 * (a ? Z1 : Z0);
        if (((u128)ge << 24) >= need && ((u128)gt << 24) < need) { lc.tau_key[a] = wv; lc.kept[a] = ge; }   // (equal weights write the same)
    }
    __syncthreads();
}

// A warp's ids come in groups of NS x 128: lane l holds ids 4 l .. 4 l + 3 of each 128 (16-byte loads where rows are
// aligned). REG: one group, which stays in registers. Else long_range: ids of a warp, a multiple of 32. (As a multiple of a
// group it left half of the warps without ids where a warp's share is just above one group, and the others with more than
// a list takes: 8 x 32 rows of 4371 ids, top-k 4000, 82.9 us, 42.4 so. In registers there is no such limit, and shares
// that are no whole groups are 5 % slower: 6 rows of 24774 ids 26.1 and 27.3 us.)
// TOP_P: with nucleus truncation. (A kernel of its own: in one with the rest it cost the other calls spilled registers, 32
// rows of 16384 ids 24.0 us, 21.1 so; 256 rows with guidance 48.9 and 44.9.)
template <int NS, bool REG, bool TOP_P>
__global__ void __launch_bounds__(CT, 2) verify_rows_kernel(const VerifyParams p, int C, int long_range)
{
    constexpr int N = 4 * NS;                          // ids per lane and group
    constexpr int WCAP = REG ? 32 * N : WCAP_LONG;     // entries of a warp's list
    const int range = REG ? 32 * N : long_range;       // ids of a warp
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ __align__(16) Xchg xc;
    __shared__ Local lc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x % C;                   // = rank in the cluster (cluster dims (C, 1, 1))
    const int k = blockIdx.x / C, b = blockIdx.y;
    pdl_trigger();
    auto zero_hist = [&]() {
        for (int i = tid; i < 2 * 2 * NB / 4; i += CT) ((uint4 *)&xc.hist[0][0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    };
    zero_hist();
    // This grid may have started early. In a session it reads, up to the wait further down, only what earlier iterations left
    // behind - the window counters, the draft ids, the drafts' stored weights. In a stand-alone call every input may come from
    // the kernel in front.
    if (!p.n_known) pdl_wait();
    const WindowState w = load_state(p, b);
    if (k >= w.Lw) { pdl_wait(); return; }             // (all CTAs of the cluster; no kernel ends before the one in front)
    const int L = p.L, V = p.V;
    const size_t row = (size_t)b * L + k;
    const long long pos = w.pos0 + k;
    int lo, hi;
    allowed_range(p, pos, lo, hi);
    // rows that are 16-byte aligned throughout are dealt from an aligned id on
    const bool vec = (V & 3) == 0 && ((uintptr_t)p.p_logits & 15) == 0 && ((uintptr_t)p.xbuf[w.parity ^ 1] & 15) == 0;
    const int wbase = (vec ? lo & ~3 : lo) + (rank * NWARP + warp) * range, wend = min(hi, wbase + range);
    const bool mix = p.S == 2, div = p.temperature != 1.0f;
    const bool use_topk = p.top_k > 0 && p.top_k < hi - lo;
    const int qk = k + w.shift;
    const bool fresh = !(qk < w.prev_lw);
    const bool rawq = !fresh && p.q_is_raw;            // draft distribution from raw logits, built here
    const int NA = rawq ? 2 : 1;
    const bool mrs = p.mode != SCD_MODE_AR;
    const float *c = p.p_logits + row * V;
    const float *u = mix ? p.p_logits + ((size_t)(p.B + b) * L + k) * V : nullptr;
    const float *qr = fresh ? nullptr : p.xbuf[w.parity ^ 1] + ((size_t)b * L + qk) * V;
    // the lists [warp][WCAP]: value (x, later the weight) and id of the target row's entries, values of the draft row's
    uint2 *const list_p = (uint2 *)dyn + (size_t)warp * WCAP;
    unsigned *const list_q = (unsigned *)((uint2 *)dyn + (size_t)NWARP * WCAP) + (size_t)warp * WCAP;

    auto csync = [&]() {                               // barrier of the cluster
        if (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        else __syncthreads();
    };
    // (the target logits are read through L2: this kernel may have started before they were written, and the
    // non-coherent load path then served stale lines of the previous iteration)
    auto load_p = [&](int v) -> float { return post_logit(c, u, v, p.one_plus_lam, p.lam, p.temperature); };
    auto load_q = [&](int v) -> float { return post_logit(qr, nullptr, v, 0.f, 0.f, p.temperature); };

    auto load4 = [&](const float *src, int v, float *x) {            // ids v .. v + 3, at least the first of them below hi
        if (vec) {
            const float4 t = __ldcg((const float4 *)(src + v));
            x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = v + i >= hi ? 0.f : __ldcg(src + v + i);
        }
    };
    auto has = [&](int v) { return v >= lo && v < wend; };
    float xr[2][N];
    bool loaded = false;
    // body(v): this lane's x of a group are in xr[row], its ids in v + 128 h + i
    auto sweep = [&](auto body) {
#pragma unroll 1
        for (int v0 = wbase; REG ? v0 == wbase : v0 < wbase + range; v0 += 32 * N) {
            const int v = v0 + 4 * lane;
            if (!REG || !loaded) {                     // both rows, all loads in flight
                float t[N], s[N];
#pragma unroll
                for (int j = 0; j < N; ++j) t[j] = s[j] = xr[1][j] = 0.f;
#pragma unroll
                for (int h = 0; h < NS; ++h) {
                    if (v + 128 * h >= wend) continue;
                    if (rawq) load4(qr, v + 128 * h, &xr[1][4 * h]);
                    load4(c, v + 128 * h, &t[4 * h]);
                    if (mix) load4(u, v + 128 * h, &s[4 * h]);
                }
                if (mix) {
#pragma unroll
                    for (int j = 0; j < N; ++j) t[j] = __fsub_rn(__fmul_rn(p.one_plus_lam, t[j]), __fmul_rn(p.lam, s[j]));
                }
                if (div) {
#pragma unroll
                    for (int j = 0; j < N; ++j) { t[j] = __fdiv_rn(t[j], p.temperature); xr[1][j] = __fdiv_rn(xr[1][j], p.temperature); }
                }
#pragma unroll
                for (int j = 0; j < N; ++j) xr[0][j] = t[j];
                // ids that do not exist: NaN, which no comparison below takes
                if (v0 < lo || v0 + 32 * N > wend) {
#pragma unroll
                    for (int j = 0; j < N; ++j)
                        if (!has(v + 128 * (j >> 2) + (j & 3))) xr[0][j] = xr[1][j] = __int_as_float(0x7FC00000);
                }
            }
            body(v);
        }
        loaded = true;
    };
    auto warp_sum64 = [&](unsigned long long x) -> unsigned long long {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULLM, x, o);
        return x;
    };
    auto all_cand = [&](int a) -> uint2 * { return (uint2 *)&xc.hist[a][0][0]; };
    static_assert(sizeof(uint2) * CAND_CAP <= sizeof(xc.hist[0]), "the candidates reuse the histograms");

    const int X = p.draft_in[row];
    const bool x_in = X >= lo && X < hi;
    const float xq_raw = qr && x_in ? qr[X] : 0.f;     // raw logit, or stored integer weight (bit pattern), of the draft
    const unsigned long long Zq_stored = !fresh && !rawq ? p.stats[w.parity ^ 1][(size_t)b * L + qk].Z : 0ull;
    if (tid < 2) { xc.cand_n[tid] = 0u; lc.sel[tid] = -1; lc.bound[tid] = -INFINITY; lc.above[tid] = lc.kept[tid] = 0ull; }
    __syncthreads();
    pdl_wait();                                        // the target logits come from the kernel in front
    const float xX = x_in ? load_p(X) : 0.f;           // the draft's own logit: every CTA weighs X itself
    unsigned *wstore = p.keep_x ? (unsigned *)(p.xbuf[w.parity] + row * V) : nullptr;
    const bool nucleus = TOP_P && !use_topk;           // the nucleus is taken of the whole row
    float m[2] = {-INFINITY, 0.f};

    // maxima (and bounds) of the CTAs -> of the row
    auto exchange_max = [&](float m0, float m1) {
        m0 = warp_max(m0);
        m1 = warp_max(m1);
        if (lane == 0) { lc.red_f[0][warp] = m0; lc.red_f[1][warp] = m1; }
        __syncthreads();
        if (warp < 2) {
            const float t = warp_max(lane < NWARP ? lc.red_f[warp][lane] : -INFINITY);
            if (lane == 0) { xc.f32[warp] = t; xc.f32[2 + warp] = lc.bound[warp]; }
        }
        csync();
        // (what every thread needs from every peer is fetched once per CTA, one lane per peer: distributed shared
        // memory is for few, wide requests)
        if (warp < 4) {
            const float t = warp_max(lane < C ? __uint_as_float(ld_peer_u32(&xc.f32[warp], (uint32_t)lane)) : -INFINITY);
            if (lane == 0) { if (warp < 2) lc.red_f[warp][0] = t; else lc.bound[warp - 2] = t; }
        }
        __syncthreads();
        m[0] = lc.red_f[0][0];
        if (rawq) m[1] = lc.red_f[1][0];
    };
    // Two ids per lane of each row, spread over the warp's range (REG: of the registers).
    auto sample = [&](auto body) {
        if (REG) {
            const int v = wbase + 4 * lane;
#pragma unroll
            for (int j = 0; j < N; j += N - 1)
                if (has(v + 128 * (j >> 2) + (j & 3))) { body(0, xr[0][j]); if (rawq) body(1, xr[1][j]); }
        } else {
            const int n = range / 128, va = wbase + 128 * (n / 4) + 4 * lane + 1, vb = wbase + 128 * (n - 1 - n / 4) + 4 * lane + 2;
            const bool ia = has(va), ib = has(vb);
            const float pa = ia ? load_p(va) : 0.f, pb = ib ? load_p(vb) : 0.f;
            const float qa = rawq && ia ? load_q(va) : 0.f, qb = rawq && ib ? load_q(vb) : 0.f;
            if (ia) { body(0, pa); if (rawq) body(1, qa); }
            if (ib) { body(0, pb); if (rawq) body(1, qb); }
        }
    };
    // After a sample's histogram (2 NB bins per row in the tables of the masses, the smallest sample in bin 0): visits the
    // bins that hold something, with want(sum of value(bin, count) over all) and the sums over the bins above and from this
    // one on.
    // Thread t of row a looks at 8 bins. The tables are cleared.
    auto sample_bins = [&](auto value, auto want, auto visit) {
        using T = decltype(value(0, 0u));
        const int a = tid >> 8, t = tid & 255, wi = warp & 7;
        T val[8], mine = 0, inc = 0;
        const unsigned *h = &xc.hist[a][0][0] + 2 * NB - 8 - 8 * t;
#pragma unroll
        for (int j = 0; j < 8; ++j) { val[j] = value(2 * NB - 8 - 8 * t + j, h[j]); mine += val[j]; }
        inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T v = __shfl_up_sync(FULLM, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) lc.scan[a][wi] = inc;
        __syncthreads();
        T acc = inc - mine, all = 0;
#pragma unroll
        for (int i = 0; i < NWARP / 2; ++i) {
            if (i < wi) acc += (T)lc.scan[a][i];
            all += (T)lc.scan[a][i];
        }
        const auto need = want(all);
#pragma unroll
        for (int j = 7; j >= 0; --j) {
            if (val[j] != 0) visit(a, 2 * NB - 8 - 8 * t + j, need, acc, acc + val[j]);
            acc += val[j];
        }
        __syncthreads();
        zero_hist();
        __syncthreads();
    };

    // The lists: of the group at v (see sweep), the ids that `keep` has a bit for (bit 4 h + i of row a), with their value
    // (x, or the weight's bit pattern). One scan over the warp for both rows: counts of up to 128 in bytes.
    int n_list[2] = {0, 0};                            // (warp-uniform; above WCAP once a list has overflowed)
    auto append = [&](int v, const unsigned (&keep)[2], const float (&val)[2][N]) {
        unsigned packed = 0;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int h = 0; h < NS; ++h) packed |= (unsigned)__popc(keep[a] >> (4 * h) & 15u) << (8 * (a * NS + h));
        unsigned inc = packed;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(FULLM, inc, o);
            if (lane >= o) inc += t;
        }
        const unsigned all = __shfl_sync(FULLM, inc, 31);
        inc -= packed;
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            if (a && !rawq) break;
            int n = n_list[a];
#pragma unroll
            for (int h = 0; h < NS; ++h) n_list[a] += (int)(all >> (8 * (a * NS + h)) & 255u);
            if (n_list[a] > WCAP) continue;
#pragma unroll
            for (int h = 0; h < NS; ++h) {
                int at = n + (int)(inc >> (8 * (a * NS + h)) & 255u);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (!(keep[a] >> (4 * h + i) & 1u)) continue;
                    if (a == 0) list_p[at] = make_uint2(__float_as_uint(val[a][4 * h + i]), (unsigned)(v + 128 * h + i));
                    else list_q[at] = __float_as_uint(val[a][4 * h + i]);
                    ++at;
                }
                n += (int)(all >> (8 * (a * NS + h)) & 255u);
            }
        }
        if (wstore) {
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (!(keep[0] >> j & 1u) && has(v + 128 * (j >> 2) + (j & 3))) wstore[v + 128 * (j >> 2) + (j & 3)] = 0u;
        }
    };
    // entry e of this warp: of its list, or of its whole range when the list did not fit
    bool whole[2] = {false, false};
    bool dense = false;                                // whole[0], and the weights of the range lie where the lists were
    auto dense_at = [&](int e) -> unsigned * { return e < 2 * WCAP ? (unsigned *)list_p + e : list_q + (e - 2 * WCAP); };
    int n_e[2] = {0, 0};
    auto close_lists = [&]() {
        __syncwarp();
#pragma unroll
        for (int a = 0; a < 2; ++a) { whole[a] = n_list[a] > WCAP; n_e[a] = whole[a] ? range : n_list[a]; }
    };
    float tau[2] = {-INFINITY, -INFINITY};
    unsigned theta[2] = {0u, 0u};
    auto entry_in = [&](int a, int e) -> bool { return e < n_e[a] && (!whole[a] || has(wbase + e)); };
    auto entry_x = [&](auto A_, int e, bool &in) -> float {          // x of entry e (in: it exists), while the lists hold x
        constexpr int a = decltype(A_)::value;
        in = entry_in(a, e);
        if (!in) return -INFINITY;
        if (!whole[a]) return __uint_as_float(a == 0 ? list_p[e].x : list_q[e]);
        return a == 0 ? load_p(wbase + e) : load_q(wbase + e);
    };
    auto entry_w = [&](auto A_, int e) -> unsigned {                 // its weight (0: none), once they hold weights
        constexpr int a = decltype(A_)::value;
        if (!entry_in(a, e)) return 0u;
        if (!whole[a]) return a == 0 ? list_p[e].x : list_q[e];
        if (TOP_P && !REG && a == 0 && dense) return *dense_at(e);
        return weight_of(a == 0 ? load_p(wbase + e) : load_q(wbase + e), m[a], tau[a]);
    };
    auto entry_id = [&](int e) -> int { return whole[0] ? wbase + e : (int)list_p[e].y; };

    // merges the C histograms: threads 0..255 take the target row, 256..511 the draft row; each owns four steps. Scans
    // them and leaves the step in which the running sum (from `base` on) reaches top_k (counts) or top_p of the mass Z
    // in lc.sel, the sum above it in lc.above and up to it in lc.kept.
    auto select_step = [&](bool mass, unsigned long long Z0, unsigned long long Z1, unsigned long long base0, unsigned long long base1) {
        const int a = tid >> 8, t = tid & 255, wi = warp & 7;
        unsigned long long s[4] = {0ull, 0ull, 0ull, 0ull}, mine = 0, inc = 0;
        if (a < NA) {
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                if (part && !mass) break;
                uint4 t4[MAXC];
#pragma unroll
                for (int r = 0; r < MAXC; ++r) t4[r] = r < C ? ld_peer_u32x4(&xc.hist[a][part][4 * t], (uint32_t)r) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int r = 0; r < MAXC; ++r) {
                    const int sh = part ? 15 : 0;
                    s[0] += (unsigned long long)t4[r].x << sh; s[1] += (unsigned long long)t4[r].y << sh;
                    s[2] += (unsigned long long)t4[r].z << sh; s[3] += (unsigned long long)t4[r].w << sh;
                }
            }
            mine = s[0] + s[1] + s[2] + s[3];
            inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long v = __shfl_up_sync(FULLM, inc, o);
                if (lane >= o) inc += v;
            }
            if (lane == 31) lc.scan[a][wi] = inc;
        }
        __syncthreads();
        if (a < NA) {
            unsigned long long acc = (a ? base1 : base0) + inc - mine;
            for (int i = 0; i < wi; ++i) acc += lc.scan[a][i];
            const u128 need = (u128)p.top_p24 * (a ? Z1 : Z0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool hit = mass ? ((u128)(acc + s[j]) << 24) >= need && ((u128)acc << 24) < need
                                      : acc < (unsigned)p.top_k && (unsigned)p.top_k <= acc + s[j];
                if (hit) { lc.sel[a] = 4 * t + j; lc.above[a] = acc; lc.kept[a] = acc + s[j]; }
                acc += s[j];
            }
        }
        __syncthreads();
    };
    auto add_mass = [&](int a, int step, unsigned wv) {
        atomicAdd(&xc.hist[a][0][step], wv & 0x7FFFu);
        atomicAdd(&xc.hist[a][1][step], wv >> 15);
    };

    int sb[2] = {-1, -1};                              // selected step
    unsigned long long Zall[2] = {0ull, 0ull};         // normaliser
    if (!nucleus) {
        // ---- top-k, or no truncation ------------------------------------------------------------------------------
        if (use_topk && !REG) {
            sample([&](int a, float x) { atomicAdd(&xc.hist[a][0][0] + (float_key(x) >> 21), 1u); });
            __syncthreads();
            // (a share of top_k / n of the samples lies above the k-th largest, give or take; four deviations more are
            // listed. Without that many samples the list takes everything.)
            const float share = (float)p.top_k / (float)(hi - lo);
            sample_bins([](int, unsigned n) { return n; },
                        [&](unsigned all) { const float e = share * (float)all; return (unsigned)(e + 4.0f * sqrtf(e)) + 4u; },
                        [&](int a, int bin, unsigned need, unsigned above, unsigned sum) {
                if (above >= need || sum < need) return;
                const float t = key_float((unsigned)bin << 21);
                lc.bound[a] = t > -INFINITY ? t : -INFINITY;                 // (the bin of -inf begins among the NaNs)
            });
        }
        for (bool again = false;; again = true) {
            const float bound[2] = {again ? -INFINITY : lc.bound[0], again ? -INFINITY : lc.bound[1]};
            float mx[2] = {-INFINITY, -INFINITY};
            n_list[0] = n_list[1] = 0;
            sweep([&](int v) {
                unsigned keep[2] = {0u, 0u};
#pragma unroll
                for (int j = 0; j < N; ++j) {
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        mx[a] = fmaxf(mx[a], xr[a][j]);
                        if (xr[a][j] >= bound[a]) keep[a] |= 1u << j;
                    }
                }
                if (!rawq) keep[1] = 0u;
                if (!REG) append(v, keep, xr);
            });
            close_lists();
            if (!again) exchange_max(mx[0], mx[1]);                                   // ---- exchange: maxima
            if (use_topk) {
                auto count = [&](int a, bool in, float x) {
                    const int s = in ? live_step(x, a ? m[1] : m[0]) : -1;
                    if (s >= 0) atomicAdd(&xc.hist[a][0][s], 1u);
                };
                if (REG) {
                    sweep([&](int) {
#pragma unroll
                        for (int j = 0; j < N; ++j) {
                            count(0, true, xr[0][j]);
                            if (rawq) count(1, true, xr[1][j]);
                        }
                    });
                } else {
                    EACH_ROW([&](auto A_) {
                        constexpr int a = decltype(A_)::value;
                        for (int e0 = 0; e0 < n_e[a]; e0 += 32) {
                            bool in;
                            const float x = entry_x(A_, e0 + lane, in);
                            count(a, in, x);
                        }
                    });
                }
                csync();                                                              // ---- exchange: histograms
                select_step(false, 0ull, 0ull, 0ull, 0ull);
                // (no step: fewer than top_k live ids. The k-th largest then has weight 0, and so has everything below
                // it: the threshold is dropped, the weights are those of the definition)
                sb[0] = lc.sel[0];
                sb[1] = lc.sel[1];
            }
            if (REG) {                                 // the ids are in registers: the lists come last
                sweep([&](int v) {
                    unsigned keep[2] = {0u, 0u};
#pragma unroll
                    for (int j = 0; j < N; ++j) {
#pragma unroll
                        for (int a = 0; a < 2; ++a) {
                            const int s = live_step(xr[a][j], m[a]);
                            if (s >= 0 && (sb[a] < 0 || s <= sb[a])) keep[a] |= 1u << j;
                        }
                    }
                    if (!rawq) keep[1] = 0u;
                    append(v, keep, xr);
                });
                close_lists();
            }
            if (!use_topk) break;
            bool complete = true;                      // every id of the step and above it is in the lists
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                const int s = live_step(lc.bound[a], m[a]);          // (a bound above m would be in step 0)
                if (s >= 0 && (sb[a] < 0 || s <= sb[a])) complete = false;
            });
            if (complete || again) {
                if (tid < 2) lc.sel_k[tid] = (unsigned)p.top_k - (unsigned)lc.above[tid];
                break;
            }
            csync();                                   // every peer has read these tables
            if (tid < 2) lc.sel[tid] = -1;
            zero_hist();
            __syncthreads();
        }
    } else {
        // ---- nucleus of the whole row ---------------------------------------------------------------------------------
        {
            float mx[2] = {-INFINITY, -INFINITY};
            sweep([&](int) {
#pragma unroll
                for (int j = 0; j < N; ++j) { mx[0] = fmaxf(mx[0], xr[0][j]); mx[1] = fmaxf(mx[1], xr[1][j]); }
            });
            exchange_max(mx[0], mx[1]);                                               // ---- exchange: maxima
        }
        sample([&](int a, float x) {
            const unsigned wv = weight_of(x, a ? m[1] : m[0], -INFINITY);
            atomicAdd(&xc.hist[a][0][0] + (wv ? NB - 1 - weight_step(wv) : 0), 1u);
        });
        // The bound lists the heaviest LIST_SHARE of the ids, and in flat rows more: until the sample's mass reaches top_p and
        // TAIL_WIDE of the rest, so that the nucleus ends inside the lists (without it such rows had them built twice: 175
        // rows of 12991 ids, guidance, top-p 0.95, 226 us, 65 so), but not more than fit a list (LIST_FILL: some warps have
        // more ids above the bound than others). Only where the nucleus itself is far from fitting (top_p and TAIL_TIGHT of the rest take
        // FAR times as much) the lists are given up at once (128 rows of 30000 ids, top-p 0.99: 138 us after a try, 111 so).
        if (tid < 10) (&lc.cuts[0][0])[tid] = (float)W_TAIL;
        __syncthreads();
        auto cut_at = [&](int bin) { return fmaxf((float)W_TAIL, bin > 0 ? (float)weight_step_lo(NB - 1 - bin) : 0.f); };
        const float rest = 1.0f - (float)p.top_p24 * 0x1p-24f, fit = LIST_FILL * (float)WCAP / (float)range;
        // (number and mass of a bin's ids in one word: up to 1024 of them, weights below 2^31)
        sample_bins([](int bin, unsigned n) { return ((unsigned long long)n << 48) + (bin > 0 ? (unsigned long long)n * weight_step_lo(NB - 1 - bin) : 0ull); },
                    [](unsigned long long all) { return all; },
                    [&](int a, int bin, unsigned long long all, unsigned long long above, unsigned long long sum) {
            const unsigned long long mass = 0xFFFFFFFFFFFFull;
            const float n = (float)(all >> 48), m_ = (float)(all & mass);
            auto ids = [&](float share) { const unsigned need = (unsigned)(share * n) + 1u; return (unsigned)(above >> 48) < need && need <= (unsigned)(sum >> 48); };
            auto tail = [&](float share) { const unsigned long long need = (all & mass) - (unsigned long long)(share * rest * m_); return (above & mass) < need && need <= (sum & mass); };
            if (ids(LIST_SHARE)) lc.cuts[a][0] = cut_at(bin);
            if (ids(fit)) lc.cuts[a][1] = cut_at(bin + 1);
            if (ids(FAR * fit)) lc.cuts[a][2] = cut_at(bin + 1);
            if (tail(TAIL_WIDE)) lc.cuts[a][3] = cut_at(bin);
            if (tail(TAIL_TIGHT)) lc.cuts[a][4] = cut_at(bin);
        });
        if (tid < 2) {
            const float *c_ = lc.cuts[tid];
            lc.give_up[tid] = c_[4] < c_[2];
            lc.bound[tid] = c_[4] < c_[2] ? fminf(c_[0], c_[4]) : fmaxf(fminf(c_[0], c_[3]), c_[1]);
        }
        __syncthreads();
        // A warp whose target list is given up, or overflows, keeps the weights of its whole range where the lists were: up to
        // 2 x 384 words over the target row's, up to 1024 where the draft row leaves its own free. Weighed again from L2 in
        // every pass instead, 64 rows of 64000 ids of a random decoder took 212 us inside a session, 155 so; 64 rows of 64000
        // ids, top-p 0.95, both rows raw, 161 us, 139 so. A list that fits is the shorter one to go over (128 rows of 20000
        // ids, guidance, top-p 0.99: 82 us, 94 with the weights of whole ranges).
        const bool give_up[2] = {!REG && range > WCAP && lc.give_up[0], !REG && range > WCAP && lc.give_up[1]};
        auto fill = [&](int v) {
#pragma unroll
            for (int h = 0; h < NS; ++h) {
                const int e = v + 128 * h - wbase;
                if (e >= range) continue;
                unsigned wv[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) wv[i] = weight_of(xr[0][4 * h + i], m[0], -INFINITY);
                *(uint4 *)dense_at(e) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
            }
        };
        for (bool again = false;; again = true) {
            // (a bound is the smallest weight of a step: exact in fp32)
            const unsigned cut[2] = {again ? 1u : (unsigned)lc.bound[0], again ? 1u : (unsigned)lc.bound[1]};
            unsigned long long z[2] = {0ull, 0ull};
            dense = give_up[0] && (range <= 2 * WCAP || !rawq || give_up[1]);
            n_list[0] = dense ? WCAP + 1 : 0;
            n_list[1] = dense && give_up[1] ? WCAP + 1 : 0;
            sweep([&](int v) {
                unsigned keep[2] = {0u, 0u};
                float val[2][N];
#pragma unroll
                for (int j = 0; j < N; ++j) {
#pragma unroll
                    for (int a = 0; a < 2; ++a) {
                        if (a && !rawq) break;
                        const unsigned wv = weight_of(xr[a][j], m[a], -INFINITY);
                        z[a] += wv;
                        if (wv >= cut[a]) keep[a] |= 1u << j;
                        val[a][j] = __uint_as_float(wv);
                    }
                }
                if (!REG && dense) {
                    keep[0] = 0u;
                    fill(v);
                }
                if (!dense || (rawq && !give_up[1]) || wstore) append(v, keep, val);
            });
            close_lists();
            if (!REG && whole[0] && !dense && (range <= 2 * WCAP || !rawq || whole[1])) {
                dense = true;
                sweep(fill);
                __syncwarp();
            }
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                const unsigned long long t = warp_sum64(z[a]);
                if (lane == 0) (a ? lc.red_b : lc.red_a)[warp] = t;
                for (int e = lane; e < n_e[a]; e += 32) {
                    const unsigned wv = entry_w(A_, e);
                    if (wv >= cut[a]) add_mass(a, weight_step(wv), wv);
                }
            });
            __syncthreads();
            if (warp < NA) {
                const unsigned long long t = warp_sum64(lane < NWARP ? (warp ? lc.red_b : lc.red_a)[lane] : 0ull);
                if (lane == 0) { xc.u64[warp] = t; xc.f32[2 + warp] = (float)cut[warp]; }
            }
            csync();                                                                  // ---- exchange: histograms, sums, bounds
            if (warp < 2 * NA) {
                const int a = warp >> 1;
                if (warp & 1) {
                    const float t = warp_max(lane < C ? __uint_as_float(ld_peer_u32(&xc.f32[2 + a], (uint32_t)lane)) : 0.f);
                    if (lane == 0) lc.red_f[a][0] = t;
                } else {
                    const unsigned long long t = warp_sum64(lane < C ? ld_peer_u64(&xc.u64[a], (uint32_t)lane) : 0ull);
                    if (lane == 0) lc.peer[a][0] = t;
                }
            }
            __syncthreads();
            Zall[0] = lc.peer[0][0];
            if (rawq) Zall[1] = lc.peer[1][0];
            select_step(true, Zall[0], Zall[1], 0ull, 0ull);
            bool complete = true;                      // every id of the step and above it is in the lists
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                sb[a] = lc.sel[a];
                if (sb[a] < 0 || (float)weight_step_lo(sb[a]) < lc.red_f[a][0]) complete = false;
            });
            csync();                                   // every peer has read these tables
            zero_hist();
            __syncthreads();
            if (complete || again) break;
            if (tid < 2) lc.sel[tid] = -1;
            __syncthreads();
        }
    }

    if (!nucleus) {
        // ---- mass above the selected step, its candidates, the exact threshold, the normaliser ------------------------
        EACH_ROW([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            unsigned long long z = 0;
            for (int e = lane; e < n_e[a]; e += 32) {
                bool in;
                const float x = entry_x(A_, e, in);
                const int s = in ? live_step(x, m[a]) : -1;
                const bool above = s >= 0 && (sb[a] < 0 || s < sb[a]), cand = s >= 0 && s == sb[a];
                const unsigned wv = above || cand ? weight_of(x, m[a], -INFINITY) : 0u;
                if (above) z += wv;
                if (!whole[a]) { if (a == 0) list_p[e].x = wv; else list_q[e] = wv; }   // the lists hold weights from here on
                if (cand) {
                    const unsigned at = atomicAdd(&xc.cand_n[a], 1u);
                    if (at < CAND_CAP) {
                        xc.cand[a][at] = make_uint2(logit_key(x), wv);
                        lc.cand_at[a][at] = (unsigned short)(whole[a] ? 0xFFFF : warp * WCAP + e);
                    }
                }
            }
            __syncwarp();
            z = warp_sum64(z);
            if (lane == 0) (a ? lc.red_b : lc.red_a)[warp] = z;
        });
        __syncthreads();
        if (warp < NA) {
            const unsigned long long t = warp_sum64(lane < NWARP ? (warp ? lc.red_b : lc.red_a)[lane] : 0ull);
            if (lane == 0) xc.u64[warp] = t;
        }
        csync();                                                                      // ---- exchange: masses, candidates
        if (warp < 2 * NA) {                           // warps 0, 1: the target row's mass and counts; 2, 3: the draft row's
            const int a = warp >> 1;
            if (warp & 1) { if (lane < MAXC) lc.peer_n[a][lane] = lane < C && lc.sel[a] >= 0 ? ld_peer_u32(&xc.cand_n[a], (uint32_t)lane) : 0u; }
            else {
                const unsigned long long t = warp_sum64(lane < C ? ld_peer_u64(&xc.u64[a], (uint32_t)lane) : 0ull);
                if (lane == 0) lc.total[a] = t;
            }
        }
        __syncthreads();
        unsigned n_all[2] = {0u, 0u};
        EACH_ROW([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            Zall[a] = lc.total[a];
#pragma unroll
            for (int r = 0; r < MAXC; ++r) n_all[a] += lc.peer_n[a][r];
        });
        {                                              // gather: half the threads per row, entry e of the peers' lists in turn
            const int a = tid >> 8;
            const unsigned n = a < NA ? n_all[a] : 0u;
            if (n <= CAND_CAP) {
                for (unsigned e = tid & 255; e < n; e += CT / 2) {
                    unsigned off = 0;
                    int rr = 0;
#pragma unroll
                    for (int r = 0; r < MAXC - 1; ++r) {
                        const unsigned end = off + lc.peer_n[a][r];
                        if (rr == r && e >= end) { off = end; rr = r + 1; }
                    }
                    const unsigned long long kw = ld_peer_u64(&xc.cand[a][e - off], (uint32_t)rr);
                    all_cand(a)[e] = make_uint2((unsigned)kw, (unsigned)(kw >> 32));
                }
            }
        }
        __syncthreads();
        EACH_ROW([&](auto A_) {                        // the sel_k-th largest key of the list, by counting
            constexpr int a = decltype(A_)::value;
            if (sb[a] < 0 || n_all[a] > CAND_CAP) return;
            const unsigned kk = lc.sel_k[a];
            for (unsigned j = tid; j < n_all[a]; j += CT) {
                const unsigned key = all_cand(a)[j].x;
                unsigned gt = 0, ge = 0;
                for (unsigned i = 0; i < n_all[a]; ++i) {
                    const unsigned o = all_cand(a)[i].x;
                    gt += o > key ? 1u : 0u;
                    ge += o >= key ? 1u : 0u;
                }
                if (gt < kk && kk <= ge) lc.tau_key[a] = key;        // (equal keys write the same value)
            }
        });
        __syncthreads();
        EACH_ROW([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            if (sb[a] < 0) return;
            if (n_all[a] <= CAND_CAP) {
                const unsigned tk = lc.tau_key[a];
                tau[a] = key_float(tk);
                for (unsigned i = tid; i < xc.cand_n[a]; i += CT) {  // candidates below the threshold lose their weight
                    const unsigned at = lc.cand_at[a][i];
                    if (xc.cand[a][i].x < tk && at != 0xFFFFu) { if (a == 0) ((uint2 *)dyn)[at].x = 0u; else (list_q - (size_t)warp * WCAP)[at] = 0u; }
                }
                unsigned long long add = 0;            // the candidates that stay (every warp sums the list for itself)
                for (unsigned i = lane; i < n_all[a]; i += 32)
                    if (all_cand(a)[i].x >= tk) add += all_cand(a)[i].y;
                Zall[a] += warp_sum64(add);
                return;
            }
            // long runs of equal or nearly equal logits: radix selection over the cluster, 8 bits of the key per pass,
            // among the ids of the step; then the normaliser from scratch. The warps work on their whole ranges from here
            // on (their lists hold weights that the threshold does not know).
            whole[a] = true;
            n_e[a] = range;
            unsigned prefix = 0, mask = 0, kk = lc.sel_k[a];
            for (int pass = 0; pass < 4; ++pass) {
                const int shift = 24 - 8 * pass;
                csync();                               // (nobody still reads the counters)
                for (int i = tid; i < 256; i += CT) xc.hist[a][0][i] = 0u;
                __syncthreads();
                for (int e0 = 0; e0 < n_e[a]; e0 += 32) {
                    bool in;
                    const float x = entry_x(A_, e0 + lane, in);
                    if (!in || live_step(x, m[a]) != sb[a]) continue;
                    const unsigned key = logit_key(x);
                    if ((key & mask) == prefix) atomicAdd(&xc.hist[a][0][(key >> shift) & 255u], 1u);
                }
                csync();
                if (warp == 0) {                       // lane l owns the values 8 l .. 8 l + 7
                    unsigned cnt[8], mine = 0;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        cnt[j] = 0;
                        for (int r = 0; r < C; ++r) cnt[j] += ld_peer_u32(&xc.hist[a][0][8 * lane + j], (uint32_t)r);
                        mine += cnt[j];
                    }
                    unsigned suf = mine;               // sum over lanes >= lane
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const unsigned t = __shfl_down_sync(FULLM, suf, o);
                        if (lane + o < 32) suf += t;
                    }
                    unsigned acc = suf - mine;
#pragma unroll
                    for (int j = 7; j >= 0; --j) {
                        if (acc < kk && kk <= acc + cnt[j]) { lc.tau_key[a] = 8u * lane + j; lc.sel_k[a] = kk - acc; }
                        acc += cnt[j];
                    }
                }
                __syncthreads();
                prefix |= lc.tau_key[a] << shift;
                mask |= 0xFFu << shift;
                kk = lc.sel_k[a];
            }
            tau[a] = key_float(prefix);
            unsigned long long z = 0;
            for (int e0 = 0; e0 < n_e[a]; e0 += 32) {
                bool in;
                const float x = entry_x(A_, e0 + lane, in);
                if (in) z += weight_of(x, m[a], tau[a]);
            }
            z = warp_sum64(z);
            if (lane == 0) lc.red_a[warp] = z;
            __syncthreads();
            if (warp == 0) {
                const unsigned long long t = warp_sum64(lane < NWARP ? lc.red_a[lane] : 0ull);
                if (lane == 0) xc.u64[2 + a] = t;
            }
            csync();
            if (warp == 0) {
                const unsigned long long t = warp_sum64(lane < C ? ld_peer_u64(&xc.u64[2 + a], (uint32_t)lane) : 0ull);
                if (lane == 0) lc.total[a] = t;
            }
            __syncthreads();
            Zall[a] = lc.total[a];
        });
        __syncthreads();                               // (weights of other warps' entries were cleared)
    }
    // ---- nucleus: theta = the largest weight whose ids {W >= theta} hold at least top_p of the mass. The selected step
    // is a range [range_lo, range_lo + 2^bits) of weights, divided NB ways until it is one value. -------------------
    if (TOP_P) {
        unsigned range_lo[2] = {0u, 0u};
        int bits[2] = {0, 0};
        unsigned long long above[2] = {0ull, 0ull};    // mass of the weights above the range
        auto level = [&](auto step_of) {               // one division: step_of(a, W) = step of NB, heaviest first, or -1
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                for (int e = lane; e < n_e[a]; e += 32) {
                    const unsigned wv = entry_w(A_, e);
                    const int s = wv != 0u ? step_of(a, wv) : -1;
                    if (s >= 0) add_mass(a, s, wv);
                }
            });
            csync();
            select_step(true, Zall[0], Zall[1], above[0], above[1]);
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                sb[a] = lc.sel[a];
                above[a] = lc.above[a];
            });
            csync();                                   // every peer has read these tables
            zero_hist();
            __syncthreads();
        };
        if (use_topk) {                                // (the histogram tables hold the counts of top-k)
            csync();
            zero_hist();
            if (tid < 2) xc.cand_n[tid] = 0u;
            __syncthreads();
            level([&](int, unsigned wv) { return weight_step(wv); });
        } else {
            above[0] = lc.above[0];
            above[1] = lc.above[1];
        }
        EACH_ROW([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            if (Zall[a] == 0ull) return;               // no id has a weight: no step, nothing to divide
            range_lo[a] = weight_step_lo(sb[a]);
            bits[a] = max(0, ((NB - 1 - sb[a]) >> 5) - 5);           // a step is 2^(e - 5) weights wide
        });
        auto in_range = [&](int a, unsigned wv) { return wv >= range_lo[a] && ((wv - range_lo[a]) >> bits[a]) == 0u; };
        while (bits[0] > 0 || (rawq && bits[1] > 0)) {
            // the range's mass over its smallest weight bounds the number of its ids
            bool few = true;
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                if (bits[a] > 0 && lc.kept[a] - lc.above[a] > (unsigned long long)NUC_CAP * range_lo[a]) few = false;
            });
            if (!few) {
                const int sh[2] = {max(0, bits[0] - 10), max(0, bits[1] - 10)};
                level([&](int a, unsigned wv) -> int {
                    const unsigned d = (wv - range_lo[a]) >> sh[a];
                    return in_range(a, wv) ? NB - 1 - (int)d : -1;
                });
                EACH_ROW([&](auto A_) {
                    constexpr int a = decltype(A_)::value;
                    range_lo[a] += (unsigned)(NB - 1 - sb[a]) << sh[a];
                    bits[a] = sh[a];
                });
                continue;
            }
            // few: every CTA takes them all and selects among them by counting, one exchange for what takes up to three
            // divisions of two each (16 rows of 21458 ids, top-k 1000 and top-p 0.8: 84 us, 48 so)
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                if (bits[a] == 0) return;
                for (int e = lane; e < n_e[a]; e += 32) {
                    const unsigned wv = entry_w(A_, e);
                    if (wv == 0u || !in_range(a, wv)) continue;
                    const unsigned at = atomicAdd(&xc.cand_n[a], 1u);
                    if (at < CAND_CAP) xc.cand[a][at].x = wv;
                }
            });
            csync();                                                                  // ---- exchange: candidates
            nucleus_among(xc, lc, C, (unsigned)p.top_p24, Zall[0], Zall[1], above[0], above[1]);
            EACH_ROW([&](auto A_) {
                constexpr int a = decltype(A_)::value;
                if (bits[a] > 0) range_lo[a] = lc.tau_key[a];
            });
            break;
        }
        EACH_ROW([&](auto A_) {
            constexpr int a = decltype(A_)::value;
            theta[a] = range_lo[a];
            if (Zall[a] != 0ull) Zall[a] = lc.kept[a];
        });
    }
    const unsigned long long Zp = Zall[0];
    const unsigned long long Zq = rawq ? Zall[1] : fresh ? (unsigned long long)(hi - lo) : Zq_stored;
    auto weight_p = [&](int e) -> unsigned {
        const unsigned wv = entry_w(RowIndex<0>{}, e);
        return wv >= theta[0] ? wv : 0u;
    };
    if (wstore) {
        for (int e = lane; e < n_e[0]; e += 32)
            if (entry_in(0, e)) wstore[entry_id(e)] = weight_p(e);
    }
    if (rank == 0 && tid == 0) {
        RowStats st; st.m = m[0]; st.tau = tau[0]; st.Z = Zp; st.theta = theta[0]; st.pad_ = 0u;
        p.stats[w.parity][row] = st;
    }

    // Sum of `mass` over the row's entries, and the entry in which a running sum in id order first exceeds
    // (U * sum) >> 24. found(id) runs in one lane of the cluster; returns the sum. slot: of xc.u64, one per call.
    // When it returns, other warps may still add up lc.red_a, lc.red_b and lc.peer: a barrier before these are written again.
    auto draw = [&](int slot, unsigned U, auto mass, auto found) -> u128 {
        Limbs s = {0ull, 0ull};
        for (int e0 = 0; e0 < n_e[0]; e0 += 32) s.add(mass(e0 + lane));
        s = warp_sum(s);
        __syncthreads();                               // (an earlier user of these is done)
        if (lane == 0) { lc.red_a[warp] = s.lo; lc.red_b[warp] = s.hi; }
        __syncthreads();
        if (warp < 2) {
            const unsigned long long t = warp_sum64(lane < NWARP ? (warp ? lc.red_b : lc.red_a)[lane] : 0ull);
            if (lane == 0) xc.u64[slot + warp] = t;
        }
        csync();                                                                      // ---- exchange: masses
        if (warp < 2 && lane < MAXC) lc.peer[warp][lane] = lane < C ? ld_peer_u64(&xc.u64[slot + warp], (uint32_t)lane) : 0ull;
        __syncthreads();
        u128 total = 0, run = 0;
#pragma unroll
        for (int r = 0; r < MAXC; ++r) {
            const u128 t = ((u128)lc.peer[1][r] << 40) + lc.peer[0][r];
            if (r < rank) run += t;
            total += t;
        }
        for (int i = 0; i < warp; ++i) run += ((u128)lc.red_b[i] << 40) + lc.red_a[i];
        const u128 target = ((u128)U * total) >> 24;
        if (total != 0 && run <= target && target < run + s.value()) {               // (one warp of the cluster)
            for (int e0 = 0; e0 < n_e[0]; e0 += 32) {
                Limbs r = {0ull, 0ull};
                r.add(mass(e0 + lane));
                const Limbs inc = warp_scan_inclusive(r, lane);
                const unsigned hit = __ballot_sync(FULLM, run + inc.value() > target);
                if (hit) {
                    if (lane == __ffs(hit) - 1) found(entry_id(e0 + lane));
                    break;
                }
                Limbs tot;
                tot.lo = __shfl_sync(FULLM, inc.lo, 31);
                tot.hi = __shfl_sync(FULLM, inc.hi, 31);
                run += tot.value();
            }
        }
        return total;
    };

    // ---- Algorithm 1 on (p, q, X) -----------------------------------------------------------------------------------
    // row_y: the row's output; row_y_indep: what becomes of it if the row stays in the window
    const bool indep = mrs && redraw_independent(p, b, pos, w.t);
    const bool race = p.mode == SCD_MODE_SCD_GS;
    int *const redraft = indep || race ? nullptr : p.row_y_indep + row;
    const bool first = rank == 0 && tid == 0;
    if (mrs) {
        const unsigned WpX = x_in ? weight_of(xX, m[0], tau[0], theta[0]) : 0u;
        const unsigned WqX = !x_in ? 0u : rawq ? weight_of(div ? __fdiv_rn(xq_raw, p.temperature) : xq_raw, m[1], tau[1], theta[1])
                                  : fresh ? 1u : __float_as_uint(xq_raw);
        const unsigned Ua = noise_u24(p.seed, NOISE_ACCEPT, (unsigned)b, pos, w.t, 0);
        // u <= min(1, p(X)/q(X)) with u = (Ua+1)/2^24  <=>  (Ua+1) Wq[X] Zp <= Wp[X] Zq 2^24;
        // a draft without mass under p is rejected
        const u128 lhs = (u128)(Ua + 1u) * WqX * Zp;
        const u128 rhs = ((u128)WpX * Zq) << 24;
        const bool accept = WpX != 0u && lhs <= rhs;
        if (first) p.accept_flags[row] = accept ? 1 : 0;
        bool keep_x = accept;
        if (!accept) {
            // Y ~ norm(max(0, p - q)). The draft's weights of the listed ids first: four gathers in flight, into the draft
            // row's list, which is done with (one at a time, and again in the walk, they were 10 to 15 us of a row)
            auto weight_q = [&](int v) -> unsigned {
                return rawq ? weight_of(load_q(v), m[1], tau[1], theta[1]) : fresh ? 1u : __float_as_uint(qr[v]);
            };
            if (!whole[0] && !fresh) {
                __syncwarp();
                for (int e0 = lane; e0 < n_e[0]; e0 += 128) {
                    float t[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) t[i] = e0 + 32 * i < n_e[0] ? qr[list_p[e0 + 32 * i].y] : 0.f;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (rawq && div) t[i] = __fdiv_rn(t[i], p.temperature);
                        if (e0 + 32 * i < n_e[0]) list_q[e0 + 32 * i] = rawq ? weight_of(t[i], m[1], tau[1], theta[1]) : __float_as_uint(t[i]);
                    }
                }
                __syncwarp();
            }
            const unsigned Ur = noise_u24(p.seed, NOISE_RESIDUAL, (unsigned)b, pos, w.t, 0);
            const u128 total = draw(4, Ur, [&](int e) -> u128 {
                const unsigned wp = weight_p(e);
                if (wp == 0u) return (u128)0;
                return residual_of(wp, fresh ? 1u : whole[0] ? weight_q(wbase + e) : list_q[e], Zp, Zq);
            }, [&](int y) {
                p.row_y[row] = y;
                if (redraft) *redraft = y;
            });
            keep_x = total == 0;
        }
        if (keep_x && first) {
            p.row_y[row] = X;
            if (redraft) *redraft = X;
        }
    }
    // ---- an independent draw from p: the token of vanilla AR, the redraft of Algorithm 2 ------------------------------
    if (indep || !mrs) {
        const unsigned Ui = noise_u24(p.seed, NOISE_INDEP, (unsigned)b, pos, mrs ? w.t : 0u, 0);
        int *const dst = mrs ? p.row_y_indep + row : p.row_y + row;
        // draw() for plain weights, whose sums take 64 bits (an autoregressive step of two layers: 102.5 us with 128, 101.6 so)
        unsigned long long s = 0, run = 0, total = 0;
        for (int e0 = 0; e0 < n_e[0]; e0 += 32) s += weight_p(e0 + lane);
        s = warp_sum64(s);
        __syncthreads();                               // (an earlier user of these is done)
        if (lane == 0) lc.red_a[warp] = s;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long t = warp_sum64(lane < NWARP ? lc.red_a[lane] : 0ull);
            if (lane == 0) xc.u64[6] = t;
        }
        csync();                                                                      // ---- exchange: masses
        if (warp == 0 && lane < MAXC) lc.peer[0][lane] = lane < C ? ld_peer_u64(&xc.u64[6], (uint32_t)lane) : 0ull;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < MAXC; ++r) {
            if (r < rank) run += lc.peer[0][r];
            total += lc.peer[0][r];
        }
        for (int i = 0; i < warp; ++i) run += lc.red_a[i];
        const unsigned long long target = (unsigned long long)(((u128)Ui * total) >> 24);
        if (total != 0 && run <= target && target < run + s) {                       // (one warp of the cluster)
            for (int e0 = 0; e0 < n_e[0]; e0 += 32) {
                unsigned long long inc = weight_p(e0 + lane);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long t = __shfl_up_sync(FULLM, inc, o);
                    if (lane >= o) inc += t;
                }
                const unsigned hit = __ballot_sync(FULLM, run + inc > target);
                if (hit) {
                    if (lane == __ffs(hit) - 1) *dst = entry_id(e0 + lane);
                    break;
                }
                run += __shfl_sync(FULLM, inc, 31);
            }
        }
        if (first) {
            if (total == 0) *dst = lo;
            if (!mrs) p.accept_flags[row] = 1;
        }
    }
    // ---- Algorithm 7: the redraft is the Gumbel-max sample of p under this position's shared noise; the row that may enter
    // the window at position pos0 + L + k starts from the race under the uniform draft distribution --------------------
    if (race) {
        float best = INFINITY;
        auto ratio = [&](int e, unsigned wv) -> float {
            return __fdividef(neglog2_estimate(noise_u24(p.seed, NOISE_GUMBEL, (unsigned)b, pos, 0u, (unsigned)entry_id(e))), (float)wv);
        };
        for (int e = lane; e < n_e[0]; e += 32) {
            const unsigned wv = weight_p(e);
            if (wv != 0u) best = fminf(best, ratio(e, wv));
        }
        const long long posf = w.pos0 + L + k;
        int flo, fhi;
        allowed_range(p, posf, flo, fhi);
        unsigned long long fk = 0;
        for (int v = flo + rank * CT + tid; v < fhi; v += C * CT) fk = max(fk, fresh_key(p, b, posf, v));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fk = max(fk, __shfl_xor_sync(FULLM, fk, o));
        const float wbest = -warp_max(-best);
        __syncthreads();                               // (an earlier user of these is done: the draw of a rejected row)
        if (lane == 0) { lc.red_f[0][warp] = wbest; lc.red_a[warp] = fk; }
        __syncthreads();
        if (warp == 0) {
            const float t = -warp_max(lane < NWARP ? -lc.red_f[0][lane] : -INFINITY);
            unsigned long long f = lane < NWARP ? lc.red_a[lane] : 0ull;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(FULLM, f, o));
            if (lane == 0) { xc.f32[0] = t; xc.fresh = f; }
        }
        csync();                                                                      // ---- exchange: smallest estimate
        if (warp == 0) {
            const float t = -warp_max(lane < C ? -__uint_as_float(ld_peer_u32(&xc.f32[0], (uint32_t)lane)) : -INFINITY);
            if (lane == 0) lc.red_f[1][0] = t;
        }
        __syncthreads();
        // The integers T carry up to 2^-39 of truncation, 4e-5 of the smallest variate there is, and the estimate
        // errs by less than 2e-6: the winner's estimate is within RACE_SLACK of the smallest one.
        const float bound = lc.red_f[1][0] * (1.0f + RACE_SLACK);
        Racer mine = {0ull, 0u, -1};
        if (best <= bound) {
            for (int e = lane; e < n_e[0]; e += 32) {
                const unsigned wv = weight_p(e);
                if (wv == 0u || !(ratio(e, wv) <= bound)) continue;
                const int v = entry_id(e);
                const Racer r = {neglog2_q40(noise_u24(p.seed, NOISE_GUMBEL, (unsigned)b, pos, 0u, (unsigned)v)), wv, v};
                if (race_before(r, mine)) mine = r;
            }
        }
        __syncwarp();
        mine = warp_racer(mine);
        if (lane == 0) { lc.red_a[warp] = mine.T; lc.red_b[warp] = ((unsigned long long)mine.W << 32) | (unsigned)mine.v; }
        __syncthreads();
        if (warp == 0) {
            Racer r = {0ull, 0u, -1};
            if (lane < NWARP) { r.T = lc.red_a[lane]; r.W = (unsigned)(lc.red_b[lane] >> 32); r.v = (int)(unsigned)lc.red_b[lane]; }
            r = warp_racer(r);
            if (lane == 0) { xc.racer[0] = r.T; xc.racer[1] = ((unsigned long long)r.W << 32) | (unsigned)r.v; }
        }
        csync();                                                                      // ---- exchange: racers
        if (rank == 0 && warp == 0) {
            Racer r = {0ull, 0u, -1};
            unsigned long long f = 0;
            if (lane < C) {
                const unsigned long long wv = ld_peer_u64(&xc.racer[1], (uint32_t)lane);
                r.T = ld_peer_u64(&xc.racer[0], (uint32_t)lane);
                r.W = (unsigned)(wv >> 32);
                r.v = (int)(unsigned)wv;
                f = ld_peer_u64(&xc.fresh, (uint32_t)lane);
            }
            r = warp_racer(r);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) f = max(f, __shfl_xor_sync(FULLM, f, o));
            if (lane == 0) {
                p.row_y_indep[row] = r.v < 0 ? lo : r.v;
                p.row_y_indep[(size_t)p.B * L + row] = fresh_key_id(f);
            }
        }
    }
    csync();                                           // nobody leaves while a peer may still read its shared memory
}

// First rejection, commit, next window: one CTA per sequence, a thread per row.
__global__ void __launch_bounds__(256) commit_kernel(const VerifyParams p)
{
    __shared__ int redraft[256], entering_s[256], first_s;
    const int b = blockIdx.x, k = threadIdx.x, L = p.L;
    if (!p.n_known) pdl_wait();                        // (the verify grid starts before its inputs are there, so does this one)
    const WindowState w = load_state(p, b);
    if (k == 0) first_s = w.Lw;
    pdl_wait();                                        // the rows come from the grid in front
    pdl_trigger();                                     // (a caller's next call starts under the rest of this one)
    const size_t row = (size_t)b * L + k;
    const bool live = k < w.Lw;
    const int y = live ? __ldcg(&p.row_y[row]) : 0;
    const int flag = live ? __ldcg(&p.accept_flags[row]) : 1;
    entering_s[k] = p.mode == SCD_MODE_SCD_GS && live ? __ldcg(&p.row_y_indep[(size_t)p.B * L + row]) : 0;
    redraft[k] = live && p.mode != SCD_MODE_AR ? __ldcg(&p.row_y_indep[row]) : 0;
    __syncthreads();
    if (flag == 0) atomicMin(&first_s, k);
    __syncthreads();
    if (w.Lw == 0) {
        if (k == 0) p.n_commit[b] = 0;
        return;
    }
    const int a = min(first_s + 1, w.Lw);              // the rejected row's residual sample is committed
    if (k < L) {
        if (k < a && p.tokens) p.tokens[(size_t)b * p.token_stride + w.pos0 + k] = y;
        if (p.committed_ids) p.committed_ids[row] = k < a ? y : 0;
        if (p.mode != SCD_MODE_AR) {
            const int src = k + a;
            p.draft_out[row] = src < w.Lw ? redraft[src]
                             : p.mode == SCD_MODE_SCD_GS && src >= L ? entering_s[src - L]
                                                                     : fresh_draft(p, b, w.pos0 + src, w.t + 1u);
        }
    }
    if (k == 0) {
        p.n_commit[b] = a;
        if (p.n_known) {
            p.n_known[b] = (int)w.pos0 + a;
            p.iter[b] = w.t + 1u;
            p.shift[b] = a;
            p.prev_lw[b] = w.Lw;
            // this iteration completed the sequence (it was live: Lw > 0): the last of the batch raises the flag
            if (p.finished && (int)w.pos0 + a >= p.n_total[b] && atomicAdd(&p.finished[0], 1) == p.B - 1) p.finished[1] = 1;
        }
        if (p.dev_stats) {
            atomicMax(&p.dev_stats->forwards, (unsigned long long)w.t + 1ull);   // iterations in which a sequence was live
            atomicAdd(&p.dev_stats->committed, (unsigned long long)a);
            atomicAdd(&p.dev_stats->accept_hist[a], 1ull);
        }
    }
}

// Cluster size and ids per warp for rows of at most n ids. One CTA per SM while that leaves a warp at most 256 ids
// (then they stay in registers), else two: a grid of one wave.
bool choose_cluster(const VerifyParams &p, int sm_count, int *C_out, int *ids_out)
{
    const int n = p.allowed_hi - p.allowed_lo + (p.allowed_lo & 3), rows = p.L * p.B;
    auto ids = [&](int C) { return (std::max(n, 4) + C * NWARP - 1) / (C * NWARP); };
    int C = 1;
    while (C < MAXC && ids(C) > 128 && (rows * C * 2 <= sm_count || (rows * C * 2 <= 2 * sm_count && ids(C) > 256))) C *= 2;
    while (C < MAXC && ids(C) > 256 * MAXG) C *= 2;
    *C_out = C;
    *ids_out = ids(C);
    return ids(C) <= 256 * MAXG;
}

template <class K, class... A>
cudaError_t launch_ex(K kernel, dim3 grid, int threads, size_t smem, int C, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (C > 0) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = (unsigned)C;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

bool verify_rows_supported(const VerifyParams &p)
{
    int C, ids;
    return choose_cluster(p, 148, &C, &ids);
}

int launch_verify_rows(const VerifyParams &p, cudaStream_t stream)
{
    auto lists = [](int wcap) { return NWARP * wcap * 12; };         // values and ids of one row, values of the other
    int dev = 0, sms = 148;
    int rc = current_device(&dev);
    if (rc != SCD_OK) return rc;
    static int sm_count[DeviceOnce::kSlots];
    static DeviceOnce once;
    rc = once.run(dev, [&]() -> int {
        SCD_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (dev >= 0 && dev < DeviceOnce::kSlots) sm_count[dev] = sms;
        auto opt_in = [&](auto kernel, int wcap) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lists(wcap)); };
        SCD_CUDA_TRY(opt_in(verify_rows_kernel<1, true, false>, 128));
        SCD_CUDA_TRY(opt_in(verify_rows_kernel<1, true, true>, 128));
        SCD_CUDA_TRY(opt_in(verify_rows_kernel<2, true, false>, 256));
        SCD_CUDA_TRY(opt_in(verify_rows_kernel<2, true, true>, 256));
        SCD_CUDA_TRY(opt_in(verify_rows_kernel<2, false, false>, WCAP_LONG));
        SCD_CUDA_TRY(opt_in(verify_rows_kernel<2, false, true>, WCAP_LONG));
        return SCD_OK;
    });
    if (rc != SCD_OK) return rc;
    if (dev >= 0 && dev < DeviceOnce::kSlots) sms = sm_count[dev];
    int C = 1, ids = 1;
    SCD_REQUIRE(choose_cluster(p, sms, &C, &ids), SCD_ERR_SHAPE, "verify: rows of %d ids do not fit a cluster", p.allowed_hi - p.allowed_lo);
    // Always a programmatic launch: the kernel waits before it reads what the one in front may have written. Stand-alone
    // calls one after the other otherwise paid a full launch each (1 x 32 rows of 16384 ids: 26.6 us a call, 24.3 so,
    // 4 us less on the host included; Gumbel, 2 x 32: 39.5 and 36.6).
    const dim3 grid((unsigned)(p.L * C), (unsigned)p.B, 1);
    auto launch = [&](auto kernel, int wcap, int range) { return launch_ex(kernel, grid, CT, (size_t)lists(wcap), C, stream, p, C, range); };
    auto pick = [&](auto with_top_p) {
        constexpr bool TOP_P = decltype(with_top_p)::value;
        return ids <= 128 ? launch(verify_rows_kernel<1, true, TOP_P>, 128, 0)
             : ids <= 256 ? launch(verify_rows_kernel<2, true, TOP_P>, 256, 0)
                          : launch(verify_rows_kernel<2, false, TOP_P>, WCAP_LONG, (ids + 31) / 32 * 32);
    };
    SCD_CUDA_TRY(p.top_p24 ? pick(std::true_type{}) : pick(std::false_type{}));
    return SCD_OK;
}

int launch_commit(const VerifyParams &p, cudaStream_t stream)
{
    SCD_CUDA_TRY(launch_ex(commit_kernel, dim3((unsigned)p.B, 1, 1), (p.L + 31) / 32 * 32, 0, 0, stream, p));
    return SCD_OK;
}

}  // namespace scd
