// GEMM of a forward with more than 128 rows (prefill chunks, large batches; up to 256 rows only where choose_shape in
// gemm_tcgen05.cu finds it faster): y[m, n] = sum_k x[m, k] * w[n, k],
// x in one or two bf16 planes, fp32 accumulation in tensor memory, output operations fused.
//
// Such a GEMM is bound by the tensor cores (two planes: 2 x 2 flop per weight and row), and next by the copies
// from L2 into shared memory. A pair of CTAs (cta_group::2, the two SMs of a TPC) therefore works on one tile of
// 256 x rows by 256 weight rows: x on the UMMA M axis (128 rows per CTA), weights on N (each CTA holds 128 of
// them, the tensor core reads both halves), and a K block of 64 weights is multiplied with BOTH planes of x into
// the same accumulator: 48 KB copied per CTA for 1024 cycles of MMA.
//   warps 0, 6, 7 : TMA producers of the weights, of x and of x's remainder plane (one lane each, in each CTA),
//               ring of 4 slots of 48 KB (one plane: 6 of 32 KB). One lane for all of them took 1135 cycles per K
//               block, more than its MMAs: a lane needs some 250 cycles per copy that it issues.
//   warp 1    : tensor memory; in the leader CTA one lane issues the MMAs for both CTAs
//   warps 2-5 : epilogue, one thread per x row (tensor-memory lane): rows leave as runs of 32 columns
// Two accumulators of 256 columns: the epilogue of a tile runs under the MMAs of the next.
//
// The grid is one CTA per SM and the K blocks of all tiles are dealt out evenly: pair p takes the units
// [p U / P, (p + 1) U / P) of the U = tiles x k_blocks, whatever tile borders they cross, so that no last wave is
// half empty. A tile that is cut is finished from partial tiles in global memory (they stay in L2): every
// contributor stores its part and counts itself in; a pair whose LAST segment the tile is waits for the others
// and adds up its share of the columns, its own part first and the others' in order - the result does not depend on
// scheduling. A pair that has work left never waits, and none waits for long: with the kernels of other streams on the
// device the pairs that are waited for may have no SM while these hold them. One that has waited PATIENCE polls stores
// its share too, says so and leaves; who is counted in last adds up the shares left to it, in the same order.
// Every other wait is bounded; on expiry the error word is raised, the roles run out and the outputs are not written.
//
// Measured on a B200 (before: 256 rows at a time through the weight-streaming kernel, or an earlier step of this one):
// 2560 x 12288 x 3072, two planes: 247 us with one producer lane, 207 with one per operand;
// 2560 x 9216 x 3072, one plane: 179, 111; 256 x 22016 x 4096 SwiGLU: 112 with parts loaded through registers, 65 by
// bulk copies. 2560 tokens of prefill through 28 layers of 3072: 73 ms by passes of 128 rows, 32 ms.
#include <algorithm>
#include <cstring>

#include "gemm_pair.cuh"
#include "model.cuh"
#include "ptx.cuh"

namespace scd {

namespace {

constexpr int PAIR_THREADS = 256;
constexpr int BK = 64;
constexpr int MAX_PAIR_STAGES = 6;
constexpr uint32_t TILE_BYTES = 128 * BK * 2;                        // 128 rows of one operand, one K block
constexpr size_t PAIR_SMEM = 227 * 1024 - 8192;                      // all of an SM: no other kernel's CTA beside it
constexpr int PAIR_UNITS = PAIR_COLS / PAIR_UNIT;                    // 8 runs of 32 accumulator columns
constexpr size_t RUN_FLOATS = (size_t)128 * PAIR_UNIT;               // 32 columns of the CTA's 128 rows: [column / 8][row][8]
constexpr size_t SLOT_FLOATS = PAIR_UNITS * RUN_FLOATS;              // one CTA's part of a cut tile
constexpr int RED_SLOTS = 12;                                        // runs of other pairs' parts in flight (in the ring's memory)
constexpr unsigned PATIENCE = 1u << 11;                              // polls for the other parts of a tile: a millisecond or two

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void arrive_cluster(uint32_t addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Copies of the pair: into this CTA's shared memory, counted on the leader's barrier.
__device__ __forceinline__ void tma_pair_2d(const CUtensorMap *map, uint32_t bar, void *dst, int x, int y, uint64_t pol)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
                 " [%0], [%1, {%3, %4}], [%2], %5;"
                 ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y), "l"(pol) : "memory");
}
__device__ __forceinline__ void tma_pair_3d(const CUtensorMap *map, uint32_t bar, void *dst, int x, int y, int z, uint64_t pol)
{
    asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
                 " [%0], [%1, {%3, %4, %5}], [%2], %6;"
                 ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(pol) : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
}
// arrives on the barrier at this offset in both CTAs once the MMAs issued so far are complete
__device__ __forceinline__ void commit_pair(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}

// 32 consecutive floats of a row, through L2 (other SMs write them)
__device__ __forceinline__ void ld32(const float *src, float *v, bool vec)
{
    if (vec) {
#pragma unroll
        for (int j = 0; j < 32; j += 8)
            asm volatile("ld.relaxed.gpu.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=f"(v[j]), "=f"(v[j + 1]), "=f"(v[j + 2]), "=f"(v[j + 3]), "=f"(v[j + 4]), "=f"(v[j + 5]),
                           "=f"(v[j + 6]), "=f"(v[j + 7]) : "l"(src + j) : "memory");
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __ldcg(src + j);
    }
}
__device__ __forceinline__ void st32(float *dst, const float *v, int n, bool vec)
{
    if (vec && n == 32) {
#pragma unroll
        for (int j = 0; j < 32; j += 8)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                         ::"l"(dst + j), "f"(v[j]), "f"(v[j + 1]), "f"(v[j + 2]), "f"(v[j + 3]), "f"(v[j + 4]), "f"(v[j + 5]),
                           "f"(v[j + 6]), "f"(v[j + 7]) : "memory");
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) if (j < n) dst[j] = v[j];
    }
}
// a run of a part, 8 columns at a time: a warp writes 1 KB in one piece
__device__ __forceinline__ void st_run(float *run, int row, const float *v)
{
#pragma unroll
    for (int j = 0; j < 32; j += 8)
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(run + (size_t)(j >> 3) * 1024 + row * 8), "f"(v[j]), "f"(v[j + 1]), "f"(v[j + 2]), "f"(v[j + 3]),
                       "f"(v[j + 4]), "f"(v[j + 5]), "f"(v[j + 6]), "f"(v[j + 7]) : "memory");
}
__device__ __forceinline__ void add_run_global(const float *run, int row, float *v)
{
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
        float t[8];
        asm volatile("ld.relaxed.gpu.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(t[0]), "=f"(t[1]), "=f"(t[2]), "=f"(t[3]), "=f"(t[4]), "=f"(t[5]), "=f"(t[6]), "=f"(t[7])
                     : "l"(run + (size_t)(j >> 3) * 1024 + row * 8) : "memory");
#pragma unroll
        for (int i = 0; i < 8; ++i) v[j + i] += t[i];
    }
}
__device__ __forceinline__ void add_run(const float *run, int row, float *v)   // (in shared memory)
{
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        const float4 t = *(const float4 *)(run + (j >> 3) * 1024 + row * 8 + (j & 4));
        v[j] += t.x; v[j + 1] += t.y; v[j + 2] += t.z; v[j + 3] += t.w;
    }
}
__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
    return *(const uint32_t *)&t;
}
__device__ __forceinline__ float rest(float x) { return x - __bfloat162float(__float2bfloat16_rn(x)); }
// v as two bf16 planes: hi = bf16(v), lo = bf16(v - hi)
__device__ __forceinline__ void st32_planes(__nv_bfloat16 *dst, long long plane, const float *v, int n)
{
    if (n == 32) {                                                   // (row pitches are multiples of 64, runs of 32: 32-byte aligned)
#pragma unroll
        for (int pl = 0; pl < 2; ++pl) {
#pragma unroll
            for (int j = 0; j < 32; j += 16) {
                uint32_t w[8];
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    w[k] = pl ? pack2(rest(v[j + 2 * k]), rest(v[j + 2 * k + 1])) : pack2(v[j + 2 * k], v[j + 2 * k + 1]);
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                             ::"l"(dst + pl * plane + j), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                             : "memory");
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (j < n) { dst[j] = __float2bfloat16_rn(v[j]); dst[plane + j] = __float2bfloat16_rn(rest(v[j])); }
    }
}

// One pair's walk over its units: the segment of tile `tile` from K block k0 to k1 (exclusive).
struct Walk {
    long long u, end;
    int kb, tile, k0, k1;
    __device__ Walk(const PairParams &p, int pair)
    {
        const long long U = (long long)p.w_tiles * p.x_tiles * p.k_blocks;
        kb = p.k_blocks;
        u = U * pair / p.pairs;
        end = U * (pair + 1) / p.pairs;
    }
    __device__ bool next()
    {
        if (u >= end) return false;
        tile = (int)(u / kb);
        k0 = (int)(u - (long long)tile * kb);
        k1 = (int)min((long long)kb, k0 + (end - u));
        u += k1 - k0;
        return true;
    }
    __device__ bool last() const { return u >= end; }
};
__device__ __forceinline__ int pair_of(const PairParams &p, long long unit)   // the pair whose range holds `unit`
{
    const long long U = (long long)p.w_tiles * p.x_tiles * p.k_blocks;
    return (int)(((unit + 1) * p.pairs - 1) / U);
}

__global__ void __launch_bounds__(PAIR_THREADS, 1) gemm_pair_kernel(const __grid_constant__ PairParams p)
{
    extern __shared__ __align__(1024) uint8_t ring[];
    __shared__ uint64_t full_bar[MAX_PAIR_STAGES], empty_bar[MAX_PAIR_STAGES], tfull[2], tempty[2], red_bar[RED_SLOTS];
    __shared__ float scale_s[PAIR_MAX_X_TILES][128];                 // 1 / rms of this CTA's rows of each x tile
    __shared__ uint32_t tmem_base_s;
    __shared__ unsigned ticket_s;
    __shared__ volatile int failed;

    if (p.skip && *p.skip) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1;
    if (p.stamp && tid == 0 && blockIdx.x < STAMP_CTAS) p.stamp[blockIdx.x] = global_timer_ns();
    if (tid == 0) {
        if ((smem_u32(ring) & 1023u) != 0u) atomicExch(p.err, 6);
        for (int s = 0; s < MAX_PAIR_STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], 8); }
        for (int b = 0; b < RED_SLOTS; ++b) mbar_init(&red_bar[b], 1);
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();                                              // both CTAs: barriers ready, tensor memory held
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    pdl_trigger();                                                   // (only now: the kernel behind allocates tensor memory too)
    const uint32_t tmem = tmem_base_s;

    const uint32_t stage_bytes = TILE_BYTES * (1u + (uint32_t)p.planes);
    const int stages = p.planes == 2 ? 4 : 6;
    const bool swiglu = p.epi == PAIR_EPI_SWIGLU;
    auto wait = [&](uint64_t *bar, unsigned parity, int code) -> bool {
        const uint32_t a = smem_u32(bar);
        for (unsigned i = 0; i < SPIN_LIMIT; ++i) {
            unsigned ok;
            asm volatile("{\n\t.reg .pred p;\n\t"
                         "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(a), "r"(parity) : "memory");
            if (ok) return true;
            if ((i & 1023u) == 1023u && failed) return false;
        }
        atomicExch(p.err, code);
        failed = 1;
        return false;
    };
    auto all_epilogue = [](bool mine) -> bool {                       // barrier of the four epilogue warps, with the AND of `mine`
        unsigned r;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                     : "=r"(r) : "r"(mine ? 1u : 0u) : "memory");
        return r != 0;
    };
    auto segment_of = [&](int wt) { int s = 0; while (s + 1 < p.n_seg && wt >= p.seg_tile0[s + 1]) ++s; return s; };

    const bool w_lane = warp == 0 && lane == 0, x_lane = lane == 0 && (warp == 6 || (warp == 7 && p.planes == 2));
    if (w_lane || x_lane) {
        // ---------------- TMA producers ----------------
        // The full barrier of a slot takes one arrival, the leader's weight lane with the bytes of all copies; copies
        // of the other lanes may land before it.
        uint64_t pol_w, pol_x;
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_w));
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_x));
        if (p.x_tiles > 1) pol_w = pol_x;                            // the tiles of the other x rows read it again
        const uint32_t full0 = map_rank(smem_u32(&full_bar[0]), 0);
        const int plane = warp == 7 ? 1 : 0;
        uint8_t *dst0 = ring + (w_lane ? 0u : TILE_BYTES * (1u + (uint32_t)plane));
        if (x_lane) pdl_wait();                                      // x is written by the kernel in front; the weights by none
        Walk w(p, pair);
        int s = 0;
        unsigned round = 0;
        bool ok = true;
        while (ok && w.next()) {
            const int wt = w.tile / p.x_tiles;
            const int seg = swiglu ? (int)rank : segment_of(wt);
            const CUtensorMap *map = w_lane ? &p.tmap_w[seg] : &p.tmap_x;
            const int row = !w_lane ? (w.tile - wt * p.x_tiles) * PAIR_ROWS + (int)rank * 128
                            : swiglu ? p.seg_row0[0] + wt * 128
                                     : p.seg_row0[seg] + (wt - p.seg_tile0[seg]) * PAIR_COLS + (int)rank * 128;
            for (int k = w.k0; k < w.k1; ++k) {
                if (round > 0 && !wait(&empty_bar[s], (round & 1u) ^ 1u, 1)) { ok = false; break; }
                uint8_t *dst = dst0 + (size_t)s * stage_bytes;
                if (w_lane) {
                    if (rank == 0) mbar_expect_tx(&full_bar[s], 2 * stage_bytes);
                    tma_pair_2d(map, full0 + 8u * s, dst, k * BK, row, pol_w);
                } else {
                    tma_pair_3d(map, full0 + 8u * s, dst, k * BK, row, plane, pol_x);
                }
                if (++s == stages) { s = 0; ++round; }
            }
        }
        if (!ok) {                                                   // give copies in flight time to land before the CTA exits
            const unsigned long long t0 = global_timer_ns();
            while (global_timer_ns() - t0 < 1000000ull) { }
        }
    } else if (warp == 1 && lane == 0 && rank == 0) {
        // ---------------- MMA issuer (both CTAs' tensor cores) ----------------
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(PAIR_COLS >> 3) << 17) | ((uint32_t)(PAIR_ROWS >> 4) << 24);
        Walk w(p, pair);
        int s = 0, seg_i = 0;
        unsigned round = 0;
        bool ok = true;
        for (; ok && w.next(); ++seg_i) {
            const int b = seg_i & 1;
            if (seg_i >= 2) ok = wait(&tempty[b], (unsigned)((seg_i >> 1) - 1) & 1u, 3);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc = tmem + (uint32_t)b * PAIR_COLS;
            for (int k = w.k0; ok && k < w.k1; ++k) {
                ok = wait(&full_bar[s], round & 1u, 2);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = smem_u32(ring + (size_t)s * stage_bytes);
                const uint64_t db = umma_desc(base), da = umma_desc(base + TILE_BYTES), da2 = umma_desc(base + 2 * TILE_BYTES);
#pragma unroll
                for (int j = 0; j < BK / 16; ++j) umma_pair(acc, da + j * 2, db + j * 2, idesc, (k > w.k0 || j > 0) ? 1u : 0u);
                if (p.planes == 2) {
#pragma unroll
                    for (int j = 0; j < BK / 16; ++j) umma_pair(acc, da2 + j * 2, db + j * 2, idesc, 1u);
                }
                commit_pair(&empty_bar[s]);
                if (++s == stages) { s = 0; ++round; }
            }
            commit_pair(&tfull[b]);
        }
    } else if (warp >= 2 && warp < 6) {
        // ---------------- epilogue: thread = x row ----------------
        const int quarter = warp & 3, row = quarter * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const uint32_t tempty_leader[2] = {map_rank(smem_u32(&tempty[0]), 0), map_rank(smem_u32(&tempty[1]), 0)};
        pdl_wait();                                                  // statistics, residual rows and outputs belong to kernels in front
        Walk w(p, pair);
        const int limit_units = swiglu ? PAIR_UNITS / 2 : PAIR_UNITS;
        if (p.ss_in) {
            // once for all tiles, under the first tile's main loop; 16 loads in flight (tile by tile and one after the
            // other they cost 20 us and more per tile: 264 against 111 us for 2560 x 9216 x 3072)
            const int t0 = (int)(w.u / w.kb), n_t = min(p.x_tiles, (int)((w.end - 1) / w.kb) - t0 + 1);
            for (int i = 0; i < n_t; ++i) {
                const int xt = (t0 + i) % p.x_tiles, m = min(xt * PAIR_ROWS + (int)rank * 128 + row, p.rows - 1);
                const float *src = p.ss_in + m;
                float ss = 0.f;
                for (int part = 0; part < p.ss_parts; part += 16) {
                    float t[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) t[j] = part + j < p.ss_parts ? __ldcg(src + (size_t)(part + j) * p.ss_stride) : 0.f;
#pragma unroll
                    for (int j = 0; j < 16; ++j) ss += t[j];
                }
                scale_s[xt][row] = rsqrtf(ss * p.inv_k + p.eps);     // (read by this thread only)
            }
        }
        const bool vec_out = (p.ldo & 7) == 0 && ((uintptr_t)p.out & 31) == 0;
        for (int seg_i = 0; w.next(); ++seg_i) {
            const int b = seg_i & 1;
            const int wt = w.tile / p.x_tiles, m = (w.tile % p.x_tiles) * PAIR_ROWS + (int)rank * 128 + row;
            const bool live = m < p.rows;
            const int seg = swiglu ? 0 : segment_of(wt);
            const int wrow0 = swiglu ? p.seg_row0[0] + wt * 128 : p.seg_row0[seg] + (wt - p.seg_tile0[seg]) * PAIR_COLS;
            const int n_cols = p.seg_end[seg] - wrow0;               // output columns from the tile's first one on
            const int col0 = p.seg_col0[seg] + wrow0;
            const float scale = p.ss_in ? scale_s[w.tile % p.x_tiles][row] : 1.0f;
            // the residual rows that columns [32 u, 32 u + 32) of the tile are added to
            auto load_resid = [&](int u, float *g) {
                const int n = min(32, n_cols - 32 * u);
                const float *src = (const float *)p.out + (size_t)m * p.ldo + col0 + 32 * u;
                if (live && n == 32 && vec_out) { ld32(src, g, true); return; }
#pragma unroll
                for (int j = 0; j < 32; ++j) g[j] = live && j < n ? __ldcg(src + j) : 0.f;
            };
            // the output operation on these columns (SwiGLU: features; g = gate, v = up; residual: g = the rows)
            auto finish = [&](int u, float *v, float *g) {
                const int n = min(32, n_cols - 32 * u);
                if (!live || n <= 0) return;
                const int col = col0 + 32 * u;
                if (swiglu) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float gj = g[j] * scale, uj = v[j] * scale;
                        // (the fast division: 2 ulp, right up to 2^128. What is stored has two bf16 planes: rms error against
                        // 64 bits 2.450e-6, 2.450e-6 with an IEEE division too, which costs 256 rows x 30 layers 3 %)
                        v[j] = __fdividef(gj, 1.0f + expf(-gj)) * uj;
                    }
                    st32_planes((__nv_bfloat16 *)p.out + (size_t)m * p.ldo + col, p.out_plane, v, n);
                    return;
                }
                float *dst = (float *)p.out + (size_t)m * p.ldo + col;
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] *= scale;
                if (p.epi == PAIR_EPI_RESID) {
                    float sq = 0.f;
#pragma unroll
                    for (int j = 0; j < 32; ++j) { v[j] = j < n ? v[j] + g[j] : 0.f; sq += v[j] * v[j]; }
                    st32(dst, v, n, vec_out && (col & 7) == 0);
                    if (p.xg_out) {
                        const __nv_bfloat16 *gn = p.gain_next + col;
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] *= j < n ? __bfloat162float(gn[j]) : 0.f;
                        st32_planes(p.xg_out + (size_t)m * p.ldo + col, p.out_plane, v, n);
                        p.ss_out[(size_t)(col >> 5) * p.ss_stride + m] = sq;
                    }
                } else {
                    st32(dst, v, n, vec_out && (col & 7) == 0);
                }
            };
            const bool ok = wait(&tfull[b], (unsigned)(seg_i >> 1) & 1u, 3);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            int errw = 0;
            if (lane == 0) errw = *(volatile int *)p.err;
            errw = __shfl_sync(0xffffffffu, errw, 0);
            const bool healthy = __all_sync(0xffffffffu, ok) && errw == 0 && !failed;
            if (!all_epilogue(healthy)) { failed = 1; break; }       // (the same decision in all four warps: they meet at barriers)
            const uint32_t acc = tmem + lane_addr + (uint32_t)b * PAIR_COLS;
            const bool whole = w.k0 == 0 && w.k1 == w.kb;
            const int q0 = whole ? pair : pair_of(p, (long long)w.tile * w.kb);
            float v[32], g[32];
            if (whole) {
#pragma unroll 1
                for (int u = 0; u < limit_units; ++u) {
                    if (32 * u >= n_cols) break;                     // (warp-uniform)
                    if (p.epi == PAIR_EPI_RESID) load_resid(u, g);
                    if (swiglu) { tmem_ld32(acc + 32u * u, g); tmem_ld32(acc + 128u + 32u * u, v); }
                    else tmem_ld32(acc + 32u * u, v);
                    finish(u, v, g);
                }
            }
            if (whole) {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) arrive_cluster(tempty_leader[b]);     // the accumulator may be overwritten
                continue;
            }
            // ---- a cut tile: this part goes to memory and is counted in - but for the columns that this pair itself
            // adds up, which it does if nothing is left for it to do ----
            const long long U = (long long)p.w_tiles * p.x_tiles * p.k_blocks;
            const long long tile_u0 = (long long)w.tile * w.kb, tile_u1 = tile_u0 + w.kb;
            const int q1 = pair_of(p, tile_u1 - 1), n_parts = q1 - q0 + 1;
            // contributors that end on this tile, as many as there are runs of columns to add up
            const int n_red = min(limit_units, U * (q1 + 1) / p.pairs == tile_u1 ? n_parts : n_parts - 1), me = pair - q0;
            const bool reduces = w.last() && me < n_red;
            auto part_of = [&](int q) -> const float * {             // (its second slot if it had a tile in front of this one)
                return p.scratch + ((size_t)(q * 2 + (U * q / p.pairs >= tile_u0 ? 0 : 1)) * 2 + rank) * SLOT_FLOATS;
            };
            float *slot = p.scratch + ((size_t)(pair * 2 + (seg_i == 0 ? 0 : 1)) * 2 + rank) * SLOT_FLOATS;
#pragma unroll 1
            for (int u = 0; u < PAIR_UNITS; ++u) {
                if (reduces && (u % limit_units) % n_red == me) continue;
                tmem_ld32(acc + 32u * u, v);
                st_run(slot + u * RUN_FLOATS, row, v);
            }
            // counters of a tile: [0] parts that are there, from bit 16 on the shares that were left; [1] shares that are done
            unsigned *cnt = p.counters + (size_t)w.tile * 4 + rank * 2;
            auto count_in = [&](unsigned what) -> unsigned {         // (what was there before, in all four warps)
                __threadfence();
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (tid == 64) ticket_s = atomicAdd(cnt, what);
                asm volatile("bar.sync 1, 128;" ::: "memory");
                return ticket_s;
            };
            auto done = [&](unsigned shares) {                       // the last one clears the tile's counters for the next launch
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (tid == 64 && atomicAdd(cnt + 1, shares) + shares == (unsigned)n_red) { cnt[0] = 0u; cnt[1] = 0u; }
            };
            auto add_left = [&](unsigned left) {                     // shares that their pairs left to the last one to come
                __threadfence();
#pragma unroll 1
                for (int sh = 0; sh < n_red; ++sh) {
                    if (!(left >> sh & 1u)) continue;
                    auto sum_parts = [&](int u, float *sum) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) sum[j] = 0.f;
                        add_run_global(part_of(q0 + sh) + (size_t)u * RUN_FLOATS, row, sum);
#pragma unroll 1
                        for (int q = q0; q <= q1; ++q)
                            if (q != q0 + sh) add_run_global(part_of(q) + (size_t)u * RUN_FLOATS, row, sum);
                    };
#pragma unroll 1
                    for (int u = sh; u < limit_units; u += n_red) {
                        if (p.epi == PAIR_EPI_RESID) load_resid(u, g);
                        if (swiglu) sum_parts(u, g);
                        sum_parts(swiglu ? u + PAIR_UNITS / 2 : u, v);
                        finish(u, v, g);
                    }
                }
                done((unsigned)__popc(left));
            };
            const unsigned ticket = count_in(1u);
            const bool all_here = (ticket & 0xFFFFu) + 1u == (unsigned)n_parts;
            const unsigned left = all_here ? ticket >> 16 : 0u;
            if (!reduces) {
                if (lane == 0) arrive_cluster(tempty_leader[b]);
                if (left) add_left(left);
                continue;
            }
            if (!all_here) {
                unsigned seen = (unsigned)n_parts;
                if (tid == 64) {
                    seen = 0;
                    for (unsigned i = 0; i < PATIENCE && seen < (unsigned)n_parts; ++i) {
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(cnt) : "memory");
                        seen &= 0xFFFFu;
                        if ((i & 1023u) == 1023u && failed) break;
                    }
                }
                if (!all_epilogue(!failed)) break;
                if (!all_epilogue(seen == (unsigned)n_parts)) {
#pragma unroll 1
                    for (int u = me; u < PAIR_UNITS; ++u) {
                        if ((u % limit_units) % n_red != me) continue;
                        tmem_ld32(acc + 32u * u, v);
                        st_run(slot + u * RUN_FLOATS, row, v);
                    }
                    // (unless the last one has come meanwhile, and found nothing left to it)
                    if ((count_in(0x10000u << me) & 0xFFFFu) != (unsigned)n_parts) break;
                }
            }
            __threadfence();
            // The runs to add, in order: for each of this pair's runs of columns (SwiGLU: gate, then up) the parts of the
            // other contributors. They come by bulk copies into the ring, which this CTA's MMAs no longer need, twelve
            // at a time: with register loads, one or two in flight, a tile took 8 to 27 us.
            const int n_oth = n_parts - 1, per_unit = swiglu ? 2 * n_oth : n_oth;
            const int my_units = (limit_units - me + n_red - 1) / n_red, n_runs = my_units * per_unit;
            auto request = [&](int first) {
                asm volatile("fence.proxy.async;" ::: "memory");
                for (int r = first; r < min(n_runs, first + RED_SLOTS); ++r) {
                    const int k = r % per_unit, i = k % n_oth;
                    const int u = me + (r / per_unit) * n_red + (k >= n_oth ? PAIR_UNITS / 2 : 0);
                    const int q = q0 + i + (i >= me ? 1 : 0);
                    const float *src = part_of(q) + (size_t)u * RUN_FLOATS;
                    uint64_t *bar = &red_bar[r - first];
                    mbar_expect_tx(bar, (unsigned)(RUN_FLOATS * sizeof(float)));
                    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(smem_u32(ring + (size_t)(r - first) * RUN_FLOATS * sizeof(float))), "l"(src),
                                   "r"((unsigned)(RUN_FLOATS * sizeof(float))), "r"(smem_u32(bar)) : "memory");
                }
            };
            if (tid == 64 && n_runs > 0) request(0);
            int r = 0;
            unsigned red_parity = 0;
            bool good = true;
            auto add_parts = [&](float *sum) {
#pragma unroll 1
                for (int i = 0; i < n_oth; ++i, ++r) {
                    const int sl = r % RED_SLOTS;
                    if (r > 0 && sl == 0) {                          // the next twelve, once all threads have read these
                        asm volatile("bar.sync 1, 128;" ::: "memory");
                        if (tid == 64) request(r);
                        red_parity ^= 1u;
                    }
                    good = wait(&red_bar[sl], red_parity, 3) && good;
                    add_run((const float *)ring + (size_t)sl * RUN_FLOATS, row, sum);
                }
            };
#pragma unroll 1
            for (int u = me; u < limit_units; u += n_red) {
                if (p.epi == PAIR_EPI_RESID) load_resid(u, g);
                if (swiglu) { tmem_ld32(acc + 32u * u, g); add_parts(g); }
                tmem_ld32(acc + 32u * (swiglu ? u + PAIR_UNITS / 2 : u), v);
                add_parts(v);
                __syncwarp();
                if (good) finish(u, v, g);
            }
            done(1u);
            if (left) add_left(left);
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync_all();                                              // no MMA reads, no barrier arrives in a CTA that has left
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    if (p.stamp && tid == 0 && blockIdx.x < STAMP_CTAS) p.stamp[STAMP_CTAS + blockIdx.x] = global_timer_ns();
}

}  // namespace

size_t pair_scratch_bytes(int pairs) { return (size_t)pairs * 4 * SLOT_FLOATS * sizeof(float); }
size_t pair_counter_count(int w_tiles, int x_tiles) { return (size_t)w_tiles * x_tiles * 4; }

// The pairs of one cut tile wait for each other, for a while, so the grid never has more pairs than fit at once.
int pair_grid_limit(int *pairs)
{
    SCD_CUDA_TRY(cudaFuncSetAttribute(gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PAIR_SMEM));
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(PAIR_THREADS, 1, 1);
    cfg.dynamicSmemBytes = PAIR_SMEM;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    SCD_CUDA_TRY(cudaOccupancyMaxActiveClusters(pairs, gemm_pair_kernel, &cfg));
    SCD_REQUIRE(*pairs >= 1, SCD_ERR_CUDA, "the device holds no CTA pair of the GEMM");
    return SCD_OK;
}

int launch_gemm_pair(PairParams &p, int max_pairs, cudaStream_t st)
{
    // (a pair takes at least four K blocks: below that the parts of a tile cost more than they save)
    const long long units = (long long)p.w_tiles * p.x_tiles * p.k_blocks;
    p.pairs = (int)std::max(1ll, std::min((long long)max_pairs, units / 4));
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(2 * p.pairs), 1, 1);
    cfg.blockDim = dim3(PAIR_THREADS, 1, 1);
    cfg.dynamicSmemBytes = PAIR_SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = 2;
    attrs[1].val.clusterDim.y = 1;
    attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = 2;
    SCD_REQUIRE(p.x_tiles <= PAIR_MAX_X_TILES, SCD_ERR_SHAPE, "GEMM: %d rows, at most %d", p.rows, PAIR_MAX_X_TILES * PAIR_ROWS);
    SCD_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_pair_kernel, p));
    count_launches(1);
    return SCD_OK;
}

}  // namespace scd
