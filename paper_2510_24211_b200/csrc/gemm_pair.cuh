// Launch interface of the CTA-pair GEMM for forwards of more than 128 rows (gemm_pair.cu).
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace scd {

constexpr int PAIR_ROWS = 256;         // x rows of a tile (128 per CTA of the pair)
constexpr int PAIR_COLS = 256;         // weight rows of a tile (SwiGLU: 128 gate rows + 128 up rows)
constexpr int PAIR_UNIT = 32;          // output columns that one partial sum of squares covers
constexpr int PAIR_MAX_SEG = 3;
constexpr int PAIR_MAX_X_TILES = 10;   // 2560 rows

enum { PAIR_EPI_F32 = 0, PAIR_EPI_RESID = 1, PAIR_EPI_SWIGLU = 2 };

struct PairParams {
    CUtensorMap tmap_w[PAIR_MAX_SEG];  // weight segments, boxes of 128 rows; SwiGLU: [0] gate, [1] up
    CUtensorMap tmap_x;                // [planes][rows][K], box of 128 rows of one plane
    int seg_tile0[PAIR_MAX_SEG + 1];   // first weight tile of each segment
    int seg_row0[PAIR_MAX_SEG];        // weight row of the segment's first tile
    int seg_end[PAIR_MAX_SEG];         // end (exclusive) of the segment's rows in its weight matrix
    int seg_col0[PAIR_MAX_SEG];        // output column of row 0 of the segment's weight matrix
    int n_seg;
    int rows;                          // live x rows
    int x_tiles, w_tiles;
    int planes;                        // planes of x to multiply with (1 or 2)
    int k_blocks;                      // K / 64
    int pairs;                         // CTA pairs of the grid
    int epi;
    void *out;                         // fp32 [rows][ldo]; SwiGLU: bf16 hi plane [rows][ldo]
    int ldo;
    long long out_plane;               // elements from the hi plane to the lo plane (SwiGLU, xg_out)
    const float *ss_in;                // optional: [ss_parts][ss_stride] partial sums of squares of the x rows
    int ss_parts, ss_stride;
    float inv_k, eps;
    const __nv_bfloat16 *gain_next;    // RESID: norm input of the next GEMM
    __nv_bfloat16 *xg_out;
    float *ss_out;                     // [columns / 32][ss_stride]
    float *scratch;                    // partial tiles: pair_scratch_bytes() bytes
    unsigned *counters;                // zero between launches: pair_counter_count() words
    int *err;
    const int *skip;
    unsigned long long *stamp;
};

size_t pair_scratch_bytes(int pairs);
size_t pair_counter_count(int w_tiles, int x_tiles);
int pair_grid_limit(int *pairs);       // CTA pairs the current device holds at the same time
int launch_gemm_pair(PairParams &p, int max_pairs, cudaStream_t st);

}  // namespace scd
