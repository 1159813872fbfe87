// What the steps kernel of the delayed-update path (prune_lazy.cu) and its tensor-core update
// (prune_lazy_tc.cu) share: the packed operands of the update.
//
// P[l][g][a][row][64] (bfloat16): g the group of 32 steps (a block has one or two), a = 0: [U1 | U2],
// 1: [U3 | Z3], 2: [Z1 | Z2], each half of a row the 32 steps of one part of the pending vectors; a row is a
// position (zero from the last position to the next multiple of 128), and behind lazy_tc_rows_pad(d) rows a
// row index of W with its scaled pivot columns C in the place of U and zeros in the place of Z.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"

namespace ziplm {

constexpr int kPackSteps = 32;     // pending steps per group of packed operands
constexpr int kPackGroups = 2;     // groups a block may have
constexpr int kPackArrays = 3;     // per group
constexpr int kPackTile = 128;

inline int lazy_tc_rows_pad(int d) { return round_up_int(d, kPackTile); }
inline int lazy_tc_rows_tot(int d, int rp) { return lazy_tc_rows_pad(d) + round_up_int(rp, kPackTile); }

// size of the packed operands in floats (a row is 2 * kPackSteps bfloat16)
inline size_t lazy_tc_pack_floats(int L, int d, int rp) {
    return (size_t)L * kPackGroups * kPackArrays * lazy_tc_rows_tot(d, rp) * kPackSteps;
}

bool lazy_tc_make_map(CUtensorMap* m, const float* P, int L, int d, int rp);
bool lazy_tc_make_matrix_map(CUtensorMap* m, const float* M, int L, int d, int cols);

// The packed pending steps (`groups` groups of 32) applied to H^-1, Q and W^T with every position left in place.
ziplm_status run_lazy_update_aq_tc(const CUtensorMap& map, const CUtensorMap& map_a,
                                   const CUtensorMap& map_q, const CUtensorMap& map_w, int L, int groups, int n_pos,
                                   int d, int rp, float* A2, float* Q2, float* W2, int* counter,
                                   int* layer_status, unsigned slot_spin_limit, cudaStream_t st);

// The three bfloat16 parts of two values, each the nearest bfloat16 of what the earlier ones left (the
// remainders are exact).
__device__ __forceinline__ void split_bf16x3(float x, float y, __nv_bfloat162 (&p)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = __floats2bfloat162_rn(x, y);
        x -= __low2float(p[k]);
        y -= __high2float(p[k]);
    }
}

}  // namespace ziplm
