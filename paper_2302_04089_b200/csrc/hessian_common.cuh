// What the two tensor-core product kernels of the Hessian share (hessian_tc.cu, hessian_pair.cu).
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace ziplm {

// One product launch: H[layer0 + l] = beta H + alpha X X^T for `layers` layers of a K-major operand.
struct HessianProduct {
    CUtensorMap hi, lo;          // 16-bit operand, or the two fp16 parts of fp32 input (split)
    float* H;
    int d, layers, num_kb;       // K blocks of 64 tokens
    float alpha, beta;
    int layer0, L;               // L: all layers of the call
    unsigned long long* err_word; unsigned long long call;     // the word a wait that runs out sets to `call`
    uint32_t fmt16, spin;        // operand format of the instruction; poll limit of the producer
    const unsigned* amax;        // split: largest magnitudes of the feature rows
    bool split;
};

// Whether the kernel on CTA pairs takes a launch of that many layers (split: fp32 input in two parts).
bool hessian_pair_fits(int layers, int d, long long N, bool split);
// CTAs that share a 128 x 128 tile of the other one.
int hessian_tile_split(long long tiles, long long num_kb);
// Scratch that such a launch uses.
size_t hessian_pair_scratch_bytes(int layers, int d, long long N, bool split);
ziplm_status run_hessian_pair(const HessianProduct& p, void* scratch, size_t scratch_bytes, cudaStream_t st);

// A product kernel that gives up on a wait leaves NaN in H[l][0][0] of every layer of the call, so that
// whichever stage reads H next reports ZIPLM_ERR_NONFINITE.  The thread that gives up records the call's
// number first and poisons the layers then; the CTA that writes an entry (0, 0) looks for the number
// afterwards (hessian_check): whichever of the two comes second sees the other.  The number is new for
// every call, so the word needs no clearing, except in a captured call, whose replays share it.
__device__ __forceinline__ void hessian_give_up(float* H, int L, int d, unsigned long long* err_word,
                                                unsigned long long call) {
    atomicExch(err_word, call);
    __threadfence();
    for (int l = 0; l < L; ++l) *reinterpret_cast<volatile float*>(H + (size_t)l * d * d) = __int_as_float(0x7fc00000);
}
__device__ __forceinline__ void hessian_check(float* entry, const unsigned long long* err_word,
                                              unsigned long long call) {
    __threadfence();
    if (*reinterpret_cast<const volatile unsigned long long*>(err_word) == call)
        *reinterpret_cast<volatile float*>(entry) = __int_as_float(0x7fc00000);
}

// Power-of-two scale of a feature row from the bit pattern of its largest magnitude m: the largest
// scaled entry lies in [2^13, 2^14).  inverse = true gives 1 / scale.  Rows of zeros and
// non-finite rows are left alone; the exponent is clamped so that the scale is a normal number.
__device__ __forceinline__ float row_scale(unsigned amax_bits, bool inverse) {
    const int e = (int)((amax_bits >> 23) & 255u);
    if (amax_bits == 0u || e == 255) return 1.f;
    int k = 140 - e;                       // m in [2^(e-127), 2^(e-126))  ->  m 2^k < 2^14
    k = k > 100 ? 100 : (k < -100 ? -100 : k);
    return __int_as_float((127 + (inverse ? -k : k)) << 23);
}

}  // namespace ziplm
