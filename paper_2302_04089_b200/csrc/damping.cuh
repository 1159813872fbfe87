// The damping of a layer's Hessian (caption of Algorithm 1), as the damped inverse and the endgame use it.
#pragma once

#include <math.h>

#include "common.cuh"

namespace ziplm {

// lambda = damp_frac * mean(diag H) of layer l, by a CTA of 256 threads; every thread returns it.  A non-finite
// diagonal and, with damping, a mean that is not positive give 1 and are reported by the caller that is to do so.
__device__ __forceinline__ double mean_diag_lambda(const float* Hl, int d, float damp_frac, int* layer_status,
                                                   int l, bool report) {
    __shared__ double red[256];
    __shared__ int sbad;
    const int tid = threadIdx.x;
    double s = 0.0;
    bool bad = false;
    for (int i = tid; i < d; i += 256) {
        const float v = Hl[(size_t)i * d + i];
        if (!isfinite(v)) bad = true;
        s += (double)v;
    }
    if (tid == 0) sbad = 0;
    __syncthreads();
    if (bad) sbad = 1;
    red[tid] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (tid < o) red[tid] += red[tid + o];
        __syncthreads();
    }
    const double mean = red[0] / (double)d;
    double lm = (double)damp_frac * mean;
    int code = ZIPLM_OK;
    if (sbad || !isfinite(mean)) code = ZIPLM_ERR_NONFINITE;
    else if (damp_frac > 0.f && !(mean > 0.0)) code = ZIPLM_ERR_NOT_PD;
    if (code != ZIPLM_OK) {
        lm = 1.0;
        if (report && tid == 0) set_layer_status(layer_status, l, code);
    }
    return lm;
}

}  // namespace ziplm
