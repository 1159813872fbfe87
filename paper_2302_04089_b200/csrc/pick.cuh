// Device-side argmin of the saliencies rho = Q[k,k] / H^-1[k,k], shared by the neuron-path kernels.
#pragma once

#include <math.h>

#include "common.cuh"

namespace ziplm {

// Candidate of the argmin of rho = q / a (q = Q[k,k], a = H^-1[k,k]).  Candidates are compared by
// cross-multiplication (q_x a_y < q_y a_x), which needs no float64 division on the critical path;
// the quotient is formed once, for the winner.  An entry whose a is not positive or whose values
// are not finite sorts first, so that it is picked -- and its layer flagged -- at once.
struct Cand {
    double a, q;
    int org, pos;
};

__device__ __forceinline__ bool cand_valid(const Cand& x) {
    return x.a > 0.0 && isfinite(x.a) && isfinite(x.q);
}

__device__ __forceinline__ bool better(const Cand& x, const Cand& y) {   // x strictly before y
    const bool vx = cand_valid(x), vy = cand_valid(y);
    if (vx != vy) return !vx;
    if (!vx) return x.org < y.org;
    const double lhs = x.q * y.a, rhs = y.q * x.a;
    return lhs < rhs || (lhs == rhs && x.org < y.org);
}

__device__ __forceinline__ void merge_cand(Cand& best, const Cand& o) {
    if (o.pos >= 0 && (best.pos < 0 || better(o, best))) best = o;
}

__device__ __forceinline__ Cand bcast_cand(const Cand& c, int src_lane) {
    Cand o;
    o.a = __shfl_sync(0xffffffffu, c.a, src_lane);
    o.q = __shfl_sync(0xffffffffu, c.q, src_lane);
    o.org = __shfl_sync(0xffffffffu, c.org, src_lane);
    o.pos = __shfl_sync(0xffffffffu, c.pos, src_lane);
    return o;
}

// fp32 quotient that orders candidates coarsely: +inf for "none", -inf for an invalid entry.
__device__ __forceinline__ float cand_quotient(const Cand& c) {
    if (c.pos < 0) return INFINITY;
    return cand_valid(c) ? __fdividef((float)c.q, (float)c.a) : -INFINITY;
}

// Best candidate of a warp (every lane returns it).  The cheap fp32 quotient r orders the lanes;
// only the lanes within 1e-5 of the fp32 minimum (almost always a single one) go through the exact
// float64 comparison, so the common case costs one reduction and six 32-bit shuffles instead of
// five rounds of 64-bit exchanges.
__device__ __forceinline__ Cand warp_best(const Cand& mine, float r, float* warp_min = nullptr) {
    // warp minimum in one reduction instruction, on keys that order like the floats they encode
    const unsigned bits = __float_as_uint(r);
    const unsigned key = bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u);
    const unsigned kmin = __reduce_min_sync(0xffffffffu, key);
    const float rmin = __uint_as_float(kmin ^ ((kmin >> 31) ? 0x80000000u : 0xffffffffu));
    if (warp_min) *warp_min = rmin;
    const bool near_min = mine.pos >= 0 && (r == rmin || r <= rmin + fabsf(rmin) * 1e-5f);
    unsigned mask = __ballot_sync(0xffffffffu, near_min);
    Cand best;
    best.a = 1.0; best.q = 0.0; best.org = 0x7fffffff; best.pos = -1;
    while (mask) {
        const int b = __ffs(mask) - 1;
        mask &= mask - 1;
        merge_cand(best, bcast_cand(mine, b));
    }
    return best;
}

__device__ __forceinline__ Cand warp_best(const Cand& mine) { return warp_best(mine, cand_quotient(mine)); }

// What a warp, or a CTA, offers as its next pick.
struct __align__(16) Offer {
    Cand c;
};

// Pick among n <= 32 offers by their fp32 keys (good to 1e-5): when exactly one key lies within 4e-5 of
// the smallest, that offer is the pick and is read directly; otherwise -- near ties, an invalid entry,
// nothing left -- all of them go through the exact comparison.  Every lane returns the pick and its index.
__device__ __forceinline__ Cand pick_offer(const Offer* offers, const float* keys, int n, int lane, int* which) {
    const float k = lane < n ? keys[lane] : INFINITY;
    const unsigned bits = __float_as_uint(k);
    const unsigned kmin = __reduce_min_sync(0xffffffffu, bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u));
    const float rmin = __uint_as_float(kmin ^ ((kmin >> 31) ? 0x80000000u : 0xffffffffu));
    const unsigned near_min = __ballot_sync(0xffffffffu, k <= rmin + fabsf(rmin) * 4e-5f);
    if (fabsf(rmin) < INFINITY && __popc(near_min) == 1) {
        *which = __ffs(near_min) - 1;
        return offers[*which].c;
    }
    Cand g;
    g.a = 1.0; g.q = 0.0; g.org = 0x7fffffff; g.pos = -1;
    if (lane < n) g = offers[lane].c;
    const Cand best = warp_best(g);
    const unsigned mine = __ballot_sync(0xffffffffu, lane < n && best.pos >= 0 && g.pos == best.pos);
    *which = mine ? __ffs(mine) - 1 : 0;
    return best;
}

}  // namespace ziplm
