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

// An fp32 quotient as an integer of the same order.  Quotients of float64 values rounded to fp32 and divided
// approximately are good to 1e-5, 84 to 168 units of the key: candidates within kKeyNear of each other have
// to be compared exactly, and so have offers within kKeyFar (4e-5 at least) of each other, which are the
// best of their warps or CTAs up to kKeyNear.
constexpr unsigned kKeyNegInf = 0x007fffffu, kKeyInf = 0xff800000u, kKeyNone = 0xffffffffu;
constexpr unsigned kKeyNear = 256u, kKeyFar = 700u;
__device__ __forceinline__ unsigned order_key(float r) {
    const unsigned bits = __float_as_uint(r);
    return bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ unsigned cand_key(bool alive, double a, double q) {
    const int ha = __double2hiint(a), hq = __double2hiint(q);
    const bool ok = (unsigned)(ha - 1) < 0x7fefffffu && (hq & 0x7fffffff) < 0x7ff00000;   // a > 0, finite
    const float x = __fdividef((float)q, (float)a);
    return alive ? (ok ? order_key(x) : kKeyNegInf) : kKeyNone;
}

// What a warp, or a CTA, offers as its next pick.
struct __align__(16) Bid {
    double a, q;
    int org, pos;
    unsigned key, pad;
};
__device__ __forceinline__ Cand cand_of(const Bid& b) {
    Cand c;
    c.a = b.a; c.q = b.q; c.org = b.org; c.pos = b.pos;
    return c;
}

// Index of the best of n <= 32 bids: the one whose key is alone within kKeyFar of the smallest, otherwise --
// near ties, an invalid entry, nothing left -- by the exact comparison.  Every lane returns it.
__device__ __forceinline__ int best_bid(const Bid* bids, int n, int lane) {
    const unsigned k = lane < n ? bids[lane].key : kKeyNone;
    const unsigned kmin = __reduce_min_sync(0xffffffffu, k);
    const unsigned near_min = __ballot_sync(0xffffffffu, k - kmin <= kKeyFar);
    int which = __ffs(near_min) - 1;
    if ((near_min & (near_min - 1)) || kmin <= kKeyNegInf || kmin >= kKeyInf) {
        Cand best;
        best.pos = -1; best.a = 1.0; best.q = 0.0; best.org = 0x7fffffff;
        which = 0;
        for (int c = 0; c < n; ++c) {
            const Cand o = cand_of(bids[c]);
            if (o.pos >= 0 && (best.pos < 0 || better(o, best))) { best = o; which = c; }
        }
    }
    return which;
}

}  // namespace ziplm
