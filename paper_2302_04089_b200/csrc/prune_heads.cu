// Greedy structured OBS for attention heads: structures of g consecutive columns, g a multiple of 16
// from 32 to 128 (prune_block.cu serves the other widths).
//
// With S the columns of the selected head and B = (H^-1)[S,S], everything a step needs follows from
//     T  = B^-1 (H^-1)[S,:]                                  (g x d)
//     H^-1 <- H^-1 - (H^-1)[:,S] T                           (Eq. 4)
//     W    <- W    - W[:,S] T                                (Eq. 3)
// and the saliency rho_S = tr(W[:,S] B^-1 W[:,S]^T) = <B^-1, Q[S,S]> (Eq. 2) from the Gram matrix
// Q = W^T W, which is carried along instead of being formed again from W for every head and step:
//     Q <- Q - V^T T - T^T V,   V = Q[S,:] - 1/2 Q[S,S] T.
// The whole state (H^-1, Q, W) is float64.  Removed heads stay in place and are skipped.
//
// A layer has 8 to 16 heads, so the loop is short and used to be bound by latency: a Cholesky
// factorisation with three barriers per column, a forward substitution and a Gram product over all
// rows of W for every head and step (232 us a step for 12 layers of 12 heads of 64), then another
// 250 us for the update on the float64 FMA pipe.  Here every product is a g x g x g tile product on
// the float64 tensor-core instruction, the inverse of a head's block goes by 16 x 16 blocks (two
// barriers per block), and a step is two launches (programmatic dependent ones): `solve` (which also selects) and `update` (whose
// diagonal tiles go on to score their head for the next step, and whose tiles of W write the
// snapshot).
#include <math.h>

#include "common.cuh"
#include "factor16.cuh"
#include "inverse_i8.cuh"
#include "tc_common.cuh"

namespace ziplm {
namespace {

constexpr int HT = 256;          // threads per CTA
constexpr int KCH = 32;          // k-chunk of a tile product
constexpr int P_MK = KCH + 4;    // pitch of a chunk stored [m][k]; like g + 4 it is 4 mod 16, so that the
                                 // 16 lanes of a half-warp's fragment load hit 16 different 8-byte banks

// Shape of the tile products of heads of 8 * G8 columns.  A warp owns UN units of one row of 8 x 8
// fragments by half of the columns; all its units lie in the same half and share its fragments.
template <int G8>
struct HeadShape {
    static constexpr int g = 8 * G8, CF = G8 / 2, UN = (2 * G8 + 7) / 8, P_KM = g + 4;
    static constexpr int kOperand = KCH * P_KM > g * P_MK ? KCH * P_KM : g * P_MK;     // doubles
    static constexpr int kScore = g * P_KM + (g + 16) * PB;                            // a head's block, panel
    static constexpr size_t kSmem = sizeof(double) * (4 * kOperand > kScore ? 4 * kOperand : kScore);   // two stages
};

template <int G8>
struct HeadAcc {
    using S = HeadShape<G8>;
    double d[S::UN][S::CF][2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int u = 0; u < S::UN; ++u)
#pragma unroll
            for (int j = 0; j < S::CF; ++j) d[u][j][0] = d[u][j][1] = 0.0;
    }
    // f(row, col, pair) with col even, for every pair this thread holds
    template <typename F>
    __device__ __forceinline__ void visit(F f) const {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int u = 0; u < S::UN; ++u) {
            const int rf = (warp + 8 * u) >> 1;
            if (rf >= G8) continue;
#pragma unroll
            for (int j = 0; j < S::CF; ++j)
                f(8 * rf + (lane >> 2), 8 * ((warp & 1) * S::CF + j) + 2 * (lane & 3),
                  make_double2(d[u][j][0], d[u][j][1]));
        }
    }
};

__device__ __forceinline__ void h_cp16(double* dst, const double* src, bool ok) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(src), "r"(ok ? 16u : 0u) : "memory");
}

// Start the copy of one chunk of an operand: KM: P[k * ld + m], m < g, kept [k][m], rows k >= k_valid
// zero; otherwise P[m * ld + k], kept [m][k], rows m >= m_valid and columns k >= k_valid zero.
template <int G8, bool KM>
__device__ __forceinline__ void h_chunk(double* s, const double* P, size_t ld, int k0, int k_valid, int m_valid) {
    using S = HeadShape<G8>;
    for (int e = threadIdx.x; e < S::g * KCH / 2; e += HT) {
        if (KM) {
            const int k = e / (S::g / 2), m = 2 * (e % (S::g / 2));
            const bool ok = k0 + k < k_valid;
            h_cp16(s + k * S::P_KM + m, P + (ok ? (size_t)(k0 + k) * ld + m : 0), ok);
        } else {
            const int m = e / (KCH / 2), k = 2 * (e % (KCH / 2));
            const bool ok = m < m_valid && k0 + k < k_valid;
            h_cp16(s + m * P_MK + k, P + (ok ? (size_t)m * ld + k0 + k : 0), ok);
        }
    }
}

template <int G8, bool KM>
__device__ __forceinline__ double h_frag(const double* s, int m0, int kk, int lane) {
    return KM ? s[(kk * 4 + (lane & 3)) * HeadShape<G8>::P_KM + m0 + (lane >> 2)]
              : s[(m0 + (lane >> 2)) * P_MK + kk * 4 + (lane & 3)];
}

// acc += one chunk's product of `steps` mma steps.
template <int G8, bool XKM, bool YKM>
__device__ __forceinline__ void h_chunk_mma(HeadAcc<G8>& acc, const double* sx, const double* sy, int steps, int warp,
                                            int lane) {
    using S = HeadShape<G8>;
#pragma unroll 4
    for (int kk = 0; kk < steps; ++kk) {
        double b[S::CF];
#pragma unroll
        for (int j = 0; j < S::CF; ++j) b[j] = h_frag<G8, YKM>(sy, 8 * ((warp & 1) * S::CF + j), kk, lane);
#pragma unroll
        for (int u = 0; u < S::UN; ++u) {
            const int rf = (warp + 8 * u) >> 1;
            if (rf >= G8) continue;
            const double a = h_frag<G8, XKM>(sx, 8 * rf, kk, lane);
#pragma unroll
            for (int j = 0; j < S::CF; ++j) dmma884(acc.d[u][j], a, b[j]);
        }
    }
}

// acc(g x g) += X (g x K) Y (K x g).  XKM: X(m,k) = X[k * ldx + m], else X[m * ldx + k] with rows from
// x_rows on zero; YKM: Y(k,n) = Y[k * ldy + n], else Y[n * ldy + k].  K is a multiple of 16 unless both
// are stored by k.  Starts with every thread past its use of smem and ends with a barrier.
template <int G8, bool XKM, bool YKM>
__device__ __forceinline__ void h_product(HeadAcc<G8>& acc, const double* X, size_t ldx, int x_rows,
                                          const double* Y, size_t ldy, int K, double* smem) {
    using S = HeadShape<G8>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nch = (K + KCH - 1) / KCH;
    auto start = [&](int c) {
        double* s = smem + (c & 1) * 2 * S::kOperand;
        h_chunk<G8, XKM>(s, X, ldx, c * KCH, K, x_rows);
        h_chunk<G8, YKM>(s + S::kOperand, Y, ldy, c * KCH, K, S::g);
    };
    start(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int c = 0; c < nch; ++c) {
        if (c + 1 < nch) start(c + 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const double* sx = smem + (c & 1) * 2 * S::kOperand;
        const double* sy = sx + S::kOperand;
        const int steps = (min(KCH, K - c * KCH) + 3) / 4;        // (a row past K is zero)
        h_chunk_mma<G8, XKM, YKM>(acc, sx, sy, steps, warp, lane);
        __syncthreads();
    }
}

// As h_product (both operands stored by k, K = g) for `n` products in a row: operands(i, X, Y) gives those
// of the i-th, done(i) runs when it is complete.  The copies of the next product run beside `done`.
template <int G8, typename Ops, typename Done>
__device__ __forceinline__ void h_products(HeadAcc<G8>& acc, int n, size_t ld, double* smem, Ops operands, Done done) {
    using S = HeadShape<G8>;
    constexpr int NC = (S::g + KCH - 1) / KCH;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto start = [&](int c) {
        const double *X, *Y;
        operands(c / NC, X, Y);
        double* s = smem + (c & 1) * 2 * S::kOperand;
        h_chunk<G8, true>(s, X, ld, (c % NC) * KCH, S::g, S::g);
        h_chunk<G8, true>(s + S::kOperand, Y, ld, (c % NC) * KCH, S::g, S::g);
    };
    start(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int c = 0; c < n * NC; ++c) {
        if (c + 1 < n * NC) start(c + 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        const double* sx = smem + (c & 1) * 2 * S::kOperand;
        h_chunk_mma<G8, true, true>(acc, sx, sx + S::kOperand, min(KCH, S::g - (c % NC) * KCH) / 4, warp, lane);
        __syncthreads();
        if (c % NC == NC - 1) done(c / NC);
    }
}

// use(row, col, product, load(row, col)) for every pair of the thread's.  The loads of CF pairs (after(),
// or with kAhead of all, before the product) are in flight together: a load behind a store it may alias
// waits for it, and one such pair after the other took 10000 clocks.
template <int G8, bool kAhead, typename P, typename Ld, typename Use>
__device__ __forceinline__ void h_combine(HeadAcc<G8>& acc, P product, Ld load, Use use) {
    using S = HeadShape<G8>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    decltype(load(0, 0)) v[kAhead ? S::UN : 1][S::CF];
    auto fetch = [&](int u) {
#pragma unroll
        for (int j = 0; j < S::CF; ++j)
            v[kAhead ? u : 0][j] = load(8 * ((warp + 8 * u) >> 1) + (lane >> 2), 8 * ((warp & 1) * S::CF + j) + 2 * (lane & 3));
    };
    if (kAhead) {
#pragma unroll
        for (int u = 0; u < S::UN; ++u)
            if ((warp + 8 * u) >> 1 < G8) fetch(u);
    }
    product();
#pragma unroll
    for (int u = 0; u < S::UN; ++u) {
        if ((warp + 8 * u) >> 1 >= G8) continue;
        if (!kAhead) fetch(u);
#pragma unroll
        for (int j = 0; j < S::CF; ++j)
            use(8 * ((warp + 8 * u) >> 1) + (lane >> 2), 8 * ((warp & 1) * S::CF + j) + 2 * (lane & 3),
                make_double2(acc.d[u][j][0], acc.d[u][j][1]), v[kAhead ? u : 0][j]);
    }
}

// Everything the kernels of a call work on.
struct Heads {
    int L, G, r, d;
    const float* W; const float* H;
    double* A; double* Q; double* W64;      // [d][d] (Q and, after the first step, A: lower blocks), [r][d]
    double* P; double* T; double* V;        // [g][d]: (H^-1)[S,:], T, V of the step
    double* Bneg;                           // [G][g][g]: -(head's block of H^-1)^-1
    double* rho;                            // [G]: saliencies of the live heads
    double* rho_sel;                        // [G]: of the removed ones, by step
    double* dw2;                            // [n_levels + 1]: ||W - W_snap||^2 by level, then 2 * base loss
    int* alive;                             // [2][G], by step parity
    int* chosen;                            // [1]
    int* steps_of;                          // [n_levels], shared by the layers: removals of a level
    float* W_snap; int n_levels;
    int pairs;                              // W and W_snap start on 8 bytes
    int* order; float* saliency; int* layer_status;
};

// Row block i >= j of a lower-triangular pair index.
__device__ __forceinline__ void pair_index(int x, int& i, int& j) {
    i = (int)((sqrtf(8.f * (float)x + 1.f) - 1.f) * 0.5f);
    while (i * (i + 1) / 2 > x) --i;
    while ((i + 1) * (i + 2) / 2 <= x) ++i;
    j = x - i * (i + 1) / 2;
}

// Sum over the CTA, in thread 0.
__device__ __forceinline__ double h_sum(double v, double* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < HT / 32; ++w) t += red[w];
    return t;
}

// rho of head s of layer l and -(H^-1)[S,S]^-1, from the diagonal blocks of H^-1 and Q.  With M the inverse
// of the Cholesky factor of B = (H^-1)[S,S]: B^-1 = M^T M.
// M by elimination of [B | I] in 16 x 16 blocks, in place in shared memory (block (i, j), j < b, of the
// lower triangle holds X_ij, the others what is left of B): one warp turns the diagonal block into M_bb,
// then L_ib = B_ib M_bb^T (kept aside) and X_bj = M_bb X_bj, then B_ik -= L_ib L_kb^T, X_ij -= L_ib X_bj
// and X_ib = -L_ib M_bb, a warp and 16 mma instructions per block; warp 0 updates the next diagonal block
// and goes on with it while the others do the rest.  The chain is the pivots'.  Heads of 64: 20000 clocks
// (symmetric sweeps in registers, one barrier per column, took 45000).
template <int G8>
__device__ void h_score(const Heads& w, int l, int s, double* red, double* smem) {
    using S = HeadShape<G8>;
    constexpr int NB = S::g / 16, PG = S::P_KM;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double* m = smem;                                     // [g][PG]
    double* pan = smem + S::g * PG;                       // [g][PB]: L_ib
    double* blk = pan + S::g * PB;                        // [16][PB]: M_bb
    const size_t at = (size_t)l * w.d * w.d + (size_t)s * S::g * w.d + (size_t)s * S::g;
    for (int e = tid; e < S::g * S::g / 2; e += HT) {
        const int i = e / (S::g / 2), j = 2 * (e % (S::g / 2));
        *reinterpret_cast<double2*>(m + i * PG + j) =
            j >> 4 <= i >> 4 ? *reinterpret_cast<const double2*>(w.A + at + (size_t)i * w.d + j) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    auto X = [&](int i, int j) { return m + 16 * i * PG + 16 * j; };
    int flag = 0;
#pragma unroll 1
    for (int b = 0; b < NB; ++b) {
        if (warp == 0) {
            __syncwarp();
            const int f = warp_factor16(X(b, b), PG, blk);
            if (!flag) flag = f;
        }
        __syncthreads();
        const int n = NB - 1 - b;
        for (int q = warp; q < NB; q += HT / 32) {
            double c[2][2][2] = {};
            if (q < n) {
                warp_mma16<true>(c, X(b + 1 + q, b), PG, blk, PB);
                warp_put16<false>(c, pan + 16 * (b + 1 + q) * PB, PB);
            } else if (q < n + b) {
                double* x = X(b, q - n);
                warp_mma16<false>(c, blk, PB, x, PG);
                __syncwarp();
                warp_put16<false>(c, x, PG);
            } else {
                for (int e = lane; e < 256; e += 32) X(b, b)[(e >> 4) * PG + (e & 15)] = blk[(e >> 4) * PB + (e & 15)];
            }
        }
        __syncthreads();
        const int n_a = n * (n + 1) / 2, n_all = n_a + n * (b + 1);
        for (int q = warp; q < n_all; q += warp == 0 ? n_all : HT / 32 - 1) {
            double c[2][2][2] = {};
            if (q < n_a) {
                int ii, kk;
                pair_index(q, ii, kk);
                const int i = b + 1 + ii, k = b + 1 + kk;
                warp_mma16<true>(c, pan + 16 * i * PB, PB, pan + 16 * k * PB, PB);
                warp_put16<true>(c, X(i, k), PG);
            } else {
                const int i = b + 1 + (q - n_a) / (b + 1), j = (q - n_a) % (b + 1);
                warp_mma16<false>(c, pan + 16 * i * PB, PB, X(b, j), PG);
                if (j == b) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) c[e >> 2][(e >> 1) & 1][e & 1] = -c[e >> 2][(e >> 1) & 1][e & 1];
                    warp_put16<false>(c, X(i, j), PG);
                } else {
                    warp_put16<true>(c, X(i, j), PG);
                }
            }
        }
    }
    // B^-1 = M^T M: both operands are M stored by k, whose rows above a column's are zero
    HeadAcc<G8> acc;
    acc.zero();
#pragma unroll
    for (int u = 0; u < S::UN; ++u) {
        const int rf = (warp + 8 * u) >> 1;
        if (rf >= G8) continue;
#pragma unroll 2
        for (int kk = 2 * max(rf, (warp & 1) * S::CF); kk < S::g / 4; ++kk) {
            const double a = m[(kk * 4 + (lane & 3)) * PG + 8 * rf + (lane >> 2)];
#pragma unroll
            for (int j = 0; j < S::CF; ++j)
                dmma884(acc.d[u][j], a, m[(kk * 4 + (lane & 3)) * PG + 8 * ((warp & 1) * S::CF + j) + (lane >> 2)]);
        }
    }
    double part = 0.0;
    double* B = w.Bneg + ((size_t)l * w.G + s) * S::g * S::g;
    acc.visit([&](int i, int j, double2 x) {
        const double2 q = *reinterpret_cast<const double2*>(w.Q + at + (size_t)i * w.d + j);
        *reinterpret_cast<double2*>(B + i * S::g + j) = make_double2(-x.x, -x.y);
        part = fma(x.x, q.x, fma(x.y, q.y, part));
    });
    const double rho = h_sum(part, red);
    if (tid == 0) {
        w.rho[(size_t)l * w.G + s] = rho;
        if (flag) set_layer_status(w.layer_status, l, flag);
    }
}

__global__ void __launch_bounds__(HT) k_heads_init(Heads w) {
    const size_t count = (size_t)w.L * w.r * w.d;
    for (size_t i = (size_t)blockIdx.x * HT + threadIdx.x; i < count; i += (size_t)gridDim.x * HT)
        w.W64[i] = (double)w.W[i];
    for (int i = blockIdx.x * HT + threadIdx.x; i < w.L * w.G; i += gridDim.x * HT)
        w.alive[(size_t)(i / w.G) * 2 * w.G + i % w.G] = 1;
}

// Block (i, j), i >= j, of Q = W^T W.
template <int G8>
__global__ void __launch_bounds__(HT) k_heads_gram(Heads w) {
    using S = HeadShape<G8>;
    extern __shared__ __align__(16) double smem[];
    const int l = blockIdx.y;
    int i, j;
    pair_index(blockIdx.x, i, j);
    const double* Wl = w.W64 + (size_t)l * w.r * w.d;
    HeadAcc<G8> acc;
    acc.zero();
    h_product<G8, true, true>(acc, Wl + i * S::g, w.d, S::g, Wl + j * S::g, w.d, w.r, smem);
    const size_t at = (size_t)l * w.d * w.d + (size_t)i * S::g * w.d + (size_t)j * S::g;
    acc.visit([&](int row, int col, double2 x) {
        *reinterpret_cast<double2*>(w.Q + at + (size_t)row * w.d + col) = x;
    });
}

// <Q, H> = 2 ||W X||^2 from the lower triangles.
__global__ void __launch_bounds__(HT) k_heads_base(Heads w) {
    __shared__ double red[HT / 32];
    const int l = blockIdx.y;
    double part = 0.0;
    for (int i = blockIdx.x; i < w.d; i += gridDim.x) {
        const size_t row = ((size_t)l * w.d + i) * w.d;
        for (int j = threadIdx.x; j <= i; j += HT) part += (j < i ? 2.0 : 1.0) * w.Q[row + j] * (double)w.H[row + j];
    }
    const double t = h_sum(part, red);
    if (threadIdx.x == 0) atomicAdd(w.dw2 + (size_t)l * (w.n_levels + 1) + w.n_levels, t);
}

template <int G8>
__global__ void __launch_bounds__(HT) k_heads_score(Heads w) {
    extern __shared__ __align__(16) double smem[];
    __shared__ double red[HT / 32];
    h_score<G8>(w, blockIdx.y, blockIdx.x, red, smem);
}

// Selection (argmin of rho over the live heads, ties to the lowest index; every CTA makes it for
// itself) and, for the columns of head blockIdx.x, P = (H^-1)[S,:], T = B^-1 P, V = Q[S,:] - Q[S,S] T / 2.
template <int G8>
__global__ void __launch_bounds__(HT) k_heads_solve(Heads w, int t) {
    using S = HeadShape<G8>;
    extern __shared__ __align__(16) double smem[];
    __shared__ int s_pick;
    const int l = blockIdx.y, j = blockIdx.x, tid = threadIdx.x;
    const int* alive = w.alive + ((size_t)l * 2 + (t & 1)) * w.G;
    tc::grid_trigger();
    tc::grid_wait();
    if (tid < 32) {
        double best = INFINITY;
        int at = 0x7fffffff;
        for (int s = tid; s < w.G; s += 32) {
            if (!alive[s]) continue;
            double x = w.rho[(size_t)l * w.G + s];
            if (!(x == x)) x = INFINITY;
            if (x < best || (x == best && s < at)) { best = x; at = s; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double x = __shfl_xor_sync(0xffffffffu, best, o);
            const int s = __shfl_xor_sync(0xffffffffu, at, o);
            if (x < best || (x == best && s < at)) { best = x; at = s; }
        }
        if (tid == 0) s_pick = at;
        if (j == 0) {
            for (int s = tid; s < w.G; s += 32)
                w.alive[((size_t)l * 2 + ((t + 1) & 1)) * w.G + s] = s == at ? 0 : alive[s];
            if (tid == 0) {
                if (!isfinite(best)) set_layer_status(w.layer_status, l, ZIPLM_ERR_NONFINITE);
                w.chosen[l] = at;
                w.rho_sel[(size_t)l * w.G + t] = isfinite(best) ? best : 0.0;
                w.order[(size_t)l * w.G + t] = at;
                if (w.saliency) w.saliency[(size_t)l * w.G + t] = (float)best;
            }
        }
    }
    __syncthreads();
    const int s = s_pick;
    if (!alive[j] || j == s) return;
    const size_t lay = (size_t)l * w.d * w.d, out = (size_t)l * S::g * w.d + (size_t)j * S::g;
    const bool below = j > s;       // the block is stored as (j, s): transposed
    const size_t blk = lay + (below ? (size_t)j * S::g * w.d + (size_t)s * S::g
                                    : (size_t)s * S::g * w.d + (size_t)j * S::g);
    const double* Bn = w.Bneg + ((size_t)l * w.G + s) * S::g * S::g;
    HeadAcc<G8> acc;
    constexpr bool kAhead = G8 <= 8;     // one CTA per SM here, so registers are to be had
    auto block = [&](const double* M) {
        return [=](int k, int n) {
            const double* o = M + (below ? blk + (size_t)n * w.d + k : blk + (size_t)k * w.d + n);
            return below ? make_double2(o[0], o[w.d]) : *reinterpret_cast<const double2*>(o);
        };
    };
    acc.zero();
    // B^-1 is symmetric: stored by k as well as by m
    h_combine<G8, kAhead>(acc, [&] {
        if (below) h_product<G8, true, false>(acc, Bn, S::g, S::g, w.A + blk, w.d, S::g, smem);
        else h_product<G8, true, true>(acc, Bn, S::g, S::g, w.A + blk, w.d, S::g, smem);
    }, block(w.A), [&](int k, int n, double2 x, double2 p) {
        *reinterpret_cast<double2*>(w.T + out + (size_t)k * w.d + n) = make_double2(-x.x, -x.y);
        *reinterpret_cast<double2*>(w.P + out + (size_t)k * w.d + n) = p;
    });
    __syncthreads();                // T is read back below, by the whole CTA
    const size_t ss = lay + (size_t)s * S::g * w.d + (size_t)s * S::g;
    acc.zero();
    h_combine<G8, kAhead>(acc, [&] {
        h_product<G8, true, true>(acc, w.Q + ss, w.d, S::g, w.T + out, w.d, S::g, smem);
    }, block(w.Q), [&](int k, int n, double2 x, double2 q) {
        *reinterpret_cast<double2*>(w.V + out + (size_t)k * w.d + n) =
            make_double2(fma(-0.5, x.x, q.x), fma(-0.5, x.y, q.y));
    });
}

// CTAs 0 .. G - 1 of every layer: diagonal blocks of H^-1 and Q, then the head's next score; the next G (G - 1) / 2:
// blocks below the diagonal; the rest: blocks of g rows of W and, when `slot` is a level, of the snapshot.  The
// longest CTAs come first, those of all layers before the next kind (layer after layer the last layer's scores, a chain
// of 20000 clocks, began when the rest was nearly done: twelve updates of 12 x 768 x 768 took 910 us, now 749).
template <int G8>
__global__ void __launch_bounds__(HT) k_heads_update(Heads w, int t, int slot, int rescore) {
    using S = HeadShape<G8>;
    extern __shared__ __align__(16) double smem[];
    __shared__ double red[HT / 32];
    const int l = blockIdx.x % w.L, x = blockIdx.x / w.L, n_pairs = w.G * (w.G + 1) / 2;
    tc::grid_trigger();
    tc::grid_wait();
    if (slot >= 0 && x == 0 && l == 0 && threadIdx.x == 0) w.steps_of[slot] = t + 1;
    const int* alive = w.alive + ((size_t)l * 2 + ((t + 1) & 1)) * w.G;
    const size_t ops = (size_t)l * S::g * w.d;
    HeadAcc<G8> acc;
    if (x < n_pairs) {
        int i = x, j = x;
        if (x >= w.G) { pair_index(x - w.G, i, j); ++i; }
        if (!alive[i] || !alive[j]) return;
        const size_t at = (size_t)l * w.d * w.d + (size_t)i * S::g * w.d + (size_t)j * S::g;
        const double *Pi = w.P + ops + i * S::g, *Ti = w.T + ops + i * S::g, *Tj = w.T + ops + j * S::g;
        const double *Vi = w.V + ops + i * S::g, *Vj = w.V + ops + j * S::g;
        acc.zero();
        h_products<G8>(acc, 3, w.d, smem, [&](int q, const double*& X, const double*& Y) {
            X = q == 0 ? Pi : q == 1 ? Vi : Ti;
            Y = q == 2 ? Vj : Tj;
        }, [&](int q) {
            if (q == 1) return;
            double* M = (q == 0 ? w.A : w.Q) + at;
            h_combine<G8, false>(acc, [] {}, [=](int row, int col) {
                return *reinterpret_cast<const double2*>(M + (size_t)row * w.d + col);
            }, [=](int row, int col, double2 d, double2 cur) {
                *reinterpret_cast<double2*>(M + (size_t)row * w.d + col) = make_double2(cur.x - d.x, cur.y - d.y);
            });
            acc.zero();
        });
        if (i == j && rescore) {
            __syncthreads();
            h_score<G8>(w, l, i, red, smem);
        }
        return;
    }
    const int j = (x - n_pairs) % w.G, b = (x - n_pairs) / w.G, row0 = b * S::g;
    const int rows = min(S::g, w.r - row0);
    const float* W0 = w.W + ((size_t)l * w.r + row0) * w.d + (size_t)j * S::g;
    float* snap = slot < 0 ? nullptr
                           : w.W_snap + (((size_t)l * w.n_levels + slot) * w.r + row0) * w.d + (size_t)j * S::g;
    double part = 0.0;
    if (!alive[j]) {
        if (!snap) return;
        for (int e = threadIdx.x; e < rows * (S::g / 4); e += HT) {
            const size_t o = (size_t)(e / (S::g / 4)) * w.d + 4 * (e % (S::g / 4));
            for (int c = 0; c < 4; ++c) {
                part += (double)W0[o + c] * (double)W0[o + c];
                snap[o + c] = 0.f;
            }
        }
    } else {
        double* Wl = w.W64 + ((size_t)l * w.r + row0) * w.d;
        acc.zero();
        h_product<G8, false, true>(acc, Wl + (size_t)w.chosen[l] * S::g, w.d, rows, w.T + ops + j * S::g, w.d, S::g,
                                   smem);
        struct Cur { double2 w; float2 w0; };
        h_combine<G8, false>(acc, [] {}, [&](int row, int col) {
            const size_t o = (size_t)min(row, rows - 1) * w.d + col;
            return Cur{*reinterpret_cast<const double2*>(Wl + (size_t)j * S::g + o),
                       !snap ? make_float2(0.f, 0.f)
                             : w.pairs ? *reinterpret_cast<const float2*>(W0 + o) : make_float2(W0[o], W0[o + 1])};
        }, [&](int row, int col, double2 d, Cur cur) {
            if (row >= rows) return;
            const size_t o = (size_t)row * w.d + col;
            cur.w.x -= d.x; cur.w.y -= d.y;
            *reinterpret_cast<double2*>(Wl + (size_t)j * S::g + o) = cur.w;
            if (snap) {
                const float f0 = (float)cur.w.x, f1 = (float)cur.w.y, e0 = cur.w0.x - f0, e1 = cur.w0.y - f1;
                if (w.pairs) *reinterpret_cast<float2*>(snap + o) = make_float2(f0, f1);
                else { snap[o] = f0; snap[o + 1] = f1; }
                part += (double)e0 * e0 + (double)e1 * e1;
            }
        });
    }
    if (!snap) return;
    const double sum = h_sum(part, red);
    if (threadIdx.x == 0 && sum != 0.0) atomicAdd(w.dw2 + (size_t)l * (w.n_levels + 1) + slot, sum);
}

// Losses of all levels (half the sum of the saliencies removed so far, less the damping's share: every
// rho is twice the increase of the damped objective) and the base loss.  One warp per layer.
__global__ void __launch_bounds__(32) k_heads_loss(Heads w, const double* __restrict__ lam, float* __restrict__ loss,
                                                   float* __restrict__ base_loss) {
    const int l = blockIdx.x;
    const double* dw2 = w.dw2 + (size_t)l * (w.n_levels + 1);
    for (int q = threadIdx.x; q < w.n_levels; q += 32) {
        double sum = 0.0;
        for (int t = 0; t < w.steps_of[q]; ++t) sum += w.rho_sel[(size_t)l * w.G + t];
        const double x = 0.5 * sum - 0.5 * lam[l] * dw2[q];
        loss[(size_t)l * w.n_levels + q] = (float)(x > 0.0 ? x : 0.0);
    }
    if (threadIdx.x == 0 && base_loss) base_loss[l] = (float)(0.5 * dw2[w.n_levels]);
}

struct HeadsWs {
    Heads h;
    double* lam; void* inv_ws; size_t inv_bytes, zero_bytes; void* zero; size_t total;
};

// Q = W^T W in digits on the int8 tensor cores when that is quicker (12 x 768 x 768: 262 -> 195 us); the
// float64 kernel runs at 0.65 of its instruction's rate, and a CTA's chain is 4500 clocks per 64^3.
bool gram_on_i8(int L, int r, int d, int g) {
    const double G = d / g, ctas = L * G * (G + 1) / 2, cta = (double)r * g * g / 64 * 1.1 + 4000;
    return i8_symmetric_pays(L, d, r, cta > ctas * cta / (kSMs * 0.65) ? cta : ctas * cta / (kSMs * 0.65));
}

HeadsWs carve_heads(void* ws, int L, int r, int d, int g, int n_levels) {
    HeadsWs w = {};
    const int G = d / g;
    w.h.L = L; w.h.G = G; w.h.r = r; w.h.d = d; w.h.n_levels = n_levels;
    Carver c(ws);
    w.h.A = c.take<double>((size_t)L * d * d);
    w.h.Q = c.take<double>((size_t)L * d * d);
    w.h.W64 = c.take<double>((size_t)L * r * d);
    w.h.P = c.take<double>((size_t)L * g * d);
    w.h.T = c.take<double>((size_t)L * g * d);
    w.h.V = c.take<double>((size_t)L * g * d);
    w.h.Bneg = c.take<double>((size_t)L * G * g * g);
    w.h.rho = c.take<double>((size_t)L * G);
    w.h.rho_sel = c.take<double>((size_t)L * G);
    w.h.alive = c.take<int>((size_t)L * 2 * G);
    w.h.chosen = c.take<int>((size_t)L);
    const size_t z0 = c.off;                               // zeroed together
    w.h.dw2 = c.take<double>((size_t)L * (n_levels + 1));
    w.h.steps_of = c.take<int>((size_t)n_levels);
    w.zero = w.h.dw2;
    w.zero_bytes = c.off - z0;
    w.lam = c.take<double>((size_t)L);
    w.inv_bytes = inverse_workspace_bytes(L, d);
    if (gram_on_i8(L, r, d, g)) w.inv_bytes = max(w.inv_bytes, carve_i8_operand(nullptr, nullptr, L, d, r));
    w.inv_ws = c.take<char>(w.inv_bytes);
    w.total = c.off;
    return w;
}

template <int G8>
ziplm_status run_heads(HeadsWs& ws, float damp_frac, const int* levels, float* loss, float* base_loss,
                       cudaStream_t st) {
    Heads& w = ws.h;
    const int L = w.L, G = w.G, g = 8 * G8, n_levels = w.n_levels;
    constexpr int smem = (int)HeadShape<G8>::kSmem;
    ziplm_status s;
    {
        PhaseScope ps(PH_INVERSE, st);
        s = run_damped_inverse(w.H, L, w.d, damp_frac, w.A, nullptr, 0, 0, nullptr, ws.lam, w.layer_status,
                               ws.inv_ws, ws.inv_bytes, st);
    }
    if (s != ZIPLM_OK) return s;
    const int n_steps = n_levels > 0 ? G - levels[n_levels - 1] : 0;
    int slot = 0;
    {
        PhaseScope ps(PH_INIT, st);
        ZIPLM_CHECK_CUDA(cudaMemsetAsync(w.order, 0xFF, sizeof(int) * (size_t)L * G, st));
        if (w.saliency) ZIPLM_CHECK_CUDA(cudaMemsetAsync(w.saliency, 0, sizeof(float) * (size_t)L * G, st));
        ZIPLM_CHECK_CUDA(cudaMemsetAsync(ws.zero, 0, ws.zero_bytes, st));
        k_heads_init<<<4 * kSMs, HT, 0, st>>>(w);
        ZIPLM_CHECK_LAUNCH();
        if (n_steps > 0 || base_loss) {
            if (gram_on_i8(L, w.r, w.d, g)) {
                I8Operand x;
                carve_i8_operand(&x, ws.inv_ws, L, w.d, w.r);        // the inverse is done with it
                s = i8_digits_of_columns(x, w.W, (size_t)w.r * w.d, w.d, w.r, w.d, L, st);
                if (s != ZIPLM_OK) return s;
                I8Product p = {};
                p.alpha = 1.0; p.krange = K_ALL; p.lower = 1;
                p.d = w.d; p.out64 = w.Q; p.layer_status = w.layer_status;
                s = i8_product(x, x, p, L, st);
                if (s != ZIPLM_OK) return s;
            } else {
                ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_heads_gram<G8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      smem));
                k_heads_gram<G8><<<dim3(G * (G + 1) / 2, L), HT, smem, st>>>(w);
                ZIPLM_CHECK_LAUNCH();
            }
            if (base_loss) {
                k_heads_base<<<dim3(min(64, w.d), L), HT, 0, st>>>(w);
                ZIPLM_CHECK_LAUNCH();
            }
        }
        if (n_levels > 0 && levels[0] == G) {              // the unpruned level: loss 0
            const size_t n = (size_t)w.r * w.d;
            for (int l = 0; l < L; ++l)
                ZIPLM_CHECK_CUDA(cudaMemcpyAsync(w.W_snap + (size_t)l * n_levels * n, w.W + l * n, n * sizeof(float),
                                                 cudaMemcpyDeviceToDevice, st));
            ++slot;
        }
    }
    if (n_steps > 0) {
        PhaseScope ps(PH_BLOCK_SCORE, st);
        ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_heads_score<G8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        k_heads_score<G8><<<dim3(G, L), HT, smem, st>>>(w);
        ZIPLM_CHECK_LAUNCH();
    }
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_heads_solve<G8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_heads_update<G8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const int ctas = G * (G + 1) / 2 + G * ((w.r + g - 1) / g);
    for (int t = 0; t < n_steps; ++t) {
        {
            PhaseScope ps(PH_BLOCK_SCORE, st);
            if ((s = launch_dependent(k_heads_solve<G8>, dim3(G, L), HT, smem, st, w, t)) != ZIPLM_OK) return s;
        }
        const bool level = levels[slot] == G - t - 1;
        if (G - t > 1 || level) {
            PhaseScope ps(PH_BLOCK_UPDATE, st);
            s = launch_dependent(k_heads_update<G8>, dim3((unsigned)ctas * (unsigned)L), HT, smem, st, w, t,
                                 level ? slot : -1, t + 1 < n_steps ? 1 : 0);
            if (s != ZIPLM_OK) return s;
        }
        if (level) ++slot;
    }
    k_heads_loss<<<L, 32, 0, st>>>(w, ws.lam, loss, base_loss);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace

bool heads_path_supported(int g) { return g >= 32 && g <= 128 && g % 16 == 0; }

size_t heads_workspace_bytes(int L, int r, int d, int g, int n_levels) {
    return carve_heads(nullptr, L, r, d, g, n_levels).total;
}

ziplm_status run_prune_heads(const float* W, const float* H, int L, int r, int d, int g, float damp_frac,
                             const int* levels, int n_levels, float* W_snap, float* loss, float* base_loss,
                             int* order, float* saliency, int* layer_status, void* ws, size_t ws_bytes,
                             cudaStream_t st) {
    if (!heads_path_supported(g)) return ZIPLM_ERR_UNSUPPORTED;
    HeadsWs w = carve_heads(ws, L, r, d, g, n_levels);
    if (ws_bytes < w.total) return ZIPLM_ERR_WORKSPACE;
    w.h.W = W; w.h.H = H; w.h.W_snap = W_snap; w.h.order = order; w.h.saliency = saliency;
    w.h.pairs = (reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(W_snap)) % 8 == 0;    // g is even
    w.h.layer_status = layer_status;
    switch (g / 8) {
        case 4: return run_heads<4>(w, damp_frac, levels, loss, base_loss, st);
        case 6: return run_heads<6>(w, damp_frac, levels, loss, base_loss, st);
        case 8: return run_heads<8>(w, damp_frac, levels, loss, base_loss, st);
        case 10: return run_heads<10>(w, damp_frac, levels, loss, base_loss, st);
        case 12: return run_heads<12>(w, damp_frac, levels, loss, base_loss, st);
        case 14: return run_heads<14>(w, damp_frac, levels, loss, base_loss, st);
        default: return run_heads<16>(w, damp_frac, levels, loss, base_loss, st);
    }
}

}  // namespace ziplm
