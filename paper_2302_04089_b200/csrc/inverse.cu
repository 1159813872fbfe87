// Damped float64 inverse of the calibration Hessian (caption of Algorithm 1:
// H^-1 = (2 X X^T + lambda I)^-1), batched over layers.
//
// Route: H + lambda I = F F^T (Cholesky), M = F^-1, H^-1 = M^T M, all on 64 x 64 tiles.  The
// factor and its inverse are built together by recursive halving of the tile range [lo, hi):
//     factor [lo, mid);   F21 = A21 M11^T;   A22 -= F21 F21^T;   factor [mid, hi);
//     M21 = -M22 (F21 M11)
// so that nearly all of the work sits in large, wide products (thousands of independent tiles
// per launch) and only the 64 x 64 leaves are sequential.  Everything has float64 accuracy: the
// greedy loop that follows needs the diagonal of H^-1 to roughly 1e-7 relative, which an fp32
// factorisation of a matrix with condition number 1e3 .. 1e5 does not give.  Products of blocks of
// at least eight tiles a side run in digits on the int8 tensor cores (inverse_i8.cu), the others and
// the ranges of up to four tiles on the float64 instruction.  The matrix is padded to a multiple of
// 64 with an identity block, whose inverse is again the identity.
#include <cooperative_groups.h>
#include <math.h>

#include <mutex>

#include "common.cuh"
#include "damping.cuh"
#include "factor16.cuh"
#include "inverse_i8.cuh"

// Built-in scratch of ziplm_damped_inverse_noalloc: lives in every GPU that loads this library
// until the process exits.  In host code this name is only a handle for cudaGetSymbolAddress,
// never a device address.
constexpr size_t kBuiltinScratchBytes = (size_t)12 << 20;
static __device__ __align__(256) unsigned char g_builtin_scratch[kBuiltinScratchBytes];

namespace ziplm {
namespace {
constexpr int KC = 16;          // k-chunk staged in shared memory per pipeline stage
constexpr int MTM = 128;        // rows of the macro tile one CTA computes (two tiles)
constexpr int MTN = 64;         // columns of the macro tile (one tile)
constexpr int GT = 256;         // threads of a product CTA: 8 warps, 32 x 32 outputs per warp; two CTAs per SM
constexpr int kSmallThreads = 512;   // threads of the base-case kernel
constexpr int kStages = 3;      // cp.async pipeline depth
// Shared-memory pitches (doubles).  All are 4 mod 16, so that the 16 threads of a half-warp
// (4 m-indices x 4 k-indices of an operand fragment) hit 16 different 8-byte banks, and all keep
// rows 16-byte aligned for cp.async.
constexpr int P_MK = KC + 4;    // chunk stored [m][k] (k contiguous in global memory)
__host__ __device__ constexpr int pitch_km(int rows) { return rows + 4; }   // chunk stored [k][m] (m contiguous)
__host__ __device__ constexpr int stage_doubles(int rows) {
    return rows * P_MK > KC * pitch_km(rows) ? rows * P_MK : KC * pitch_km(rows);
}
constexpr int kStageA = stage_doubles(MTM), kStageB = stage_doubles(MTN);
constexpr size_t kProductSmemBytes = sizeof(double) * kStages * (kStageA + kStageB);

__device__ __forceinline__ void cp_async16(double* smem_dst, const double* gmem_src) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Start the copy of one ROWS x KC operand chunk into a pipeline stage; rows m >= m_valid (tiles
// beyond the edge of the task) are not touched.
//   KM == false: op(m,k) = P[m*ld + k], kept as s[m][k] (pitch P_MK);
//   KM == true : op(m,k) = P[k*ld + m], kept as s[k][m] (pitch ROWS + 4).
template <bool KM, int ROWS>
__device__ __forceinline__ void chunk_async(double* s, const double* P, int ld, int k0, int m_valid) {
    constexpr int PIECES = ROWS * KC / 2;                 // pieces of 16 bytes
#pragma unroll
    for (int e = 0; e < PIECES / GT; ++e) {
        const int piece = threadIdx.x + e * GT;
        if (KM) {
            const int k = piece / (ROWS / 2), m = (piece % (ROWS / 2)) * 2;
            if (m < m_valid) cp_async16(s + k * pitch_km(ROWS) + m, P + (size_t)(k0 + k) * ld + m);
        } else {
            const int m = piece >> 3, k = (piece & 7) * 2;
            if (m < m_valid) cp_async16(s + m * P_MK + k, P + (size_t)m * ld + k0 + k);
        }
    }
}

// Operand fragment of the k-step kk (4 k's) for the 8 m-indices starting at m0.
template <bool KM, int ROWS>
__device__ __forceinline__ double frag(const double* s, int m0, int kk, int lane) {
    return KM ? s[(kk * 4 + (lane & 3)) * pitch_km(ROWS) + m0 + (lane >> 2)]
              : s[(m0 + (lane >> 2)) * P_MK + kk * 4 + (lane & 3)];
}

// Accumulators of one warp: 4 x 4 fragments of 8 x 8 = a 32 x 32 block of the macro tile.
struct WarpAcc {
    double d[4][4][2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) d[i][j][0] = d[i][j][1] = 0.0;
    }
};

// acc(128 x 64 macro tile) += opA(128 x K) opB(K x 64) over the tile range [kt_lo, kt_hi) of K (in
// tiles of 64), operands streamed through a three-stage cp.async pipeline with one barrier per
// chunk.  Warp w owns rows 32 (w / 2) .. and columns 32 (w % 2) .. of the macro tile and only
// multiplies the chunks of its own range [my_lo, my_hi) (the triangular operands cut the range
// per 64 x 64 tile; what the other warps' ranges bring into shared memory may be uninitialised
// and is never read by this warp).  rows_valid crops the macro tile at the edge of the task.
// A and B point at k = 0 of the macro tile's rows / columns.
//   TA == false: A stored m x K row-major; true: stored K x m.
//   TB == false: B stored K x n row-major; true: stored n x K.
// The operand pointers are deliberately not __restrict__: callers read tiles written earlier in
// the same launch sequence.
template <bool TA, bool TB>
__device__ __forceinline__ void dgemm_macro(WarpAcc& acc, const double* A, int lda, const double* B,
                                            int ldb, int kt_lo, int kt_hi, int my_lo, int my_hi,
                                            int rows_valid, double* smem) {
    constexpr bool KA = TA, KB = !TB;       // orientation in memory: true = stored K x m
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = 32 * (warp >> 1), c0 = 32 * (warp & 1);
    double* sa = smem;
    double* sb = smem + kStages * kStageA;
    const int nchunks = (kt_hi - kt_lo) * (kTile / KC);
    const int kbase = kt_lo * kTile;
    for (int c = 0; c < kStages - 1; ++c) {
        if (c < nchunks) {
            chunk_async<KA, MTM>(sa + c * kStageA, A, lda, kbase + c * KC, rows_valid);
            chunk_async<KB, MTN>(sb + c * kStageB, B, ldb, kbase + c * KC, MTN);
        }
        cp_async_commit();
    }
    for (int c = 0; c < nchunks; ++c) {
        cp_async_wait<kStages - 2>();       // chunk c has landed (this thread's pieces)
        __syncthreads();                    // ... everyone's; and chunk c - 1 has been consumed
        const int nx = c + kStages - 1;
        if (nx < nchunks) {
            const int st = nx % kStages;
            chunk_async<KA, MTM>(sa + st * kStageA, A, lda, kbase + nx * KC, rows_valid);
            chunk_async<KB, MTN>(sb + st * kStageB, B, ldb, kbase + nx * KC, MTN);
        }
        cp_async_commit();
        const int ktile = kt_lo + c / (kTile / KC);
        if (ktile < my_lo || ktile >= my_hi) continue;
        const double* pa = sa + (c % kStages) * kStageA;
        const double* pb = sb + (c % kStages) * kStageB;
#pragma unroll
        for (int kk = 0; kk < KC / 4; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = frag<KA, MTM>(pa, r0 + 8 * i, kk, lane);
                b[i] = frag<KB, MTN>(pb, c0 + 8 * i, kk, lane);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dmma884(acc.d[i][j], a[i], b[j]);
        }
    }
    cp_async_wait<0>();
}

// Macro tiles (I, J) of a lower-triangular region of T x T tiles: row block I (tiles 2I, 2I+1)
// meets the column tiles J <= 2I + 1.  Count, and linear index -> (I, J) in row-block order.
__host__ __device__ inline int lower_macro_count(int T) {
    int n = 0;
    for (int I = 0; 2 * I < T; ++I) n += (2 * I + 2 < T) ? 2 * I + 2 : T;
    return n;
}
__device__ __forceinline__ void lower_macro_index(int idx, int T, int& I, int& J) {
    I = 0;
    for (;;) {
        const int w = (2 * I + 2 < T) ? 2 * I + 2 : T;
        if (idx < w) break;
        idx -= w; ++I;
    }
    J = idx;
}

// eq (may be null): powers of two that bring the diagonal of the damped matrix to [1, 4).
// lambda[l] = damp_frac * mean(diag H[l]); flags non-finite diagonals and non-positive means.
__global__ void __launch_bounds__(256) k_mean_diag(const float* __restrict__ H, int d,
                                                   float damp_frac, double* __restrict__ lam,
                                                   double* __restrict__ eq, int* layer_status) {
    const int l = blockIdx.x;
    const float* Hl = H + (size_t)l * d * d;
    const double lm = mean_diag_lambda(Hl, d, damp_frac, layer_status, l, true);
    if (threadIdx.x == 0) lam[l] = lm;
    if (!eq) return;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        const int hi = __double2hiint((double)Hl[(size_t)i * d + i] + lm), e = hi >> 20;
        const int half = (e - 1023) >> 1;
        eq[(size_t)l * d + i] = e > 0 && e < 2047 ? __hiloint2double((1023 - half) << 20, 0) : 1.0;
    }
}

// C = H + lambda I on the d x d corner, identity on the padding (dp x dp, float64); with eq, rows and columns
// scaled by it (exactly).  All of H is read, for the check, but of C only what is used is written: the factorisation
// works on the lower tiles, and its products reach up to 256 columns behind the diagonal.  A warp takes 128 columns, four
// neighbouring ones a lane (QUADS: 16 bytes of H), and has four rows in flight.  Bound by memory: 24 x 4096 1559 us with
// single elements and all of C written, 574 now (5.6 TB/s).
constexpr int FILL_COLS = 128, FILL_ROWS = 32, FILL_BAND = 256;      // (tiles of a product on the diagonal: 256 wide)
template <bool QUADS>
__global__ void __launch_bounds__(256) k_fill_damped(const float* __restrict__ H, int d, int dp,
                                                     const double* __restrict__ lam,
                                                     const double* __restrict__ eq,
                                                     double* __restrict__ C, int* layer_status) {
    const int l = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row0 = blockIdx.y * FILL_ROWS + warp, col = blockIdx.x * FILL_COLS + 4 * lane;
    if (col >= dp) return;                       // (dp and col are multiples of four)
    const float* Hl = H + (size_t)l * d * d;
    double* Cl = C + (size_t)l * dp * dp;
    const double lm = lam[l];
    double ec[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) ec[q] = eq && col + q < d ? eq[(size_t)l * d + col + q] : 1.0;
    float h[FILL_ROWS / 8][4];
#pragma unroll
    for (int k = 0; k < FILL_ROWS / 8; ++k) {
        const int row = row0 + 8 * k;
        const float* from = Hl + (size_t)row * d + col;
        if (QUADS) {
            const float4 x = row < d && col < d ? __ldcs(reinterpret_cast<const float4*>(from)) : make_float4(0.f, 0.f, 0.f, 0.f);
            h[k][0] = x.x; h[k][1] = x.y; h[k][2] = x.z; h[k][3] = x.w;
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) h[k][q] = row < d && col + q < d ? __ldcs(from + q) : 0.f;
        }
    }
    bool bad = false;
#pragma unroll
    for (int k = 0; k < FILL_ROWS / 8; ++k) {
        const int row = row0 + 8 * k;
        if (row >= dp) break;
        const double er = eq && row < d ? eq[(size_t)l * d + row] : 1.0;
        double v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (!isfinite(h[k][q])) bad = true;
            const bool in = row < d && col + q < d;
            v[q] = in ? ((double)h[k][q] + (row == col + q ? lm : 0.0)) * (er * ec[q]) : row == col + q ? 1.0 : 0.0;
        }
        if (col >= row + FILL_BAND) continue;
        double2* to = reinterpret_cast<double2*>(Cl + (size_t)row * dp + col);
        to[0] = make_double2(v[0], v[1]);
        to[1] = make_double2(v[2], v[3]);
    }
    if (bad) set_layer_status(layer_status, l, ZIPLM_ERR_NONFINITE);
}

// One launch of the recursion: C_out[tile (ti,tj)] = beta * C_out + alpha * sum_k opA(ti,k) opB(k,tj)
// over a rectangle of mt x nt tiles, with the k range cut to the non-zero tiles of a triangular
// operand.  All matrices are dp x dp float64 per layer; coordinates are in tiles.
struct GemmTask {
    const double* A; int a_r, a_c;      // TA == false: tile (ti,k) at (a_r + ti, a_c + k); true: (a_r + k, a_c + ti)
    const double* B; int b_r, b_c;      // TB == false: tile (k,tj) at (b_r + k, b_c + tj); true: (b_r + tj, b_c + k)
    double* C; int c_r, c_c;
    int mt, nt, kt;
    int kmode;                          // 0: all k; 1: k <= tj; 2: k <= ti; 3: k >= tj
    int lower_only;                     // square region: only tiles ti >= tj
    double alpha; int beta;             // beta in {0, 1}
};

// k range (in tiles) of output tile (ti, tj) under the task's kmode.
__device__ __forceinline__ void task_krange(const GemmTask& t, int ti, int tj, int& klo, int& khi) {
    klo = 0; khi = t.kt;
    if (t.kmode == 1) khi = min(t.kt, tj + 1);
    else if (t.kmode == 2) khi = min(t.kt, ti + 1);
    else if (t.kmode == 3) klo = tj;
}

// One CTA per 128 x 64 macro tile (two tiles high); blockIdx.x runs over the macro tiles of the
// task (those that reach the lower triangle when lower_only), blockIdx.y over the layers.
template <bool TA, bool TB>
__device__ __forceinline__ void dgemm_task(const GemmTask& t, int dp, int bx, int l, double* smem) {
    const int mmt = (t.mt + 1) / 2;
    // macro tiles with the longest k range come first, so that the last wave is the lightest
    int I, J;
    if (t.lower_only) lower_macro_index(bx, t.mt, I, J);
    else if (t.kmode == 1) { J = t.nt - 1 - bx / mmt; I = bx % mmt; }
    else if (t.kmode == 3) { J = bx / mmt; I = bx % mmt; }
    else if (t.kmode == 2) { I = mmt - 1 - bx / t.nt; J = bx % t.nt; }
    else { I = bx / t.nt; J = bx % t.nt; }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ti = 2 * I + (warp >> 2), tj = J;                          // this warp's tile
    const bool mine = ti < t.mt && (!t.lower_only || ti >= tj);
    // CTA range: union over its valid tiles; warp range: its own tile's
    int kt_lo = t.kt, kt_hi = 0;
    for (int a = 0; a < 2; ++a) {
        const int si = 2 * I + a;
        if (si >= t.mt || (t.lower_only && si < tj)) continue;
        int lo, hi;
        task_krange(t, si, tj, lo, hi);
        kt_lo = min(kt_lo, lo); kt_hi = max(kt_hi, hi);
    }
    int my_lo = 0, my_hi = 0;
    if (mine) task_krange(t, ti, tj, my_lo, my_hi);
    const int rows_valid = min(MTM, (t.mt - 2 * I) * kTile);
    const size_t lay = (size_t)l * dp * dp;
    const double* A = t.A + lay + (TA ? ((size_t)t.a_r * kTile * dp + (size_t)(t.a_c + 2 * I) * kTile)
                                      : ((size_t)(t.a_r + 2 * I) * kTile * dp + (size_t)t.a_c * kTile));
    const double* B = t.B + lay + (TB ? ((size_t)(t.b_r + J) * kTile * dp + (size_t)t.b_c * kTile)
                                      : ((size_t)t.b_r * kTile * dp + (size_t)(t.b_c + J) * kTile));
    WarpAcc acc;
    acc.zero();
    dgemm_macro<TA, TB>(acc, A, dp, B, dp, kt_lo, kt_hi, my_lo, my_hi, rows_valid, smem);
    if (!mine) return;
    double* out = t.C + lay + (size_t)((t.c_r + 2 * I) * kTile + 32 * (warp >> 1)) * dp +
                  (size_t)(t.c_c + J) * kTile + 32 * (warp & 1);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        double2* o = reinterpret_cast<double2*>(out + (size_t)(8 * i + (lane >> 2)) * dp + 2 * (lane & 3));
        double2 cur[4];                        // four old values in flight, not each behind the store before it
#pragma unroll
        for (int j = 0; j < 4; ++j) cur[j] = t.beta ? o[4 * j] : make_double2(0.0, 0.0);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o[4 * j] = make_double2(fma(t.alpha, acc.d[i][j][0], cur[j].x), fma(t.alpha, acc.d[i][j][1], cur[j].y));
    }
}

template <bool TA, bool TB>
__global__ void __launch_bounds__(GT, 2) k_dgemm_tiles(GemmTask t, int dp) {
    extern __shared__ __align__(16) double smem[];
    dgemm_task<TA, TB>(t, dp, blockIdx.x, blockIdx.y, smem);
}

// Two independent products in one launch: the first n1 CTAs of a layer run t1 (A B^T form), the
// rest t2 (A B form).  Used for A22 -= F21 F21^T and scratch = F21 M11, which both depend on F21
// only: one launch fills the other's last wave.
__global__ void __launch_bounds__(GT, 2) k_dgemm_pair(GemmTask t1, int n1, GemmTask t2, int dp) {
    extern __shared__ __align__(16) double smem[];
    if ((int)blockIdx.x < n1) dgemm_task<false, true>(t1, dp, blockIdx.x, blockIdx.y, smem);
    else dgemm_task<false, false>(t2, dp, blockIdx.x - n1, blockIdx.y, smem);
}

// ---- base case of the recursion: a range of up to kSmallMax tiles, one cluster per layer -------
constexpr int kSmallMax = 4;
constexpr int PS = kTile + 4;    // pitch of a 64 x 64 operand tile in shared memory (4 mod 16)

struct SmallSmem {
    double ta[kTile * PS];       // operand tiles, as stored (row-major)
    double tb[kTile * PS];
    double blk[16 * 20];         // leaf: inverse factor of the current 16 x 16 diagonal block
    int flag;                    // first error seen by this CTA
};

// Start the copy of a 64 x 64 tile (row-major, leading dimension ld) into a shared-memory tile.
__device__ __forceinline__ void tile_async(double* dst, const double* src, int ld) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int piece = threadIdx.x + e * kSmallThreads;            // 2048 pieces of 16 bytes
        const int r = piece >> 5, c = (piece & 31) * 2;
        cp_async16(dst + r * PS + c, src + (size_t)r * ld + c);
    }
}

// Fragment of a shared-memory tile: KM == false: op(m,k) = s[m][k]; true: op(m,k) = s[k][m].
template <bool KM>
__device__ __forceinline__ double tile_frag(const double* s, int m0, int kk, int lane) {
    return KM ? s[(kk * 4 + (lane & 3)) * PS + m0 + (lane >> 2)]
              : s[(m0 + (lane >> 2)) * PS + kk * 4 + (lane & 3)];
}

// Accumulators of one warp of the small kernel: 2 x 2 fragments = a 16 x 16 block of a tile;
// warp w owns rows 16 (w / 4) .. and columns 16 (w % 4) ...
struct SmallAcc {
    double d[2][2][2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) d[i][j][0] = d[i][j][1] = 0.0;
    }
};

// acc += opA(64 x 64) opB(64 x 64), both operands in shared memory.
//   AKM: opA(m,k) = sa[k][m], else sa[m][k];  BKN: opB(k,n) = sb[k][n], else sb[n][k].
template <bool AKM, bool BKN>
__device__ __forceinline__ void tile_mma(SmallAcc& acc, const double* sa, const double* sb) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = 16 * (warp >> 2), c0 = 16 * (warp & 3);
#pragma unroll 4
    for (int kk = 0; kk < kTile / 4; ++kk) {
        double a[2], b[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            a[i] = tile_frag<AKM>(sa, r0 + 8 * i, kk, lane);
            b[i] = tile_frag<BKN>(sb, c0 + 8 * i, kk, lane);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) dmma884(acc.d[i][j], a[i], b[j]);
    }
}

// Visit the elements of a warp's accumulators: f(row, col, pair) with col even.
template <typename Fn>
__device__ __forceinline__ void small_epilogue(const SmallAcc& acc, Fn f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r0 = 16 * (warp >> 2) + (lane >> 2), c0 = 16 * (warp & 3) + 2 * (lane & 3);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
            f(r0 + 8 * i, c0 + 8 * j, make_double2(acc.d[i][j][0], acc.d[i][j][1]));
}

// Leaf: the inverse M of the Cholesky factor of the 64 x 64 tile at Ag (null: it is in sm.ta) -> Mg (lower, upper
// part zeroed), and left in sm.tb.  The factor itself is not needed.  Starts and ends with a barrier.
// The same elimination by 16 x 16 blocks: one warp turns the diagonal block into M_bb, then
// L_ib = A_ib M_bb^T and X_bj = M_bb X_bj, then A_ik -= L_ib L_kb^T and X_ij -= L_ib X_bj, a warp and 16
// float64 mma instructions per block.  Warp 0 updates the next diagonal block and goes on with it while
// the others do the rest: two barriers a block.  15000 clocks, of which 4 x 2200 are the chain of the
// pivots; column by column on all threads it was 36000, 560 a column (a barrier, ten shared-memory reads
// and the CTA's instructions on every column's chain).  12 x 1024 inverse 0.87 -> 0.78 ms.
__device__ __forceinline__ void leaf_factor(const double* Ag, double* Mg, int dp, SmallSmem& sm) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    __syncthreads();                          // earlier readers of the shared arrays are done
#pragma unroll
    for (int e = tid; e < kTile * kTile; e += kSmallThreads) {
        const int i = e >> 6, j = e & 63;     // the lower triangle is the valid one
        if (Ag && j <= i) {
            const double v = Ag[(size_t)i * dp + j];
            sm.ta[i * PS + j] = v;
            sm.ta[j * PS + i] = v;
        }
        sm.tb[i * PS + j] = 0.0;
    }
    __syncthreads();
    auto A = [&](int i, int j) { return sm.ta + 16 * i * PS + 16 * j; };
    auto X = [&](int i, int j) { return sm.tb + 16 * i * PS + 16 * j; };
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        if (warp == 0) {                      // warp 0 updated A_bb itself and goes on without a barrier
            __syncwarp();
            const int flag = warp_factor16(A(b, b), PS, sm.blk);
            if (lane == 0 && flag && !sm.flag) sm.flag = flag;
        }
        __syncthreads();
        const int n = 3 - b;
        double acc[2][2][2] = {};
        if (warp < n) {                                       // L_ib, in A's place
            double* a = A(b + 1 + warp, b);
            warp_mma16<true>(acc, a, PS, sm.blk, PB);
            __syncwarp();
            warp_put16<false>(acc, a, PS);
        } else if (warp < n + b) {
            double* x = X(b, warp - n);
            warp_mma16<false>(acc, sm.blk, PB, x, PS);
            __syncwarp();
            warp_put16<false>(acc, x, PS);
        } else if (warp == 3) {
            for (int e = lane; e < 256; e += 32) X(b, b)[(e >> 4) * PS + (e & 15)] = sm.blk[(e >> 4) * PB + (e & 15)];
        }
        __syncthreads();
        const int n_a = n * (n + 1) / 2;
        if (warp < n_a) {
            int ii = 0, kk = warp;
            while (kk > ii) { kk -= ii + 1; ++ii; }
            const int i = b + 1 + ii, k = b + 1 + kk;
            double c[2][2][2] = {};
            warp_mma16<true>(c, A(i, b), PS, A(k, b), PS);
            warp_put16<true>(c, A(i, k), PS);
        } else if (warp < n_a + n * (b + 1)) {
            const int q = warp - n_a, i = b + 1 + q / (b + 1), j = q % (b + 1);
            double c[2][2][2] = {};
            warp_mma16<false>(c, A(i, b), PS, X(b, j), PS);
            warp_put16<true>(c, X(i, j), PS);
        }
    }
#pragma unroll
    for (int e = tid; e < kTile * kTile; e += kSmallThreads)
        Mg[(size_t)(e >> 6) * dp + (e & 63)] = sm.tb[(e >> 6) * PS + (e & 63)];
    __syncthreads();
}

// Factor the tile range [lo, lo + nt), nt <= kSmallMax, of every layer with one cluster of four CTAs per
// layer: right-looking elimination of [A | I] by tiles.  Stage j: rank 0 turns the diagonal tile into
// M_jj; then F_ij = A_ij M_jj^T below it and M_jk = M_jj X_jk left of it; then A_ik -= F_ij F_kj^T and
// X_ik -= F_ij M_jk (X_ik, kept in M's tile, is what M_ik is before its own row's stage).  The tiles of a
// phase are independent and dealt out to the ranks; rank 0 updates the next diagonal tile first, out of its own
// F and without a detour through memory, and goes on to its leaf without waiting for the others, so the chain is
// leaf, two products, leaf, ...: one cluster barrier a stage, and the arrival at another.  Every product is a
// 64 x 64 x 64 tile product of a whole CTA on the float64 tensor core, its operands fetched from global memory (the
// L2) into shared memory; on one CTA alone the 32 products of four tiles took 150 us of 184.
constexpr int kSmallCluster = 4;
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__global__ void __launch_bounds__(kSmallThreads, 1) k_factor_small(double* A, double* F, double* M, int dp, int lo,
                                                        int nt, int* layer_status) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem& sm = *reinterpret_cast<SmallSmem*>(smem_raw);
    const int rank = (int)cluster.block_rank();
    const int l = blockIdx.x / kSmallCluster;
    const size_t lay = (size_t)l * dp * dp;
    auto tile = [&](double* base, int i, int j) {
        return base + lay + (size_t)(lo + i) * kTile * dp + (size_t)(lo + j) * kTile;
    };
    if (threadIdx.x == 0) sm.flag = 0;
    // operands into shared memory: ta = x, tb = y
    auto fetch = [&](const double* x, const double* y) {
        __syncthreads();                                   // the previous product's readers are done
        tile_async(sm.ta, x, dp);
        tile_async(sm.tb, y, dp);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
    };
    // what is at `out`: requested before the product that is to be taken from it
    struct Old { double2 v[4]; };
    auto load = [&](const double* out) {
        Old old;
        int e = 0;
        small_epilogue(SmallAcc(), [&](int r, int c, double2) {
            old.v[e++] = *reinterpret_cast<const double2*>(out + (size_t)r * dp + c);
        });
        return old;
    };
    auto store = [&](const SmallAcc& acc, double* out) {
        small_epilogue(acc, [&](int r, int c, double2 v) {
            *reinterpret_cast<double2*>(out + (size_t)r * dp + c) = v;
        });
    };
    auto subtract = [&](const SmallAcc& acc, double* out, const Old& old) {
        int e = 0;
        small_epilogue(acc, [&](int r, int c, double2 v) {
            const double2 cur = old.v[e++];
            *reinterpret_cast<double2*>(out + (size_t)r * dp + c) = make_double2(cur.x - v.x, cur.y - v.y);
        });
    };
    static_assert(kSmallMax <= kSmallCluster, "a rank has one tile of a row and column");
    for (int j = 0; j < nt; ++j) {
        SmallAcc acc;
        if (rank == 0) {
            leaf_factor(j == 0 ? tile(A, j, j) : nullptr, tile(M, j, j), dp, sm);
            if (j > 0) cluster_wait();
        }
        cluster.sync();
        if (rank == 0 && j + 1 < nt) {
            // F_{j+1,j} from the M_jj in shared memory, then the next diagonal tile from that F, into the
            // place where the leaf wants it
            const Old old = load(tile(A, j + 1, j + 1));
            tile_async(sm.ta, tile(A, j + 1, j), dp);
            cp_async_commit();
            cp_async_wait<0>();
            __syncthreads();
            acc.zero();
            tile_mma<false, false>(acc, sm.ta, sm.tb);
            store(acc, tile(F, j + 1, j));
            cluster_arrive();                              // the others need F; rank 0 waits after its leaf
            __syncthreads();
            small_epilogue(acc, [&](int r, int c, double2 v) {
                *reinterpret_cast<double2*>(sm.ta + r * PS + c) = v;
            });
            __syncthreads();
            acc.zero();
            tile_mma<false, false>(acc, sm.ta, sm.ta);
            __syncthreads();
            int e = 0;
            small_epilogue(acc, [&](int r, int c, double2 v) {
                const double2 cur = old.v[e++];
                if (c <= r) sm.ta[r * PS + c] = sm.ta[c * PS + r] = cur.x - v.x;
                if (c + 1 <= r) sm.ta[r * PS + c + 1] = sm.ta[(c + 1) * PS + r] = cur.y - v.y;
            });
            continue;
        }
        // ---- row and column j
        if (rank < nt - 1) {
            acc.zero();
            if (rank < nt - 1 - j) {
                const int i = j + 1 + rank;
                fetch(tile(A, i, j), tile(M, j, j));
                tile_mma<false, false>(acc, sm.ta, sm.tb);
                store(acc, tile(F, i, j));
            } else {
                const int k = rank - (nt - 1 - j);
                fetch(tile(M, j, j), tile(M, j, k));
                tile_mma<false, true>(acc, sm.ta, sm.tb);
                store(acc, tile(M, j, k));
            }
        }
        if (j + 1 == nt) break;
        cluster_arrive();
        cluster_wait();
        // ---- what is behind them: tile 0 is the next diagonal tile and rank 0's
        const int rest = nt - 1 - j, n_a = rest * (rest + 1) / 2, n_all = n_a + rest * (j + 1);
        for (int q = rank; q < n_all; q += kSmallCluster - 1) {
            acc.zero();
            if (q < n_a) {
                int ii = 0, kk = q;
                while (kk > ii) { kk -= ii + 1; ++ii; }
                const int i = j + 1 + ii, k = j + 1 + kk;
                const Old old = load(tile(A, i, k));
                fetch(tile(F, i, j), tile(F, k, j));
                tile_mma<false, false>(acc, sm.ta, sm.tb);
                subtract(acc, tile(A, i, k), old);
            } else {
                const int i = j + 1 + (q - n_a) / (j + 1), k = (q - n_a) % (j + 1);
                Old old = {};
                if (k < j) old = load(tile(M, i, k));
                fetch(tile(F, i, j), tile(M, j, k));
                tile_mma<false, true>(acc, sm.ta, sm.tb);
                subtract(acc, tile(M, i, k), old);
            }
        }
    }
    if (threadIdx.x == 0 && sm.flag) set_layer_status(layer_status, l, sm.flag);
}

// H^-1 = M^T M on the lower tiles (i >= j): sum over k >= i of M_ki^T M_kj; writes the cropped
// d x d result as float64 (mirrored to the upper triangle) and/or fp32 off-diagonal (both
// triangles) + fp64 diag.
// One CTA per 128 x 64 macro tile that reaches the lower triangle.
__global__ void __launch_bounds__(GT, 2) k_lauum(const double* M, int dp, int T, int d, double* out64,
                                                 float* tri32, int pitch32, int rows32, double* diag64) {
    extern __shared__ __align__(16) double smem[];
    const int l = blockIdx.y;
    int I, J;
    lower_macro_index(blockIdx.x, T, I, J);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ti = 2 * I + (warp >> 2), tj = J;
    const bool mine = ti < T && ti >= tj;
    const double* Ml = M + (size_t)l * dp * dp;
    const int rows_valid = min(MTM, (T - 2 * I) * kTile);
    WarpAcc acc;
    acc.zero();
    // (M^T M)_ij: opA(i,k) = M[k][i] (stored K x m), opB(k,j) = M[k][j]; tile (ti, .) starts at k = ti
    dgemm_macro<true, false>(acc, Ml + (size_t)(2 * I) * kTile, dp, Ml + (size_t)J * kTile, dp,
                             2 * I, T, mine ? ti : 0, mine ? T : 0, rows_valid, smem);
    if (!mine) return;
    const int row0 = 2 * I * kTile + 32 * (warp >> 1) + (lane >> 2);
    const int col0 = J * kTile + 32 * (warp & 1) + 2 * (lane & 3);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int row = row0 + 8 * i, col = col0 + 8 * j + e;
                if (row >= d || col >= d) continue;
                const double v = acc.d[i][j][e];
                if (out64 && row >= col) {
                    double* o = out64 + (size_t)l * d * d;
                    o[(size_t)row * d + col] = v;
                    o[(size_t)col * d + row] = v;
                }
                if (tri32 && row > col) {       // both triangles: a column can then be read as a row
                    float* t = tri32 + (size_t)l * rows32 * pitch32;
                    t[(size_t)row * pitch32 + col] = (float)v;
                    t[(size_t)col * pitch32 + row] = (float)v;
                }
                if (diag64 && row == col) diag64[(size_t)l * rows32 + row] = v;
            }
}

struct InvCtx {
    double* A;   // damped Hessian, updated in place (Schur complements); dead blocks serve as scratch
    double* F;   // Cholesky factor
    double* M;   // inverse of the factor
    int dp, L;
    int* layer_status;
    cudaStream_t st;
    const double* eq;      // int8 products: equilibration, and two operands in digits (rows and K set per use)
    I8Operand X, Y;
};

// Products of blocks of at least eight tiles a side, and M^T M from sixteen tiles on, run on the int8 tensor
// cores: below, the passes that write the digits and the few 256 x 128 tiles cost what the products save.
// M^T M sums over the whole width, which the exactness of the int32 sums limits; wider matrices stay on the
// float64 instruction.
constexpr int kI8Tiles = 8;
bool uses_i8(int T) { return T >= 2 * kI8Tiles && T * kTile <= kI8MostK; }

int task_ctas(const GemmTask& t) {
    const int mm = (t.mt + 1) / 2;                           // macro tiles: mm x t.nt
    return t.lower_only ? lower_macro_count(t.mt) : mm * t.nt;
}

ziplm_status launch_pair(const InvCtx& c, const GemmTask& t1, const GemmTask& t2) {
    const int n1 = task_ctas(t1), n2 = task_ctas(t2);
    const cudaError_t attr = cudaFuncSetAttribute(
        k_dgemm_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProductSmemBytes);
    if (attr != cudaSuccess) return ZIPLM_ERR_CUDA;
    PhaseScope ps(PH_INV_PRODUCTS, c.st);
    k_dgemm_pair<<<dim3(n1 + n2, c.L), GT, kProductSmemBytes, c.st>>>(t1, n1, t2, c.dp);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

template <bool TA, bool TB>
ziplm_status launch_gemm(const InvCtx& c, const GemmTask& t) {
    const int ctas = task_ctas(t);
    if (ctas <= 0 || t.kt <= 0) return ZIPLM_OK;
    const cudaError_t attr = cudaFuncSetAttribute(
        k_dgemm_tiles<TA, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProductSmemBytes);
    if (attr != cudaSuccess) return ZIPLM_ERR_CUDA;
    PhaseScope ps(PH_INV_PRODUCTS, c.st);
    k_dgemm_tiles<TA, TB><<<dim3(ctas, c.L), GT, kProductSmemBytes, c.st>>>(t, c.dp);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

// Factor the tile range [lo, hi): on return F holds the Cholesky factor of the (updated) block
// and M its inverse.
ziplm_status factor_range(const InvCtx& c, int lo, int hi) {
    if (hi - lo <= kSmallMax) {
        const cudaError_t attr = cudaFuncSetAttribute(
            k_factor_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem));
        if (attr != cudaSuccess) return ZIPLM_ERR_CUDA;
        PhaseScope ps(PH_INV_LEAVES, c.st);
        // A few CTAs per layer and a long dependent chain: launched at the highest priority, so that
        // it does not queue behind the wide kernels of other layer groups.
        static int prio = [] {
            int least = 0, greatest = 0;
            return cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess ? greatest : 0;
        }();
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c.L * kSmallCluster);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.dynamicSmemBytes = sizeof(SmallSmem);
        cfg.stream = c.st;
        cudaLaunchAttribute la[2];
        la[0].id = cudaLaunchAttributePriority;
        la[0].val.priority = prio;
        la[1].id = cudaLaunchAttributeClusterDimension;
        la[1].val.clusterDim.x = kSmallCluster;
        la[1].val.clusterDim.y = la[1].val.clusterDim.z = 1;
        cfg.attrs = la;
        cfg.numAttrs = 2;
        ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k_factor_small, c.A, c.F, c.M, c.dp, lo, hi - lo,
                                            c.layer_status));
        ZIPLM_CHECK_LAUNCH();
        return ZIPLM_OK;
    }
    const int mid = lo + (hi - lo) / 2;
    const int n1 = mid - lo, n2 = hi - mid;
    ziplm_status s = factor_range(c, lo, mid);
    if (s != ZIPLM_OK) return s;
    if (c.X.dig && n1 >= kI8Tiles && n2 >= kI8Tiles) {
        const size_t lay = (size_t)c.dp * c.dp;
        auto block = [&](double* m, int i, int j) { return m + (size_t)i * kTile * c.dp + (size_t)j * kTile; };
        auto operand = [&](I8Operand o, int rows, int K) { o.rows = rows * kTile; o.K = K * kTile; return o; };
        auto product = [&](const I8Operand& x, const I8Operand& y, double* C, double alpha, int beta, int krange,
                           int lower) {
            I8Product p = {};
            p.C = C; p.layer_stride = lay; p.ld = c.dp;
            p.alpha = alpha; p.beta = beta; p.krange = krange; p.lower = lower;
            p.layer_status = c.layer_status;
            return i8_product(x, y, p, c.L, c.st);
        };
        {
            PhaseScope ps(PH_INV_PRODUCTS, c.st);
            // F21 = A21 M11^T
            I8Operand x = operand(c.X, n2, n1), y = operand(c.Y, n1, n1);
            if ((s = i8_digits(x, block(c.A, mid, lo), lay, c.dp, false, false, c.L, c.st)) != ZIPLM_OK) return s;
            if ((s = i8_digits(y, block(c.M, lo, lo), lay, c.dp, false, true, c.L, c.st)) != ZIPLM_OK) return s;
            if ((s = product(x, y, block(c.F, mid, lo), 1.0, 0, K_TO_COL, 0)) != ZIPLM_OK) return s;
            // A22 -= F21 F21^T, scratch (the dead A21 block) = F21 M11
            if ((s = i8_digits(x, block(c.F, mid, lo), lay, c.dp, false, false, c.L, c.st)) != ZIPLM_OK) return s;
            if ((s = product(x, x, block(c.A, mid, mid), -1.0, 1, K_ALL, 1)) != ZIPLM_OK) return s;
            if ((s = i8_digits(y, block(c.M, lo, lo), lay, c.dp, true, true, c.L, c.st)) != ZIPLM_OK) return s;
            if ((s = product(x, y, block(c.A, mid, lo), 1.0, 0, K_FROM_COL, 0)) != ZIPLM_OK) return s;
        }
        if ((s = factor_range(c, mid, hi)) != ZIPLM_OK) return s;
        PhaseScope ps(PH_INV_PRODUCTS, c.st);
        // M21 = -M22 scratch
        I8Operand x = operand(c.X, n2, n2), y = operand(c.Y, n1, n2);
        if ((s = i8_digits(x, block(c.M, mid, mid), lay, c.dp, false, true, c.L, c.st)) != ZIPLM_OK) return s;
        if ((s = i8_digits(y, block(c.A, mid, lo), lay, c.dp, true, false, c.L, c.st)) != ZIPLM_OK) return s;
        return product(x, y, block(c.M, mid, lo), -1.0, 0, K_TO_ROW, 0);
    }
    GemmTask t;
    // F21 = A21 M11^T   (M11 lower triangular: opB(k,j) = M11[j,k] vanishes for k > j)
    t = GemmTask{c.A, mid, lo, c.M, lo, lo, c.F, mid, lo, n2, n1, n1, 1, 0, 1.0, 0};
    if ((s = launch_gemm<false, true>(c, t)) != ZIPLM_OK) return s;
    // A22 -= F21 F21^T  (lower tiles), and in the same launch
    // scratch (the dead A21 block) = F21 M11   (M11 lower: opB(k,j) vanishes for k < j):
    // its operands are final here and only the M21 product below reads it
    {
        const GemmTask syrk{c.F, mid, lo, c.F, mid, lo, c.A, mid, mid, n2, n2, n1, 0, 1, -1.0, 1};
        const GemmTask scr{c.F, mid, lo, c.M, lo, lo, c.A, mid, lo, n2, n1, n1, 3, 0, 1.0, 0};
        if ((s = launch_pair(c, syrk, scr)) != ZIPLM_OK) return s;
    }
    if ((s = factor_range(c, mid, hi)) != ZIPLM_OK) return s;
    // M21 = -M22 scratch  (M22 lower: opA(i,k) vanishes for k > i)
    t = GemmTask{c.M, mid, mid, c.A, mid, lo, c.M, mid, lo, n2, n1, n2, 2, 0, -1.0, 0};
    return launch_gemm<false, false>(c, t);
}

}  // namespace

namespace {

// Carves the workspace; with ws == nullptr it only measures.
size_t carve_inverse(InvCtx* ctx, double** lam, double** eq, void* ws, int L, int d) {
    const int dp = round_up_int(d, kTile), T = dp / kTile;
    Carver c(ws);
    ctx->A = c.take<double>((size_t)L * dp * dp);      // damped Hessian / Schur complements
    ctx->F = c.take<double>((size_t)L * dp * dp);      // off-diagonal blocks of the Cholesky factor
    ctx->M = c.take<double>((size_t)L * dp * dp);      // inverse of the factor
    *lam = c.take<double>((size_t)L);
    *eq = nullptr;
    ctx->X = ctx->Y = I8Operand{};
    if (uses_i8(T)) {
        const size_t h = (size_t)(T - T / 2) * kTile;  // the widest blocks: both halves of the whole range
        *eq = c.take<double>((size_t)L * d);
        for (I8Operand* o : {&ctx->X, &ctx->Y}) {
            o->dig = c.take<signed char>((size_t)L * 8 * h * h);
            o->scale = c.take<double>((size_t)L * dp);
            o->exps = c.take<int>((size_t)L * dp);
        }
    }
    ctx->eq = *eq;
    ctx->dp = dp;
    ctx->L = L;
    return c.off;
}

// Factorisation of ctx.A and M^T M.
ziplm_status invert(const InvCtx& ctx, int d, double* out64, float* tri32, int pitch32, int rows32,
                    double* diag64) {
    const int T = ctx.dp / kTile;
    const ziplm_status s = factor_range(ctx, 0, T);
    if (s != ZIPLM_OK) return s;
    PhaseScope ps(PH_INV_LAUUM, ctx.st);
    if (ctx.X.dig) {
        // the digits of all of M take the place of the dead A
        const size_t lay = (size_t)ctx.dp * ctx.dp;
        I8Operand x = ctx.X;
        x.dig = reinterpret_cast<signed char*>(ctx.A);
        x.rows = x.K = ctx.dp;
        const ziplm_status e = i8_digits(x, ctx.M, lay, ctx.dp, true, true, ctx.L, ctx.st);
        if (e != ZIPLM_OK) return e;
        I8Product p = {};
        p.alpha = 1.0; p.krange = K_FROM_ROW; p.lower = 1;
        p.d = d; p.eq = ctx.eq; p.out64 = out64; p.tri32 = tri32; p.pitch32 = pitch32; p.rows32 = rows32;
        p.diag64 = diag64; p.layer_status = ctx.layer_status;
        return i8_product(x, x, p, ctx.L, ctx.st);
    }
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_lauum, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kProductSmemBytes));
    k_lauum<<<dim3(lower_macro_count(T), ctx.L), GT, kProductSmemBytes, ctx.st>>>(ctx.M, ctx.dp, T, d, out64, tri32,
                                                                                pitch32, rows32, diag64);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace

size_t inverse_workspace_bytes(int L, int d) {
    InvCtx ctx = {};
    double *lam, *eq;
    return carve_inverse(&ctx, &lam, &eq, nullptr, L, d);
}

double* inverse_matrix(void* ws) { return static_cast<double*>(ws); }     // the first piece of the workspace

ziplm_status run_inverse_of(void* ws, int L, int d, double* out64, int* layer_status, cudaStream_t st) {
    InvCtx ctx = {};
    double *lam, *eq;
    carve_inverse(&ctx, &lam, &eq, ws, L, d);
    ctx.layer_status = layer_status;
    ctx.st = st;
    ctx.eq = nullptr;
    ctx.X.dig = nullptr;               // the caller's matrix is not equilibrated
    return invert(ctx, d, out64, nullptr, 0, 0, nullptr);
}

ziplm_status run_damped_inverse(const float* H, int L, int d, float damp_frac, double* out64,
                                float* tri32, int pitch32, int rows32, double* diag64, double* lam_out,
                                int* layer_status, void* ws, size_t ws_bytes, cudaStream_t st) {
    if (ws_bytes < inverse_workspace_bytes(L, d)) return ZIPLM_ERR_WORKSPACE;
    InvCtx ctx = {};
    double *lam, *eq;
    carve_inverse(&ctx, &lam, &eq, ws, L, d);
    ctx.layer_status = layer_status;
    ctx.st = st;
    k_mean_diag<<<L, 256, 0, st>>>(H, d, damp_frac, lam, eq, layer_status);
    ZIPLM_CHECK_LAUNCH();
    const bool quads = d % 4 == 0 && reinterpret_cast<uintptr_t>(H) % 16 == 0;
    auto fill = quads ? k_fill_damped<true> : k_fill_damped<false>;
    fill<<<dim3((ctx.dp + FILL_COLS - 1) / FILL_COLS, (ctx.dp + FILL_ROWS - 1) / FILL_ROWS, L), 256, 0, st>>>(
        H, d, ctx.dp, lam, eq, ctx.A, layer_status);
    ZIPLM_CHECK_LAUNCH();
    const ziplm_status s = invert(ctx, d, out64, tri32, pitch32, rows32, diag64);
    if (s != ZIPLM_OK) return s;
    if (lam_out) {
        ZIPLM_CHECK_CUDA(cudaMemcpyAsync(lam_out, lam, sizeof(double) * L, cudaMemcpyDeviceToDevice, st));
    }
    return ZIPLM_OK;
}

}  // namespace ziplm

// ---------------------------------------------------------------------------------------------
// Variant of the damped inverse for callers that cannot allocate device memory.
namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_addr[kMaxDevices] = {};   // device address of g_builtin_scratch, per device
}  // namespace

extern "C" ziplm_status ziplm_damped_inverse_noalloc(const float* H, int L, int d, float damp_frac,
                                                     double* Hinv, int* layer_status,
                                                     void* cuda_stream) {
    using namespace ziplm;
    if (L < 1 || d < 1 || !H || !Hinv || !layer_status) return ZIPLM_ERR_INVALID_ARG;
    if (!(damp_frac >= 0.f) || !isfinite(damp_frac)) return ZIPLM_ERR_INVALID_ARG;
    if (inverse_workspace_bytes(L, d) > kBuiltinScratchBytes) return ZIPLM_ERR_UNSUPPORTED;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ZIPLM_ERR_CUDA;
    void* scratch = nullptr;
    {
        // once per device, with that device current: turn the symbol into its device address
        std::lock_guard<std::mutex> lk(g_scratch_mu);
        if (!g_scratch_addr[dev]) {
            void* addr = nullptr;
            if (cudaGetSymbolAddress(&addr, g_builtin_scratch) != cudaSuccess || !addr)
                return ZIPLM_ERR_CUDA;
            g_scratch_addr[dev] = addr;
        }
        scratch = g_scratch_addr[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    ZIPLM_CHECK_CUDA(cudaMemsetAsync(layer_status, 0, sizeof(int) * L, st));
    // Every part of the scratch that a kernel reads is written earlier in the same call (the
    // damped copy, the factor, the lower tiles of its inverse, lambda), so nothing left behind
    // by the previous call needs clearing.
    return run_damped_inverse(H, L, d, damp_frac, Hinv, nullptr, 0, 0, nullptr, nullptr, layer_status,
                              scratch, kBuiltinScratchBytes, st);
}
