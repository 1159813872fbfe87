// Float64 products of the factorisation on the int8 tensor cores (tcgen05.mma kind::i8).
//
// The float64 instruction runs at 37 TFLOP/s, the int8 one a hundred times faster.  Following Ozaki, Ogita,
// Oishi and Rump ("Error-free transformations of matrix multiplication", 2012) an operand row is written as
// a fixed-point number, x = 2^(E - 62) q with |q| < 2^62 and E the exponent of the row's largest entry, and
// q as eight signed digits of radix 256.  Products of digit matrices are exact in int32 (8 * 2^14 * K stays
// below 2^31 up to kI8MostK, the leading digits being 64 at most); of the 64 pairs the 36 whose weight is at least
// 256^7 are formed, those of one weight into the same accumulator, and the accumulators are joined exactly in
// int64 and then rounded once.  Digits and dropped pairs leave an error below 2^-60 of the largest entries per
// term, less than the 2^-53 of every partial sum that a float64 chain makes; the matrices are equilibrated by
// powers of two beforehand (k_fill_damped), so that a row's entries and the columns they meet are of one scale.
//
// A pair of CTAs computes a tile of 256 x 128: the eight accumulators take two passes of four (512 columns
// of tensor memory), first the digits 4 .. 7 (10 products), then all (26).  A K block is 64 digits (64-byte
// swizzle): eight slices of both operands fill half of the shared-memory ring, 96 KB for 3328 clocks of
// MMAs, so the operand traffic stays at 30 bytes per clock and SM.
// Inverse of 12 x 3072: 14.7 -> 8.8 ms, of 24 x 4096: 57 -> 31 ms (float64 instruction before).  The tensor
// pipe bounds it: an MMA of M = 256, N = 128, K = 32 takes some 92 clocks in place of 64.  Neither an operand kept in
// the collector for up to four MMAs nor a ring of 16 single slices (12 of them in flight) changes that; tiles of
// 256 x 256 (163 clocks an MMA in place of 128, a quarter of the drains four times as often through scratch) were
// slower, 128-byte swizzled rows of two digits the same.
#include <cuda.h>

#include "common.cuh"
#include "inverse_i8.cuh"
#include "tc_common.cuh"

namespace ziplm {
namespace {
using namespace tc;

constexpr int SL = 8;                          // digits
constexpr int KB = 64;                         // digits per K block
constexpr int PM = 256, PN = 128;              // tile of a CTA pair
constexpr int A_BYTES = 128 * KB, B_BYTES = 64 * KB;          // one slice of a CTA's half of the operands
constexpr int STAGE = SL * (A_BYTES + B_BYTES);               // 96 KiB
constexpr int STAGES = 2;
constexpr int I8_SMEM = STAGES * STAGE + 1024;
constexpr int EPI = 16;
constexpr int I8_THREADS = 32 * (2 + EPI);

// ------------------------------------------------------------------------------------------ digits
// Biased exponent of the largest entry (kept away from the ends of the range) -> the factors 2^(62 - E) that
// makes q, and 2^(E - 34): the joined accumulators weigh 2^(Ex + Ey - 68).
__device__ __forceinline__ int clamp_exp(int e) { return max(e, 64); }
__device__ __forceinline__ double pow2_field(int f) { return __hiloint2double(f << 20, 0); }

// The eight digits of four neighbouring entries as one word per slice.
__device__ __forceinline__ void digits4(const double (&x)[4], double to_q, unsigned (&w)[SL]) {
    unsigned lo[4], hi[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        // adding 128 to every lower digit makes them unsigned bytes without carries; the XOR takes it back
        const long long q = __double2ll_rn(x[e] * to_q) + 0x0080808080808080ll;
        lo[e] = (unsigned)q ^ 0x80808080u;
        hi[e] = (unsigned)(q >> 32) ^ 0x00808080u;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const unsigned *v = h ? hi : lo;
        const unsigned a = __byte_perm(v[0], v[1], 0x5140), b = __byte_perm(v[2], v[3], 0x5140);   // bytes 0 0' 1 1'
        const unsigned c = __byte_perm(v[0], v[1], 0x7362), d = __byte_perm(v[2], v[3], 0x7362);   // bytes 2 2' 3 3'
        w[4 * h] = __byte_perm(a, b, 0x5410);
        w[4 * h + 1] = __byte_perm(a, b, 0x7632);
        w[4 * h + 2] = __byte_perm(c, d, 0x5410);
        w[4 * h + 3] = __byte_perm(c, d, 0x7632);
    }
}

// Operand rows = matrix rows.  tri: row i is zero behind the tile of its diagonal entry (block of a lower
// triangular matrix whose upper tiles are not written).  One CTA per row.
__global__ void __launch_bounds__(256) k_digits_rows(const double* __restrict__ src, size_t layer_stride, int ld,
                                                     int rows, int K, int tri, signed char* __restrict__ dig,
                                                     double* __restrict__ scale) {
    __shared__ int red[8];
    const int l = blockIdx.y, i = blockIdx.x, tid = threadIdx.x;
    const double* s = src + l * layer_stride + (size_t)i * ld;
    const int valid = tri ? min(K, (i / kTile + 1) * kTile) : K;
    int e = 0;
    for (int k = 2 * tid; k < valid; k += 512) {
        const double2 x = *reinterpret_cast<const double2*>(s + k);
        e = max(e, max((__double2hiint(x.x) >> 20) & 2047, (__double2hiint(x.y) >> 20) & 2047));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if ((tid & 31) == 0) red[tid >> 5] = e;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) e = max(e, red[w]);
    e = clamp_exp(e);
    if (tid == 0) scale[(size_t)l * rows + i] = pow2_field(e - 33);
    const double to_q = pow2_field(2107 - e);
    signed char* d = dig + ((size_t)l * SL * rows + i) * K;
    for (int k = 4 * tid; k < K; k += 1024) {
        double x[4] = {0.0, 0.0, 0.0, 0.0};
        if (k < valid) {
            const double2 a = *reinterpret_cast<const double2*>(s + k), b = *reinterpret_cast<const double2*>(s + k + 2);
            x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
        }
        unsigned w[SL];
        digits4(x, to_q, w);
#pragma unroll
        for (int q = 0; q < SL; ++q) *reinterpret_cast<unsigned*>(d + (size_t)q * rows * K + k) = w[q];
    }
}

// Operand rows = matrix columns: largest exponents first (exps zeroed beforehand), then the digits through a
// 64 x 64 tile.  tri: column j is zero above the tile of its diagonal entry.  Entries from k_valid and
// column_valid on (the padding of the operand) are zero and not read.
constexpr int EXP_ROWS = 64;                     // of a CTA (256, eight reads in flight: 12 x 3072 382 us in all, now 164)
template <typename T>
__global__ void __launch_bounds__(256) k_column_exponents(const T* __restrict__ src, size_t layer_stride, int ld,
                                                          int cols, int k_valid, int column_valid, int tri,
                                                          int* __restrict__ exps) {
    __shared__ int red[256];
    const int l = blockIdx.z, tid = threadIdx.x, c = tid & 63, k0 = blockIdx.y * EXP_ROWS;
    const int j = blockIdx.x * 64 + c;
    const T* s = src + l * layer_stride + j;
    if (tri && k0 < (int)blockIdx.x * 64) return;
    const int end = j < column_valid ? min(k_valid, k0 + EXP_ROWS) : 0;
    int e = 0;
#pragma unroll
    for (int i = 0; i < EXP_ROWS / 4; ++i) {                 // all reads in flight
        const int k = k0 + (tid >> 6) + 4 * i;
        if (k < end) e = max(e, (__double2hiint((double)s[(size_t)k * ld]) >> 20) & 2047);
    }
    red[tid] = e;
    __syncthreads();
    if (tid < 64) {
        e = max(max(red[tid], red[tid + 64]), max(red[tid + 128], red[tid + 192]));
        atomicMax(exps + (size_t)l * cols + j, e);
    }
}
template <typename T>
__global__ void __launch_bounds__(256) k_digits_columns(const T* __restrict__ src, size_t layer_stride, int ld,
                                                        int cols, int K, int k_valid, int column_valid, int tri,
                                                        const int* __restrict__ exps, signed char* __restrict__ dig,
                                                        double* __restrict__ scale) {
    __shared__ double tile[64][65];              // [k][column]
    const int l = blockIdx.z, tid = threadIdx.x, j0 = blockIdx.x * 64, k0 = blockIdx.y * 64;
    const bool zero = tri && k0 < j0;
    const T* s = src + l * layer_stride + (size_t)k0 * ld + j0;
    if (!zero)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int k = (tid >> 6) + 4 * e, c = tid & 63;
            tile[k][c] = k0 + k < k_valid && j0 + c < column_valid ? (double)s[(size_t)k * ld + c] : 0.0;
        }
    __syncthreads();
    const int kq = 4 * (tid & 15);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int c = (tid >> 4) + 16 * h;
        const int e = clamp_exp(exps[(size_t)l * cols + j0 + c]);
        if (blockIdx.y == 0 && (tid & 15) == 0) scale[(size_t)l * cols + j0 + c] = pow2_field(e - 33);
        double x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = zero ? 0.0 : tile[kq + q][c];
        unsigned w[SL];
        digits4(x, pow2_field(2107 - e), w);
        signed char* d = dig + ((size_t)l * SL * cols + j0 + c) * K + k0 + kq;
#pragma unroll
        for (int q = 0; q < SL; ++q) *reinterpret_cast<unsigned*>(d + (size_t)q * cols * K) = w[q];
    }
}

// ---------------------------------------------------------------------------------------- products
__device__ __forceinline__ void umma_i8_pair(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// K-major tile with 64-byte rows and the 64-byte swizzle: eight-row groups of 512 bytes.
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | (1ull << 16) | (32ull << 32) | (1ull << 46) | (4ull << 61);
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
}

// The MMAs of a K block in one pass: products of weight 256^t, t = qa + qb from T0 to T0 + 3, each weight with an
// accumulator of its own.  Unrolled, so that the one issuing thread adds constants only (with its descriptors' arithmetic
// between the MMAs M^T M of 12 x 3072 took 2.19 ms, now 2.08).
template <int T0>
__device__ __forceinline__ void issue_block(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, bool add) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int qa = T0 + c - 7; qa <= 7; ++qa)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                umma_i8_pair(tmem + (uint32_t)(c * PN), a + (uint32_t)(qa * (A_BYTES / 16) + 2 * h),
                             b + (uint32_t)((T0 + c - qa) * (B_BYTES / 16) + 2 * h), idesc,
                             add || h || qa > T0 + c - 7 ? 1u : 0u);
}

__global__ void __launch_bounds__(I8_THREADS, 1) __cluster_dims__(2, 1, 1)
k_i8_product(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_y,
             const __grid_constant__ I8Product p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_acc_full, bar_acc_empty, bar_final, bar_report;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, reported;
    const uint32_t raw = smem_u32(smem_raw), ring = (raw + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = blockIdx.x & 1u;
    const int l = blockIdx.y;
    // tile (I, J): the ones with the longest K ranges first
    const int nI = (p.rows + PM - 1) / PM, nJ = (p.cols + PN - 1) / PN;
    int I, J, x = (int)(blockIdx.x >> 1);
    if (p.lower) {
        I = 0;
        for (;; ++I) {
            const int w = min(2 * I + 2, nJ);
            if (x < w) break;
            x -= w;
        }
        J = x;
    } else if (p.krange == K_TO_COL) { J = nJ - 1 - x / nI; I = x % nI; }
    else if (p.krange == K_FROM_COL) { J = x / nI; I = x % nI; }
    else { I = nI - 1 - x / nJ; J = x % nJ; }
    const int i0 = I * PM, j0 = J * PN;
    int kb0 = 0, kb1 = p.K / KB;
    if (p.krange == K_TO_COL) kb1 = min(kb1, (j0 + PN) / KB);
    else if (p.krange == K_TO_ROW) kb1 = min(kb1, (i0 + PM) / KB);
    else if (p.krange == K_FROM_COL) kb0 = j0 / KB;
    else if (p.krange == K_FROM_ROW) kb0 = i0 / KB;
    const int n_kb = kb1 - kb0;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_acc_full), 1);
        mbar_init(smem_u32(&bar_acc_empty), 2 * EPI);
        mbar_init(smem_u32(&bar_final), 1);
        mbar_init(smem_u32(&bar_report), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_barrier();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    bool failed = false;
    int issued = 0;                              // K blocks whose copies were started (thread 0)
    auto first_digit = [&](int it) { return it >= n_kb ? 0 : 4; };
    auto bytes = [&](int it) { return (uint32_t)((SL - first_digit(it)) * (A_BYTES + B_BYTES)); };   // per CTA

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer: pass 0 brings the digits 4 .. 7, pass 1 all of them
            const int ya = i0 + (int)rank * 128, yb = j0 + (int)rank * 64;
            const uint32_t full0 = cluster_addr(smem_u32(&bar_full[0]), 0);
            int s = 0;
            uint32_t ph = 1u;
            for (int it = 0; it < 2 * n_kb; ++it) {
                const int pass = it >= n_kb, kx = (kb0 + it - (pass ? n_kb : 0)) * KB;
                if (!mbar_wait_limit(smem_u32(&bar_empty[s]), ph, abortp, p.spin)) { failed = true; break; }
                const uint32_t full = full0 + 8u * (uint32_t)s, base = ring + (uint32_t)s * STAGE;
                if (rank == 0) mbar_expect_tx(smem_u32(&bar_full[s]), 2u * bytes(it));
                for (int q = first_digit(it); q < SL; ++q) {
                    tma_load_4d_pair(base + q * A_BYTES, &map_x, full, kx, ya, q, l);
                    tma_load_4d_pair(base + SL * A_BYTES + q * B_BYTES, &map_y, full, kx, yb, q, l);
                }
                issued = it + 1;
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            if (rank == 1)
                pair_report(cluster_addr(smem_u32(&reported), 0), cluster_addr(smem_u32(&bar_report), 0), issued);
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // ---------------- MMA issuer: int8 x int8 -> int32, M = 256, N = 128, K = 32
            constexpr uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(PN >> 3) << 17) |
                                       ((uint32_t)(PM >> 4) << 24);
            constexpr uint16_t both = 3;
            const uint64_t a0 = desc64(ring), b0 = desc64(ring + SL * A_BYTES);
            int s = 0;
            uint32_t ph = 0u;
            for (int pass = 0; pass < 2 && !failed; ++pass) {
                // the accumulators of pass 0 have been taken out by both CTAs
                if (pass && !mbar_wait(smem_u32(&bar_acc_empty), 0u, abortp)) { failed = true; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int kb = 0; kb < n_kb; ++kb) {
                    if (!mbar_wait(smem_u32(&bar_full[s]), ph, abortp)) { failed = true; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t a = a0 + (uint32_t)(s * (STAGE / 16)), b = b0 + (uint32_t)(s * (STAGE / 16));
                    if (pass) issue_block<7>(tmem_base, a, b, idesc, kb > 0);
                    else issue_block<11>(tmem_base, a, b, idesc, kb > 0);
                    umma_commit_pair(smem_u32(&bar_empty[s]), both);
                    if (++s == STAGES) { s = 0; ph ^= 1u; }
                }
                if (!failed) umma_commit_pair(smem_u32(&bar_acc_full), both);
            }
            umma_commit_pair(smem_u32(&bar_final), both);
            mbar_wait_quiet(smem_u32(&bar_final), 0u);
        }
    } else {
        // ---------------- epilogue: lane quarter = warp % 4, 32 columns by warp
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(cq * 32);
        const uint32_t acc_empty = cluster_addr(smem_u32(&bar_acc_empty), 0);
        double v[32];
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (!mbar_wait(smem_u32(&bar_acc_full), (uint32_t)pass, abortp)) failed = true;
            failed = __any_sync(0xffffffffu, failed);
            if (failed) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                int a[4][8];
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld8(taddr + (uint32_t)(c * PN + 8 * g), a[c]);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const long long j = (((long long)a[3][e] * 256 + a[2][e]) * 256 + a[1][e]) * 256 + a[0][e];
                    v[8 * g + e] = pass ? fma(v[8 * g + e], 4294967296.0, (double)j) : (double)j;
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0 && pass == 0) mbar_arrive_cluster(acc_empty);
        }
        if (!failed) {
            // The ring is free (every MMA has completed): 32 x 32 results pass through it, rows leave whole.
            double* buf = reinterpret_cast<double*>(smem_raw + (ring - raw)) + (size_t)(warp - 2) * 32 * 33;
            const int r0 = i0 + (int)rank * 128 + 32 * q, c0 = j0 + 32 * cq;
            if (r0 < p.rows && c0 < p.cols) {
                const double sx = p.x_scale[(size_t)l * p.rows + r0 + lane] * p.alpha;
#pragma unroll
                for (int e = 0; e < 32; ++e) buf[lane * 33 + e] = v[e] * sx;
                __syncwarp();
                const int col = c0 + lane;
                const double sy = p.y_scale[(size_t)l * p.cols + col];
                if (p.C) {
                    double* C = p.C + l * p.layer_stride + (size_t)r0 * p.ld + col;
                    if (p.beta) {
                        // all old values requested together (behind one another's stores: 22000 clocks)
                        double old[32];
#pragma unroll
                        for (int rr = 0; rr < 32; ++rr) old[rr] = C[(size_t)rr * p.ld];
#pragma unroll
                        for (int rr = 0; rr < 32; ++rr) C[(size_t)rr * p.ld] = fma(buf[rr * 33 + lane], sy, old[rr]);
                    } else {
#pragma unroll 8
                        for (int rr = 0; rr < 32; ++rr) C[(size_t)rr * p.ld] = buf[rr * 33 + lane] * sy;
                    }
                } else {
                    // M^T M: the cropped result, with the equilibration taken back
                    const double dc = p.eq && col < p.d ? p.eq[(size_t)l * p.d + col] * sy : sy;
                    const double dr = p.eq && r0 + lane < p.d ? p.eq[(size_t)l * p.d + r0 + lane] : 1.0;
#pragma unroll 4
                    for (int rr = 0; rr < 32; ++rr) {
                        const int row = r0 + rr;
                        const double x = buf[rr * 33 + lane] * dc * __shfl_sync(0xffffffffu, dr, rr);
                        buf[rr * 33 + lane] = x;
                        if (row >= p.d || col > row) continue;
                        if (p.out64) p.out64[(size_t)l * p.d * p.d + (size_t)row * p.d + col] = x;
                        if (p.tri32 && col < row) p.tri32[((size_t)l * p.rows32 + row) * p.pitch32 + col] = (float)x;
                        if (p.diag64 && col == row) p.diag64[(size_t)l * p.rows32 + row] = x;
                    }
                    __syncwarp();
                    const int row = r0 + lane;               // mirrored: lanes along the rows
#pragma unroll 4
                    for (int e = 0; e < 32; ++e) {
                        const int cc = c0 + e;
                        if (row >= p.d || cc >= row) continue;
                        const double x = buf[lane * 33 + e];
                        if (p.out64) p.out64[(size_t)l * p.d * p.d + (size_t)cc * p.d + row] = x;
                        if (p.tri32) p.tri32[((size_t)l * p.rows32 + cc) * p.pitch32 + row] = (float)x;
                    }
                }
            }
        }
    }

    if (failed) {
        set_layer_status(p.layer_status, l, ZIPLM_ERR_TIMEOUT);
        for (uint32_t r = 0; r < 2; ++r) cluster_store(cluster_addr(smem_u32(&abort_flag), r), 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && rank == 0 && abort_flag)
        pair_land<STAGES>(bar_full, issued, smem_u32(&bar_report), &reported, bytes);
    __syncwarp();
    cluster_barrier();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

template <typename T>
ziplm_status column_digits(const I8Operand& o, const T* src, size_t layer_stride, int ld, int k_valid, int column_valid,
                           bool tri, int L, cudaStream_t st) {
    ZIPLM_CHECK_CUDA(cudaMemsetAsync(o.exps, 0, sizeof(int) * (size_t)L * o.rows, st));
    k_column_exponents<T><<<dim3(o.rows / 64, (k_valid + EXP_ROWS - 1) / EXP_ROWS, L), 256, 0, st>>>(
        src, layer_stride, ld, o.rows, k_valid, column_valid, tri, o.exps);
    ZIPLM_CHECK_LAUNCH();
    k_digits_columns<T><<<dim3(o.rows / 64, o.K / 64, L), 256, 0, st>>>(
        src, layer_stride, ld, o.rows, o.K, k_valid, column_valid, tri, o.exps, o.dig, o.scale);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

bool make_digit_map(CUtensorMap* m, const signed char* dig, int L, int rows, int K, int box_rows) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[4] = {(cuuint64_t)K, (cuuint64_t)rows, SL, (cuuint64_t)L};
    cuuint64_t strides[3] = {(cuuint64_t)K, (cuuint64_t)rows * K, (cuuint64_t)SL * rows * K};
    cuuint32_t box[4] = {KB, (cuuint32_t)box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<signed char*>(dig), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

ziplm_status i8_digits(const I8Operand& o, const double* src, size_t layer_stride, int ld, bool columns, bool tri,
                       int L, cudaStream_t st) {
    if (!columns) {
        k_digits_rows<<<dim3(o.rows, L), 256, 0, st>>>(src, layer_stride, ld, o.rows, o.K, tri, o.dig, o.scale);
        ZIPLM_CHECK_LAUNCH();
        return ZIPLM_OK;
    }
    return column_digits(o, src, layer_stride, ld, o.K, o.rows, tri, L, st);
}

ziplm_status i8_digits_of_columns(const I8Operand& o, const float* src, size_t layer_stride, int ld, int k_valid,
                                  int column_valid, int L, cudaStream_t st) {
    return column_digits(o, src, layer_stride, ld, k_valid, column_valid, false, L, st);
}

size_t carve_i8_operand(I8Operand* o, void* ws, int L, int rows, int K) {
    Carver c(ws);
    I8Operand x = {};
    x.rows = round_up_int(rows, 64);
    x.K = round_up_int(K, 64);
    x.dig = c.take<signed char>((size_t)L * SL * x.rows * x.K);
    x.scale = c.take<double>((size_t)L * x.rows);
    x.exps = c.take<int>((size_t)L * x.rows);
    if (o) *o = x;
    return c.off;
}

bool i8_symmetric_pays(int L, int rows, int K, double float64_clocks) {
    if (K > kI8MostK) return false;
    const int nI = (rows + PM - 1) / PM, nJ = (rows + PN - 1) / PN;
    double tiles = 0;
    for (int I = 0; I < nI; ++I) tiles += 2 * I + 2 < nJ ? 2 * I + 2 : nJ;
    const double waves = ceil(L * tiles / (kSMs / 2));     // two SMs to a tile
    return 20000.0 + waves * ((K + KB - 1) / KB * 7000.0 + 30000.0) < float64_clocks;
}

ziplm_status i8_product(const I8Operand& x, const I8Operand& y, I8Product p, int L, cudaStream_t st) {
    CUtensorMap mx, my;
    if (x.K > kI8MostK) return ZIPLM_ERR_UNSUPPORTED;      // (no caller asks for it)
    p.rows = x.rows; p.cols = y.rows; p.K = x.K;
    p.x_scale = x.scale; p.y_scale = y.scale;
    const int spin = option_value(ZIPLM_OPT_SPIN_LIMIT);
    p.spin = spin > 0 ? (unsigned)spin : kSpinLimit;
    if (!make_digit_map(&mx, x.dig, L, x.rows, x.K, 128) || !make_digit_map(&my, y.dig, L, y.rows, y.K, 64))
        return ZIPLM_ERR_CUDA;
    const int nI = (p.rows + PM - 1) / PM, nJ = (p.cols + PN - 1) / PN;
    int tiles = nI * nJ;
    if (p.lower) {
        tiles = 0;
        for (int I = 0; I < nI; ++I) tiles += 2 * I + 2 < nJ ? 2 * I + 2 : nJ;
    }
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_i8_product, cudaFuncAttributeMaxDynamicSharedMemorySize, I8_SMEM));
    k_i8_product<<<dim3(2 * tiles, L), I8_THREADS, I8_SMEM, st>>>(mx, my, p);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace ziplm
