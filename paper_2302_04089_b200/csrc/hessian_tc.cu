// Calibration Hessian H = beta H + alpha X X^T (caption of Algorithm 1) on the 5th-generation
// tensor cores: TMA-fed 128-byte-swizzled K-major tiles, tcgen05.mma issued by one thread,
// fp32 accumulator in tensor memory, read back with tcgen05.ld for the symmetric store.
//
// Both operands of X X^T are row blocks of the same K-major matrix (tokens contiguous), so one
// tensor map serves A and B.  Only the 128 x 128 tiles on or below the diagonal are computed; an
// off-diagonal tile is stored twice (as is, and transposed).
//
//   bf16 / fp16 X : kind::f16 (both operands of the same 16-bit type, exact products, fp32
//            accumulate), K block of 64 tokens.
//   fp32 X : a pre-pass scales every feature row by a power of two s_i (so that its largest
//            entry lies in [2^13, 2^14): the whole fp16 range is used whatever the row's
//            magnitude) and writes two fp16 parts, X_1 = fp16(s x) and X_2 = fp16(s x - X_1);
//            the kernel accumulates X_1 X_1^T + X_1 X_2^T + X_2 X_1^T with kind::f16 (exact
//            products, fp32 accumulate), which keeps ~21 mantissa bits per product, and the
//            epilogue multiplies entry (i, j) by 1 / (s_i s_j) (exact).  K block of 64 tokens:
//            half the operand bytes and half the MMAs of a TF32 hi / lo split of the same
//            accuracy, which matters because the kernel is bound by the L2 -> shared-memory
//            operand traffic.
//
// One CTA per tile, or a cluster of up to eight where the tiles are few, each CTA a range of the
// tile's K blocks (problems of many tiles go to hessian_pair.cu).  Warp 0 = TMA producer, warp 1 =
// TMEM owner + MMA issuer, warps 2..9 = epilogue (two per TMEM lane quarter; they drain the
// accumulator every few K blocks, see below).  Every mbarrier wait is bounded; if one runs out the
// kernel raises the error word and every role leaves its loop; the issuer then waits (one more commit)
// for the MMAs it has issued, the producer for the copies it has started, and the CTA leaves through
// the normal exit (TMEM freed), so a lost copy can never hang the GPU.  H[l][0][0] of every layer is
// NaN then (hessian_common.cuh).
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <chrono>

#include "common.cuh"
#include "hessian_common.cuh"
#include "tc_common.cuh"

namespace cg = cooperative_groups;

namespace ziplm {
namespace {
using namespace tc;

constexpr int TM = 128;                 // tile rows / cols
constexpr int ROW_BYTES = 128;          // one swizzle row
constexpr int TILE_BYTES = TM * ROW_BYTES;   // 16 KiB per operand tile per K block

template <bool SPLIT> struct Cfg;   // SPLIT: two fp16 parts per operand (fp32 inputs)
template <> struct Cfg<true>  { static constexpr int BK = 64, UK = 16, STAGES = 3, TILES = 4; };
template <> struct Cfg<false> { static constexpr int BK = 64, UK = 16, STAGES = 5, TILES = 2; };

// Tensor-memory accumulators truncate when they add (measured: the error of a chain of S
// accumulating MMAs grows like S * 3e-8, always toward zero), so a chain is kept short: the main
// accumulator is double-buffered, and after every CHUNK K blocks (8 MMAs) the epilogue warps
// drain it into fp32 registers, where the partial sums are added with round-to-nearest in two
// levels (a running sum that is folded into the total every FOLD drains, so that neither level
// adds more than a few dozen terms).  The cross terms X_1 X_2^T + X_2 X_1^T of the split are
// 2^-11 of the main term; they get an accumulator of their own that is only read at the end, so
// their truncation is negligible.
constexpr int CHUNK = 2;
constexpr int FOLD = 32;
constexpr int EPI_WARPS = 8;                  // two warps per TMEM lane quarter, 64 columns each
constexpr int THREADS = 32 * (2 + EPI_WARPS);
constexpr int OUT_PITCH = TM + 1;             // floats of a row of the finished tile in shared memory
constexpr int PART_PITCH = TM + 4;            // ... of a part of it, whose rows are read 16 bytes a lane

// The end of a tile that S CTAs of a cluster have shared, their parts in out_tile of each: a CTA finishes 128 / S
// rows.  Sums over the parts in rank order, rows [i][j] written along j, mirrored rows [j][i] along i.
// A warp takes R rows at a time, the parts and the old values of all of them requested together, and eight
// mirrored pieces at a time: one after the other the two took 22000 clocks of a tile's 32000 (13 x 1145 features,
// 324 bf16 tokens: 70 -> 54 us a call).
// Parts are read 16 bytes a lane, four columns, and the scales wait in shared memory: 1 x 256 x 2048 fp32 on clusters of
// eight 12.8 us, against 15.5 with 4 bytes a lane and the scales from global memory behind the last barrier.  H is read
// and written with lanes along the columns, 128 bytes an instruction, also where its rows start on 16 bytes: four columns
// a lane took 18.5 us in place of 16.6 (1 x 1322 x 600 fp16, rows at any element, written in four passes of half-empty
// sectors), 18.5 and 16.7 (4 x 576 x 693), 16.4 and 14.8 (8 x 80 x 2178 bf16); 20.8 and 22.2 the other way (2 x 408 x 1267
// fp32).
struct TileEnd {
    float* out_tile; float* mirror;
    int rank, i0, j0, d;
    float alpha, beta;
    float* Hl; const float* scales;           // inverse scales of the tile's rows and columns [2][TM]
    const unsigned long long* err_word; unsigned long long call;

    // rows of `mirror`: this CTA's share
    template <int S, int R, bool SPLIT>
    __device__ __forceinline__ void rows_of_parts() const {
        constexpr int N_ROWS = TM / S, WARPS = THREADS / 32, NH = TM / 32;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, first = rank * N_ROWS, cc = 4 * lane;
        const float4 scale = SPLIT ? *reinterpret_cast<const float4*>(scales + TM + cc) : make_float4(1.f, 1.f, 1.f, 1.f);
#pragma unroll 1
        for (int at = warp * R; at < N_ROWS && i0 + first + at < d; at += WARPS * R) {
            float4 part[S][R];
            float old[R][NH];
            float* own = out_tile + (first + at) * PART_PITCH;
#pragma unroll
            for (int p = 0; p < S; ++p) {
                const float* from = cg::this_cluster().map_shared_rank(own + cc, p);
#pragma unroll
                for (int k = 0; k < R; ++k) part[p][k] = *reinterpret_cast<const float4*>(from + k * PART_PITCH);
            }
#pragma unroll
            for (int k = 0; k < R; ++k)
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    const int row = i0 + first + at + k, col = j0 + 32 * h + lane;
                    old[k][h] = beta != 0.f && row < d && col <= row ? Hl[(size_t)row * d + col] : 0.f;
                }
            // the scaled sums go back to the place of this CTA's own part, which nobody else reads
#pragma unroll
            for (int k = 0; k < R; ++k) {
                float v[4] = {part[0][k].x, part[0][k].y, part[0][k].z, part[0][k].w};
#pragma unroll
                for (int p = 1; p < S; ++p) { v[0] += part[p][k].x; v[1] += part[p][k].y; v[2] += part[p][k].z; v[3] += part[p][k].w; }
                const float sc[4] = {scale.x, scale.y, scale.z, scale.w}, mul = SPLIT ? scales[first + at + k] : 1.f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    v[e] *= alpha;
                    if (SPLIT) v[e] = (v[e] * mul) * sc[e];
                }
                *reinterpret_cast<float4*>(own + k * PART_PITCH + cc) = make_float4(v[0], v[1], v[2], v[3]);
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const int row = i0 + first + at + k;
                float* out = Hl + (size_t)row * d + j0 + lane;
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    const int c = 32 * h + lane, col = j0 + c;
                    if (row >= d || col > row) continue;             // (col <= row < d)
                    const float v = own[k * PART_PITCH + c] + old[k][h];
                    out[32 * h] = v;
                    if ((row | col) == 0) hessian_check(out, err_word, call);
                    mirror[(at + k) * OUT_PITCH + c] = v;
                }
            }
        }
    }

    template <int R, bool SPLIT>
    __device__ __forceinline__ void rows_of_tile() const {
        constexpr int NH = TM / 32, WARPS = THREADS / 32;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        // split route: undo the power-of-two scales of the two feature rows (exact)
        float scale[NH];
#pragma unroll
        for (int h = 0; h < NH; ++h) scale[h] = SPLIT ? scales[TM + 32 * h + lane] : 1.f;
#pragma unroll 1
        for (int at = warp * R; at < TM && i0 + at < d; at += WARPS * R) {
            float part[R][NH], old[R][NH];
#pragma unroll
            for (int k = 0; k < R; ++k)
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    const int row = i0 + at + k, col = j0 + 32 * h + lane;
                    part[k][h] = out_tile[(at + k) * OUT_PITCH + 32 * h + lane];
                    old[k][h] = beta != 0.f && row < d && col <= row ? Hl[(size_t)row * d + col] : 0.f;
                }
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const int row = i0 + at + k;
                float* out = Hl + (size_t)row * d + j0 + lane;
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    const int cc = 32 * h + lane, col = j0 + cc;
                    if (row >= d || col > row) continue;             // (col <= row < d)
                    float v = part[k][h] * alpha;
                    if (SPLIT) v = (v * scales[at + k]) * scale[h];
                    v += old[k][h];
                    out[32 * h] = v;
                    if ((row | col) == 0) hessian_check(out, err_word, call);
                    mirror[(at + k) * OUT_PITCH + cc] = v;
                }
            }
        }
    }

    template <int S, int R, bool SPLIT>
    __device__ __forceinline__ void finish() const {
        constexpr int N_ROWS = TM / S, WARPS = THREADS / 32;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, first = rank * N_ROWS;
        if constexpr (S > 1) rows_of_parts<S, R, SPLIT>();
        else rows_of_tile<R, SPLIT>();
        __syncthreads();
        // lanes along the rows of this share (32, or all of them where there are fewer), then along columns
        constexpr int LANES = N_ROWS < 32 ? N_ROWS : 32, PER = 32 / LANES, SEG = N_ROWS / LANES, FLY = 8;
        constexpr int PIECES = TM / PER * SEG;                       // (PER columns) x (LANES rows)
        const int sub = lane / LANES, ln = lane % LANES;
#pragma unroll 1
        for (int x = warp; x < PIECES; x += FLY * WARPS) {
            float v[FLY];
#pragma unroll
            for (int k = 0; k < FLY; ++k) {
                const int y = min(x + k * WARPS, PIECES - 1), c = y / SEG * PER + sub, rr = y % SEG * LANES + ln;
                v[k] = mirror[rr * OUT_PITCH + c];
            }
#pragma unroll
            for (int k = 0; k < FLY; ++k) {
                const int y = x + k * WARPS, c = y / SEG * PER + sub, rr = y % SEG * LANES + ln;
                const int row = i0 + first + rr, col = j0 + c;
                if (y < PIECES && row < d && col < row) Hl[(size_t)col * d + row] = v[k];
            }
        }
    }
};

template <bool SPLIT>
__global__ void __launch_bounds__(THREADS, 1)
k_syrk_tc(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
          float* __restrict__ H, int d, int num_kb_all, int n_split, float alpha, float beta, int layer0,
          int L, unsigned long long* err_word, unsigned long long call, uint32_t fmt16, uint32_t empty_spin_limit,
          const unsigned* __restrict__ amax) {
    using C = Cfg<SPLIT>;
    constexpr int STAGE_BYTES = C::TILES * TILE_BYTES;
    constexpr uint32_t TMEM_COLS = SPLIT ? 512u : 256u;   // main x2 (+ cross terms), power of two
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[C::STAGES], bar_empty[C::STAGES], bar_acc_full[2], bar_acc_empty[2], bar_final;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float scales[2 * TM];

    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;       // swizzled tiles need 1024-byte alignment
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l = blockIdx.y;                             // layer within the launched chunk
    // a cluster of n_split CTAs shares a tile, each a range of its K blocks
    const int rank = (int)blockIdx.x % n_split;
    const int kb_begin = (int)((long long)num_kb_all * rank / n_split);
    const int num_kb = (int)((long long)num_kb_all * (rank + 1) / n_split) - kb_begin;
    int ti = 0, rem = (int)blockIdx.x / n_split;
    while (rem > ti) { rem -= ti + 1; ++ti; }
    const int tj = rem;
    const int i0 = ti * TM, j0 = tj * TM;
    const bool diag = (ti == tj);
    const int num_chunks = (num_kb + CHUNK - 1) / CHUNK;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_acc_full[b]), 1);
            mbar_init(smem_u32(&bar_acc_empty[b]), EPI_WARPS);   // one arrival per epilogue warp
        }
        mbar_init(smem_u32(&bar_final), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    grid_wait();                                          // the operands are there
    const uint32_t tmem_base = tmem_base_slot;            // main[0] = +0, main[1] = +128, cross = +256
    volatile int* abortp = &abort_flag;
    float* out_tile = reinterpret_cast<float*>(smem_raw + (tiles - raw));    // [TM][OUT_PITCH], over the ring
    float* mirror = n_split > 1 ? out_tile + TM * PART_PITCH : out_tile;     // finished rows of this CTA
    if (SPLIT && threadIdx.x >= THREADS - 2 * TM) {       // the epilogue's threads; read behind the barrier at the end
        const int e = (int)threadIdx.x - (THREADS - 2 * TM), row = (e < TM ? i0 : j0 - TM) + e;
        scales[e] = row < d ? row_scale(__ldcg(amax + (size_t)l * d + row), true) : 1.f;
    }
    bool failed = false;
    int issued = 0;                                       // K blocks whose copies were started (thread 0)

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer
            const uint32_t bytes = (uint32_t)((diag ? C::TILES / 2 : C::TILES) * TILE_BYTES);
            int s = 0;
            uint32_t ph = 1u;
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!mbar_wait_limit(smem_u32(&bar_empty[s]), ph, abortp, empty_spin_limit)) {
                    failed = true;
                    break;
                }
                const uint32_t full = smem_u32(&bar_full[s]);
                const uint32_t base = tiles + (uint32_t)s * STAGE_BYTES;
                mbar_expect_tx(full, bytes);
                const int x = (kb_begin + kb) * C::BK;
                tma_load_3d(base, &map_hi, full, x, i0, l);
                if (!diag) tma_load_3d(base + TILE_BYTES, &map_hi, full, x, j0, l);
                if (SPLIT) {
                    tma_load_3d(base + 2 * TILE_BYTES, &map_lo, full, x, i0, l);
                    if (!diag) tma_load_3d(base + 3 * TILE_BYTES, &map_lo, full, x, j0, l);
                }
                issued = kb + 1;
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---------------- MMA issuer
            // operand format of the instruction: 1 = BF16, 0 = F16 (A and B alike; the split is fp16)
            const uint32_t idesc = make_idesc(SPLIT ? 0u : fmt16, TM, TM);
            const uint32_t tmem_cross = tmem_base + 256u;
            int kb = 0, s = 0;
            uint32_t ph = 0u;
            for (int c = 0; c < num_chunks && !failed; ++c) {
                const int b = c & 1;
                const uint32_t tmem_main = tmem_base + (uint32_t)b * 128u;
                // the epilogue must have drained this buffer (first use of each buffer passes)
                if (!mbar_wait(smem_u32(&bar_acc_empty[b]), (((uint32_t)c >> 1) & 1u) ^ 1u, abortp)) {
                    failed = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int kb_end = (kb + CHUNK < num_kb) ? kb + CHUNK : num_kb;
                const int kb_first = kb;
                for (; kb < kb_end; ++kb) {
                    if (!mbar_wait(smem_u32(&bar_full[s]), ph, abortp)) { failed = true; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t base = tiles + (uint32_t)s * STAGE_BYTES;
                    const uint64_t a_hi = make_desc(base);
                    const uint64_t b_hi = diag ? a_hi : make_desc(base + TILE_BYTES);
                    const uint64_t a_lo = make_desc(base + 2 * TILE_BYTES);
                    const uint64_t b_lo = diag ? a_lo : make_desc(base + 3 * TILE_BYTES);
#pragma unroll
                    for (int k = 0; k < C::BK / C::UK; ++k) {
                        const uint64_t adv = (uint64_t)(k * 32 / 16);   // 32 bytes per MMA along K
                        const uint32_t acc_main = ((kb - kb_first) | k) ? 1u : 0u;
                        if (SPLIT) {
                            umma_bf16(tmem_main, a_hi + adv, b_hi + adv, idesc, acc_main);
                            umma_bf16(tmem_cross, a_hi + adv, b_lo + adv, idesc, (kb | k) ? 1u : 0u);
                            umma_bf16(tmem_cross, a_lo + adv, b_hi + adv, idesc, 1u);
                        } else {
                            umma_bf16(tmem_main, a_hi + adv, b_hi + adv, idesc, acc_main);
                        }
                    }
                    umma_commit(smem_u32(&bar_empty[s]));     // stage free once these MMAs have read it
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
                if (!failed) umma_commit(smem_u32(&bar_acc_full[b]));   // chunk (and all before) done
            }
            // Whatever was issued has completed before tensor memory is given back and the CTA
            // retires, also when a role has given up: one more commit, to a barrier of its own.
            umma_commit(smem_u32(&bar_final));
            mbar_wait_quiet(smem_u32(&bar_final), 0u);
        }
    } else {
        // ---------------- epilogue: warps 2..9; TMEM lane quarter = warp % 4, column half by warp
        const int q = warp & 3;
        const int half = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        constexpr int NC = TM / 2;                      // columns owned by this thread
        float acc[NC], tot[NC];
#pragma unroll
        for (int e = 0; e < NC; ++e) { acc[e] = 0.f; tot[e] = 0.f; }
        for (int c = 0; c < num_chunks; ++c) {
            const int b = c & 1;
            if (!mbar_wait(smem_u32(&bar_acc_full[b]), ((uint32_t)c >> 1) & 1u, abortp)) failed = true;
            failed = __any_sync(0xffffffffu, failed);
            if (failed) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int cc = 0; cc < NC / 32; ++cc) {
                uint32_t v[32];
                tmem_ld32(tmem_base + lane_base + (uint32_t)(b * 128 + half * NC + cc * 32), v);
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[cc * 32 + e] += __uint_as_float(v[e]);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[b]));
            if ((c % FOLD) == FOLD - 1) {
#pragma unroll
                for (int e = 0; e < NC; ++e) { tot[e] += acc[e]; acc[e] = 0.f; }
            }
        }
        if (!failed) {
            if (SPLIT) {
                // the last chunk's commit also covers every cross-term MMA (16 columns at a time: 32 spill)
#pragma unroll
                for (int cc = 0; cc < NC / 16; ++cc) {
                    uint32_t v[16];
                    tmem_ld16(tmem_base + lane_base + (uint32_t)(256 + half * NC + cc * 16), v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[cc * 16 + e] += __uint_as_float(v[e]);
                }
            }
            // The operand ring is free (every MMA has completed): the partial tile goes there.
            const int row = q * 32 + lane;
            if (n_split > 1) {
#pragma unroll
                for (int e = 0; e < NC; e += 4)
                    *reinterpret_cast<float4*>(out_tile + row * PART_PITCH + half * NC + e) =
                        make_float4(tot[e] + acc[e], tot[e + 1] + acc[e + 1], tot[e + 2] + acc[e + 2], tot[e + 3] + acc[e + 3]);
            } else {
#pragma unroll
                for (int e = 0; e < NC; ++e) out_tile[row * OUT_PITCH + half * NC + e] = tot[e] + acc[e];
            }
        }
    }

    if (failed) {
        abort_flag = 1;
        hessian_give_up(H, L, d, err_word, call);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) {
        // Copies that were started land in this CTA's shared memory: wait for them (bounded) before
        // the CTA retires.  The last STAGES K blocks started are the latest phases of their barriers.
        for (int kb = issued > C::STAGES ? issued - C::STAGES : 0; kb < issued; ++kb)
            mbar_wait_quiet(smem_u32(&bar_full[kb % C::STAGES]), (uint32_t)(kb / C::STAGES) & 1u);
    }
    __syncwarp();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS)
                     : "memory");
    }
    cg::cluster_group cluster = cg::this_cluster();
    if (n_split > 1) cluster.sync();

    // Every CTA of the cluster finishes its share of the rows.
    float* Hl = H + (size_t)(layer0 + l) * d * d;
    const TileEnd end{out_tile, mirror, rank, i0, j0, d, alpha, beta, Hl, scales, err_word, call};
    if (n_split == 1) end.finish<1, 4, SPLIT>();
    else if (n_split == 2) end.finish<2, 4, SPLIT>();
    else if (n_split == 4) end.finish<4, 4, SPLIT>();
    else end.finish<8, 2, SPLIT>();
    if (n_split > 1) cluster.sync();                         // no CTA retires while others read its tile
}

// Largest magnitude of every feature row of a token-contiguous X (bit pattern of |x|, which
// orders like the value for non-negative floats; a NaN sorts above everything and switches the
// scaling of its row off).
__global__ void __launch_bounds__(256) k_row_absmax(const float* __restrict__ X, long long ldx, long long N,
                                                    unsigned* __restrict__ amax) {
    __shared__ unsigned red[8];
    const size_t row = blockIdx.x;
    const float* src = X + row * (size_t)ldx;
    unsigned m = 0u;
    for (long long k = threadIdx.x; k < N; k += 256) m = max(m, __float_as_uint(src[k]) & 0x7fffffffu);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = max(m, red[w]);
        amax[row] = m;
    }
}

// The same for token-major input A [layers, N, lda] (one token per row): every thread walks one feature over a slab of
// tokens with AM_FLY reads in flight, the slabs meet through atomicMax (amax zeroed beforehand).  Slabs are as short
// as it takes to fill the SMs, and no longer than 256 tokens: 6 x 7265 x 317 23.2 -> 14.0 us, 1 x 9000 x 65 19.1 -> 4.8
// (slabs of 256 always, four reads in flight); 12 x 16384 x 768 as before, 95 us (6.4 TB/s): without branches and with
// indexes held at the edge 119, a warp to 32 features with 32 tokens in flight 140.
constexpr int AM_FLY = 16, AM_SLAB = 256;
__global__ void __launch_bounds__(256) k_tokens_absmax(const float* __restrict__ A, long long lda,
                                                       long long N, int d, long long slab,
                                                       unsigned* __restrict__ amax) {
    const int l = blockIdx.z;
    const int f = blockIdx.x * 256 + threadIdx.x;
    if (f >= d) return;
    const long long t0 = (long long)blockIdx.y * slab, t1 = min(N, t0 + slab);
    unsigned m = 0u;
    const float* src = A + ((size_t)l * (size_t)N + (size_t)t0) * (size_t)lda + f;
    long long t = t0;
    for (; t + AM_FLY <= t1; t += AM_FLY) {
        unsigned v[AM_FLY];
#pragma unroll
        for (int k = 0; k < AM_FLY; ++k, src += lda) v[k] = __float_as_uint(*src) & 0x7fffffffu;
#pragma unroll
        for (int k = 0; k < AM_FLY; ++k) m = max(m, v[k]);
    }
    for (; t < t1; ++t, src += lda) m = max(m, __float_as_uint(*src) & 0x7fffffffu);
    atomicMax(amax + (size_t)l * d + f, m);
}

// The two fp16 parts of four scaled fp32 values: y_1 = fp16(y), y_2 = fp16(y - y_1) (the difference is exact in fp32),
// by packed conversions.
__device__ __forceinline__ void split_f16x2(const float (&y)[4], uint2& p1, uint2& p2) {
    union { uint2 v; __half2 e[2]; } a, b;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        a.e[e] = __floats2half2_rn(y[2 * e], y[2 * e + 1]);
        const float2 f = __half22float2(a.e[e]);
        b.e[e] = __floats2half2_rn(y[2 * e] - f.x, y[2 * e + 1] - f.y);
    }
    p1 = a.v;
    p2 = b.v;
}

// X_1, X_2 of a token-contiguous fp32 X, four tokens per thread; np (a multiple of 8) is the row
// pitch of the parts, zero past N.
__global__ void __launch_bounds__(256) k_split_f16(const float* __restrict__ X, long long ldx,
                                                   long long N, long long np, size_t rows,
                                                   const unsigned* __restrict__ amax,
                                                   __half* __restrict__ hi, __half* __restrict__ lo) {
    grid_trigger();
    const size_t row = blockIdx.y;
    const long long k = ((long long)blockIdx.x * 256 + threadIdx.x) * 4;
    if (row >= rows || k >= np) return;
    const float* src = X + row * (size_t)ldx + k;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (k + 3 < N) {
        const float4 t = *reinterpret_cast<const float4*>(src);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        for (int e = 0; e < 4; ++e) if (k + e < N) v[e] = src[e];
    }
    const float sc = row_scale(amax[row], false);
    const float y[4] = {v[0] * sc, v[1] * sc, v[2] * sc, v[3] * sc};
    split_f16x2(y, *reinterpret_cast<uint2*>(hi + row * (size_t)np + k),
                *reinterpret_cast<uint2*>(lo + row * (size_t)np + k));
}

// Both pre-passes in one for rows of at most 256 * 4 * VEC tokens: a CTA keeps its feature row in
// registers (VEC 16-byte loads per thread, all in flight together), finds the largest magnitude,
// and writes the two scaled fp16 parts -- X is read once instead of twice.  Values and layout are
// those of k_row_absmax followed by k_split_f16.
template <int VEC>
__global__ void __launch_bounds__(256) k_row_absmax_split(const float* __restrict__ X, long long ldx,
                                                          long long N, long long np,
                                                          unsigned* __restrict__ amax,
                                                          __half* __restrict__ hi, __half* __restrict__ lo) {
    grid_trigger();
    __shared__ unsigned red[8];
    __shared__ unsigned row_max;
    const size_t row = blockIdx.x;
    const float* src = X + row * (size_t)ldx;
    float v[VEC][4];
    unsigned m = 0u;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        const long long k = ((long long)j * 256 + threadIdx.x) * 4;
        v[j][0] = v[j][1] = v[j][2] = v[j][3] = 0.f;
        if (k + 3 < N) {
            const float4 t = *reinterpret_cast<const float4*>(src + k);
            v[j][0] = t.x; v[j][1] = t.y; v[j][2] = t.z; v[j][3] = t.w;
        } else {
            for (int e = 0; e < 4; ++e) if (k + e < N) v[j][e] = src[k + e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) m = max(m, __float_as_uint(v[j][e]) & 0x7fffffffu);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = max(m, red[w]);
        amax[row] = m;
        row_max = m;
    }
    __syncthreads();
    const float sc = row_scale(row_max, false);
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        const long long k = ((long long)j * 256 + threadIdx.x) * 4;
        if (k >= np) continue;
        const float y[4] = {v[j][0] * sc, v[j][1] * sc, v[j][2] * sc, v[j][3] * sc};
        split_f16x2(y, *reinterpret_cast<uint2*>(hi + row * (size_t)np + k),
                    *reinterpret_cast<uint2*>(lo + row * (size_t)np + k));
    }
}

// Token-major fp32 input (one calibration token per row, as a forward pass emits activations): A is [layers, N, lda]
// with the feature index contiguous.  A 64 x 64 tile goes through shared memory, so the reads run along features and
// the writes along tokens, both coalesced; the scaled fp16 parts X_1 / X_2 leave in the K-major [layers * d, np]
// matrices that the product kernel loads (same values as k_split_f16; amax holds the features' largest magnitudes).
// QUADS: rows of A start on 16 bytes (A aligned, lda % 4 == 0); otherwise a warp reads 32 neighbouring features,
// sixteen tokens a thread in flight.  np is a multiple of 8, so a quad that starts below np ends below it.
// Bound by memory: 6 x 7265 x 320 20 us, x 317 35.3 -> 19.3 (32 x 32 tiles, entries one by one before).
template <bool QUADS>
__global__ void __launch_bounds__(256) k_tokens_to_kmajor(const float* __restrict__ A, long long lda, long long N,
                                                             int d, long long np, const unsigned* __restrict__ amax,
                                                             __half* __restrict__ hi, __half* __restrict__ lo) {
    grid_trigger();
    __shared__ float tile[64][65];                       // [token][feature]
    const int l = blockIdx.z;
    const long long t0 = (long long)blockIdx.x * 64;
    const int f0 = blockIdx.y * 64;
    const int q = threadIdx.x & 15, rr = threadIdx.x >> 4;
    const float* Al = A + (size_t)l * (size_t)N * (size_t)lda;
    if (QUADS) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int tl = rr + 16 * k;
            const long long t = t0 + tl;
            const int f = f0 + 4 * q;
            float u[4];
            if (t < N && f + 3 < d) {
                const float4 x = *reinterpret_cast<const float4*>(Al + (size_t)t * (size_t)lda + f);
                u[0] = x.x; u[1] = x.y; u[2] = x.z; u[3] = x.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) u[e] = (t < N && f + e < d) ? Al[(size_t)t * (size_t)lda + f + e] : 0.f;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) tile[tl][4 * q + e] = u[e];
        }
    } else {
        const int fl = threadIdx.x & 63, r0 = threadIdx.x >> 6;
        const float* src = Al + ((size_t)t0 + r0) * (size_t)lda + f0 + fl;
        float u[16];
#pragma unroll
        for (int k = 0; k < 16; ++k, src += 4 * (size_t)lda)
            u[k] = t0 + r0 + 4 * k < N && f0 + fl < d ? *src : 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k) tile[r0 + 4 * k][fl] = u[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int fl = rr + 16 * k;
        const int f = f0 + fl;
        const long long t = t0 + 4 * q;
        if (f >= d || t >= np) continue;
        const float sc = row_scale(amax[(size_t)l * d + f], false);
        float y[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) y[e] = tile[4 * q + e][fl] * sc;
        const size_t o = ((size_t)l * d + f) * (size_t)np + (size_t)t;
        split_f16x2(y, *reinterpret_cast<uint2*>(hi + o), *reinterpret_cast<uint2*>(lo + o));
    }
}

// The same move of 16-bit elements (raw bits of bf16 or fp16), pairs of features at a time: 128 tokens x 64
// features, 16 loads in flight per thread (a warp reads 128 bytes of a row; PAIRS: rows start on 4 bytes, lda
// even, otherwise a pair is two loads), and eight tokens of
// two features per thread put together from eight words, so that 256 bytes of a feature leave together.  The
// words of a token lie permuted by the group of eight tokens: no bank conflicts on either side.
// 4099 x 1322: 10.7 -> 6.7 us, 19 x 2186 x 1203 79.6 -> 46 (32 x 32 elements one by one before).
// TOKENS of a tile: 128, or 32 without PAIRS where tiles of 128 leave SMs idle and the chain of a thread's loads is what
// counts (a call 1 x 700 x 513 18.2 -> 16.6 us, 2 x 2402 x 89 16.0 -> 14.6; with PAIRS 1 x 600 x 1322 16.7 -> 17.9).
template <bool PAIRS, int TOKENS>
__global__ void __launch_bounds__(256) k_tokens16_to_kmajor(const uint16_t* __restrict__ A, long long lda, long long N,
                                                            int d, long long np, uint16_t* __restrict__ out) {
    grid_trigger();
    constexpr int GROUPS = TOKENS / 8;                   // of eight tokens; a thread reads a token of each
    constexpr int SHIFT = TOKENS == 128 ? 0 : 3;         // place of word w in group k: w ^ (k << SHIFT)
    static_assert(TOKENS == 128 || TOKENS == 32, "the places below are worked out for these");
    __shared__ uint32_t tile[TOKENS * 32];
    const int l = blockIdx.z, f0 = blockIdx.y * 64, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long t0 = (long long)blockIdx.x * TOKENS;
    {
        const int f = f0 + 2 * lane;
        const long long left = N - 1 - t0;               // tokens behind the tile's first, which is below N
        const uint16_t* src = A + ((size_t)l * (size_t)N + (size_t)t0) * (size_t)lda;
        uint32_t v[GROUPS];
        if (PAIRS) {
            src += warp * (size_t)lda + f;
#pragma unroll
            for (int k = 0; k < GROUPS; ++k, src += 8 * (size_t)lda) {
                v[k] = 0u;
                if (warp + 8 * k <= left && f < d)
                    v[k] = f + 1 < d ? *reinterpret_cast<const uint32_t*>(src) : (uint32_t)*src;
            }
        } else {                                         // (read again past the ends: no branches around the loads)
            const int c0 = min(f, d - 1), c1 = min(f + 1, d - 1);
            uint16_t x0[GROUPS], x1[GROUPS];
#pragma unroll
            for (int k = 0; k < GROUPS; ++k) {
                const uint16_t* row = src + (size_t)min((long long)(warp + 8 * k), left) * (size_t)lda;
                x0[k] = row[c0];
                x1[k] = row[c1];
            }
#pragma unroll
            for (int k = 0; k < GROUPS; ++k)
                v[k] = warp + 8 * k > left || f >= d ? 0u : x0[k] | (f + 1 < d ? (uint32_t)x1[k] << 16 : 0u);
        }
#pragma unroll
        for (int k = 0; k < GROUPS; ++k) tile[(warp + 8 * k) * 32 + (lane ^ (k << SHIFT))] = v[k];
    }
    __syncthreads();
    const int tg = threadIdx.x & (GROUPS - 1);
    const long long t = t0 + 8 * tg;
#pragma unroll
    for (int h = 0; h < (TOKENS == 128 ? 2 : 1); ++h) {
        const int w = TOKENS == 128 ? warp + 8 * h + 16 * (lane >> 4) : threadIdx.x / GROUPS, f = f0 + 2 * w;
        if (w >= 32) break;
        uint32_t x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = tile[(8 * tg + k) * 32 + (w ^ (tg << SHIFT))];
        if (t >= np || f >= d) continue;
        uint16_t* o = out + ((size_t)l * d + f) * (size_t)np + (size_t)t;
        *reinterpret_cast<uint4*>(o) = make_uint4(__byte_perm(x[0], x[1], 0x5410), __byte_perm(x[2], x[3], 0x5410),
                                                  __byte_perm(x[4], x[5], 0x5410), __byte_perm(x[6], x[7], 0x5410));
        if (f + 1 < d)
            *reinterpret_cast<uint4*>(o + np) = make_uint4(__byte_perm(x[0], x[1], 0x7632), __byte_perm(x[2], x[3], 0x7632),
                                                           __byte_perm(x[4], x[5], 0x7632), __byte_perm(x[6], x[7], 0x7632));
    }
}

// Both pre-passes of token-major fp32 batches in one: a cluster of up to eight CTAs takes 32 features of
// all N tokens, each CTA a range of tokens that it keeps in shared memory; the features' largest magnitudes
// meet through distributed shared memory, and the scaled fp16 parts leave K-major.  A is read once instead
// of twice and nothing has to be zeroed beforehand (for a small batch it is one launch instead of three).
// VEC: rows of A start on 16 bytes.  12 x 2048 x 3072: 168 -> 124 us (4.9 TB/s) by the bank-conflict-free
// rows below, packed conversions (37 instructions an entry before) and no fence behind the stores.
// In shared memory a feature's tokens lie in a row, in quads whose place is permuted by the feature, so that
// a warp's stores of 8 x 4 features by 4 tokens and its loads of a row's quads meet no bank conflict.
constexpr int TS_FEATURES = 32, TS_THREADS = 4 * TS_FEATURES;
constexpr int TS_TOKENS = 768;                   // most tokens per CTA: 96 KiB of shared memory
__device__ __forceinline__ int ts_at(int f, int t, int pitch) { return f * pitch + (t ^ (f & 28)); }
template <bool VEC>
__global__ void __launch_bounds__(TS_THREADS) k_tokens_split(const float* __restrict__ A, long long lda, int N, int d,
                                                      long long np, int tokens, unsigned* __restrict__ amax,
                                                      __half* __restrict__ hi, __half* __restrict__ lo) {
    grid_trigger();
    extern __shared__ __align__(16) float ts_tile[];     // [TS_FEATURES][pitch]
    __shared__ unsigned s_max[TS_FEATURES];
    __shared__ float s_scale[TS_FEATURES];
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int l = blockIdx.z, f0 = blockIdx.y * TS_FEATURES;
    const int t0 = rank * tokens, t1 = min(N, t0 + tokens), pitch = (tokens + 31) & ~31;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = lane & 7, rr = (lane >> 3) + 4 * warp;
    const float* Al = A + (size_t)l * (size_t)N * (size_t)lda;
    if (tid < TS_FEATURES) s_max[tid] = 0u;
    __syncthreads();
    unsigned m[4] = {0u, 0u, 0u, 0u};
    const int f = f0 + 4 * q;
    const bool whole = VEC && f + 3 < d;
    // places of the tokens rr + 16 k: the permutation takes rr's low bits and exchanges k's parity
    const int swz = (4 * q) & 28;
    float* place = ts_tile + 4 * q * pitch + (rr ^ (swz & 15));
    const int odd = swz & 16;
    constexpr int FLY = 16;                      // 16-byte loads in flight per thread
    for (int t = t0 + rr; t < t1; t += 16 * FLY) {
        float4 v[FLY];
        const float* src = Al + (size_t)t * (size_t)lda + f;
        const size_t step = 16 * (size_t)lda;
        const int n = (t1 - t + 15) >> 4;        // tokens of this thread in the turn, at most FLY
#pragma unroll
        for (int k = 0; k < FLY; ++k, src += step) {
            v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k >= n) continue;
            if (whole) {
                v[k] = __ldcs(reinterpret_cast<const float4*>(src));
            } else {
                if (f < d) v[k].x = src[0];
                if (f + 1 < d) v[k].y = src[1];
                if (f + 2 < d) v[k].z = src[2];
                if (f + 3 < d) v[k].w = src[3];
            }
        }
        float* to = place + (t - t0 - rr);
#pragma unroll
        for (int k = 0; k < FLY; ++k) {
            if (k >= n) break;
            float* o = to + 16 * (k & ~1) + (k & 1 ? 16 - odd : odd);
            m[0] = max(m[0], __float_as_uint(v[k].x) & 0x7fffffffu);
            m[1] = max(m[1], __float_as_uint(v[k].y) & 0x7fffffffu);
            m[2] = max(m[2], __float_as_uint(v[k].z) & 0x7fffffffu);
            m[3] = max(m[3], __float_as_uint(v[k].w) & 0x7fffffffu);
            o[0] = v[k].x;
            o[pitch] = v[k].y;
            o[2 * pitch] = v[k].z;
            o[3 * pitch] = v[k].w;
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {                // the four tokens of a warp's features first
        m[e] = max(m[e], __shfl_xor_sync(0xffffffffu, m[e], 8));
        m[e] = max(m[e], __shfl_xor_sync(0xffffffffu, m[e], 16));
        if (lane < 8) atomicMax(&s_max[4 * q + e], m[e]);
    }
    if (CS > 1) cluster.sync();
    else __syncthreads();
    {
        const int fl = tid >> 2;
        unsigned mx = 0u;
        for (int r = tid & 3; r < CS; r += 4) mx = max(mx, cluster.map_shared_rank(s_max, r)[fl]);
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        if ((tid & 3) == 0) {
            s_scale[fl] = row_scale(mx, false);
            if (rank == 0 && f0 + fl < d) amax[(size_t)l * d + f0 + fl] = mx;
        }
    }
    // The magnitudes stay readable until all have them.  (Nothing else to order: a releasing arrival behind
    // the stores below would wait for them.)
    __syncwarp();
    if (CS > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    __syncthreads();
    // four tokens per lane, a feature per warp and turn
    const int p1 = (int)min(np, (long long)(t0 + tokens));       // the last range also writes the padding
    for (int fl = warp; fl < TS_FEATURES; fl += TS_THREADS / 32) {
        if (f0 + fl >= d) break;
        const float sc = s_scale[fl];
        const size_t row = ((size_t)l * d + f0 + fl) * (size_t)np;
#pragma unroll 2
        for (int t = t0 + 4 * lane; t < p1; t += 128) {
            const float4 x4 = *reinterpret_cast<const float4*>(ts_tile + ts_at(fl, t - t0, pitch));
            const float x[4] = {x4.x, x4.y, x4.z, x4.w};
            float y[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) y[e] = (t + e < t1 ? x[e] : 0.f) * sc;
            uint2 h, w;
            split_f16x2(y, h, w);
            *reinterpret_cast<uint2*>(hi + row + t) = h;
            *reinterpret_cast<uint2*>(lo + row + t) = w;
        }
    }
    __syncwarp();
    if (CS > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// Launch of k_tokens_split: ranges of about 256 tokens (a multiple of 8), more per CTA where eight of them
// do not reach.
ziplm_status run_tokens_split(const float* A, long long lda, int N, int d, long long np, int layers,
                              unsigned* amax, __half* hi, __half* lo, cudaStream_t st) {
    int cs = 1;
    while (cs < 8 && cs * 256 < N) cs *= 2;
    const int tokens = round_up_int((int)((np + cs - 1) / cs), 8);
    const bool vec = (reinterpret_cast<uintptr_t>(A) % 16) == 0 && lda % 4 == 0;
    auto kernel = vec ? k_tokens_split<true> : k_tokens_split<false>;
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          TS_TOKENS * TS_FEATURES * (int)sizeof(float)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, (d + TS_FEATURES - 1) / TS_FEATURES, layers);
    cfg.blockDim = dim3(TS_THREADS);
    cfg.dynamicSmemBytes = (size_t)round_up_int(tokens, 32) * TS_FEATURES * sizeof(float);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kernel, A, lda, N, d, np, tokens, amax, hi, lo));
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

bool quad_rows(const void* A, long long lda) {
    return (reinterpret_cast<uintptr_t>(A) % 16) == 0 && lda % 4 == 0;
}

// 3-D map over a 16-bit [layers, rows, K] with box {128 bytes of K, 128 rows, 1 layer}, 128-byte swizzle,
// zero fill outside the tensor (ragged d and ragged token counts contribute zeros).
bool make_map(CUtensorMap* m, const void* base, ziplm_dtype dt, long long K, int rows, int layers,
              long long pitch_elems) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    const size_t esz = 2;
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)layers};
    cuuint64_t strides[2] = {(cuuint64_t)pitch_elems * esz, (cuuint64_t)pitch_elems * esz * rows};
    cuuint32_t box[3] = {(cuuint32_t)(ROW_BYTES / esz), (cuuint32_t)TM, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(m, dt == ZIPLM_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3,
                     const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

constexpr size_t kSplitCapBytes = (size_t)8 << 30;   // bound on the hi/lo scratch of one chunk

long long padded_tokens_bf16(long long N) { return (N + 7) / 8 * 8; }   // 16-byte row pitch

// Layers per chunk of the K-major bf16 copy of a token-major input.
int transpose_chunk_layers(int L, int d, long long N) {
    const size_t per_layer = (size_t)d * (size_t)padded_tokens_bf16(N) * 2;
    size_t lc = kSplitCapBytes / (per_layer ? per_layer : 1);
    if (lc < 1) lc = 1;
    if (lc > 65535) lc = 65535;
    return (int)(lc < (size_t)L ? lc : (size_t)L);
}

int split_chunk_layers(int L, int d, long long N) {
    const size_t per_layer = 2 * (size_t)d * (size_t)padded_tokens_bf16(N) * 2;
    size_t lc = kSplitCapBytes / (per_layer ? per_layer : 1);
    if (lc < 1) lc = 1;
    return (int)(lc < (size_t)L ? lc : (size_t)L);
}

// Most layers of one product launch.
int product_layers(int L, int d, long long N, ziplm_dtype dt, bool token_major) {
    if (dt == ZIPLM_F32) return split_chunk_layers(L, d, N);
    if (token_major) return transpose_chunk_layers(L, d, N);
    return L < 65535 ? L : 65535;
}

// Scratch of the pair kernel over all product launches of a call.  Kernel and pairs per tile are chosen for the
// layers of a launch, so the last, smaller one may use more than the others (48 x 1600 features of 131072 fp32
// tokens: 10 layers 73 MB, the last 8, with two pairs a tile, 117) or be the only one to use any.
size_t product_scratch_bytes(int L, int d, long long N, ziplm_dtype dt, bool token_major) {
    const int full = product_layers(L, d, N, dt, token_major), last = L % full;
    size_t b = 0;
    for (int layers : {full, last})
        if (layers > 0 && hessian_pair_fits(layers, d, N, dt == ZIPLM_F32)) {
            const size_t need = hessian_pair_scratch_bytes(layers, d, N, dt == ZIPLM_F32);
            if (need > b) b = need;
        }
    return b;
}

}  // namespace

// Where the 128 x 128 tiles leave half of the SMs idle, up to eight CTAs share a tile: the largest power of
// two with which all fit and each keeps four K blocks (one layer of 256 features, 2048 tokens: three tiles,
// a chain of 32 K blocks on one CTA).  `most`: the occupancy calculator's room for clusters of 2, 4 and 8 CTAs on the
// kSMs of a B200, whose GPCs differ in size: what does not fit would wait for a second round (calls with 18
// tiles on clusters of eight and of four: 3 x 333 x 2276 bf16 25.3 and 20.0 us, 18 x 93 x 2000 25.9 and 19.5; with 34
// and 36 on four and on two: 34 x 100 x 1030 fp16 26.0 and 20.4, 6 x 353 x 1142 26.7 and 20.6, 36 x 100 x 1200 fp32
// 39.3 and 33.0).
int hessian_tile_split(long long tiles, long long num_kb) {
    constexpr int most[9] = {0, kSMs, kSMs / 2, 0, 33, 0, 0, 0, 15};
    int split = 1;
    while (split < 8 && tiles <= most[split * 2] && num_kb / (split * 2) >= 4) split *= 2;
    return split;
}

size_t hessian_tc_workspace_bytes(int L, int d, long long N, ziplm_dtype dt, bool token_major) {
    size_t b = kAlign;   // error word
    if (dt == ZIPLM_F32) {
        const int lc = split_chunk_layers(L, d, N);
        b += align_up((size_t)lc * d * sizeof(unsigned));                            // row magnitudes
        b += 2 * align_up((size_t)lc * d * (size_t)padded_tokens_bf16(N) * 2);       // the two fp16 parts
    } else if (token_major) {
        const int lc = transpose_chunk_layers(L, d, N);
        b += align_up((size_t)lc * d * (size_t)padded_tokens_bf16(N) * 2);
    }
    return b + align_up(product_scratch_bytes(L, d, N, dt, token_major));
}

namespace {

// A number that no call had before and that stale scratch does not hold by accident.
unsigned long long next_call() {
    static std::atomic<unsigned long long> calls{
        (unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count() * 0x9e3779b97f4a7c15ull};
    return calls.fetch_add(0x9e3779b97f4a7c15ull) | 1ull;
}

// One product launch on the kernel that suits its number of tiles.
ziplm_status run_product(const HessianProduct& p, void* scratch, size_t scratch_bytes, cudaStream_t st) {
    if (hessian_pair_fits(p.layers, p.d, (long long)p.num_kb * 64, p.split))
        return run_hessian_pair(p, scratch, scratch_bytes, st);
    const int T = (p.d + TM - 1) / TM;
    const long long tiles = (long long)T * (T + 1) / 2 * p.layers;
    const int split = hessian_tile_split(tiles, p.num_kb);
    constexpr int smem2 = Cfg<true>::STAGES * Cfg<true>::TILES * TILE_BYTES + 1024;
    constexpr int smem1 = Cfg<false>::STAGES * Cfg<false>::TILES * TILE_BYTES + 1024;
    static_assert(TM * (PART_PITCH + OUT_PITCH) * (int)sizeof(float) + 1024 <= smem1, "finished tiles fit the operand ring");
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_syrk_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2));
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_syrk_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(T * (T + 1) / 2 * split, p.layers);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = p.split ? smem2 : smem1;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = split;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, p.split ? k_syrk_tc<true> : k_syrk_tc<false>, p.hi,
                                        p.split ? p.lo : p.hi, p.H, p.d, p.num_kb, split, p.alpha, p.beta,
                                        p.layer0, p.L, p.err_word, p.call, p.fmt16, p.spin, p.amax));
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace

ziplm_status run_hessian_tc(float* H, const void* X, ziplm_dtype dt, bool token_major, int L, int d,
                            long long N, long long ldx, float alpha, float beta, void* ws,
                            size_t ws_bytes, cudaStream_t st) {
    if (ws_bytes < hessian_tc_workspace_bytes(L, d, N, dt, token_major)) return ZIPLM_ERR_WORKSPACE;
    const bool f32 = (dt == ZIPLM_F32);
    const uint32_t fmt16 = (dt == ZIPLM_F16) ? 0u : 1u;
    Carver c(ws);
    unsigned long long* err_word = c.take<unsigned long long>(1);
    // A captured call is replayed under one number: there the word is cleared first, so that a replay whose wait
    // ran out does not mark the ones behind it.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    ZIPLM_CHECK_CUDA(cudaStreamIsCapturing(st, &capture));
    if (capture != cudaStreamCaptureStatusNone) ZIPLM_CHECK_CUDA(cudaMemsetAsync(err_word, 0, sizeof(*err_word), st));
    const int spin_opt = option_value(ZIPLM_OPT_SPIN_LIMIT);
    const uint32_t spin = spin_opt > 0 ? (uint32_t)spin_opt : kSpinLimit;
    HessianProduct prod = {};
    prod.H = H; prod.d = d; prod.alpha = alpha; prod.beta = beta; prod.err_word = err_word;
    prod.L = L; prod.call = next_call();
    prod.num_kb = (int)((N + Cfg<false>::BK - 1) / Cfg<false>::BK);
    prod.fmt16 = fmt16; prod.spin = spin; prod.split = f32;
    const size_t scratch_bytes = product_scratch_bytes(L, d, N, dt, token_major);
    void* scratch = nullptr;             // of the pair kernel, behind the operands
    auto take_scratch = [&] { scratch = c.take<char>(scratch_bytes); };
    if (f32) {
        const long long np = padded_tokens_bf16(N);
        const int lc = split_chunk_layers(L, d, N);
        unsigned* amax = c.take<unsigned>((size_t)lc * d);
        __half* hi = c.take<__half>((size_t)lc * d * np);
        __half* lo = c.take<__half>((size_t)lc * d * np);
        take_scratch();
        prod.amax = amax;
        for (int l0 = 0; l0 < L; l0 += lc) {
            const int ln = (L - l0 < lc) ? (L - l0) : lc;
            const size_t rows = (size_t)ln * d;
            if (token_major) {
                const float* Ac = static_cast<const float*>(X) + (size_t)l0 * (size_t)N * ldx;
                const bool one_pass = np <= 8ll * TS_TOKENS;
                if (!one_pass) ZIPLM_CHECK_CUDA(cudaMemsetAsync(amax, 0, sizeof(unsigned) * rows, st));
                // slabs of AM_SLAB tokens, shorter ones where those would leave SMs idle, at most 65535 of them (grid.y)
                const long long columns = (long long)((d + 255) / 256) * ln;
                long long slab = (N * columns / (8 * kSMs) + AM_FLY) / AM_FLY * AM_FLY;
                if (slab > AM_SLAB) slab = AM_SLAB;
                if (slab < N / 65535 + 1) slab = N / 65535 + 1;
                // grid.z is limited to 65535 layers per launch
                for (int z0 = 0; z0 < ln; z0 += 65535) {
                    const int zn = ln - z0 < 65535 ? ln - z0 : 65535;
                    if (one_pass) {
                        const ziplm_status s = run_tokens_split(Ac + (size_t)z0 * N * ldx, ldx, (int)N, d, np, zn,
                                                                amax + (size_t)z0 * d, hi + (size_t)z0 * d * np,
                                                                lo + (size_t)z0 * d * np, st);
                        if (s != ZIPLM_OK) return s;
                        continue;
                    }
                    k_tokens_absmax<<<dim3((unsigned)((d + 255) / 256), (unsigned)((N + slab - 1) / slab),
                                           (unsigned)zn), 256, 0, st>>>(Ac + (size_t)z0 * N * ldx, ldx, N, d, slab,
                                                                        amax + (size_t)z0 * d);
                    ZIPLM_CHECK_LAUNCH();
                    auto move = quad_rows(X, ldx) ? k_tokens_to_kmajor<true> : k_tokens_to_kmajor<false>;
                    move<<<dim3((unsigned)((np + 63) / 64), (unsigned)((d + 63) / 64), (unsigned)zn), 256, 0, st>>>(
                        Ac + (size_t)z0 * N * ldx, ldx, N, d, np, amax + (size_t)z0 * d, hi + (size_t)z0 * d * np,
                        lo + (size_t)z0 * d * np);
                    ZIPLM_CHECK_LAUNCH();
                }
            } else {
                const float* Xc = static_cast<const float*>(X) + (size_t)l0 * d * ldx;
                // rows of up to 16384 tokens stay in registers: 1, 4 or 16 quads per thread
                if (np <= 256ll * 4 * 16) {
                    for (size_t r0 = 0; r0 < rows; r0 += (size_t)1 << 30) {
                        const size_t rn = rows - r0 < ((size_t)1 << 30) ? rows - r0 : ((size_t)1 << 30);
                        const float* xs = Xc + r0 * ldx;
                        if (np <= 256ll * 4)
                            k_row_absmax_split<1><<<(unsigned)rn, 256, 0, st>>>(xs, ldx, N, np, amax + r0,
                                                                                hi + r0 * np, lo + r0 * np);
                        else if (np <= 256ll * 4 * 4)
                            k_row_absmax_split<4><<<(unsigned)rn, 256, 0, st>>>(xs, ldx, N, np, amax + r0,
                                                                                hi + r0 * np, lo + r0 * np);
                        else
                            k_row_absmax_split<16><<<(unsigned)rn, 256, 0, st>>>(xs, ldx, N, np, amax + r0,
                                                                                 hi + r0 * np, lo + r0 * np);
                        ZIPLM_CHECK_LAUNCH();
                    }
                } else {
                    for (size_t r0 = 0; r0 < rows; r0 += (size_t)1 << 30) {
                        const size_t rn = rows - r0 < ((size_t)1 << 30) ? rows - r0 : ((size_t)1 << 30);
                        k_row_absmax<<<(unsigned)rn, 256, 0, st>>>(Xc + r0 * ldx, ldx, N, amax + r0);
                        ZIPLM_CHECK_LAUNCH();
                    }
                    // grid.y is limited to 65535 rows per launch
                    for (size_t r0 = 0; r0 < rows; r0 += 65535) {
                        const size_t rn = rows - r0 < 65535 ? rows - r0 : 65535;
                        k_split_f16<<<dim3((unsigned)((np / 4 + 255) / 256), (unsigned)rn), 256, 0, st>>>(
                            Xc + r0 * ldx, ldx, N, np, rn, amax + r0, hi + r0 * np, lo + r0 * np);
                        ZIPLM_CHECK_LAUNCH();
                    }
                }
            }
            if (!make_map(&prod.hi, hi, ZIPLM_F16, N, d, ln, np) || !make_map(&prod.lo, lo, ZIPLM_F16, N, d, ln, np))
                return ZIPLM_ERR_CUDA;
            prod.layer0 = l0; prod.layers = ln;
            const ziplm_status s = run_product(prod, scratch, scratch_bytes, st);
            if (s != ZIPLM_OK) return s;
        }
    } else if (token_major) {
        // K-major bf16 copy of a chunk of layers, then the same product kernel
        const long long np = padded_tokens_bf16(N);
        const int lc = transpose_chunk_layers(L, d, N);
        uint16_t* xt = c.take<uint16_t>((size_t)lc * d * np);
        take_scratch();
        for (int l0 = 0; l0 < L; l0 += lc) {
            const int ln = (L - l0 < lc) ? (L - l0) : lc;
            const uint16_t* Ac = static_cast<const uint16_t*>(X) + (size_t)l0 * (size_t)N * ldx;
            const bool pairs = ldx % 2 == 0 && reinterpret_cast<uintptr_t>(X) % 4 == 0;
            const bool small = !pairs && (np + 127) / 128 * ((d + 63) / 64) * ln < kSMs;
            auto move = pairs ? k_tokens16_to_kmajor<true, 128>
                              : small ? k_tokens16_to_kmajor<false, 32> : k_tokens16_to_kmajor<false, 128>;
            const int tokens = small ? 32 : 128;
            move<<<dim3((unsigned)((np + tokens - 1) / tokens), (unsigned)((d + 63) / 64), (unsigned)ln), 256, 0, st>>>(
                Ac, ldx, N, d, np, xt);
            ZIPLM_CHECK_LAUNCH();
            if (!make_map(&prod.hi, xt, dt, N, d, ln, np)) return ZIPLM_ERR_CUDA;
            prod.lo = prod.hi; prod.layer0 = l0; prod.layers = ln;
            const ziplm_status s = run_product(prod, scratch, scratch_bytes, st);
            if (s != ZIPLM_OK) return s;
        }
    } else {
        take_scratch();
        // tensor-map dimensions are 32-bit boxes over up to 2^32 elements; chunk layers so that the
        // grid stays within limits
        for (int l0 = 0; l0 < L; l0 += 65535) {
            const int ln = (L - l0 < 65535) ? (L - l0) : 65535;
            const __nv_bfloat16* Xc = static_cast<const __nv_bfloat16*>(X) + (size_t)l0 * d * ldx;
            if (!make_map(&prod.hi, Xc, dt, N, d, ln, ldx)) return ZIPLM_ERR_CUDA;
            prod.lo = prod.hi; prod.layer0 = l0; prod.layers = ln;
            const ziplm_status s = run_product(prod, scratch, scratch_bytes, st);
            if (s != ZIPLM_OK) return s;
        }
    }
    return ZIPLM_OK;
}

}  // namespace ziplm
