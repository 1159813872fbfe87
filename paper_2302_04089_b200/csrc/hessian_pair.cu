// Calibration Hessian on CTA pairs: the product kernel for problems of many tiles.
//
// Same contraction, operands and numerics as k_syrk_tc (hessian_tc.cu), on tiles of 256 x 256 that a
// pair of CTAs computes together with tcgen05.mma.cta_group::2 (M = N = 256): each CTA holds 128 rows of
// both operands in its shared memory and 128 rows of the product in its tensor memory.  The 128 x 128
// kernel was bound by its operand traffic from L2 (64 KB per K block of split fp32 against 800 clocks of
// MMAs, about 40 B per clock and SM arrive): a pair moves the same bytes per CTA for twice the products.
//
// Tensor memory holds two accumulators of 256 columns, drained in turn after every chunk of K into fp32
// registers (accumulation in tensor memory truncates, so a chain is kept to at most eight MMAs of the
// main term).  There is no room for a third accumulator for the cross terms X_1 X_2^T + X_2 X_1^T of
// split fp32: they go first into the chunk's own accumulator, where they meet nothing but each other
// (2^-11 of the main term, so what their truncation loses is negligible), and the main term follows on
// top.  The partial sums are added in two levels; 64 columns of running sums per thread fill the
// registers, so the second level is a tile of scratch in global memory (in L2) that every FOLD drains
// are added to with red.add: one writer per address, so the sums are the same on every run.
//
// Roles of a CTA: warp 0 loads its own half of the operands by TMA (no multicast; the bytes of both
// halves are counted on the leader's barrier), one thread of warp 1 of the leader issues the MMAs for
// both CTAs, warps 2 .. 17 drain (four TMEM lane quarters x four quarters of the columns).  Every wait
// is bounded; a role that gives up raises the abort flag of both CTAs.
#include <cuda.h>

#include "common.cuh"
#include "hessian_common.cuh"
#include "tc_common.cuh"

namespace ziplm {
namespace {
using namespace tc;

constexpr int PT = 256;                       // tile rows / columns of a pair
constexpr int HALF = 128;                     // rows of an operand per CTA
constexpr int BK = 64;                        // K block: one 128-byte swizzle row of 16-bit elements
constexpr int OP_BYTES = HALF * 128;          // one operand half, one part, one K block: 16 KiB
constexpr int PAIR_EPI = 16;                  // epilogue warps
constexpr int PAIR_THREADS = 32 * (2 + PAIR_EPI);
constexpr int FOLD = 32;                      // drains between additions to the second level
constexpr int NC = 64;                        // columns per epilogue thread
constexpr int OUT_PITCH = NC + 4;             // of the results in shared memory: rows on 16 bytes
constexpr int FLY = 8;                        // rows whose old values are requested together

template <bool SPLIT> struct PairCfg;         // SPLIT: two fp16 parts per operand (fp32 inputs)
template <> struct PairCfg<true>  { static constexpr int STAGES = 3, PARTS = 2, CHUNK = 1; };
template <> struct PairCfg<false> { static constexpr int STAGES = 6, PARTS = 1, CHUNK = 2; };
template <bool SPLIT>
constexpr int kStageBytes = 2 * PairCfg<SPLIT>::PARTS * OP_BYTES;      // A half and B half
template <bool SPLIT>
constexpr int kPairSmem = PairCfg<SPLIT>::STAGES * kStageBytes<SPLIT> + 1024;

__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}

// The end of a tile that n_parts pairs have shared.  Every thread of the cluster's CTAs comes here once the
// parts' sums are in shared memory, [16 quads][512 threads].  Part p finishes the quads [16 p / n, 16 (p + 1) / n)
// of every epilogue thread's 64 columns: sums over the parts in order, rows along the columns, mirrored rows
// along the rows.
template <bool SPLIT>
__device__ __forceinline__ void finish_parts(uint8_t* ring, int n_parts, int part, int rank, int i0, int j0, int d,
                                             float alpha, float beta, float* Hl, const unsigned* am,
                                             const unsigned long long* err_word, unsigned long long call, bool give_up) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, et = (int)threadIdx.x - 64;
    const int g0 = 16 * part / n_parts, n = 16 * (part + 1) / n_parts - g0;      // at most eight quads
    float4 sum[8];
    if (warp >= 2) {
        const uint32_t mine = smem_u32(ring) + 16u * (uint32_t)(g0 * (32 * PAIR_EPI) + et);
#pragma unroll
        for (int e = 0; e < 8; ++e) sum[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p = 0; p < n_parts; ++p) {
            const uint32_t from = cluster_addr(mine, 2u * (uint32_t)p + (uint32_t)rank);
            float4 x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (e < n)
                    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                                 : "=f"(x[e].x), "=f"(x[e].y), "=f"(x[e].z), "=f"(x[e].w)
                                 : "r"(from + 16u * (uint32_t)(e * 32 * PAIR_EPI)) : "memory");
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (e < n) { sum[e].x += x[e].x; sum[e].y += x[e].y; sum[e].z += x[e].z; sum[e].w += x[e].w; }
        }
    }
    __syncwarp();
    cluster_barrier();                                    // all have read: the sums' place is free
    if (warp < 2 || give_up) return;
    const int q = warp & 3, cols = 4 * n;
    const int r0 = i0 + rank * HALF + q * 32, c0 = j0 + ((warp - 2) >> 2) * NC + 4 * g0;
    float* buf = reinterpret_cast<float*>(ring) + (warp - 2) * (32 * 33);
    const float mul = (SPLIT && r0 + lane < d) ? row_scale(am[r0 + lane], true) : 1.f;
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (e < n) {
            float* b = buf + lane * 33 + 4 * e;
            b[0] = (alpha * sum[e].x) * mul;
            b[1] = (alpha * sum[e].y) * mul;
            b[2] = (alpha * sum[e].z) * mul;
            b[3] = (alpha * sum[e].w) * mul;
        }
    __syncwarp();
    const int col = c0 + lane;
    const float sc = SPLIT && lane < cols && col < d ? row_scale(am[col], true) : 1.f;
#pragma unroll 1
    for (int g = 0; g < 32; g += 16) {
        float old[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int row = r0 + g + k;
            old[k] = beta != 0.f && lane < cols && row < d && col <= row ? Hl[(size_t)row * d + col] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int row = r0 + g + k;
            if (lane >= cols || row >= d || col > row) continue;
            const float v = buf[(g + k) * 33 + lane] * sc + old[k];
            buf[(g + k) * 33 + lane] = v;
            float* p = Hl + (size_t)row * d + col;
            *p = v;
            if ((row | col) == 0) hessian_check(p, err_word, call);
        }
    }
    __syncwarp();
    const int row = r0 + lane;
#pragma unroll 4
    for (int e = 0; e < cols; ++e)
        if (row < d && c0 + e < row) Hl[(size_t)(c0 + e) * d + row] = buf[lane * 33 + e];
}

template <bool SPLIT>
__global__ void __launch_bounds__(PAIR_THREADS, 1)
k_syrk_pair(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
            float* __restrict__ H, int d, int num_kb_all, int n_parts, float alpha, float beta, int layer0,
            int L, unsigned long long* err_word, unsigned long long call, uint32_t fmt16, uint32_t empty_spin_limit,
            const unsigned* __restrict__ amax, float4* __restrict__ level2, int quads) {
    using C = PairCfg<SPLIT>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_full[C::STAGES], bar_empty[C::STAGES], bar_acc_full[2], bar_acc_empty[2], bar_final;
    __shared__ uint64_t bar_report;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, reported;

    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles = (raw + 1023u) & ~1023u;        // swizzled tiles need 1024-byte alignment
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a cluster of n_parts pairs shares a tile, each a range of its K blocks
    const uint32_t rank = blockIdx.x & 1u;                // CTA of the pair; 0 leads
    const int part = (int)(blockIdx.x >> 1) % n_parts;
    const uint32_t lead = 2u * (uint32_t)part;            // cluster rank of the pair's leader
    const uint16_t both = (uint16_t)(3u << lead);
    const int kb_begin = (int)((long long)num_kb_all * part / n_parts);
    const int num_kb = (int)((long long)num_kb_all * (part + 1) / n_parts) - kb_begin;
    const int l = blockIdx.y;                             // layer within the launched chunk
    int ti = 0, rem = (int)(blockIdx.x >> 1) / n_parts;
    while (rem > ti) { rem -= ti + 1; ++ti; }
    const int tj = rem;
    const int i0 = ti * PT, j0 = tj * PT;
    const bool diag = (ti == tj);
    const int num_chunks = (num_kb + C::CHUNK - 1) / C::CHUNK;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_acc_full[b]), 1);
            mbar_init(smem_u32(&bar_acc_empty[b]), 2 * PAIR_EPI);     // every epilogue warp of both CTAs
        }
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
    cluster_barrier();                                    // both CTAs' barriers are initialised
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    grid_wait();                                          // the operands are there
    const uint32_t tmem_base = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    bool failed = false;
    int issued = 0;                                       // K blocks whose copies were started (thread 0)
    auto bytes = [&](int) { return (uint32_t)((diag ? 1 : 2) * C::PARTS * OP_BYTES); };     // of a K block, per CTA

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer (each CTA its own half of the operands)
            const int ya = i0 + (int)rank * HALF, yb = j0 + (int)rank * HALF;
            const uint32_t full0 = cluster_addr(smem_u32(&bar_full[0]), lead);
            int s = 0;
            uint32_t ph = 1u;
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!mbar_wait_limit(smem_u32(&bar_empty[s]), ph, abortp, empty_spin_limit)) {
                    failed = true;
                    break;
                }
                const uint32_t full = full0 + 8u * (uint32_t)s;
                const uint32_t base = tiles + (uint32_t)s * kStageBytes<SPLIT>;
                if (rank == 0) mbar_expect_tx(smem_u32(&bar_full[s]), 2 * bytes(kb));
                const int x = (kb_begin + kb) * BK;
                tma_load_3d_pair(base, &map_hi, full, x, ya, l);
                if (SPLIT) tma_load_3d_pair(base + OP_BYTES, &map_lo, full, x, ya, l);
                if (!diag) {
                    tma_load_3d_pair(base + C::PARTS * OP_BYTES, &map_hi, full, x, yb, l);
                    if (SPLIT) tma_load_3d_pair(base + 3 * OP_BYTES, &map_lo, full, x, yb, l);
                }
                issued = kb + 1;
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
            if (rank == 1)
                pair_report(cluster_addr(smem_u32(&reported), lead), cluster_addr(smem_u32(&bar_report), lead), issued);
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // ---------------- MMA issuer (the leader, for both CTAs)
            const uint32_t idesc = make_idesc(SPLIT ? 0u : fmt16, PT, PT);
            // One thread issues every MMA of the pair, 128 clocks of tensor-core time each, so the code
            // between two MMAs has to be short: stage and phase are counted, descriptors are one addition.
            const uint64_t desc0 = make_desc(tiles);
            const uint32_t b_off = diag ? 0u : (uint32_t)(C::PARTS * OP_BYTES / 16);
            int s = 0, kb = 0;
            uint32_t ph = 0u;
            for (int c = 0; c < num_chunks && !failed; ++c) {
                const int b = c & 1;
                const uint32_t acc = tmem_base + (uint32_t)b * PT;
                // both CTAs must have drained this buffer (first use of each buffer passes)
                if (!mbar_wait(smem_u32(&bar_acc_empty[b]), (((uint32_t)c >> 1) & 1u) ^ 1u, abortp)) {
                    failed = true;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int j = 0; j < C::CHUNK; ++j) {
                    if (j > 0 && kb >= num_kb) break;
                    if (!mbar_wait(smem_u32(&bar_full[s]), ph, abortp)) { failed = true; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t a_hi = desc0 + (uint32_t)(s * (kStageBytes<SPLIT> / 16)), b_hi = a_hi + b_off;
                    if (SPLIT) {
                        const uint64_t a_lo = a_hi + OP_BYTES / 16, b_lo = b_hi + OP_BYTES / 16;
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {       // 32 bytes per MMA along K
                            umma_pair(acc, a_hi + 2u * k, b_lo + 2u * k, idesc, k > 0 || j > 0);
                            umma_pair(acc, a_lo + 2u * k, b_hi + 2u * k, idesc, 1u);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        umma_pair(acc, a_hi + 2u * k, b_hi + 2u * k, idesc, SPLIT || k > 0 || j > 0);
                    umma_commit_pair(smem_u32(&bar_empty[s]), both);     // stage free once these MMAs have read it
                    ++kb;
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
                if (!failed) umma_commit_pair(smem_u32(&bar_acc_full[b]), both);
            }
            // whatever was issued has completed before tensor memory is given back
            umma_commit_pair(smem_u32(&bar_final), both);
            mbar_wait_quiet(smem_u32(&bar_final), 0u);
        }
    } else {
        // ---------------- epilogue: lane quarter = warp % 4, quarter of the columns by warp
        const int q = warp & 3, cq = (warp - 2) >> 2;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        const uint32_t empty0 = cluster_addr(smem_u32(&bar_acc_empty[0]), lead);
        const uint32_t empty1 = cluster_addr(smem_u32(&bar_acc_empty[1]), lead);
        const int et = (int)threadIdx.x - 64;
        float4* l2 = level2 + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * (HALF * PT / 4) + et;
        float acc[NC];
#pragma unroll
        for (int e = 0; e < NC; ++e) acc[e] = 0.f;
        bool folded = false;
        for (int c = 0; c < num_chunks; ++c) {
            const int b = c & 1;
            if (!mbar_wait(smem_u32(&bar_acc_full[b]), ((uint32_t)c >> 1) & 1u, abortp)) failed = true;
            failed = __any_sync(0xffffffffu, failed);
            if (failed) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int cc = 0; cc < NC / 16; ++cc) {
                uint32_t v[16];
                tmem_ld16(tmem_base + lane_base + (uint32_t)(b * PT + cq * NC + cc * 16), v);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) acc[cc * 16 + e] += __uint_as_float(v[e]);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(b ? empty1 : empty0);
            if ((c % FOLD) == FOLD - 1 && c + 1 < num_chunks) {
                // second level, [16 quads][512 threads]
#pragma unroll
                for (int e = 0; e < NC / 4; ++e) {
                    float4* p = l2 + (size_t)e * (32 * PAIR_EPI);
                    if (folded)
                        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(acc[4 * e]),
                                     "f"(acc[4 * e + 1]), "f"(acc[4 * e + 2]), "f"(acc[4 * e + 3]) : "memory");
                    else
                        __stcg(p, make_float4(acc[4 * e], acc[4 * e + 1], acc[4 * e + 2], acc[4 * e + 3]));
                    acc[4 * e] = acc[4 * e + 1] = acc[4 * e + 2] = acc[4 * e + 3] = 0.f;
                }
                folded = true;
            }
        }
        if (!failed) {
            if (folded)
#pragma unroll
                for (int e = 0; e < NC / 4; ++e) {
                    const float4 t = __ldcg(l2 + (size_t)e * (32 * PAIR_EPI));
                    acc[4 * e] += t.x; acc[4 * e + 1] += t.y; acc[4 * e + 2] += t.z; acc[4 * e + 3] += t.w;
                }
            if (n_parts > 1) {
                // The operand ring is free (every MMA has completed): the part's sums wait there for finish_parts.
                float4* mine = reinterpret_cast<float4*>(smem_raw + (tiles - raw)) + et;
#pragma unroll
                for (int e = 0; e < NC / 4; ++e)
                    mine[e * (32 * PAIR_EPI)] = make_float4(acc[4 * e], acc[4 * e + 1], acc[4 * e + 2], acc[4 * e + 3]);
            } else {
                // The operand ring is free (every MMA has completed): the warp's 32 x 64 results pass
                // through it, so that rows [i][j] leave along j and mirrored rows [j][i] along i.  The old values
                // of several rows are requested together: a load behind every row's store made a call with
                // beta = 1 take 1056 us where beta = 0 took 667 (12 x 3072 x 2048 fp32).
                float* buf = reinterpret_cast<float*>(smem_raw + (tiles - raw)) + (size_t)(warp - 2) * 32 * OUT_PITCH;
                float* Hl = H + (size_t)(layer0 + l) * d * d;
                const int r0 = i0 + (int)rank * HALF + q * 32, c0 = j0 + cq * NC;
                const unsigned* am = SPLIT ? amax + (size_t)l * d : nullptr;
                // split route: undo the power-of-two scales of the two feature rows (exact)
                const float mul = (SPLIT && r0 + lane < d) ? row_scale(am[r0 + lane], true) : 1.f;
#pragma unroll
                for (int e = 0; e < NC; e += 4)
                    *reinterpret_cast<float4*>(buf + lane * OUT_PITCH + e) =
                        make_float4((alpha * acc[e]) * mul, (alpha * acc[e + 1]) * mul, (alpha * acc[e + 2]) * mul,
                                    (alpha * acc[e + 3]) * mul);
                __syncwarp();
                if (!diag && quads && r0 + 32 <= d) {
                    // whole rows below the diagonal that start on 16 bytes: 16 lanes take one, 16 bytes each
                    const int cc = 4 * (lane & 15);
                    float sc[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) sc[e] = SPLIT ? row_scale(am[c0 + cc + e], true) : 1.f;
                    float4* out = reinterpret_cast<float4*>(Hl + (size_t)(r0 + (lane >> 4)) * d + c0 + cc);
                    float4* in = reinterpret_cast<float4*>(buf + (lane >> 4) * OUT_PITCH + cc);
#pragma unroll
                    for (int g = 0; g < 16; g += FLY) {
                        float4 old[FLY];
                        if (beta != 0.f)
#pragma unroll
                            for (int k = 0; k < FLY; ++k) old[k] = out[(size_t)(g + k) * (2 * (d / 4))];
#pragma unroll
                        for (int k = 0; k < FLY; ++k) {
                            float4 v = in[(g + k) * (2 * OUT_PITCH / 4)];
                            v.x *= sc[0]; v.y *= sc[1]; v.z *= sc[2]; v.w *= sc[3];
                            if (beta != 0.f) { v.x += old[k].x; v.y += old[k].y; v.z += old[k].z; v.w += old[k].w; }
                            out[(size_t)(g + k) * (2 * (d / 4))] = v;
                            in[(g + k) * (2 * OUT_PITCH / 4)] = v;
                        }
                    }
                    __syncwarp();
                    float* mir = Hl + (size_t)c0 * d + r0 + lane;
#pragma unroll
                    for (int e = 0; e < NC; e += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(buf + lane * OUT_PITCH + e);
                        mir[(size_t)e * d] = v.x;
                        mir[(size_t)(e + 1) * d] = v.y;
                        mir[(size_t)(e + 2) * d] = v.z;
                        mir[(size_t)(e + 3) * d] = v.w;
                    }
                } else {
                    float sc[NC / 32];
#pragma unroll
                    for (int h = 0; h < NC / 32; ++h)
                        sc[h] = SPLIT && c0 + 32 * h + lane < d ? row_scale(am[c0 + 32 * h + lane], true) : 1.f;
#pragma unroll 1
                    for (int g = 0; g < 32; g += FLY) {
                        float old[FLY][NC / 32];
#pragma unroll
                        for (int k = 0; k < FLY; ++k)
#pragma unroll
                            for (int h = 0; h < NC / 32; ++h) {
                                const int row = r0 + g + k, col = c0 + 32 * h + lane;
                                old[k][h] = beta != 0.f && row < d && col <= row ? Hl[(size_t)row * d + col] : 0.f;
                            }
#pragma unroll
                        for (int k = 0; k < FLY; ++k)
#pragma unroll
                            for (int h = 0; h < NC / 32; ++h) {
                                const int row = r0 + g + k, col = c0 + 32 * h + lane;
                                if (row >= d || col > row) continue;
                                float* b = buf + (g + k) * OUT_PITCH + 32 * h + lane;
                                const float v = *b * sc[h] + old[k][h];
                                *b = v;
                                float* p = Hl + (size_t)row * d + col;
                                *p = v;
                                if ((row | col) == 0) hessian_check(p, err_word, call);
                            }
                    }
                    __syncwarp();
                    const int row = r0 + lane;
#pragma unroll 4
                    for (int e = 0; e < NC; ++e) {
                        const int col = c0 + e;
                        if (row < d && col < row) Hl[(size_t)col * d + row] = buf[lane * OUT_PITCH + e];
                    }
                }
            }
        }
    }

    if (failed) {
        hessian_give_up(H, L, d, err_word, call);
        for (uint32_t r = 0; r < 2; ++r) cluster_store(cluster_addr(smem_u32(&abort_flag), lead + r), 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && rank == 0 && abort_flag)
        pair_land<C::STAGES>(bar_full, issued, smem_u32(&bar_report), &reported, bytes);
    __syncwarp();
    cluster_barrier();            // the pair's MMAs, copies and remote arrivals are over
    if (n_parts > 1)
        finish_parts<SPLIT>(smem_raw + (tiles - raw), n_parts, part, (int)rank, i0, j0, d, alpha, beta,
                            H + (size_t)(layer0 + l) * d * d, SPLIT ? amax + (size_t)l * d : nullptr, err_word, call,
                            abort_flag != 0);
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

int pair_count(int d) {
    const int T = (d + PT - 1) / PT;
    return T * (T + 1) / 2;
}

// Pairs that share a tile: the number with the shortest chain of K blocks over all waves, where the tiles leave
// SMs idle or a second wave nearly empty (most_clusters: the occupancy calculator's room for clusters of that
// many pairs on the kSMs of a B200, whose GPCs differ in size); the ends of a tile weigh 14 to 28 K blocks.
// Four K blocks each at least.  8 x 512 features, 2048 bf16 tokens: 39.8 -> 29.7 us a call, 2 x 1100 of 500
// fp32 37.7 -> 27.6, 1 x 1322 of 4099 64.5 -> 58.3, 1 x 3072 of 8192 (78 tiles) 347 -> 304.
int most_clusters(int parts) {
    constexpr int n[5] = {0, kSMs / 2, 33, 22, 15};
    return n[parts];
}
int parts_of(long long pairs, long long kb) {
    int parts = 1;
    long long best = 0;
    for (int p = 1; p <= 4; ++p) {
        if (p > 1 && kb / p < 4) break;
        const long long cost = (pairs + most_clusters(p) - 1) / most_clusters(p) * ((kb + p - 1) / p + 20);
        if (p == 1 || cost < best) { best = cost; parts = p; }
    }
    return parts;
}

template <bool SPLIT>
ziplm_status launch_pair(const HessianProduct& p, float4* level2, cudaStream_t st) {
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_syrk_pair<SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          kPairSmem<SPLIT>));
    const int parts = parts_of((long long)pair_count(p.d) * p.layers, p.num_kb);
    const int quads = p.d % 4 == 0 && reinterpret_cast<uintptr_t>(p.H) % 16 == 0;     // rows of H start on 16 bytes
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * parts * pair_count(p.d), p.layers);
    cfg.blockDim = dim3(PAIR_THREADS);
    cfg.dynamicSmemBytes = kPairSmem<SPLIT>;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2 * parts;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k_syrk_pair<SPLIT>, p.hi, p.lo, p.H, p.d, p.num_kb, parts, p.alpha,
                                        p.beta, p.layer0, p.L, p.err_word, p.call, p.fmt16, p.spin, p.amax, level2,
                                        quads));
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace

// A K block of a 256 x 256 tile takes a pair about 4/3 of the time that one of a 128 x 128 tile takes a CTA
// (12 MMAs of 128 clocks against 12 of 92, where the shared-memory reads of a 128 x 128 MMA bound it).  The end of a
// tile of 16-bit input weighs as much as eight of its K blocks, six where a pair has a tile to itself.  The lines lie where
// the device times of the two kernels' calls cross (us, pairs and CTAs): 1 x 1000 x 4000 27.0 and 34.7, 1 x 1322 x 4099
// 28.7 and 29.3, 1 x 1700 x 2000 25.5 and 29.4, 1 x 1884 x 15943 123 and 138, 13 x 237 x 4318 45.9 and 47.3;
// 2 x 1000 x 2000 25.3 and 22.6, 2 x 1400 x 2000 34.5 and 30.8, 2 x 502 x 19169 61.1 and 54.8, 5 x 314 x 750 20.6 and
// 16.4.  Of fp32 the K blocks alone count: pairs sum it the more exactly (6 x 287 x 843: 1.4e-8 of the diagonal in the
// mean square against 2.7e-8, 28.2 us against 22.6; 1 x 1000 x 4000: 7e-9 against 15e-9, 41.1 us against 47.3).
bool hessian_pair_fits(int layers, int d, long long N, bool split) {
    const long long kb = (N + BK - 1) / BK, T = (d + HALF - 1) / HALF, tiles = T * (T + 1) / 2 * layers;
    const long long pairs = (long long)pair_count(d) * layers, parts = parts_of(pairs, kb);
    const long long share = hessian_tile_split(tiles, kb);
    const long long end = split ? 0 : parts > 1 ? 8 : 6, other_end = split ? 0 : 8;
    const long long cost = (pairs + most_clusters(parts) - 1) / most_clusters(parts) * ((kb + parts - 1) / parts + end);
    return 4 * cost < 3 * ((tiles * share + kSMs - 1) / kSMs * ((kb + share - 1) / share + other_end));
}

// Scratch of the second summation level, for the layers of one launch; none where FOLD drains are
// never reached.
size_t hessian_pair_scratch_bytes(int layers, int d, long long N, bool split) {
    const long long kb = (N + BK - 1) / BK, per = split ? PairCfg<true>::CHUNK : PairCfg<false>::CHUNK;
    const long long pairs = (long long)pair_count(d) * layers, parts = parts_of(pairs, kb);
    if (((kb + parts - 1) / parts + per - 1) / per <= FOLD) return 0;
    return (size_t)2 * pairs * parts * HALF * PT * sizeof(float);
}

ziplm_status run_hessian_pair(const HessianProduct& p, void* scratch, size_t scratch_bytes, cudaStream_t st) {
    if (hessian_pair_scratch_bytes(p.layers, p.d, (long long)p.num_kb * BK, p.split) > scratch_bytes)
        return ZIPLM_ERR_WORKSPACE;
    float4* l2 = static_cast<float4*>(scratch);
    return p.split ? launch_pair<true>(p, l2, st) : launch_pair<false>(p, l2, st);
}

}  // namespace ziplm
