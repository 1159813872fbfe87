// Greedy one-column-at-a-time structured OBS with delayed (blocked) updates.
//
// Same arithmetic as the streaming neuron path (Algorithm 1 with |M_S| = 1; Eq. 2, 3, 4), but
// the rank-1 updates of a block of up to B steps are kept pending and applied together:
//
//   * Only three things are needed exactly at every step: the saliencies, the pivot column of
//     H^-1 and the pivot column of W.  With Q = W^T W (Gram matrix of the weight columns)
//         rho_k = Q[k,k] / H^-1[k,k]                                               (Eq. 2)
//     and one step (pivot p, h = H^-1[p,p], u = H^-1[:,p]/sqrt(h), q = Q[:,p]/sqrt(h),
//     z = q - Q[p,p]/(2h) u) acts as
//         H^-1 <- H^-1 - u u^T                                                     (Eq. 4)
//         Q    <- Q - z u^T - u z^T      (the Gram matrix of W - c u^T, c = W[:,p]/sqrt(h): Eq. 3)
//     so both diagonals are downdated exactly (float64) from the pivot columns alone, and a
//     pivot column of the true matrix is the stale column minus the pending terms evaluated at
//     p -- O(n * pending) work instead of a pass over n^2 entries.
//   * At the end of a block the pending terms are applied to H^-1, Q and W as rank-B updates
//     (one read + write of each matrix per B steps instead of per step).  Removed positions stay in
//     place for a few blocks (idx = -1), then a block squeezes them out by a stable, out-of-place
//     compaction, so the live problem is again the leading n x n corner in original column order.
//
// B is 64 where the pending vectors of a slice fit shared memory on up to eight CTAs (up to 3072 positions),
// less above (48 up to 4096), and 32 in a block that squeezes: the update moves the same bytes for twice the
// steps (12 x 3072: 27.3 -> 24.4 ms with all other work, 24 x 4096: 107 -> 99, 12 x 1814: 12.1 -> 11.1).
//
// Launches per block, for all L layers at once: one "steps" kernel (one thread-block cluster per
// layer runs the B greedy steps back to back; its CTAs exchange their offers by asynchronous stores,
// and layers are independent, so a step has neither a cluster barrier nor a grid-wide one) and one
// update kernel, or two where the block squeezes removed positions out.  Block boundaries are placed
// on the requested levels, where W is up to date and can be snapshotted.
//
// Layout per layer: A, Q fp32 [d, d], off-diagonal entries in both triangles (two buffers each, ping-pong),
// Wt = W^T fp32 [d, rp] (two buffers), float64 diagonals, pending U, Z [B, d] and C [B, rp].
#include <cooperative_groups.h>
#include <math.h>

#include <cuda.h>

#include "common.cuh"
#include "lazy_common.cuh"
#include "pick.cuh"
#include "tc_common.cuh"

namespace ziplm {

namespace {

constexpr int GS = kPackSteps;   // steps per group of packed operands, and at most in a compaction block
constexpr int BMAX = kPackGroups * GS;   // pending steps per dense block, at most
constexpr int STEP_THREADS = 256; // threads per CTA of the steps kernel, four positions each
constexpr int SLICE_MAX = 768;   // positions per CTA
constexpr int SLICE_WIDE = 384;  // ... up to which BMAX steps are pending
constexpr int STEPS_SMEM = 2 * BMAX * (SLICE_WIDE + 4) * 4;    // bytes of pending vectors per CTA
constexpr int CLUSTER_MAX = 8;   // portable cluster size
// Removed positions tolerated in the arrays before they are squeezed out, or this fraction of all positions,
// whichever comes first.  12 x 3072 / 24 x 4096 / 12 x 1814: 24.6 / 98 / 11.4 ms with 256 and a twelfth, 24.4 / 99 /
// 11.1 with 320 and an eighth or 384 and an eighth, 24.4 / 100 / 11.1 with 512 and a sixth.
constexpr int kDeadMax = 320;
constexpr int kDeadFraction = 8;

struct LazyState {
    double sumrho;
    double dw2;
};

// Wt = W^T (zero padded to rp), float64 column norms, identity index, state reset.  Positions d .. ld - 1
// (ld: d rounded up to 4, the pitch of the matrices) get index -1 and zero weights: they are removed from
// the start.
__global__ void __launch_bounds__(256) k_lazy_init(const float* __restrict__ W, int r, int d, int ld, int rp,
                                                   float* __restrict__ Wt, double* __restrict__ dQ,
                                                   double* __restrict__ norm2, int* __restrict__ idx,
                                                   LazyState* __restrict__ state) {
    __shared__ float tile[32][33];
    const int l = blockIdx.y;
    const int c0 = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const float* Wl = W + (size_t)l * r * d;
    float* Wtl = Wt + (size_t)l * ld * rp;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i0 = 0; i0 < rp; i0 += 32) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int rr = ty + 8 * m;
            const int i = i0 + rr, c = c0 + tx;
            tile[rr][tx] = (i < r && c < d) ? Wl[(size_t)i * d + c] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int cc = ty + 8 * m;
            const int c = c0 + cc, i = i0 + tx;
            const float v = tile[tx][cc];
            if (c < ld && i < rp) Wtl[(size_t)c * rp + i] = v;
            acc[m] += (double)v * (double)v;
        }
        __syncthreads();
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        double s = acc[m];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const int c = c0 + ty + 8 * m;
        if (tx == 0 && c < ld) {
            dQ[(size_t)l * ld + c] = s;
            norm2[(size_t)l * ld + c] = s;
            idx[(size_t)l * ld + c] = c < d ? c : -1;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state[l].sumrho = 0.0; state[l].dw2 = 0.0;
    }
}

// Every CTA of a cluster sends its offers of all steps, also past a give-up.  Once all have been sent (behind the
// last cluster barrier) those from step `first` on, which the CTA has not waited for, land before it leaves, or run
// out once more: barriers of even and odd steps, armed up to step first + 1.
template <typename Bytes>
__device__ __forceinline__ void land_offers(uint64_t (&bar_step)[2], int first, int nsteps, const Bytes& step_bytes) {
    for (int m = first; m < nsteps; ++m) {
        const uint32_t bar = tc::smem_u32(&bar_step[m & 1]);
        if (!tc::mbar_wait_quiet(bar, (uint32_t)(m >> 1) & 1u)) return;
        if (m + 2 < nsteps) tc::mbar_expect_tx(bar, step_bytes(m + 2));
    }
}

// nsteps (at most cap) greedy steps of one layer, run by a thread-block cluster of CS CTAs (CS = 1, 2, 4 or 8,
// chosen so that a CTA's slice of positions fits its shared memory).  CTA `rank` owns the
// positions [rank * S, rank * S + S); each of its 256 threads owns four consecutive ones and
// keeps their float64 diagonal entries of H^-1 and Q in registers for the whole block.  The
// pending vectors u_s, z_s of the block live in shared memory, sliced the same way (pitch Sp), so the
// correction of a pivot column touches no global memory.
//
// A step is a chain of latencies, so its parts are as short as they can be made and nothing waits for a
// hand-over that it can do without: the fp32 quotients of a thread's four positions are formed without
// branches and ordered as integers (the exact float64 comparison only sees candidates within 1e-5 of each
// other), every warp offers its best, and after the barrier every warp makes the pick for itself and
// requests the pivot rows at once.  On a cluster (MULTI) the CTA's best is picked first and warp c sends
// it to CTA c, with the pending entries at its position, which the winner's column needs, by asynchronous
// stores that complete on a barrier of the receiving CTA.  No step writes to global memory:
// a cluster barrier, and every fence, would wait for it.  What the update kernels need -- u, z and the
// step order -- goes out at the end of the block, for a dense block as the packed operands themselves.
// (Clocks per step at 3072 positions: 5200 with the comparisons one after the other and the pending
// entries fetched after the pick; 3700 with a cluster barrier and u, z stored step by step; 2800 to
// 3300 now, on twice the CTAs and for 64 steps with as many clocks for the pending terms.)
//
// The scaled pivot columns of W (c_s) do not feed the selection; they are solved for at the end
// of the block by forward substitution with the triangle T[m][s] = u_s[p_m].
// Finally the per-position vectors are compacted (stable) across the cluster.
template <bool MULTI>
__global__ void __launch_bounds__(STEP_THREADS, 1)
k_lazy_steps(int n0, int S, int Sp, int cap, int t0, int nsteps, int compact, int d, int G, int r, int rp,
             const float* __restrict__ A, const float* __restrict__ Q, const float* __restrict__ Wt,
             const double* __restrict__ dA_in, const double* __restrict__ dQ_in,
             const int* __restrict__ idx_in, double* __restrict__ dA_out,
             double* __restrict__ dQ_out, int* __restrict__ idx_out, int* __restrict__ src,
             float* __restrict__ U, float* __restrict__ Z, float* __restrict__ C,
             __nv_bfloat16* __restrict__ P, int rows_pad, int rows_tot,
             LazyState* __restrict__ state, int* __restrict__ order, float* __restrict__ saliency,
             int* layer_status) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = MULTI ? (int)cluster.num_blocks() : 1;
    const int rank = MULTI ? (int)cluster.block_rank() : 0;
    const int l = blockIdx.x / CS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = STEP_THREADS / 32;

    extern __shared__ float4 dyn_smem4[];
    float* sU = reinterpret_cast<float*>(dyn_smem4);       // [cap][Sp]
    float* sZ = sU + (size_t)cap * Sp;                     // [cap][Sp]
    double (*sTd)[BMAX + 4] = reinterpret_cast<double (*)[BMAX + 4]>(dyn_smem4);   // T in float64, after the last step
    __shared__ Bid s_warp[2][NW];                          // the warps' offers, by step parity
    __shared__ Bid s_cta[2][CLUSTER_MAX];                  // the CTAs' offers, and the pending entries
    __shared__ __align__(16) float2 s_pend[2][CLUSTER_MAX][BMAX];   // (u_s[p], z_s[p]) at their positions
    __shared__ uint64_t bar_step[2];
    __shared__ float sT[BMAX][BMAX];                       // T[m][s] = u_s[p_m]
    __shared__ int s_pm[BMAX], s_org[BMAX];
    __shared__ double s_rsm[BMAX], s_rho[BMAX];
    __shared__ int s_count, s_wsum[NW];
    __shared__ int abort_flag;

    const float* Al = A + (size_t)l * d * d;
    const float* Ql = Q + (size_t)l * d * d;
    const float* Wl = Wt + (size_t)l * d * rp;

    const int kloc = 4 * tid;                  // first owned position within the slice
    const int k0 = rank * S + kloc;            // ... and globally
    const bool owner_thread = (kloc < S) && (k0 < n0);
    double da[4], dq[4];
    int org[4];
    bool alive[4];
    // what step m brings to a CTA: offers and the pending entries, in groups of 32
    auto step_bytes = [&](int m) { return (uint32_t)(CS * (sizeof(Bid) + (m > GS ? BMAX : GS) * sizeof(float2))); };
    if (MULTI) {
        if (tid == 0) {
            abort_flag = 0;
            tc::mbar_init(tc::smem_u32(&bar_step[0]), 1);
            tc::mbar_init(tc::smem_u32(&bar_step[1]), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            tc::mbar_expect_tx(tc::smem_u32(&bar_step[0]), step_bytes(0));
        }
        cluster.sync();
    }
    // where warp c sends to in CTA c
    uint32_t to_bid = 0, to_pend = 0, to_bar = 0;
    if (MULTI && warp < CS) {
        to_bid = tc::map_rank(&s_cta[0][rank], warp);
        to_pend = tc::map_rank(&s_pend[0][rank][lane], warp);
        to_bar = tc::map_rank(&bar_step[0], warp);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = k0 + e;
        // a position removed in an earlier block that has not been squeezed out yet carries
        // index -1: it stays dead
        const int o = (owner_thread && k < n0) ? idx_in[(size_t)l * d + k] : -1;
        alive[e] = o >= 0;
        da[e] = alive[e] ? dA_in[(size_t)l * d + k] : 1.0;
        dq[e] = alive[e] ? dQ_in[(size_t)l * d + k] : 0.0;
        org[e] = alive[e] ? o : 0x7fffffff;
    }
    int first_bad = ZIPLM_OK;                  // meaningful in lane 0 of the last warp
    int gave_up = nsteps;                      // the first step whose offers did not come in time
    // row indices of W that this CTA solves for
    const int w_per = ((rp + CS - 1) / CS + 7) / 8 * 8, w_first = rank * w_per, w_end = min(rp, w_first + w_per);

    for (int m = 0; m < nsteps; ++m) {
        const int par = m & 1;
        // ---- best of the four owned positions of rho = Q[k,k] / H^-1[k,k] (ties: lowest original index)
        unsigned key[4], kmine = kKeyNone;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            key[e] = cand_key(alive[e], da[e], dq[e]);
            kmine = min(kmine, key[e]);
        }
        unsigned near_mine = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) near_mine |= (alive[e] && key[e] - kmine <= kKeyNear) ? 1u << e : 0u;
        const unsigned kmin = __reduce_min_sync(0xffffffffu, kmine);
        Cand best;
        best.a = near_mine & 1 ? da[0] : near_mine & 2 ? da[1] : near_mine & 4 ? da[2] : da[3];
        best.q = near_mine & 1 ? dq[0] : near_mine & 2 ? dq[1] : near_mine & 4 ? dq[2] : dq[3];
        best.org = near_mine & 1 ? org[0] : near_mine & 2 ? org[1] : near_mine & 4 ? org[2] : org[3];
        best.pos = near_mine ? k0 + __ffs(near_mine) - 1 : -1;
        if (near_mine & (near_mine - 1)) {         // several within 1e-5: the exact comparison
            best.pos = -1;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (!(near_mine >> e & 1)) continue;
                Cand c;
                c.a = da[e]; c.q = dq[e]; c.org = org[e]; c.pos = k0 + e;
                merge_cand(best, c);
            }
        }
        // ---- the warp's offer, written by the lane that holds it
        const unsigned near_warp = __ballot_sync(0xffffffffu, best.pos >= 0 && kmine - kmin <= kKeyNear);
        int holder = near_warp ? __ffs(near_warp) - 1 : 0;
        if (near_warp & (near_warp - 1)) {
            Cand b = bcast_cand(best, holder);
            for (unsigned left = near_warp & (near_warp - 1); left; left &= left - 1)
                merge_cand(b, bcast_cand(best, __ffs(left) - 1));
            best = b;                              // (every lane has it)
        }
        if (lane == holder) {
            Bid b;
            b.a = best.a; b.q = best.q; b.org = best.org; b.pos = best.pos; b.key = kmin; b.pad = 0;
            s_warp[par][warp] = b;
        }
        __syncthreads();
        // ---- the pick: made by every warp for itself
        const Bid* bid;
        const float2* pend = nullptr;              // pending entries at the pivot
        if (MULTI) {
            // the CTA's own offer, sent to every CTA (warp c to CTA c) with its pending entries
            const Bid own = s_warp[par][best_bid(s_warp[par], NW, lane)];
            if (warp < CS) {
                const int pl = own.pos >= 0 ? own.pos - rank * S : 0;
                float2 uz[BMAX / GS];
#pragma unroll
                for (int g = 0; g < BMAX / GS; ++g) {
                    const int s = g * GS + lane;
                    uz[g] = s < m ? make_float2(sU[(size_t)s * Sp + pl], sZ[(size_t)s * Sp + pl]) : make_float2(0.f, 0.f);
                }
                const uint32_t bar = to_bar + 8u * par;
                if (lane == 0) {
                    const uint32_t to = to_bid + (uint32_t)(par * CLUSTER_MAX * sizeof(Bid));
                    tc::send2(to, own.a, own.q, bar);
                    tc::send2(to + 16u, ((long long)own.pos << 32) | (unsigned)own.org, (long long)own.key, bar);
                }
#pragma unroll
                for (int g = 0; g < BMAX / GS; ++g)
                    if (g == 0 || m > g * GS)
                        tc::send1(to_pend + (uint32_t)((par * CLUSTER_MAX * BMAX + g * GS) * sizeof(float2)),
                                  ((long long)__float_as_uint(uz[g].y) << 32) | __float_as_uint(uz[g].x), bar);
            }
            // (past a give-up the barrier may still be in an older phase)
            if (tid == 0 && m + 1 < nsteps && gave_up == nsteps)
                tc::mbar_expect_tx(tc::smem_u32(&bar_step[par ^ 1]), step_bytes(m + 1));
            if (!tc::mbar_wait(tc::smem_u32(&bar_step[par]), (uint32_t)(m >> 1) & 1u, &abort_flag)) {
                gave_up = min(gave_up, m);         // (the waits that follow give up at once)
                abort_flag = 1;
            }
            const int which = best_bid(s_cta[par], CS, lane);
            bid = &s_cta[par][which];
            pend = s_pend[par][which];
        } else {
            bid = &s_warp[par][best_bid(s_warp[par], NW, lane)];
        }
        const int p = min(max(bid->pos, 0), n0 - 1);
        // both triangles of H^-1 and Q are kept, so the pivot column is the contiguous row p
        float4 a4 = make_float4(0.f, 0.f, 0.f, 0.f), q4 = a4;
        if (owner_thread) {
            a4 = *reinterpret_cast<const float4*>(Al + (size_t)p * d + k0);
            q4 = *reinterpret_cast<const float4*>(Ql + (size_t)p * d + k0);
        }
        const double gq = bid->q;
        double h = bid->a;
        int bad = 0;
        if (!isfinite(gq) || !isfinite(h)) { bad = ZIPLM_ERR_NONFINITE; h = 1.0; }
        else if (!(h > 0.0)) { bad = ZIPLM_ERR_NOT_PD; h = 1.0; }
        const double rs = rsqrt(h), half = 0.5 * gq * rs * rs;
        const float *pu = sU + p, *pz = sZ + p;    // pending entries of one CTA: in its own slice
        if (warp == NW - 1) {                      // (the last warp: the others may own more positions)
#pragma unroll
            for (int s = lane; s < BMAX; s += 32) sT[m][s] = s < m ? (MULTI ? pend[s].x : pu[(size_t)s * Sp]) : 0.f;
            // this CTA's part of the pivot column of W, which the end of the block reads, on its way to L2
            for (int i = w_first + 32 * lane; i < w_end; i += 1024)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(Wl + (size_t)p * rp + i));
            if (lane == 0) {
                s_pm[m] = p;
                s_rsm[m] = rs;
                s_rho[m] = bad ? 0.0 : gq * rs * rs;
                s_org[m] = bid->org;
                if (bad && first_bad == ZIPLM_OK) first_bad = bad;
            }
        }
        // ---- true pivot columns of H^-1 and Q on the owned positions; float64 diagonal downdate
        if (owner_thread) {
            // pending terms at the pivot, summed while the gathered entries are still in flight
            float ca[4] = {0.f, 0.f, 0.f, 0.f}, cq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int s = 0; s < m; ++s) {
                const float4 u4 = *reinterpret_cast<const float4*>(sU + (size_t)s * Sp + kloc);
                const float4 z4 = *reinterpret_cast<const float4*>(sZ + (size_t)s * Sp + kloc);
                float up, zp;
                if (MULTI) {
                    const float2 uz = pend[s];
                    up = uz.x; zp = uz.y;
                } else {
                    up = pu[(size_t)s * Sp]; zp = pz[(size_t)s * Sp];
                }
                const float uu[4] = {u4.x, u4.y, u4.z, u4.w}, zz[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    ca[e] = fmaf(uu[e], up, ca[e]);
                    cq[e] = fmaf(zz[e], up, cq[e]);
                    cq[e] = fmaf(uu[e], zp, cq[e]);
                }
            }
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, q[4] = {q4.x, q4.y, q4.z, q4.w};
            float u32[4], z32[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                // removed positions and the pivot itself: zero, which leaves the diagonals as they are
                alive[e] = alive[e] && k0 + e != p;
                const float ae = alive[e] ? a[e] - ca[e] : 0.f, qe = alive[e] ? q[e] - cq[e] : 0.f;
                const double u = (double)ae * rs;
                const double z = (double)qe * rs - half * u;
                da[e] -= u * u;
                dq[e] -= 2.0 * z * u;
                u32[e] = alive[e] ? (float)u : 0.f;
                z32[e] = alive[e] ? (float)z : 0.f;
            }
            *reinterpret_cast<float4*>(sU + (size_t)m * Sp + kloc) = make_float4(u32[0], u32[1], u32[2], u32[3]);
            *reinterpret_cast<float4*>(sZ + (size_t)m * Sp + kloc) = make_float4(z32[0], z32[1], z32[2], z32[3]);
        }
        // no barrier here: the next step's barrier orders these writes before any read
    }
    if (gave_up < nsteps) set_layer_status(layer_status, l, ZIPLM_ERR_TIMEOUT);
    __syncthreads();

    // ---- what the update kernels read: u, z as they are for a compaction block, packed for a dense one
    const int n_own = max(0, min(S, n0 - rank * S));
    if (compact) {
        float* Ul = U + (size_t)l * GS * d + rank * S;
        float* Zl = Z + (size_t)l * GS * d + rank * S;
        for (int s = warp; s < nsteps; s += NW)
            for (int k = lane; k < n_own; k += 32) {
                Ul[(size_t)s * d + k] = sU[(size_t)s * Sp + k];
                Zl[(size_t)s * d + k] = sZ[(size_t)s * Sp + k];
            }
    } else {
        // two positions per warp, two steps per lane: 64-byte pieces (a position per thread with 16-byte stores
        // touches 32 lines an instruction and takes 1.7 times as long); the last CTA zeroes the rows up to the
        // next whole tile
        const size_t arr = (size_t)rows_tot * 2 * GS;
        const int end = rank == CS - 1 ? (n0 + kPackTile - 1) / kPackTile * kPackTile - rank * S : n_own;
        for (int g = 0; g * GS < nsteps; ++g) {
            __nv_bfloat16* Pl = P + ((size_t)l * kPackGroups + g) * kPackArrays * arr;
            const int sl = 2 * (lane & 15), sp = g * GS + sl;
#pragma unroll 2
            for (int k = 2 * warp + (lane >> 4); k < end; k += 2 * NW) {
                const bool i0 = k < n_own && sp < nsteps, i1 = k < n_own && sp + 1 < nsteps;
                __nv_bfloat162 u[3], z[3];
                split_bf16x3(i0 ? sU[(size_t)sp * Sp + k] : 0.f, i1 ? sU[(size_t)(sp + 1) * Sp + k] : 0.f, u);
                split_bf16x3(i0 ? sZ[(size_t)sp * Sp + k] : 0.f, i1 ? sZ[(size_t)(sp + 1) * Sp + k] : 0.f, z);
                __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(Pl + (size_t)(rank * S + k) * 2 * GS + sl);
                o[0] = u[0];       o[GS / 2] = u[1];
                o += arr / 2;
                o[0] = u[2];       o[GS / 2] = z[2];
                o += arr / 2;
                o[0] = z[0];       o[GS / 2] = z[1];
            }
        }
    }
    if (rank == 0) {
        if (tid < nsteps) {
            order[(size_t)l * G + t0 + tid] = s_org[tid];
            if (saliency) saliency[(size_t)l * G + t0 + tid] = (float)s_rho[tid];
        }
        if (warp == NW - 1 && lane == 0) {
            double sum = 0.0;
            for (int m = 0; m < nsteps; ++m) sum += s_rho[m];
            state[l].sumrho += sum;
            if (first_bad != ZIPLM_OK) set_layer_status(layer_status, l, first_bad);
        }
    }
    __syncthreads();                           // sU, sZ are done with

    // ---- c_m = (W[:,p_m] - sum_{s<m} c_s T[m][s]) / sqrt(h_m), forward substitution for every row index i
    //      of W (each CTA a slice of them), in 8 x 8 blocks on the float64 tensor-core instruction: the
    //      diagonal blocks of the triangle are inverted first, a lane for a column; then a warp takes
    //      eight row indices and 32 steps at a time: C_b = D_b^-1 W_b, W_q -= T_qb C_b for q > b, the second 32
    //      steps behind the first.  C_b is rounded to fp32, as it is stored and applied, before it is used.
    //      (One thread per row index ran 500 FMAs and as many loads of straight-line code from a cold
    //      instruction cache: 21000 to 36000 clocks a block of 32 steps, a fifth of it.)
    //      It reads this CTA's own shared memory only and runs last, when the per-position state is dead.
    auto solve_c = [&]() {
        double (*sD)[9] = reinterpret_cast<double (*)[9]>(sTd + BMAX);     // [BMAX][8]: D_b^-1, row m, column m % 8
        const int groups = (nsteps + GS - 1) / GS;
        for (int e = tid; e < groups * GS * BMAX; e += STEP_THREADS)
            sTd[e / BMAX][e % BMAX] = e / BMAX < nsteps ? (double)sT[e / BMAX][e % BMAX] : 0.0;
        __syncthreads();
        if (warp < groups) {
            const int b8 = warp * GS + (lane & 24), j = lane & 7;
            double x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                double acc = i == j ? 1.0 : 0.0;
#pragma unroll
                for (int k = 0; k < i; ++k) acc = fma(-sTd[b8 + i][b8 + k], x[k], acc);
                x[i] = i >= j && b8 + i < nsteps ? acc * s_rsm[b8 + i] : 0.0;
                sD[b8 + i][j] = x[i];
            }
        }
        __syncthreads();
        float* Cl = C + (size_t)l * GS * rp;
        const size_t arr = (size_t)rows_tot * 2 * GS;
        const int gr = lane >> 2, qd = lane & 3;         // accumulator: row gr, columns 2 qd, 2 qd + 1
        constexpr int NT = 3;                            // tiles of eight row indices side by side
        // a block as the second operand: element (k = 4 kk + qd, n = gr) of it
        auto operand = [&](double v0, double v1, int kk) {
            const int from = (4 * kk + qd) * 4 + (gr >> 1);
            const double x = __shfl_sync(0xffffffffu, v0, from), y = __shfl_sync(0xffffffffu, v1, from);
            return gr & 1 ? y : x;
        };
        for (int i0 = w_first + 8 * warp; i0 < w_end; i0 += 8 * NW * NT) {
            float done[NT][4][2] = {};                   // C of the first group
#pragma unroll 1
            for (int g = 0; g < groups; ++g) {
                const int m0 = g * GS;
                __nv_bfloat16* Pc = P + ((size_t)l * kPackGroups + g) * kPackArrays * arr + (size_t)rows_pad * 2 * GS;
                double acc[NT][4][2];
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        // (rows are zero from r to rp; what lies past the slice or the last step is not used)
                        const int i = min(i0 + 8 * NW * t + 2 * qd, rp - 2), m = m0 + 8 * b + gr;
                        const float2 w = *reinterpret_cast<const float2*>(Wl + (size_t)s_pm[min(m, nsteps - 1)] * rp + i);
                        acc[t][b][0] = m < nsteps ? (double)w.x : 0.0;
                        acc[t][b][1] = m < nsteps ? (double)w.y : 0.0;
                    }
                if (g)
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk) {
                            double tq[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) tq[q] = -sTd[m0 + 8 * q + gr][8 * b + 4 * kk + qd];
#pragma unroll
                            for (int t = 0; t < NT; ++t) {
                                const double x = operand((double)done[t][b][0], (double)done[t][b][1], kk);
#pragma unroll
                                for (int q = 0; q < 4; ++q) dmma884(acc[t][q], tq[q], x);
                            }
                        }
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const double d0 = sD[m0 + 8 * b + gr][qd], d1 = sD[m0 + 8 * b + gr][4 + qd];
                    double tq[3][2];
#pragma unroll
                    for (int q = b + 1; q < 4; ++q) {
                        tq[q - 1][0] = -sTd[m0 + 8 * q + gr][m0 + 8 * b + qd];
                        tq[q - 1][1] = -sTd[m0 + 8 * q + gr][m0 + 8 * b + 4 + qd];
                    }
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        double c[2] = {0.0, 0.0};
                        dmma884(c, d0, operand(acc[t][b][0], acc[t][b][1], 0));
                        dmma884(c, d1, operand(acc[t][b][0], acc[t][b][1], 1));
                        const float c0 = (float)c[0], c1 = (float)c[1];
                        done[t][b][0] = c0; done[t][b][1] = c1;
                        const int i = i0 + 8 * NW * t + 2 * qd, sl = 8 * b + gr;
                        if (i < w_end) {                     // (rp and the slices are even)
                            if (compact) {
                                if (sl < nsteps) *reinterpret_cast<float2*>(Cl + (size_t)sl * rp + i) = make_float2(c0, c1);
                            } else {
                                // rows of the packed operands behind the positions: [C1 | C2], [C3 | 0] (the rest
                                // was zeroed before the first block)
                                __nv_bfloat162 x[3];
                                split_bf16x3(c0, c1, x);
                                __nv_bfloat16* o = Pc + (size_t)i * 2 * GS + sl;
                                o[0] = __low2bfloat16(x[0]); o[GS] = __low2bfloat16(x[1]); o[arr] = __low2bfloat16(x[2]);
                                o += 2 * GS;
                                o[0] = __high2bfloat16(x[0]); o[GS] = __high2bfloat16(x[1]); o[arr] = __high2bfloat16(x[2]);
                            }
                        }
                        if (b == 3) continue;
                        const double b0 = operand((double)c0, (double)c1, 0), b1 = operand((double)c0, (double)c1, 1);
#pragma unroll
                        for (int q = b + 1; q < 4; ++q) {
                            dmma884(acc[t][q], tq[q - 1][0], b0);
                            dmma884(acc[t][q], tq[q - 1][1], b1);
                        }
                    }
                }
            }
        }
    };

    // ---- end of the block.  Either the removed positions are squeezed out (stable compaction of
    //      the per-position vectors across the cluster; src[new] = old), or every position stays
    //      where it is (src = identity) and the removed ones are marked with index -1: the update
    //      kernels then move nothing and a later block does the squeezing.
    if (!compact) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = k0 + e;
            if (owner_thread && k < n0) {
                dA_out[(size_t)l * d + k] = da[e];
                dQ_out[(size_t)l * d + k] = dq[e];
                idx_out[(size_t)l * d + k] = alive[e] ? org[e] : -1;
            }
        }
        solve_c();
        if (MULTI) cluster.sync();      // no CTA leaves while others may send to it
        if (MULTI && tid == 0) land_offers(bar_step, gave_up, nsteps, step_bytes);
        return;
    }
    const int f0 = alive[0] ? 1 : 0, f1 = alive[1] ? 1 : 0, f2 = alive[2] ? 1 : 0, f3 = alive[3] ? 1 : 0;
    const int mine = f0 + f1 + f2 + f3;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_wsum[warp] = incl;
    __syncthreads();
    if (tid == 0) {
        int t = 0;
        for (int w2 = 0; w2 < NW; ++w2) { const int v = s_wsum[w2]; s_wsum[w2] = t; t += v; }
        s_count = t;
    }
    if (MULTI) cluster.sync();
    else __syncthreads();
    int base = 0;
    if (MULTI)
        for (int c2 = 0; c2 < rank; ++c2) base += *cluster.map_shared_rank(&s_count, c2);
    int np = base + s_wsum[warp] + incl - mine;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (alive[e]) {
            src[(size_t)l * d + np] = k0 + e;
            dA_out[(size_t)l * d + np] = da[e];
            dQ_out[(size_t)l * d + np] = dq[e];
            idx_out[(size_t)l * d + np] = org[e];
            ++np;
        }
    }
    // After a give-up the CTAs may have removed more than one position a step between them: what is left without
    // an owner becomes column 0 at position 0, so that the kernels behind this one stay in bounds.  (Otherwise
    // this lies past the live positions.)
    if (MULTI && rank == CS - 1)
        for (int k = base + s_count + tid; k < n0; k += STEP_THREADS) {
            const size_t o = (size_t)l * d + k;
            src[o] = 0; idx_out[o] = 0; dA_out[o] = 1.0; dQ_out[o] = 0.0;
        }
    if (MULTI) cluster.sync();      // no CTA may retire while another can still read its shared memory
    if (MULTI && tid == 0) land_offers(bar_step, gave_up, nsteps, step_bytes);
    solve_c();
}

// 4-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros without reading.
__device__ __forceinline__ void cp_async4(float* smem_dst, const float* gmem_src, unsigned src_bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sa), "l"(gmem_src), "r"(src_bytes)
                 : "memory");
}

__device__ __forceinline__ void cp_async16_zfill(float4* smem_dst, const float* gmem_src, unsigned src_bytes) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gmem_src), "r"(src_bytes)
                 : "memory");
}

// Rank-m update of the off-diagonal entries of H^-1 and Q with compaction (out of place):
//   A'[i,j] = A[si,sj] - sum_s U[s,si] U[s,sj],
//   Q'[i,j] = Q[si,sj] - sum_s (Z[s,si] U[s,sj] + U[s,si] Z[s,sj]),    si = src[i] > sj = src[j].
// 64 x 64 tiles of the new index space, 128 threads, 8 rows x 4 columns of both matrices per
// thread: per pending step six 128-bit shared-memory loads feed 96 FMAs.  Every entry is stored
// twice, at [i][j] and [j][i]: the steps kernel reads a pivot column as a contiguous row.
__global__ void __launch_bounds__(128, 5) k_lazy_update_aq(int n_new, int m, int d,
                                                        const float* __restrict__ A,
                                                        const float* __restrict__ Q,
                                                        float* __restrict__ A2, float* __restrict__ Q2,
                                                        const int* __restrict__ src,
                                                        const float* __restrict__ U,
                                                        const float* __restrict__ Z) {
    __shared__ __align__(16) float stage[4][GS][64];   // pending slabs of the tile's rows and columns
    float (*sUr)[64] = stage[0];
    float (*sZr)[64] = stage[1];
    float (*sUc)[64] = stage[2];
    float (*sZc)[64] = stage[3];
    __shared__ int srow[64], scol[64];
    const int l = blockIdx.y;
    // linear index -> (ti, tj) of the lower triangle: ti = floor((sqrt(8 x + 1) - 1) / 2), fixed up
    int ti = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while (ti * (ti + 1) / 2 > (int)blockIdx.x) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.x) ++ti;
    const int tj = (int)blockIdx.x - ti * (ti + 1) / 2;
    const int i0 = ti * 64, j0 = tj * 64;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;     // rows 4ty + 32h + e, cols 4tx + e
    // a tile strictly below the diagonal and inside the live range needs no per-entry checks
    const bool interior = tj < ti && i0 + 64 <= n_new;
    const int* sl = src + (size_t)l * d;
    if (tid < 64) srow[tid] = (i0 + tid < n_new) ? sl[i0 + tid] : -1;
    else scol[tid - 64] = (j0 + tid - 64 < n_new) ? sl[j0 + tid - 64] : -1;
    __syncthreads();
    // The pending slabs of the tile's rows and columns go straight to shared memory with
    // asynchronous 4-byte copies (zero-filled past the last live row), so that all of them and the
    // gathered old entries below are in flight together.
    const float* Ul = U + (size_t)l * GS * d;
    const float* Zl = Z + (size_t)l * GS * d;
    {
        const int c = tid & 63;
        const int idx = (tid < 64) ? srow[c] : scol[c];
        float (*dU)[64] = (tid < 64) ? sUr : sUc;
        float (*dZ)[64] = (tid < 64) ? sZr : sZc;
        const unsigned nbytes = idx >= 0 ? 4u : 0u;
        const size_t off = idx >= 0 ? (size_t)idx : 0;
        for (int s = 0; s < m; ++s) {
            cp_async4(&dU[s][c], Ul + (size_t)s * d + off, nbytes);
            cp_async4(&dZ[s][c], Zl + (size_t)s * d + off, nbytes);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const float* Al = A + (size_t)l * d * d;
    const float* Ql = Q + (size_t)l * d * d;
    int cs[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) cs[y] = scol[4 * tx + y];
    float a[8][4], q[8][4];
    if (interior) {
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const unsigned roff = (unsigned)(srow[4 * ty + 32 * (x >> 2) + (x & 3)] * d);   // d * d < 2^31
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                a[x][y] = __ldcs(Al + (roff + (unsigned)cs[y]));
                q[x][y] = __ldcs(Ql + (roff + (unsigned)cs[y]));
            }
        }
    } else {
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const int il = 4 * ty + 32 * (x >> 2) + (x & 3), i = i0 + il;
            const int sr = srow[il];
            const size_t roff = (size_t)(sr >= 0 ? sr : 0) * d;
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int j = j0 + 4 * tx + y;
                if (sr >= 0 && j < i) {
                    a[x][y] = __ldcs(Al + roff + cs[y]);
                    q[x][y] = __ldcs(Ql + roff + cs[y]);
                } else {
                    a[x][y] = 0.f; q[x][y] = 0.f;
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int s = 0; s < m; ++s) {
        float ur[8], zr[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 v0 = *reinterpret_cast<const float4*>(&sUr[s][4 * ty + 32 * h]);
            const float4 v1 = *reinterpret_cast<const float4*>(&sZr[s][4 * ty + 32 * h]);
            ur[4 * h] = v0.x; ur[4 * h + 1] = v0.y; ur[4 * h + 2] = v0.z; ur[4 * h + 3] = v0.w;
            zr[4 * h] = v1.x; zr[4 * h + 1] = v1.y; zr[4 * h + 2] = v1.z; zr[4 * h + 3] = v1.w;
        }
        const float4 u4 = *reinterpret_cast<const float4*>(&sUc[s][4 * tx]);
        const float4 z4 = *reinterpret_cast<const float4*>(&sZc[s][4 * tx]);
        const float uc[4] = {u4.x, u4.y, u4.z, u4.w}, zc[4] = {z4.x, z4.y, z4.z, z4.w};
#pragma unroll
        for (int x = 0; x < 8; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                a[x][y] = fmaf(-ur[x], uc[y], a[x][y]);
                q[x][y] = fmaf(-zr[x], uc[y], q[x][y]);
                q[x][y] = fmaf(-ur[x], zc[y], q[x][y]);
            }
    }
    float* Ao = A2 + (size_t)l * d * d;
    float* Qo = Q2 + (size_t)l * d * d;
    const int j = j0 + 4 * tx;
    if (interior) {
        float* ao = Ao + (size_t)(i0 + 4 * ty) * d + j;
        float* qo = Qo + (size_t)(i0 + 4 * ty) * d + j;
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const unsigned o = (unsigned)((32 * (x >> 2) + (x & 3)) * d);
            *reinterpret_cast<float4*>(ao + o) = make_float4(a[x][0], a[x][1], a[x][2], a[x][3]);
            *reinterpret_cast<float4*>(qo + o) = make_float4(q[x][0], q[x][1], q[x][2], q[x][3]);
        }
        // mirror ([j][i]): the tile goes through shared memory (the staging arrays are free now),
        // so that the transposed rows leave as contiguous 256-byte pieces
        float* tbuf = &stage[0][0][0];                 // 64 x 65 floats of the 4 x 32 x 64
        const int lane = tid & 31, wrp = tid >> 5;
#pragma unroll
        for (int mat = 0; mat < 2; ++mat) {
            __syncthreads();                           // the arrays' previous readers are done
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    tbuf[(4 * tx + y) * 65 + 4 * ty + 32 * (x >> 2) + (x & 3)] = mat ? q[x][y] : a[x][y];
            __syncthreads();
            float* mo = (mat ? Qo : Ao) + (size_t)j0 * d + i0 + 2 * lane;
#pragma unroll 4
            for (int jl = wrp; jl < 64; jl += 4)
                *reinterpret_cast<float2*>(mo + (size_t)jl * d) =
                    make_float2(tbuf[jl * 65 + 2 * lane], tbuf[jl * 65 + 2 * lane + 1]);
        }
        return;
    }
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const int i = i0 + 4 * ty + 32 * (x >> 2) + (x & 3);
        if (i >= n_new || j >= i) continue;
        for (int e = 0; e < 4; ++e)          // tile on the diagonal or at the ragged edge: entry by entry
            if (j + e < i) {
                Ao[(size_t)i * d + j + e] = a[x][e]; Ao[(size_t)(j + e) * d + i] = a[x][e];
                Qo[(size_t)i * d + j + e] = q[x][e]; Qo[(size_t)(j + e) * d + i] = q[x][e];
            }
    }
}

// Rank-m update of W^T with row compaction (out of place): Wt'[i,:] = Wt[si,:] - sum_s U[s,si] C[s,:].
// A CTA owns 64 rows x 256 columns; the C panel and the rows' U entries are staged in shared
// memory once per CTA, each thread carries 16 consecutive rows of one float4 column (per pending
// step: one 128-bit load of C and four broadcast 128-bit loads of U for 64 FMAs).
__global__ void __launch_bounds__(256, 3) k_lazy_update_w(int n_new, int m, int d, int rp,
                                                       const float* __restrict__ Wt,
                                                       float* __restrict__ Wt2,
                                                       const int* __restrict__ src,
                                                       const float* __restrict__ U,
                                                       const float* __restrict__ C) {
    __shared__ float4 sC[GS][64];       // C[s][col0 .. col0+255]
    __shared__ __align__(16) float sUr[GS][64];       // U[s][src[row]]
    __shared__ int srow[64];
    const int l = blockIdx.z;
    const int i0 = blockIdx.x * 64, c0 = blockIdx.y * 256;
    const int tid = threadIdx.x, tx = tid & 63, ty = tid >> 6;      // ty: rows 16 ty .. 16 ty + 15
    if (tid < 64) srow[tid] = (i0 + tid < n_new) ? src[(size_t)l * d + i0 + tid] : -1;
    __syncthreads();
    const float* Ul = U + (size_t)l * GS * d;
    const float* Cl = C + (size_t)l * GS * rp;
    // asynchronous copies (zero-filled where there is nothing to read), in flight together with
    // the gathered rows below
    for (int e = tid; e < m * 64; e += 256) {
        const int s = e >> 6, c = e & 63;
        const int sr = srow[c];
        cp_async4(&sUr[s][c], Ul + (size_t)s * d + (sr >= 0 ? sr : 0), sr >= 0 ? 4u : 0u);
        const int col = c0 + 4 * c;
        cp_async16_zfill(&sC[s][c], Cl + (size_t)s * rp + (col < rp ? col : 0), col < rp ? 16u : 0u);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int col = c0 + 4 * tx;
    const bool col_ok = col < rp;
    float4 w[16];                                  // rows 16 ty + x of this CTA's 64
#pragma unroll
    for (int x = 0; x < 16; ++x) {
        const int sr = srow[16 * ty + x];
        w[x] = (sr >= 0 && col_ok)
                   ? __ldcs(reinterpret_cast<const float4*>(Wt + (size_t)l * d * rp + (size_t)sr * rp + col))
                   : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int s = 0; s < m; ++s) {
        const float4 c = sC[s][tx];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 u4 = *reinterpret_cast<const float4*>(&sUr[s][16 * ty + 4 * k]);   // broadcast
            const float nu[4] = {-u4.x, -u4.y, -u4.z, -u4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float4& t = w[4 * k + e];
                t.x = fmaf(nu[e], c.x, t.x); t.y = fmaf(nu[e], c.y, t.y);
                t.z = fmaf(nu[e], c.z, t.z); t.w = fmaf(nu[e], c.w, t.w);
            }
        }
    }
    if (col_ok) {
#pragma unroll
        for (int x = 0; x < 16; ++x) {
            const int i = i0 + 16 * ty + x;
            if (i < n_new)
                *reinterpret_cast<float4*>(Wt2 + (size_t)l * d * rp + (size_t)i * rp + col) = w[x];
        }
    }
}

__global__ void __launch_bounds__(256) k_lazy_pos_of(int n, int d, const int* __restrict__ idx,
                                                     int* __restrict__ pos_of) {
    const int l = blockIdx.x;
    for (int c = threadIdx.x; c < d; c += blockDim.x) pos_of[(size_t)l * d + c] = -1;
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const int o = idx[(size_t)l * d + k];
        if (o >= 0) pos_of[(size_t)l * d + o] = k;      // -1: removed, not squeezed out yet
    }
}

// W_snap = current weights in original column order, removed columns exactly zero; accumulates
// ||W - W_snap||_F^2 over the kept columns for the loss identity (the removed ones' share is their norms).
// 64 columns x 128 rows per CTA through shared memory, VEC columns per lane.  Bound by memory: W_snap is
// written whole, W and W^T are read where a column is kept; all of a thread's 16-byte reads of W^T, then its
// sixteen reads of W, are in flight together (32 x 32 tiles with four 4-byte reads in flight and all of W
// read moved 2.8 TB/s: twelve levels of 12 x 768 x 3072 took 1.3 ms).
constexpr int SNAP_C = 64, SNAP_R = 128;
template <int VEC>
__global__ void __launch_bounds__(256) k_lazy_snapshot(int r, int d, int ld, int rp,
                                                       const float* __restrict__ W,
                                                       const float* __restrict__ Wt,
                                                       const int* __restrict__ pos_of,
                                                       float* __restrict__ W_snap, int n_levels,
                                                       int slot, LazyState* __restrict__ state) {
    __shared__ float tile[SNAP_C][SNAP_R + 1];
    __shared__ int s_pos[SNAP_C];
    __shared__ double red[8];
    const int l = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c0 = blockIdx.x * SNAP_C, i0 = blockIdx.y * SNAP_R;
    const float* Wtl = Wt + (size_t)l * ld * rp;
    if (tid < SNAP_C) s_pos[tid] = c0 + tid < d ? pos_of[(size_t)l * ld + c0 + tid] : -1;
    __syncthreads();
    float4 v[SNAP_C / 8];
#pragma unroll
    for (int k = 0; k < SNAP_C / 8; ++k) {
        const int pos = s_pos[warp + 8 * k], i = i0 + 4 * lane;       // (rp is a multiple of four)
        v[k] = pos >= 0 && i < rp ? __ldcs(reinterpret_cast<const float4*>(Wtl + (size_t)pos * rp + i))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < SNAP_C / 8; ++k) {
        float* t = &tile[warp + 8 * k][4 * lane];
        t[0] = v[k].x; t[1] = v[k].y; t[2] = v[k].z; t[3] = v[k].w;
    }
    __syncthreads();
    const float* Wl = W + (size_t)l * r * d;
    float* out = W_snap + ((size_t)l * n_levels + slot) * (size_t)r * d;
    double acc = 0.0;
    constexpr int H = SNAP_C / (32 * VEC);         // column groups of a row
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int cc = h * 32 * VEC + lane * VEC, c = c0 + cc;
        bool kept[VEC], any = false;
#pragma unroll
        for (int e = 0; e < VEC; ++e) { kept[e] = s_pos[cc + e] >= 0; any |= kept[e]; }
        float w[SNAP_R / 8][VEC];
#pragma unroll
        for (int k = 0; k < SNAP_R / 8; ++k) {
            const int i = i0 + warp + 8 * k;
            const float* from = Wl + (size_t)i * d + c;
            const bool in = any && i < r;
            if (VEC == 2) {
                const float2 x = in ? __ldcs(reinterpret_cast<const float2*>(from)) : make_float2(0.f, 0.f);
                w[k][0] = x.x; w[k][VEC - 1] = x.y;
            } else {
                w[k][0] = in ? __ldcs(from) : 0.f;
            }
        }
#pragma unroll
        for (int k = 0; k < SNAP_R / 8; ++k) {
            const int i = i0 + warp + 8 * k;
            if (i >= r || c >= d) continue;
            float x[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                x[e] = tile[cc + e][i - i0];
                const float df = kept[e] ? w[k][e] - x[e] : 0.f;
                acc += (double)df * (double)df;
            }
            float* o = out + (size_t)i * d + c;
            if (VEC == 2) __stcs(reinterpret_cast<float2*>(o), make_float2(x[0], x[VEC - 1]));
            else __stcs(o, x[0]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += red[k];
        if (t != 0.0) atomicAdd(&state[l].dw2, t);
    }
}

// One CTA per layer.
__global__ void __launch_bounds__(256) k_lazy_loss(int d, int ld, int n_levels, int slot,
                                                   const double* __restrict__ lam,
                                                   const int* __restrict__ pos_of,
                                                   const double* __restrict__ norm2,
                                                   LazyState* __restrict__ state, float* __restrict__ loss) {
    __shared__ double red[8];
    const int l = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double acc = 0.0;
    for (int c = threadIdx.x; c < d; c += 256)
        if (pos_of[(size_t)l * ld + c] < 0) acc += norm2[(size_t)l * ld + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double dw2 = state[l].dw2;
    for (int k = 0; k < 8; ++k) dw2 += red[k];
    const double v = 0.5 * state[l].sumrho - 0.5 * lam[l] * dw2;
    loss[(size_t)l * n_levels + slot] = (float)(v > 0.0 ? v : 0.0);
    state[l].dw2 = 0.0;
}

// base_loss = ||W X||_F^2 = 1/2 tr(W H W^T) = 1/2 <W^T W, H>: one elementwise pass over the Gram
// matrix (pitch ld, full symmetric right after the product kernel) and the undamped Hessian (pitch d).
__global__ void __launch_bounds__(256) k_lazy_base_loss(int d, int ld, const float* __restrict__ Q,
                                                        const float* __restrict__ H,
                                                        double* __restrict__ acc64) {
    __shared__ double red[8];
    const int l = blockIdx.y;
    const float* Ql = Q + (size_t)l * ld * ld;
    const float* Hl = H + (size_t)l * d * d;
    double acc = 0.0;
    if (d == ld) {
        const size_t count = (size_t)d * d / 4;
        const float4* q4 = reinterpret_cast<const float4*>(Ql);
        const float4* h4 = reinterpret_cast<const float4*>(Hl);
        for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < count; e += (size_t)gridDim.x * 256) {
            const float4 a = __ldg(q4 + e), b = __ldg(h4 + e);
            acc += (double)a.x * b.x + (double)a.y * b.y + (double)a.z * b.z + (double)a.w * b.w;
        }
    } else {
        const int lane = threadIdx.x & 31;
        for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < d; i += gridDim.x * 8)
            for (int j = lane; j < d; j += 32)
                acc += (double)Ql[(size_t)i * ld + j] * Hl[(size_t)i * d + j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        atomicAdd(acc64 + l, t);
    }
}

__global__ void k_lazy_base_finish(int L, const double* __restrict__ acc64,
                                   float* __restrict__ base_loss) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l < L) base_loss[l] = (float)(0.5 * acc64[l]);
}

struct LazyWs {
    float* A[2]; float* Q[2]; float* Wt[2];
    double* dA[2]; double* dQ[2]; double* norm2; int* idx[2];
    int* src; int* pos_of; float* U; float* Z; float* C;
    float* P; int* sched;              // packed operands and work counter of the tensor-core update
    LazyState* state; double* lam; double* base_acc;
    void* aux; size_t aux_bytes;       // shared by the inverse, the Gram-matrix product and the endgame
    int rp, ld; size_t total;
};

LazyWs carve_lazy(void* ws, int L, int r, int d, int n_levels) {
    LazyWs w;
    w.rp = round_up_int(r, 4);
    w.ld = round_up_int(d, 4);
    const int ld = w.ld;
    Carver c(ws);
    for (int b = 0; b < 2; ++b) w.A[b] = c.take<float>((size_t)L * ld * ld);
    for (int b = 0; b < 2; ++b) w.Q[b] = c.take<float>((size_t)L * ld * ld);
    for (int b = 0; b < 2; ++b) w.Wt[b] = c.take<float>((size_t)L * ld * w.rp);
    for (int b = 0; b < 2; ++b) w.dA[b] = c.take<double>((size_t)L * ld);
    for (int b = 0; b < 2; ++b) w.dQ[b] = c.take<double>((size_t)L * ld);
    w.norm2 = c.take<double>((size_t)L * ld);
    for (int b = 0; b < 2; ++b) w.idx[b] = c.take<int>((size_t)L * ld);
    w.src = c.take<int>((size_t)L * ld);
    w.pos_of = c.take<int>((size_t)L * ld);
    w.U = c.take<float>((size_t)L * GS * ld);
    w.Z = c.take<float>((size_t)L * GS * ld);
    w.C = c.take<float>((size_t)L * GS * w.rp);
    w.P = c.take<float>(lazy_tc_pack_floats(L, ld, w.rp));
    w.sched = c.take<int>(2);
    w.state = c.take<LazyState>((size_t)L);
    w.lam = c.take<double>((size_t)L);
    w.base_acc = c.take<double>((size_t)L);
    const size_t inv = inverse_workspace_bytes(L, d);
    const size_t gram = hessian_tc_workspace_bytes(L, ld, w.rp, ZIPLM_F32, false);
    const size_t tail = endgame_workspace_bytes(L, r, kEndgame, n_levels);
    w.aux_bytes = inv > gram ? inv : gram;
    if (tail > w.aux_bytes) w.aux_bytes = tail;
    w.aux = c.take<char>(w.aux_bytes);
    w.total = c.off;
    return w;
}

}  // namespace

// Pitch of the pending vectors in the steps kernel: four more than a multiple of 32, so that the entries at
// one position (one per pending step) lie in eight different banks instead of one.
static int steps_pitch(int S) { return round_up_int(S, 32) + 4; }
// Steps that may be pending on slices of S positions, whole groups of 16 (the K of an MMA of the update).
static int steps_cap(int S) {
    const int fit = STEPS_SMEM / (2 * steps_pitch(S) * (int)sizeof(float));
    return fit >= BMAX ? BMAX : fit / 16 * 16;
}
static int steps_smem(int S, int cap) {
    const int b = 2 * cap * steps_pitch(S) * (int)sizeof(float), t = BMAX * (BMAX + 4 + 9) * (int)sizeof(double);
    return b > t ? b : t;
}

bool lazy_path_supported(int d) { return d >= 1 && d <= CLUSTER_MAX * SLICE_MAX; }

size_t lazy_workspace_bytes(int L, int r, int d, int n_levels) {
    if (d <= kEndgame) return endgame_workspace_bytes(L, r, d, n_levels);
    return carve_lazy(nullptr, L, r, d, n_levels).total;
}

ziplm_status run_prune_lazy(const float* W, const float* H, int L, int r, int d, float damp_frac,
                            const int* levels, int n_levels, float* W_snap, float* loss,
                            float* base_loss, int* order, float* saliency, int* layer_status,
                            void* ws, size_t ws_bytes, cudaStream_t st) {
    if (!lazy_path_supported(d)) return ZIPLM_ERR_UNSUPPORTED;
    if (ws_bytes < lazy_workspace_bytes(L, r, d, n_levels)) return ZIPLM_ERR_WORKSPACE;
    if (d <= kEndgame)
        return run_endgame_whole(W, H, L, r, d, damp_frac, levels, n_levels, W_snap, loss, base_loss, order,
                                 saliency, layer_status, ws, ws_bytes, st);
    LazyWs w = carve_lazy(ws, L, r, d, n_levels);
    // The matrices have the pitch ld = d rounded up to 4, so that every row starts on 16 bytes (128-bit
    // loads, TMA); the up to three positions behind d are treated as removed ones.
    const int G = d, rp = w.rp, ld = w.ld;
    ziplm_status s;
    {
        PhaseScope ps(PH_INVERSE, st);
        s = run_damped_inverse(H, L, d, damp_frac, nullptr, w.A[0], ld, ld, w.dA[0], w.lam, layer_status,
                               w.aux, w.aux_bytes, st);
    }
    if (s != ZIPLM_OK) return s;
    auto init = [&]() -> ziplm_status {
        PhaseScope ps(PH_INIT, st);
        ZIPLM_CHECK_CUDA(cudaMemsetAsync(order, 0xFF, sizeof(int) * (size_t)L * G, st));
        if (saliency)
            ZIPLM_CHECK_CUDA(cudaMemsetAsync(saliency, 0, sizeof(float) * (size_t)L * G, st));
        k_lazy_init<<<dim3((ld + 31) / 32, L), 256, 0, st>>>(W, r, d, ld, rp, w.Wt[0], w.dQ[0], w.norm2, w.idx[0],
                                                           w.state);
        ZIPLM_CHECK_LAUNCH();
        // Q = W^T W: the symmetric product kernel of the Hessian with X = W^T (K = d_row)
        ziplm_status g = run_hessian_tc(w.Q[0], w.Wt[0], ZIPLM_F32, false, L, ld, rp, rp, 1.0f, 0.0f, w.aux,
                                        w.aux_bytes, st);
        if (g != ZIPLM_OK) return g;
        if (base_loss) {
            ZIPLM_CHECK_CUDA(cudaMemsetAsync(w.base_acc, 0, sizeof(double) * L, st));
            k_lazy_base_loss<<<dim3(kSMs, L), 256, 0, st>>>(d, ld, w.Q[0], H, w.base_acc);
            ZIPLM_CHECK_LAUNCH();
            k_lazy_base_finish<<<(L + 63) / 64, 64, 0, st>>>(L, w.base_acc, base_loss);
            ZIPLM_CHECK_LAUNCH();
        }
        return ZIPLM_OK;
    };
    s = init();
    if (s != ZIPLM_OK) return s;

    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_lazy_steps<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          STEPS_SMEM));
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_lazy_steps<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          STEPS_SMEM));
    int cur = 0;
    auto snapshot = [&](int n, int slot) -> ziplm_status {
        PhaseScope ps(PH_SNAPSHOT, st);
        k_lazy_pos_of<<<L, 256, 0, st>>>(n, ld, w.idx[cur], w.pos_of);
        ZIPLM_CHECK_LAUNCH();
        const bool pairs = d % 2 == 0 && (reinterpret_cast<uintptr_t>(W) | reinterpret_cast<uintptr_t>(W_snap)) % 8 == 0;
        auto kernel = pairs ? k_lazy_snapshot<2> : k_lazy_snapshot<1>;
        kernel<<<dim3((d + SNAP_C - 1) / SNAP_C, (r + SNAP_R - 1) / SNAP_R, L), 256, 0, st>>>(
            r, d, ld, rp, W, w.Wt[cur], w.pos_of, W_snap, n_levels, slot, w.state);
        ZIPLM_CHECK_LAUNCH();
        k_lazy_loss<<<L, 256, 0, st>>>(d, ld, n_levels, slot, w.lam, w.pos_of, w.norm2, w.state, loss);
        ZIPLM_CHECK_LAUNCH();
        return ZIPLM_OK;
    };

    int slot = 0, t = 0;
    int n = G;
    int prio_least = 0, prio_greatest = 0;
    ZIPLM_CHECK_CUDA(cudaDeviceGetStreamPriorityRange(&prio_least, &prio_greatest));
    const int steps_priority = prio_greatest;
    if (slot < n_levels && levels[slot] == n) {
        s = snapshot(ld, slot++);
        if (s != ZIPLM_OK) return s;
    }
    const int n_min = n_levels > 0 ? levels[n_levels - 1] : G;
    // n = live structures, npos = positions of the arrays (live ones and those removed since the
    // last block that squeezed the removed positions out)
    int npos = ld;
    const bool every_block = option_value(ZIPLM_OPT_COMPACT_EVERY_BLOCK) == 1;
    const unsigned spin = (unsigned)option_value(ZIPLM_OPT_SPIN_LIMIT);
    CUtensorMap map_p, map_a[2], map_q[2], map_w[2];
    if (!lazy_tc_make_map(&map_p, w.P, L, ld, rp)) return ZIPLM_ERR_CUDA;
    for (int b = 0; b < 2; ++b)
        if (!lazy_tc_make_matrix_map(&map_a[b], w.A[b], L, ld, ld) ||
            !lazy_tc_make_matrix_map(&map_q[b], w.Q[b], L, ld, ld) ||
            !lazy_tc_make_matrix_map(&map_w[b], w.Wt[b], L, ld, rp))
            return ZIPLM_ERR_CUDA;
    ZIPLM_CHECK_CUDA(cudaMemsetAsync(w.sched, 0, sizeof(int) * 2, st));
    ZIPLM_CHECK_CUDA(cudaMemsetAsync(w.P, 0, sizeof(float) * lazy_tc_pack_floats(L, ld, rp), st));
    // The last kEndgame structures go to the float64 endgame unless only a few of them are to be removed
    // (its set-up costs as much as two blocks).
    const bool endgame = n_min <= kEndgame - 2 * GS;
    while (n > n_min) {
        int stop = (slot < n_levels) ? levels[slot] : n_min;         // next block boundary
        if (endgame && stop < kEndgame) stop = kEndgame;             // ... and where the endgame begins
        const int nxt = cur ^ 1;
        // Up to four CTAs a layer as long as a CTA has more than 256 positions: the pending terms of a step are
        // bound by shared-memory bandwidth, 24 clocks per pending step and 384 positions, which outweighs
        // the exchange.  Eight where a slice of BMAX pending steps would not fit shared memory (from 1537
        // positions on), whatever the number of layers: four with as many steps as then fit take longer in
        // all, 28.7 ms where eight take 26.3 (12 x 3072), 48.7 and 43.8 (24 x 3072), 102 and 97 (24 x 4096), or as
        // long (24 x 1814 and 24 x 2048, to 1 %), although 15 clusters of eight fit the part at a time: with all 24
        // layers in one group 53.3 and 48.9 (3072), 18.15 and 18.14 (1814), 19.97 and 20.32 (2048).  The steps
        // of 4 x 4096 by themselves: 9.5 ms on four CTAs up to 3072, 9.2 on eight, 8.8 with never more than 32 pending.
        int cs = 1;
        while (cs < CLUSTER_MAX && (npos + cs - 1) / cs > (cs < 4 ? 256 : SLICE_WIDE)) cs *= 2;
        const int S = round_up_int((npos + cs - 1) / cs, 4), cap = steps_cap(S);
        // Squeezing removed positions out makes the update kernels gather through a map; leaving
        // them in place keeps their reads and writes dense at the price of dead rows and columns.
        // They are squeezed out, by a block of at most 32 steps, once they make up kDeadMax positions or an
        // eighth of all.
        int nsteps = (n - stop < GS) ? (n - stop) : GS;
        const int dead_after = npos - (n - nsteps);
        const bool last = endgame && n - nsteps == kEndgame;
        const int compact = (every_block || last || dead_after >= kDeadMax ||
                             dead_after * kDeadFraction >= npos || npos <= 1) ? 1 : 0;
        if (!compact) {
            nsteps = (n - stop < cap) ? (n - stop) : cap;
            // (the block that reaches the endgame squeezes)
            if (endgame && n - nsteps == kEndgame) nsteps -= GS;
        }
        {
            PhaseScope ps(PH_LAZY_STEPS, st);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(L * cs);
            cfg.blockDim = dim3(STEP_THREADS);
            cfg.dynamicSmemBytes = (size_t)steps_smem(S, cap);
            cfg.stream = st;
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = cs;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            // The steps kernel is the latency chain of a layer group and needs whole SMs for its
            // clusters: at the highest launch priority its CTAs go ahead of the queued CTAs of the
            // other groups' wide update kernels as SMs drain.
            attr[1].id = cudaLaunchAttributePriority;
            attr[1].val.priority = steps_priority;
            cfg.attrs = attr;
            cfg.numAttrs = 2;
            ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(
                &cfg, cs > 1 ? k_lazy_steps<true> : k_lazy_steps<false>, npos, S, steps_pitch(S), cap, t, nsteps, compact, ld, G, r, rp, (const float*)w.A[cur],
                (const float*)w.Q[cur], (const float*)w.Wt[cur], (const double*)w.dA[cur],
                (const double*)w.dQ[cur], (const int*)w.idx[cur], w.dA[nxt], w.dQ[nxt], w.idx[nxt],
                w.src, w.U, w.Z, w.C, reinterpret_cast<__nv_bfloat16*>(w.P), lazy_tc_rows_pad(ld),
                lazy_tc_rows_tot(ld, rp), w.state, order, saliency, layer_status));
            ZIPLM_CHECK_LAUNCH();
        }
        const int n_new = compact ? n - nsteps : npos;      // positions after this block
        // The update of W goes first: measured, the step is 2 ms shorter than with the wide update
        // of H^-1 and Q in front (the next steps kernel then follows the kernel with the longer,
        // finer-grained tail).
        if (n_new > 0 && compact) {     // a dense block updates W^T in the tensor-core kernel
            PhaseScope ps(PH_LAZY_UPDATE_W, st);
            k_lazy_update_w<<<dim3((n_new + 63) / 64, (rp + 255) / 256, L), 256, 0, st>>>(
                n_new, nsteps, ld, rp, w.Wt[cur], w.Wt[nxt], w.src, w.U, w.C);
            ZIPLM_CHECK_LAUNCH();
        }
        if (!compact) {
            // every position stays in place: dense tiles, tensor-core kernel
            PhaseScope ps(PH_LAZY_UPDATE_AQ, st);
            s = run_lazy_update_aq_tc(map_p, map_a[cur], map_q[cur], map_w[cur], L, (nsteps + GS - 1) / GS, n_new, ld, rp,
                                      w.A[nxt], w.Q[nxt], w.Wt[nxt], w.sched, layer_status, spin, st);
            if (s != ZIPLM_OK) return s;
        } else if (n_new > 1) {
            PhaseScope ps(PH_LAZY_UPDATE_AQ, st);
            const int T = (n_new + 63) / 64;
            k_lazy_update_aq<<<dim3(T * (T + 1) / 2, L), 128, 0, st>>>(
                n_new, nsteps, ld, w.A[cur], w.Q[cur], w.A[nxt], w.Q[nxt], w.src, w.U, w.Z);
            ZIPLM_CHECK_LAUNCH();
        }
        cur = nxt;
        npos = n_new;
        n -= nsteps;
        t += nsteps;
        if (slot < n_levels && levels[slot] == n) {
            s = snapshot(npos, slot++);
            if (s != ZIPLM_OK) return s;
        }
        if (last) {
            EndgameTail tail = {};
            tail.L = L; tail.r = r; tail.d = d;
            tail.W = W; tail.H = H;
            tail.Wt = w.Wt[cur]; tail.wt_rows = ld; tail.rp = rp;
            tail.idx = w.idx[cur]; tail.idx_pitch = ld;
            tail.norm2 = w.norm2; tail.norm2_pitch = ld;
            tail.sumrho = &w.state->sumrho; tail.sumrho_stride = (int)(sizeof(LazyState) / sizeof(double));
            tail.lam = w.lam;
            tail.W_snap = W_snap; tail.loss = loss; tail.order = order; tail.saliency = saliency;
            tail.layer_status = layer_status;
            return run_endgame_tail(tail, levels, n_levels, slot, w.aux, st);
        }
    }
    return ZIPLM_OK;
}

}  // namespace ziplm
