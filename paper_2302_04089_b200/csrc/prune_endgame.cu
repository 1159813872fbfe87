// The last steps of a greedy run over neurons (up to kEndgame = 256 live structures), and whole runs of
// layers that are no wider.
//
// The delayed-update path (prune_lazy.cu) pays two or three dependent launches for every 32 steps and a chain
// of 2800 to 3300 clocks a step, whatever the size: a layer of 64 x 256 took 0.7 ms, nearly all of it latency.
// With 256 structures or fewer the state fits the registers of a cluster of eight CTAs, in float64:
//
//   k_endgame_setup   H_lambda restricted to the live structures (by the remark after Eq. 4 its inverse is
//                     H^-1 restricted to them: an exact rebuild, whatever happened before) and the Gram
//                     matrix Q of the current weight columns, both in float64; then the float64 inverse;
//   k_endgame_steps   all remaining steps in one launch: every CTA holds its rows of H^-1 and Q in
//                     registers and applies each step's rank-1 updates (Eq. 4, and the Gram matrix's form
//                     of Eq. 3) at once, so there are no pending terms, nothing is stored and nothing
//                     drifts; the step order, u_s and the pivots go to memory;
//   k_endgame_weights W replayed over those steps, a CTA for 32 rows of W: the scaled pivot columns c_s by
//                     forward substitution, rank-32 updates, and the snapshot of every level on the way;
//   k_endgame_loss    losses.
//
// One layer of 64 x 256 (192 steps, three levels): 1.08 -> 0.36 ms a whole call, of which the steps 0.205 and the
// factorisation 0.07 (0.72 ms for the loop alone with pending updates, a launch every 32 steps).
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"
#include "damping.cuh"
#include "pick.cuh"
#include "tc_common.cuh"

namespace cg = cooperative_groups;

namespace ziplm {
namespace {

constexpr int kMaxN = kEndgame;
constexpr int WORKERS = 16;                       // warps that hold rows of the state
constexpr int STEP_THREADS = 32 * (WORKERS + 1);  // ... and one that keeps the diagonals
constexpr int CHUNK = 32;                         // steps per rank update of W
constexpr int WT = 512;                           // threads of the kernel that replays W

struct Levels {
    int count;                  // levels reached here
    int slot0;                  // ... the first one's slot
    short done[kMaxN + 1];      // steps done when it is reached
};

struct Endgame {
    int L, r, d, n0, n_steps, t0;      // n0 live structures, n_steps of them to be removed, t0 removed before
    const float* W; const float* H;    // the caller's
    const float* Wt; int wt_rows, rp;  // current W^T by position ([wt_rows][rp] per layer), or null: W itself
    const int* idx; int idx_pitch;     // original column of a position, or null: the position
    const double* norm2; int norm2_pitch;   // ||W[:,c]||^2 of the caller's W by column, or null: diagonal of Q
    const double* sumrho; int sumrho_stride;    // sum of the saliencies so far, or null: 0
    double* lam; float damp_frac; bool own_lam;
    double* A64;                       // [dp][dp] H_lambda for the inverse
    double* inv; double* Q;            // [n0][n0]
    double* base_part;                 // [gram tiles]
    float* U; int u_pitch;             // [n_steps][u_pitch], u_pitch = n0 rounded up to 4
    int* piv; double* rs; double* rho; int* removed;     // by step, by step, by step; step by position
    double* dw2;                       // [levels][slabs]
    float* W_snap; int n_levels; float* loss; float* base_loss;
    int* order; float* saliency; int* layer_status;
    Levels lv;
};

// ------------------------------------------------------------------------------------------ set-up
// CTAs 0 .. n_gram - 1: a 32 x 32 tile (on or below the diagonal) of Q = W^T W over the live columns, and
// its share of <Q, H> when the run starts here; the rest: 16 rows of H_lambda, identity on the padding.
__global__ void __launch_bounds__(256) k_endgame_setup(const __grid_constant__ Endgame w, int n_gram, int dp) {
    constexpr int P = 36;                    // pitch of a chunk [position][k], 4 mod 16 doubles
    __shared__ double sa[32 * P], sb[32 * P];
    __shared__ double red8[8];
    const int l = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = w.n0;
    const float* Hl = w.H + (size_t)l * w.d * w.d;
    if ((int)blockIdx.x < n_gram) {
        int ti = 0, tj = blockIdx.x;
        while (tj > ti) { tj -= ti + 1; ++ti; }
        const int i0 = 32 * ti, j0 = 32 * tj;
        const float* src = w.Wt ? w.Wt + (size_t)l * w.wt_rows * w.rp : w.W + (size_t)l * w.r * w.d;
        double acc[2][2] = {};
        float va[4], vb[4];
        auto fetch = [&](int k0) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                // W^T: lanes along k; W: lanes along the columns
                const int m = w.Wt ? warp + 8 * e : lane, k = k0 + (w.Wt ? lane : warp + 8 * e);
                const bool in = k < w.r;
                const size_t oa = w.Wt ? (size_t)(i0 + m) * w.rp + k : (size_t)k * w.d + i0 + m;
                const size_t ob = w.Wt ? (size_t)(j0 + m) * w.rp + k : (size_t)k * w.d + j0 + m;
                va[e] = in && i0 + m < n ? src[oa] : 0.f;
                vb[e] = in && j0 + m < n ? src[ob] : 0.f;
            }
        };
        fetch(0);
        for (int k0 = 0; k0 < w.r; k0 += 32) {
            __syncthreads();
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = w.Wt ? warp + 8 * e : lane, k = w.Wt ? lane : warp + 8 * e;
                sa[m * P + k] = (double)va[e];
                sb[m * P + k] = (double)vb[e];
            }
            __syncthreads();
            if (k0 + 32 < w.r) fetch(k0 + 32);
            // warp: rows 8 (warp / 2) .., columns 16 (warp % 2) ..
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const double a = sa[(8 * (warp >> 1) + (lane >> 2)) * P + 4 * kk + (lane & 3)];
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    dmma884(acc[j], a, sb[(16 * (warp & 1) + 8 * j + (lane >> 2)) * P + 4 * kk + (lane & 3)]);
            }
        }
        double* Ql = w.Q + (size_t)l * n * n;
        double part = 0.0;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int row = i0 + 8 * (warp >> 1) + (lane >> 2), col = j0 + 16 * (warp & 1) + 8 * j + 2 * (lane & 3) + e;
                if (row >= n || col > row) continue;
                Ql[(size_t)row * n + col] = acc[j][e];
                Ql[(size_t)col * n + row] = acc[j][e];
                if (!w.Wt && w.base_loss)
                    part += (row == col ? 1.0 : 2.0) * acc[j][e] * (double)Hl[(size_t)row * w.d + col];
            }
        if (!w.Wt && w.base_loss) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            if (lane == 0) red8[warp] = part;
            __syncthreads();
            if (tid == 0) {
                double t = 0.0;
                for (int q = 0; q < 8; ++q) t += red8[q];
                w.base_part[(size_t)l * n_gram + blockIdx.x] = t;
            }
        }
        return;
    }
    const int x = (int)blockIdx.x - n_gram;
    const double lm = w.own_lam ? mean_diag_lambda(Hl, w.d, w.damp_frac, w.layer_status, l, x == 0) : w.lam[l];
    if (x == 0 && w.own_lam) {
        if (tid == 0) w.lam[l] = lm;
        // what no step of the run writes
        for (int c = tid; c < w.d; c += 256) {
            if (c >= w.n_steps) {
                w.order[(size_t)l * w.d + c] = -1;
                if (w.saliency) w.saliency[(size_t)l * w.d + c] = 0.f;
            }
        }
    }
    double* A = w.A64 + (size_t)l * dp * dp;
    const int* idx = w.idx ? w.idx + (size_t)l * w.idx_pitch : nullptr;
    bool bad = false;
    for (int e = tid; e < 16 * dp; e += 256) {
        const int i = 16 * x + e / dp, j = e % dp;
        double v = i == j ? 1.0 : 0.0;
        if (i < n && j < n) {
            const float h = idx ? Hl[(size_t)idx[i] * w.d + idx[j]] : Hl[(size_t)i * w.d + j];
            if (!isfinite(h)) bad = true;
            v = (double)h + (i == j ? lm : 0.0);
        }
        A[(size_t)i * dp + j] = v;
    }
    if (bad) set_layer_status(w.layer_status, l, ZIPLM_ERR_NONFINITE);
}

// ------------------------------------------------------------------------------------------- steps
// A cluster of CS CTAs per layer; CTA `rank` owns S rows of H^-1 and Q, held in the registers of its 16
// worker warps (4 rows x 32 CPL columns each).  Lane t of the control warp owns the rows' diagonals.
// What the CTAs exchange in a step is small: every one's best offer for the next pick, and u, z of its own
// rows, which it can form by itself because the pivot column restricted to its rows is a column of its own
// block.  Both go out as asynchronous stores that complete on a barrier of the receiving CTA:
//   wait for the step's data; every warp picks p from the offers; the workers that hold column p lay it
//   out; barrier
//   control: column p brought up to date by the step before, u and z of its rows, their diagonals, the
//            next offer; sends both             | workers: the rank-1 updates of the step before
// u, z are in three buffers by step: a CTA may send step m while another's workers still apply step m - 2.
// u and the bookkeeping of all steps are kept in shared memory and written out at the end.
// One layer of 256: a version that pushed every CTA's offered row of 2 x 256 doubles to all others took
// 2.5 us a step, half of it those stores and the cluster barrier behind them; with this exchange and a
// cluster barrier 1.8 us; as it stands 1.05 us.
template <int CS, int S, int CPL> struct StepsCfg {
    static constexpr int RG = S / 4, CG = WORKERS / RG, NP = CG * 32 * CPL, E = (S + 31) / 32;
};

template <int CS, int S, int CPL>
__global__ void __launch_bounds__(STEP_THREADS, 1) k_endgame_steps(const __grid_constant__ Endgame w) {
    using C = StepsCfg<CS, S, CPL>;
    constexpr int NP = C::NP, E = C::E;
    static_assert(CS * S == NP && NP <= kMaxN, "rows and columns cover the same positions");
    extern __shared__ float dyn_hist[];                        // [n_steps][S] u of the own rows
    __shared__ __align__(16) double2 s_uz[3][NP];              // u, z by step
    __shared__ __align__(16) double2 s_col[S];                 // column p of H^-1 and Q, own rows
    __shared__ Bid s_bid[2][CS];                               // by step parity
    __shared__ uint64_t bar_step[2];
    __shared__ int h_piv[kMaxN], h_org[kMaxN];
    __shared__ double h_rs[kMaxN], h_rho[kMaxN];
    __shared__ int abort_flag, s_stopped;                      // step of a give-up
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = CS > 1 ? (int)cluster.block_rank() : 0;
    const int l = blockIdx.x / CS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = w.n0, row0 = rank * S;
    const bool control = warp == WORKERS;
    const int rg = warp / C::CG, col0 = (warp % C::CG) * 32 * CPL;        // workers: rows row0 + 4 rg + x
    const double* Ag = w.inv + (size_t)l * n * n;
    const double* Qg = w.Q + (size_t)l * n * n;
    const int* idx = w.idx ? w.idx + (size_t)l * w.idx_pitch : nullptr;

    double A[4][CPL], Q[4][CPL];             // workers
    double da[E], dq[E];                     // control: row lane + 32 e
    int org[E];
    bool alive[E];
    int first_bad = ZIPLM_OK;
    uint32_t to_uz[CS], to_bid = 0;          // control: where the CTAs take u, z and the bid
    const uint32_t uz_to_bar = tc::smem_u32(&bar_step[0]) - tc::smem_u32(&s_uz[0][row0 + min(lane, S - 1)]);
    const uint32_t bid_to_bar = tc::smem_u32(&bar_step[0]) - tc::smem_u32(&s_bid[0][rank]);

    // control: the CTA's best offer for step m, sent to every CTA
    auto offer = [&](int m) {
        unsigned k[E], kmine = kKeyNone;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            k[e] = cand_key(alive[e], da[e], dq[e]);
            kmine = min(kmine, k[e]);
        }
        const unsigned kmin = __reduce_min_sync(0xffffffffu, kmine);
        Cand mine;
        mine.a = da[0]; mine.q = dq[0]; mine.org = org[0]; mine.pos = alive[0] ? row0 + lane : -1;
#pragma unroll
        for (int e = 1; e < E; ++e) {
            if (!alive[e] || (alive[0] && k[e] > k[0] + kKeyNear)) continue;      // beyond a tie of the fp32 quotients
            Cand c;
            c.a = da[e]; c.q = dq[e]; c.org = org[e]; c.pos = row0 + lane + 32 * e;
            merge_cand(mine, c);
        }
        unsigned near_min = __ballot_sync(0xffffffffu, mine.pos >= 0 && kmine - kmin <= kKeyNear);
        Cand best = bcast_cand(mine, near_min ? __ffs(near_min) - 1 : 0);
        if (near_min & (near_min - 1)) {          // several: the exact comparison
            near_min &= near_min - 1;
            while (near_min) {
                const int b = __ffs(near_min) - 1;
                near_min &= near_min - 1;
                merge_cand(best, bcast_cand(mine, b));
            }
        }
        if (lane < CS) {
            const long long ids = ((long long)best.pos << 32) | (unsigned)best.org;
            if (CS > 1) {
                const uint32_t to = to_bid + (uint32_t)((m & 1) * CS * sizeof(Bid)), bar = to_bid + bid_to_bar + 8u * (m & 1);
                tc::send2(to, best.a, best.q, bar);
                tc::send2(to + 16u, ids, (long long)kmin, bar);
            } else {
                Bid b;
                b.a = best.a; b.q = best.q; b.org = best.org; b.pos = best.pos; b.key = kmin; b.pad = 0;
                s_bid[m & 1][0] = b;
            }
        }
    };

    if (tid == 0) {
        abort_flag = 0;
        tc::mbar_init(tc::smem_u32(&bar_step[0]), 1);
        tc::mbar_init(tc::smem_u32(&bar_step[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (CS > 1) cluster.sync();              // every CTA of the cluster has started
    if (control) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int k = row0 + lane + 32 * e;
            alive[e] = lane + 32 * e < S && k < n;
            da[e] = alive[e] ? Ag[(size_t)k * n + k] : 1.0;
            dq[e] = alive[e] ? Qg[(size_t)k * n + k] : 0.0;
            org[e] = !alive[e] ? 0x7fffffff : idx ? idx[k] : k;
        }
        if (CS > 1) {
#pragma unroll
            for (int c = 0; c < CS; ++c) {
                to_uz[c] = tc::map_rank(&s_uz[0][row0 + min(lane, S - 1)], c);
            }
            to_bid = tc::map_rank(&s_bid[0][rank], lane < CS ? lane : 0);
            if (lane == 0) tc::mbar_expect_tx(tc::smem_u32(&bar_step[0]), CS * sizeof(Bid));
        }
        for (int k = lane; k < NP; k += 32) s_uz[2][k] = make_double2(0.0, 0.0);
        offer(0);
    } else {
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int q = 0; q < CPL; ++q) {
                const int i = row0 + 4 * rg + x, j = col0 + 32 * q + lane;
                const bool in = i < n && j < n;
                A[x][q] = in ? Ag[(size_t)i * n + j] : 0.0;
                Q[x][q] = in ? Qg[(size_t)i * n + j] : 0.0;
            }
    }
    __syncthreads();

    // The pick of step m.
    bool failed = false;
    auto pick = [&](int m) -> const Bid* {
        const int par = m & 1;
        int which = 0;
        if (CS > 1) {
            if (!tc::mbar_wait(tc::smem_u32(&bar_step[par]), (uint32_t)(m >> 1) & 1u, &abort_flag)) {
                failed = true;
                abort_flag = 1;
            }
            which = best_bid(s_bid[par], CS, lane);
        }
        return &s_bid[par][which];
    };
    // two loops, so that the workers' state and the control warp's share registers
    int cur = 0, last = 2;                   // buffers of step m and step m - 1
    if (!control) {
        for (int m = 0; m < w.n_steps; ++m) {
            const double2* prev = s_uz[last];
            const int p = min(max(pick(m)->pos, 0), NP - 1);
            if (p / (32 * CPL) == warp % C::CG && (p & 31) == lane) {
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    int pc = (p / 32) % CPL;
                    asm volatile("" : "+r"(pc));      // a test per column: an indexed A would live in local memory
                    if (pc == c) {
#pragma unroll
                        for (int x = 0; x < 4; ++x) s_col[4 * rg + x] = make_double2(A[x][c], Q[x][c]);
                    }
                }
            }
            if (__syncthreads_or(failed)) { failed = true; s_stopped = m; break; }
            double2 ui[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) ui[x] = prev[row0 + 4 * rg + x];
            // the float64 pipe belongs to the control warp until it has sent u and z
            asm volatile("bar.sync 1, %0;" ::"n"(STEP_THREADS) : "memory");
#pragma unroll
            for (int q = 0; q < CPL; ++q) {
                const double2 uj = prev[col0 + 32 * q + lane];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    A[x][q] = fma(-ui[x].x, uj.x, A[x][q]);
                    Q[x][q] = fma(-ui[x].y, uj.x, fma(-ui[x].x, uj.y, Q[x][q]));
                }
            }
            if (CS == 1) __syncthreads();
            last = cur;
            cur = cur == 2 ? 0 : cur + 1;
        }
    } else {
        for (int m = 0; m < w.n_steps; ++m) {
            const int par = m & 1;
            const double2* prev = s_uz[last];
            const Bid* bid = pick(m);
            const int p = min(max(bid->pos, 0), NP - 1);
            const double ga = bid->a, gq = bid->q;
            const double2 pp = prev[p];
            double2 pj[E];
#pragma unroll
            for (int e = 0; e < E; ++e) pj[e] = prev[row0 + min(lane + 32 * e, S - 1)];
            if (CS > 1 && lane == 0)
                tc::mbar_expect_tx(tc::smem_u32(&bar_step[par ^ 1]), NP * sizeof(double2) + CS * sizeof(Bid));
            double h = ga;
            int bad = 0;
            if (!isfinite(gq) || !isfinite(h)) { bad = ZIPLM_ERR_NONFINITE; h = 1.0; }
            else if (!(h > 0.0)) { bad = ZIPLM_ERR_NOT_PD; h = 1.0; }
            const double rs = rsqrt(h), half = 0.5 * gq * rs * rs;
            if (__syncthreads_or(failed)) { failed = true; break; }
            float uh[E];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int j = lane + 32 * e;
                alive[e] = alive[e] && row0 + j != p;
                const double2 col = s_col[min(j, S - 1)];
                const double a = fma(-pj[e].x, pp.x, col.x);
                const double q = fma(-pj[e].y, pp.x, fma(-pj[e].x, pp.y, col.y));
                const double u = alive[e] ? a * rs : 0.0;
                const double z = alive[e] ? fma(q, rs, -half * u) : 0.0;
                if (j < S) {
                    if (CS > 1) {
                        static_assert(CS == 1 || E == 1, "one row per lane on a cluster");
#pragma unroll
                        for (int c = 0; c < CS; ++c)
                            tc::send2(to_uz[c] + (uint32_t)(cur * NP * sizeof(double2)), u, z,
                                  to_uz[c] + uz_to_bar + 8u * (par ^ 1));
                    } else {
                        s_uz[cur][j] = make_double2(u, z);
                    }
                }
                da[e] = fma(-u, u, da[e]);
                dq[e] = fma(-2.0 * z, u, dq[e]);
                uh[e] = (float)u;
            }
            asm volatile("bar.arrive 1, %0;" ::"n"(STEP_THREADS) : "memory");
            offer(m + 1);
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (lane + 32 * e < S) dyn_hist[m * S + lane + 32 * e] = uh[e];
            if (bad && first_bad == ZIPLM_OK) first_bad = bad;
            if (lane == 0) {
                h_piv[m] = p;
                h_org[m] = bid->org;
                h_rs[m] = rs;
                h_rho[m] = bad ? 0.0 : gq * rs * rs;
            }
            if (CS == 1) __syncthreads();
            last = cur;
            cur = cur == 2 ? 0 : cur + 1;
        }
    }
    if (failed && tid == 0) set_layer_status(w.layer_status, l, ZIPLM_ERR_TIMEOUT);
    if (CS > 1 && !failed && tid == 0)       // what the last step sent has landed before any CTA leaves
        tc::mbar_wait_quiet(tc::smem_u32(&bar_step[w.n_steps & 1]), (uint32_t)(w.n_steps >> 1) & 1u);
    __syncthreads();
    if (CS > 1) cluster.sync();
    // After a give-up: what the others had sent by then, for this step and the next, lands or runs out once more.
    if (CS > 1 && failed && tid == 0)
        for (int m = s_stopped; m < s_stopped + 2; ++m)
            if (!tc::mbar_wait_quiet(tc::smem_u32(&bar_step[m & 1]), (uint32_t)(m >> 1) & 1u)) break;

    for (int e = tid; e < w.n_steps * S; e += STEP_THREADS) {
        const int m = e / S, k = row0 + e % S;
        if (k < n) w.U[((size_t)l * w.n_steps + m) * w.u_pitch + k] = dyn_hist[e];
    }
    if (rank == 0) {
        for (int k = tid; k < n; k += STEP_THREADS) w.removed[(size_t)l * n + k] = 0x7fffffff;
        __syncthreads();
        for (int m = tid; m < w.n_steps; m += STEP_THREADS) {
            const size_t at = (size_t)l * w.n_steps + m;
            const int p = failed ? min(m, n - 1) : h_piv[m];
            w.piv[at] = p;
            w.rs[at] = h_rs[m];
            w.rho[at] = h_rho[m];
            w.removed[(size_t)l * n + p] = m;
            w.order[(size_t)l * w.d + w.t0 + m] = failed ? -1 : h_org[m];
            if (w.saliency) w.saliency[(size_t)l * w.d + w.t0 + m] = (float)h_rho[m];
        }
        if (control && lane == 0 && first_bad != ZIPLM_OK) set_layer_status(w.layer_status, l, first_bad);
    }
}

// ----------------------------------------------------------------------------------------- weights
// A CTA replays 32 rows of W over all steps: chunks of up to 32 steps that end at the levels.  The scaled
// pivot columns c_m = (W[:,p_m] - sum_{s<m} c_s u_s[p_m]) / sqrt(h_m) of its rows are solved by one warp
// (a lane per row, sums in float64, every c_m subtracted from the later ones as soon as it is known, so that
// the chain is one product and two conversions a step; by all warps side by side it took twice as long, bound
// by their reads of T).  The rank update takes four positions at a time, so that a broadcast load of u feeds
// four FMAs and four chains run side by side.  The u of the next chunk arrive meanwhile.
__global__ void __launch_bounds__(WT) k_endgame_weights(const __grid_constant__ Endgame w) {
    extern __shared__ __align__(16) float dyn_w[];
    const int n = w.n0, l = blockIdx.y, i0 = blockIdx.x * 32, pitch = w.u_pitch;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* sU = dyn_w;                                   // [2][32][pitch] u_s of two chunks
    double* sT = reinterpret_cast<double*>(sU + 2 * CHUNK * pitch);      // [s][m] T = u_s[p_m], widened once (a
                                                         // conversion costs as much as eight FMAs)
    float* sW = reinterpret_cast<float*>(sT + CHUNK * CHUNK);            // [pitch][33] current weights, by position
    float* sO = sW + pitch * 33;                         // [n][33] original ones
    int* sRem = reinterpret_cast<int*>(sO + n * 33);     // [n] step that removes a position
    short* sPos = reinterpret_cast<short*>(sRem + n);    // [d] position of a column, -1: none
    __shared__ int s_all_piv[kMaxN + CHUNK];
    __shared__ double s_all_rs[kMaxN + CHUNK], red[WT / 32];
    __shared__ float sC[CHUNK][32];
    const int* idx = w.idx ? w.idx + (size_t)l * w.idx_pitch : nullptr;
    const float* Wl = w.W + (size_t)l * w.r * w.d;
    const float* Ul = w.U + (size_t)l * w.n_steps * pitch;
    // chunk of steps [t, t + m_n) into a buffer; steps past m_n are zero
    auto stage = [&](int b, int t, int m_n) {
        const int quads = pitch / 4;
        float* to = sU + b * CHUNK * pitch;
        for (int e = tid; e < CHUNK * quads; e += WT) {
            const int s = e / quads, k = 4 * (e % quads);
            const unsigned sa = tc::smem_u32(to + s * pitch + k);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa),
                         "l"(Ul + (size_t)(s < m_n ? t + s : 0) * pitch + k), "r"(s < m_n ? 16u : 0u) : "memory");
        }
    };
    // the chunk that follows step t: ends at a level or after 32 steps
    auto chunk_len = [&](int t, int q) {
        while (q < w.lv.count && w.lv.done[q] <= t) ++q;
        return q < w.lv.count ? min(CHUNK, (int)w.lv.done[q] - t) : 0;
    };
    int m_n = chunk_len(0, 0), buf = 0;
    if (m_n > 0) stage(0, 0, m_n);
    asm volatile("cp.async.commit_group;" ::: "memory");
    for (int m = tid; m < kMaxN + CHUNK; m += WT) {
        s_all_piv[m] = m < w.n_steps ? w.piv[(size_t)l * w.n_steps + m] : 0;
        s_all_rs[m] = m < w.n_steps ? w.rs[(size_t)l * w.n_steps + m] : 0.0;
    }
    for (int c = tid; c < w.d; c += WT) sPos[c] = (short)(idx ? -1 : c);
    for (int e = tid; e < (pitch - n) * 33; e += WT) sW[n * 33 + e] = 0.f;
    __syncthreads();
    for (int k = tid; k < n; k += WT) {
        sRem[k] = w.n_steps > 0 ? w.removed[(size_t)l * n + k] : 0x7fffffff;
        if (idx) sPos[idx[k]] = (short)k;
    }
    if (w.Wt) {
        const float* Wtl = w.Wt + (size_t)l * w.wt_rows * w.rp;
        for (int k = warp; k < n; k += WT / 32) {
            const int i = i0 + lane;
            sW[k * 33 + lane] = i < w.r ? Wtl[(size_t)k * w.rp + i] : 0.f;
            sO[k * 33 + lane] = i < w.r ? Wl[(size_t)i * w.d + (idx ? idx[k] : k)] : 0.f;
        }
    } else {
        for (int e = tid; e < 32 * n; e += WT) {
            const int i = e / n, k = e % n;
            const float v = i0 + i < w.r ? Wl[(size_t)(i0 + i) * w.d + k] : 0.f;
            sW[k * 33 + i] = v;
            sO[k * 33 + i] = v;
        }
    }
    int t = 0;
    for (int q = 0; q < w.lv.count; ++q) {
        const int stop = w.lv.done[q];
        while (t < stop) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            const int* s_piv = s_all_piv + t;
            const double* s_rs = s_all_rs + t;
            const float* U = sU + buf * CHUNK * pitch;
            const int next = chunk_len(t + m_n, q);
            if (next > 0) stage(buf ^ 1, t + m_n, next);
            asm volatile("cp.async.commit_group;" ::: "memory");
            for (int e = tid; e < CHUNK * CHUNK; e += WT) sT[e] = (double)U[(e >> 5) * pitch + s_piv[e & 31]];
            __syncthreads();
            if (warp == 0) {
                double c[CHUNK];
#pragma unroll
                for (int m = 0; m < CHUNK; ++m) c[m] = m < m_n ? (double)sW[s_piv[m] * 33 + lane] : 0.0;
#pragma unroll
                for (int s = 0; s < CHUNK; ++s) {
                    const float f = s < m_n ? (float)(c[s] * s_rs[s]) : 0.f;
                    const double cs = (double)f;
                    sC[s][lane] = f;
#pragma unroll
                    for (int m = s + 1; m < CHUNK; ++m) c[m] = fma(-cs, sT[s * CHUNK + m], c[m]);
                }
            }
            __syncthreads();
            float cf[CHUNK];
#pragma unroll
            for (int s = 0; s < CHUNK; ++s) cf[s] = sC[s][lane];
            for (int k = 4 * warp; k < pitch; k += WT / 8) {
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = sW[(k + e) * 33 + lane];
#pragma unroll
                for (int s = 0; s < CHUNK; ++s) {
                    const float4 u = *reinterpret_cast<const float4*>(U + s * pitch + k);
                    v[0] = fmaf(-u.x, cf[s], v[0]);
                    v[1] = fmaf(-u.y, cf[s], v[1]);
                    v[2] = fmaf(-u.z, cf[s], v[2]);
                    v[3] = fmaf(-u.w, cf[s], v[3]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) sW[(k + e) * 33 + lane] = v[e];
            }
            t += m_n;
            m_n = next;
            buf ^= 1;
        }
        __syncthreads();
        // ---- level: rows i0 .. of the snapshot in original column order, removed columns exactly zero
        const int slot = w.lv.slot0 + q;
        float* out = w.W_snap + (((size_t)l * w.n_levels + slot) * w.r + i0) * w.d;
        for (int i = warp; i < 32 && i0 + i < w.r; i += WT / 32)
#pragma unroll 4
            for (int c = lane; c < w.d; c += 32) {
                const int k = sPos[c];
                out[(size_t)i * w.d + c] = k >= 0 && sRem[k] >= t ? sW[k * 33 + i] : 0.f;
            }
        double part = 0.0;
        for (int k = warp; k < n; k += WT / 32)
            if (sRem[k] >= t) {
                const float df = sO[k * 33 + lane] - sW[k * 33 + lane];
                part += (double)df * (double)df;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) red[warp] = part;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int v = 0; v < WT / 32; ++v) s += red[v];
            w.dw2[((size_t)l * w.lv.count + q) * gridDim.x + blockIdx.x] = s;
        }
        m_n = chunk_len(t, q + 1);
    }
}

// loss = half the sum of the saliencies of the removed structures, less the damping's share; one CTA per
// level and layer.  ||W - W_snap||^2 is the norms of the removed columns and what the kept ones moved.
__global__ void __launch_bounds__(128) k_endgame_loss(const __grid_constant__ Endgame w, int slabs, int n_gram) {
    __shared__ double red[4];
    __shared__ unsigned char kept[6144];
    const int l = blockIdx.y, tid = threadIdx.x, n = w.n0;
    if (blockIdx.x == 0 && w.base_loss && !w.Wt && tid == 0) {
        double t = 0.0;
        for (int q = 0; q < n_gram; ++q) t += w.base_part[(size_t)l * n_gram + q];
        w.base_loss[l] = (float)(0.5 * t);
    }
    if ((int)blockIdx.x >= w.lv.count) return;
    const int q = blockIdx.x, t = w.lv.done[q];
    const int* idx = w.idx ? w.idx + (size_t)l * w.idx_pitch : nullptr;
    for (int c = tid; c < w.d; c += 128) kept[c] = 0;
    __syncthreads();
    for (int k = tid; k < n; k += 128)
        if (w.n_steps == 0 || w.removed[(size_t)l * n + k] >= t) kept[idx ? idx[k] : k] = 1;
    __syncthreads();
    double dw = 0.0, rho = 0.0;
    for (int c = tid; c < w.d; c += 128)
        if (!kept[c]) dw += w.norm2 ? w.norm2[(size_t)l * w.norm2_pitch + c] : w.Q[(size_t)l * n * n + (size_t)c * n + c];
    for (int s = tid; s < slabs; s += 128) dw += w.dw2[((size_t)l * w.lv.count + q) * slabs + s];
    for (int s = tid; s < t; s += 128) rho += w.rho[(size_t)l * w.n_steps + s];
    double v = 0.5 * rho - 0.5 * w.lam[l] * dw;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
        double s = w.sumrho ? 0.5 * w.sumrho[(size_t)l * w.sumrho_stride] : 0.0;
        for (int e = 0; e < 4; ++e) s += red[e];
        w.loss[(size_t)l * w.n_levels + w.lv.slot0 + q] = (float)(s > 0.0 ? s : 0.0);
    }
}

int gram_tiles(int n) {
    const int T = (n + 31) / 32;
    return T * (T + 1) / 2;
}

size_t weights_smem(int n, int d) {
    const int pitch = round_up_int(n, 4);
    return sizeof(float) * (size_t)(2 * CHUNK * pitch + 2 * CHUNK * CHUNK + pitch * 33 + n * 33 + n) +
           sizeof(short) * (size_t)d;
}

// Carves the scratch; with ws == nullptr it only measures.
size_t carve_endgame(Endgame* w, void** inv_ws, void* ws, int L, int r, int n0, int n_levels) {
    Carver c(ws);
    Endgame dummy;
    if (!w) w = &dummy;
    *inv_ws = c.take<char>(inverse_workspace_bytes(L, n0));
    w->inv = c.take<double>((size_t)L * n0 * n0);
    w->Q = c.take<double>((size_t)L * n0 * n0);
    w->base_part = c.take<double>((size_t)L * gram_tiles(n0));
    w->u_pitch = round_up_int(n0, 4);
    w->U = c.take<float>((size_t)L * n0 * w->u_pitch);
    w->piv = c.take<int>((size_t)L * n0);
    w->rs = c.take<double>((size_t)L * n0);
    w->rho = c.take<double>((size_t)L * n0);
    w->removed = c.take<int>((size_t)L * n0);
    w->dw2 = c.take<double>((size_t)L * (n_levels + 1) * ((r + 31) / 32));
    w->lam = c.take<double>((size_t)L);
    return c.off;
}

template <int CS, int S, int CPL>
ziplm_status launch_steps(const Endgame& w, cudaStream_t st) {
    auto kernel = k_endgame_steps<CS, S, CPL>;
    const int smem = w.n_steps * S * (int)sizeof(float);
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          kMaxN * S * (int)sizeof(float)));
    int least = 0, greatest = 0;
    ZIPLM_CHECK_CUDA(cudaDeviceGetStreamPriorityRange(&least, &greatest));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(w.L * CS);
    cfg.blockDim = dim3(STEP_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributePriority;        // a latency chain: ahead of other groups' wide kernels
    attr[1].val.priority = greatest;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kernel, w));
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

ziplm_status run(Endgame& w, void* inv_ws, cudaStream_t st) {
    const int n = w.n0, dp = round_up_int(n, kTile), tiles = gram_tiles(n), slabs = (w.r + 31) / 32;
    ziplm_status s;
    w.A64 = inverse_matrix(inv_ws);
    {
        PhaseScope ps(PH_INIT, st);
        k_endgame_setup<<<dim3(tiles + dp / 16, w.L), 256, 0, st>>>(w, tiles, dp);
        ZIPLM_CHECK_LAUNCH();
    }
    {
        PhaseScope ps(PH_INVERSE, st);
        s = run_inverse_of(inv_ws, w.L, n, w.inv, w.layer_status, st);
        if (s != ZIPLM_OK) return s;
    }
    if (w.n_steps > 0) {
        PhaseScope ps(PH_LAZY_STEPS, st);
        // the smallest cluster that holds the state
        s = n <= 64 ? launch_steps<1, 64, 2>(w, st) : n <= 128 ? launch_steps<4, 32, 2>(w, st) : launch_steps<8, 32, 4>(w, st);
        if (s != ZIPLM_OK) return s;
    }
    if (w.lv.count > 0) {
        PhaseScope ps(PH_LAZY_UPDATE_W, st);
        const size_t smem = weights_smem(n, w.d);
        ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_endgame_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_endgame_weights<<<dim3(slabs, w.L), WT, smem, st>>>(w);
        ZIPLM_CHECK_LAUNCH();
    }
    if (w.lv.count > 0 || w.base_loss) {
        PhaseScope ps(PH_SNAPSHOT, st);
        k_endgame_loss<<<dim3(w.lv.count > 0 ? w.lv.count : 1, w.L), 128, 0, st>>>(w, slabs, tiles);
        ZIPLM_CHECK_LAUNCH();
    }
    return ZIPLM_OK;
}

void set_levels(Endgame& w, const int* levels, int n_levels, int slot0) {
    w.lv.slot0 = slot0;
    w.lv.count = n_levels - slot0;
    for (int q = 0; q < w.lv.count; ++q) w.lv.done[q] = (short)(w.n0 - levels[slot0 + q]);
    w.n_steps = w.lv.count > 0 ? w.lv.done[w.lv.count - 1] : 0;
    w.n_levels = n_levels;
}

}  // namespace

size_t endgame_workspace_bytes(int L, int r, int n0, int n_levels) {
    void* inv_ws;
    return carve_endgame(nullptr, &inv_ws, nullptr, L, r, n0, n_levels);
}

ziplm_status run_endgame_whole(const float* W, const float* H, int L, int r, int d, float damp_frac,
                               const int* levels, int n_levels, float* W_snap, float* loss, float* base_loss,
                               int* order, float* saliency, int* layer_status, void* ws, size_t ws_bytes,
                               cudaStream_t st) {
    if (d > kEndgame) return ZIPLM_ERR_UNSUPPORTED;
    if (ws_bytes < endgame_workspace_bytes(L, r, d, n_levels)) return ZIPLM_ERR_WORKSPACE;
    Endgame w = {};
    void* inv_ws;
    carve_endgame(&w, &inv_ws, ws, L, r, d, n_levels);
    w.L = L; w.r = r; w.d = d; w.n0 = d;
    w.W = W; w.H = H; w.damp_frac = damp_frac; w.own_lam = true;
    w.W_snap = W_snap; w.loss = loss; w.base_loss = base_loss; w.order = order; w.saliency = saliency;
    w.layer_status = layer_status;
    set_levels(w, levels, n_levels, 0);
    return run(w, inv_ws, st);
}

ziplm_status run_endgame_tail(const EndgameTail& t, const int* levels, int n_levels, int slot0, void* ws,
                              cudaStream_t st) {
    Endgame w = {};
    void* inv_ws;
    carve_endgame(&w, &inv_ws, ws, t.L, t.r, kEndgame, n_levels);
    w.L = t.L; w.r = t.r; w.d = t.d; w.n0 = kEndgame; w.t0 = t.d - kEndgame;
    w.W = t.W; w.H = t.H; w.Wt = t.Wt; w.wt_rows = t.wt_rows; w.rp = t.rp;
    w.idx = t.idx; w.idx_pitch = t.idx_pitch;
    w.norm2 = t.norm2; w.norm2_pitch = t.norm2_pitch;
    w.sumrho = t.sumrho; w.sumrho_stride = t.sumrho_stride;
    w.lam = const_cast<double*>(t.lam);
    w.W_snap = t.W_snap; w.loss = t.loss; w.order = t.order; w.saliency = t.saliency;
    w.layer_status = t.layer_status;
    set_levels(w, levels, n_levels, slot0);
    return run(w, inv_ws, st);
}

}  // namespace ziplm
