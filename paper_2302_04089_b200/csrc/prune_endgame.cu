// The last steps of a greedy run over neurons (up to kEndgame = 256 live structures), and whole runs of
// layers that are no wider.
//
// The delayed-update path (prune_lazy.cu) pays three dependent launches for every 32 steps and a chain of
// about 3700 clocks a step, whatever the size: a layer of 64 x 256 took 0.7 ms, nearly all of it latency.
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
// One layer of 64 x 256 (192 steps, three levels): 0.715 -> MEASURED ms.
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"
#include "pick.cuh"

namespace cg = cooperative_groups;

namespace ziplm {
namespace {

constexpr int kMaxN = kEndgame;
constexpr int WORKERS = 16;                       // warps that hold rows of the state
constexpr int STEP_THREADS = 32 * (WORKERS + 1);  // ... and one that keeps the diagonals
constexpr int CHUNK = 32;                         // steps per rank update of W

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
    float* U;                          // [n_steps][n0]
    int* piv; double* rs; double* rho; int* removed;     // by step, by step, by step; step by position
    double* dw2;                       // [levels][slabs]
    float* W_snap; int n_levels; float* loss; float* base_loss;
    int* order; float* saliency; int* layer_status;
    Levels lv;
};

// ------------------------------------------------------------------------------------------ set-up
// lambda of a layer as the damped inverse defines it; every thread returns it.
__device__ double mean_diag_lambda(const float* Hl, int d, float damp_frac, int* layer_status, int l, bool report) {
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

__device__ __forceinline__ void dmma(double (&d)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                 : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

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
                    dmma(acc[j], a, sb[(16 * (warp & 1) + 8 * j + (lane >> 2)) * P + 4 * kk + (lane & 3)]);
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
// worker warps (8 rows x 32 CPL columns each).  Lane t of the control warp owns the rows' diagonals.
// What the CTAs exchange in a step is small: every one's best offer for the next pick, and u, z of its own
// rows, which it can form by itself because the pivot column restricted to its rows is a column of its own
// block.  Both go out with one cluster barrier a step:
//   every warp picks p from the offers; the workers that hold column p lay it out; barrier
//   control: column p brought up to date by the step before, u and z of its rows, their diagonals, the
//            next offer; pushes both            | workers: the rank-1 updates of the step before
//   cluster barrier
// u, z and the bookkeeping of all steps are kept in shared memory and written out at the end: a store to
// global memory in front of a cluster barrier makes the barrier wait for it (1060 instead of 590 clocks).
// A first version pushed every CTA's offered row of 2 x 256 doubles to all others: 2.5 us a step, half of it
// those stores and the barrier behind them.
template <int CS, int S, int CPL> struct StepsCfg {
    static constexpr int RG = S / 8, CG = WORKERS / RG, NP = CG * 32 * CPL, E = (S + 31) / 32;
};

template <int CS, int S, int CPL>
__global__ void __launch_bounds__(STEP_THREADS, 1) k_endgame_steps(const __grid_constant__ Endgame w) {
    using C = StepsCfg<CS, S, CPL>;
    constexpr int NP = C::NP, E = C::E;
    static_assert(CS * S == NP && NP <= kMaxN, "rows and columns cover the same positions");
    extern __shared__ float dyn_hist[];                        // [n_steps][S] u of the own rows
    __shared__ __align__(16) double2 s_uz[2][NP];              // u, z by step parity
    __shared__ __align__(16) double2 s_col[S];                 // column p of H^-1 and Q, own rows
    __shared__ Offer s_offer[2][CS];
    __shared__ float s_key[2][CS];
    __shared__ int h_piv[kMaxN], h_org[kMaxN];
    __shared__ double h_rs[kMaxN], h_rho[kMaxN];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = CS > 1 ? (int)cluster.block_rank() : 0;
    const int l = blockIdx.x / CS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = w.n0, row0 = rank * S;
    const bool control = warp == WORKERS;
    const int rg = warp / C::CG, col0 = (warp % C::CG) * 32 * CPL;        // workers: rows row0 + 8 rg + x
    const double* Ag = w.inv + (size_t)l * n * n;
    const double* Qg = w.Q + (size_t)l * n * n;
    const int* idx = w.idx ? w.idx + (size_t)l * w.idx_pitch : nullptr;

    double A[8][CPL], Q[8][CPL];             // workers
    double da[E], dq[E];                     // control: row lane + 32 e
    int org[E];
    bool alive[E];
    int first_bad = ZIPLM_OK;

    // control: the CTA's best offer for step m, pushed to every CTA
    auto offer = [&](int m) {
        float rq[E], rmin = INFINITY;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int ha = __double2hiint(da[e]), hq = __double2hiint(dq[e]);
            const bool ok = (unsigned)(ha - 1) < 0x7fefffffu && (hq & 0x7fffffff) < 0x7ff00000;   // a > 0, finite
            const float x = __fdividef((float)dq[e], (float)da[e]);
            rq[e] = alive[e] ? (ok ? x : -INFINITY) : INFINITY;
            rmin = fminf(rmin, rq[e]);
        }
        Cand mine;
        mine.a = da[0]; mine.q = dq[0]; mine.org = org[0]; mine.pos = alive[0] ? row0 + lane : -1;
#pragma unroll
        for (int e = 1; e < E; ++e) {
            if (!alive[e]) continue;
            Cand c;
            c.a = da[e]; c.q = dq[e]; c.org = org[e]; c.pos = row0 + lane + 32 * e;
            merge_cand(mine, c);
        }
        float key;
        const Cand best = warp_best(mine, rmin, &key);
        if (lane < CS) {
            Offer* o = &s_offer[m & 1][rank];
            float* k = &s_key[m & 1][rank];
            if (CS > 1) {
                o = cluster.map_shared_rank(o, lane);
                k = cluster.map_shared_rank(k, lane);
            }
            o->c = best;
            *k = key;
        }
    };

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
        for (int k = lane; k < NP; k += 32) s_uz[1][k] = make_double2(0.0, 0.0);
        offer(0);
    } else {
#pragma unroll
        for (int x = 0; x < 8; ++x)
#pragma unroll
            for (int q = 0; q < CPL; ++q) {
                const int i = row0 + 8 * rg + x, j = col0 + 32 * q + lane;
                const bool in = i < n && j < n;
                A[x][q] = in ? Ag[(size_t)i * n + j] : 0.0;
                Q[x][q] = in ? Qg[(size_t)i * n + j] : 0.0;
            }
    }
    if (CS > 1) cluster.sync();
    else __syncthreads();

    for (int m = 0; m < w.n_steps; ++m) {
        const int par = m & 1;
        const double2* prev = s_uz[par ^ 1];
        int which;
        const Cand g = CS > 1 ? pick_offer(s_offer[par], s_key[par], CS, lane, &which) : s_offer[par][0].c;
        const int p = g.pos < 0 ? 0 : g.pos;
        if (!control) {
            if (p / (32 * CPL) == warp % C::CG && (p & 31) == lane) {
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    double a = A[x][0], q = Q[x][0];
#pragma unroll
                    for (int c = 1; c < CPL; ++c)
                        if ((p / 32) % CPL == c) { a = A[x][c]; q = Q[x][c]; }
                    s_col[8 * rg + x] = make_double2(a, q);
                }
            }
            __syncthreads();
            double2 uj[CPL];
#pragma unroll
            for (int q = 0; q < CPL; ++q) uj[q] = prev[col0 + 32 * q + lane];
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const double2 ui = prev[row0 + 8 * rg + x];
#pragma unroll
                for (int q = 0; q < CPL; ++q) {
                    A[x][q] = fma(-ui.x, uj[q].x, A[x][q]);
                    Q[x][q] = fma(-ui.y, uj[q].x, fma(-ui.x, uj[q].y, Q[x][q]));
                }
            }
        } else {
            double h = g.a;
            int bad = 0;
            if (!isfinite(g.q) || !isfinite(h)) { bad = ZIPLM_ERR_NONFINITE; h = 1.0; }
            else if (!(h > 0.0)) { bad = ZIPLM_ERR_NOT_PD; h = 1.0; }
            if (bad && first_bad == ZIPLM_OK) first_bad = bad;
            const double rs = rsqrt(h), half = 0.5 * g.q * rs * rs;
            const double2 pp = prev[p];
            double2 pj[E];
#pragma unroll
            for (int e = 0; e < E; ++e) pj[e] = prev[min(row0 + lane + 32 * e, NP - 1)];
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int j = lane + 32 * e;
                alive[e] = alive[e] && row0 + j != p;
                const double2 col = s_col[min(j, S - 1)];
                const double a = fma(-pj[e].x, pp.x, col.x);
                const double q = fma(-pj[e].y, pp.x, fma(-pj[e].x, pp.y, col.y));
                const double u = alive[e] ? a * rs : 0.0;
                const double z = alive[e] ? q * rs - half * u : 0.0;
                da[e] -= u * u;
                dq[e] -= 2.0 * z * u;
                if (j < S) {
                    dyn_hist[m * S + j] = (float)u;
                    if (CS > 1) {
#pragma unroll
                        for (int c = 0; c < CS; ++c)
                            *cluster.map_shared_rank(&s_uz[par][row0 + j], c) = make_double2(u, z);
                    } else {
                        s_uz[par][j] = make_double2(u, z);
                    }
                }
            }
            offer(m + 1);
            if (lane == 0) {
                h_piv[m] = p;
                h_org[m] = g.org;
                h_rs[m] = rs;
                h_rho[m] = bad ? 0.0 : g.q * rs * rs;
            }
        }
        if (CS > 1) cluster.sync();
        else __syncthreads();
    }

    for (int e = tid; e < w.n_steps * S; e += STEP_THREADS) {
        const int m = e / S, k = row0 + e % S;
        if (k < n) w.U[((size_t)l * w.n_steps + m) * n + k] = dyn_hist[e];
    }
    if (rank == 0) {
        for (int k = tid; k < n; k += STEP_THREADS) w.removed[(size_t)l * n + k] = 0x7fffffff;
        __syncthreads();
        for (int m = tid; m < w.n_steps; m += STEP_THREADS) {
            const size_t at = (size_t)l * w.n_steps + m;
            w.piv[at] = h_piv[m];
            w.rs[at] = h_rs[m];
            w.rho[at] = h_rho[m];
            w.removed[(size_t)l * n + h_piv[m]] = m;
            w.order[(size_t)l * w.d + w.t0 + m] = h_org[m];
            if (w.saliency) w.saliency[(size_t)l * w.d + w.t0 + m] = (float)h_rho[m];
        }
        if (control && lane == 0 && first_bad != ZIPLM_OK) set_layer_status(w.layer_status, l, first_bad);
    }
}

// ----------------------------------------------------------------------------------------- weights
// A CTA replays 32 rows of W over all steps: chunks of up to 32 steps that end at the levels.  The scaled
// pivot columns c_m = (W[:,p_m] - sum_{s<m} c_s u_s[p_m]) / sqrt(h_m) of its rows are solved by every warp
// for itself (a lane per row, sums in float64), so that they are in registers for the rank update.
__global__ void __launch_bounds__(256) k_endgame_weights(const __grid_constant__ Endgame w) {
    extern __shared__ float dyn_w[];
    const int n = w.n0, l = blockIdx.y, i0 = blockIdx.x * 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int np4 = (n + 3) & ~3;
    float* sW = dyn_w;                                   // [n][33] current weights, by position
    float* sO = sW + n * 33;                             // [n][33] original ones
    float* sU = sW + ((2 * n * 33 + 3) & ~3);            // [n][36] u_s of the chunk, by position; on 16 bytes
    double* sT = reinterpret_cast<double*>(sU + n * 36);       // [32][32] T[m][s] = u_s[p_m], widened once: a
                                                         // conversion costs as much as eight FMAs
    int* sRem = reinterpret_cast<int*>(sT + CHUNK * CHUNK);    // [n] step that removes a position
    short* sPos = reinterpret_cast<short*>(sRem + np4);  // [d] position of a column, -1: none
    __shared__ int s_piv[CHUNK];
    __shared__ double s_rs[CHUNK], red[8];
    const int* idx = w.idx ? w.idx + (size_t)l * w.idx_pitch : nullptr;
    const float* Wl = w.W + (size_t)l * w.r * w.d;
    const float* Ul = w.U + (size_t)l * w.n_steps * n;
    for (int c = tid; c < w.d; c += 256) sPos[c] = (short)(idx ? -1 : c);
    __syncthreads();
    for (int k = tid; k < n; k += 256) {
        sRem[k] = w.n_steps > 0 ? w.removed[(size_t)l * n + k] : 0x7fffffff;
        if (idx) sPos[idx[k]] = (short)k;
    }
    if (w.Wt) {
        const float* Wtl = w.Wt + (size_t)l * w.wt_rows * w.rp;
        for (int k = warp; k < n; k += 8) {
            const int i = i0 + lane;
            sW[k * 33 + lane] = i < w.r ? Wtl[(size_t)k * w.rp + i] : 0.f;
            sO[k * 33 + lane] = i < w.r ? Wl[(size_t)i * w.d + (idx ? idx[k] : k)] : 0.f;
        }
    } else {
        for (int e = tid; e < 32 * n; e += 256) {
            const int i = e / n, k = e % n;
            const float v = i0 + i < w.r ? Wl[(size_t)(i0 + i) * w.d + k] : 0.f;
            sW[k * 33 + i] = v;
            sO[k * 33 + i] = v;
        }
    }
    __syncthreads();
    int t = 0;
    for (int q = 0; q < w.lv.count; ++q) {
        const int stop = w.lv.done[q];
        while (t < stop) {
            const int m_n = min(CHUNK, stop - t);
            if (tid < CHUNK) {
                s_piv[tid] = tid < m_n ? w.piv[(size_t)l * w.n_steps + t + tid] : 0;
                s_rs[tid] = tid < m_n ? w.rs[(size_t)l * w.n_steps + t + tid] : 0.0;
            }
            for (int s = warp; s < CHUNK; s += 8)
                for (int k = lane; k < n; k += 32) sU[k * 36 + s] = s < m_n ? Ul[(size_t)(t + s) * n + k] : 0.f;
            __syncthreads();
            for (int e = tid; e < CHUNK * CHUNK; e += 256) {
                const int m = e >> 5, s = e & 31;
                sT[m * CHUNK + s] = (double)sU[s_piv[m] * 36 + s];
            }
            __syncthreads();
            double c[CHUNK];                              // the fp32 values, widened
#pragma unroll
            for (int m = 0; m < CHUNK; ++m) {
                double acc[4] = {m < m_n ? (double)sW[s_piv[m] * 33 + lane] : 0.0, 0.0, 0.0, 0.0};
#pragma unroll
                for (int s = 0; s < m; ++s) acc[s & 3] = fma(-c[s], sT[m * CHUNK + s], acc[s & 3]);
                c[m] = (double)(float)(((acc[0] + acc[1]) + (acc[2] + acc[3])) * s_rs[m]);
            }
            float cf[CHUNK];
#pragma unroll
            for (int m = 0; m < CHUNK; ++m) cf[m] = (float)c[m];
            __syncthreads();                              // everyone has read the pivot rows
            for (int k = warp; k < n; k += 8) {
                const float4* u4 = reinterpret_cast<const float4*>(sU + k * 36);
                float v = sW[k * 33 + lane];
#pragma unroll
                for (int s = 0; s < CHUNK / 4; ++s) {
                    const float4 u = u4[s];
                    v = fmaf(-u.x, cf[4 * s], v);
                    v = fmaf(-u.y, cf[4 * s + 1], v);
                    v = fmaf(-u.z, cf[4 * s + 2], v);
                    v = fmaf(-u.w, cf[4 * s + 3], v);
                }
                sW[k * 33 + lane] = v;
            }
            t += m_n;
            __syncthreads();
        }
        // ---- level: rows i0 .. of the snapshot in original column order, removed columns exactly zero
        const int slot = w.lv.slot0 + q;
        float* out = w.W_snap + (((size_t)l * w.n_levels + slot) * w.r + i0) * w.d;
        for (int i = warp; i < 32 && i0 + i < w.r; i += 8)
            for (int c = lane; c < w.d; c += 32) {
                const int k = sPos[c];
                out[(size_t)i * w.d + c] = k >= 0 && sRem[k] >= t ? sW[k * 33 + i] : 0.f;
            }
        double part = 0.0;
        for (int k = warp; k < n; k += 8)
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
            for (int v = 0; v < 8; ++v) s += red[v];
            w.dw2[((size_t)l * w.lv.count + q) * gridDim.x + blockIdx.x] = s;
        }
        __syncthreads();
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
    return sizeof(float) * (size_t)(round_up_int(2 * n * 33, 4) + n * 36 + 2 * CHUNK * CHUNK + round_up_int(n, 4)) +
           sizeof(short) * (size_t)round_up_int(d, 2);
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
    w->U = c.take<float>((size_t)L * n0 * n0);
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
        s = n <= 64 ? launch_steps<1, 64, 1>(w, st) : n <= 128 ? launch_steps<4, 32, 1>(w, st) : launch_steps<8, 32, 2>(w, st);
        if (s != ZIPLM_OK) return s;
    }
    if (w.lv.count > 0) {
        PhaseScope ps(PH_LAZY_UPDATE_W, st);
        const size_t smem = weights_smem(n, w.d);
        ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_endgame_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_endgame_weights<<<dim3(slabs, w.L), 256, smem, st>>>(w);
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
