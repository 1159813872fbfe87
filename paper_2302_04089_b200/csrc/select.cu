// Budgeted choice of one database level per module (Sec. 3.2, "Finding the optimal sparsity
// configuration" and "Structured SPDY search"): given, for every module m and every level s of its
// database, the run time t[m][s] from the latency table and the prior p[m][s] = loss[m][s] /
// base_loss[m] (relative layer-wise squared error, 1 for a dropped module), and sensitivity
// coefficients c[m], find the levels that minimise sum_m c[m] p[m][s_m] subject to
// sum_m t[m][s_m] <= budget.  The search of the paper solves this problem once per candidate
// coefficient vector (1000 mutation steps), so the kernel solves K candidates per launch.
//
// Time is discretised into n_buckets units of budget / n_buckets, every option rounded UP, so a
// selection that fits in units also fits in real time.  A CTA runs a candidate's dynamic
// programme over modules with the two value rows f[0 .. n_buckets] in shared memory (float64):
//     f_{m+1}[b] = min over options s with u[m][s] <= b of  f_m[b - u[m][s]] + c[m] p[m][s]
// (ties: lowest s), stores the argmin per (module, b) in global scratch and walks it back from
// b = n_buckets.  All comparisons are on float64 sums formed in module order, which is what makes
// the chosen levels reproducible bit for bit.
//
// What bounds it: instruction issue (one addition and one comparison per option and bucket), so the
// programme evaluates only what can matter, without changing any value it returns:
//   * Buckets.  Row m is needed from lo[m] = n_buckets - (largest units of modules m, m + 1, ...)
//     on, because no walk back reaches below, and is constant from hi[m] = (largest units of
//     modules 0 .. m - 1) on, where every option fits; only lo .. hi is computed and reads beyond
//     hi are clamped to it.  With a budget of half the dense run time that is half of the buckets.
//   * Options.  f_m does not increase with b (a larger budget keeps every choice), so over a block
//     of buckets [b0, b1] option s costs at least f_m[b1 - u_s] + c_s, and the best option of any
//     bucket costs at most min_s f_m[b0 - u_s] + c_s.  Options whose lower bound lies above that
//     are skipped (rounding is monotone, so the bounds hold for the rounded sums too).  A warp takes
//     64 buckets: its lanes test one option each, then all lanes evaluate the 3 to 6 of (on the
//     paper's grid) 13 or 44 options that are left.  32 buckets leave fewer options but pay the
//     test twice as often, 128 leave twice as many.
#include <math.h>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace ziplm {
namespace {

constexpr int SEL_THREADS = 1024;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_BLK = 64;               // buckets a warp works on at a time
constexpr int SEL_MAX_OPT = 255;          // options per module (argmin stored in a byte)
constexpr int SEL_MAX_BUCKETS = 12000;    // two float64 rows of n_buckets + 1 fit shared memory
constexpr int SEL_MAX_MOD = 512;          // modules per search (coefficient vectors in shared memory)
constexpr int SEL_MAX_CLUSTER = 16;       // CTAs (steps at a time) of one search
constexpr int SEL_SMEM_MOD = 1024;        // up to here the per-module bounds are in shared memory
constexpr int SEL_SMEM_MAX = 227 * 1024 - 8192;      // dynamic shared memory a kernel here may use

// Everything a CTA keeps in shared memory is addressed as elements of this array, never through stored
// pointers: the compiler then knows the address space, and a load is one shared-memory instruction.
//   two value rows, each behind a guard entry of +inf (the value of a negative bucket);
//   the priors and units of every option, or of one module at a time where not all fit;
//   per-module bounds; argmins of the last modules in what is left.
extern __shared__ double sel_smem[];

__device__ __forceinline__ int* sel_ints() { return reinterpret_cast<int*>(sel_smem); }
__device__ __forceinline__ unsigned char* sel_bytes() { return reinterpret_cast<unsigned char*>(sel_smem); }

__host__ __device__ __forceinline__ int sel_pitch(int n_buckets) { return (n_buckets + 16) & ~15; }

// Where the parts are (bytes); the same arithmetic on host and device.
struct DpLayout {
    int rows, p, u, row_cost, bounds, argmin, total;
    bool resident, bounds_in_smem;
    __host__ __device__ DpLayout(int n_mod, int max_opt, int n_buckets) {
        rows = 2 * (n_buckets + 2) * (int)sizeof(double);
        rows = (rows + 15) & ~15;
        bounds_in_smem = n_mod <= SEL_SMEM_MOD;
        const int b = bounds_in_smem ? (3 * n_mod + 2) * (int)sizeof(int) : 0;
        const int costs = 2 * ((max_opt + 1) & ~1) * (int)sizeof(double2);
        const long long all = (long long)n_mod * max_opt;
        resident = rows + costs + b + all * (int)(sizeof(double) + sizeof(int)) <= SEL_SMEM_MAX;
        const int n = resident ? (int)all : 0;
        row_cost = rows;
        p = row_cost + costs;
        u = p + n * (int)sizeof(double);
        bounds = u + n * (int)sizeof(int);
        argmin = (bounds + b + 15) & ~15;
        total = SEL_SMEM_MAX;
    }
};

// What one CTA works with.
struct DpCta {
    const float* loss; const float* base_loss; const float* time; const int* n_opt;
    int n_mod, max_opt, n_buckets;
    double per_unit;
    int p, u, cost;                  // elements of sel_smem as double, int, double2
    int* lo; int* hi;                // [n_mod + 1] each: row m is computed on lo[m] .. hi[m]
    int* at;                         // [n_mod]: where bucket 0 of module m's argmins is in sel_bytes()
    int direct, fetched;             // modules >= direct keep them there, those >= fetched are copied there
    unsigned char* ch;               // [n_mod][sel_pitch] argmins (global)
    bool resident;                   // all modules' tables at once
};

// Prior and units of one option; raises *nonfinite for a NaN (a coefficient is checked when used).
__device__ __forceinline__ void dp_option(const DpCta& w, int m, int s, double* p, int* u, int* nonfinite) {
    const size_t at = (size_t)m * w.max_opt + s;
    *p = (double)w.loss[at] / (double)w.base_loss[m];
    const double t = ceil((double)w.time[at] * w.per_unit);
    // an option that cannot fit (or has a negative time) is never taken
    *u = (t >= 0.0 && t <= (double)w.n_buckets) ? (int)t : w.n_buckets + 1;
    if (t != t) *nonfinite = 1;
}

__device__ __forceinline__ int dp_units(const DpCta& w, int m, int s) {
    return w.resident ? sel_ints()[w.u + m * w.max_opt + s]
                      : (int)ceil((double)w.time[(size_t)m * w.max_opt + s] * w.per_unit);
}

__device__ __forceinline__ int dp_count(const DpCta& w, int m) { return min(max(w.n_opt[m], 0), w.max_opt); }

// Tables (when resident), bounds and places of a CTA; ends with a barrier.
__device__ void dp_setup(DpCta& w, const DpLayout& lay, int* nonfinite) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int m = tid >> 5; m < w.n_mod; m += SEL_WARPS) {
        const int no = dp_count(w, m);
        int most = 0;
        for (int s = lane; s < no; s += 32) {
            double p;
            int u;
            dp_option(w, m, s, &p, &u, nonfinite);
            if (w.resident) { sel_smem[w.p + m * w.max_opt + s] = p; sel_ints()[w.u + m * w.max_opt + s] = u; }
            if (u <= w.n_buckets) most = max(most, u);
        }
        most = __reduce_max_sync(0xffffffffu, most);
        if (lane == 0) w.hi[m + 1] = most;
    }
    __syncthreads();
    __shared__ int s_direct, s_fetched;
    if (tid == 0) {
        int lo = w.n_buckets, hi = 0;
        w.lo[w.n_mod] = lo;
        for (int m = w.n_mod - 1; m >= 0; --m) w.lo[m] = lo = max(0, lo - w.hi[m + 1]);
        w.hi[0] = 0;
        for (int m = 1; m <= w.n_mod; ++m) w.hi[m] = hi = min(w.n_buckets, hi + w.hi[m]);
        int m = w.n_mod - 1, used = lay.argmin;
        for (; m >= 0; --m) {
            const int first = min(w.lo[m + 1], w.hi[m + 1]), n = w.hi[m + 1] - first + 1;
            if (used + n > lay.total) break;
            w.at[m] = used - first;
            used += n;
        }
        s_direct = m + 1;
        for (used = 0; m >= 0; --m) {            // over the value rows, when these are done with
            const int first = min(w.lo[m + 1], w.hi[m + 1]) & ~15, n = (w.hi[m + 1] + 16 - first) & ~15;
            if (used + n > lay.rows) break;
            w.at[m] = used - first;
            used += n;
        }
        s_fetched = m + 1;
    }
    __syncthreads();
    w.direct = s_direct;
    w.fetched = s_fetched;
}

// The upper word of a float64 as an integer that does not decrease with the value.
__device__ __forceinline__ int value_order(double v) {
    const int i = __double2hiint(v);
    return i ^ ((i >> 31) & 0x7fffffff);
}

// One row of the programme, buckets [lo, hi], by the whole CTA; f0 and f1 are the rows' places in
// sel_smem, cost that of the module's (cost, units) pairs.  R: options a lane tests.
template <int R>
__device__ __forceinline__ void dp_row(int f0, int f1, int cost, int no, int lo, int hi, int hi_prev,
                                       unsigned char* ch, int at) {
    const int lane = threadIdx.x & 31;
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    const double2* table = reinterpret_cast<const double2*>(sel_smem) + cost;
    double c[R];
    int us[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int s = r * 32 + lane;
        // a lane without an option holds a NaN, which sorts behind every bound
        const double2 t = s < no ? table[s] : make_double2(__longlong_as_double(0x7ff8000000000000LL), 0.0);
        c[r] = t.x;
        us[r] = __double2loint(t.y);
    }
    for (int b0 = lo + (threadIdx.x >> 5) * SEL_BLK; b0 <= hi; b0 += SEL_WARPS * SEL_BLK) {
        const int b1 = min(b0 + SEL_BLK - 1, hi);
        int low[R];
        int bound = 0x7ff00000;                                   // +inf
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r > 0 && r * 32 >= no) break;
            const double up = sel_smem[f0 + max(min(b0 - us[r], hi_prev), -1)] + c[r];
            low[r] = value_order(sel_smem[f0 + max(min(b1 - us[r], hi_prev), -1)] + c[r]);
            if (up == up) bound = min(bound, value_order(up));
        }
        bound = __reduce_min_sync(0xffffffffu, bound);
        double best0 = inf, best1 = inf;
        int arg0 = 0, arg1 = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r > 0 && r * 32 >= no) break;
            unsigned left = __ballot_sync(0xffffffffu, low[r] <= bound);
            if (left) {       // the next option's pair is requested while this one is tested (1024 candidates: 751 -> 741 us)
                int s = r * 32 + __ffs(left) - 1;
                double2 t = table[s];
                for (;;) {
                    left &= left - 1;
                    const int q = left ? r * 32 + __ffs(left) - 1 : s;
                    const double2 x = table[q];
                    const int i = b0 + lane - __double2loint(t.y);
                    const double v0 = sel_smem[f0 + max(min(i, hi_prev), -1)] + t.x;
                    const double v1 = sel_smem[f0 + max(min(i + 32, hi_prev), -1)] + t.x;
                    if (v0 < best0) { best0 = v0; arg0 = s; }
                    if (v1 < best1) { best1 = v1; arg1 = s; }
                    if (!left) break;
                    s = q; t = x;
                }
            }
        }
        const int b = b0 + lane;
        if (b <= hi) sel_smem[f1 + b] = best0;
        if (b + 32 <= hi) sel_smem[f1 + b + 32] = best1;
        if (ch) {
            if (b <= hi) ch[b] = (unsigned char)arg0;
            if (b + 32 <= hi) ch[b + 32] = (unsigned char)arg1;
        } else {
            if (b <= hi) sel_bytes()[at + b] = (unsigned char)arg0;
            if (b + 32 <= hi) sel_bytes()[at + b + 32] = (unsigned char)arg1;
        }
    }
}

// (cost, units) pairs of module m into half m & 1 of the cost table, by the whole CTA.
__device__ __forceinline__ void dp_costs(const DpCta& w, int m, const float* coef, int* nonfinite) {
    const int no = dp_count(w, m);
    double2* table = reinterpret_cast<double2*>(sel_smem) + w.cost + (m & 1) * ((w.max_opt + 1) & ~1);
    // the last threads: where warps have unequal numbers of blocks, theirs have fewer
    for (int s = SEL_THREADS - 1 - (int)threadIdx.x; s < no; s += SEL_THREADS) {
        double p;
        int u;
        if (w.resident) {
            p = sel_smem[w.p + m * w.max_opt + s];
            u = sel_ints()[w.u + m * w.max_opt + s];
        } else {
            dp_option(w, m, s, &p, &u, nonfinite);
        }
        const double c = (double)coef[m] * p;
        if (c != c) *nonfinite = 1;
        table[s] = make_double2(c, __hiloint2double(0, u));
    }
}

// The dynamic programme and its walk back for one coefficient vector (global or shared memory), run
// by the whole CTA.  Returns the minimal cost (inf: nothing fits) in every thread; then sel[0 ..
// n_mod) (global) holds the chosen options.  *nonfinite is a shared flag that is raised when a cost
// is NaN.  Ends with a barrier.
template <int R>
__device__ double dp_solve(const DpCta& w, const float* coef, int* nonfinite, int* sel) {
    const int tid = threadIdx.x, lane = tid & 31, B = w.n_buckets, pitch = sel_pitch(B);
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    int f0 = 1, f1 = B + 3;
    if (tid == 0) {
        sel_smem[f0 - 1] = sel_smem[f1 - 1] = inf;
        sel_smem[f0] = 0.0;                      // row 0 is 0 everywhere: hi[0] = 0
    }
    dp_costs(w, 0, coef, nonfinite);
    __syncthreads();
    int hi = 0;
    for (int m = 0; m < w.n_mod; ++m) {
        const int next = w.hi[m + 1];
        if (m + 1 < w.n_mod) dp_costs(w, m + 1, coef, nonfinite);
        const bool direct = m >= w.direct;
        dp_row<R>(f0, f1, w.cost + (m & 1) * ((w.max_opt + 1) & ~1), dp_count(w, m), min(w.lo[m + 1], next), next,
                  hi, direct ? nullptr : w.ch + (size_t)m * pitch, direct ? w.at[m] : 0);
        __syncthreads();
        const int t = f0; f0 = f1; f1 = t;
        hi = next;
    }
    const double total = sel_smem[f0 + hi];
    __syncthreads();
    if (total < inf) {
        // the walk is a chain of one look-up per module: bring the argmins that are in global memory
        // over the value rows first, two warps a module
        for (int m = w.direct - 1 - (tid >> 6); m >= w.fetched; m -= SEL_THREADS / 64) {
            const int first = min(w.lo[m + 1], w.hi[m + 1]) & ~15, n = (w.hi[m + 1] + 16 - first) / 16;
            const uint4* src = reinterpret_cast<const uint4*>(w.ch + (size_t)m * pitch + first);
            uint4* dst = reinterpret_cast<uint4*>(sel_bytes() + w.at[m] + first);
#pragma unroll 4
            for (int e = tid & 63; e < n; e += 64) dst[e] = src[e];
        }
        __syncthreads();
        if (tid < 32) {
            int b = B;
            for (int m = w.n_mod - 1; m >= 0; --m) {
                const int i = min(b, w.hi[m + 1]);
                const int s = m >= w.fetched ? sel_bytes()[w.at[m] + i] : w.ch[(size_t)m * pitch + i];
                if (lane == 0) sel[m] = s;
                b -= dp_units(w, m, s);
            }
        }
    }
    __syncthreads();
    return total;
}

// Sum of row[m][sel[m]] over the modules, float64, in the order first, first + step, ...; warp 0 (the
// warp that wrote sel) calls it and every lane has the sum.
__device__ double dp_sum(const DpCta& w, const float* row, const int* sel, bool descending) {
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int k0 = 0; k0 < w.n_mod; k0 += 32) {
        const int k = k0 + lane, m = descending ? w.n_mod - 1 - k : k;
        const double v = k < w.n_mod ? (double)row[(size_t)m * w.max_opt + sel[m]] : 0.0;
        const int n = min(32, w.n_mod - k0);
        for (int j = 0; j < n; ++j) acc += __shfl_sync(0xffffffffu, v, j);
    }
    return acc;
}

__device__ __forceinline__ void dp_bind(DpCta& w, const DpLayout& lay, const float* loss, const float* base_loss,
                                        const float* time, const int* n_opt, int n_mod, int max_opt,
                                        int n_buckets, double per_unit, unsigned char* choice, int* bounds) {
    w.loss = loss; w.base_loss = base_loss; w.time = time; w.n_opt = n_opt;
    w.n_mod = n_mod; w.max_opt = max_opt; w.n_buckets = n_buckets; w.per_unit = per_unit;
    w.p = lay.p / (int)sizeof(double);
    w.u = lay.u / (int)sizeof(int);
    w.cost = lay.row_cost / (int)sizeof(double2);
    w.lo = lay.bounds_in_smem ? sel_ints() + lay.bounds / (int)sizeof(int)
                              : bounds + blockIdx.x * (3 * (size_t)n_mod + 2);
    w.hi = w.lo + n_mod + 1;
    w.at = w.hi + n_mod + 1;
    w.ch = choice + blockIdx.x * ((size_t)n_mod * sel_pitch(n_buckets));
    w.resident = lay.resident;
}

// One CTA per SM takes candidates blockIdx.x, blockIdx.x + gridDim.x, ...: the tables are formed once
// and the argmins of a CTA's candidates share one piece of scratch, which then stays in L2.
template <int R>
__global__ void __launch_bounds__(SEL_THREADS)
k_select_levels(const float* __restrict__ loss, const float* __restrict__ base_loss,
                const float* __restrict__ time, const int* __restrict__ n_opt, int n_mod, int max_opt,
                const float* __restrict__ coef, int K, double budget, int n_buckets, unsigned char* choice,
                int* bounds, int* selected, double* __restrict__ cost_out, double* __restrict__ time_out,
                int* __restrict__ status) {
    __shared__ int s_table_bad, s_nonfinite;
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    const DpLayout lay(n_mod, max_opt, n_buckets);
    DpCta w;
    dp_bind(w, lay, loss, base_loss, time, n_opt, n_mod, max_opt, n_buckets, (double)n_buckets / budget, choice,
            bounds);
    if (threadIdx.x == 0) s_table_bad = 0;
    __syncthreads();
    dp_setup(w, lay, &s_table_bad);
    for (int k = blockIdx.x; k < K; k += gridDim.x) {
        if (threadIdx.x == 0) s_nonfinite = s_table_bad;
        __syncthreads();
        int* sel = selected + (size_t)k * n_mod;
        const double total = dp_solve<R>(w, coef + (size_t)k * n_mod, &s_nonfinite, sel);
        if (threadIdx.x < 32) {
            const bool ok = !s_nonfinite && total < inf;      // no NaN came in, and the budget can be met
            const double tsum = ok ? dp_sum(w, time, sel, true) : 0.0;
            if (!ok)
                for (int m = threadIdx.x; m < n_mod; m += 32) sel[m] = -1;
            if (threadIdx.x == 0) {
                status[k] = ok ? (int)ZIPLM_OK : s_nonfinite ? (int)ZIPLM_ERR_NONFINITE : (int)ZIPLM_ERR_INVALID_ARG;
                cost_out[k] = ok ? total : inf;
                time_out[k] = tsum;
            }
        }
        __syncthreads();
    }
}

// The mutation search of "Structured SPDY search": starting from coef0, every step replaces the
// coefficients marked in mask[step] by values[step] (the caller draws both: a mark with
// probability 0.1 per coefficient gives the paper's "10 % in expectation"), solves the dynamic
// programme, scores the selection and keeps the mutated vector when the score is strictly lower.
// The score of a selection is sum_m objective[m][s_m]: a separable stand-in for the calibration
// loss of the stitched model, which only the caller's model can give.
//
// A step needs the vector that the steps before it left, but few steps are accepted (16 of 1000 on
// the paper's grid).  So a cluster of CTAs runs one search, every CTA the whole programme of another
// step, all from the current best vector: the first accepted step in step order counts, the ones
// behind it are evaluated again from the new vector, and the outcome is that of one step at a time.
template <int R>
__global__ void __launch_bounds__(SEL_THREADS)
k_search_levels(const float* __restrict__ loss, const float* __restrict__ base_loss,
                const float* __restrict__ time, const int* __restrict__ n_opt, int n_mod, int max_opt,
                const float* __restrict__ objective, const float* __restrict__ coef0,
                const double* __restrict__ budgets, int n_buckets, const unsigned char* __restrict__ mask,
                const float* __restrict__ values, int n_steps, unsigned char* choice, int* trial_sel,
                int* bounds, int* __restrict__ best_sel, float* __restrict__ best_coef,
                double* __restrict__ best_obj, int* __restrict__ n_accepted, int* __restrict__ status) {
    __shared__ float c_best[SEL_MAX_MOD], c_try[SEL_MAX_MOD];
    __shared__ int s_nonfinite;
    __shared__ double s_score[2][SEL_MAX_CLUSTER];       // scores of even and odd rounds (inf: nothing fits)
    __shared__ int s_bad[2][SEL_MAX_CLUSTER];            // whether a NaN came in
    cg::cluster_group cluster = cg::this_cluster();
    const int P = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int k = blockIdx.x / P, tid = threadIdx.x;
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    const DpLayout lay(n_mod, max_opt, n_buckets);
    DpCta w;
    dp_bind(w, lay, loss, base_loss, time, n_opt, n_mod, max_opt, n_buckets, (double)n_buckets / budgets[k], choice,
            bounds);
    int* trial = trial_sel + (size_t)blockIdx.x * n_mod;
    const unsigned char* mk = mask + (size_t)k * n_steps * n_mod;
    const float* val = values + (size_t)k * n_steps * n_mod;
    if (tid == 0) s_nonfinite = 0;
    for (int m = tid; m < n_mod; m += SEL_THREADS) c_best[m] = coef0[(size_t)k * n_mod + m];
    __syncthreads();
    dp_setup(w, lay, &s_nonfinite);
    const int table_bad = s_nonfinite;
    double best = inf;
    bool bad = false;
    int accepted = 0, round = 0;
    for (int step = 0; step <= n_steps; ++round) {         // step 0 scores coef0 itself
        const int mine = step + rank;
        if (mine <= n_steps) {
            for (int m = tid; m < n_mod; m += SEL_THREADS) {
                float c = c_best[m];
                if (mine > 0 && mk[(size_t)(mine - 1) * n_mod + m]) c = val[(size_t)(mine - 1) * n_mod + m];
                c_try[m] = c;
            }
            if (tid == 0) s_nonfinite = table_bad;
            __syncthreads();
            const double total = dp_solve<R>(w, c_try, &s_nonfinite, trial);
            if (tid < 32) {
                const double score = total < inf ? dp_sum(w, objective, trial, false) : inf;
                if (tid < P) {
                    cluster.map_shared_rank(&s_score[round & 1][0], tid)[rank] = score;
                    cluster.map_shared_rank(&s_bad[round & 1][0], tid)[rank] = s_nonfinite;
                }
            }
        }
        cluster.sync();
        // every CTA reads the same scores and comes to the same end of the round
        const int n = min(P, n_steps - step + 1);
        int winner = -1;
        for (int q = 0; q < n && winner < 0; ++q) {
            const double score = s_score[round & 1][q];
            if (s_bad[round & 1][q]) bad = true;
            if (!bad && score < best) { best = score; winner = q; }
        }
        if (winner >= 0) {
            const int at = step + winner;
            if (at > 0) {
                ++accepted;
                for (int m = tid; m < n_mod; m += SEL_THREADS)
                    if (mk[(size_t)(at - 1) * n_mod + m]) c_best[m] = val[(size_t)(at - 1) * n_mod + m];
            }
            if (rank == winner)
                for (int m = tid; m < n_mod; m += SEL_THREADS) best_sel[(size_t)k * n_mod + m] = trial[m];
            step = at + 1;
        } else {
            step += n;
        }
        __syncthreads();
        if (bad) break;                                    // nothing is accepted any more
    }
    cluster.sync();                                        // no CTA leaves while others may write to it
    const bool ok = best < inf;
    if (rank == 0) {
        for (int m = tid; m < n_mod; m += SEL_THREADS) {
            best_coef[(size_t)k * n_mod + m] = c_best[m];
            if (!ok) best_sel[(size_t)k * n_mod + m] = -1;
        }
        if (tid == 0) {
            best_obj[k] = best;
            n_accepted[k] = accepted;
            status[k] = bad ? (int)ZIPLM_ERR_NONFINITE : ok ? (int)ZIPLM_OK : (int)ZIPLM_ERR_INVALID_ARG;
        }
    }
}
// Pieces of scratch of a search call: a search runs on 16 CTAs at most, and on several only while
// there are SMs for all searches.
int search_slices(int S) { return S > 16 * SEL_MAX_CLUSTER ? S : S * SEL_MAX_CLUSTER < 256 ? S * SEL_MAX_CLUSTER : 256; }

// The kernels are instantiated for the options a lane holds: 32, 64 or 255 options per module.
template <typename F>
F by_options(int max_opt, F r1, F r2, F r8) { return max_opt <= 32 ? r1 : max_opt <= 64 ? r2 : r8; }

}  // namespace

size_t select_workspace_bytes(int K, int n_mod, int n_buckets) {
    return align_up((size_t)K * n_mod * (size_t)sel_pitch(n_buckets)) +
           align_up((size_t)K * (3 * (size_t)n_mod + 2) * sizeof(int));
}

ziplm_status run_select_levels(const float* loss, const float* base_loss, const float* time,
                               const int* n_opt, int n_mod, int max_opt, const float* coef, int K,
                               double budget, int n_buckets, int* selected, double* cost, double* time_sum,
                               int* status, void* ws, size_t ws_bytes, cudaStream_t st) {
    if (max_opt > SEL_MAX_OPT || n_buckets > SEL_MAX_BUCKETS) return ZIPLM_ERR_UNSUPPORTED;
    if (ws_bytes < select_workspace_bytes(K, n_mod, n_buckets)) return ZIPLM_ERR_WORKSPACE;
    Carver c(ws);
    unsigned char* choice = c.take<unsigned char>((size_t)K * n_mod * (size_t)sel_pitch(n_buckets));
    int* bounds = c.take<int>((size_t)K * (3 * (size_t)n_mod + 2));
    int dev = 0, sms = 0;
    ZIPLM_CHECK_CUDA(cudaGetDevice(&dev));
    ZIPLM_CHECK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = DpLayout(n_mod, max_opt, n_buckets).total;
    auto kernel = by_options(max_opt, k_select_levels<1>, k_select_levels<2>, k_select_levels<8>);
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kernel<<<K < sms ? K : sms, SEL_THREADS, smem, st>>>(loss, base_loss, time, n_opt, n_mod, max_opt, coef, K,
                                                         budget, n_buckets, choice, bounds, selected, cost,
                                                         time_sum, status);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

size_t search_workspace_bytes(int S, int n_mod, int n_buckets) {
    const size_t n = (size_t)search_slices(S);
    return align_up(n * n_mod * (size_t)sel_pitch(n_buckets)) + align_up(n * n_mod * sizeof(int)) +
           align_up(n * (3 * (size_t)n_mod + 2) * sizeof(int));
}

ziplm_status run_search_levels(const float* loss, const float* base_loss, const float* time,
                               const int* n_opt, int n_mod, int max_opt, const float* objective,
                               const float* coef0, const double* budgets, int S, int n_buckets,
                               const unsigned char* mask, const float* values, int n_steps, int* best_sel,
                               float* best_coef, double* best_obj, int* n_accepted, int* status, void* ws,
                               size_t ws_bytes, cudaStream_t st) {
    if (max_opt > SEL_MAX_OPT || n_buckets > SEL_MAX_BUCKETS || n_mod > SEL_MAX_MOD) return ZIPLM_ERR_UNSUPPORTED;
    if (ws_bytes < search_workspace_bytes(S, n_mod, n_buckets)) return ZIPLM_ERR_WORKSPACE;
    const int slices = search_slices(S);
    Carver c(ws);
    unsigned char* choice = c.take<unsigned char>((size_t)slices * n_mod * (size_t)sel_pitch(n_buckets));
    int* trial = c.take<int>((size_t)slices * n_mod);
    int* bounds = c.take<int>((size_t)slices * (3 * (size_t)n_mod + 2));
    const size_t smem = DpLayout(n_mod, max_opt, n_buckets).total;
    auto kernel = by_options(max_opt, k_search_levels<1>, k_search_levels<2>, k_search_levels<8>);
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(SEL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // the largest cluster with which all searches still run at once
    int P = SEL_MAX_CLUSTER;
    for (; P > 1; P /= 2) {
        if ((long long)S * P > slices || P > n_steps + 1) continue;
        int most = 0;
        attr[0].val.clusterDim.x = P;
        cfg.gridDim = dim3(S * P);
        if (cudaOccupancyMaxActiveClusters(&most, kernel, &cfg) == cudaSuccess && most >= S) break;
        (void)cudaGetLastError();
    }
    attr[0].val.clusterDim.x = P;
    cfg.gridDim = dim3(S * P);
    ZIPLM_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kernel, loss, base_loss, time, n_opt, n_mod, max_opt, objective,
                                        coef0, budgets, n_buckets, mask, values, n_steps, choice, trial, bounds,
                                        best_sel, best_coef, best_obj, n_accepted, status));
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace ziplm
