// Model reshaping (Sec. 3.1, "Pruned structures"): once the columns of removed structures are
// zero, they are dropped from this matrix and the matching rows are dropped from the previous
// layer (FC1 rows and bias for neurons; the Q, K, V rows of a head) without any output change.
//
//   k_kept_structures   order[l][0 .. G-level) -> ascending list of the `level` survivors
//   k_gather_columns    out[l][i][k*g + c] = M[l][i][kept[l][k]*g + c]
//   k_gather_rows       out[l][k*g + c][:] = M[l][kept[l][k]*g + c][:]
//
// All three only move data: results are bit-exact.
//
// A level is three launches of 5 to 25 us, so they are programmatic dependent launches: a kernel lets the next one
// start once all of its own CTAs run, and the next one's CTAs take the SMs that the last ones leave and wait there for
// its end (griddepcontrol.wait, by every thread before it reads or writes anything; loads are coherent ones, which
// nothing moves in front of it).  Eleven levels of 12 x 768 x 3072, 33 launches: 634 -> 561 us.
#include "common.cuh"
#include "tc_common.cuh"

namespace ziplm {
namespace {

constexpr int KEEP_THREADS = 1024;

// One CTA per layer.  The removed structures are marked in a bitmap in shared memory; every thread then
// owns whole words of it, counts their survivors, a scan over the threads (within the warps by shuffles,
// then over the warps' totals) gives its first output slot, and the words are written in order.
// bad[l] is ZIPLM_ERR_INVALID_ARG when order[l][0 .. G-level) is not a list of distinct indices in [0, G),
// else 0.
__global__ void __launch_bounds__(KEEP_THREADS) k_kept_structures(const int* __restrict__ order, int G,
                                                                  int level, int* __restrict__ kept,
                                                                  int* __restrict__ bad) {
    extern __shared__ unsigned int bits[];                    // ceil(G / 32) words
    __shared__ int warp_sum[KEEP_THREADS / 32];
    __shared__ int fail;
    const int words = (G + 31) / 32;
    const int l = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int* ord = order + (size_t)l * G;
    tc::grid_trigger();
    tc::grid_wait();
    if (tid == 0) fail = 0;
    for (int w = tid; w < words; w += KEEP_THREADS)
        bits[w] = (w + 1) * 32 <= G ? 0u : ~0u << (G & 31);   // what lies past G counts as removed
    __syncthreads();
    const int n_removed = G - level;
    for (int t = tid; t < n_removed; t += KEEP_THREADS) {
        const int s = __ldca(ord + t);
        if (s < 0 || s >= G) {
            fail = 1;
        } else {
            const unsigned int m = 1u << (s & 31);
            if (atomicOr(&bits[s >> 5], m) & m) fail = 1;     // listed twice
        }
    }
    __syncthreads();
    const int chunk = (words + KEEP_THREADS - 1) / KEEP_THREADS;
    const int lo = tid * chunk, hi = min(lo + chunk, words);
    int cnt = 0;
    for (int w = lo; w < hi; ++w) cnt += __popc(~bits[w]);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int before = lane < warp ? warp_sum[lane] : 0;
    before = __reduce_add_sync(0xffffffffu, before);
    int pos = before + incl - cnt;
    if (tid == KEEP_THREADS - 1 && before + incl != level) fail = 1;
    __syncthreads();
    if (tid == 0) bad[l] = fail ? (int)ZIPLM_ERR_INVALID_ARG : 0;
    if (fail) return;
    int* out = kept + (size_t)l * level;
    for (int w = lo; w < hi; ++w)
        for (unsigned int left = ~bits[w]; left; left &= left - 1) out[pos++] = 32 * w + __ffs(left) - 1;
}

// Columns: a thread keeps its source columns for 16 rows and has the reads of eight rows in flight; VEC
// neighbouring columns of the output are one store.  Bound by memory: a sparse gather reads whole 32-byte
// sectors of the source row, so a level that keeps a twelfth of the columns still reads half of it.
constexpr int COL_ROWS = 16;
template <int VEC>
__global__ void __launch_bounds__(256) k_gather_columns(const float* __restrict__ M, long long ld,
                                                        long long layer_stride,
                                                        const int* __restrict__ kept, int rows, int G,
                                                        int g, int level, float* __restrict__ out) {
    const int l = blockIdx.z;
    const int n_out = level * g;
    const int j = (blockIdx.x * 256 + threadIdx.x) * VEC;
    tc::grid_trigger();
    tc::grid_wait();
    if (j >= n_out) return;
    int src[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        const int s = __ldca(kept + (size_t)l * level + (j + e) / g);
        src[e] = (unsigned)s < (unsigned)G ? s * g + (j + e) % g : -1;      // an index outside [0, G) gives zeros
    }
    const int i0 = blockIdx.y * COL_ROWS;
    const float* Ml = M + (size_t)l * (size_t)layer_stride + (size_t)i0 * (size_t)ld;
    float* Ol = out + (size_t)l * rows * n_out + (size_t)i0 * n_out + j;
    const int n = min(COL_ROWS, rows - i0);
#pragma unroll
    for (int h = 0; h < COL_ROWS; h += 8) {
        float v[8][VEC];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                v[i][e] = h + i < n && src[e] >= 0 ? __ldca(Ml + (size_t)(h + i) * (size_t)ld + src[e]) : 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (h + i >= n) break;
            float* o = Ol + (size_t)(h + i) * n_out;
            if (VEC == 4) __stcs(reinterpret_cast<float4*>(o), make_float4(v[i][0], v[i][1], v[i][2], v[i][3]));
            else if (VEC == 2) __stcs(reinterpret_cast<float2*>(o), make_float2(v[i][0], v[i][1]));
            else __stcs(o, v[i][0]);
        }
    }
}

// Rows: a warp copies a row, eight 16-byte (or 4-byte) pieces per lane in flight.
template <typename V>
__global__ void __launch_bounds__(256) k_gather_rows(const float* __restrict__ M, long long ld,
                                                     long long layer_stride,
                                                     const int* __restrict__ kept, int cols, int G,
                                                     int g, int level, float* __restrict__ out) {
    constexpr int N = sizeof(V) / sizeof(float);
    const int l = blockIdx.y, lane = threadIdx.x & 31;
    const int k = blockIdx.x * 8 + (threadIdx.x >> 5);         // output row
    tc::grid_trigger();
    tc::grid_wait();
    if (k >= level * g) return;
    const int s = __ldca(kept + (size_t)l * level + k / g);
    const bool ok = (unsigned)s < (unsigned)G;                 // an index outside [0, G) gives zeros
    const V* row = reinterpret_cast<const V*>(M + (size_t)l * (size_t)layer_stride +
                                              (size_t)(ok ? s * g + k % g : 0) * (size_t)ld);
    V* dst = reinterpret_cast<V*>(out + ((size_t)l * level * g + k) * (size_t)cols);
    const int n = cols / N;
    for (int c0 = lane; c0 < n; c0 += 256) {
        V v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = ok && c0 + 32 * e < n ? __ldca(row + c0 + 32 * e) : V();
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (c0 + 32 * e < n) __stcs(dst + c0 + 32 * e, v[e]);
    }
}

}  // namespace

ziplm_status run_kept_structures(const int* order, int L, int G, int level, int* kept, int* bad,
                                 cudaStream_t st) {
    const size_t smem = (size_t)(G + 31) / 32 * 4;
    if (smem > 200 * 1024) return ZIPLM_ERR_UNSUPPORTED;
    if (smem > 48 * 1024)
        ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_kept_structures, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)smem));
    return launch_dependent(k_kept_structures, dim3(L), KEEP_THREADS, smem, st, order, G, level, kept, bad);
}

ziplm_status run_gather_columns(const float* M, long long ld, long long layer_stride, const int* kept,
                                int L, int rows, int G, int g, int level, float* out, cudaStream_t st) {
    if (level == 0 || rows == 0) return ZIPLM_OK;
    const int n_out = level * g;
    for (int l0 = 0; l0 < L; l0 += 65535) {
        const int ln = (L - l0 < 65535) ? (L - l0) : 65535;
        // stores of two or four columns where they stay aligned and leave enough threads
        const long long threads = (long long)n_out * ((rows + COL_ROWS - 1) / COL_ROWS) * ln;
        const bool al = reinterpret_cast<uintptr_t>(out) % 16 == 0;
        const int vec = al && n_out % 4 == 0 && threads >= 4ll * kSMs * 1024 ? 4
                        : al && n_out % 2 == 0 && threads >= 2ll * kSMs * 1024 ? 2 : 1;
        auto kernel = vec == 4 ? k_gather_columns<4> : vec == 2 ? k_gather_columns<2> : k_gather_columns<1>;
        const dim3 grid((unsigned)((n_out + 256 * vec - 1) / (256 * vec)), (unsigned)((rows + COL_ROWS - 1) / COL_ROWS),
                        (unsigned)ln);
        if (grid.y > 65535) return ZIPLM_ERR_UNSUPPORTED;
        const ziplm_status s = launch_dependent(kernel, grid, 256, 0, st, M + (size_t)l0 * (size_t)layer_stride, ld,
                                                layer_stride, kept + (size_t)l0 * level, rows, G, g, level,
                                                out + (size_t)l0 * rows * n_out);
        if (s != ZIPLM_OK) return s;
    }
    return ZIPLM_OK;
}

ziplm_status run_gather_rows(const float* M, long long ld, long long layer_stride, const int* kept,
                             int L, int cols, int G, int g, int level, float* out, cudaStream_t st) {
    if (level == 0 || cols == 0) return ZIPLM_OK;
    for (int l0 = 0; l0 < L; l0 += 65535) {
        const int ln = (L - l0 < 65535) ? (L - l0) : 65535;
        const bool quads = cols % 4 == 0 && ld % 4 == 0 && layer_stride % 4 == 0 &&
                           (reinterpret_cast<uintptr_t>(M) | reinterpret_cast<uintptr_t>(out)) % 16 == 0;
        auto kernel = quads ? k_gather_rows<float4> : k_gather_rows<float>;
        const ziplm_status s = launch_dependent(kernel, dim3((unsigned)((level * g + 7) / 8), (unsigned)ln), 256, 0, st,
                                                M + (size_t)l0 * (size_t)layer_stride, ld, layer_stride,
                                                kept + (size_t)l0 * level, cols, G, g, level,
                                                out + (size_t)l0 * level * g * (size_t)cols);
        if (s != ZIPLM_OK) return s;
    }
    return ZIPLM_OK;
}

}  // namespace ziplm
