// Rank-32 or rank-64 update of H^-1, of the Gram matrix Q = W^T W and of W^T itself (delayed Eq. 4 / Eq. 3)
// for the blocks that leave the removed positions in place, on the 5th-generation tensor cores,
// as one persistent kernel:
//
//   A'[i,j] = A[i,j] - sum_s U[s,i] U[s,j]
//   Q'[i,j] = Q[i,j] - sum_s (Z[s,i] U[s,j] + U[s,i] Z[s,j]),       i > j positions of the arrays
//   Wt'[i,c] = Wt[i,c] - sum_s U[s,i] C[s,c],                         c row indices of W
//
// (the tiles of W^T follow the tiles of their row strip: the same packed rows of U, the packed C
// in the place of the column operand, one accumulator, no mirrored store)
// (the pending vectors are zero at removed positions, whose rows and columns are carried along
// unchanged).  Nothing is gathered: tiles are plain rectangles, read by TMA and written densely.
// The steps kernel leaves the pending vectors K-major ([position][step], lazy_common.cuh), each
// value split into three bfloat16 parts x = x1 + x2 + x3 (every part the nearest bfloat16 of what
// the earlier ones left, so |x - x1 - x2 - x3| <= 2^-27 |x|).  Products of two bfloat16 values are
// exact in the fp32 accumulator, and the six partial products x_a y_b with a + b <= 4 are kept
// (the others are below 2^-26 of the product), so a product is as good as an fp32 one.
//
// Two groups of 32 steps: the operands of a group at a time fill their shared memory, each group has an
// accumulator of its own and the two are joined in fp32 (one chain of both would truncate more).  12 x 3072 with two
// groups 487 us on two thirds of the SMs, where one group took 365: the MMAs of a tile's groups follow one another, each
// behind its operands (545 us with slices of 16 columns, 515 with 32, whole lines of 128 bytes; the rest is operands
// requested array by array and descriptors a tile ahead).  Rows of both groups kept in shared memory beside a ring of
// narrower slices: 547 us; old entries read into registers from the other side of the diagonal, with operands of both
// groups in shared memory: 740 us (loads queue behind the stores).
//
// The update kernel runs one CTA on each of two thirds of the SMs.  Work is cut into tiles of
// 128 x 128 entries on or below the diagonal; runs of consecutive tiles of one row strip
// ("segments") are handed out through an atomic counter, so a CTA that starts late (another kernel
// holds its SM) simply finds less left to do.  Inside a CTA three kinds of warps work as a pipeline,
// linked by mbarriers only:
//   warp 0      one thread fetches segments, publishes one descriptor per tile (layer, tile origin), a tile
//               ahead, and loads the tile's packed operands by TMA (rows that are there already stay).  One thread
//               throughout: as a whole warp whose lane 0 issued the copies, the other lanes ran ahead of it into the
//               next tile, and lane 0 met their values;
//   warp 1      one thread issues the 36 tcgen05.mma (kind::f16, bfloat16, M = N = 128, K = 16)
//               of a tile and group (12 for a tile of W^T), the smallest partial products first, so that the truncating
//               accumulation meets them while the accumulator is small, into one of two
//               accumulator regions in tensor memory;
//   warps 2-17  each owns 32 rows x 64 columns of one matrix (H^-1 or Q) in every tile, worked
//               on as two slices of 32 columns: one lane brings the old entries of a slice in
//               by TMA (128-byte swizzle) into a ring of two slices of the warp's own, a tile ahead, the warp
//               reads the accumulators with tcgen05.ld (one row per lane), subtracts, stores the mirrored
//               entries [j][i] straight from registers (lanes run along i: 128-byte pieces) and the entries
//               [i][j] after a pass through its slice (eight lanes along a row: 128-byte pieces).
// No CTA-wide barrier exists between set-up and exit.  Every mbarrier wait is bounded; a wait that
// runs out raises an abort flag that all roles poll, the issuer still commits and waits for the
// MMAs it has issued, every lane that started copies waits for them, and the CTA leaves through
// the normal exit (tensor memory freed) with ZIPLM_ERR_TIMEOUT in the layers' status.
#include <cuda_bf16.h>

#include "common.cuh"
#include "lazy_common.cuh"
#include "tc_common.cuh"

namespace ziplm {
namespace {
using namespace tc;

constexpr int PK = kPackSteps;
constexpr int RM = 128, CN = 128;            // tile rows, tile columns (new index space)
constexpr int NARR = kPackArrays;            // packed arrays: [U1|U2], [U3|Z3], [Z1|Z2], 128-byte rows
constexpr int BOX_ROWS = 64;                 // rows per TMA box
constexpr int BOX_BYTES = BOX_ROWS * 128;    // 8 KiB
constexpr int ARR_BYTES = 2 * BOX_BYTES;     // one packed array, 128 positions
constexpr int ROWS_BYTES = NARR * ARR_BYTES; // 48 KiB
constexpr int COLS_BYTES = NARR * ARR_BYTES; // 48 KiB
constexpr int ACC_STAGES = 2;                // accumulator regions: the groups of the tiles in turn
constexpr int N_EPI = 16;                    // epilogue warps: 4 lane quarters x 2 matrices x 2 column halves
constexpr int SUBS = 2;                      // slices of 32 columns per warp and tile
constexpr int RING = 2;                      // slices per epilogue warp
constexpr int SLICE_FLOATS = 32 * 32;        // 32 rows x 32 columns
constexpr int RING_BYTES = N_EPI * RING * SLICE_FLOATS * 4;   // 128 KiB
constexpr int AQ_SMEM = ROWS_BYTES + COLS_BYTES + RING_BYTES + 1024;
constexpr int AQ_THREADS = 32 * (2 + N_EPI);
constexpr uint32_t AQ_TMEM_COLS = 512;       // two stages of (H^-1: 128 columns, Q: 128 columns)
constexpr int DESC_RING = 4;
constexpr int MAX_STRIPS = 48;               // d <= 6144
enum { TILE_STOP = 1, TILE_W = 2 };

// Work list of one launch: the row strips from the longest to the shortest; prefix[k] = number
// of segments (over all layers) of the k longest strips.
struct AqSched {
    int n_strips, seg, n_segments, L;
    int groups;               // groups of 32 pending steps
    int n_wt;                 // tiles of 128 columns of W^T that follow the tiles of a row strip
    int rows_pad;             // first row of the packed C in P
    int prefix[MAX_STRIPS + 1];
};

struct __align__(16) TileSlot {
    int l, i0, j0, flags;
};

__global__ void __launch_bounds__(AQ_THREADS, 1)
k_lazy_update_aq_tc(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap map_a,
                    const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_w,
                    const __grid_constant__ AqSched sch, int n_pos, int d, int rp,
                    float* __restrict__ A2, float* __restrict__ Q2, float* __restrict__ W2,
                    int* __restrict__ counter, int* __restrict__ layer_status, uint32_t slot_spin_limit) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_tile_full[DESC_RING], bar_tile_empty[DESC_RING];
    __shared__ uint64_t bar_ops_full[NARR], bar_ops_free[NARR], bar_acc_full[ACC_STAGES], bar_acc_empty[ACC_STAGES], bar_final;
    __shared__ uint64_t bar_slice[N_EPI][RING];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ TileSlot slots[DESC_RING];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t ops = (raw + 1023u) & ~1023u;          // swizzled tiles need 1024-byte alignment
    const uint32_t rows_smem = ops, cols_smem = ops + ROWS_BYTES;
    const uint32_t rings_smem = cols_smem + COLS_BYTES;
    float* rings_ptr = reinterpret_cast<float*>(smem_raw + (rings_smem - raw));

    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int i = 0; i < DESC_RING; ++i) {
            mbar_init(smem_u32(&bar_tile_full[i]), 1);
            mbar_init(smem_u32(&bar_tile_empty[i]), 1 + N_EPI);
        }
        for (int a = 0; a < NARR; ++a) {
            mbar_init(smem_u32(&bar_ops_full[a]), 1);
            mbar_init(smem_u32(&bar_ops_free[a]), 1);
        }
        for (int i = 0; i < ACC_STAGES; ++i) {
            mbar_init(smem_u32(&bar_acc_full[i]), 1);
            mbar_init(smem_u32(&bar_acc_empty[i]), N_EPI);
        }
        mbar_init(smem_u32(&bar_final), 1);
        for (int i = 0; i < N_EPI * RING; ++i) mbar_init(smem_u32(&bar_slice[0][0]) + 8u * i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_slot)), "r"(AQ_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    bool failed = false;

    if (warp == 0) {
        // ---------------- scheduler and TMA producer (one thread) ----------------
        if (lane == 0) {
            int published = 0;               // descriptors so far
            int issued = 0;                  // groups whose copies were issued
            int copies[NARR] = {0, 0, 0};    // ... by packed array, the one under way counted
            auto publish = [&](int l, int i0, int j0, int flags) {
                const int slot = published & (DESC_RING - 1);
                if (published >= DESC_RING &&
                    !mbar_wait_limit(smem_u32(&bar_tile_empty[slot]), (uint32_t)(((published >> 2) - 1) & 1), abortp,
                                     slot_spin_limit))
                    return false;
                TileSlot& ts = slots[slot];
                ts.l = l; ts.i0 = i0; ts.j0 = j0; ts.flags = flags;
                mbar_arrive(smem_u32(&bar_tile_full[slot]));
                ++published;
                return true;
            };
            // The operands of a tile, group after group, an array as soon as the MMAs of the group before are done
            // with it.  Rows that are there already stay; the order of two groups alternates from tile to tile.
            int rows_l = -1, rows_i0 = -1, rows_g = -1;      // the rows in shared memory
            auto load = [&](int t, int l, int i0, int j0) {
                for (int k2 = 0; k2 < sch.groups; ++k2) {
                    const int g = sch.groups > 1 ? k2 ^ (t & 1) : 0;
                    const bool rows = l != rows_l || i0 != rows_i0 || g != rows_g;
                    rows_l = l; rows_i0 = i0; rows_g = g;
                    for (int k = 0; k < NARR; ++k) {
                        const int a = k + 1 < NARR ? k + 1 : 0;         // 1, 2, 0: the order in which they are done with
                        if (issued > 0 && !mbar_wait(smem_u32(&bar_ops_free[a]), (uint32_t)((issued - 1) & 1), abortp))
                            return false;
                        const uint32_t full = smem_u32(&bar_ops_full[a]);
                        const uint32_t to_rows = rows_smem + (uint32_t)(a * ARR_BYTES), to_cols = cols_smem + (uint32_t)(a * ARR_BYTES);
                        mbar_expect_tx(full, (uint32_t)((rows ? 2 : 1) * ARR_BYTES));
                        ++copies[a];
                        for (int b = 0; b < 2; ++b) {
                            if (rows) tma_load_4d(to_rows + b * BOX_BYTES, &map, full, 0, i0 + b * BOX_ROWS, g * NARR + a, l);
                            tma_load_4d(to_cols + b * BOX_BYTES, &map, full, 0, j0 + b * BOX_ROWS, g * NARR + a, l);
                        }
                    }
                    ++issued;
                }
                return true;
            };
            // descriptors run a tile ahead of the operands, so that nobody waits for one
            int t = 0, pl = 0, pi0 = 0, pj0 = 0;           // tile t: published, its operands are next
            bool pending = false;
            int s = atomicAdd(counter, 1);
            while (s < sch.n_segments && !failed) {
                const int s_next = atomicAdd(counter, 1);   // in flight while this segment is set up
                int k = 0;
                while (k + 1 < sch.n_strips && sch.prefix[k + 1] <= s) ++k;
                const int I = sch.n_strips - 1 - k;
                const int within = s - sch.prefix[k];
                const int segs_strip = (sch.prefix[k + 1] - sch.prefix[k]) / sch.L;
                const int l = within / segs_strip, sidx = within - l * segs_strip;
                const int nJ = I + 1 + sch.n_wt;      // tiles J = 0 .. I (the last one holds the diagonal), then W^T
                const int Jb = sidx * sch.seg, Je = min(Jb + sch.seg, nJ);
                const int i0 = I * RM;
                for (int J = Jb; J < Je; ++J) {
                    // a tile of W^T takes its column operand from the rows of P that hold C
                    const bool wtile = J > I;
                    const int j0 = wtile ? sch.rows_pad + (J - I - 1) * CN : J * CN;
                    if (!publish(l, i0, j0, wtile ? TILE_W : 0) || (pending && !load(t, pl, pi0, pj0))) { failed = true; break; }
                    t += pending;
                    pl = l; pi0 = i0; pj0 = j0;
                    pending = true;
                }
                s = s_next;
            }
            if (!failed) failed = !publish(0, 0, 0, TILE_STOP) || (pending && !load(t, pl, pi0, pj0));
            if (failed) abort_flag = 1;
            // The copies land in this CTA's shared memory before it leaves, also where another role gives up and
            // the issuer no longer waits for them.
            for (int a = 0; a < NARR; ++a)
                if (copies[a] > 0) mbar_wait_quiet(smem_u32(&bar_ops_full[a]), (uint32_t)((copies[a] - 1) & 1));
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer (one thread) ----------------
        if (lane == 0) {
            constexpr uint32_t idesc = make_idesc(1u, RM, CN);     // bfloat16 operands, fp32 accumulate
            // descriptor of part p of the rows (r) and of the columns (c): U1 U2 U3 Z1 Z2 Z3
            const uint32_t part_off[6] = {0u, 64u, (uint32_t)ARR_BYTES, 2u * ARR_BYTES, 2u * ARR_BYTES + 64u,
                                          (uint32_t)ARR_BYTES + 64u};
            uint64_t r[6], c[6];
#pragma unroll
            for (int p = 0; p < 6; ++p) {
                r[p] = make_desc(rows_smem + (part_off[p] & ~127u)) + (uint64_t)((part_off[p] & 127u) >> 4);
                c[p] = make_desc(cols_smem + (part_off[p] & ~127u)) + (uint64_t)((part_off[p] & 127u) >> 4);
            }
            enum { U1 = 0, U2 = 1, U3 = 2, Z1 = 3, Z2 = 4, Z3 = 5 };
            int unit = 0;                // groups of 32 steps so far
            for (int t = 0;; ++t) {
                const int slot = t & (DESC_RING - 1);
                if (!mbar_wait(smem_u32(&bar_tile_full[slot]), (uint32_t)((t >> 2) & 1), abortp)) { failed = true; break; }
                const int flags = *reinterpret_cast<volatile int*>(&slots[slot].flags);
                mbar_arrive(smem_u32(&bar_tile_empty[slot]));
                if (flags & TILE_STOP) break;
                for (int g = 0; g < sch.groups; ++g, ++unit) {
                    const int st = unit & 1;
                    for (int a = 0; a < NARR && !failed; ++a)
                        if (!mbar_wait(smem_u32(&bar_ops_full[a]), (uint32_t)(unit & 1), abortp)) failed = true;
                    if (failed) break;
                    if (unit >= ACC_STAGES &&
                        !mbar_wait(smem_u32(&bar_acc_empty[st]), (uint32_t)(((unit >> 1) - 1) & 1), abortp)) {
                        failed = true;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t t_a = tmem_base + (uint32_t)(st * 2 * CN), t_q = t_a + (uint32_t)CN;
                    // one partial product x_a y_b over the 32 steps: two MMAs of K = 16 (32 bytes each)
                    auto prod = [&](uint32_t acc, int pr, int pc2, bool first) {
                        umma_bf16(acc, r[pr], c[pc2], idesc, first ? 0u : 1u);
                        umma_bf16(acc, r[pr] + 2u, c[pc2] + 2u, idesc, 1u);
                    };
                    // H^-1: U U^T, Q: Z U^T + U Z^T (a tile of W^T has no second matrix: its column operand is C
                    // in the place of U, and the products of the first are the whole update U^T C); smallest terms
                    // first, and arranged so that the arrays with the third parts and with Z are done with early
                    const bool w = flags & TILE_W;
                    prod(t_a, U1, U3, true);  prod(t_a, U3, U1, false);
                    if (!w) {
                        prod(t_q, Z1, U3, true);  prod(t_q, Z3, U1, false);
                        prod(t_q, U1, Z3, false); prod(t_q, U3, Z1, false);
                    }
                    umma_commit(smem_u32(&bar_ops_free[1]));
                    if (!w) {
                        prod(t_q, Z2, U2, false); prod(t_q, U2, Z2, false);
                        prod(t_q, Z1, U2, false); prod(t_q, Z2, U1, false); prod(t_q, U1, Z2, false);
                        prod(t_q, U2, Z1, false); prod(t_q, Z1, U1, false); prod(t_q, U1, Z1, false);
                    }
                    umma_commit(smem_u32(&bar_ops_free[2]));
                    prod(t_a, U2, U2, false);
                    prod(t_a, U1, U2, false); prod(t_a, U2, U1, false); prod(t_a, U1, U1, false);
                    umma_commit(smem_u32(&bar_ops_free[0]));
                    umma_commit(smem_u32(&bar_acc_full[st]));
                }
                if (failed) break;
            }
            if (failed) abort_flag = 1;
            // whatever was issued has completed before tensor memory is given back
            umma_commit(smem_u32(&bar_final));
            mbar_wait_quiet(smem_u32(&bar_final), 0u);
        }
        __syncwarp();
    } else {
        // ---------------- epilogue warps ----------------
        // warp -> TMEM lane quarter q (rows 32 q ..), matrix, column half h (columns 64 h ..)
        const int ew = warp - 2, q = warp & 3, mat = ew >> 3, h = (ew >> 2) & 1;
        const CUtensorMap* min_map = mat ? &map_q : &map_a;
        float* Mout = mat ? Q2 : A2;
        float* ring = rings_ptr + (size_t)ew * RING * SLICE_FLOATS;
        const uint32_t ring_u32 = rings_smem + (uint32_t)(ew * RING * SLICE_FLOATS * 4);
        const uint32_t bar0 = smem_u32(&bar_slice[ew][0]);
        const uint32_t lane_taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(mat * CN + 64 * h);
        const size_t dd = (size_t)d * d;
        // A slice is [32 rows][32 columns] as TMA writes it with the 128-byte swizzle: 128-byte rows,
        // the 16-byte unit index of row r XORed with r & 7: a lane per row and eight lanes
        // per row both reach it without bank conflicts.

        // Copy cursor: tile pt (descriptor in its ring slot), next slice psub.  One call starts
        // the copy of one slice (lane 0: expect_tx + TMA; the slice's earlier readers and writers,
        // this warp, are done and have fenced their accesses against the asynchronous proxy);
        // after the last slice of a tile the slot is given back and the next descriptor awaited.
        int pt = 0, psub = 0, pflags = TILE_STOP;
        int nl = 0, ni0 = 0, nj0 = 0;                        // tile pt
        int issued = 0;                                      // slices whose copies were started
        auto open_tile = [&]() -> bool {
            const int slot = pt & (DESC_RING - 1);
            // (the limit is for what the pipeline leaves behind, not for the kernel's first descriptor)
            const bool ok = __all_sync(0xffffffffu, mbar_wait_limit(smem_u32(&bar_tile_full[slot]), (uint32_t)((pt >> 2) & 1),
                                                                    abortp, pt > 0 ? slot_spin_limit : kSpinLimit));
            if (!ok) { pflags = TILE_STOP; return false; }
            const TileSlot& ts = slots[slot];
            nl = ts.l; ni0 = ts.i0; nj0 = ts.j0;
            pflags = *reinterpret_cast<volatile const int*>(&ts.flags);
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_tile_empty[slot]));      // the descriptor is in registers
            return true;
        };
        auto copy_next = [&]() -> bool {
            bool ok = true;
            if (!(pflags & TILE_STOP)) {
                const int c = SUBS * pt + psub;
                if (lane == 0) {
                    const uint32_t bar = bar0 + 8u * (uint32_t)(c % RING);
                    mbar_expect_tx(bar, (uint32_t)(SLICE_FLOATS * 4));
                    // a tile of W^T: both matrices' warps bring the same slices in (the second
                    // copy is served by L2) and work on one of the two each
                    if (pflags & TILE_W)
                        tma_load_3d(ring_u32 + (uint32_t)((c % RING) * SLICE_FLOATS * 4), &map_w, bar,
                                    nj0 - sch.rows_pad + 64 * h + 32 * psub, ni0 + 32 * q, nl);
                    else
                        tma_load_3d(ring_u32 + (uint32_t)((c % RING) * SLICE_FLOATS * 4), min_map, bar,
                                    nj0 + 64 * h + 32 * psub, ni0 + 32 * q, nl);
                }
                issued = c + 1;
                if (++psub == SUBS) {
                    psub = 0;
                    ++pt;
                    ok = open_tile();
                }
            }
            return ok;
        };

        failed = !open_tile();
        int cl = nl, ci0 = ni0, cj0 = nj0, cflags = pflags;   // tile being worked on
        failed = failed || !copy_next() || !copy_next();
        int unit = 0;
        for (int t = 0; !(cflags & TILE_STOP) && !failed; ++t) {
            for (int g = 0; g < sch.groups && !failed; ++g)
                if (!mbar_wait(smem_u32(&bar_acc_full[(unit + g) & 1]), (uint32_t)(((unit + g) >> 1) & 1), abortp))
                    failed = true;
            failed = __any_sync(0xffffffffu, failed);
            if (failed) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int sub = 0; sub < SUBS; ++sub) {
                const int c = SUBS * t + sub;
                // ---- the update of the slice, summed over the groups (each in an accumulator of its own and
                //      joined in fp32 here: a longer chain in tensor memory would truncate more)
                // (a tile of W^T has one accumulator, which both matrices' warps read)
                const uint32_t from = lane_taddr - ((cflags & TILE_W) ? (uint32_t)(mat * CN) : 0u) + (uint32_t)(32 * sub);
                float upd[32];
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                    uint32_t v[16];
                    tmem_ld16(from + (uint32_t)((unit & 1) * 2 * CN + 16 * cc), v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) upd[16 * cc + e] = __uint_as_float(v[e]);
                    if (sch.groups > 1) {
                        tmem_ld16(from + (uint32_t)(((unit + 1) & 1) * 2 * CN + 16 * cc), v);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; ++e) upd[16 * cc + e] += __uint_as_float(v[e]);
                    }
                }
                if (sub == SUBS - 1) {                   // all of the tile's entries are in registers
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0)
                        for (int g = 0; g < sch.groups; ++g) mbar_arrive(smem_u32(&bar_acc_empty[(unit + g) & 1]));
                }
                if (!mbar_wait(bar0 + 8u * (uint32_t)(c % RING), (uint32_t)((c / RING) & 1), abortp)) failed = true;
                failed = __any_sync(0xffffffffu, failed);
                if (failed) break;
                float* buf = ring + (size_t)(c % RING) * SLICE_FLOATS;
                float4* b4 = reinterpret_cast<float4*>(buf);
                const int ib = ci0 + 32 * q;             // first row of the slice
                const int jc = cj0 + 64 * h + 32 * sub;  // first column of the slice
                // ---- new entries: old - update, one matrix row per lane
                //      (tile of W^T: the two warps that share a quarter of the rows and a half of the columns
                //      take one of its two slices each)
                if (!(cflags & TILE_W) || sub == mat) {
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        float4& o = b4[lane * 8 + (g ^ (lane & 7))];
                        upd[4 * g] = o.x - upd[4 * g];
                        upd[4 * g + 1] = o.y - upd[4 * g + 1];
                        upd[4 * g + 2] = o.z - upd[4 * g + 2];
                        upd[4 * g + 3] = o.w - upd[4 * g + 3];
                        o = make_float4(upd[4 * g], upd[4 * g + 1], upd[4 * g + 2], upd[4 * g + 3]);
                    }
                }
                if (cflags & TILE_W) {
                    // ---- tile of W^T: rows = positions, columns = row indices of W; no mirror
                    __syncwarp();
                    if (sub == mat) {
                        float* Wo = W2 + (size_t)cl * d * rp;
#pragma unroll
                        for (int it = 0; it < 8; ++it) {
                            const int row = 4 * it + (lane >> 3), u = lane & 7;
                            const float4 x = b4[row * 8 + (u ^ (row & 7))];
                            const int gi = ib + row, gj = jc - sch.rows_pad + 4 * u;
                            if (gi < n_pos && gj < rp) *reinterpret_cast<float4*>(Wo + (size_t)gi * rp + gj) = x;
                        }
                    }
                } else {
                    float* Mo = Mout + (size_t)cl * dd;
                    // ---- mirror [j][i]: lanes run along i
                    {
                        const int i = ib + lane;
                        const int jlim = (i < n_pos) ? i - jc : 0;     // entries e < jlim lie below the diagonal
                        float* mp = Mo + (size_t)jc * d + i;
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            if (e < jlim) *mp = upd[e];
                            mp += d;
                        }
                    }
                    __syncwarp();
                    // ---- [i][j]: four rows per instruction, eight lanes along a row
#pragma unroll
                    for (int it = 0; it < 8; ++it) {
                        const int row = 4 * it + (lane >> 3), u = lane & 7;
                        const float4 x = b4[row * 8 + (u ^ (row & 7))];
                        const int gi = ib + row, gj = jc + 4 * u;
                        if (gi < n_pos) {
                            float* p = Mo + (size_t)gi * d + gj;
                            if (gj + 3 < gi) {
                                *reinterpret_cast<float4*>(p) = x;
                            } else {
                                if (gj < gi) p[0] = x.x;
                                if (gj + 1 < gi) p[1] = x.y;
                                if (gj + 2 < gi) p[2] = x.z;
                            }
                        }
                    }
                }
                // the slice is refilled: fence this lane's accesses, then the warp; the copy of the slice two ahead
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                // (the cursor is in the next tile; with the last slice's copy it moves on to the one behind)
                if (sub == SUBS - 1) { cl = nl; ci0 = ni0; cj0 = nj0; cflags = pflags; }
                if (!copy_next()) { failed = true; break; }
            }
            unit += sch.groups;
        }
        // every copy this warp started has landed before the CTA leaves (the last RING slices
        // started are the latest phases of their barriers)
        if (lane == 0)
            for (int c = max(issued - RING, 0); c < issued; ++c)
                mbar_wait_quiet(bar0 + 8u * (uint32_t)(c % RING), (uint32_t)((c / RING) & 1));
        __syncwarp();
        if (failed) abort_flag = 1;
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (abort_flag)
        for (int l = threadIdx.x; l < sch.L; l += AQ_THREADS) set_layer_status(layer_status, l, ZIPLM_ERR_TIMEOUT);
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(AQ_TMEM_COLS)
                     : "memory");
    }
    // the last CTA to leave puts the work counter back to zero for the next launch
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(counter + 1, 1) == (int)gridDim.x - 1) {
            counter[0] = 0;
            counter[1] = 0;
            __threadfence();
        }
    }
}

int sm_count() {
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        cached[dev] = n;
    }
    return cached[dev];
}

}  // namespace

// Tensor map over the packed operands P[L][2][3][rows_tot][64] (bfloat16): box = 64 rows of one array.
bool lazy_tc_make_map(CUtensorMap* m, const float* P, int L, int d, int rp) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    const int rows_pad = lazy_tc_rows_tot(d, rp);
    cuuint64_t dims[4] = {(cuuint64_t)2 * PK, (cuuint64_t)rows_pad, kPackGroups * NARR, (cuuint64_t)L};
    cuuint64_t strides[3] = {(cuuint64_t)128, (cuuint64_t)rows_pad * 128,
                             (cuuint64_t)kPackGroups * NARR * rows_pad * 128};
    cuuint32_t box[4] = {(cuuint32_t)2 * PK, (cuuint32_t)BOX_ROWS, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<float*>(P), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map over one of the fp32 matrices M[L][d][cols] (cols a multiple of 4; d for H^-1 and Q,
// the padded row count of W for W^T): box = 32 rows x 32 columns, 128-byte swizzle; what lies
// outside the matrix reads as zero.
bool lazy_tc_make_matrix_map(CUtensorMap* m, const float* M, int L, int d, int cols) {
    EncodeTiledFn enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)d, (cuuint64_t)L};
    cuuint64_t strides[2] = {(cuuint64_t)cols * 4, (cuuint64_t)d * cols * 4};
    cuuint32_t box[3] = {32, 32, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(M), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// One block of pending steps applied to H^-1 and Q with every position left in place: map_a /
// map_q cover the matrices as they stand (n_pos positions), A2 / Q2 receive the result.
// `counter` points at two ints (work counter, CTAs that have left) that are zero before the first
// launch; every launch leaves them zero again.  slot_spin_limit = 0 selects the default poll
// limit of the waits for descriptors: the producer's for a free slot, the epilogue's for the next one.
ziplm_status run_lazy_update_aq_tc(const CUtensorMap& map, const CUtensorMap& map_a,
                                   const CUtensorMap& map_q, const CUtensorMap& map_w, int L, int groups, int n_pos,
                                   int d, int rp, float* A2, float* Q2, float* W2, int* counter,
                                   int* layer_status, unsigned slot_spin_limit, cudaStream_t st) {
    ZIPLM_CHECK_CUDA(cudaFuncSetAttribute(k_lazy_update_aq_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          AQ_SMEM));
    const int sms = sm_count();
    if (sms <= 0) return ZIPLM_ERR_CUDA;
    const int rows_pad = lazy_tc_rows_pad(d);
    const int rows_used = round_up_int(n_pos, RM);
    if (rows_used / RM > MAX_STRIPS) return ZIPLM_ERR_UNSUPPORTED;
    // Two thirds of the SMs; the others are left to the kernels of other layer groups and batches that run beside it.
    // With two groups of steps the kernel is not bound by memory (0.47 of the copy rate on 99 CTAs) and all SMs make
    // it shorter: a call whose layers are one group takes 27.5 ms on 99 CTAs and 25.7 on 148 (12 x 768 x 3072), 18.1 and
    // 17.2 (24 x 768 x 1814), 108 and 102 (24 x 1024 x 4096).  With six groups beside one another both are the same to
    // about 1.5 %: 26.3 and 26.4, 16.4 and 16.6, 43.8 and 43.8 (24 x 768 x 3072), 96.7 and 95.7; one layer 11.4 and 11.1.
    const int ctas = (2 * sms + 2) / 3;
    AqSched sch;
    sch.n_strips = rows_used / RM;
    sch.L = L;
    sch.groups = groups;
    sch.n_wt = (rp + CN - 1) / CN;
    sch.rows_pad = rows_pad;
    const long long tiles = (long long)L * sch.n_strips * ((sch.n_strips + 1) / 2 + sch.n_wt);   // about
    // about six segments per CTA, so that the last ones to finish differ by a fraction of the run
    long long seg = tiles / ((long long)ctas * 6);
    sch.seg = (int)(seg < 1 ? 1 : (seg > 8 ? 8 : seg));
    sch.prefix[0] = 0;
    for (int k = 0; k < sch.n_strips; ++k) {
        const int nJ = sch.n_strips - k + sch.n_wt;   // strip I = n_strips - 1 - k: I + 1 tiles, then W^T
        sch.prefix[k + 1] = sch.prefix[k] + L * ((nJ + sch.seg - 1) / sch.seg);
    }
    for (int k = sch.n_strips + 1; k <= MAX_STRIPS; ++k) sch.prefix[k] = sch.prefix[sch.n_strips];
    sch.n_segments = sch.prefix[sch.n_strips];
    const int grid = sch.n_segments < ctas ? sch.n_segments : ctas;
    k_lazy_update_aq_tc<<<grid, AQ_THREADS, AQ_SMEM, st>>>(map, map_a, map_q, map_w, sch, n_pos, d, rp, A2, Q2,
                                                          W2, counter, layer_status,
                                                          slot_spin_limit ? slot_spin_limit : kSpinLimit);
    ZIPLM_CHECK_LAUNCH();
    return ZIPLM_OK;
}

}  // namespace ziplm
