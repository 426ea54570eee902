// Merge-path compute kernel for sm_103a (Section 4.2, Algorithm 1): one warp
// per tile of the merge path, joined per CTA at the end.
#pragma once

#include <climits>

#include "kernels.cuh"

namespace spmm {

constexpr int kMergeWarps = 4;  // per CTA, one merge-path tile each
constexpr int kMergeThreads = kMergeWarps * 32;

// Steps of gathers in flight per lane (at most the W steps of a batch): 32
// registers of them for accesses of 16 bytes, 16 for narrower ones.
template <typename TB, int VEC, int E, int W>
__host__ __device__ constexpr int merge_unroll() {
    constexpr int bytes = VEC * (int)sizeof(TB);
    constexpr int u = E >= 4 ? 4 : E > 1 || bytes >= 8 ? 8 : 16;
    return u < W ? u : W;
}

// CTAs of 4 warps per SM, as the registers of the gathers in flight and of the
// row bookkeeping of several lane groups need: 72, 64 or 48 per thread.  Up to 12
// words are spilled where it is 48 (one element per lane and 16 lanes, two and 32)
// and, in 16 bits, up to 7 of the 16-byte layouts.
template <typename TB, int VEC, int E, int W>
__host__ __device__ constexpr int merge_min_blocks() {
    constexpr int bytes = VEC * E * (int)sizeof(TB) * merge_unroll<TB, VEC, E, W>();
    return bytes > 64 ? (W < 32 ? 7 : 8) : (VEC == 2 && W == 32) || W < 32 ? 10 : 8;
}

// Phase 2 of Algorithm 1.  A warp walks its tile (rows [r0, r1) that end in
// it, nonzeros [z0, z1)) in order, all lanes on the same row: W lanes hold the
// W * VEC * E columns of the slab, and the warp's NG = 32 / W lane groups take
// consecutive nonzeros of one step.  So row ends are warp-uniform events (no
// lane waits for another lane's row), and the walk needs no barrier and no
// search.  What bounds it is the gathers of B: their requests to L2 and, where B
// is larger than L2, the DRAM behind it.
//
// The nonzeros come in batches of 32.  Their (column, value) pairs are loaded
// coalesced, one per lane, a batch ahead of their use, and handed out through a
// warp-private slot of shared memory: one 16-byte read serves four steps, where
// every step would need two shuffles of the same pipe.  U steps of gathers are
// issued before the first is accumulated.  Four steps without a row end are
// accumulated unchecked; otherwise each step is split at the row ends in it.
// Tile bounds and row ends are kept in uniform registers (redux results), so
// the checks are uniform branches and cost no vector registers.
//
// A row that began in an earlier tile leaves its last part in s_head, the row
// unfinished at the tile's end its part in s_carry.  The warps of a CTA join
// theirs in tile order at the end, and only rows that cross CTAs go through
// head / carry in global memory to the fix-up.  The unfinished row counts as
// ending at z1, and what the last batch's slots past z1 add goes to a row after
// it that is never stored.
//
// Measured on GB300 (CUDA events, one call, float32) against one CTA per tile
// with the lane groups on separate shares of it (staged by bulk copies, joined
// through barriers): 500,000-row graph of mean degree 20, n = 256, two slabs:
// 1.12 -> 0.74 ms (6.0 TB/s of DRAM traffic); 250,000-row graph, n = 47 (not 16-byte
// aligned): 0.315 -> 0.118 ms; 300,000 rows of Poisson 8, n = 128: 0.167 ->
// 0.147 ms; 200,000 rows of 32, n = 32: 0.094 -> 0.074 ms.
template <typename TV, typename TB, typename TC, int VEC, int E, int W, typename SR = PlusTimes>
__global__ void __launch_bounds__(kMergeThreads, merge_min_blocks<TB, VEC, E, W>()) merge_kernel(MergeArgs a) {
    constexpr int NG = 32 / W;                        // nonzeros per step; a batch is W steps
    constexpr int U = merge_unroll<TB, VEC, E, W>();  // steps in flight
    constexpr int SS = U >= 4 ? 4 : U;                // steps per shared-memory read
    constexpr int GS = NG * U;                        // nonzeros per round of U steps
    constexpr int R = 32 / GS;                        // rounds per batch
    __shared__ __align__(16) int s_col[kMergeWarps][32];
    __shared__ __align__(16) float s_val[kMergeWarps][32];
    __shared__ __align__(16) float s_head[kMergeWarps][W * VEC * E], s_carry[kMergeWarps][W * VEC * E];
    __shared__ int s_carry_row[kMergeWarps];
    pdl_wait();               // the partition (launched just before) has finished writing limits
    pdl_launch_dependents();  // the fix-up may be scheduled; it waits for this grid to finish
    const int lane = threadIdx.x & 31;
    const int warp = uniform(threadIdx.x >> 5);
    const int tile = blockIdx.x * kMergeWarps + warp;  // empty past the last one
    int* const w_col = s_col[warp];
    float* const w_val = s_val[warp];
    const int sl = lane & (W - 1), grp = lane / W;
    const int2 l0 = __ldcg(a.limits + min(tile, a.num_tiles)), l1 = __ldcg(a.limits + min(tile + 1, a.num_tiles));
    const int r0 = uniform(l0.x), z0 = uniform(l0.y), r1 = uniform(l1.x), z1 = uniform(l1.y);
    const TV* __restrict__ vals = static_cast<const TV*>(a.vals);
    const TB* __restrict__ B = static_cast<const TB*>(a.B);
    const int col0 = (int)blockIdx.y * (W * VEC * E) + sl * VEC;  // chunk e: col0 + e * W * VEC
    bool col_ok[E];
#pragma unroll
    for (int e = 0; e < E; ++e) col_ok[e] = col0 + e * W * VEC < a.n;
    // row 0 of B; lanes past n read along with the slab's first column, which the warp reads anyway
    const TB* const b_col = B + (col_ok[0] ? col0 : (int)blockIdx.y * (W * VEC * E));
    const unsigned ldb_bytes = (unsigned)(a.ldb * (long long)sizeof(TB));

    int mc;
    float mv;
    auto fetch = [&](int base) {  // this lane's pair of the batch starting at nonzero base (base <= z1)
        const bool ok = lane < z1 - base;
        mc = ok ? __ldg(a.col_ind + base + lane) : 0;  // slots past z1: column 0, a row that exists
        mv = ok ? load_f(vals + base + lane) : 0.0f;
    };
    // nonzero i of a batch goes to lane group i % NG, step i / NG; a lane group's steps of a round lie together
    const int slot = lane / GS * GS + lane % NG * U + lane / NG % U;

    const int rows = r1 - r0;
    const int row_start = uniform(__ldg(a.row_ptr + r0));
    const bool head_exists = rows > 0 && row_start < z0;  // row r0 began in an earlier tile
    const bool carry_exists = r1 < a.m && z1 > uniform(__ldg(a.row_ptr + r1));
    const int num_ends = rows + (carry_exists ? 1 : 0);
    auto load_end = [&](int i) {
        return i < rows ? __ldg(a.row_ptr + r0 + 1 + i) : (i == rows && carry_exists) ? z1 : INT_MAX;
    };
    fetch(z0);
    int ends = load_end(lane), ends_next = load_end(lane + 32);
    int i_row = 0;                         // current row is r0 + i_row
    int special = head_exists ? 0 : rows;  // the next row that does not go to C: the head, then the carry
    int rend = uniform(__shfl_sync(kFullMask, ends, 0));
    TC* out = static_cast<TC*>(a.C) + (long long)r0 * a.ldc + col0;

    float acc[E][VEC];
    auto clear = [&]() {
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int i = 0; i < VEC; ++i) acc[e][i] = SR::identity();
    };
    clear();
    auto combine = [&]() {  // the lane groups' partial sums of the current row
#pragma unroll
        for (int off = W; off < 32; off <<= 1)
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int i = 0; i < VEC; ++i) acc[e][i] = SR::add(acc[e][i], __shfl_xor_sync(kFullMask, acc[e][i], off));
    };
    // Long rows are summed in blocks (as many nonzeros in sequence would round further off): from
    // sum_from on in acc, what came before in s_carry.
    int sum_from = z0;
    bool summed = false;
    auto add_summed = [&]() {
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int i = 0; i < VEC; ++i)
                if (grp == 0) acc[e][i] = SR::add(s_carry[warp][(e * W + sl) * VEC + i], acc[e][i]);
    };
    auto emit = [&]() {  // the current row ends here
        combine();
        if (summed) add_summed();
        summed = false;
        sum_from = rend;
        if (i_row == special) {
            float* const part = (head_exists && i_row == 0 ? s_head : s_carry)[warp] + sl * VEC;
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (grp == 0) store_vec<float, VEC>(part + e * W * VEC, acc[e]);
            special = rows;
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (grp == 0 && col_ok[e]) store_vec<TC, VEC>(out + e * W * VEC, acc[e]);
        }
        clear();
        out += a.ldc;
        if ((++i_row & 31) == 0) {
            ends = ends_next;
            ends_next = load_end(i_row + lane + 32);
        }
        rend = __reduce_min_sync(kFullMask, lane >= (i_row & 31) ? ends : INT_MAX);  // ends do not decrease
    };

    for (int base = z0; base < z1;) {
        if (base - sum_from >= 64) {
            combine();
            if (summed) add_summed();
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (grp == 0) store_vec<float, VEC>(s_carry[warp] + (e * W + sl) * VEC, acc[e]);
            clear();
            summed = true;
            sum_from = base;
        }
        __syncwarp();
        w_col[slot] = mc;
        w_val[slot] = mv;
        __syncwarp();
        const int left = z1 - base;  // nonzeros from this batch on
        if (left > 32) fetch(base + 32);
#pragma unroll 1
        for (int rd = 0; rd < R; ++rd) {
            if (left <= rd * GS) break;
            Raw<TB, VEC> bv[U][E];
#pragma unroll
            for (int u0 = 0; u0 < U; u0 += SS) {
                int c[SS];
                lds_words<SS>(w_col + rd * GS + grp * U + u0, c);
#pragma unroll
                for (int i = 0; i < SS; ++i)
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        bv[u0 + i][e] = e == 0 || col_ok[e] ? load_raw<TB, VEC>(row_at(b_col, c[i], ldb_bytes) + e * W * VEC)
                                                            : zero_raw<TB, VEC>();
            }
            const int gb = base + rd * GS;
            int rel = rend - gb;  // the current row's end, counted from the round's first nonzero
#pragma unroll
            for (int u0 = 0; u0 < U; u0 += SS) {
                float v[SS];
                lds_words<SS>(w_val + rd * GS + grp * U + u0, v);
                auto accumulate = [&](int i) {
#pragma unroll
                    for (int e = 0; e < E; ++e) accum_raw<SR, TB, VEC>(acc[e], v[i], bv[u0 + i][e]);
                };
                if (rel >= (u0 + SS) * NG) {  // no row ends in these steps
#pragma unroll
                    for (int i = 0; i < SS; ++i) accumulate(i);
                    continue;
                }
#pragma unroll
                for (int i = 0; i < SS; ++i) {
                    const int step_end = (u0 + i + 1) * NG;
                    if constexpr (NG == 1) {
                        while (rel < step_end) {  // rows (possibly empty) that end before this nonzero
                            emit();
                            rel = rend - gb;
                        }
                        accumulate(i);
                    } else if (rel >= step_end) {
                        accumulate(i);
                    } else {
                        const int t = (u0 + i) * NG + grp;  // this lane group's nonzero
                        int lo = 0;
                        do {  // the part of the step that belongs to the ending row
                            if (t >= lo && t < rel) accumulate(i);
                            lo = max(lo, rel);
                            emit();
                            rel = rend - gb;
                        } while (rel < step_end);
                        if (t >= lo) accumulate(i);
                    }
                }
            }
        }
        if (left <= 32) break;
        base += 32;
    }
    while (i_row < num_ends) emit();  // row ends at or after the tile's last nonzero
    if (lane == 0) s_carry_row[warp] = carry_exists ? r1 : -1;
    __syncthreads();

    // rows that cross warps: the carries of the warps before this one that worked on the same row, in
    // order, then `last`; from = the first of those warps
    auto join = [&](int row, const float* last, int* from, float (&sum)[E][VEC]) {
        int t = warp;
        while (t > 0 && s_carry_row[t - 1] == row) --t;
        *from = t;
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                const int at = e * W * VEC + sl * VEC + i;
                float x = SR::identity();
                for (int u = t; u < warp; ++u) x = SR::add(x, s_carry[u][at]);
                sum[e][i] = SR::add(x, last[at]);
            }
    };
    const int2 c0 = __ldcg(a.limits + blockIdx.x * kMergeWarps);  // the CTA's first tile begins here
    if (head_exists) {
        float sum[E][VEC];
        int from;
        join(r0, s_head[warp], &from, sum);
        const bool began_here = from > 0 || row_start >= c0.y;
        if (grp == 0) {
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (!col_ok[e]) continue;
                const int c = col0 + e * W * VEC;
                if (began_here) store_vec<TC, VEC>(static_cast<TC*>(a.C) + (long long)r0 * a.ldc + c, sum[e]);
                else store_vec<float, VEC>(a.head + (size_t)blockIdx.x * a.n + c, sum[e]);
            }
        }
    }
    if (warp == kMergeWarps - 1) {
        if (carry_exists) {
            float sum[E][VEC];
            int from;
            join(r1, s_carry[warp], &from, sum);
            if (grp == 0) {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (col_ok[e]) store_vec<float, VEC>(a.carry + (size_t)blockIdx.x * a.n + col0 + e * W * VEC, sum[e]);
            }
        }
        if (blockIdx.y == 0 && lane == 0) {
            a.carry_row[blockIdx.x] = carry_exists ? r1 : -1;
            a.head_row[blockIdx.x] = c0.x < r1 && __ldg(a.row_ptr + c0.x) < c0.y ? c0.x : -1;
        }
    }
}

}  // namespace spmm
