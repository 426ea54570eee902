// Operations of the backward pass of C = A B with respect to the stored
// values of A and to B (the paper's SpMM_T, named as future work in
// Section 6, plus the sampled dense-dense product):
//   dB    = A^T dC      : spmm_csr_ex on A^T, built once by spmm_csr_transpose
//   dvals = SDDMM(dC, B): dvals[p] = <dC[row(p), :], B[col(p), :]>
//
// CSR transpose: a stable sort of the nonzeros by column index (LSD radix
// sort, 8 bits per pass, the original position as payload), so row c of A^T
// lists the nonzeros of column c in increasing original position.  Every step
// is deterministic; the permutation lets vals^T be refreshed with one gather
// when the values change but the pattern does not.
//
// SDDMM: balanced by nonzero split (Section 4 item 2(a)): every lane group
// takes an equal run of consecutive nonzeros and finds its first row by a
// binary search on row_ptr, so a long row is shared by many groups.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <climits>

#include "launch.cuh"

namespace spmm {
namespace {

constexpr int kRadix = 256;
constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kScanThreads = 1024;

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

int status_of(cudaError_t e) {
    if (e == cudaSuccess) return SPMM_OK;
    if (e == cudaErrorMemoryAllocation) return SPMM_ERR_ALLOC;
    if (e == cudaErrorInvalidConfiguration || e == cudaErrorLaunchOutOfResources || e == cudaErrorInvalidValue)
        return SPMM_ERR_LAUNCH;
    return SPMM_ERR_CUDA;
}

int launched(cudaError_t e) {
    if (e == cudaSuccess) g_launches.fetch_add(1, std::memory_order_relaxed);
    return status_of(e);
}

// Passes of the radix sort over column indices below k, and the bits of a
// digit: the passes share the bits equally, since a digit of fewer bits leaves
// longer runs of equal digits in a tile (k = 500,000: three digits of 7 bits).
void radix_shape(int k, int* passes, int* bits) {
    int total = 0;
    while (total < 31 && ((long long)(k > 0 ? k - 1 : 0) >> total) > 0) ++total;
    *passes = std::max(1, (total + 7) / 8);
    *bits = std::max(1, (total + *passes - 1) / *passes);
}

struct TransposeLayout {
    int tiles;
    size_t off_k0, off_k1, off_v, off_hist, off_tot, total;
};

TransposeLayout transpose_layout(long long nnz) {
    TransposeLayout L{};
    L.tiles = (int)((nnz + kSortTile - 1) / kSortTile);
    size_t off = 0;
    L.off_k0 = off;
    off = a256(off + (size_t)nnz * 4);
    L.off_k1 = off;
    off = a256(off + (size_t)nnz * 4);
    L.off_v = off;
    off = a256(off + (size_t)nnz * 4);
    L.off_hist = off;
    off = a256(off + (size_t)kRadix * (L.tiles > 0 ? L.tiles : 1) * 4);
    L.off_tot = off;
    off = a256(off + (size_t)kRadix * 4);
    L.total = off;
    return L;
}

// Per-tile histogram of one digit of at most 8 bits; hist is digit-major
// [mask + 1][tiles].  A thread's keys are loaded before the first is counted.
__global__ void radix_hist_kernel(const int* __restrict__ keys, long long n, int shift, int mask, int tiles,
                                  int* __restrict__ hist) {
    __shared__ int cnt[kRadix];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const long long base = (long long)blockIdx.x * kSortTile + threadIdx.x;
    int key[kSortItems];
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) key[i] = base + i * kSortThreads < n ? __ldg(keys + base + i * kSortThreads) : 0;
#pragma unroll
    for (int i = 0; i < kSortItems; ++i)
        if (base + i * kSortThreads < n) atomicAdd(&cnt[(key[i] >> shift) & mask], 1);
    __syncthreads();
    if ((int)threadIdx.x <= mask) hist[(long long)threadIdx.x * tiles + blockIdx.x] = cnt[threadIdx.x];
}

// Exclusive prefix sums of the digit-major histogram: one CTA per digit scans
// its row in place (chunks of kScanThreads coalesced elements, warp shuffles, a
// running carry) and leaves the row's total in totals[d].  The scatter turns the
// totals into the digits' first positions and adds them to each row's prefix.
__global__ void digit_scan_kernel(int* __restrict__ hist, int tiles, int* __restrict__ totals) {
    constexpr int kWarps = kScanThreads / 32;
    __shared__ int warp_sum[kWarps];
    __shared__ int carry;
    int* row = hist + (long long)blockIdx.x * tiles;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < tiles; base += kScanThreads) {
        const int i = base + tid;
        const int v = i < tiles ? row[i] : 0;
        int x = v;  // inclusive scan inside the warp
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(kFullMask, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        if (warp == 0) {  // inclusive scan of the warp sums
            int w = warp_sum[lane];
#pragma unroll
            for (int off = 1; off < kWarps; off <<= 1) {
                const int y = __shfl_up_sync(kFullMask, w, off);
                if (lane >= off) w += y;
            }
            warp_sum[lane] = w;
        }
        __syncthreads();
        if (i < tiles) row[i] = carry + (warp > 0 ? warp_sum[warp - 1] : 0) + x - v;
        __syncthreads();
        if (tid == 0) carry += warp_sum[kWarps - 1];
        __syncthreads();
    }
    if (tid == 0) totals[blockIdx.x] = carry;
}

// Exclusive prefix sums of two values per thread over a block of kRadix threads.
__device__ __forceinline__ void block_scan2(int& a, int& b, int (*warp_sum)[kRadix / 32]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = a, y = b;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int xs = __shfl_up_sync(kFullMask, x, off), ys = __shfl_up_sync(kFullMask, y, off);
        if (lane >= off) {
            x += xs;
            y += ys;
        }
    }
    if (lane == 31) {
        warp_sum[0][warp] = x;
        warp_sum[1][warp] = y;
    }
    __syncthreads();
    a = x - a;
    b = y - b;
    for (int w = 0; w < warp; ++w) {
        a += warp_sum[0][w];
        b += warp_sum[1][w];
    }
}

// Stable scatter of one radix pass.  The tile is first sorted by digit in
// shared memory, then written out in that order, so a run of equal digits goes
// to consecutive global positions.  A warp ranks the kSortItems x 32 consecutive
// elements that it holds in registers: the rank among equal digits comes from
// ballots of the digit's bits within 32 of them and from the warp's own digit
// counts across the steps, without a barrier; one scan over warps and digits
// then gives every element its place.  (Ranking a step of the whole tile at a
// time took three barriers for every 256 elements, and __match_any_sync in the
// place of the ballots a third longer.)  Element order is kept among equal
// digits.  10M keys of 7 bits: 0.12 -> 0.088 ms, the transpose 0.55 -> 0.36.
// payload_in == nullptr means the payload is the element's own index.  Four CTAs
// per SM leave 64 registers, which hold all but 17 words of a thread's keys and
// ranks.
__global__ void __launch_bounds__(kSortThreads, 4) radix_scatter_kernel(
    const int* __restrict__ keys_in, const int* __restrict__ payload_in, long long n, int shift, int mask, int tiles,
    const int* __restrict__ offsets, const int* __restrict__ totals, int* __restrict__ keys_out,
    int* __restrict__ payload_out) {
    constexpr int kWarps = kSortThreads / 32;
    __shared__ int s_key[kSortTile];
    __shared__ int s_pay[kSortTile];
    __shared__ int s_cnt[kWarps][kRadix];  // digit counts of each warp, then the warp's offset within the digit
    __shared__ int local[kRadix];          // tile-local first position of each digit
    __shared__ int global[kRadix];         // global position of a tile-local position of the digit, less the latter
    __shared__ int warp_sum[2][kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long tile0 = (long long)blockIdx.x * kSortTile;
    const int count = n - tile0 < kSortTile ? (int)(n - tile0) : kSortTile;
    const int first = warp * kSortItems * 32 + lane;  // this lane's elements: first + 32 r
    int key[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) key[r] = first + 32 * r < count ? __ldg(keys_in + tile0 + first + 32 * r) : 0;
#pragma unroll
    for (int d = lane; d < kRadix; d += 32) s_cnt[warp][d] = 0;
    __syncwarp();
    const unsigned lt_mask = (1u << lane) - 1u;
    int rank[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const bool valid = first + 32 * r < count;
        const int d = (key[r] >> shift) & mask;
        unsigned peers = __ballot_sync(kFullMask, valid);  // the lanes of the same digit: those that agree in every bit
        for (int b = 0; mask >> b; ++b) {
            const bool set = (d >> b) & 1;
            const unsigned ball = __ballot_sync(kFullMask, set);
            peers &= set ? ball : ~ball;
        }
        const int before = valid ? s_cnt[warp][d] : 0;
        rank[r] = before + __popc(peers & lt_mask);
        __syncwarp();
        if (valid && lane == 31 - __clz(peers)) s_cnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {  // thread d: digit d (kSortThreads == kRadix)
        int in_tile = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const int c = s_cnt[w][tid];
            s_cnt[w][tid] = in_tile;
            in_tile += c;
        }
        int in_all = tid <= mask ? totals[tid] : 0;
        block_scan2(in_tile, in_all, warp_sum);
        local[tid] = in_tile;
        if (tid <= mask) global[tid] = offsets[(long long)tid * tiles + blockIdx.x] + in_all - in_tile;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        if (first + 32 * r < count) {
            const int d = (key[r] >> shift) & mask;
            const int pos = local[d] + s_cnt[warp][d] + rank[r];
            s_key[pos] = key[r];
            s_pay[pos] = payload_in ? __ldg(payload_in + tile0 + first + 32 * r) : (int)(tile0 + first + 32 * r);
        }
    }
    __syncthreads();
    for (int i = tid; i < count; i += kSortThreads) {
        const int k = s_key[i];
        const int pos = global[(k >> shift) & mask] + i;
        keys_out[pos] = k;
        payload_out[pos] = s_pay[i];
    }
}

// row_ptr_t[c] = first position of column c in the sorted keys (lower bound).
__global__ void transpose_rowptr_kernel(const int* __restrict__ sorted_keys, long long nnz, int k,
                                        int* __restrict__ row_ptr_t) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c > k) return;
    long long lo = 0, hi = nnz;
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        if (__ldg(sorted_keys + mid) < c) lo = mid + 1;
        else hi = mid;
    }
    row_ptr_t[c] = (int)lo;
}

// rows[p] = the row of A holding nonzero p, for every p: a CTA per tile of
// nonzeros marks where its rows begin and spreads the marks with a running
// maximum.  A tile with more than two rows per nonzero, most of them empty, looks
// each nonzero up among them instead, so that the work of a CTA is bounded: a
// transpose with 4M empty rows between two nonzeros 6.8 -> 0.13 ms, with 20M
// 33.7 -> 0.18 (a warp per row: 0.41 and 1.55).
constexpr int kMostRows = 2 * kSortTile;
__global__ void __launch_bounds__(kSortThreads) expand_rows_kernel(const int* __restrict__ row_ptr, int m, int nnz,
                                                                   int* __restrict__ rows) {
    __shared__ __align__(16) int s_row[kSortTile];  // row beginning at this nonzero, counted from the tile's first
    __shared__ int s_first[2];
    __shared__ int warp_max[kSortThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile0 = blockIdx.x * kSortTile;
    const int last = nnz - tile0 > kSortTile ? tile0 + kSortTile - 1 : nnz - 1;
    for (int i = tid; i < kSortTile; i += kSortThreads) s_row[i] = 0;
    if (warp < 2) {  // the rows of the tile's first and last nonzero: the largest r with row_ptr[r] <= p
        const int p = warp == 0 ? tile0 : last;
        int lo = 0, hi = m;
        while (hi - lo > 1) {
            const long long span = hi - lo;
            const int x = lo + (int)((span * lane) / 32);
            const int cnt = __popc(__ballot_sync(kFullMask, __ldg(row_ptr + x) <= p));
            const int x_last = lo + (int)((span * (cnt - 1)) / 32);
            hi = cnt < 32 ? lo + (int)((span * cnt) / 32) : hi;
            lo = x_last;
        }
        if (lane == 0) s_first[warp] = lo;
    }
    __syncthreads();
    const int ra = s_first[0], rb = s_first[1];
    if (rb - ra > kMostRows) {  // the largest r with row_ptr[r] <= p, for all of a thread's nonzeros at once
        int lo[kSortItems], step = 1 << (31 - __clz(rb - ra));
#pragma unroll
        for (int i = 0; i < kSortItems; ++i) lo[i] = ra;
        for (; step > 0; step >>= 1) {
#pragma unroll
            for (int i = 0; i < kSortItems; ++i)
                if (step <= rb - lo[i] && __ldg(row_ptr + lo[i] + step) <= min(tile0 + i * kSortThreads + tid, last))
                    lo[i] += step;
        }
#pragma unroll
        for (int i = 0; i < kSortItems; ++i)
            if (i * kSortThreads + tid <= last - tile0) rows[tile0 + i * kSortThreads + tid] = lo[i];
        return;
    }
    for (int r = ra + 1 + tid; r <= rb; r += kSortThreads)  // empty rows begin where the next one does: the last wins
        atomicMax(&s_row[__ldg(row_ptr + r) - tile0], r - ra);
    __syncthreads();
    int v[kSortItems];
    int best = 0;
#pragma unroll
    for (int i = 0; i < kSortItems; i += 4) {
        const int4 x = *reinterpret_cast<const int4*>(s_row + tid * kSortItems + i);
        const int w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) v[i + e] = best = max(best, w[e]);
    }
    int incl = best;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFullMask, incl, off);
        if (lane >= off) incl = max(incl, y);
    }
    if (lane == 31) warp_max[warp] = incl;
    int before = __shfl_up_sync(kFullMask, incl, 1);
    if (lane == 0) before = 0;
    __syncthreads();
    for (int w = 0; w < warp; ++w) before = max(before, warp_max[w]);
#pragma unroll
    for (int i = 0; i < kSortItems; i += 4)
        *reinterpret_cast<int4*>(s_row + tid * kSortItems + i) =
            make_int4(ra + max(before, v[i]), ra + max(before, v[i + 1]), ra + max(before, v[i + 2]), ra + max(before, v[i + 3]));
    __syncthreads();
    for (int i = tid; i <= last - tile0; i += kSortThreads) rows[tile0 + i] = s_row[i];
}

template <typename T>
__global__ void gather_values_kernel(const int* __restrict__ perm, long long nnz, const T* __restrict__ vals,
                                     T* __restrict__ out) {
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < nnz; q += (long long)gridDim.x * blockDim.x)
        out[q] = vals[__ldg(perm + q)];
}

// ------------------------------------------------------------------------------------- SDDMM

struct SddmmArgs {
    int m, n;
    long long nnz;
    const int* row_ptr;
    const int* col_ind;
    const void* dC;
    long long lddc;
    const void* B;
    long long ldb;
    void* out;
    int chunk;  // nonzeros per lane group
};

// One lane group of W lanes per run of `chunk` consecutive nonzeros; each lane
// owns the columns chunk j = sl, sl + W, ... (VEC elements each) of both rows;
// kUnroll nonzeros are processed together and their partial dot products are
// reduced across the group with xor shuffles.
template <typename TD, typename TO, int VEC, int W>
__global__ void __launch_bounds__(kThreads) sddmm_kernel(SddmmArgs a) {
    constexpr int U = kUnroll;
    const int lane = threadIdx.x & 31, sl = lane & (W - 1);
    const long long g = ((long long)blockIdx.x * kThreads + threadIdx.x) / W;
    const long long p0 = g * a.chunk;
    const long long p1 = p0 + a.chunk < a.nnz ? p0 + a.chunk : a.nnz;
    const TD* __restrict__ dC = static_cast<const TD*>(a.dC);
    const TD* __restrict__ B = static_cast<const TD*>(a.B);
    const int nchunks = (a.n + VEC - 1) / VEC;
    int row = 0, row_end = 0;
    if (p0 < p1) {  // last row whose start is <= p0
        int lo = 0, hi = a.m;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(a.row_ptr + mid) <= p0) lo = mid;
            else hi = mid - 1;
        }
        row = lo;
        row_end = __ldg(a.row_ptr + row + 1);
    }
    const int nb = p0 < p1 ? (int)((p1 - p0 + U - 1) / U) : 0;
    const int nb_max = __reduce_max_sync(kFullMask, nb);
    for (int b = 0; b < nb_max; ++b) {
        float part[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long p = p0 + (long long)b * U + u;
            part[u] = 0.0f;
            if (p < p1) {
                while (p >= row_end) row_end = __ldg(a.row_ptr + (++row) + 1);
                const TD* brow = gather_row(B, 0, __ldg(a.col_ind + p), a.ldb);
                const TD* drow = dC + (long long)row * a.lddc;
                for (int j = sl; j < nchunks; j += W) {
                    const Raw<TD, VEC> x = load_raw<TD, VEC>(brow + (long long)j * VEC);
                    float y[VEC];
                    load_vec<TD, VEC>(drow + (long long)j * VEC, y);
                    float t[VEC];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) t[e] = 0.0f;
                    fma_raw<TD, VEC>(t, 1.0f, x);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) part[u] = fmaf(t[e], y[e], part[u]);
                }
            }
        }
#pragma unroll
        for (int off = W / 2; off > 0; off >>= 1)
#pragma unroll
            for (int u = 0; u < U; ++u) part[u] += __shfl_xor_sync(kFullMask, part[u], off, W);
        if (sl == 0) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long long p = p0 + (long long)b * U + u;
                if (p < p1) static_cast<TO*>(a.out)[p] = Elem<TO>::from_f(part[u]);
            }
        }
    }
}

// Wide and unaligned rows: a warp per run of `chunk` consecutive nonzeros, 32
// lanes on one nonzero at a time, E column chunks of VEC elements per lane from
// column col0 on.  U rows of B are gathered before the first is used, whatever
// rows of A they belong to; the current row of dC stays in registers and changes
// at the row ends, which are warp-uniform (redux results, kept in uniform
// registers), with the next row's already on its way.  The U dot products are
// reduced together: each exchange halves the products a lane holds, so that U =
// 8 of them take 9 shuffles and not 40.  With `accumulate` a pass adds to what
// the passes over the columns before col0 left in out (float32).
//
// What bounds it is the gathers of B, as in the forward product.  Measured on
// GB300 (CUDA events, float32) against the kernel that cut its batches at row
// ends and reduced each product on its own: 500,000-node graph
// of mean degree 20, n = 256 (two passes), 0.963 -> 0.907 ms (5.1 TB/s of DRAM
// traffic), n = 128 0.582 -> 0.432; 250,000 nodes, n = 47, 0.710 -> 0.151;
// 60,000 rows of Poisson 15, n = 128, 0.072 -> 0.045 ms.
template <typename TD, int VEC, int E>
__host__ __device__ constexpr int sddmm_unroll() {
    constexpr int bytes = VEC * E * (int)sizeof(TD);
    return bytes <= 16 ? 8 : bytes <= 32 ? 4 : bytes <= 64 ? 2 : 1;
}

// CTAs of 4 warps per SM: 64 registers, more where a lane holds more than 16
// columns of the row of dC (and of the next one).
template <int VEC, int E>
__host__ __device__ constexpr int sddmm_min_blocks() { return VEC * E <= 16 ? 8 : VEC * E <= 32 ? 4 : 2; }

template <typename TD, typename TO, int VEC, int E>
__global__ void __launch_bounds__(128, sddmm_min_blocks<VEC, E>()) sddmm_warp_kernel(SddmmArgs a, int col0, int accumulate) {
    constexpr int U = sddmm_unroll<TD, VEC, E>();
    constexpr int SS = U >= 4 ? 4 : U;  // columns per shared-memory read
    __shared__ __align__(16) int s_col[4][32];
    const int lane = threadIdx.x & 31;
    const int warp = uniform(threadIdx.x >> 5);
    const long long first = ((long long)blockIdx.x * 4 + warp) * a.chunk;
    if (first >= a.nnz) return;  // whole warps leave together
    const int p0 = uniform((int)first);
    const int p1 = uniform((int)(first + a.chunk < a.nnz ? first + a.chunk : a.nnz));
    int* const w_col = s_col[warp];
    bool col_ok[E];
#pragma unroll
    for (int e = 0; e < E; ++e) col_ok[e] = (e * 32 + lane) * VEC < a.n - col0;  // a.n may be near 2^31
    // lanes past n read along with the pass's first column, which the warp reads anyway, and add nothing
    const int my_col = col_ok[0] ? col0 + lane * VEC : col0;
    const TD* const b_col = static_cast<const TD*>(a.B) + my_col;
    const TD* const d_col = static_cast<const TD*>(a.dC) + my_col;
    const unsigned ldb_bytes = (unsigned)(a.ldb * (long long)sizeof(TD));

    // first row: the largest r with row_ptr[r] <= p0 (row_ptr[0] = 0 <= p0 always holds)
    int lo = 0, hi = a.m;  // answer in [lo, hi)
    while (hi - lo > 1) {
        const long long span = hi - lo;
        const int x = lo + (int)((span * lane) / 32);
        const unsigned ball = __ballot_sync(kFullMask, __ldg(a.row_ptr + x) <= p0);
        const int cnt = __popc(ball);  // a prefix of the lanes, at least lane 0
        const int x_last = lo + (int)((span * (cnt - 1)) / 32);
        hi = cnt < 32 ? lo + (int)((span * cnt) / 32) : hi;
        lo = x_last;
    }
    // row ends from row window on, one per lane; next_row(q) finds the first row that ends after nonzero q
    int window = uniform(lo);
    auto load_ends = [&]() { return lane < a.m - window ? __ldg(a.row_ptr + window + 1 + lane) : INT_MAX; };
    int ends = load_ends();
    int row = window, rend = 0;
    auto next_row = [&](int q) {
        unsigned after = __ballot_sync(kFullMask, ends > q);
        while (after == 0u) {
            window += 32;
            ends = load_ends();
            after = __ballot_sync(kFullMask, ends > q);
        }
        row = min(window + __ffs(after) - 1, a.m - 1);
        rend = __reduce_min_sync(kFullMask, ends > q && ends < p1 ? ends : INT_MAX);  // p1 on: no other row here
    };
    float y[E][VEC];
    Raw<TD, VEC> y_next[E];
    auto load_y = [&](int r) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            y_next[e] = col_ok[e] ? load_raw<TD, VEC>(d_col + (long long)r * a.lddc + e * 32 * VEC) : zero_raw<TD, VEC>();
    };
    auto take_y = [&]() {
#pragma unroll
        for (int e = 0; e < E; ++e) widen_raw<TD, VEC>(y_next[e], y[e]);
    };
    next_row(p0);
    load_y(row);
    take_y();
    int y_row = -1;  // the row in y_next
    if (row + 1 < a.m) load_y(y_row = row + 1);

    int mc = lane < p1 - p0 ? __ldg(a.col_ind + p0 + lane) : 0;
    for (int base = p0;;) {
        __syncwarp();
        w_col[lane] = mc;  // slots past p1: column 0, a row that exists
        __syncwarp();
        const int left = p1 - base;
        if (left > 32) mc = lane < left - 32 ? __ldg(a.col_ind + base + 32 + lane) : 0;
#pragma unroll 1
        for (int rd = 0; rd < 32 / U; ++rd) {
            const int gl = left - rd * U;  // nonzeros from this group on
            if (gl <= 0) break;
            const int q0 = base + rd * U;
            Raw<TD, VEC> x[U][E];
#pragma unroll
            for (int u0 = 0; u0 < U; u0 += SS) {
                int c[SS];
                lds_words<SS>(w_col + rd * U + u0, c);
#pragma unroll
                for (int i = 0; i < SS; ++i)
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        x[u0 + i][e] = e == 0 || col_ok[e] ? load_raw<TD, VEC>(row_at(b_col, c[i], ldb_bytes) + e * 32 * VEC)
                                                           : zero_raw<TD, VEC>();
            }
            float part[U];
            auto product = [&](int u) {
                part[u] = 0.0f;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    float t[VEC];
                    widen_raw<TD, VEC>(x[u][e], t);
#pragma unroll
                    for (int i = 0; i < VEC; ++i) part[u] = fmaf(t[i], y[e][i], part[u]);
                }
            };
#pragma unroll
            for (int u0 = 0; u0 < U; u0 += SS) {
                if (rend - q0 >= u0 + SS) {  // no row ends in these products
#pragma unroll
                    for (int i = 0; i < SS; ++i) product(u0 + i);
                    continue;
                }
#pragma unroll
                for (int i = 0; i < SS; ++i) {
                    while (rend - q0 <= u0 + i) {  // this nonzero belongs to a later row (once at most)
                        next_row(q0 + u0 + i);
                        if (row != y_row) load_y(row);
                        take_y();
                        y_row = -1;
                        if (row + 1 < a.m) load_y(y_row = row + 1);
                    }
                    product(u0 + i);
                }
            }
            if (!col_ok[0]) {
#pragma unroll
                for (int u = 0; u < U; ++u) part[u] = 0.0f;
            }
            // lane l ends up with product l / (32 / U)
            int off = 16;
#pragma unroll
            for (int cnt = U; cnt > 1; cnt >>= 1, off >>= 1) {
                const bool upper = (lane & off) != 0;
#pragma unroll
                for (int i = 0; i < cnt / 2; ++i) {
                    const float send = upper ? part[i] : part[i + cnt / 2], keep = upper ? part[i + cnt / 2] : part[i];
                    part[i] = keep + __shfl_xor_sync(kFullMask, send, off);
                }
            }
#pragma unroll
            for (; off > 0; off >>= 1) part[0] += __shfl_xor_sync(kFullMask, part[0], off);
            const int mine = lane / (32 / U);
            if (lane % (32 / U) == 0 && mine < gl) {
                TO* const o = static_cast<TO*>(a.out) + q0 + mine;
                *o = Elem<TO>::from_f(accumulate ? Elem<TO>::to_f(*o) + part[0] : part[0]);
            }
        }
        if (left <= 32) break;
        base += 32;
    }
}

template <typename TD, typename TO, int VEC, int E>
cudaError_t sddmm_warp_launch(const SddmmArgs& a0, cudaStream_t st, int k = 0) {
    SddmmArgs a = a0;
    // nonzeros per warp: about 256, in whole waves of the 32 warps that an SM runs at once (up to 16
    // columns of dC per lane; the wider layouts run 16 or 8, and two or four waves for one)
    const long long wave = 256LL * 32 * 152, waves = std::max<long long>(1, (a.nnz + wave / 2) / wave);
    const long long per_warp = (a.nnz + waves * 32 * 152 - 1) / (waves * 32 * 152);
    a.chunk = (int)std::max<long long>(32, (per_warp + 31) / 32 * 32);
    const long long blocks = (a.nnz + 4LL * a.chunk - 1) / (4LL * a.chunk);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    long long c = 0;
    auto pass = [&](auto chunks) {
        constexpr int EP = decltype(chunks)::value;
        sddmm_warp_kernel<TD, TO, VEC, EP><<<(unsigned)blocks, 128, 0, st>>>(a, (int)c, c > 0);
        if (c > 0) g_launches.fetch_add(1, std::memory_order_relaxed);  // the caller counts one
        c += 32 * VEC * EP;
        return cudaGetLastError();
    };
    while (c < a.n) {
        cudaError_t e;
        const long long left = a.n - c;
        if constexpr (sizeof(TD) == 4 && VEC == 4 && E == 1) {
            // A short last pass costs nearly a full one, and joins the pass before it: up to 52 columns,
            // and any short one where L2 (129 MB) does not hold a pass's columns of B.  Below 5 nonzeros
            // per row, where every pass loads a row of dC for a few products, passes go two by two.  Against two passes
            // and against one with the products reduced one by one (us): 500,000 rows of Poisson 6,
            // n = 132, 310 / 421 / 363, n = 200, 412 / 490 / 457, n = 256, 488 / 463 / 519; 150,000 of
            // 15, n = 132, 169 / 199 / 199, n = 200, 236 / 222 / 224.
            const bool short_rows = a.nnz < 5LL * a.m;
            if (left > 128 && (short_rows || (left < 256 && (left <= 180 || k * 512LL > (129LL << 20)))))
                e = pass(std::integral_constant<int, 2>());
            else
                e = pass(std::integral_constant<int, 1>());
        } else {
            e = pass(std::integral_constant<int, E>());
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// W: up to 8 lanes for the narrow and short rows that sddmm_run leaves to the lane
// groups, 32 for the wide ones with 16-bit results.
template <typename TD, typename TO, int VEC>
cudaError_t sddmm_launch_vec(const SddmmArgs& a, int W, long long groups, cudaStream_t st) {
    const long long blocks = (groups * W + kThreads - 1) / kThreads;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    switch (W) {
        case 1: sddmm_kernel<TD, TO, VEC, 1><<<(unsigned)blocks, kThreads, 0, st>>>(a); break;
        case 2: sddmm_kernel<TD, TO, VEC, 2><<<(unsigned)blocks, kThreads, 0, st>>>(a); break;
        case 4: sddmm_kernel<TD, TO, VEC, 4><<<(unsigned)blocks, kThreads, 0, st>>>(a); break;
        case 8: sddmm_kernel<TD, TO, VEC, 8><<<(unsigned)blocks, kThreads, 0, st>>>(a); break;
        default:
            if constexpr (sizeof(TO) == 2) {
                sddmm_kernel<TD, TO, VEC, 32><<<(unsigned)blocks, kThreads, 0, st>>>(a);
                break;
            }
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <typename TD, typename TO>
int sddmm_run(const SddmmArgs& a0, int k, cudaStream_t st) {
    SddmmArgs a = a0;
    constexpr int V = Elem<TD>::kVec;
    auto aligned = [&](int v) {
        return a.n % v == 0 && a.lddc % v == 0 && a.ldb % v == 0 && ((uintptr_t)a.dC % (v * sizeof(TD))) == 0 &&
               ((uintptr_t)a.B % (v * sizeof(TD))) == 0;
    };
    const bool vec_ok = aligned(V);
    const int vec = vec_ok ? V : 1;
    const long long nchunks = ((long long)a.n + vec - 1) / vec;
    int W = 1;
    while (W < nchunks && W < 32) W <<= 1;
    // A warp per nonzero, with the narrowest access that covers the row in one pass of 32 lanes, or
    // the widest aligned one and several passes (float32 results) or column chunks (16-bit results,
    // which cannot be added up in place).  The lane groups stay for up to 3 columns and, up to 32
    // aligned ones (or 8), for rows of A of fewer than 4 nonzeros (4.75 for up to 7 unaligned columns),
    // where the warp changes rows at every other nonzero: 600,000 rows of 3, n = 32, 119 us against
    // 129; 2M nonzeros of a graph, n = 32, 80 against 64; 900,000 of Poisson 15, n = 8, 72 against 31.
    // They also stay for rows of up to 4 lanes where many nonzeros fill their waves (of 4 CTAs per SM,
    // about as long as they are empty), the groups / the warps (us): n = 16, 500,000 rows of 9.5, 120 /
    // 146, of 6, 115 / 119, 800,000 of 7 (1.1 waves) 228 / 197; n = 8, 1M of 6, 154 / 187, bf16 n = 16,
    // 1M of 9, 175 / 238; n = 4, 1M of 9, 169 / 234; bf16 n = 4 (unaligned), 500,000 of 8, 97 / 120, of
    // 4.5, 87 / 89.
    constexpr bool kPasses = sizeof(TO) == 4;
    const int n = a.n;
    int w = V;
    while (w > 1 && !aligned(w)) w >>= 1;
    const bool short_rows = n <= 32 && (n < 8 && !vec_ok && a.nnz >= 2000000 ? 4 * a.nnz < 19LL * a.m : a.nnz < 4LL * a.m) && (n <= 8 || vec_ok);
    const long long wave = 4LL * 152 * (kThreads / W) * 128;  // nonzeros of the lane groups' CTAs
    const bool full = !vec_ok   ? n == 4 && a.nnz >= 2500000
                      : W == 1  ? a.nnz >= 7000000
                      : W <= 4  ? a.nnz >= 3600000 && (a.nnz <= wave || a.nnz * 100 >= (a.nnz + wave - 1) / wave * wave * (W == 2 ? 69 : 90))
                                : false;
    const bool by_groups = n < 4 || short_rows || full || (!kPasses && n > (w == V ? 256 * V : 128));
    if (!by_groups) {
        if (n <= 32) return launched(sddmm_warp_launch<TD, TO, 1, 1>(a, st));
        if (w >= 2 && n <= 64) return launched(sddmm_warp_launch<TD, TO, 2, 1>(a, st));
        if constexpr (V == 8) {
            if (w >= 4 && n <= 128) return launched(sddmm_warp_launch<TD, TO, 4, 1>(a, st));
        }
        if (w == V && (n <= 32 * V || kPasses)) return launched(sddmm_warp_launch<TD, TO, V, 1>(a, st, k));
        if constexpr (!kPasses) {
            if (w == V && n <= 64 * V) return launched(sddmm_warp_launch<TD, TO, V, 2>(a, st));
            if (w == V && n <= 128 * V) return launched(sddmm_warp_launch<TD, TO, V, 4>(a, st));
            if (w == V) return launched(sddmm_warp_launch<TD, TO, V, 8>(a, st));
        }
        if (w >= 2) return launched(sddmm_warp_launch<TD, TO, 2, 2>(a, st));
        if (n <= 64) return launched(sddmm_warp_launch<TD, TO, 1, 2>(a, st));
        return launched(sddmm_warp_launch<TD, TO, 1, 4>(a, st));
    }
    a.chunk = 128;  // nonzeros per lane group: longer runs amortise the row search (n = 32: 0.38 -> 0.35 ms)
    const long long groups = (a.nnz + a.chunk - 1) / a.chunk;
    const cudaError_t e = vec_ok ? sddmm_launch_vec<TD, TO, V>(a, W, groups, st) : sddmm_launch_vec<TD, TO, 1>(a, W, groups, st);
    return launched(e);
}

}  // namespace
}  // namespace spmm

using namespace spmm;

extern "C" {

size_t spmm_csr_transpose_workspace_size(int m, int k, long long nnz) {
    if (m < 0 || k < 0 || nnz < 0) return 0;
    return transpose_layout(nnz).total;
}

int spmm_csr_transpose(int m, int k, long long nnz, const int* row_ptr, const int* col_ind, int* row_ptr_t,
                       int* col_ind_t, int* perm, void* workspace, size_t workspace_bytes, void* stream) {
    if (m < 0 || k < 0 || nnz < 0 || nnz > 0x7fffffffLL) return SPMM_ERR_INVALID_VALUE;
    if (!row_ptr_t || (nnz > 0 && (!row_ptr || !col_ind || !col_ind_t || !perm))) return SPMM_ERR_INVALID_VALUE;
    if (nnz > 0 && m == 0) return SPMM_ERR_INVALID_VALUE;
    cudaStream_t s = (cudaStream_t)stream;
    const TransposeLayout L = transpose_layout(nnz);
    if (nnz == 0) {
        const cudaError_t e = cudaMemsetAsync(row_ptr_t, 0, (size_t)(k + 1) * 4, s);
        return status_of(e);
    }
    bool own = false;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    if (!ws) {
        if (workspace_bytes != 0) return SPMM_ERR_WORKSPACE;
        void* p = nullptr;
        if (cudaMallocAsync(&p, L.total, s) != cudaSuccess) return SPMM_ERR_ALLOC;
        ws = static_cast<unsigned char*>(p);
        own = true;
    } else if (workspace_bytes < L.total) {
        return SPMM_ERR_WORKSPACE;
    }
    int* kbuf[2] = {reinterpret_cast<int*>(ws + L.off_k0), reinterpret_cast<int*>(ws + L.off_k1)};
    int* vtmp = reinterpret_cast<int*>(ws + L.off_v);
    int* hist = reinterpret_cast<int*>(ws + L.off_hist);
    int* totals = reinterpret_cast<int*>(ws + L.off_tot);
    int passes = 0, bits = 0;
    radix_shape(k, &passes, &bits);
    const int mask = (1 << bits) - 1;
    const int* kin = col_ind;
    const int* vin = nullptr;  // payload of the first pass: the element index
    int st = SPMM_OK;
    for (int pass = 0; pass < passes && st == SPMM_OK; ++pass) {
        const int shift = bits * pass;
        int* kout = kbuf[pass & 1];
        int* vout = ((passes - 1 - pass) % 2 == 0) ? perm : vtmp;  // the last pass lands in perm
        radix_hist_kernel<<<L.tiles, kSortThreads, 0, s>>>(kin, nnz, shift, mask, L.tiles, hist);
        st = launched(cudaGetLastError());
        if (st != SPMM_OK) break;
        digit_scan_kernel<<<mask + 1, kScanThreads, 0, s>>>(hist, L.tiles, totals);
        st = launched(cudaGetLastError());
        if (st != SPMM_OK) break;
        radix_scatter_kernel<<<L.tiles, kSortThreads, 0, s>>>(kin, vin, nnz, shift, mask, L.tiles, hist, totals, kout, vout);
        st = launched(cudaGetLastError());
        kin = kout;
        vin = vout;
    }
    if (st == SPMM_OK) {
        transpose_rowptr_kernel<<<(unsigned)(((long long)k + 1 + 255) / 256), 256, 0, s>>>(kin, nnz, k, row_ptr_t);
        st = launched(cudaGetLastError());
    }
    if (st == SPMM_OK) {  // col_ind_t[q] = row of perm[q]: rows expanded into the free key buffer, then gathered
        int* rows = kbuf[passes & 1];
        expand_rows_kernel<<<L.tiles, kSortThreads, 0, s>>>(row_ptr, m, (int)nnz, rows);
        st = launched(cudaGetLastError());
        if (st == SPMM_OK) {
            gather_values_kernel<int><<<(unsigned)std::min<long long>((nnz + 255) / 256, 152LL * 16), 256, 0, s>>>(
                perm, nnz, rows, col_ind_t);
            st = launched(cudaGetLastError());
        }
    }
    if (own) {
        const cudaError_t e = cudaFreeAsync(ws, s);
        if (st == SPMM_OK && e != cudaSuccess) st = status_of(e);
    }
    return st;
}

int spmm_gather_values(long long nnz, const int* perm, const void* vals, int vals_type, void* out, void* stream) {
    if (nnz < 0 || (nnz > 0 && (!perm || !vals || !out))) return SPMM_ERR_INVALID_VALUE;
    if (vals_type != SPMM_F32 && vals_type != SPMM_BF16 && vals_type != SPMM_F16) return SPMM_ERR_UNSUPPORTED;
    if (nnz == 0) return SPMM_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned blocks = (unsigned)std::min<long long>((nnz + 255) / 256, 152LL * 16);
    if (vals_type == SPMM_F32)
        gather_values_kernel<float><<<blocks, 256, 0, s>>>(perm, nnz, (const float*)vals, (float*)out);
    else
        gather_values_kernel<unsigned short><<<blocks, 256, 0, s>>>(perm, nnz, (const unsigned short*)vals,
                                                                     (unsigned short*)out);
    return launched(cudaGetLastError());
}

int sddmm_csr(int m, int k, int n, long long nnz, const int* row_ptr, const int* col_ind, const void* dC, int dc_type,
              long long lddc, const void* B, int b_type, long long ldb, void* out, int out_type, void* stream) {
    if (m < 0 || k < 0 || n < 0 || nnz < 0 || nnz > 0x7fffffffLL) return SPMM_ERR_INVALID_VALUE;
    if (nnz == 0) return SPMM_OK;
    if (!row_ptr || !col_ind || !out || m == 0 || k == 0) return SPMM_ERR_INVALID_VALUE;
    if (n > 0 && (!dC || !B || lddc < n || ldb < n)) return SPMM_ERR_INVALID_VALUE;
    if (dc_type != b_type) return SPMM_ERR_UNSUPPORTED;
    if (ldb * (b_type == SPMM_F32 ? 4LL : 2LL) > 0xffffffffLL) return SPMM_ERR_INVALID_VALUE;  // rows of B < 4 GiB apart
    SddmmArgs a{m, n, nnz, row_ptr, col_ind, dC, lddc, B, ldb, out, 32};
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) {  // empty dot products
        const int es = out_type == SPMM_F32 ? 4 : 2;
        return status_of(cudaMemsetAsync(out, 0, (size_t)nnz * es, s));
    }
    if (b_type == SPMM_F32 && out_type == SPMM_F32) return sddmm_run<float, float>(a, k, s);
    if (b_type == SPMM_BF16 && out_type == SPMM_BF16) return sddmm_run<__nv_bfloat16, __nv_bfloat16>(a, k, s);
    if (b_type == SPMM_BF16 && out_type == SPMM_F32) return sddmm_run<__nv_bfloat16, float>(a, k, s);
    if (b_type == SPMM_F16 && out_type == SPMM_F16) return sddmm_run<__half, __half>(a, k, s);
    if (b_type == SPMM_F16 && out_type == SPMM_F32) return sddmm_run<__half, float>(a, k, s);
    return SPMM_ERR_UNSUPPORTED;
}

}  // extern "C"
