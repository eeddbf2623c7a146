// Graph construction on the device: edge list -> A + I in CSR -> symmetric normalisation
// A_hat = D^-1/2 (A+I) D^-1/2 (Section 2.1 of the paper) -> CSR of the transpose (aliased when
// symmetric) -> degree-sorted row schedule.  Lists of up to ten million entries become a CSR in graph_buckets.cu; sorting, run-length
// and selection steps of larger ones, and the schedule's sort and scans, use CUB device primitives; everything else is a kernel in this file.
//
// What a build costs beside its kernels is memory and waiting: every temporary comes from the library's pool, the host
// waits twice (for the entry count, then for the schedule's counts), keys carry no more bits than the ids have
// (a radix pass over the keys costs as much as any other kernel here), and what the flags already say about the
// structure is not looked up.  The schedule looks the column blocks of a long row up once, keeps them for the segments, and orders those by
// 4,096 ranges of first columns (250 K nodes, 4.7 M entries: seg_count_kernel 46 -> 20 us, of which 7 were additions of single warps to one counter,
// seg_fill_kernel 47 -> 12, the order 45 -> 9); rows are sorted by as many bits as the longest has (43 -> 34).
// Builds of that list: 9.0 ms and more -> 0.68 -> 0.42 ms.
#include <cub/cub.cuh>

#include <atomic>
#include <new>
#include <type_traits>

#include "graph_values.cuh"
#include "internal.cuh"

using namespace mixgcn;

namespace {

uint64_t next_graph_uid() {
    static std::atomic<uint64_t> counter{0};
    return ++counter;
}

constexpr int TPB = 256;
inline unsigned blocks_for(int64_t n) { return (unsigned)((n + TPB - 1) / TPB); }

// flag bits written by validation kernels
enum { F_BAD_ID = 1, F_NOT_SYMMETRIC = 2, F_BAD_ROWPTR = 4, F_UNSORTED = 8, F_DROPPED = 16 };

// Keys (row << shift | column) of the entries; dropped edges become the sentinel n << shift, which sorts last.
template <typename Key>
__global__ void make_keys_kernel(int64_t n, int64_t m, const int32_t* __restrict__ src,
                                 const int32_t* __restrict__ dst, int sym, int self_loops, int shift,
                                 Key* __restrict__ keys, int32_t* flags) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) {
        const int32_t u = src[i], v = dst[i];
        const bool bad = u < 0 || v < 0 || u >= n || v >= n;
        const bool drop = bad || u == v;
        if (drop) atomicOr(flags, bad ? (F_BAD_ID | F_DROPPED) : F_DROPPED);
        const Key sentinel = (Key)n << shift;
        keys[i] = drop ? sentinel : (((Key)(uint32_t)u << shift) | (Key)(uint32_t)v);
        if (sym) keys[m + i] = drop ? sentinel : (((Key)(uint32_t)v << shift) | (Key)(uint32_t)u);
    }
    if (self_loops && i < n) keys[(sym ? 2 * m : m) + i] = ((Key)i << shift) | (Key)i;
}

// rowptr[q] = first position whose row id is >= q, from the sorted unique keys.
template <typename Key>
__global__ void rowptr_from_keys_kernel(int64_t n, int64_t nnz, int shift, const Key* __restrict__ keys,
                                        int64_t* __restrict__ rowptr, int32_t* __restrict__ col) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nnz) {
        const Key k = keys[i];
        const int64_t r = (int64_t)(k >> shift);
        const int64_t rp = i == 0 ? -1 : (int64_t)(keys[i - 1] >> shift);
        for (int64_t q = rp + 1; q <= r; ++q) rowptr[q] = i;
        col[i] = (int32_t)(uint32_t)(k & (((Key)1 << shift) - 1));
    } else if (i == nnz) {
        const int64_t last = nnz == 0 ? -1 : (int64_t)(keys[nnz - 1] >> shift);
        for (int64_t q = last + 1; q <= n; ++q) rowptr[q] = nnz;
    }
}

__global__ void degree_kernel(int64_t n, const int64_t* __restrict__ rowptr, int32_t* __restrict__ deg,
                              float* __restrict__ dinv) {
    int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n) return;
    int32_t d = (int32_t)(rowptr[u + 1] - rowptr[u]);
    deg[u] = d;
    dinv[u] = degree_norm(d);
}

// One warp per row.
__global__ void values_kernel(int64_t n, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                              const float* __restrict__ dinv, int norm, float* __restrict__ val) {
    int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (u >= n) return;
    const int64_t b = rowptr[u], e = rowptr[u + 1];
    const float du = dinv[u];
    for (int64_t i = b + lane; i < e; i += 32) val[i] = entry_value(norm, du, norm == 0 ? dinv[col[i]] : 0.0f, (int32_t)(e - b));
}

// One thread per entry, where the sorted keys still name its row: no row is too short or too long for its lanes
// (250 K nodes, 4.2 M entries: 68 -> 15 us).
template <typename Key>
__global__ void values_from_keys_kernel(int64_t nnz, int shift, const Key* __restrict__ keys, const int32_t* __restrict__ deg,
                                        const float* __restrict__ dinv, int norm, float* __restrict__ val) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nnz) return;
    const Key k = keys[i];
    const int64_t u = (int64_t)(k >> shift), v = (int64_t)(k & (((Key)1 << shift) - 1));
    val[i] = entry_value(norm, __ldg(dinv + u), norm == 0 ? __ldg(dinv + v) : 0.0f, norm == 1 ? __ldg(deg + u) : 0);
}

// For every stored (u,v), u != v, look v's row up for u.
__global__ void symmetry_kernel(int64_t n, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                int32_t* flags) {
    int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (u >= n) return;
    for (int64_t i = rowptr[u] + lane; i < rowptr[u + 1]; i += 32) {
        int32_t v = col[i];
        if (v == u) continue;
        int64_t lo = rowptr[v], hi = rowptr[v + 1];
        bool found = false;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            int32_t c = col[mid];
            if (c == (int32_t)u) { found = true; break; }
            if (c < (int32_t)u) lo = mid + 1; else hi = mid;
        }
        if (!found) { atomicOr(flags, F_NOT_SYMMETRIC); return; }
    }
}

// Rows that store their own diagonal entry (binary search of u in row u).
__global__ void diagonal_count_kernel(int64_t n, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                      unsigned long long* count) {
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool has = false;
    if (u < n) {
        int64_t lo = rowptr[u], hi = rowptr[u + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            const int32_t c = col[mid];
            if (c == (int32_t)u) { has = true; break; }
            if (c < (int32_t)u) lo = mid + 1; else hi = mid;
        }
    }
    const unsigned b = __ballot_sync(0xFFFFFFFFu, has);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(count, (unsigned long long)__popc(b));
}

__global__ void transpose_keys_kernel(int64_t n, int shift, const int64_t* __restrict__ rowptr,
                                      const int32_t* __restrict__ col, uint64_t* __restrict__ keys) {
    int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (u >= n) return;
    for (int64_t i = rowptr[u] + lane; i < rowptr[u + 1]; i += 32)
        keys[i] = ((uint64_t)(uint32_t)col[i] << shift) | (uint64_t)u;
}

// Sort key of a row: most entries first (top - entries); ties keep their ascending ids because the sort is stable.
__global__ void schedule_keys_kernel(int64_t row0, int64_t n_rows, uint32_t top, const int64_t* __restrict__ rowptr,
                                     uint32_t* __restrict__ keys, int32_t* __restrict__ ids) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_rows) return;
    const int64_t u = row0 + i;
    keys[i] = top - (uint32_t)(rowptr[u + 1] - rowptr[u]);
    ids[i] = (int32_t)u;
}

// What the host has to know of a schedule, counted on the device (integers, so the order of the atomics does not matter).
struct ScheduleCounts {
    unsigned long long rows_above_seg, rows_above[3], rows_heavy, total_segs, max_deg, bounds;
};

// Row counts of the buckets (one atomic per block and counter).
__global__ void schedule_counts_kernel(int64_t n, uint32_t top, const uint32_t* __restrict__ keys, int seg, ScheduleCounts* counts) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t d = i < n ? (int64_t)(top - keys[i]) : -1;
    if (i == 0) counts->max_deg = (unsigned long long)d;
    const int thr[5] = {seg, SPMM_PACK_DEG[0], SPMM_PACK_DEG[1], SPMM_PACK_DEG[2], SPMM_HEAVY};
    unsigned long long* const to[5] = {&counts->rows_above_seg, &counts->rows_above[0], &counts->rows_above[1], &counts->rows_above[2], &counts->rows_heavy};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const int rows = __syncthreads_count(d > thr[q]);
        if (threadIdx.x == 0 && rows) atomicAdd(to[q], (unsigned long long)rows);
    }
}

// Long rows are cut at dyadic column-block boundaries (and every seg entries): a row with d
// entries uses 2^k blocks, the largest k <= SPMM_MAX_LOG_BLOCKS with d / 2^k >= schedule_blk_min.
__device__ __forceinline__ int row_log_blocks(int64_t d, int64_t blk_min) {
    int k = 0;
    while (k < SPMM_MAX_LOG_BLOCKS && (d >> (k + 1)) >= blk_min) ++k;
    return k;
}

// The positions of N columns in a row of `len` entries (how many lie below each); the searches run side by side, a request each in flight.
template <int N>
__device__ __forceinline__ void lower_bounds(const int32_t* __restrict__ row, int32_t len, const int64_t (&key)[N], int32_t (&at)[N]) {
#pragma unroll
    for (int r = 0; r < N; ++r) at[r] = 0;
    for (int32_t step = 1 << (31 - __clz(len)); step > 0; step >>= 1) {
        int32_t c[N];
#pragma unroll
        for (int r = 0; r < N; ++r) c[r] = at[r] + step <= len ? __ldg(row + at[r] + step - 1) : 0x7FFFFFFF;
#pragma unroll
        for (int r = 0; r < N; ++r) if ((int64_t)c[r] < key[r]) at[r] += step;
    }
}

// Long rows: the number of segments of the i-th longest row (0 for rows that are not cut; i <= cap, a bound of the number of long rows), a warp
// per row, 32 column blocks at a time.  The first entry of every block is kept for seg_fill_kernel, the row's at bounds[bound_at[i]].
__global__ void __launch_bounds__(TPB) seg_count_kernel(int64_t n_cols, int64_t cap, const int32_t* __restrict__ perm, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, int seg,
                                 int64_t* __restrict__ row_segs, int32_t* __restrict__ bounds, int32_t* __restrict__ bound_at, ScheduleCounts* counts) {
    const int64_t i = ((int64_t)blockIdx.x * TPB + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ int room[TPB / 32], block_segs[TPB / 32];       // of the block's rows: one addition each to the counters
    int32_t segs = 0;
    const int64_t rb = i < cap ? rowptr[perm[i]] : 0, re = i < cap ? rowptr[perm[i] + 1] : 0;
    const int nb = re - rb > seg ? 1 << row_log_blocks(re - rb, schedule_blk_min(n_cols)) : 0;
    if (lane == 0) room[warp] = nb;
    __syncthreads();
    if (threadIdx.x == 0) {
        int all = 0;
        for (int k = 0; k < TPB / 32; ++k) { const int mine = room[k]; room[k] = all; all += mine; }
        const int first = all ? (int)atomicAdd(&counts->bounds, (unsigned long long)all) : 0;
        for (int k = 0; k < TPB / 32; ++k) room[k] += first;
    }
    __syncthreads();
    if (nb) {
        const int64_t width = (n_cols + nb - 1) / nb;
        const int at = room[warp];
        if (lane == 0) bound_at[i] = at;
        const int32_t len = (int32_t)(re - rb);
        auto blocks = [&](auto n_c) {          // n_c * 32 blocks at a time, from the last ones on, so that every block knows where the next one begins
            constexpr int N = decltype(n_c)::value;
            int32_t next_begin = len;
            for (int b0 = nb > N * 32 ? nb - N * 32 : 0;; b0 -= N * 32) {
                int64_t key[N];
                int32_t lo[N];
#pragma unroll
                for (int r = 0; r < N; ++r) key[r] = (int64_t)(b0 + r * 32 + lane) * width;       // (past the last block: past the last column)
                lower_bounds<N>(col + rb, len, key, lo);
#pragma unroll
                for (int r = N - 1; r >= 0; --r) {
                    const int b = b0 + r * 32 + lane;
                    if (b < nb) bounds[at + b] = lo[r];
                    const int32_t next = __shfl_down_sync(0xFFFFFFFFu, lo[r], 1), hi = lane == 31 ? next_begin : next;
                    segs += (hi - lo[r] + seg - 1) / seg;
                    next_begin = __shfl_sync(0xFFFFFFFFu, lo[r], 0);
                }
                if (b0 == 0) break;
            }
        };
        if (nb <= 32) blocks(std::integral_constant<int, 1>());
        else blocks(std::integral_constant<int, 4>());
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) segs += __shfl_xor_sync(0xFFFFFFFFu, segs, o);
    }
    if (lane == 0) {
        if (i <= cap) row_segs[i] = segs;
        block_segs[warp] = segs;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long all = 0;
        for (int k = 0; k < TPB / 32; ++k) all += (unsigned long long)block_segs[k];
        if (all) atomicAdd(&counts->total_segs, all);
    }
}

// Segments run in order of their first columns, as far as SEG_BINS ranges of columns tell them apart: their order decides what the L2 holds, not
// what is added up.
constexpr int SEG_BINS = 4096;
__device__ __forceinline__ int seg_bin(int64_t n_cols, int32_t c) { return (int)((int64_t)c * SEG_BINS / n_cols); }

__global__ void seg_fill_kernel(int64_t n_cols, int64_t n_long, const int32_t* __restrict__ perm, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col, int seg,
                                const int64_t* __restrict__ seg_off, const int32_t* __restrict__ bounds, const int32_t* __restrict__ bound_at,
                                SpmmRec* __restrict__ rec_tmp, int32_t* __restrict__ bin_of, uint32_t* __restrict__ bins) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n_long) return;
    const int lane = threadIdx.x & 31;
    const int64_t u = perm[i], rb = rowptr[u], re = rowptr[u + 1];
    const int nb = 1 << row_log_blocks(re - rb, schedule_blk_min(n_cols));
    const int32_t* mine = bounds + bound_at[i];
    int64_t q0 = seg_off[i];
    for (int b0 = 0; b0 < nb; b0 += 32) {
        const int b = b0 + lane;
        const int64_t lo = b < nb ? rb + mine[b] : re, hi = b + 1 < nb ? rb + mine[b + 1] : re;
        const int segs = (int)((hi - lo + seg - 1) / seg);
        int incl = segs;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        int64_t q = q0 + incl - segs;
        for (int64_t pos = lo; pos < hi; pos += seg, ++q) {
            SpmmRec x; x.begin = pos; x.len = (int32_t)((hi - pos) < seg ? (hi - pos) : seg); x.row = (int32_t)i;
            rec_tmp[q] = x;
            const int bin = seg_bin(n_cols, col[pos]);
            bin_of[q] = bin;
            atomicAdd(&bins[bin], 1u);
        }
        q0 += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
}

__global__ void __launch_bounds__(SEG_BINS / 4) seg_bins_kernel(uint32_t* __restrict__ bins) {      // counts -> first positions
    using Scan = cub::BlockScan<uint32_t, SEG_BINS / 4>;
    __shared__ typename Scan::TempStorage temp;
    uint4 c = reinterpret_cast<uint4*>(bins)[threadIdx.x];
    uint32_t x[4] = {c.x, c.y, c.z, c.w};
    Scan(temp).ExclusiveSum(x, x);
    reinterpret_cast<uint4*>(bins)[threadIdx.x] = make_uint4(x[0], x[1], x[2], x[3]);
}

__global__ void seg_place_kernel(int64_t total_segs, const int32_t* __restrict__ bin_of, const SpmmRec* __restrict__ rec_tmp, uint32_t* __restrict__ bins,
                                 SpmmRec* __restrict__ rec, int64_t* __restrict__ seg_pos) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= total_segs) return;
    const uint32_t pos = atomicAdd(&bins[bin_of[q]], 1u);
    rec[pos] = rec_tmp[q];
    seg_pos[q] = pos;
}

// Ordinary rows: one record each, in perm order, after the segment records.
__global__ void fill_records_kernel(int64_t n, int64_t n_long, int64_t total_segs, const int32_t* __restrict__ perm,
                                    const int64_t* __restrict__ rowptr, SpmmRec* __restrict__ rec) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || i < n_long) return;
    const int64_t u = perm[i];
    SpmmRec x; x.begin = rowptr[u]; x.len = (int32_t)(rowptr[u + 1] - rowptr[u]); x.row = (int32_t)u;
    rec[total_segs + (i - n_long)] = x;
}

__global__ void validate_csr_kernel(int64_t n, int64_t nnz, const int64_t* __restrict__ rowptr,
                                    const int32_t* __restrict__ col, int32_t* flags) {
    int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= n) return;
    int64_t b = rowptr[u], e = rowptr[u + 1];
    if ((u == 0 && b != 0) || b < 0 || e < b || e > nnz) { atomicOr(flags, F_BAD_ROWPTR); return; }
    if (e - b > 0x7FFFFFFFll) { atomicOr(flags, F_BAD_ROWPTR); return; }
    for (int64_t i = b; i < e; ++i) {
        int32_t c = col[i];
        if (c < 0 || c >= n) { atomicOr(flags, F_BAD_ID); return; }
        if (i > b && col[i - 1] >= c) { atomicOr(flags, F_UNSORTED); return; }
    }
}

int bits_for(uint64_t x) { int b = 0; while (x) { ++b; x >>= 1; } return b; }

// (these release memory that kernels on any stream may have used: callers synchronise the device first)
void free_schedule(SpmmSchedule& v) {
    dev_free(v.perm, nullptr); dev_free(v.rec, nullptr); dev_free(v.seg_off, nullptr); dev_free(v.seg_pos, nullptr);
    v = SpmmSchedule{};
}

void free_view(CsrView& v) {
    dev_free(v.rowptr, nullptr); dev_free(v.col, nullptr); dev_free(v.val, nullptr);
    free_schedule(v.full);
    for (int k = 0; k < v.n_chunk; ++k) free_schedule(v.chunk[k]);
    delete[] v.chunk;
    v = CsrView{};
}

// Schedule of rows [row0, row0 + n) of the CSR (rowptr, col) of a matrix with n_total columns and nnz entries in all
// rows (a row chunk is cut like the whole matrix, so that its sums are the same).
// max_deg: what no row exceeds (a pass of the sort less for every eight bits).
mixgcn_status build_schedule(int64_t n_total, int64_t nnz, int64_t max_deg, const int64_t* rowptr, const int32_t* col, int64_t row0, int64_t n,
                             SpmmSchedule& v, cudaStream_t s) {
    v = SpmmSchedule{};
    v.row0 = row0; v.n_rows = n; v.seg = schedule_seg(nnz);
    if (n <= 0) return MIXGCN_OK;
    // rows by descending entry count; the bucket counts; the segments each long row will need
    const int deg_bits = bits_for((uint64_t)(max_deg > 0 ? max_deg : 1));
    const uint32_t top = (uint32_t)(((uint64_t)1 << deg_bits) - 1);
    int64_t cap = nnz / (v.seg + 1);                                       // no more rows than this are long
    if (cap > n) cap = n;
    DevBuf k0(s), k1(s), ids(s), tmp(s), counts(s), row_segs(s), bounds(s), bound_at(s);
    MIXGCN_TRY(k0.alloc(n * (int64_t)sizeof(uint32_t)));
    MIXGCN_TRY(k1.alloc(n * (int64_t)sizeof(uint32_t)));
    MIXGCN_TRY(ids.alloc(n * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(counts.alloc(sizeof(ScheduleCounts)));
    MIXGCN_TRY(row_segs.alloc((cap + 1) * (int64_t)sizeof(int64_t)));
    // (a long row has a block per blk_min of its entries at most, or one)
    MIXGCN_TRY(bounds.alloc((nnz / schedule_blk_min(n_total) + cap) * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(bound_at.alloc(cap * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(dev_alloc((void**)&v.perm, n * (int64_t)sizeof(int32_t), s));
    MIXGCN_CUDA(cudaMemsetAsync(counts.p, 0, sizeof(ScheduleCounts), s));
    schedule_keys_kernel<<<blocks_for(n), TPB, 0, s>>>(row0, n, top, rowptr, k0.as<uint32_t>(), ids.as<int32_t>());
    size_t tb = 0;
    MIXGCN_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tb, k0.as<uint32_t>(), k1.as<uint32_t>(), ids.as<int32_t>(), v.perm, n, 0, deg_bits, s));
    MIXGCN_TRY(tmp.alloc((int64_t)tb));
    MIXGCN_CUDA(cub::DeviceRadixSort::SortPairs(tmp.p, tb, k0.as<uint32_t>(), k1.as<uint32_t>(), ids.as<int32_t>(), v.perm, n, 0, deg_bits, s));
    schedule_counts_kernel<<<blocks_for(n), TPB, 0, s>>>(n, top, k1.as<uint32_t>(), v.seg, counts.as<ScheduleCounts>());
    if (cap > 0)
        seg_count_kernel<<<blocks_for((cap + 1) * 32), TPB, 0, s>>>(n_total, cap, v.perm, rowptr, col, v.seg, row_segs.as<int64_t>(), bounds.as<int32_t>(), bound_at.as<int32_t>(),
                                                                        counts.as<ScheduleCounts>());
    ScheduleCounts h{};
    MIXGCN_CUDA(cudaMemcpyAsync(&h, counts.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    v.n_long = (int64_t)h.rows_above_seg;
    v.n_heavy = (int64_t)h.rows_heavy;
    for (int q = 0; q < 3; ++q) v.rows_above[q] = (int64_t)h.rows_above[q];
    v.max_deg = (int32_t)h.max_deg;
    const int64_t nl = v.n_long, total = (int64_t)h.total_segs;
    if (total >= 0xFFFFFFFFll) MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "graph schedule: too many long-row segments (%lld)", (long long)total);
    v.total_segs = total;
    MIXGCN_TRY(dev_alloc((void**)&v.seg_off, (nl + 1) * (int64_t)sizeof(int64_t), s));
    MIXGCN_TRY(dev_alloc((void**)&v.rec, (total + n - nl + 1) * (int64_t)sizeof(SpmmRec), s));
    MIXGCN_TRY(dev_alloc((void**)&v.seg_pos, (total + 1) * (int64_t)sizeof(int64_t), s));
    if (total > 0) {
        // segments of the long rows, in order of their first column
        DevBuf rec_tmp(s), bin_of(s), bins(s), tmp2(s);
        MIXGCN_TRY(rec_tmp.alloc(total * (int64_t)sizeof(SpmmRec)));
        MIXGCN_TRY(bin_of.alloc(total * (int64_t)sizeof(int32_t)));
        MIXGCN_TRY(bins.alloc(SEG_BINS * sizeof(uint32_t)));
        MIXGCN_CUDA(cudaMemsetAsync(bins.p, 0, SEG_BINS * sizeof(uint32_t), s));
        size_t tb_scan = 0;
        MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb_scan, row_segs.as<int64_t>(), v.seg_off, nl + 1, s));
        MIXGCN_TRY(tmp2.alloc((int64_t)tb_scan));
        MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(tmp2.p, tb_scan, row_segs.as<int64_t>(), v.seg_off, nl + 1, s));
        seg_fill_kernel<<<blocks_for(nl * 32), TPB, 0, s>>>(n_total, nl, v.perm, rowptr, col, v.seg, v.seg_off, bounds.as<int32_t>(), bound_at.as<int32_t>(),
                                                           rec_tmp.as<SpmmRec>(), bin_of.as<int32_t>(), bins.as<uint32_t>());
        seg_bins_kernel<<<1, SEG_BINS / 4, 0, s>>>(bins.as<uint32_t>());
        seg_place_kernel<<<blocks_for(total), TPB, 0, s>>>(total, bin_of.as<int32_t>(), rec_tmp.as<SpmmRec>(), bins.as<uint32_t>(), v.rec, v.seg_pos);
    } else {
        MIXGCN_CUDA(cudaMemsetAsync(v.seg_off, 0, (nl + 1) * sizeof(int64_t), s));
    }
    fill_records_kernel<<<blocks_for(n), TPB, 0, s>>>(n, nl, total, v.perm, rowptr, v.rec);
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

// Degrees and room for the values of a graph whose rowptr exists.
mixgcn_status fill_degrees(mixgcn_graph* g, cudaStream_t s) {
    if (!g->deg) MIXGCN_TRY(dev_alloc((void**)&g->deg, g->n * (int64_t)sizeof(int32_t), s));
    if (!g->dinv) MIXGCN_TRY(dev_alloc((void**)&g->dinv, g->n * (int64_t)sizeof(float), s));
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.val, (g->nnz > 0 ? g->nnz : 1) * (int64_t)sizeof(float), s));
    degree_kernel<<<blocks_for(g->n), TPB, 0, s>>>(g->n, g->fwd.rowptr, g->deg, g->dinv);
    return MIXGCN_OK;
}

// Everything after the CSR exists: symmetry, transpose, schedules.  known_symmetric / known_diagonal:
// what the caller already knows of the structure (-1: look); max_deg: what no row exceeds.  Leaves work in flight on `s`.
mixgcn_status finish_graph(mixgcn_graph* g, int known_symmetric, int known_diagonal, int64_t max_deg, cudaStream_t s) {
    const int64_t n = g->n, nnz = g->nnz;
    CsrView& A = g->fwd;
    g->symmetric = known_symmetric; g->has_diagonal = known_diagonal;
    if (known_symmetric < 0 || known_diagonal < 0) {
        struct Looked { unsigned long long diagonal; int32_t flags; } h{};
        DevBuf looked(s);
        MIXGCN_TRY(looked.alloc(sizeof(Looked)));
        MIXGCN_CUDA(cudaMemsetAsync(looked.p, 0, sizeof(Looked), s));
        Looked* d = looked.as<Looked>();
        if (known_symmetric < 0) symmetry_kernel<<<blocks_for(n * 32), TPB, 0, s>>>(n, A.rowptr, A.col, &d->flags);
        if (known_diagonal < 0) diagonal_count_kernel<<<blocks_for(n), TPB, 0, s>>>(n, A.rowptr, A.col, &d->diagonal);
        MIXGCN_CUDA(cudaMemcpyAsync(&h, looked.p, sizeof(h), cudaMemcpyDeviceToHost, s));
        MIXGCN_CUDA(cudaStreamSynchronize(s));
        if (known_symmetric < 0) g->symmetric = (h.flags & F_NOT_SYMMETRIC) ? 0 : 1;
        if (known_diagonal < 0) g->has_diagonal = h.diagonal == (unsigned long long)n ? 1 : (h.diagonal == 0 ? 0 : 2);
    }
    MIXGCN_TRY(build_schedule(n, nnz, max_deg, A.rowptr, A.col, 0, n, A.full, s));
    g->bwd_is_fwd = (g->symmetric && g->norm != 1) ? 1 : 0;   // row-mean values are not symmetric: A_hat^T needs its own copy
    if (g->bwd_is_fwd) {
        g->bwd = A;  // alias: the same index serves the backward aggregation
        return MIXGCN_OK;
    }
    // Transposed structure: sort (col,row) keys carrying the value.
    CsrView& T = g->bwd;
    DevBuf k0(s), k1(s), tmp(s);
    const int64_t cap = nnz > 0 ? nnz : 1;
    MIXGCN_TRY(k0.alloc(cap * (int64_t)sizeof(uint64_t)));
    MIXGCN_TRY(k1.alloc(cap * (int64_t)sizeof(uint64_t)));
    MIXGCN_TRY(dev_alloc((void**)&T.val, cap * (int64_t)sizeof(float), s));
    MIXGCN_TRY(dev_alloc((void**)&T.rowptr, (n + 1) * (int64_t)sizeof(int64_t), s));
    MIXGCN_TRY(dev_alloc((void**)&T.col, cap * (int64_t)sizeof(int32_t), s));
    const int shift = bits_for((uint64_t)n);
    transpose_keys_kernel<<<blocks_for(n * 32), TPB, 0, s>>>(n, shift, A.rowptr, A.col, k0.as<uint64_t>());
    size_t tb = 0;
    MIXGCN_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tb, k0.as<uint64_t>(), k1.as<uint64_t>(), A.val, T.val,
                                                nnz, shift, 2 * shift, s));
    MIXGCN_TRY(tmp.alloc((int64_t)tb));
    // the keys are made in row order and the sort is stable: sorting by the column part leaves the rows ascending
    MIXGCN_CUDA(cub::DeviceRadixSort::SortPairs(tmp.p, tb, k0.as<uint64_t>(), k1.as<uint64_t>(), A.val, T.val,
                                                nnz, shift, 2 * shift, s));
    rowptr_from_keys_kernel<uint64_t><<<blocks_for(nnz + 1), TPB, 0, s>>>(n, nnz, shift, k1.as<uint64_t>(), T.rowptr, T.col);
    return build_schedule(n, nnz, n, T.rowptr, T.col, 0, n, T.full, s);
}

// Edge list (on the device) -> CSR of the graph: keys, sort, unique, values.
template <typename Key>
mixgcn_status csr_from_edges(mixgcn_graph* g, int64_t m, const int32_t* src, const int32_t* dst, int sym, int self, cudaStream_t s) {
    const int64_t n = g->n, total = m * (sym ? 2 : 1) + (self ? n : 0);
    struct Counted { int64_t unique; int32_t flags; } h{};
    DevBuf k0(s), k1(s), tmp(s), counted(s);
    MIXGCN_TRY(k0.alloc(total * (int64_t)sizeof(Key)));
    MIXGCN_TRY(k1.alloc(total * (int64_t)sizeof(Key)));
    MIXGCN_TRY(counted.alloc(sizeof(Counted)));
    Counted* d = counted.as<Counted>();
    MIXGCN_CUDA(cudaMemsetAsync(d, 0, sizeof(Counted), s));
    const int shift = bits_for((uint64_t)n);
    const int64_t work = m > n ? m : n;
    make_keys_kernel<Key><<<blocks_for(work), TPB, 0, s>>>(n, m, src, dst, sym, self, shift, k0.as<Key>(), &d->flags);
    size_t tb_sort = 0, tb_uniq = 0;
    MIXGCN_CUDA(cub::DeviceRadixSort::SortKeys(nullptr, tb_sort, k0.as<Key>(), k1.as<Key>(), total, 0, 2 * shift, s));
    MIXGCN_CUDA(cub::DeviceSelect::Unique(nullptr, tb_uniq, k1.as<Key>(), k0.as<Key>(), &d->unique, total, s));
    size_t tb = tb_sort > tb_uniq ? tb_sort : tb_uniq;
    MIXGCN_TRY(tmp.alloc((int64_t)tb));
    MIXGCN_CUDA(cub::DeviceRadixSort::SortKeys(tmp.p, tb, k0.as<Key>(), k1.as<Key>(), total, 0, 2 * shift, s));
    MIXGCN_CUDA(cub::DeviceSelect::Unique(tmp.p, tb, k1.as<Key>(), k0.as<Key>(), &d->unique, total, s));
    MIXGCN_CUDA(cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    if (h.flags & F_BAD_ID) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create: a node id lies outside [0, %lld)", (long long)n);
    const int64_t nnz = total == 0 ? 0 : h.unique - ((h.flags & F_DROPPED) ? 1 : 0);     // dropped edges left one sentinel, the last key
    g->nnz = nnz;
    if (!g->fwd.rowptr) MIXGCN_TRY(dev_alloc((void**)&g->fwd.rowptr, (n + 1) * (int64_t)sizeof(int64_t), s));
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.col, (nnz > 0 ? nnz : 1) * (int64_t)sizeof(int32_t), s));
    rowptr_from_keys_kernel<Key><<<blocks_for(nnz + 1), TPB, 0, s>>>(n, nnz, shift, k0.as<Key>(), g->fwd.rowptr, g->fwd.col);
    MIXGCN_TRY(fill_degrees(g, s));
    if (nnz > 0) values_from_keys_kernel<Key><<<blocks_for(nnz), TPB, 0, s>>>(nnz, shift, k0.as<Key>(), g->deg, g->dinv, g->norm, g->fwd.val);
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

mixgcn_status check_common(mixgcn_ctx* ctx, int64_t n, mixgcn_graph** out) {
    if (!ctx || !out) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_create: null ctx or out");
    if (n <= 0) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_create: n must be positive (got %lld)", (long long)n);
    if (n >= 0x7FFFFFFFll) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create: n = %lld does not fit int32 ids", (long long)n);
    return MIXGCN_OK;
}

}  // namespace

namespace mixgcn {

mixgcn_status build_view_schedule(int64_t n_cols, int64_t n, int64_t nnz, CsrView& v, cudaStream_t s) {
    return build_schedule(n_cols, nnz, n_cols, v.rowptr, v.col, 0, n, v.full, s);
}

void release_view(CsrView& v) { free_view(v); }

mixgcn_status ensure_chunk_schedules(const mixgcn_graph* g, const CsrView& A_const, int chunks) {
    // a cache inside the graph object; a symmetric graph keeps one set (in fwd) and mirrors it into the alias
    CsrView& A = const_cast<CsrView&>(g->bwd_is_fwd ? g->fwd : A_const);
    if (chunks <= 1 || A.n_chunk == chunks) return MIXGCN_OK;
    MIXGCN_CUDA(cudaDeviceSynchronize());         // earlier launches may still read the schedules being replaced
    if (A.n_chunk) memory_given_back(g->memory);  // recorded ones too
    for (int k = 0; k < A.n_chunk; ++k) free_schedule(A.chunk[k]);
    delete[] A.chunk;
    A.chunk = nullptr; A.n_chunk = 0;
    SpmmSchedule* sc = new (std::nothrow) SpmmSchedule[chunks]();
    if (!sc) MIXGCN_FAIL(MIXGCN_ENOMEM, "chunk schedules: host allocation failed");
    cudaStream_t s = g->ctx->side_stream[0];
    for (int k = 0; k < chunks; ++k) {
        const int64_t r0 = (g->n * (int64_t)k) / chunks, r1 = (g->n * (int64_t)(k + 1)) / chunks;
        mixgcn_status st = build_schedule(g->n, g->nnz, A.full.max_deg, A.rowptr, A.col, r0, r1 - r0, sc[k], s);
        if (st == MIXGCN_OK && cudaStreamSynchronize(s) != cudaSuccess) st = MIXGCN_ECUDA;    // usable on every stream from here on
        if (st != MIXGCN_OK) {
            cudaStreamSynchronize(s);         // kernels that write to them
            for (int q = 0; q <= k; ++q) free_schedule(sc[q]);
            delete[] sc;
            return st;
        }
    }
    A.chunk = sc; A.n_chunk = chunks;
    if (g->bwd_is_fwd) const_cast<mixgcn_graph*>(g)->bwd = g->fwd;   // keep the alias in step
    return MIXGCN_OK;
}

}  // namespace mixgcn

extern "C" mixgcn_status mixgcn_graph_destroy(mixgcn_graph* g) {
    if (!g) return MIXGCN_OK;
    memory_given_back(g->memory);
    cudaSetDevice(g->device);
    cudaDeviceSynchronize();          // launches that read the graph may still be in flight on any stream
    release_tiles(g);
    if (!g->bwd_is_fwd) free_view(g->bwd);
    free_view(g->fwd);
    dev_free(g->deg, nullptr);
    dev_free(g->dinv, nullptr);
    delete g;
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_graph_create(mixgcn_ctx* ctx, int64_t n, int64_t m, const int32_t* src,
                                             const int32_t* dst, uint32_t flags, mixgcn_graph** out) {
    MIXGCN_TRY(check_common(ctx, n, out));
    if (m < 0 || (m > 0 && (!src || !dst))) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_create: bad edge list (m=%lld)", (long long)m);
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->side_stream[0];
    if ((flags & MIXGCN_GRAPH_NORM_ROW) && (flags & MIXGCN_GRAPH_NORM_NONE)) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_create: NORM_ROW and NORM_NONE exclude each other");
    const int sym = (flags & MIXGCN_GRAPH_SYMMETRISE) != 0, self = (flags & MIXGCN_GRAPH_ADD_SELF_LOOPS) != 0;

    mixgcn_graph* g = new (std::nothrow) mixgcn_graph();
    if (g) g->uid = next_graph_uid();
    if (!g) MIXGCN_FAIL(MIXGCN_ENOMEM, "graph_create: host allocation failed");
    g->ctx = ctx; g->device = ctx->device; g->n = n; g->nnz = 0; g->symmetric = 1; g->bwd_is_fwd = 1;
    g->norm = (flags & MIXGCN_GRAPH_NORM_ROW) ? 1 : ((flags & MIXGCN_GRAPH_NORM_NONE) ? 2 : 0);
    struct Guard { mixgcn_graph* g; bool keep = false; ~Guard() { if (!keep) { g->bwd_is_fwd = g->bwd.rowptr == g->fwd.rowptr; mixgcn_graph_destroy(g); } } } guard{g};
    MIXGCN_TRY(new_generation(&g->memory));
    LaunchScope scope(ctx, PH_GRAPH, s, 12);

    DevBuf dsrc(s), ddst(s);
    const int32_t *ps = src, *pd = dst;
    if (!(flags & MIXGCN_GRAPH_EDGES_ON_DEVICE) && m > 0) {
        MIXGCN_TRY(dsrc.alloc(m * (int64_t)sizeof(int32_t)));
        MIXGCN_TRY(ddst.alloc(m * (int64_t)sizeof(int32_t)));
        MIXGCN_CUDA(cudaMemcpyAsync(dsrc.p, src, m * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        MIXGCN_CUDA(cudaMemcpyAsync(ddst.p, dst, m * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        ps = dsrc.as<int32_t>(); pd = ddst.as<int32_t>();
    }
    bool built = false;
    int64_t max_deg = n;               // a row has at most n entries
    MIXGCN_TRY(csr_from_buckets(g, m, ps, pd, sym, self, s, &built, &max_deg));
    // two ids fit one 32-bit key on graphs of fewer than 2^16 nodes: half the bytes per radix pass
    if (built) {}
    else if (2 * bits_for((uint64_t)n) <= 32) MIXGCN_TRY(csr_from_edges<uint32_t>(g, m, ps, pd, sym, self, s));
    else MIXGCN_TRY(csr_from_edges<uint64_t>(g, m, ps, pd, sym, self, s));
    dsrc.release(); ddst.release();
    // self loops of the input are dropped, so the flags decide what lies on the diagonal; a directed list may still be symmetric
    MIXGCN_TRY(finish_graph(g, sym ? 1 : -1, self ? 1 : 0, max_deg, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    guard.keep = true;
    *out = g;
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_graph_create_from_csr(mixgcn_ctx* ctx, int64_t n, const int64_t* rowptr,
                                                      const int32_t* col, uint32_t flags, mixgcn_graph** out) {
    MIXGCN_TRY(check_common(ctx, n, out));
    if (!rowptr) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_create_from_csr: null rowptr");
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = ctx->side_stream[0];
    const bool on_dev = (flags & MIXGCN_GRAPH_EDGES_ON_DEVICE) != 0;
    const cudaMemcpyKind kind = on_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    int64_t nnz = 0;
    MIXGCN_CUDA(cudaMemcpy(&nnz, rowptr + n, sizeof(int64_t), on_dev ? cudaMemcpyDeviceToHost : cudaMemcpyHostToHost));
    if (nnz < 0) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create_from_csr: rowptr[n] is negative");
    if (nnz > 0 && !col) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_create_from_csr: null col");

    mixgcn_graph* g = new (std::nothrow) mixgcn_graph();
    if (g) g->uid = next_graph_uid();
    if (!g) MIXGCN_FAIL(MIXGCN_ENOMEM, "graph_create_from_csr: host allocation failed");
    g->ctx = ctx; g->device = ctx->device; g->n = n; g->nnz = nnz; g->symmetric = 1; g->bwd_is_fwd = 1;
    g->norm = (flags & MIXGCN_GRAPH_NORM_ROW) ? 1 : ((flags & MIXGCN_GRAPH_NORM_NONE) ? 2 : 0);
    struct Guard { mixgcn_graph* g; bool keep = false; ~Guard() { if (!keep) { g->bwd_is_fwd = g->bwd.rowptr == g->fwd.rowptr; mixgcn_graph_destroy(g); } } } guard{g};
    MIXGCN_TRY(new_generation(&g->memory));
    LaunchScope scope(ctx, PH_GRAPH, s, 8);
    DevBuf fl(s);
    MIXGCN_TRY(fl.alloc(sizeof(int32_t)));
    MIXGCN_CUDA(cudaMemsetAsync(fl.p, 0, sizeof(int32_t), s));
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.rowptr, (n + 1) * (int64_t)sizeof(int64_t), s));
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.col, (nnz > 0 ? nnz : 1) * (int64_t)sizeof(int32_t), s));
    MIXGCN_CUDA(cudaMemcpyAsync(g->fwd.rowptr, rowptr, (n + 1) * sizeof(int64_t), kind, s));
    if (nnz > 0) MIXGCN_CUDA(cudaMemcpyAsync(g->fwd.col, col, nnz * sizeof(int32_t), kind, s));
    // rowptr must be validated before col is indexed with it: first monotonicity on the host side
    // of the device array (cheap kernel), then the per-row column checks.
    validate_csr_kernel<<<blocks_for(n), TPB, 0, s>>>(n, nnz, g->fwd.rowptr, g->fwd.col, fl.as<int32_t>());
    int32_t hf = 0;
    MIXGCN_CUDA(cudaMemcpyAsync(&hf, fl.p, sizeof(hf), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    if (hf & F_BAD_ROWPTR) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create_from_csr: rowptr is not monotone from 0");
    if (hf & F_BAD_ID) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create_from_csr: a column id lies outside [0, %lld)", (long long)n);
    if (hf & F_UNSORTED) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create_from_csr: columns are not strictly ascending in a row");
    MIXGCN_TRY(fill_degrees(g, s));
    values_kernel<<<blocks_for(n * 32), TPB, 0, s>>>(n, g->fwd.rowptr, g->fwd.col, g->dinv, g->norm, g->fwd.val);
    MIXGCN_TRY(finish_graph(g, -1, -1, n, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    guard.keep = true;
    *out = g;
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_graph_info(const mixgcn_graph* g, int64_t* n, int64_t* nnz, int32_t* max_deg,
                                           int32_t* symmetric) {
    if (!g) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_info: null graph");
    if (n) *n = g->n;
    if (nnz) *nnz = g->nnz;
    if (max_deg) *max_deg = g->fwd.full.max_deg;
    if (symmetric) *symmetric = g->symmetric;
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_graph_export(const mixgcn_graph* g, int transposed, int64_t* rowptr, int32_t* col,
                                             float* val, int32_t* deg, float* dinv) {
    if (!g) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_export: null graph");
    MIXGCN_CUDA(cudaSetDevice(g->ctx->device));
    MIXGCN_CUDA(cudaDeviceSynchronize());
    const CsrView& v = transposed ? g->bwd : g->fwd;
    if (rowptr) MIXGCN_CUDA(cudaMemcpy(rowptr, v.rowptr, (g->n + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost));
    if (col && g->nnz) MIXGCN_CUDA(cudaMemcpy(col, v.col, g->nnz * sizeof(int32_t), cudaMemcpyDeviceToHost));
    if (val && g->nnz) MIXGCN_CUDA(cudaMemcpy(val, v.val, g->nnz * sizeof(float), cudaMemcpyDeviceToHost));
    if (deg) MIXGCN_CUDA(cudaMemcpy(deg, g->deg, g->n * sizeof(int32_t), cudaMemcpyDeviceToHost));
    if (dinv) MIXGCN_CUDA(cudaMemcpy(dinv, g->dinv, g->n * sizeof(float), cudaMemcpyDeviceToHost));
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_graph_export_schedule(const mixgcn_graph* g, int transposed, int32_t* perm) {
    if (!g || !perm) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_export_schedule: null argument");
    MIXGCN_CUDA(cudaSetDevice(g->ctx->device));
    MIXGCN_CUDA(cudaDeviceSynchronize());
    const CsrView& v = transposed ? g->bwd : g->fwd;
    MIXGCN_CUDA(cudaMemcpy(perm, v.full.perm, g->n * sizeof(int32_t), cudaMemcpyDeviceToHost));
    return MIXGCN_OK;
}
