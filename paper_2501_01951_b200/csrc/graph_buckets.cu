// Edge list -> CSR for graphs of up to ten million entries: rows in buckets that a block of threads sorts in shared memory.
//
// A radix sort of the keys of the whole list passes over them five times and more (250 K nodes, 4.7 M entries: 302 us, with unique,
// row pointers and values 365), because every pass goes by eight bits.  Here an entry goes to the bucket of its row at once, as (row in the
// bucket, column) in 32 bits, in no particular order; a block then sorts a bucket, drops duplicates and counts its rows, and once the host
// knows how many entries there are the buckets are read once more into columns and values.  Two passes over the edges, two over
// the entries: 14 + 34 + 60 + 9 + 45 us of the same list.  The result is a sorted set, so it does not depend on the order in which entries arrived.
//
// Rows are spread over the buckets by a multiplicative hash (a bijection of the ids), so that neighbouring hubs do not meet.  In a bucket a
// row of n entries has a power of two between n / 4 and n / 2 of bins, by the highest bits of the columns; entries are counted into bins
// and put there, a thread sorts a bin of up to eight, and a warp what ids that lie close together make larger (bitonic, 128 at a time in
// registers).  Where a bucket has no room for its longest rows they are marked in a bitmap of the columns instead, one after the other.
//
// Bound: short dependent kernels, latency of scattered requests and shared-memory atomics.  Buckets hold 5,000 entries at most on average,
// so that every SM has several blocks; there are at most 2,048, whose counters a block keeps in shared memory while it scatters.  That
// is where the line to the radix sort lies.  Lists with a bucket of more than 64 K entries go there as well (a hub of as many neighbours: a
// block would pass over them alone, a star of a million 3.0 ms against 0.77).  Whole builds, radix sort : buckets (us): 2 K nodes, 21 K entries 255 :
// 234;  5 K, 1.5 M 369 : 302;  50 K, 5.2 M 519 : 414;  250 K, 4.7 M 682 : 400;  300 K, 9.4 M 985 : 544;  1 M, 4.3 M 654 : 482;  1 M, 9.3 M 1057 : 633;  ends drawn by
// rank^-0.7, neighbouring ids, 200 K, 6 M 795 : 494;  by rank^-1, largest row 63 K, 2.7 M 689 : 668;  a star of a million, after the look at it, 764 : 796.
// (Instead of bins, for 4.7 M entries: three passes of nine bits over a bucket 147 us, rows sorted one by one in registers and shared memory
// 155; entries scattered as they come instead of in runs 48.)
#include <cub/block/block_scan.cuh>
#include <cub/device/device_scan.cuh>

#include "graph_values.cuh"
#include "internal.cuh"

using namespace mixgcn;

namespace {

constexpr int TPB = 512, EDGES = 14;                    // edges of a thread of the scatter, at most
constexpr int BUCKETS_MAX = 2048, ROWS_LOG_MAX = 11, ROWS_MAX = 1 << ROWS_LOG_MAX;
constexpr int AVERAGE = 5000, ROOM = 12288;             // entries of a bucket on average, and with room in shared memory
constexpr int BIN = 8, BINS_MAX = ROOM / 2 + ROWS_MAX;  // entries of a bin that a thread sorts
constexpr int LONG_ROW = 2048, LONGS_MAX = 32;          // entries from which a row is taken out of a bucket without room; such rows of a bucket
constexpr int64_t LONG_WORK = 4 << 20;                  // entries read for a bucket's longer rows at most (a block reads the bucket for each of them)
constexpr int BITMAP_BITS = 20;                         // bits of a node id up to which a bitmap fits shared memory
constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr uint32_t BUCKET_MAX = 1 << 16;
enum { F_BAD_ID = 1, F_FULL = 2 };

struct Counted {
    int32_t flags;
    int32_t max_deg;                                    // without duplicates
    int32_t skip;                                       // a bucket is too large: the kernels behind the first do nothing
    uint32_t done;
    uint32_t got[BUCKETS_MAX], first[BUCKETS_MAX];      // entries of a bucket as they come, and those of the buckets before
    uint32_t at[BUCKETS_MAX];                           // scattered so far
    uint16_t order[BUCKETS_MAX];                        // the large buckets first: a block that gets one late is the end of the launch
    uint32_t kept[BUCKETS_MAX];                         // without duplicates
};

// Row u is row h & (2^log - 1) of bucket h >> log, h = u * mul mod 2^bits.
struct Split {
    int64_t n;
    int bits, log, shift;                               // shift: bits of a column
    uint32_t mul, inverse;
    __host__ __device__ __forceinline__ int buckets() const { return 1 << (bits - log); }
    __device__ __forceinline__ uint32_t hash(uint32_t u) const { return u * mul & ((1u << bits) - 1); }
    __device__ __forceinline__ uint32_t node(int b, uint32_t row) const { return (((uint32_t)b << log) + row) * inverse & ((1u << bits) - 1); }     // n and above: none
};

// Entries i0, i0 + step, ... of the list, all requested before the first is looked at: an edge, or behind the m edges an entry of the diagonal (if
// self).  f(j, u, v, both ways) for those that count.
constexpr int BATCH = 7;
static_assert(EDGES % BATCH == 0, "whole batches");
template <typename F>
__device__ __forceinline__ void read_lines(const Split& sp, int64_t m, int64_t i0, int64_t step, int count, const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int sym, int self,
                                           int32_t* flags, F f) {
    int32_t u[BATCH], v[BATCH];
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {
        const int64_t i = i0 + j * step;
        const bool edge = j < count && i < m, diagonal = j < count && self && i >= m && i - m < sp.n;
        u[j] = edge ? __ldg(src + i) : diagonal ? (int32_t)(i - m) : 0;
        v[j] = edge ? __ldg(dst + i) : diagonal ? -2 : 0;       // (an edge between the same nodes does not count)
    }
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {
        const bool diagonal = i0 + j * step >= m && v[j] == -2;
        if (diagonal) { f(j, (uint32_t)u[j], (uint32_t)u[j], false); continue; }
        if ((uint32_t)u[j] >= (uint64_t)sp.n || (uint32_t)v[j] >= (uint64_t)sp.n) { atomicOr(flags, F_BAD_ID); continue; }      // (negative ids too)
        if (u[j] != v[j]) f(j, (uint32_t)u[j], (uint32_t)v[j], sym != 0);
    }
}

// Entries of every bucket; the last block adds them up.
__global__ void __launch_bounds__(TPB) count_kernel(Split sp, int64_t m, const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int sym, int self, Counted* c) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    using Scan = cub::BlockScan<uint32_t, TPB>;
    __shared__ uint32_t count[BUCKETS_MAX];
    __shared__ typename Scan::TempStorage temp;
    __shared__ bool last;
    const int nb = sp.buckets(), tid = threadIdx.x;
    for (int b = tid; b < nb; b += TPB) count[b] = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * TPB, lines = m + (self ? sp.n : 0);
    for (int64_t i = (int64_t)blockIdx.x * TPB + tid; i < lines; i += BATCH * step)
        read_lines(sp, m, i, step, BATCH, src, dst, sym, self, &c->flags, [&](int, uint32_t u, uint32_t v, bool both) {
            atomicAdd(&count[sp.hash(u) >> sp.log], 1u);
            if (both) atomicAdd(&count[sp.hash(v) >> sp.log], 1u);
        });
    __syncthreads();
    for (int b = tid; b < nb; b += TPB)
        if (count[b]) atomicAdd(&c->got[b], count[b]);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&c->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    uint32_t x[BUCKETS_MAX / TPB];
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) x[k] = tid * (BUCKETS_MAX / TPB) + k < nb ? __ldcg(&c->got[tid * (BUCKETS_MAX / TPB) + k]) : 0;
    bool large = false;
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) large |= x[k] > BUCKET_MAX;
    if (large) { c->skip = 1; atomicOr(&c->flags, F_FULL); }
    uint32_t before[BUCKETS_MAX / TPB], larges[BUCKETS_MAX / TPB], all;
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) larges[k] = x[k] > AVERAGE * 5 / 4;
    Scan(temp).ExclusiveSum(larges, before, all);
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) {
        const uint32_t b = tid * (BUCKETS_MAX / TPB) + k;
        c->order[larges[k] ? before[k] : all + b - before[k]] = (uint16_t)b;
    }
    __syncthreads();
    Scan(temp).ExclusiveSum(x, x);
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) c->first[tid * (BUCKETS_MAX / TPB) + k] = x[k];
}

struct ScatterMemory {
    uint32_t count[BUCKETS_MAX], base[BUCKETS_MAX];     // a bucket's entries of the block before its own; what to add to a place in the block for the bucket's room
    typename cub::BlockScan<uint32_t, TPB>::TempStorage scan;
    uint32_t keys[2 * EDGES * TPB];
    uint16_t bucket[2 * EDGES * TPB];
};

// Every edge (both ways round if sym), and the diagonal if self, to the room of its bucket; a thread takes `per` of them.  A block counts its own
// entries first, takes room for all of them with one addition a bucket, and puts them in order of their buckets, so that they are written
// in runs.
__global__ void __launch_bounds__(TPB, 2) scatter_kernel(Split sp, int64_t m, const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int sym, int self, int per, uint32_t* __restrict__ keys,
                                                         Counted* c) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ __align__(16) uint8_t smem_raw[];
    ScatterMemory& sm = *reinterpret_cast<ScatterMemory*>(smem_raw);
    const int nb = sp.buckets(), tid = threadIdx.x;
    for (int b = tid; b < BUCKETS_MAX; b += TPB) sm.count[b] = 0;
    __syncthreads();
    uint32_t at[EDGES];                                 // places among the block's entries of the two buckets, 16 bits each
    const int64_t i0 = (int64_t)blockIdx.x * per * TPB + tid;
#pragma unroll
    for (int e = 0; e < EDGES; e += BATCH)
        if (e < per)
            read_lines(sp, m, i0 + e * TPB, TPB, per - e, src, dst, sym, self, &c->flags, [&](int j, uint32_t u, uint32_t v, bool both) {
                at[e + j] = atomicAdd(&sm.count[sp.hash(u) >> sp.log], 1u);
                if (both) at[e + j] |= atomicAdd(&sm.count[sp.hash(v) >> sp.log], 1u) << 16;
            });
    __syncthreads();
    uint32_t x[BUCKETS_MAX / TPB], before[BUCKETS_MAX / TPB], all;
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) x[k] = sm.count[tid * (BUCKETS_MAX / TPB) + k];
    cub::BlockScan<uint32_t, TPB>(sm.scan).ExclusiveSum(x, before, all);
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) sm.count[tid * (BUCKETS_MAX / TPB) + k] = before[k];
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the buckets' rooms are known
    if (__ldcg(&c->skip)) return;
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) {            // (all additions on their way before the first is waited for)
        const int b = k * TPB + tid;
        x[k] = b < nb ? (b + 1 < BUCKETS_MAX ? sm.count[b + 1] : all) - sm.count[b] : 0;
        before[k] = b < nb ? __ldcg(&c->first[b]) : 0;
        if (x[k]) x[k] = atomicAdd(&c->at[b], x[k]);
    }
#pragma unroll
    for (int k = 0; k < BUCKETS_MAX / TPB; ++k) {
        const int b = k * TPB + tid;
        if (b < nb) sm.base[b] = before[k] + x[k] - sm.count[b];
    }
    __syncthreads();
    const uint32_t in_bucket = (1u << sp.log) - 1;
    auto put = [&](uint32_t row, uint32_t col, uint32_t at) {
        const uint32_t h = sp.hash(row), b = h >> sp.log, i = sm.count[b] + at;
        sm.keys[i] = (h & in_bucket) << sp.shift | col;
        sm.bucket[i] = (uint16_t)b;
    };
#pragma unroll
    for (int e = 0; e < EDGES; e += BATCH)
        if (e < per)
            read_lines(sp, m, i0 + e * TPB, TPB, per - e, src, dst, sym, self, &c->flags, [&](int j, uint32_t u, uint32_t v, bool both) {
                put(u, v, at[e + j] & 0xFFFFu);
                if (both) put(v, u, at[e + j] >> 16);
            });
    __syncthreads();
#pragma unroll 4
    for (uint32_t i = tid; i < all; i += TPB) keys[sm.base[sm.bucket[i]] + i] = sm.keys[i];
}

// Compares and exchanges number i = k * 32 + lane with i ^ step: the smaller one first, or last where i & size.
__device__ __forceinline__ void exchange(uint32_t (&x)[4], int step, int size) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (step >= 32) {
            const int j = k | step / 32;
            if (j == k) continue;
            const uint32_t lo = min(x[k], x[j]), hi = max(x[k], x[j]);
            const bool down = k * 32 & size;
            x[k] = down ? hi : lo;
            x[j] = down ? lo : hi;
        } else {
            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, x[k], step);
            const bool down = (k * 32 + lane) & size, upper = lane & step;
            x[k] = upper != down ? max(x[k], other) : min(x[k], other);
        }
    }
}
__device__ __forceinline__ void sort_registers(uint32_t (&x)[4]) {
#pragma unroll
    for (int size = 2; size <= 128; size <<= 1)
#pragma unroll
        for (int step = size >> 1; step > 0; step >>= 1) exchange(x, step, size);
}

// Sorts n numbers in shared memory by a warp: 128 at a time in registers, then merges; numbers past the end count as the largest, which stay
// where they are because every exchange puts the smaller number first.
__device__ __forceinline__ void sort_span(uint32_t* keys, int n) {
    const int lane = threadIdx.x & 31;
    auto swap = [&](int lo, int hi) {
        if (hi >= n) return;
        const uint32_t a = keys[lo], b = keys[hi];
        if (a > b) { keys[lo] = b; keys[hi] = a; }
    };
    for (int size = 128; size == 128 || size < 2 * n; size <<= 1) {
        if (size > 128) {
            const int pairs = (n + size - 1) / size * (size >> 1);
            for (int p = lane; p < pairs; p += 32) {
                const int off = p & ((size >> 1) - 1), at = (p - off) * 2;
                swap(at + off, at + size - 1 - off);
            }
            __syncwarp();
            for (int step = size >> 2; step >= 128; step >>= 1) {
                for (int p = lane; p < pairs; p += 32) {
                    const int off = p & (step - 1), at = (p - off) * 2 + off;
                    swap(at, at + step);
                }
                __syncwarp();
            }
        }
        for (int c = 0; c < n; c += 128) {
            uint32_t x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) x[k] = c + k * 32 + lane < n ? keys[c + k * 32 + lane] : NONE;
            if (size == 128) sort_registers(x);
            else {
#pragma unroll
                for (int step = 64; step > 0; step >>= 1) exchange(x, step, 0);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c + k * 32 + lane < n) keys[c + k * 32 + lane] = x[k];
        }
        __syncwarp();
    }
}

// Sorts up to eight numbers by themselves (Batcher's odd-even merges).
__device__ __forceinline__ void sort_bin(uint32_t* keys, int n) {
    uint32_t x[BIN];
#pragma unroll
    for (int k = 0; k < BIN; ++k) x[k] = k < n ? keys[k] : NONE;
    auto order = [&](int i, int j) { const uint32_t a = min(x[i], x[j]); x[j] = max(x[i], x[j]); x[i] = a; };
    order(0, 1); order(2, 3); order(4, 5); order(6, 7);
    order(0, 2); order(1, 3); order(4, 6); order(5, 7);
    order(1, 2); order(5, 6);
    order(0, 4); order(1, 5); order(2, 6); order(3, 7);
    order(2, 4); order(3, 5);
    order(1, 2); order(3, 4); order(5, 6);
#pragma unroll
    for (int k = 0; k < BIN; ++k)
        if (k < n) keys[k] = x[k];
}

struct SortMemory {
    typename cub::BlockScan<uint32_t, TPB>::TempStorage scan;
    uint32_t longs, long_row[LONGS_MAX];
    uint32_t count[ROWS_MAX];                           // entries of a row, then without duplicates
    uint32_t bin[ROWS_MAX];                             // its first bin << 5 | by how much a column is shifted for its bin
    uint32_t place[ROWS_MAX];                           // of its first entry in the bucket's room
    uint32_t bins[BINS_MAX];                            // entries, then the end of a bin
    uint32_t keys[ROOM];                                // (or a bitmap, as long as it is)
};

// A bucket's entries sorted and without duplicates, row by row from the beginning of its room; entry counts and normalisation of the rows.
__global__ void __launch_bounds__(TPB, 2) sort_kernel(Split sp, const uint32_t* __restrict__ keys, uint32_t* __restrict__ sorted, Counted* c, uint32_t* __restrict__ place,
                                                      int32_t* __restrict__ deg, float* __restrict__ dinv) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    SortMemory& sm = *reinterpret_cast<SortMemory*>(smem_raw);
    using Scan = cub::BlockScan<uint32_t, TPB>;
    constexpr int PER = ROWS_MAX / TPB;
    const int rows = 1 << sp.log, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t cols = (1u << sp.shift) - 1;
    for (int i = tid; i < ROWS_MAX; i += TPB) sm.count[i] = 0;
    for (int i = tid; i < BINS_MAX; i += TPB) sm.bins[i] = 0;
    if (tid == 0) sm.longs = 0;
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (__ldcg(&c->skip)) return;
    const int b = __ldcg(&c->order[blockIdx.x]);
    const uint32_t got = __ldcg(&c->got[b]), first = __ldcg(&c->first[b]);
    const uint32_t* mine = keys + first;
    uint32_t* out = sorted + first;
    // the bucket's entries, from registers where they have room there
    constexpr int HELD = ROOM / TPB;
    uint32_t held[HELD];
    const bool holds = got <= ROOM;
    if (holds) {
#pragma unroll
        for (int k = 0; k < HELD; ++k) held[k] = (uint32_t)(k * TPB + tid) < got ? __ldcg(mine + k * TPB + tid) : NONE;
    }
    auto for_entries = [&](auto f) {
        if (holds) {
#pragma unroll
            for (int k = 0; k < HELD; ++k)
                if (held[k] != NONE) f(held[k]);
        } else {
            for (uint32_t i = tid; i < got; i += TPB) f(__ldcg(mine + i));
        }
    };
    // entries of every row; a bucket without room gives up its longest ones
    for_entries([&](uint32_t key) { atomicAdd(&sm.count[key >> sp.shift], 1u); });
    __syncthreads();
    const uint32_t most = got > ROOM ? LONG_ROW : ROOM;
    uint32_t n[PER], x[PER], total = 0, n_bins, taken;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        n[k] = sm.count[tid * PER + k];
        if (n[k] > most) {
            const uint32_t l = atomicAdd(&sm.longs, 1u);
            if (l < LONGS_MAX) sm.long_row[l] = (uint32_t)(tid * PER + k);
            n[k] = 0;
        }
        total += n[k];
        x[k] = n[k] < BIN ? n[k] > 0 : 1u << min(30 - __clz(n[k]), sp.shift);
    }
    Scan(sm.scan).ExclusiveSum(total, taken, total);
    __syncthreads();
    const uint32_t longs = sm.longs;
    if (total > ROOM || longs > LONGS_MAX || (longs && (sp.bits > BITMAP_BITS || (int64_t)longs * got > LONG_WORK))) {
        if (tid == 0) atomicOr(&c->flags, F_FULL);
        return;
    }
    uint32_t at[PER];
    Scan(sm.scan).ExclusiveSum(x, at, n_bins);
#pragma unroll
    for (int k = 0; k < PER; ++k) sm.bin[tid * PER + k] = at[k] << 5 | (n[k] ? sp.shift - (31 - __clz(x[k])) : 31u);       // (31: not here)
    __syncthreads();
    // into bins
    auto bin_of = [&](uint32_t key) {
        const uint32_t f = sm.bin[key >> sp.shift];
        return (f & 31u) == 31u ? NONE : (f >> 5) + ((key & cols) >> (f & 31u));
    };
    for_entries([&](uint32_t key) {
        const uint32_t k = bin_of(key);
        if (k != NONE) atomicAdd(&sm.bins[k], 1u);
    });
    __syncthreads();
    {
        const uint32_t each = (n_bins + TPB - 1) / TPB | 1, i0 = min(tid * each, n_bins), i1 = min(i0 + each, n_bins);       // (odd: no two lanes the same bank)
        uint32_t sum = 0;
        for (uint32_t i = i0; i < i1; ++i) sum += sm.bins[i];
        Scan(sm.scan).ExclusiveSum(sum, sum);
        for (uint32_t i = i0; i < i1; ++i) { const uint32_t m = sm.bins[i]; sm.bins[i] = sum; sum += m; }
    }
    __syncthreads();
    for_entries([&](uint32_t key) {
        const uint32_t k = bin_of(key);
        if (k != NONE) sm.keys[atomicAdd(&sm.bins[k], 1u)] = key;
    });
    __syncthreads();
    // every bin by itself
    for (uint32_t i = tid; i < n_bins; i += TPB) {
        const uint32_t from = i ? sm.bins[i - 1] : 0, m = sm.bins[i] - from;
        if (m > 1 && m <= BIN) sort_bin(sm.keys + from, (int)m);
    }
    for (uint32_t i0 = 0; i0 < n_bins; i0 += TPB) {
        const uint32_t i = i0 + tid, m = i < n_bins ? sm.bins[i] - (i ? sm.bins[i - 1] : 0) : 0;
        for (uint32_t left = __ballot_sync(0xFFFFFFFFu, m > BIN); left; left &= left - 1) {
            const uint32_t j = i - lane + __ffs(left) - 1, from = j ? sm.bins[j - 1] : 0;
            const int m = (int)(sm.bins[j] - from);
            if (m <= 32) {
                uint32_t x = lane < m ? sm.keys[from + lane] : NONE;
#pragma unroll
                for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
                    for (int step = size >> 1; step > 0; step >>= 1) {
                        const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, x, step);
                        x = ((lane & step) != 0) != ((lane & size) != 0) ? max(x, other) : min(x, other);
                    }
                if (lane < m) sm.keys[from + lane] = x;
            } else sort_span(sm.keys + from, m);
        }
    }
    __syncthreads();
    for (int i = tid; i < rows; i += TPB) sm.count[i] = 0;
    // duplicates out: a warp takes entries that follow one another
    const uint32_t share = (total + TPB - 1) / TPB * 32, j0 = min(warp * share, total), j1 = min(j0 + share, total);
    auto keep = [&](uint32_t i) { return i < j1 && (i == 0 || sm.keys[i] != sm.keys[i - 1]); };
    uint32_t kept = 0;
    for (uint32_t i0 = j0; i0 < j1; i0 += 32) kept += __popc(__ballot_sync(0xFFFFFFFFu, keep(i0 + lane)));
    uint32_t before, all;
    Scan(sm.scan).ExclusiveSum(lane == 0 ? kept : 0u, before, all);
    __syncthreads();
    before = __shfl_sync(0xFFFFFFFFu, before, 0);
    for (uint32_t i0 = j0; i0 < j1; i0 += 32) {
        const uint32_t i = i0 + lane;
        const bool one = keep(i);
        const uint32_t ones = __ballot_sync(0xFFFFFFFFu, one), to = before + __popc(ones & ((1u << lane) - 1));
        if (one) {
            const uint32_t key = sm.keys[i], row = key >> sp.shift;
            out[to] = key;
            atomicAdd(&sm.count[row], 1u);
            if (i == 0 || sm.keys[i - 1] >> sp.shift != row) sm.place[row] = to;
        }
        before += __popc(ones);
    }
    __syncthreads();
    // the rows without room
    uint32_t* bitmap = sm.keys;
    const int words = (int)((sp.n + 31) >> 5);
    for (uint32_t l = 0; l < longs; ++l) {
        const uint32_t row = sm.long_row[l];
        for (int i = tid; i < words; i += TPB) bitmap[i] = 0;
        __syncthreads();
#pragma unroll 4
        for (uint32_t i = tid; i < got; i += TPB) {
            const uint32_t key = __ldcg(mine + i);
            if (key >> sp.shift == row) atomicOr(&bitmap[(key & cols) >> 5], 1u << (key & 31));
        }
        __syncthreads();
        const int each = (words + TPB - 1) / TPB | 1, w0 = min(tid * each, words), w1 = min(w0 + each, words);
        uint32_t to = 0, marked;
        for (int i = w0; i < w1; ++i) to += __popc(bitmap[i]);
        Scan(sm.scan).ExclusiveSum(to, to, marked);
        for (int i = w0; i < w1; ++i)
            for (uint32_t left = bitmap[i]; left; left &= left - 1) out[all + to++] = row << sp.shift | (uint32_t)(i * 32 + __ffs(left) - 1);
        if (tid == 0) { sm.count[row] = marked; sm.place[row] = all; }
        all += marked;
        __syncthreads();
    }
    for (int i = tid; i < rows; i += TPB) {
        place[((int64_t)b << sp.log) + i] = sm.place[i];
        const uint32_t u = sp.node(b, i);
        if (u < sp.n) { deg[u] = (int32_t)sm.count[i]; dinv[u] = degree_norm((int32_t)sm.count[i]); }
    }
    int32_t longest = 0;
    for (int i = tid; i < rows; i += TPB) longest = max(longest, (int32_t)sm.count[i]);
    longest = __reduce_max_sync(0xFFFFFFFFu, longest);
    if (lane == 0) atomicMax(&c->max_deg, longest);
    if (tid == 0) c->kept[b] = all;
}

// Columns and values of a bucket's rows.
__global__ void __launch_bounds__(TPB) fill_kernel(Split sp, int norm, const uint32_t* __restrict__ sorted, const Counted* __restrict__ c, const uint32_t* __restrict__ place,
                                                   const int32_t* __restrict__ deg, const float* __restrict__ dinv, const int64_t* __restrict__ rowptr, int32_t* __restrict__ col, float* __restrict__ val) {
    __shared__ int64_t to[ROWS_MAX];                    // where entry i of the bucket goes, less i
    __shared__ float scale[ROWS_MAX];                   // 1 / sqrt(entries of the row), or 1 / entries
    const int b = blockIdx.x, rows = 1 << sp.log;
    const uint32_t* mine = sorted + c->first[b];
    const uint32_t kept = c->kept[b], cols = (1u << sp.shift) - 1;
    for (int i = threadIdx.x; i < rows; i += TPB) {
        const uint32_t u = sp.node(b, i);
        const bool is = u < sp.n;
        to[i] = (is ? __ldg(rowptr + u) : 0) - __ldg(place + ((int64_t)b << sp.log) + i);
        scale[i] = !is ? 0.0f : norm == 1 ? __frcp_rn((float)__ldg(deg + u)) : __ldg(dinv + u);
    }
    __syncthreads();
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < kept; i += TPB) {
        const uint32_t key = __ldg(mine + i), v = key & cols, row = key >> sp.shift;
        col[to[row] + i] = (int32_t)v;
        val[to[row] + i] = norm == 0 ? entry_value(0, scale[row], __ldg(dinv + v), 0) : norm == 1 ? scale[row] : 1.0f;
    }
}

}  // namespace

namespace mixgcn {

mixgcn_status csr_from_buckets(mixgcn_graph* g, int64_t m, const int32_t* src, const int32_t* dst, int sym, int self, cudaStream_t s, bool* built, int64_t* max_deg) {
    *built = false;
    Split sp{};
    sp.n = g->n;
    const int64_t n = g->n, total = m * (sym ? 2 : 1) + (self ? n : 0);
    while (((int64_t)1 << sp.bits) < n) ++sp.bits;
    while (((int64_t)1 << sp.shift) <= n) ++sp.shift;        // (a column stays below the word of all ones)
    while (sp.log < ROWS_LOG_MAX && sp.log < sp.bits && (total << (sp.log + 1)) >> sp.bits <= AVERAGE) ++sp.log;
    if (total == 0 || sp.bits - sp.log > 11 || (total << sp.log) >> sp.bits > AVERAGE || sp.log + sp.shift > 32) return MIXGCN_OK;
    static_assert(BUCKETS_MAX == 1 << 11, "buckets that a block counts");
    sp.mul = 0x9E3779B1u;
    sp.inverse = sp.mul;
    for (int i = 0; i < 5; ++i) sp.inverse *= 2u - sp.mul * sp.inverse;       // (Newton: twice as many right bits a step, three to begin with)
    const int buckets = sp.buckets();
    DevBuf keys(s), sorted(s), counted(s), place(s), tmp(s);
    MIXGCN_TRY(keys.alloc(total * (int64_t)sizeof(uint32_t)));
    MIXGCN_TRY(sorted.alloc(total * (int64_t)sizeof(uint32_t)));
    MIXGCN_TRY(counted.alloc(sizeof(Counted)));
    MIXGCN_TRY(place.alloc(((int64_t)1 << sp.bits) * (int64_t)sizeof(uint32_t)));
    MIXGCN_TRY(dev_alloc((void**)&g->deg, (n + 1) * (int64_t)sizeof(int32_t), s));       // (one more, zero: the scan's last element is the number of entries)
    MIXGCN_TRY(dev_alloc((void**)&g->dinv, n * (int64_t)sizeof(float), s));
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.rowptr, (n + 1) * (int64_t)sizeof(int64_t), s));
    size_t tb = 0;
    MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, g->deg, g->fwd.rowptr, n + 1, s));
    MIXGCN_TRY(tmp.alloc((int64_t)tb));
    const int64_t bitmap = sp.bits <= BITMAP_BITS ? (n + 31) / 32 * 4 : 0, spare = bitmap - (int64_t)sizeof(uint32_t) * ROOM;
    const int sort_bytes = (int)(sizeof(SortMemory) + (spare > 0 ? spare : 0));
    MIXGCN_CUDA(cudaFuncSetAttribute(scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterMemory)));
    MIXGCN_CUDA(cudaFuncSetAttribute(sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_bytes));
    Counted* d = counted.as<Counted>();
    MIXGCN_CUDA(cudaMemsetAsync(d, 0, sizeof(Counted), s));
    MIXGCN_CUDA(cudaMemsetAsync(g->deg + n, 0, sizeof(int32_t), s));
    // edges of a thread of the scatter: so many that whole waves of blocks (two an SM) take them all
    const int64_t lines = m + (self ? n : 0), wave = 2 * (int64_t)g->ctx->sm_count * TPB, waves = (lines + wave * EDGES - 1) / (wave * EDGES);
    const int per = (int)((lines + wave * waves - 1) / (wave * waves));
    const int64_t blocks = (lines + (int64_t)TPB * per - 1) / ((int64_t)TPB * per), counting = (lines + TPB * 8 - 1) / (TPB * 8);
    count_kernel<<<(unsigned)(counting < 2 * g->ctx->sm_count ? counting : 2 * g->ctx->sm_count), TPB, 0, s>>>(sp, m, src, dst, sym, self, d);
    launch_chained(scatter_kernel, dim3((unsigned)blocks), TPB, sizeof(ScatterMemory), s, sp, m, src, dst, sym, self, per, keys.as<uint32_t>(), d);
    launch_chained(sort_kernel, dim3((unsigned)buckets), TPB, (size_t)sort_bytes, s, sp, keys.as<uint32_t>(), sorted.as<uint32_t>(), d, place.as<uint32_t>(), g->deg, g->dinv);
    MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(tmp.p, tb, g->deg, g->fwd.rowptr, n + 1, s));
    MIXGCN_CUDA(cudaGetLastError());
    int64_t nnz = 0;
    struct { int32_t flags, max_deg; } seen{};
    static_assert(offsetof(Counted, max_deg) == offsetof(Counted, flags) + sizeof(int32_t), "read together");
    MIXGCN_CUDA(cudaMemcpyAsync(&nnz, g->fwd.rowptr + n, sizeof(nnz), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaMemcpyAsync(&seen, &d->flags, sizeof(seen), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    if (seen.flags & F_BAD_ID) MIXGCN_FAIL(MIXGCN_EBADGRAPH, "graph_create: a node id lies outside [0, %lld)", (long long)n);
    if (seen.flags & F_FULL) return MIXGCN_OK;
    *max_deg = seen.max_deg;
    g->nnz = nnz;
    const int64_t room = nnz > 0 ? nnz : 1;
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.col, room * (int64_t)sizeof(int32_t), s));
    MIXGCN_TRY(dev_alloc((void**)&g->fwd.val, room * (int64_t)sizeof(float), s));
    fill_kernel<<<(unsigned)buckets, TPB, 0, s>>>(sp, g->norm, sorted.as<uint32_t>(), d, place.as<uint32_t>(), g->deg, g->dinv, g->fwd.rowptr, g->fwd.col, g->fwd.val);
    MIXGCN_CUDA(cudaGetLastError());
    *built = true;
    return MIXGCN_OK;
}

}  // namespace mixgcn
