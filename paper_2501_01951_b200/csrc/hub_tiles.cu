// Aggregation of the dense corner of a graph on the tensor cores.
//
// The nodes with the most entries neighbour one another: with rows and columns in order of descending entry counts, tiles of
// 256 x 128 near the corner hold thousands of the 32,768 possible entries.  The gather kernels fetch a row of Y for each of them; here a
// tile is a bitmap of 4 KB, and its product with 128 rows of Y is three tensor-core products.
//
//  * An entry's value is row_scale[u] * col_scale[v] (both normalisations and the plain sum have that form), so the matrix that is
//    multiplied holds zeros and ones only.
//  * Rows of Y are scaled by col_scale and written as whole numbers of a unit that is a column's own, 2^-31 to 2^-30 of its largest number,
//    in four signed digits of base 256, once per call, into images of the shared-memory tiles (column_range_kernel, cut_rows_kernel).
//    Whole-number products (tcgen05 kind::i8) take half the time of bf16 ones and their 32-bit sums are exact, so a row's tiles are one
//    chain: nothing is added up on the way, and the sum is rounded to fp32 once.  What is lost is half a unit a term.
//  * Where a column's numbers lie far apart (the largest more than SPREAD_MAX binades above the geometric mean, as in the gradients of a model that
//    has learnt its labels) what is left of every number goes through once or twice more, in units of 2^-31 of the ones before; infinities, NaN
//    and numbers further apart than three passes reach (71 binades) send the call's tiles to the FMA pipes.  The device decides, by whole
//    numbers: no order of blocks changes it.
//  * A stage of the product is a tile's bitmap, expanded to bytes by four warps, and one contiguous copy of the image a CTA.  64 columns of Y
//    have 256 columns of TMEM, twice: one half adds up while the epilogue empties the other.
//  * What is not in a tile is a matrix of its own, with a schedule of its own, for the gather kernels.  They run behind the tiles, and where
//    they have a row's sum add the row's pieces to it (one, or two where a pair's share ends in the row), times row_scale.
//
// Measured, R-MAT, 233 K nodes of mean degree 500 (22,224 tiles hold 75 % of the entries), 256 columns: 5.04 ms by gathers alone, 2.01 with the
// tiles (0.41 the product, 0.06 range and cut, 1.5 the rest of the matrix); with three bf16 parts of 24 bits, added up every 128 terms, 2.51 (0.73,
// 0.02, 1.7 with 20,601 tiles).
// Bound: a tile of 256 x 128 by 64 columns takes a pair of CTAs 620 cycles, 512 of which its four instructions need.  What it took: arrivals at
// the leader's barriers without a release at cluster scope (1,815 with; 1,230 with the arrivals relayed by a warp of its own), one barrier a
// tile for both operands and one commit (850 with two rings), a warp each for images and bitmaps, 64 columns at a time and two accumulators
// (128 in one: 1,690 cycles per 128 and 3,200 a piece, which rows of one or two tiles pay for: hence PIECE_COST).
// Error against fp64 relative to the gather kernels' (2-norm; N(0,1), its positive halves, what a ReLU leaves of it, softmax gradients):
// R-MAT 300 K, mean degree 31, 132 columns 0.87, 0.74, 0.88, 0.92; 60 K, 400 0.71, 0.49, 0.57, 0.76, plain sums 0.21, 0.45, 0.52, 0.25; 233 K, 170,
// 256 columns 0.72, 0.49, 0.64, 0.78.  One row in a thousand 2^15 times the others 0.2 to 0.95; exp(3 N(0,1)) 0.1 to 0.8 (300 K nodes, 64 columns
// 1.16).  Row means transposed are left out: the entries of small columns carry a row's sum there.
#include <cub/cub.cuh>

#include <algorithm>
#include <mutex>
#include <new>
#include <vector>

#include "hub_tiles.cuh"
#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"

using namespace mixgcn;
using namespace mixgcn::tc;

namespace {

constexpr int ROWS = HUB_ROWS, COLS = HUB_COLS;
constexpr int HUB_MAX = 1 << 16, CB_MAX = HUB_MAX / COLS;       // most rows and columns that are looked at
constexpr int A_BYTES = 128 * COLS;       // a CTA's rows of a tile expanded to bytes: K-major, 128-byte swizzle
constexpr int EPI_WARPS = 8, EXP_WARP = 8, EXP_WARPS = 4, TMA_WARP = 12, BITS_WARP = 13, MMA_WARP = 14, THREADS = 480;
constexpr int SLOTS = 6, B_BYTES = 128 * COLS, BITS_BYTES = 128 * 16, SLOT_BYTES = A_BYTES + B_BYTES;     // a CTA's half of the widest accumulator; its rows' bitmaps
constexpr int BOX_BYTES = 2048;
constexpr int TILES_SMEM = SLOTS * (SLOT_BYTES + BITS_BYTES) + EPI_WARPS * BOX_BYTES + 1024;
constexpr int AHEAD = 16;                       // tiles whose bitmaps are asked for in L2
constexpr int COLUMN_COST = 1200;               // entries whose gathers take as long as cutting a block of 128 rows of Y
constexpr int PIECE_COST = 3;                   // tiles that take as long as a piece does beside its tiles
constexpr int LEAST_TILES = 8;                  // of a pair of CTAs
constexpr uint32_t TMEM_COLS = 512;
constexpr int GROUP = 16, DIGITS = 4;           // columns of Y whose digits lie together, digits of a number in a pass
// Exponents between the largest number of a column and the mean of its others up to which one pass does (31 bits below the largest), by how
// many more every other pass reaches, and how many passes there are at most.
constexpr int SPREAD_MAX = 9, SPREAD_MORE = 31, PASSES_MAX = 3;

// What column_range_kernel leaves for the kernels behind it, and its own sums, which are zero between calls.
struct Ranges {
    int32_t shift[HUB_SLICE];                   // numbers are cut as multiples of 2^-shift (read by fours)
    uint32_t top[HUB_SLICE];                    // largest number of a column, as bits
    int32_t sum[HUB_SLICE], count[HUB_SLICE];   // exponents of its numbers but zeros, and how many
    int32_t passes;                             // 0: plain_pieces instead
    uint32_t done;                              // blocks that have added theirs
};
static_assert(TILES_WORD * 4 % 16 == 0 && TILES_WORD + (int)(sizeof(Ranges) / 4) <= STATUS_WORDS, "room beside the status words");

// How w columns of Y are taken: in blocks, all digits of a block's columns side by side in an accumulator; passes one behind the other.
struct Shape {
    int cols, blocks;                           // columns of a block (a multiple of GROUP), blocks
    __host__ __device__ int n() const { return DIGITS * cols; }                            // columns of the accumulator, at most 256
    __host__ __device__ int image_bytes() const { return n() / 2 * COLS; }                 // a CTA's half of a tile's image
};
Shape make_shape(int w) {
    const int most = (int)TMEM_COLS / 2 / DIGITS / GROUP * GROUP;
    Shape s;
    s.blocks = (w + most - 1) / most;
    s.cols = ((w + s.blocks - 1) / s.blocks + GROUP - 1) / GROUP * GROUP;
    return s;
}

struct TileParams {
    const HubPiece* pieces; const int32_t* first_piece; // pair i takes pieces first_piece[i] .. first_piece[i + 1] - 1
    const int32_t* tile_cb; const uint4* bits;
    float* partial; int64_t ldp;                        // row r of piece q goes to partial row q * ROWS + r
    int w4, kblocks;
    Shape shape;
    const Ranges* ranges;
    const float* Y; int64_t ldy, y_rows;
    const int32_t* nodes; const float* col_scale; int64_t n_cols;
    int32_t* status;
    uint32_t wait_limit;
    int drop_load;
};

struct Shared {
    uint64_t bits_full[SLOTS], full[SLOTS], empty[SLOTS];     // a tile: bitmap -> expansion, with the image -> MMA -> all of them
    uint64_t acc_full[2], acc_empty[2];                 // accumulators: MMA -> epilogue -> MMA
    uint32_t tmem;
    int abort_flag;
};

struct Ring {                     // position in a ring of slots and the parity of its use
    int i = 0;
    uint32_t use = 0;
    __device__ __forceinline__ void next(int n) { if (++i == n) { i = 0; use ^= 1; } }
};

__device__ __forceinline__ bool thread_wait(uint64_t* bar, uint32_t parity, Shared& b, const TileParams& p) {
    volatile int* flag = &b.abort_flag;
    if (mbar_wait(bar, parity, flag, p.wait_limit)) return true;
    *flag = 1;
    atomicMax(p.status, DEV_WAIT_EXPIRED);
    return false;
}
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, Shared& b, const TileParams& p) {
    return __all_sync(0xFFFFFFFFu, thread_wait(bar, parity, b, p)) != 0;
}
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{.reg .pred q; elect.sync _|q, 0xFFFFFFFF; selp.u32 %0, 1, 0, q;}" : "=r"(p));
    return p != 0;
}

// Where the column c (mod 32) of a tile's row has its bit: shifted right by c / 4 it is the lowest bit of byte c % 4, so that a shift and
// an AND turn a word into four bytes of zeros and ones.
__host__ __device__ constexpr int bit_of(int c) { return 8 * (c & 3) + ((c >> 2) & 7); }
__host__ __device__ constexpr int column_of(int bit) { return 4 * (bit & 7) + (bit >> 3); }

// A pair's pieces on the FMA pipes, for calls in which a row of Y holds an infinity, a NaN, or numbers too far apart: the
// expansion warps, one per row of a piece, entries in the order of their bits.
__device__ __forceinline__ void plain_pieces(const TileParams& p, int q0, int q1, int rank) {
    const int lane = threadIdx.x & 31;
    for (int i = (threadIdx.x >> 5) - EXP_WARP; i < (q1 - q0) * 128; i += EXP_WARPS) {
        const int q = q0 + i / 128, row = rank * 128 + i % 128;
        const HubPiece piece = p.pieces[q];
        float4 acc[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
        for (int t = piece.begin; t < piece.end; ++t) {
            const uint4 words = __ldg(p.bits + (int64_t)t * ROWS + row);
            const uint32_t word[4] = {words.x, words.y, words.z, words.w};
            for (int k = 0; k < 4; ++k)
                for (uint32_t left = word[k]; left; left &= left - 1) {
                    const int64_t h = (int64_t)p.tile_cb[t] * COLS + k * 32 + column_of(__ffs(left) - 1);
                    if (!index_ok(h, p.n_cols, p.status, SITE_SPMM_POS)) continue;
                    const int64_t v = __ldg(p.nodes + h);
                    if (!index_ok(v, p.y_rows, p.status, SITE_SPMM_COL)) continue;
                    const float a = __ldg(p.col_scale + h);
#pragma unroll
                    for (int c = 0; c < 2; ++c)
                        if (lane + c * 32 < p.w4) {
                            const float4 y = __ldg(reinterpret_cast<const float4*>(p.Y + v * p.ldy) + lane + c * 32);
                            acc[c].x = fmaf(a, y.x, acc[c].x); acc[c].y = fmaf(a, y.y, acc[c].y);
                            acc[c].z = fmaf(a, y.z, acc[c].z); acc[c].w = fmaf(a, y.w, acc[c].w);
                        }
                }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (lane + c * 32 < p.w4) reinterpret_cast<float4*>(p.partial + ((int64_t)q * ROWS + row) * p.ldp)[lane + c * 32] = acc[c];
    }
}

// The sums of 8 columns, digits 16 columns of the accumulator apart, from two's complement digits of base 256: exact, then rounded once.  finer:
// by how many binades this pass' unit is smaller than the first one's.
__device__ __forceinline__ void join_digits(uint32_t taddr, const int32_t* __restrict__ shift, int finer, float (&out)[8]) {
    uint32_t r[DIGITS][8];
#pragma unroll
    for (int d = 0; d < DIGITS; ++d) tc_ld8(taddr + d * GROUP, r[d]);
    tc_wait_ld();
    const int4 s0 = __ldcg(reinterpret_cast<const int4*>(shift)), s1 = __ldcg(reinterpret_cast<const int4*>(shift) + 1);
    const int32_t s[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t x = (int64_t)(int32_t)r[0][i] + (int64_t)(int32_t)r[1][i] * (1 << 8) + (int64_t)(int32_t)r[2][i] * (1 << 16) + (int64_t)(int32_t)r[3][i] * (1 << 24);
        const int down = -s[i] - finer, half = down >> 1, rest = down - half;           // (2^down itself may lie outside fp32)
        out[i] = __ll2float_rn(x) * __int_as_float((half + 127) << 23) * __int_as_float((rest + 127) << 23);
    }
}

// The accumulator of one piece and block, 16 columns at a time, through a box per warp, so that a request stores whole sectors; behind the
// first pass added to what the same threads have stored.
__device__ __forceinline__ void store_sums(const TileParams& p, uint32_t lanes, int groups, int half, int col0, int pass, float* dst, uint8_t* box) {
    const int lane = threadIdx.x & 31;
    for (int g = half; g < groups; g += 2) {
#pragma unroll
        for (int sub = 0; sub < 2; ++sub) {
            float x[8];
            join_digits(lanes + g * GROUP * DIGITS + sub * 8, p.ranges->shift + col0 + g * GROUP + sub * 8, pass * SPREAD_MORE, x);
#pragma unroll
            for (int c = 0; c < 2; ++c)
                *reinterpret_cast<float4*>(box + lane * 64 + (((sub * 2 + c) ^ ((lane >> 1) & 3)) << 4)) = make_float4(x[c * 4], x[c * 4 + 1], x[c * 4 + 2], x[c * 4 + 3]);
        }
        __syncwarp();
        const int c4 = ((col0 + g * GROUP) >> 2) + (lane & 3);
        if (c4 < p.w4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = i * 8 + (lane >> 2);
                float4 x = *reinterpret_cast<const float4*>(box + row * 64 + (((lane & 3) ^ ((row >> 1) & 3)) << 4));
                float4* to = reinterpret_cast<float4*>(dst) + row * (p.ldp >> 2) + c4;
                if (pass) { const float4 o = *to; x.x += o.x; x.y += o.y; x.z += o.z; x.w += o.w; }
                *to = x;
            }
        }
        __syncwarp();
    }
}

// A pair of CTAs (cluster of two, tcgen05 .cta_group::2) takes 256 rows, 128 each; each holds half of B.  The pair's
// tiles once for every block of the columns of Y and pass.
// The barriers full and acc_empty that count are the leader's, whose MMA warp waits on them; the others exist in both.
// Warps 0-7 epilogue (two per TMEM lane quarter, alternate groups of columns), 8-11 expansion (a thread per row of the tile),
// 12 images, 13 bitmaps, 14 MMA issue.  The expansion has its bitmaps from shared memory: its fences and its arrivals in the leader's memory would
// wait for loads from global memory that its threads have under way (1,230 cycles a tile).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1) spmm_tiles_kernel(const __grid_constant__ CUtensorMap images, const TileParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) Shared b;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank(), pair = cluster_id_x();
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* bitmaps = smem + SLOTS * SLOT_BYTES;          // (a slot: the expanded tile, the image)
    uint8_t* boxes = bitmaps + SLOTS * BITS_BYTES;
    const int q0 = p.first_piece[pair], q1 = p.first_piece[pair + 1];
    const int t0 = q0 < q1 ? p.pieces[q0].begin : 0, t1 = q0 < q1 ? p.pieces[q1 - 1].end : 0;      // the pair's tiles are consecutive
    if (threadIdx.x == 0) {
        b.abort_flag = 0;
        for (int s = 0; s < SLOTS; ++s) { mbar_init(&b.bits_full[s], 1); mbar_init(&b.full[s], 1 + 2 * EXP_WARPS); mbar_init(&b.empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&b.acc_full[s], 1); mbar_init(&b.acc_empty[s], 2 * EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == MMA_WARP) {              // (before the wait below: no kernel that this one may run beside has tensor memory)
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&b.tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                  // both CTAs' barriers exist before anything signals them
    tc_fence_after();
    const uint32_t tmem = b.tmem;
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the images are complete
    const Shape sh = p.shape;
    const int passes = __ldcg(&p.ranges->passes), blocks = passes * sh.blocks, n = sh.n();       // (the blocks of all passes)
    const uint32_t image_bytes = (uint32_t)sh.image_bytes();

    if (warp < EPI_WARPS) {
        const int quarter = warp & 3, half = warp >> 2;
        uint32_t at = 0;
        bool ok = true;
        for (int blk = 0; blk < blocks && ok; ++blk)
            for (int q = q0; q < q1; ++q, ++at) {
                const uint32_t set = at & 1, use = at >> 1 & 1;
                if (!warp_wait(&b.acc_full[set], use, b, p)) { ok = false; break; }
                tc_fence_after();
                const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16) + set * (uint32_t)n;
                float* dst = p.partial + ((int64_t)q * ROWS + rank * 128 + quarter * 32) * p.ldp;
                store_sums(p, lanes, sh.cols / GROUP, half, blk % sh.blocks * sh.cols, blk / sh.blocks, dst, boxes + warp * BOX_BYTES);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_pair(mapa_shared(smem_u32(&b.acc_empty[set]), 0));
            }
    } else if (warp < TMA_WARP) {
        if (passes == 0) plain_pieces(p, q0, q1, (int)rank);
        const int row = threadIdx.x - EXP_WARP * 32;
        Ring slot;
        for (int t = blocks * (t1 - t0); t > 0; --t, slot.next(SLOTS)) {
            if (!warp_wait(&b.bits_full[slot.i], slot.use, b, p)) break;       // (asked for when the slot was empty)
            const uint4 bits = *reinterpret_cast<const uint4*>(bitmaps + slot.i * BITS_BYTES + row * 16);
            const uint32_t word[4] = {bits.x, bits.y, bits.z, bits.w};
            uint8_t* dst = smem + slot.i * SLOT_BYTES + row * 128;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t x = word[j >> 1] >> (4 * (j & 1));
                *reinterpret_cast<uint4*>(dst + ((j ^ (row & 7)) << 4)) = make_uint4(x & 0x01010101u, x >> 1 & 0x01010101u, x >> 2 & 0x01010101u, x >> 3 & 0x01010101u);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive_pair(mapa_shared(smem_u32(&b.full[slot.i]), 0));
        }
    } else if (warp == TMA_WARP) {
        if (lane == 0) {
            Ring slot;
            bool ok = true;
            for (int blk = 0; blk < blocks && ok; ++blk)
                for (int t = t0; t < t1; ++t, slot.next(SLOTS)) {
                    const int row = ((blk * p.kblocks + __ldg(p.tile_cb + t)) * 2 + (int)rank) * (n / 2);
                    if (!thread_wait(&b.empty[slot.i], slot.use ^ 1, b, p)) { ok = false; break; }
                    if (rank == 0) mbar_expect_tx(&b.full[slot.i], 2 * image_bytes);
                    if (!(p.drop_load && blk == 0 && t == t0))
                        tma_load_2d_pair(smem + slot.i * SLOT_BYTES + A_BYTES, &images, 0, row, mapa_shared(smem_u32(&b.full[slot.i]), 0));
                }
        }
    } else if (warp == BITS_WARP) {
        if (lane == 0) {
            Ring slot;
            bool ok = true;
            for (int blk = 0; blk < blocks && ok; ++blk)
                for (int t = t0; t < t1; ++t, slot.next(SLOTS)) {
                    const uint4* bits = p.bits + (int64_t)t * ROWS + rank * 128;
                    if (t + AHEAD < t1) bulk_prefetch(bits + AHEAD * ROWS, BITS_BYTES);
                    if (!thread_wait(&b.empty[slot.i], slot.use ^ 1, b, p)) { ok = false; break; }
                    mbar_expect_tx(&b.bits_full[slot.i], BITS_BYTES);
                    bulk_load(bitmaps + slot.i * BITS_BYTES, bits, BITS_BYTES, &b.bits_full[slot.i]);
                }
        }
    } else if (warp == MMA_WARP && rank == 0) {
        const uint32_t idesc = make_idesc_u8s8(ROWS, n);
        Ring slot;
        uint32_t at = 0;
        bool ok = true;
        for (int blk = 0; blk < blocks && ok; ++blk)
            for (int q = q0; q < q1 && ok; ++q, ++at) {
                const HubPiece piece = p.pieces[q];
                const uint32_t set = at & 1, use = at >> 1 & 1;
                ok = warp_wait(&b.acc_empty[set], use ^ 1, b, p);
                for (int t = piece.begin; t < piece.end && ok; ++t, slot.next(SLOTS)) {
                    if (!warp_wait(&b.full[slot.i], slot.use, b, p)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t a = make_desc(smem_u32(smem + slot.i * SLOT_BYTES), 16, 1024, 2), bd = a + A_BYTES / 16;
                    if (elect_one()) {
#pragma unroll
                        for (int j = 0; j < COLS / 32; ++j) tc_mma_pair<KIND_I8>(tmem + set * (uint32_t)n, a + j * 2, bd + j * 2, idesc, t > piece.begin || j);
                        tc_commit_pair(&b.empty[slot.i], 3);
                        if (t + 1 == piece.end) tc_commit_pair(&b.acc_full[set], 3);
                    }
                    __syncwarp();
                }
            }
    }
    __syncwarp();
    if (threadIdx.x == 0 && b.abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);      // a wait expired: let copies in flight land
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                  // the peer is done with this CTA's shared and tensor memory
    if (warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// The range of every column of Y over the hub columns of the matrix, scaled as they are multiplied: what unit its numbers are cut in, and how
// many passes the call takes.  All whole numbers, so that neither depends on the order of the blocks.  2^lanes lanes a row.
constexpr int RANGE_THREADS = 512;
__global__ void __launch_bounds__(RANGE_THREADS) column_range_kernel(int64_t n_cols, int w, int lanes, const int32_t* __restrict__ nodes, const float* __restrict__ scale,
                                                           const float* __restrict__ Y, int64_t ldy, int64_t y_rows, Ranges* ranges, int32_t* status) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ uint32_t top[HUB_SLICE];
    __shared__ int32_t sum[HUB_SLICE], count[HUB_SLICE];
    __shared__ bool last;
    const int tid = threadIdx.x, c0 = (tid & ((1 << lanes) - 1)) * 4;
    if (tid < HUB_SLICE) { top[tid] = 0; sum[tid] = count[tid] = 0; }
    __syncthreads();
    uint32_t my_top[4] = {0, 0, 0, 0};
    int32_t my_sum[4] = {0, 0, 0, 0}, my_count[4] = {0, 0, 0, 0};
    if (c0 < w) {
        constexpr int BATCH = 4;            // rows whose numbers are on their way at once
        const int64_t step = (int64_t)gridDim.x * (RANGE_THREADS >> lanes);
        for (int64_t h0 = (int64_t)blockIdx.x * (RANGE_THREADS >> lanes) + (tid >> lanes); h0 < n_cols; h0 += BATCH * step) {
            float4 y[BATCH];
            float s[BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int64_t h = h0 + i * step, v = h < n_cols ? __ldg(nodes + h) : -1;
                const bool live = h < n_cols && index_ok(v, y_rows, status, SITE_SPMM_COL);
                y[i] = live ? __ldg(reinterpret_cast<const float4*>(Y + v * ldy + c0)) : make_float4(0.f, 0.f, 0.f, 0.f);
                s[i] = live ? __ldg(scale + h) : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const float x[4] = {y[i].x, y[i].y, y[i].z, y[i].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t bits = __float_as_uint(x[j] * s[i]) & 0x7FFFFFFFu;
                    my_top[j] = max(my_top[j], bits);
                    my_sum[j] += (int32_t)(bits >> 23);
                    my_count[j] += x[j] != 0.0f;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (c0 + j < w) { atomicMax(&top[c0 + j], my_top[j]); atomicAdd(&sum[c0 + j], my_sum[j]); atomicAdd(&count[c0 + j], my_count[j]); }
    }
    __syncthreads();
    if (tid < w) { atomicMax(&ranges->top[tid], top[tid]); atomicAdd(&ranges->sum[tid], sum[tid]); atomicAdd(&ranges->count[tid], count[tid]); }
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicInc(&ranges->done, gridDim.x - 1) == gridDim.x - 1;      // (back at zero)
    __syncthreads();
    if (!last) return;
    __threadfence();
    const bool mine = tid < HUB_SLICE;
    const uint32_t most = mine ? __ldcg(&ranges->top[tid]) : 0;
    const int32_t all = mine ? __ldcg(&ranges->sum[tid]) : 0, many = mine ? __ldcg(&ranges->count[tid]) : 0;
    const int spread = many ? (int)(most >> 23) - all / many : 0;
    int passes = 1;
    for (int k = 0; k < PASSES_MAX; ++k) passes += __syncthreads_or(spread > SPREAD_MAX + k * SPREAD_MORE) ? 1 : 0;
    if (__syncthreads_or(most >= 0x7F800000u) || passes > PASSES_MAX) passes = 0;
    if (tid == 0) ranges->passes = passes;
    if (!mine) return;
    ranges->top[tid] = 0; ranges->sum[tid] = ranges->count[tid] = 0;
    // the largest number stays below 2^31 - 2^24 units: its highest digit takes a carry from those below
    ranges->shift[tid] = 30 - (max((int)(most >> 23), 1) - 127 + ((most & 0x7FFFFFu) >= 0x7E0000u));
}

// 16 rows of a column in units -> its 16 bytes of every digit; behind the first pass of what is left, in units of 2^-31 (worked out anew: kept,
// it would take half as many registers again).  Adding 1.5 * 2^52 leaves the whole number that is nearest in the lowest bits.
__device__ __forceinline__ void cut_column(const float (&y)[16], const double* __restrict__ by, double unit, int pass, uint4 (&out)[DIGITS]) {
    constexpr uint32_t CARRIES = 0x808080u;                  // digits from -128 to 127
    constexpr double WHOLE = 6755399441055744.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t t[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            double x = (double)y[q * 4 + i] * by[q * 4 + i] * unit;
#pragma unroll 1
            for (int k = 0; k < pass; ++k) x = (x - ((x + WHOLE) - WHOLE)) * 0x1p31;
            t[i] = ((uint32_t)__double2loint(x + WHOLE) + CARRIES) ^ CARRIES;
        }
#pragma unroll
        for (int d = 0; d < DIGITS; ++d) {
            const uint32_t pick = (uint32_t)d | (uint32_t)(4 + d) << 4;
            const uint32_t r = __byte_perm(__byte_perm(t[0], t[1], pick), __byte_perm(t[2], t[3], pick), 0x5410);
            (q == 0 ? out[d].x : q == 1 ? out[d].y : q == 2 ? out[d].z : out[d].w) = r;
        }
    }
}

// Rows of Y of the hub columns -> images of their digits: images[pass][block][column block of the matrix][half of an accumulator's columns], the
// 128 numbers of a digit of a column consecutive, as the tensor core wants them in shared memory.  A block of threads takes 128 rows and 16
// columns (the blocks of the same rows run side by side), a thread 16 rows of a column.  The scaling is exact (fp64); what is below half a unit
// of the last pass is all that is lost.  Eight blocks an SM: waiting for rows is most of its time (96 registers and five: + 30 us of a 2,050 us call).
__global__ void __launch_bounds__(128, 8) cut_rows_kernel(int64_t n_cols, int kblocks, Shape sh, int w, const int32_t* __restrict__ nodes, const float* __restrict__ scale,
                                                       const float* __restrict__ Y, int64_t ldy, int64_t y_rows, uint8_t* __restrict__ images, const Ranges* ranges, int32_t* status) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ __align__(16) int32_t node[COLS];
    __shared__ __align__(16) double by[COLS];
    const int tid = threadIdx.x, kb = blockIdx.y;
    {
        const int64_t h = (int64_t)kb * COLS + tid;
        const int64_t v = h < n_cols ? __ldg(nodes + h) : -1;
        const bool live = h < n_cols && index_ok(v, y_rows, status, SITE_SPMM_COL);
        node[tid] = live ? (int32_t)v : -1;
        by[tid] = live ? (double)__ldg(scale + h) : 0.0;
    }
    __syncthreads();
    const int c = tid & 15, j = tid >> 4, col = (int)blockIdx.x * GROUP + c;
    float y[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int4 v4 = *reinterpret_cast<const int4*>(node + j * 16 + q * 4);
        const int v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) y[q * 4 + i] = v[i] >= 0 && col < w ? __ldg(Y + (int64_t)v[i] * ldy + col) : 0.0f;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the ranges are complete (Y was before them)
    const int passes = __ldcg(&ranges->passes);
    const double unit = col < w ? __hiloint2double((__ldcg(&ranges->shift[col < w ? col : 0]) + 1023) << 20, 0) : 0.0;
    const int groups = sh.cols / GROUP, blk = (int)blockIdx.x / groups, g = (int)blockIdx.x % groups;
    if (passes == 0) return;
    const int64_t image = (int64_t)sh.image_bytes();
#pragma unroll 1
    for (int pass = 0; pass < passes; ++pass) {
        uint4 out[DIGITS];
        cut_column(y, by + j * 16, unit, pass, out);
        uint8_t* base = images + ((int64_t)(pass * sh.blocks + blk) * kblocks + kb) * 2 * image;
#pragma unroll
        for (int d = 0; d < DIGITS; ++d) {
            int row = (g * DIGITS + d) * GROUP + c;
            const int rank = row >= sh.n() / 2;
            row -= rank * (sh.n() / 2);
            *reinterpret_cast<uint4*>(base + rank * image + row * 128 + ((j ^ (row & 7)) << 4)) = out[d];
        }
    }
}

// ---------------------------------------------------------------- construction

constexpr int TPB = 256;
inline unsigned blocks_for(int64_t n) { return (unsigned)((n + TPB - 1) / TPB); }

struct HubTotals { unsigned long long entries; int32_t tiles, last_row_block, last_col_block; };

// rank[perm[i]] = i for the first `hubs` of perm, `none` for the others
__global__ void rank_kernel(int64_t n, int64_t hubs, int32_t none, const int32_t* __restrict__ perm, int32_t* __restrict__ rank) {
    const int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (i < n) rank[perm[i]] = i < hubs ? (int32_t)i : none;
}

// cnt[row block][column block] += entries of one hub row (a block per row)
__global__ void __launch_bounds__(TPB) tile_count_kernel(int cbs, const int32_t* __restrict__ perm, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                                         const int32_t* __restrict__ rank, int32_t* __restrict__ cnt) {
    __shared__ int32_t hist[CB_MAX];
    const int64_t r = blockIdx.x, u = perm[r], e = rowptr[u + 1];
    for (int i = threadIdx.x; i < cbs; i += TPB) hist[i] = 0;
    __syncthreads();
    for (int64_t i = rowptr[u] + threadIdx.x; i < e; i += TPB) {
        const int32_t q = __ldg(rank + col[i]);
        if (q < cbs * COLS) atomicAdd(&hist[q / COLS], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cbs; i += TPB)
        if (hist[i]) atomicAdd(&cnt[(r / ROWS) * cbs + i], hist[i]);
}

// The tiles that pay are those of `least` entries and more, in rows and columns of tiles where what they hold beyond that is worth a row's
// piece and the cutting of a column's rows of Y.  By rows first (a block per row) ...
__global__ void __launch_bounds__(TPB) tile_rows_kernel(int cbs, int least, int worth, const int32_t* __restrict__ cnt, int32_t* __restrict__ flag) {
    const int32_t* mine = cnt + (int64_t)blockIdx.x * cbs;
    __shared__ int32_t gain;
    if (threadIdx.x == 0) gain = 0;
    __syncthreads();
    int sum = 0;
    for (int i = threadIdx.x; i < cbs; i += TPB) sum += max(mine[i] - least, 0);
    if (sum) atomicAdd(&gain, sum);
    __syncthreads();
    for (int i = threadIdx.x; i < cbs; i += TPB) flag[(int64_t)blockIdx.x * cbs + i] = gain >= worth && mine[i] >= least ? 1 : 0;
}
// ... then by columns
__global__ void __launch_bounds__(TPB) tile_cols_kernel(int rbs, int cbs, int least, int worth, const int32_t* __restrict__ cnt, int32_t* __restrict__ flag, HubTotals* totals) {
    const int cb = blockIdx.x;
    __shared__ int32_t gain;
    if (threadIdx.x == 0) gain = 0;
    __syncthreads();
    int sum = 0;
    for (int i = threadIdx.x; i < rbs; i += TPB)
        if (flag[i * cbs + cb]) sum += cnt[i * cbs + cb] - least;
    if (sum) atomicAdd(&gain, sum);
    __syncthreads();
    for (int i = threadIdx.x; i < rbs; i += TPB) {
        if (!flag[i * cbs + cb]) continue;
        if (gain < worth) { flag[i * cbs + cb] = 0; continue; }
        atomicAdd(&totals->entries, (unsigned long long)cnt[i * cbs + cb]);
        atomicAdd(&totals->tiles, 1);
        atomicMax(&totals->last_row_block, i);
        atomicMax(&totals->last_col_block, cb);
    }
    if (cb == 0 && threadIdx.x == 0) flag[rbs * cbs] = 0;        // one more than there are tiles: the scan's last element is their number
}

__global__ void tile_index_kernel(int total, int cbs, const int32_t* __restrict__ flag, const int32_t* __restrict__ first, int32_t* __restrict__ map, int32_t* __restrict__ tile_cb) {
    const int i = blockIdx.x * TPB + threadIdx.x;
    if (i >= total) return;
    map[i] = flag[i] ? first[i] : -1;
    if (flag[i]) tile_cb[first[i]] = i % cbs;
}

// Bitmaps of one row of the rows of tiles (a block per row, rows past the last node empty), and the number of its entries that are in
// no tile.
__global__ void __launch_bounds__(TPB) tile_bits_kernel(int64_t n, int cbs, const int32_t* __restrict__ perm, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                                        const int32_t* __restrict__ col_rank, const int32_t* __restrict__ map, uint4* __restrict__ bits, int64_t* __restrict__ rem_len) {
    __shared__ uint4 row_bits[CB_MAX];
    __shared__ int32_t row_map[CB_MAX], left;
    const int64_t r = blockIdx.x;
    const int64_t rb = r / ROWS;
    for (int i = threadIdx.x; i < cbs; i += TPB) { row_bits[i] = make_uint4(0, 0, 0, 0); row_map[i] = map[rb * cbs + i]; }
    if (threadIdx.x == 0) left = 0;
    __syncthreads();
    if (r < n) {
        const int64_t u = perm[r], e = rowptr[u + 1];
        int mine = 0;
        for (int64_t i = rowptr[u] + threadIdx.x; i < e; i += TPB) {
            const int32_t q = __ldg(col_rank + col[i]);
            if (q < cbs * COLS && row_map[q / COLS] >= 0) atomicOr(reinterpret_cast<uint32_t*>(row_bits) + (q >> 5), 1u << bit_of(q));
            else ++mine;
        }
        if (mine) atomicAdd(&left, mine);
        __syncthreads();
        if (threadIdx.x == 0) rem_len[u] = left;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cbs; i += TPB)
        if (row_map[i] >= 0) bits[(int64_t)row_map[i] * ROWS + r % ROWS] = row_bits[i];
}

__global__ void row_len_kernel(int64_t n, const int64_t* __restrict__ rowptr, int64_t* __restrict__ len) {
    const int64_t u = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (u <= n) len[u] = u < n ? rowptr[u + 1] - rowptr[u] : 0;
}

// The entries that are in no tile, in column order: a block per row of the rows of tiles ...
__global__ void __launch_bounds__(TPB) remainder_kernel(int cbs, const int32_t* __restrict__ perm, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                                        const float* __restrict__ val, const int32_t* __restrict__ col_rank, const int32_t* __restrict__ map,
                                                        const int64_t* __restrict__ rem_ptr, int32_t* __restrict__ rem_col, float* __restrict__ rem_val) {
    __shared__ int32_t row_map[CB_MAX];
    __shared__ int warp_sum[TPB / 32];
    const int64_t r = blockIdx.x, u = perm[r], e = rowptr[u + 1];
    const int64_t rb = r / ROWS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < cbs; i += TPB) row_map[i] = map[rb * cbs + i];
    __syncthreads();
    int64_t at = rem_ptr[u];
    for (int64_t i0 = rowptr[u]; i0 < e; i0 += TPB) {
        const int64_t i = i0 + threadIdx.x;
        int32_t c = 0;
        bool keep = false;
        if (i < e) {
            c = col[i];
            const int32_t q = __ldg(col_rank + c);
            keep = !(q < cbs * COLS && row_map[q / COLS] >= 0);
        }
        const unsigned ballot = __ballot_sync(0xFFFFFFFFu, keep);
        if (lane == 0) warp_sum[warp] = __popc(ballot);
        __syncthreads();
        int before = __popc(ballot & ((1u << lane) - 1u)), all = 0;
#pragma unroll
        for (int k = 0; k < TPB / 32; ++k) { if (k < warp) before += warp_sum[k]; all += warp_sum[k]; }
        if (keep) { rem_col[at + before] = c; rem_val[at + before] = val[i]; }
        at += all;
        __syncthreads();
    }
}
// ... and a warp per other row
__global__ void other_rows_kernel(int64_t first, int64_t n, const int32_t* __restrict__ perm, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                  const float* __restrict__ val, const int64_t* __restrict__ rem_ptr, int32_t* __restrict__ rem_col, float* __restrict__ rem_val) {
    const int64_t r = first + (((int64_t)blockIdx.x * TPB + threadIdx.x) >> 5);
    if (r >= n) return;
    const int64_t u = perm[r], b = rowptr[u], len = rowptr[u + 1] - b, at = rem_ptr[u];
    for (int64_t i = threadIdx.x & 31; i < len; i += 32) { rem_col[at + i] = col[b + i]; rem_val[at + i] = val[b + i]; }
}

// row_scale, col_scale by rank (see entry_value in graph.cu)
__global__ void hub_scale_kernel(int64_t count, int norm, int by_degree, const int32_t* __restrict__ perm, const int32_t* __restrict__ deg,
                                 const float* __restrict__ dinv, float* __restrict__ scale) {
    const int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (i >= count) return;
    const int64_t u = perm[i];
    scale[i] = norm == 0 ? dinv[u] : (norm == 1 && by_degree) ? (deg[u] > 0 ? __frcp_rn((float)deg[u]) : 0.0f) : 1.0f;
}

// CTA pairs of the product that run at once
mixgcn_status resident_pairs(const mixgcn_ctx* ctx, int* pairs) {
    *pairs = 0;
    MIXGCN_CUDA(cudaFuncSetAttribute(spmm_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_SMEM));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(ctx->sm_count & ~1), 1, 1); cfg.blockDim = dim3(THREADS, 1, 1); cfg.dynamicSmemBytes = TILES_SMEM;
    cfg.attrs = attr; cfg.numAttrs = 1;
    MIXGCN_CUDA(cudaOccupancyMaxActiveClusters(pairs, spmm_tiles_kernel, &cfg));
    return MIXGCN_OK;
}

void free_tiles(HubTiles* t) {
    if (!t) return;
    void* blocks[] = {t->rank, t->col_scale, t->row_scale, t->bits, t->tile_cb, t->pieces, t->first_piece, t->piece_first};
    for (void* b : blocks) dev_free(b, nullptr);
    release_view(t->rem);
    delete t;
}

// Tiles of one orientation.  *out stays null where there are too few, and where they pay at none of the widths (*other_widths then).
mixgcn_status build_tiles(const mixgcn_graph* g, bool transposed, int32_t n_widths, const int32_t* widths, HubTiles** out, bool* other_widths, cudaStream_t s) {
    *out = nullptr;
    *other_widths = false;
    const CsrView &A = transposed ? g->bwd : g->fwd, &At = transposed ? g->fwd : g->bwd;
    const int64_t n = g->n, hubs = n < HUB_MAX ? n : HUB_MAX;
    if (g->nnz < HUB_MIN_ENTRIES) return MIXGCN_OK;
    const int rbs = (int)((hubs + ROWS - 1) / ROWS), cbs = (int)((hubs + COLS - 1) / COLS), total = rbs * cbs;
    // (given back on a failure below only when what writes to them is through: the stream does not wait for the null stream, nor that for it)
    struct Guard { HubTiles* t; cudaStream_t s; ~Guard() { if (t) cudaStreamSynchronize(s); free_tiles(t); } } guard{new (std::nothrow) HubTiles(), s};
    HubTiles* t = guard.t;
    if (!t) MIXGCN_FAIL(MIXGCN_ENOMEM, "hub tiles: host allocation failed");
    auto take = [&](void** p, int64_t bytes) -> mixgcn_status {
        if (g->ctx->debug_fail_alloc > 0 && --g->ctx->debug_fail_alloc == 0) MIXGCN_FAIL(MIXGCN_ENOMEM, "hub tiles: allocation made to fail (MIXGCN_OPT_DEBUG_FAIL_ALLOC)");
        return dev_alloc(p, bytes > 0 ? bytes : 1, s);
    };
    DevBuf rank(s), cnt(s), flag(s), first(s), tmp(s), totals(s), map(s), rem_len(s), tmp2(s);
    MIXGCN_TRY(take(&rank.p, n * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take(&cnt.p, total * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take(&flag.p, (total + 1) * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take(&first.p, (total + 1) * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take(&totals.p, sizeof(HubTotals)));
    MIXGCN_CUDA(cudaMemsetAsync(cnt.p, 0, total * sizeof(int32_t), s));
    MIXGCN_CUDA(cudaMemsetAsync(totals.p, 0, sizeof(HubTotals), s));
    rank_kernel<<<blocks_for(n), TPB, 0, s>>>(n, hubs, 0x7FFFFFFF, At.full.perm, rank.as<int32_t>());
    tile_count_kernel<<<(unsigned)hubs, TPB, 0, s>>>(cbs, A.full.perm, A.rowptr, A.col, rank.as<int32_t>(), cnt.as<int32_t>());
    tile_rows_kernel<<<(unsigned)rbs, TPB, 0, s>>>(cbs, HUB_TILE_MIN, PIECE_COST * HUB_TILE_MIN, cnt.as<int32_t>(), flag.as<int32_t>());
    tile_cols_kernel<<<(unsigned)cbs, TPB, 0, s>>>(rbs, cbs, HUB_TILE_MIN, COLUMN_COST, cnt.as<int32_t>(), flag.as<int32_t>(), totals.as<HubTotals>());
    size_t tb = 0;
    MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, flag.as<int32_t>(), first.as<int32_t>(), total + 1, s));
    MIXGCN_TRY(take(&tmp.p, (int64_t)tb));
    MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(tmp.p, tb, flag.as<int32_t>(), first.as<int32_t>(), total + 1, s));
    HubTotals h{};
    std::vector<int32_t> host_first(total + 1);
    MIXGCN_CUDA(cudaMemcpyAsync(&h, totals.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaMemcpyAsync(host_first.data(), first.p, (total + 1) * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    if ((int64_t)h.entries < HUB_MIN_ENTRIES / 4) return MIXGCN_OK;
    t->n_tiles = h.tiles; t->entries = (int64_t)h.entries;
    t->row_blocks = h.last_row_block + 1; t->kblocks = h.last_col_block + 1;
    t->n_cols = (int64_t)t->kblocks * COLS < n ? (int64_t)t->kblocks * COLS : n;
    const int64_t covered = (int64_t)t->row_blocks * ROWS, rows = covered < n ? covered : n;
    t->nodes = At.full.perm;
    // every pair of CTAs takes consecutive tiles, as many as any other where a piece counts as PIECE_COST tiles; a piece ends where a row of tiles does
    int clusters = 0;
    MIXGCN_TRY(resident_pairs(g->ctx, &clusters));
    if (clusters < 1) return MIXGCN_OK;
    // (fewer tiles than that are not worth a pair: the pieces of a row add up one behind the other)
    if (clusters > (t->n_tiles + LEAST_TILES - 1) / LEAST_TILES) clusters = (t->n_tiles + LEAST_TILES - 1) / LEAST_TILES;
    t->clusters = clusters;
    t->rem_nnz = g->nnz - t->entries;
    *other_widths = std::none_of(widths, widths + n_widths, [&](int32_t w) { return hub_tiles_pay(t, w); });
    if (*other_widths) return MIXGCN_OK;
    std::vector<HubPiece> pieces;
    std::vector<int32_t> first_piece(clusters + 1), piece_first(t->row_blocks + 1, 0);
    int rb = 0, at = 0, rows_of_tiles = 0;
    for (int i = 0; i < t->row_blocks; ++i) rows_of_tiles += host_first[(i + 1) * cbs] > host_first[i * cbs];
    const int64_t cost = t->n_tiles + (int64_t)PIECE_COST * (rows_of_tiles + clusters - 1);       // each pair but the first continues a row, or nearly
    for (int c = 0; c < clusters; ++c) {
        first_piece[c] = (int32_t)pieces.size();
        const int64_t end = c + 1 < clusters ? cost * (c + 1) / clusters : cost + t->n_tiles;
        while (at < t->n_tiles) {
            const int64_t room = end - (at + (int64_t)PIECE_COST * ((int64_t)pieces.size() + 1));
            if (room <= 0) break;
            while (host_first[(rb + 1) * cbs] <= at) ++rb;
            const int row_end = host_first[(rb + 1) * cbs], stop = row_end - at <= room ? row_end : at + (int)room;
            pieces.push_back(HubPiece{at, stop});
            piece_first[rb + 1]++;
            at = stop;
        }
    }
    first_piece[clusters] = (int32_t)pieces.size();
    for (int i = 0; i < t->row_blocks; ++i) piece_first[i + 1] += piece_first[i];
    t->n_pieces = (int)pieces.size();
    MIXGCN_TRY(take(&map.p, total * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take(&rem_len.p, (n + 1) * (int64_t)sizeof(int64_t)));
    MIXGCN_TRY(take((void**)&t->rank, n * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take((void**)&t->pieces, t->n_pieces * (int64_t)sizeof(HubPiece)));
    MIXGCN_TRY(take((void**)&t->first_piece, (clusters + 1) * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take((void**)&t->piece_first, (t->row_blocks + 1) * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take((void**)&t->tile_cb, t->n_tiles * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take((void**)&t->bits, t->n_tiles * (int64_t)ROWS * 16));
    MIXGCN_TRY(take((void**)&t->row_scale, rows * (int64_t)sizeof(float)));
    MIXGCN_TRY(take((void**)&t->col_scale, t->n_cols * (int64_t)sizeof(float)));
    MIXGCN_TRY(take((void**)&t->rem.rowptr, (n + 1) * (int64_t)sizeof(int64_t)));
    MIXGCN_CUDA(cudaMemcpyAsync(t->pieces, pieces.data(), pieces.size() * sizeof(HubPiece), cudaMemcpyHostToDevice, s));
    MIXGCN_CUDA(cudaMemcpyAsync(t->first_piece, first_piece.data(), first_piece.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    MIXGCN_CUDA(cudaMemcpyAsync(t->piece_first, piece_first.data(), piece_first.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    rank_kernel<<<blocks_for(n), TPB, 0, s>>>(n, rows, -1, A.full.perm, t->rank);
    tile_index_kernel<<<blocks_for(total), TPB, 0, s>>>(total, cbs, flag.as<int32_t>(), first.as<int32_t>(), map.as<int32_t>(), t->tile_cb);
    hub_scale_kernel<<<blocks_for(rows), TPB, 0, s>>>(rows, g->norm, transposed ? 0 : 1, A.full.perm, g->deg, g->dinv, t->row_scale);
    hub_scale_kernel<<<blocks_for(t->n_cols), TPB, 0, s>>>(t->n_cols, g->norm, transposed ? 1 : 0, At.full.perm, g->deg, g->dinv, t->col_scale);
    row_len_kernel<<<blocks_for(n + 1), TPB, 0, s>>>(n, A.rowptr, rem_len.as<int64_t>());
    tile_bits_kernel<<<(unsigned)covered, TPB, 0, s>>>(n, cbs, A.full.perm, A.rowptr, A.col, rank.as<int32_t>(), map.as<int32_t>(), reinterpret_cast<uint4*>(t->bits), rem_len.as<int64_t>());
    tb = 0;
    MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, rem_len.as<int64_t>(), t->rem.rowptr, n + 1, s));
    MIXGCN_TRY(take(&tmp2.p, (int64_t)tb));
    MIXGCN_CUDA(cub::DeviceScan::ExclusiveSum(tmp2.p, tb, rem_len.as<int64_t>(), t->rem.rowptr, n + 1, s));
    const int64_t room = t->rem_nnz > 0 ? t->rem_nnz : 1;
    MIXGCN_TRY(take((void**)&t->rem.col, room * (int64_t)sizeof(int32_t)));
    MIXGCN_TRY(take((void**)&t->rem.val, room * (int64_t)sizeof(float)));
    remainder_kernel<<<(unsigned)rows, TPB, 0, s>>>(cbs, A.full.perm, A.rowptr, A.col, A.val, rank.as<int32_t>(), map.as<int32_t>(), t->rem.rowptr, t->rem.col, t->rem.val);
    if (rows < n) other_rows_kernel<<<blocks_for((n - rows) * 32), TPB, 0, s>>>(rows, n, A.full.perm, A.rowptr, A.col, A.val, t->rem.rowptr, t->rem.col, t->rem.val);
    MIXGCN_CUDA(cudaGetLastError());
    MIXGCN_TRY(build_view_schedule(n, n, t->rem_nnz, t->rem, s));
    MIXGCN_CUDA(cudaStreamSynchronize(s));
    guard.t = nullptr;
    *out = t;
    return MIXGCN_OK;
}

std::mutex g_build_mutex;          // two threads that prepare the same graph

}  // namespace

namespace mixgcn {

void release_tiles(mixgcn_graph* g) {
    HubTiles *f = g->tiles[0].exchange(nullptr), *t = g->tiles[1].exchange(nullptr);
    if (t != f) free_tiles(t);
    free_tiles(f);
}

// Whether an aggregation of w columns is faster with the tiles, by what both sides take (us): what the gathers of the tiles' entries would
// take, against the product, the cut and what the other entries take longer in their own kernels (add_batch; nanoseconds an
// entry, steps where the lane split changes).  Fitted to eighteen graphs at fourteen widths; taken from a 16th of the call on, an 8th below 16 M
// entries, where the fit is right about the sign (a GIN layer's aggregations over 150 K nodes of mean degree 20 took 2 % longer to 1 % less).  Measured
// without : with (us), mean degree last, entries in tiles in brackets:
//   R-MAT 233 K, 500 (75 %)    256 columns 5035 : 2012, 132 4549 : 1404, 128 3212 : 1050, 64 1908 : 623, 41 1725 : 600
//   R-MAT 2.4 M, 52 (38 %)     256 7808 : 6938, 132 6159 : 4450, 64 2862 : 2188
//   R-MAT 300 K, 100 (62 %)    256 1471 : 1030, 132 970 : 514;  300 K, 31 (48 %)  256 562 : 499, 132 469 : 367, 64 210 : 183
//   R-MAT 100 K, 106 (74 %)    256 487 : 310, 132 434 : 220, 64 190 : 118;  20 K, 300 (91 %)  256 269 : 122, 132 252 : 88, 64 104 : 57
//   R-MAT 700 K, 22 (41 %)     256 1038 : 1021, 132 823 : 744, 64 383 : 359
//   8 K of 500 K nodes joined at random (59 %)  256 4124 : 2804, 64 1990 : 1330
// and left to the gather kernels: R-MAT 1.5 M, 21 (35 %)  256 2481 : 2506;  6 M, 17 (22 %)  256 9497 : 9590, 128 4 % slower with tiles;  1 M, 8 (22 %)
// 4 to 29 % slower;  50 K, 40 (66 %)  up to 64 columns 11 to 60 % slower;  ends drawn by rank^-0.8, 1 M, 40 (13 %)  256 3564 : 3956.
bool hub_tiles_pay(const HubTiles* t, int32_t w) {
    // (narrow calls over fewer than 16 M entries are short beside the launches that tiles add, and the fit is no help: 8 columns 3 to 26 % slower
    // with less than 95 % of the entries in tiles, up to 64 columns 30 % slower to 13 % faster with less than half)
    const bool small = t->entries + t->rem_nnz < (int64_t)1 << 24;
    if (small && ((w <= 12 && t->entries < 19 * t->rem_nnz) || (w <= 64 && t->entries < t->rem_nnz))) return false;
    const double tiles = (double)t->n_tiles / t->clusters;      // of a pair
    double all = 0, gain = 0;
    auto slice = [&](int32_t c) {
        const double entry = c > 192 ? 0.040 : c > 128 ? 0.0365 : c > 96 ? 0.0285 : c > 64 ? 0.0235 : 0.0028 + 0.0002 * (c > 8 ? c : 8);
        const double other = c > 192 ? 0.0086 : c > 128 ? 0.0035 : c > 96 ? 0.0061 : c > 64 ? 0.0016 : c > 48 ? 0.0024 : 0.0008;
        const Shape sh = make_shape(c);
        const double product = sh.blocks * (0.30 * tiles * (sh.cols > 40 ? sh.cols : 40) / 64 + 3.0);
        all += entry * 1e-3 * (t->entries + t->rem_nnz);
        gain += entry * 1e-3 * t->entries - other * 1e-3 * t->rem_nnz - product - 12.0 - 3.2e-6 * t->n_cols * c;
    };
    for (int32_t c0 = 0; c0 < w; c0 += HUB_SLICE) slice(w - c0 < HUB_SLICE ? w - c0 : HUB_SLICE);
    return gain * (small ? 8 : 16) > all;
}

int64_t hub_tiles_scratch(const HubTiles* t, int32_t w, int64_t ldp, int64_t* images_at) {
    const int64_t partial = (int64_t)t->n_pieces * ROWS * ldp * (int64_t)sizeof(float);
    *images_at = (partial + 1023) & ~(int64_t)1023;
    if (w > HUB_SLICE) w = HUB_SLICE;
    const Shape sh = make_shape(w);
    return *images_at + (int64_t)t->kblocks * 2 * PASSES_MAX * sh.blocks * sh.image_bytes();
}

mixgcn_status launch_hub_tiles(mixgcn_ctx* ctx, const HubTiles* t, int phase, int32_t w, const float* Y, int64_t ldy, int64_t y_rows, float* partial, int64_t ldp,
                               uint8_t* images, cudaStream_t s) {
    TileParams p{};
    p.pieces = t->pieces; p.first_piece = t->first_piece; p.tile_cb = t->tile_cb; p.bits = reinterpret_cast<const uint4*>(t->bits);
    p.partial = partial; p.ldp = ldp;
    p.w4 = (w + 3) >> 2; p.kblocks = t->kblocks;
    p.shape = make_shape(w);
    Ranges* ranges = reinterpret_cast<Ranges*>(ctx->d_status + TILES_WORD);
    p.ranges = ranges;
    p.Y = Y; p.ldy = ldy; p.y_rows = y_rows; p.nodes = t->nodes; p.col_scale = t->col_scale; p.n_cols = t->n_cols;
    p.status = ctx->d_status;
    p.wait_limit = ctx->debug_wait_limit > 0 ? (uint32_t)ctx->debug_wait_limit : WAIT_LIMIT_DEFAULT;
    p.drop_load = ctx->debug_drop_load;
    CUtensorMap map;
    if (!encode_2d(&map, images, 2, 64, (int64_t)PASSES_MAX * p.shape.blocks * t->kblocks * p.shape.n(), 64, 64, p.shape.n() / 2, CU_TENSOR_MAP_SWIZZLE_NONE))
        MIXGCN_FAIL(MIXGCN_ECUDA, "spmm: no tensor map for the images of the hub rows");
    {
        LaunchScope scope(ctx, phase, s, 2);
        int lanes = 0;
        while ((4 << lanes) < w) ++lanes;
        const int64_t rows = RANGE_THREADS >> lanes, most = 2 * (int64_t)ctx->sm_count, blocks = (t->n_cols + rows * 4 - 1) / (rows * 4);
        column_range_kernel<<<(unsigned)(blocks < most ? blocks : most), RANGE_THREADS, 0, s>>>(t->n_cols, w, lanes, t->nodes, t->col_scale, Y, ldy, y_rows, ranges, ctx->d_status);
        launch_chained(cut_rows_kernel, dim3((unsigned)(p.shape.blocks * p.shape.cols / GROUP), (unsigned)t->kblocks), 128, 0, s, t->n_cols, t->kblocks, p.shape, w, t->nodes, t->col_scale, Y, ldy,
                       y_rows, images, ranges, ctx->d_status);
    }
    MIXGCN_CUDA(cudaFuncSetAttribute(spmm_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TILES_SMEM));
    LaunchScope scope(ctx, phase, s);
    launch_chained(spmm_tiles_kernel, dim3((unsigned)t->clusters * 2), THREADS, TILES_SMEM, s, map, p);      // it sets up beside the kernel before
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

}  // namespace mixgcn

extern "C" mixgcn_status mixgcn_graph_layout_tiles(mixgcn_ctx* ctx, mixgcn_graph* g, int32_t n_widths, const int32_t* widths, int64_t* n_tiles, int64_t* n_entries) {
    if (!g || n_widths < 0 || (n_widths > 0 && !widths)) MIXGCN_FAIL(MIXGCN_EINVAL, "graph_layout_tiles: bad argument");
    constexpr int32_t ANY[] = {HUB_SLICE, 160, 128, 64};      // one of every lane split
    const int32_t n_asked = n_widths ? n_widths : 4, *asked = n_widths ? widths : ANY;
    std::lock_guard<std::mutex> lock(g_build_mutex);
    MIXGCN_CUDA(cudaSetDevice(g->device));
    HubTiles* made[2] = {nullptr, nullptr};
    bool other_widths[2] = {false, false};
    mixgcn_status st = MIXGCN_OK;
    for (int o = 0; o < 2 && st == MIXGCN_OK; ++o) {
        if (g->tiles_tried[o]) continue;
        if (o == 1 && (g->bwd_is_fwd || g->norm == 1)) {       // (row means transposed: see the errors above)
            made[1] = g->bwd_is_fwd ? made[0] : nullptr;
            other_widths[1] = g->bwd_is_fwd && other_widths[0];
            continue;
        }
        LaunchScope scope(g->ctx, PH_GRAPH, g->ctx->side_stream[0], 6);
        try {
            st = build_tiles(g, o == 1, n_asked, asked, &made[o], &other_widths[o], g->ctx->side_stream[0]);
        } catch (const std::bad_alloc&) {
            st = MIXGCN_ENOMEM;
        }
    }
    if (st != MIXGCN_OK) {             // (the gather kernels need none of it: where there is no memory for tiles there are none)
        free_tiles(made[0]);
        made[0] = made[1] = nullptr;
        other_widths[0] = other_widths[1] = false;
        if (st != MIXGCN_ENOMEM) return st;
    }
    for (int o = 0; o < 2; ++o)
        if (!g->tiles_tried[o]) {
            g->tiles[o].store(made[o], std::memory_order_release);
            g->tiles_tried[o] = !other_widths[o];
        }
    const HubTiles* t = g->tiles[0].load(std::memory_order_acquire);
    if (n_tiles) *n_tiles = t ? t->n_tiles : 0;
    if (n_entries) *n_entries = t ? t->entries : 0;
    if (!ctx) return MIXGCN_OK;
    for (const auto& tiles : g->tiles)
        for (int32_t i = 0; i < n_widths; ++i) MIXGCN_TRY(reserve_tiles_scratch(ctx, tiles.load(std::memory_order_acquire), widths[i]));
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_graph_prepare_tiles(mixgcn_graph* g, int64_t* n_tiles, int64_t* n_entries) {
    MIXGCN_TRY(mixgcn_graph_layout_tiles(nullptr, g, 0, nullptr, n_tiles, n_entries));
    // (recorded calls of mixgcn_spmm sum in the other order)
    if (!g->tiles_in_spmm.exchange(true, std::memory_order_acq_rel) && g->tiles[0].load(std::memory_order_acquire)) memory_given_back(g->memory);
    return MIXGCN_OK;
}
