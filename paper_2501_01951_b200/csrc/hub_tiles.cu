// Aggregation of the dense corner of a graph on the tensor cores.
//
// The nodes with the most entries neighbour one another: with rows and columns in order of descending entry counts, tiles of
// 256 x 128 near the corner hold thousands of the 32,768 possible entries.  The gather kernels fetch a row of Y for each of them; here a
// tile is a bitmap of 4 KB, and its product with 128 rows of Y is three tensor-core products.
//
//  * An entry's value is row_scale[u] * col_scale[v] (both normalisations and the plain sum have that form), so the matrix that is
//    multiplied holds zeros and ones only: exact in bf16.
//  * Rows of Y are scaled by col_scale (and 2^24, see CUT_SCALE) and cut into three bf16 parts, x = x0 + x1 + x2 (24 bits, as in gemm_split.cu), once per
//    call, into images of the shared-memory tiles (split_rows_kernel): a stage of the product is one contiguous copy a CTA.
//  * The x0 (8 bits each) are summed in an accumulator of their own, the two smaller parts in another: an instruction cuts its sum off
//    at 24 bits, towards zero, and sums of a hundred 8-bit numbers have next to nothing to lose there unless their sizes lie far apart.
//    Every 128 terms (the smaller parts, 2^-8 of the others: every 1024) the epilogue warps add the accumulator to fp32 sums in registers,
//    rounding to nearest, while others take the next terms: up to 160 columns leave room for two accumulators of the x0, up to 96 for four,
//    and there every 64 terms have one (narrow gathers add up in short chains, and a tile's time is its hand-overs': + 4 % of it).
//  * What is not in a tile is a matrix of its own, with a schedule of its own, for the gather kernels.  They run behind the tiles, and where
//    they have a row's sum add the row's pieces to it (at most 64 tiles of one row of tiles each, in fp64), times row_scale.
//
// Measured, R-MAT, 233 K nodes of mean degree 500 (20,470 tiles hold 74 % of the entries), 256 columns: 5.04 ms by gathers alone, 2.49 with the
// tiles (0.82 the product, 0.03 the cut, 1.7 the rest of the matrix); more cases at hub_tiles_pay.
// Bound: a tile of 256 x 128 by 256 columns takes a pair of CTAs 4,800 cycles, 3,072 of which its 24 instructions need; the rest is adding up
// the accumulator of the x0, which nothing covers above 160 columns (every 256 terms instead: 3,700 cycles, and the error below).  One
// CTA per tile of 128 x 128 took 5,630, bound by shared memory: a stage's image is written once and read once for 128 rows, here for
// 256.  Also slow: loads of 16 columns from the accumulator; bitmaps expanded by shift and multiply and announced to the other CTA by the
// expanding threads, whose arrival there waits for the loads they have under way (2,000 of 2,500 cycles).
// Error against fp64 relative to the gather kernels' (2-norm; N(0,1), its positive halves, what a ReLU leaves of it):
// R-MAT 300 K, mean degree 31, 132 columns 0.89, 0.88, 1.03; 60 K, 400 0.78, 0.72, 0.79, plain sums 0.38, 0.80, 0.78; 4,099 nodes, half of
// their pairs joined, 64 to 256 columns 0.7 to 0.9, 0.4 to 0.7, 0.5 to 0.7.  One row in a thousand 2^15 times the others: 0.7 to 1.0, of
// one sign 0.8 to 1.05 (60 K, plain sums, 64 columns 1.3).  Numbers of one sign spread further apart (exp(3 N(0,1))) are where
// truncation shows: 1.0 to 1.7.  What it took: 256 terms an accumulator made the last three 1.2 to 2.9; pieces of any length, added up
// in fp32, 2.1 of positive plain sums; the gather kernels' chains as they were 1.26 on the 300 K nodes.  Row means transposed are left
// out: the entries of small columns carry a row's sum there.
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

constexpr int ROWS = HUB_ROWS, COLS = HUB_COLS, PARTS = 3;
constexpr int HUB_MAX = 1 << 16, CB_MAX = HUB_MAX / COLS;       // most rows and columns that are looked at
constexpr int CHUNK_BYTES = COLS * 128;         // image of 128 rows of Y x 64 columns: 128-byte rows, 128-byte swizzle
constexpr int A_BYTES = 128 * COLS * 2;         // a CTA's rows of a tile expanded to bf16: two halves of 64 columns, K-major, 128-byte swizzle
constexpr int EPI_WARPS = 8, EXP_WARP = 8, EXP_WARPS = 4, TMA_WARP = 12, MMA_WARP = 13, RELAY_WARP = 14, THREADS = 512;
constexpr int EPI_REGS = 192, OTHER_REGS = 64;  // a thread's, of the 128 it is launched with
constexpr int STAGES_MAX = 8, STAGE_SMEM = 128 * 1024, BOX_BYTES = 4096;
constexpr int AHEAD = 4;
constexpr int LEAST_TILES = 8;                  // of a pair of CTAs
constexpr int LO_TILES = 8;                     // tiles that the accumulator of the smaller parts takes; that of the largest takes one
constexpr int PIECE_MAX = 64;                   // tiles of a piece: as many fp32 additions in a row
constexpr uint32_t TMEM_COLS = 512;
constexpr float SAFE_MAX = 0x1p100f;             // sums of 2^16 such terms stay finite
// Rows of Y are cut this many times as large: bf16 has nothing below 2^-133, and the third part of a number of 2^-110 and less would
// be gone (numbers of 1e-35: error 2e-6 to 1e-5 without, 2e-8 as the gathers have it with; 2^24 brings all of fp32 above the line).
constexpr float CUT_SCALE = 0x1p24f;

struct TileParams {
    const HubPiece* pieces; const int32_t* first_piece; // pair i takes pieces first_piece[i] .. first_piece[i + 1] - 1
    const int32_t* tile_cb; const uint4* bits;
    float* partial; int64_t ldp;                        // row r of piece q goes to partial row q * ROWS + r
    int w4, bn, chunks, stages;
    // TMEM: accumulators of bn columns, those of the largest parts first.  hi_two: 1 if tiles take turns in two sets of them, hi_halves: 1 if
    // the two halves of a tile's terms have one each; lo_col: the smaller parts' one
    uint32_t hi_two, hi_halves, lo_col;
    int32_t* unsafe;                                    // flag: not zero, plain_pieces instead, from what follows; then the CTAs done with it
    const float* Y; int64_t ldy, y_rows;
    const int32_t* nodes; const float* col_scale; int64_t n_cols;
    int32_t* status;
    uint32_t wait_limit;
    int drop_load;
};

struct Shared {
    uint64_t b_full[STAGES_MAX], b_empty[STAGES_MAX];   // images: TMA -> MMA -> TMA
    uint64_t a_full[2], a_empty[2];                     // expanded tiles: expansion -> MMA -> expansion
    uint64_t hi_full[2], hi_empty[2], lo_full, lo_empty;   // the accumulators: MMA -> epilogue -> MMA
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
__device__ __forceinline__ void add2(float& x, float& y, uint32_t a, uint32_t b) {
    asm("{.reg .b64 p, q; mov.b64 p, {%0, %1}; mov.b64 q, {%2, %3}; add.rn.f32x2 p, p, q; mov.b64 {%0, %1}, p;}" : "+f"(x), "+f"(y) : "r"(a), "r"(b));
}
// Whether the accumulator of the smaller parts is added up after tile i of the n of a piece.
__device__ __forceinline__ bool lo_ends(uint32_t i, uint32_t n) { return i + 1 == n || i % LO_TILES == LO_TILES - 1; }

// Where the column c (mod 32) of a tile's row has its bit: shifted left by c / 4 it is the highest bit of byte c % 4, and one
// permutation turns the highest bits of two bytes into the masks of two bf16 (2.5 instructions a pair instead of 5).
__host__ __device__ constexpr int bit_of(int c) { return 8 * (c & 3) + 7 - ((c >> 2) & 7); }
__host__ __device__ constexpr int column_of(int bit) { return 4 * (7 - (bit & 7)) + (bit >> 3); }

// columns 8 j .. 8 j + 7 of a word as bf16 zeros and ones
__device__ __forceinline__ uint4 expand8(uint32_t word, int j) {
    uint32_t r[4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t t = word << (2 * j + i);
        asm("prmt.b32 %0, %1, 0, 0x9988;" : "=r"(r[2 * i]) : "r"(t));            // (8: the byte's highest bit eight times)
        asm("prmt.b32 %0, %1, 0, 0xBBAA;" : "=r"(r[2 * i + 1]) : "r"(t));
        r[2 * i] &= 0x3F803F80u;
        r[2 * i + 1] &= 0x3F803F80u;
    }
    return make_uint4(r[0], r[1], r[2], r[3]);
}

// A pair's pieces on the FMA pipes, for calls in which a row of Y holds an infinity, a NaN or a number above 2^76, whose parts and sums
// the tensor core would not keep apart (0 * infinity): the expansion warps, one per row of a piece, entries in the order of their bits.
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

// A pair of CTAs (cluster of two, tcgen05 .cta_group::2) takes 256 rows, 128 each; each holds half of the columns of Y.
// The barriers b_full, hi_empty and lo_empty that count are the leader's, whose MMA warp waits on them; the others exist in both.
// Warps 0-7 epilogue (two per TMEM lane quarter, half of the columns each), 8-11 expansion (a thread per row of the tile),
// 12 copies, 13 MMA issue, 14 the peer's word to the leader, 15 none (register splits go by groups of four warps).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1) spmm_tiles_kernel(const __grid_constant__ CUtensorMap images, const TileParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) Shared b;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank(), pair = cluster_id_x();
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* stages = smem + 2 * A_BYTES;
    const uint32_t stage_bytes = (uint32_t)p.chunks * CHUNK_BYTES;
    int q0 = p.first_piece[pair], q1 = p.first_piece[pair + 1];
    if (threadIdx.x == 0) {
        b.abort_flag = 0;
        for (int s = 0; s < STAGES_MAX; ++s) { mbar_init(&b.b_full[s], 1); mbar_init(&b.b_empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&b.a_full[s], rank == 0 ? EXP_WARPS + 1 : EXP_WARPS); mbar_init(&b.a_empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&b.hi_full[s], 1); mbar_init(&b.hi_empty[s], 2 * EPI_WARPS); }
        mbar_init(&b.lo_full, 1); mbar_init(&b.lo_empty, 2 * EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == MMA_WARP) {              // (before the wait below: the kernel before this one, an ordinary launch, has no tensor memory)
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&b.tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                  // both CTAs' barriers exist before anything signals them
    tc_fence_after();
    const uint32_t tmem = b.tmem;
    asm volatile("griddepcontrol.wait;" ::: "memory");       // the images are complete
    const int q1_plain = q1;
    if (*p.unsafe) q1 = q0;
    const int t0 = q0 < q1 ? p.pieces[q0].begin : 0, t1 = q0 < q1 ? p.pieces[q1 - 1].end : 0;      // the pair's tiles are consecutive

    if (warp < EPI_WARPS) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(EPI_REGS));
        const int quarter = warp & 3, half = warp >> 2;
        const int hw = ((p.bn + 1) / 2 + 31) & ~31;                      // columns of a half: a multiple of 32, at most 128
        const int n0 = half * hw, chunks = n0 >= p.bn ? 0 : (min(hw, p.bn - n0) + 31) / 32;
        const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)n0;
        uint8_t* const box = stages + (size_t)p.stages * stage_bytes + warp * BOX_BYTES;
        uint32_t at = 0, lo_use = 0;            // at: tiles of the pair so far
        bool ok = true;
        for (int q = q0; q < q1 && ok; ++q) {
            const HubPiece piece = p.pieces[q];
            float sum[4][32];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < 32; ++i) sum[k][i] = 0.0f;
            auto add = [&](uint64_t* full, uint64_t* empty, uint32_t use, uint32_t col, uint32_t col_end) {
                if (!warp_wait(full, use, b, p)) return false;
                tc_fence_after();
#pragma unroll 1
                for (; col < col_end; col += (uint32_t)p.bn) {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k < chunks) {
                            uint32_t r[32];
                            tc_ld32(lanes + col + k * 32, r);
                            tc_wait_ld();
#pragma unroll
                            for (int i = 0; i < 32; i += 2) add2(sum[k][i], sum[k][i + 1], r[i], r[i + 1]);
                        }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(empty), 0));
                return true;
            };
            const uint32_t first = at, end = at + (uint32_t)(piece.end - piece.begin);
            for (; at < end && ok; ++at) {
                if (lo_ends(at - first, end - first)) { ok = add(&b.lo_full, &b.lo_empty, lo_use, p.lo_col, p.lo_col + 1); lo_use ^= 1; }
                const uint32_t slot = at & p.hi_two, set = (uint32_t)p.bn << p.hi_halves;
                if (ok) ok = add(&b.hi_full[slot], &b.hi_empty[slot], at >> p.hi_two & 1, slot * set, slot * set + set);
            }
            if (!ok) break;
            // through a box per warp, so that a request stores whole lines (a row per lane instead: 12,000 cycles a piece)
            float4* dst = reinterpret_cast<float4*>(p.partial + ((int64_t)q * ROWS + rank * 128 + quarter * 32) * p.ldp);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < chunks) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<float4*>(box + lane * 128 + ((i ^ (lane & 7)) << 4)) = make_float4(sum[k][i * 4], sum[k][i * 4 + 1], sum[k][i * 4 + 2], sum[k][i * 4 + 3]);
                    __syncwarp();
                    const int c4 = (n0 >> 2) + k * 8 + (lane & 7);
                    if (c4 < p.w4) {
#pragma unroll 2
                        for (int i = 0; i < 8; ++i) {
                            const int row = i * 4 + (lane >> 3);
                            const float4 x = *reinterpret_cast<const float4*>(box + row * 128 + (((lane & 7) ^ (row & 7)) << 4));
                            dst[row * (p.ldp >> 2) + c4] = make_float4(x.x * (1 / CUT_SCALE), x.y * (1 / CUT_SCALE), x.z * (1 / CUT_SCALE), x.w * (1 / CUT_SCALE));
                        }
                    }
                    __syncwarp();
                }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(OTHER_REGS));
        if (warp < TMA_WARP) {
            if (q1 != q1_plain) plain_pieces(p, q0, q1_plain, (int)rank);
            const int row = threadIdx.x - EXP_WARP * 32;
            const uint4* bits = p.bits + rank * 128 + row;
            uint4 next[AHEAD];              // bitmaps of the tiles to come
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) next[i] = t0 + i < t1 ? __ldg(bits + (int64_t)(t0 + i) * ROWS) : make_uint4(0, 0, 0, 0);
            Ring buf;
            bool ok = true;
            for (int t = t0; t < t1 && ok; t += AHEAD) {
#pragma unroll
                for (int i = 0; i < AHEAD; ++i) {           // (unrolled: a register that a load is under way to is not moved)
                    if (t + i >= t1) break;
                    if (!warp_wait(&b.a_empty[buf.i], buf.use ^ 1, b, p)) { ok = false; break; }
                    const uint32_t word[4] = {next[i].x, next[i].y, next[i].z, next[i].w};
                    uint8_t* dst = smem + buf.i * A_BYTES + row * 128;
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        *reinterpret_cast<uint4*>(dst + (j >> 3) * (A_BYTES / 2) + (((j & 7) ^ (row & 7)) << 4)) = expand8(word[j >> 2], j & 3);
                    if (t + i + AHEAD < t1) next[i] = __ldg(bits + (int64_t)(t + i + AHEAD) * ROWS);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&b.a_full[buf.i]);
                    buf.next(2);
                }
            }
        } else if (warp == TMA_WARP) {
            if (lane == 0) {
                Ring st;
                bool ok = true;
                for (int t = t0; t < t1 && ok; ++t) {
                    const int kb = __ldg(p.tile_cb + t);
                    for (int part = PARTS - 1; part >= 0; --part) {
                        if (!thread_wait(&b.b_empty[st.i], st.use ^ 1, b, p)) { ok = false; break; }
                        if (rank == 0) mbar_expect_tx(&b.b_full[st.i], 2 * stage_bytes);
                        if (!(p.drop_load && t == t0 && part == 0))
                            tma_load_2d_pair(stages + (size_t)st.i * stage_bytes, &images, 0, ((kb * PARTS + part) * 2 + (int)rank) * p.chunks * COLS, mapa_shared(smem_u32(&b.b_full[st.i]), 0));
                        st.next(p.stages);
                    }
                }
            }
        } else if (warp == RELAY_WARP && rank == 1) {
            // The peer's tiles are ready: told to the leader by a thread of its own, because an arrival in another CTA's memory waits
            // for all of the arriving thread's loads, which the expansion has under way all the time.
            if (lane == 0) {
                Ring buf;
                for (int t = t0; t < t1; ++t) {
                    if (!thread_wait(&b.a_full[buf.i], buf.use, b, p)) break;
                    mbar_arrive_cluster(mapa_shared(smem_u32(&b.a_full[buf.i]), 0));
                    buf.next(2);
                }
            }
        } else if (warp == MMA_WARP && rank == 0) {
            const uint32_t idesc = make_idesc<KIND_BF16>(ROWS, p.bn, false) | (1u << 16);      // A K-major, B MN-major
            Ring st, buf;
            uint32_t lo_use = 0, lo_more = 0;       // lo_more: the accumulator holds some already
            bool ok = true;
            for (int q = q0; q < q1 && ok; ++q) {
                const HubPiece piece = p.pieces[q];
                for (int t = piece.begin; t < piece.end && ok; ++t) {
                    ok = warp_wait(&b.a_full[buf.i], buf.use, b, p) && (lo_more || warp_wait(&b.lo_empty, lo_use ^ 1, b, p));
                    const bool ends = lo_ends((uint32_t)(t - piece.begin), (uint32_t)(piece.end - piece.begin));
                    const uint32_t k = (uint32_t)(t - t0), slot = k & p.hi_two;
                    const uint64_t a = make_desc(smem_u32(smem + buf.i * A_BYTES), 16, 1024, 2);
                    for (int s = 0; s < PARTS && ok; ++s) {
                        const bool hi = s == PARTS - 1;
                        if (!warp_wait(&b.b_full[st.i], st.use, b, p) || (hi && !warp_wait(&b.hi_empty[slot], (k >> p.hi_two & 1) ^ 1, b, p))) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t d = tmem + (hi ? (slot * (uint32_t)p.bn) << p.hi_halves : p.lo_col), half = hi ? p.hi_halves : 0u, more = s ? 1u : lo_more;
                        const uint64_t bd = make_desc(smem_u32(stages + (size_t)st.i * stage_bytes), CHUNK_BYTES, 1024, 2);
                        if (elect_one()) {
#pragma unroll
                            for (int j = 0; j < COLS / 16; ++j)
                                tc_mma_pair<KIND_BF16>(d + (half & j >> 2) * (uint32_t)p.bn, a + (j >> 2) * (A_BYTES / 2 / 16) + (j & 3) * 2, bd + j * 128, idesc,
                                                       hi ? (j & (half ? 3 : 7)) != 0 : j ? 1u : more);
                            tc_commit_pair(&b.b_empty[st.i], 3);
                            if (s == PARTS - 2 && ends) tc_commit_pair(&b.lo_full, 3);
                            if (hi) tc_commit_pair(&b.a_empty[buf.i], 3);
                            if (hi) tc_commit_pair(&b.hi_full[slot], 3);
                        }
                        __syncwarp();
                        st.next(p.stages);
                    }
                    lo_use ^= ends; lo_more = !ends;
                    buf.next(2);
                }
            }
        }
    }
    __syncwarp();
    if (threadIdx.x == 0 && b.abort_flag)
        for (int i = 0; i < 200; ++i) __nanosleep(1000);      // a wait expired: let copies in flight land
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                  // the peer is done with this CTA's shared and tensor memory
    if (threadIdx.x == 0) {              // the flag is this call's alone: the last CTA that has read it clears it
        __threadfence();
        if (atomicInc(reinterpret_cast<unsigned int*>(p.unsafe) + 1, gridDim.x - 1) == gridDim.x - 1) *p.unsafe = 0;      // (back at zero itself)
    }
    if (warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Rows of Y of the hub columns -> images of their three bf16 parts: images[column block][part][half of the columns of Y][chunk of 64
// columns], a chunk as the tensor core wants it in shared memory.  Eight lanes a row and chunk, eight columns each.  The product by
// the scale is cut with its rounding error added to the last part, so the scaling itself rounds nothing.
__global__ void __launch_bounds__(256) split_rows_kernel(int64_t n_cols, int kblocks, int chunks, int nh, int w, const int32_t* __restrict__ nodes, const float* __restrict__ scale,
                                                         const float* __restrict__ Y, int64_t ldy, int64_t y_rows, uint8_t* __restrict__ images, int32_t* unsafe, int32_t* status) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int g = (int)(i & 7), k = (int)((i >> 3) & (COLS - 1));
    const int64_t kc = (i >> 3) / COLS, kb = kc / (2 * chunks);
    const int chunk = (int)(kc % (2 * chunks)), half = chunk / chunks, in_half = (chunk - half * chunks) * 64 + g * 8;
    const int c0 = in_half < nh ? half * nh + in_half : w;
    if (kb >= kblocks) return;
    float x[8], lost[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = lost[j] = 0.0f;
    const int64_t h = kb * COLS + k;
    if (h < n_cols && c0 < w) {
        const int64_t v = __ldg(nodes + h);
        if (index_ok(v, y_rows, status, SITE_SPMM_COL)) {
            const float4* src = reinterpret_cast<const float4*>(Y + v * ldy + c0);
            const float4 a = __ldg(src), c = c0 + 4 < w ? __ldg(src + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
            const float s = __ldg(scale + h) * CUT_SCALE, y[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
            bool bad = false;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (c0 + j < w) { x[j] = y[j] * s; lost[j] = fmaf(y[j], s, -x[j]); bad |= !(fabsf(x[j]) < SAFE_MAX); }
            if (bad) *unsafe = 1;
        }
    }
    uint8_t* dst = images + (kb * PARTS * 2 * chunks + chunk) * (int64_t)CHUNK_BYTES + k * 128 + ((g ^ (k & 7)) << 4);
#pragma unroll
    for (int part = 0; part < PARTS; ++part) {
        uint32_t r[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            r[j] = pack_bf16(x[2 * j], x[2 * j + 1]);
            x[2 * j] -= __uint_as_float(r[j] << 16);
            x[2 * j + 1] -= __uint_as_float(r[j] & 0xFFFF0000u);
            if (part == 1) { x[2 * j] += lost[2 * j]; x[2 * j + 1] += lost[2 * j + 1]; }
        }
        *reinterpret_cast<uint4*>(dst + (int64_t)part * 2 * chunks * CHUNK_BYTES) = make_uint4(r[0], r[1], r[2], r[3]);
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

__global__ void tile_select_kernel(int total, int cbs, int least, const int32_t* __restrict__ cnt, int32_t* __restrict__ flag, HubTotals* totals) {
    const int i = blockIdx.x * TPB + threadIdx.x;
    if (i > total) return;
    const bool on = i < total && cnt[i] >= least;
    flag[i] = on ? 1 : 0;              // one more than there are tiles: the scan's last element is their number
    if (!on) return;
    atomicAdd(&totals->entries, (unsigned long long)cnt[i]);
    atomicAdd(&totals->tiles, 1);
    atomicMax(&totals->last_row_block, i / cbs);
    atomicMax(&totals->last_col_block, i % cbs);
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

// CTA pairs of the product that run at once; none if it does not have the registers that its split hands out (an increase beyond the
// launch's registers would wait for ever)
mixgcn_status resident_pairs(const mixgcn_ctx* ctx, int* pairs) {
    *pairs = 0;
    cudaFuncAttributes fa;
    MIXGCN_CUDA(cudaFuncGetAttributes(&fa, spmm_tiles_kernel));
    if (fa.numRegs * THREADS < EPI_REGS * EPI_WARPS * 32 + OTHER_REGS * (THREADS - EPI_WARPS * 32)) return MIXGCN_OK;
    const int smem = 2 * A_BYTES + STAGE_SMEM + EPI_WARPS * BOX_BYTES + 1024;
    MIXGCN_CUDA(cudaFuncSetAttribute(spmm_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(ctx->sm_count & ~1), 1, 1); cfg.blockDim = dim3(THREADS, 1, 1); cfg.dynamicSmemBytes = smem;
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
    tile_select_kernel<<<blocks_for(total + 1), TPB, 0, s>>>(total, cbs, HUB_TILE_MIN, cnt.as<int32_t>(), flag.as<int32_t>(), totals.as<HubTotals>());
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
    // every pair of CTAs takes as many consecutive tiles as any other; a piece ends where a row of tiles does
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
    int rb = 0;
    for (int c = 0; c < clusters; ++c) {
        first_piece[c] = (int32_t)pieces.size();
        const int end = (int)((int64_t)t->n_tiles * (c + 1) / clusters);
        for (int at = (int)((int64_t)t->n_tiles * c / clusters); at < end;) {
            while (host_first[(rb + 1) * cbs] <= at) ++rb;
            const int row_end = host_first[(rb + 1) * cbs];
            int stop = row_end < end ? row_end : end;
            if (stop > at + PIECE_MAX) stop = at + PIECE_MAX;
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
// entry, steps where the lane split changes).  A pair's first 32 tiles are dearer: graphs with few tiles have them spread over many rows and
// columns, and the images come from DRAM.  Fitted to the profiles of eleven graphs; taken from a 32nd of the call on, where the fit
// is right about the sign but for 100 K nodes at 48 columns (178 : 181).  Measured without : with (us), mean degree last, entries in tiles in brackets:
//   R-MAT 233 K, 500 (74 %)    256 columns 5036 : 2494, 132 4542 : 1711, 128 3205 : 1359, 64 1907 : 1002, 32 1284 : 835
//   R-MAT 2.4 M, 52 (28 %)     256 7846 : 7629, 132 6107 : 5168, 128 4401 : 3926, 48 2766 : 2202
//   R-MAT 300 K, 31 (34 %)     192 466 : 443, 132 459 : 412;  100 K, 106 (61 %)  256 521 : 430, 128 334 : 253, 64 206 : 188
//   R-MAT 20 K, 300 (83 %)     256 276 : 165, 64 113 : 87;  8 K of 500 K nodes joined at random (51 %)  256 1907 : 1617, 64 586 : 525
// and left to the gather kernels: R-MAT 300 K, 31  256 550 : 552, 128 313 : 303, 64 205 : 218;  700 K, 22 (28 %)  256 1002 : 1072,
// 132 789 : 810, 128 527 : 581;  1.5 M, 21 (23 %)  256 2193 : 2331, 132 1721 : 1711;  ends drawn by rank^-0.6, 300 K, 100 (4 %)  256 2142 : 2396,
// 128 1022 : 1164, by rank^-0.8, 1 M, 40 (11 %)  256 3315 : 3754, 132 2362 : 2309.
bool hub_tiles_pay(const HubTiles* t, int32_t w) {
    const double tiles = (double)t->n_tiles / t->clusters, first = tiles < 32 ? tiles : 32;      // of a pair
    double all = 0, gain = 0;
    auto slice = [&](int32_t c) {
        const double entry = c > 192 ? 0.036 + 0.00003 * (c - 192) : c > 160 ? 0.036 : c > 128 ? 0.037 : c > 64 ? 0.026 : c > 24 ? 0.005 + 0.00016 * c : 0.0088;
        const double other = c > 192 ? 0.0078 : c > 128 ? 0.0045 : c > 64 ? 0.004 : 0.001;
        const double product = c > 160 ? (1.72 + 0.0076 * (c - 160)) * tiles + (2.8 + 0.0085 * (c - 160)) * first
                                       : c > 128 ? 1.72 * tiles + 2.8 * first : c > 64 ? 1.5 * tiles + 2.3 * first : 1.45 * tiles + 1.6 * first;
        all += entry * 1e-3 * (t->entries + t->rem_nnz);
        gain += entry * 1e-3 * t->entries - other * 1e-3 * t->rem_nnz - product - 10.0 - 2e-6 * t->n_cols * c;
    };
    for (int32_t c0 = 0; c0 < w; c0 += HUB_SLICE) slice(w - c0 < HUB_SLICE ? w - c0 : HUB_SLICE);
    return gain * 32 > all;
}

// columns of a half of Y, chunks of 64 of them
inline int half_cols(int32_t w) { return (w + 31) / 32 * 16; }
inline int half_chunks(int32_t w) { return (half_cols(w) + 63) / 64; }

int64_t hub_tiles_scratch(const HubTiles* t, int32_t w, int64_t ldp, int64_t* images_at) {
    const int64_t partial = (int64_t)t->n_pieces * ROWS * ldp * (int64_t)sizeof(float);
    *images_at = (partial + 1023) & ~(int64_t)1023;
    if (w > HUB_SLICE) w = HUB_SLICE;
    return *images_at + (int64_t)t->kblocks * PARTS * 2 * half_chunks(w) * CHUNK_BYTES;
}

mixgcn_status launch_hub_tiles(mixgcn_ctx* ctx, const HubTiles* t, int phase, int32_t w, const float* Y, int64_t ldy, int64_t y_rows, float* partial, int64_t ldp,
                               uint8_t* images, cudaStream_t s) {
    TileParams p{};
    p.pieces = t->pieces; p.first_piece = t->first_piece; p.tile_cb = t->tile_cb; p.bits = reinterpret_cast<const uint4*>(t->bits);
    p.partial = partial; p.ldp = ldp;
    p.w4 = (w + 3) >> 2; p.bn = half_cols(w) * 2; p.chunks = half_chunks(w);
    const int fit = STAGE_SMEM / (p.chunks * CHUNK_BYTES);
    p.stages = fit < STAGES_MAX ? fit : STAGES_MAX;
    p.hi_two = p.bn * 3 <= (int)TMEM_COLS ? 1 : 0;
    p.hi_halves = p.bn * 5 <= (int)TMEM_COLS ? 1 : 0;
    p.lo_col = (uint32_t)p.bn << (p.hi_two + p.hi_halves);
    p.unsafe = ctx->d_status + TILES_UNSAFE_WORD;
    p.Y = Y; p.ldy = ldy; p.y_rows = y_rows; p.nodes = t->nodes; p.col_scale = t->col_scale; p.n_cols = t->n_cols;
    p.status = ctx->d_status;
    p.wait_limit = ctx->debug_wait_limit > 0 ? (uint32_t)ctx->debug_wait_limit : WAIT_LIMIT_DEFAULT;
    p.drop_load = ctx->debug_drop_load;
    CUtensorMap map;
    const int64_t image_rows = (int64_t)t->kblocks * PARTS * 2 * p.chunks * COLS;
    if (!encode_2d(&map, images, 2, 64, image_rows, 64, 64, p.chunks * COLS, CU_TENSOR_MAP_SWIZZLE_NONE)) MIXGCN_FAIL(MIXGCN_ECUDA, "spmm: no tensor map for the images of the hub rows");
    {
        LaunchScope scope(ctx, phase, s);
        const int64_t threads = (int64_t)t->kblocks * COLS * 2 * p.chunks * 8;
        split_rows_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(t->n_cols, t->kblocks, p.chunks, p.bn / 2, w, t->nodes, t->col_scale, Y, ldy, y_rows, images, p.unsafe,
                                                                            ctx->d_status);
    }
    const size_t smem = 2 * A_BYTES + (size_t)p.stages * p.chunks * CHUNK_BYTES + EPI_WARPS * BOX_BYTES + 1024;
    MIXGCN_CUDA(cudaFuncSetAttribute(spmm_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    LaunchScope scope(ctx, phase, s);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)t->clusters * 2, 1, 1); cfg.blockDim = dim3(THREADS, 1, 1); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // it sets up beside the kernel before
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    MIXGCN_CUDA(cudaLaunchKernelEx(&cfg, spmm_tiles_kernel, map, p));
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
