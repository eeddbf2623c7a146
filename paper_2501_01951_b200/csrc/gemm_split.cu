// fp32 dense products on the tensor cores: every fp32 operand is cut into three bf16 parts, a = a0 + a1 + a2 with each part the
// rounded-to-nearest bf16 of what the parts before it leave.  8 + 8 + 8 bits: the three parts ARE the fp32 value (as long as
// they stay above bf16's smallest number, 2^-133), and a product of two parts is exact in fp32.  Of the nine products of parts
// the six down to 2^-16 of the largest are formed; the three left out are below 2^-25 of |a b| together, half a unit of an
// fp32 rounding, and not all of one sign.  The split of matrices into parts that multiply without error is that of Ozaki,
// Ogita, Oishi and Rump ("Error-free transformations of matrix multiplication", 2012).
//
// What the tensor core does not do is round to nearest.  An instruction aligns its 16 products and the accumulator to the
// largest of them, cuts each off 25 bits below it, towards zero, adds exactly and cuts the sum off at 24 bits (so its
// results say: bf16 operands of one instruction against fp64).  What is cut off does not average out; these things keep it small:
//  * the large products a0 b0 are accumulated over few terms only; the epilogue warps add the accumulator to fp32 sums in
//    registers, rounding to nearest, while the next terms go to a second accumulator;
//  * the five small products, at most 2^-7 of the large ones, have an accumulator of their own.
// K-major: 32 terms (two instructions) an accumulator, one chain of sums, at most 1024 terms.  Against fp64 its results are closer
// than the FMA kernel's single chain on everything a layer multiplies (activations, features and gradients by weights: 0.2 to
// 0.8 of its error).
// Weight gradient: its operands cancel -- most entries of a column of a softmax gradient are small and of one sign, a few are large
// and of the other -- and the small terms beside a large one are what is cut off.  So it accumulates 16 terms (one instruction)
// at a time; the first part of A keeps seven bits, which makes products of 15 that lose nothing down to 2^-10 of the
// largest (the three parts still hold all 24 bits; the parts left out grow to 2^-22 at most, 2^-26 in the mean, of either
// sign); and every 512 terms the sums go to a second sum in TMEM, the rounding error of that addition going on into the next sums.
// ReLU activations or 0 / 1 features by softmax gradients, error against the FMA kernel's: 256 x 40 over 170 K rows 0.43 to 0.97
// of it, 128 x 80 over 524 K 0.28 to 0.79; where it comes out above (up to 1.2, with 1 to 10 % of the rows labelled) both are below one
// rounding of the result, 2^-24.  (With 32 terms, eight bits and one chain it was up to 1.47 of it, for 156 us instead of 174 at 170 K x 256 x 256.)
// Operands of one sign, which training does not multiply, may come out at up to 1.8 of the FMA kernel's error, near one rounding.
//
// Bound: the hand-overs between the roles.  A stage of 32 terms of a 128 x 128 tile is twelve instructions, 768 cycles of the
// tensor core, and takes about 1,800: raw tile, conversion, MMA and epilogue follow one another, with the three stages of part
// tiles in flight that shared memory holds.  Tensor pipe 40 to 43 % active (of 270 TFLOP/s of fp32 products; the FMA pipes
// have 72), shared-memory banks 41 %, issue slots 40 to 54 %.
// Measured against the FMA kernel, calls back to back: 170 K x 256 x 256 forward 501 -> 162 us (138 TFLOP/s), its weight
// gradient 464 -> 174, 170 K x 40 x 256 144 -> 77, 1 M x 300 x 300 4494 -> 1482.
// Behind every such product runs the FMA kernel's grid, which reads one zero word per block and returns (see the overflow
// below): 5 us at 170 K x 256 x 256, 23 us (39 thousand blocks) at 1 M x 300 x 300, 3 us and 4 of its reduction for a weight gradient.
//
// What the layout of the work has to avoid is the latency of one stage's hand-overs in series (a wait, a proxy fence and an
// arrival each): one group of conversion warps on every stage took 212 us where two groups on alternate stages take 178;
// loads to registers before the fence instead of raw tiles by TMA, as much; the large products issued before the small ones
// (the wait for their accumulator in front), 190; issue by a divergent lane instead of an elected one of a converged warp, 10 % more.
//
// Infinities, values that round to a bf16 infinity and sums out of fp32's range do not survive the split (inf - inf): whatever is not
// finite in an operand or in a sum is a NaN or an infinity in the sums of its row.  The epilogue warps record that they met one,
// and the FMA kernel, launched behind, then computes the product over again (otherwise it returns at once).
// A value below 2^-109 keeps an absolute error of up to 2^-134, its last part being a bf16 subnormal.
//
//  * K-major form (forward, input gradient): persistent CTAs over 128 x bn tiles; the weights are cut once into three packed
//    planes, which TMA brings in; the fp32 tiles of A come by TMA too, and the conversion warps cut them into part tiles.
//  * MN-major form (weight gradient): K split over CTAs, both operands converted by the CTA that multiplies them.
// Warps 0-7 epilogue (two per TMEM lane quarter, half of the columns each), 8-15 conversion, 16 TMA, 17 MMA issue.
#include "internal.cuh"
#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"

using namespace mixgcn;
using namespace mixgcn::tc;

namespace {

constexpr int BM = 128, BN_MAX = 128, BK = 32, PARTS = 3;
constexpr int EPI_WARPS = 8, CONV_WARPS = 8, TMA_WARP = EPI_WARPS + CONV_WARPS, MMA_WARP = TMA_WARP + 1, THREADS = (MMA_WARP + 1) * 32;
constexpr int GROUPS = 2, GROUP_WARPS = CONV_WARPS / GROUPS, GROUP_THREADS = GROUP_WARPS * 32;   // groups of conversion warps, on alternate stages
constexpr int STAGES_MAX = 4, RAW_MAX = 8;      // most stages of part tiles and slots of raw fp32 tiles (a multiple of 2 * GROUPS)
static_assert(RAW_MAX % (2 * GROUPS) == 0);
// How a form adds up.  HI: accumulators of the large products per stage.  LO: stages per accumulator of the small products.
// LEVELS: 1: the sums stay in registers to the end; 2: every LO stages they are carried over to a second sum in TMEM.
// TRIM_A: 1: the first part of A keeps seven bits instead of eight.
struct KkSums { static constexpr int HI = 1, LO = 1024 / BK, LEVELS = 1, TRIM_A = 0; };
struct MmSums { static constexpr int HI = 2, LO = 512 / BK, LEVELS = 2, TRIM_A = 1; };
constexpr uint32_t TMEM_COLS = 512, BUF_COLS = 128;     // two accumulators for the large products, then
constexpr uint32_t LO_COL = 256, SUM_COL = 384;         // two for the small ones, or one and the second sum
constexpr uint32_t CVT_COLS = 256;              // the two accumulators of the bf16 form
constexpr int RAW_BYTES = BM * BK * 4, KK_PART = BM * BK * 2;       // a raw tile; K-major part tiles: 64-byte rows and swizzle
constexpr int CHUNK = BK * 128, MM_PART = BM / 64 * CHUNK;          // MN-major tiles: chunks of 64 columns, 128-byte k-rows and swizzle

struct SplitParams {
    int64_t M, N, K;
    int bn;                       // columns of a tile: a multiple of 16 up to BN_MAX
    int64_t m_tiles, n_tiles;
    int stages, raw_slots;
    int plane_rows;               // K-major: rows of one packed plane of B
    int64_t k_per_split;          // MN-major: a multiple of BK
    float* C; int64_t ldc; int vec_c;   // MN-major: partial tiles [splits][M][N] or C itself
    int raw;
    double* colsum_part;          // MN-major, nullable: [splits][m_tiles][N] column sums of B over the k-rows a CTA added up
    TcEpi epi;
    int32_t* status;
    uint32_t wait_limit;
    int drop_load;                // test hook: every CTA's first raw tile is left out (the wait for it then expires)
    int32_t* overflow;            // set when a sum is not finite
};

struct Ring {                     // position in a ring of slots and the parity of its use
    int i = 0;
    uint32_t use = 0;
    __device__ __forceinline__ void next(int n, int by = 1) { if ((i += by) >= n) { i -= n; use ^= 1; } }      // by <= n
};

// Position among the raw tiles.  They go through `raw_slots` slots, but their barriers go by eights: so all uses of one barrier are
// the same group's, which has seen the one before.  (By slots, three or five of them, a group could wait on a barrier whose last
// use, the other group's, is still in flight, and take the use before that for its own: loads land out of order.)
struct RawRing {
    uint32_t unit = 0;
    int slot = 0;
    __device__ __forceinline__ void next(int n, int by = 1) { unit += by; if ((slot += by) >= n) slot -= n; }       // by <= n
    __device__ __forceinline__ uint32_t bar() const { return unit % RAW_MAX; }
    __device__ __forceinline__ uint32_t use() const { return unit / RAW_MAX & 1; }
};

__device__ __forceinline__ void add2(float& x, float& y, float a, float b) {
    asm("{.reg .b64 p, q; mov.b64 p, {%0, %1}; mov.b64 q, {%2, %3}; add.rn.f32x2 p, p, q; mov.b64 {%0, %1}, p;}" : "+f"(x), "+f"(y) : "f"(a), "f"(b));
}
// (x, y) minus the two bf16 values of `parts`: exact
__device__ __forceinline__ void sub_parts(float& x, float& y, uint32_t parts) {
    asm("{.reg .b64 p, q, m; mov.b64 p, {%0, %1}; mov.b64 q, {%2, %3}; mov.b64 m, {%4, %4}; fma.rn.f32x2 p, q, m, p; mov.b64 {%0, %1}, p;}"
        : "+f"(x), "+f"(y) : "f"(__uint_as_float(parts << 16)), "f"(__uint_as_float(parts & 0xFFFF0000u)), "f"(-1.0f));
}

// Four floats -> their three bf16 parts at dst + t * part_bytes.
template <int TRIM>
__device__ __forceinline__ void split4(float4 v, uint8_t* dst, uint32_t part_bytes) {
#pragma unroll
    for (int t = 0; t < PARTS; ++t) {
        uint32_t lo = pack_bf16(v.x, v.y), hi = pack_bf16(v.z, v.w);
        if (TRIM && t == 0) {            // to seven bits, away from zero (a NaN is lost here and comes back in the parts behind)
            lo = (lo + 0x00010001u) & 0xFFFEFFFEu;
            hi = (hi + 0x00010001u) & 0xFFFEFFFEu;
        }
        *reinterpret_cast<uint2*>(dst + t * part_bytes) = make_uint2(lo, hi);
        if (t + 1 < PARTS) { sub_parts(v.x, v.y, lo); sub_parts(v.z, v.w, hi); }
    }
}

// This thread's share of a raw tile: the float4 t, t + 128, ...
constexpr int RAW_ITS = BM * BK / 4 / GROUP_THREADS;
template <int N>
__device__ __forceinline__ void take_raw(float4 (&v)[N], const uint8_t* tile, int t) {
#pragma unroll
    for (int it = 0; it < N; ++it) v[it] = reinterpret_cast<const float4*>(tile)[t + it * GROUP_THREADS];
}

// barriers of a CTA, TMEM address and abort flag
struct Shared {
    uint64_t raw_full[RAW_MAX], raw_empty[RAW_MAX];   // raw fp32 tiles: TMA -> conversion -> TMA
    uint64_t full[STAGES_MAX], empty[STAGES_MAX];             // part tiles: conversion (and TMA) -> MMA -> conversion
    uint64_t hi_full[2], hi_empty[2], lo_full[2], lo_empty[2];   // accumulators: MMA -> epilogue -> MMA
    uint32_t tmem;
    int abort_flag;
};

__device__ __forceinline__ uint32_t cta_begin(Shared& b, int full_count, int warp) {
    if (threadIdx.x == 0) {
        b.abort_flag = 0;
        for (int s = 0; s < RAW_MAX; ++s) { mbar_init(&b.raw_full[s], 1); mbar_init(&b.raw_empty[s], GROUP_WARPS); }
        for (int s = 0; s < STAGES_MAX; ++s) { mbar_init(&b.full[s], (uint32_t)full_count); mbar_init(&b.empty[s], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&b.hi_full[s], 1); mbar_init(&b.hi_empty[s], EPI_WARPS); mbar_init(&b.lo_full[s], 1); mbar_init(&b.lo_empty[s], EPI_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&b.tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    return b.tmem;
}

__device__ __forceinline__ void cta_end(Shared& b, int warp, uint32_t tmem) {
    if (threadIdx.x == 0 && b.abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);      // a wait expired: let copies in flight land
    }
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

__device__ __forceinline__ bool thread_wait(uint64_t* bar, uint32_t parity, Shared& b, const SplitParams& p) {
    volatile int* flag = &b.abort_flag;
    if (mbar_wait(bar, parity, flag, p.wait_limit)) return true;
    *flag = 1;
    atomicMax(p.status, DEV_WAIT_EXPIRED);
    return false;
}
// The slot of the next raw tile is free: the tile raw_slots back has been taken.
__device__ __forceinline__ bool raw_free(const RawRing& raw, Shared& b, const SplitParams& p) {
    if (raw.unit < (uint32_t)p.raw_slots) return true;
    const uint32_t last = raw.unit - p.raw_slots;
    return thread_wait(&b.raw_empty[last % RAW_MAX], last / RAW_MAX & 1, b, p);
}
// One wait of a whole warp.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, Shared& b, const SplitParams& p) {
    return __all_sync(0xFFFFFFFFu, thread_wait(bar, parity, b, p)) != 0;
}

// add an accumulator (this warp's 32 lanes, `chunks` blocks of 32 columns) to the sums in registers
__device__ __forceinline__ void add_accumulator(uint32_t taddr, int chunks, float (&acc)[2][32]) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (k < chunks) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t r[16];
                tc_ld16(taddr + (uint32_t)(k * 32 + h * 16), r);
                tc_wait_ld();
#pragma unroll
                for (int q = 0; q < 16; q += 2) add2(acc[k][h * 16 + q], acc[k][h * 16 + q + 1], __uint_as_float(r[q]), __uint_as_float(r[q + 1]));
            }
        }
}

// The sums in registers to the second sum in TMEM, s; what its rounding leaves of them stays behind (the error of a sum is the
// difference of two sums: Knuth, The Art of Computer Programming, 4.2.2), so that the second level adds no error of its own.
__device__ __forceinline__ void carry_over(uint32_t taddr, int chunks, bool first, float (&acc)[2][32]) {
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (k < chunks) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t at = taddr + (uint32_t)(k * 32 + h * 16);
                uint32_t r[16];
                if (!first) {
                    tc_ld16(at, r);
                    tc_wait_ld();
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const float a = acc[k][h * 16 + q], s = first ? 0.0f : __uint_as_float(r[q]);
                    const float t = __fadd_rn(s, a), b = __fsub_rn(t, s);
                    acc[k][h * 16 + q] = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(a, b));
                    r[q] = __float_as_uint(t);
                }
                tc_st16(at, r);
            }
        }
    tc_wait_st();
}

// Whether the sums of this warp's first `cols` columns (a multiple of 16) are all finite: 0 times anything else is NaN.
__device__ __forceinline__ bool all_finite(const float (&acc)[2][32], int cols) {
    float x = 0.0f, y = 0.0f;
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (k * 32 + h * 16 < cols) {
#pragma unroll
                for (int q = h * 16; q < h * 16 + 16; q += 2)
                    asm("{.reg .b64 p, z, s; mov.b64 p, {%2, %3}; mov.b64 z, {%4, %4}; mov.b64 s, {%0, %1}; fma.rn.f32x2 s, p, z, s; mov.b64 {%0, %1}, s;}"
                        : "+f"(x), "+f"(y) : "f"(acc[k][q]), "f"(acc[k][q + 1]), "f"(0.0f));
            }
    return x + y == 0.0f;
}

// The MMA warp's state: position in the stages and in the two pairs of accumulators.
struct MmaState {
    Ring stage;
    uint32_t hc = 0, lc = 0;
    int lo_used = 0;              // stages in the current accumulator of the small products
};

// One lane of a converged warp, always the same one.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{.reg .pred q; elect.sync _|q, 0xFFFFFFFF; selp.u32 %0, 1, 0, q;}" : "=r"(p));
    return p != 0;
}

// All products of one stage, by the whole MMA warp: uniform control flow up to the elected lane leaves the descriptors in uniform
// registers.  desc_a, desc_b: descriptors of the first part tiles, the others a_part and b_part bytes on, the second 16
// terms k_step bytes on (the address is the descriptor's low field, in units of 16 bytes).  last: no stage of this tile follows.
template <class Sums>
__device__ __forceinline__ bool mma_stage(MmaState& st, Shared& b, const SplitParams& p, uint32_t tmem, uint32_t idesc, bool last, uint64_t desc_a, uint64_t desc_b,
                                          uint32_t a_part, uint32_t b_part, uint32_t k_step) {
    if (!warp_wait(&b.full[st.stage.i], st.stage.use, b, p)) return false;
    constexpr int HI = Sums::HI;
    constexpr uint32_t LO_BUFS = Sums::LEVELS == 1 ? 2 : 1;
    const uint32_t lb = st.lc % LO_BUFS;
    if (st.lo_used == 0 && !warp_wait(&b.lo_empty[lb], ((st.lc / LO_BUFS) & 1) ^ 1, b, p)) return false;
    tc_fence_after();
    auto da = [&](int part, int k16) { return desc_a + ((part * a_part + k16 * k_step) >> 4); };
    auto db = [&](int part, int k16) { return desc_b + ((part * b_part + k16 * k_step) >> 4); };
    const uint32_t lo = tmem + LO_COL + lb * BUF_COLS;
    const bool lo_ends = st.lo_used + 1 == Sums::LO || last;
    if (elect_one()) {
        constexpr int PA[5] = {0, 1, 1, 0, 2}, PB[5] = {1, 0, 1, 2, 0};
#pragma unroll
        for (int t = 0; t < 5; ++t) {
            tc_mma<KIND_BF16>(lo, da(PA[t], 0), db(PB[t], 0), idesc, st.lo_used || t ? 1u : 0u);
            tc_mma<KIND_BF16>(lo, da(PA[t], 1), db(PB[t], 1), idesc, 1u);
        }
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < HI; ++h, ++st.hc) {
        if (!warp_wait(&b.hi_empty[st.hc & 1], ((st.hc >> 1) & 1) ^ 1, b, p)) return false;
        tc_fence_after();
        if (elect_one()) {
            const uint32_t hi = tmem + (st.hc & 1) * BUF_COLS;
            tc_mma<KIND_BF16>(hi, da(0, h), db(0, h), idesc, 0u);
            if (HI == 1) tc_mma<KIND_BF16>(hi, da(0, 1), db(0, 1), idesc, 1u);
            tc_commit(&b.hi_full[st.hc & 1]);
            if (h + 1 == HI) {
                tc_commit(&b.empty[st.stage.i]);
                if (lo_ends) tc_commit(&b.lo_full[lb]);
            }
        }
        __syncwarp();
    }
    st.lo_used = lo_ends ? 0 : st.lo_used + 1;
    st.lc += lo_ends;
    st.stage.next(p.stages);
    return true;
}

// An epilogue warp's sums of one tile over nk stages.  t_row: TMEM address of its lanes and first column.
struct EpiState { uint32_t hc = 0, lc = 0; };
template <class Sums>
__device__ __forceinline__ bool sum_tile(EpiState& st, Shared& b, const SplitParams& p, uint32_t t_row, int chunks, int nk, int lane, float (&acc)[2][32]) {
    constexpr uint32_t LO_BUFS = Sums::LEVELS == 1 ? 2 : 1;
    auto take = [&](uint64_t* full, uint64_t* empty, uint32_t& c, uint32_t bufs, uint32_t col) {
        const uint32_t i = c % bufs;
        if (!warp_wait(&full[i], (c / bufs) & 1, b, p)) return false;
        tc_fence_after();
        add_accumulator(t_row + col + i * BUF_COLS, chunks, acc);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[i]);
        ++c;
        return true;
    };
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < 32; ++q) acc[k][q] = 0.0f;
    bool second = false;                                    // the second sum holds something
    for (int ks = 1;; ++ks) {
#pragma unroll
        for (int h = 0; h < Sums::HI; ++h)
            if (!take(b.hi_full, b.hi_empty, st.hc, 2, 0)) return false;
        if ((ks % Sums::LO == 0 || ks >= nk) && !take(b.lo_full, b.lo_empty, st.lc, LO_BUFS, LO_COL)) return false;
        if (ks >= nk) break;
        if (Sums::LEVELS == 2 && ks % Sums::LO == 0) {
            carry_over(t_row + SUM_COL, chunks, !second, acc);
            second = true;
        }
    }
    if (Sums::LEVELS == 2 && second) add_accumulator(t_row + SUM_COL, chunks, acc);
    return true;
}

// The loads of a K-major kernel, by one thread: the raw tiles of A run raw_slots - 1 stages ahead of the planes of B.
__device__ __forceinline__ void load_kk(const SplitParams& p, Shared& bars, const CUtensorMap& map_a, const CUtensorMap& map_b, uint8_t* smem, uint8_t* raws,
                                        uint32_t stage_bytes, uint32_t b_offset, uint32_t b_part, int parts, int nk, int64_t tiles) {
    RawRing raw;
    Ring stage;
    int64_t a_tile = blockIdx.x;
    int a_ks = 0;
    auto load_a = [&]() {
        if (a_tile >= tiles) return true;
        if (!raw_free(raw, bars, p)) return false;
        mbar_expect_tx(&bars.raw_full[raw.bar()], RAW_BYTES);
        if (!(p.drop_load && raw.unit == 0))
            tma_load_2d(raws + (size_t)raw.slot * RAW_BYTES, &map_a, a_ks * BK, (int32_t)((uint32_t)a_tile / (uint32_t)p.n_tiles) * BM, &bars.raw_full[raw.bar()]);
        raw.next(p.raw_slots);
        if (++a_ks == nk) { a_ks = 0; a_tile += gridDim.x; }
        return true;
    };
    bool ok = true;
    for (int i = 0; i + 1 < p.raw_slots && ok; ++i) ok = load_a();
    for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int n0 = (int)((uint32_t)tile % (uint32_t)p.n_tiles) * p.bn;
        for (int ks = 0; ks < nk && ok; ++ks) {
            if (!thread_wait(&bars.empty[stage.i], stage.use ^ 1, bars, p)) return;
            uint8_t* sb = smem + (size_t)stage.i * stage_bytes + b_offset;
            mbar_expect_tx(&bars.full[stage.i], parts * b_part);
            for (int q = 0; q < parts; ++q) tma_load_2d(sb + q * b_part, &map_b, ks * BK, q * p.plane_rows + n0, &bars.full[stage.i]);
            stage.next(p.stages);
            ok = load_a();
        }
    }
}

// 32 rows from row `first`, 32 columns from nb (`here` of them the tile's), through this warp's box.
__device__ __forceinline__ void store_chunk(const SplitParams& p, const CUtensorMap& map_c, int tma_store, uint8_t* box, const float (&v)[32], int64_t first, int nb,
                                            int here, int lane) {
    if (tma_store && lane == 0) bulk_wait_read<0>();   // the store that last used this box has read it
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 8; ++q)
        *reinterpret_cast<float4*>(box + lane * 128 + ((q ^ (lane & 7)) << 4)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    if (tma_store && (nb + 32 <= p.N || (p.N & 3) == 0)) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
            tma_store_2d(&map_c, box, nb, (int32_t)first);
            bulk_commit();
        }
    } else {
        // row by row: TMA stores whole 16-byte units, and what lies behind the matrix's last column is not ours
        __syncwarp();
        if (nb + lane < p.N && lane < here)
            for (int r = 0; r < 32 && first + r < p.M; ++r)
                p.C[(first + r) * p.ldc + nb + lane] = *reinterpret_cast<const float*>(box + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4);
        __syncwarp();
    }
}

// The mask bytes and gate bits that an epilogue thread's row of the CTA's next tile will want, to the L2: their latency stood
// before every tile's sums (982 K x 63 x 91 with odd mask rows: 396 -> 372 us).
__device__ __forceinline__ void prefetch_masks(const SplitParams& p, int64_t tile, int64_t tiles, int row, int c_first, int span) {
    if (tile >= tiles || !(p.epi.drop || p.epi.gate_bits)) return;
    const int64_t m = (int64_t)((uint32_t)tile / (uint32_t)p.n_tiles) * BM + row;
    const int n = (int)((uint32_t)tile % (uint32_t)p.n_tiles) * p.bn + c_first;
    if (m >= p.M || n >= p.N) return;
    if (p.epi.drop) {
        const uint8_t* at = p.epi.drop + (p.epi.row0 + m) * p.N + n;
        const int last = (p.N - n < span ? (int)(p.N - n) : span) - 1;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(at + last));
    }
    if (p.epi.gate_bits) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.epi.gate_bits + (p.epi.row0 + m) * p.epi.ld_gate_bits + (n >> 5)));
}

// ---------------------------------------------------------------- K-major form
__global__ void __launch_bounds__(THREADS, 1) gemm_split_kk_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                                                                   const __grid_constant__ CUtensorMap map_c, const SplitParams p, const int tma_store) {
    chain_begin();
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) Shared bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bn32 = (p.bn + 31) & ~31;
    const uint32_t b_part = (uint32_t)bn32 * BK * 2, stage_bytes = PARTS * (KK_PART + b_part);
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* raws = smem + (size_t)p.stages * stage_bytes;
    uint8_t* boxes = raws + (size_t)p.raw_slots * RAW_BYTES;
    const int nk = (int)((p.K + BK - 1) / BK);
    const int64_t tiles = p.m_tiles * p.n_tiles;
    const uint32_t tmem = cta_begin(bars, GROUP_WARPS + 1, warp);

    if (warp < EPI_WARPS) {
        // 8 warps x 128 + 8 x 64 + 2 x 96 registers a thread are the 18 x 96 of the launch: the sums and the epilogue fit (191 us
        // for the forward product above with their spills, 178 without)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");
        const int quarter = warp & 3, half = warp >> 2;
        const int span = bn32 > 64 ? 64 : 32;                               // columns of this warp
        const int c_first = half * span;
        const int chunks = p.bn <= c_first ? 0 : (p.bn - c_first > 32 && span == 64) ? 2 : 1;
        const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c_first;
        const bool masks = p.epi.drop != nullptr || p.epi.gate != nullptr || p.epi.gate_bits != nullptr;
        uint8_t* const box = boxes + (size_t)warp * 4096;
        EpiState st;
        for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int64_t m0 = (int64_t)((uint32_t)tile / (uint32_t)p.n_tiles) * BM, m = m0 + quarter * 32 + lane;
            const int n0 = (int)((uint32_t)tile % (uint32_t)p.n_tiles) * p.bn;
            uint32_t dw[2] = {0xFFFFFFFFu, 0xFFFFFFFFu}, gw[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};
            if (masks && chunks) mask_words(p.epi, m0 + quarter * 32, p.M, p.N, n0 + c_first, 32, n0 + (p.bn < c_first + span ? p.bn : c_first + span), lane, dw, gw);
            prefetch_masks(p, tile + gridDim.x, tiles, quarter * 32 + lane, c_first, span);
            float acc[2][32];
            if (!sum_tile<KkSums>(st, bars, p, t_row, chunks, nk, lane, acc)) break;
            if (!all_finite(acc, p.bn - c_first)) *p.overflow = 1;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (k >= chunks) break;
                const int c0 = c_first + k * 32, nb = n0 + c0;
                if (nb >= p.N) break;
                chunk_epilogue(p.epi, acc[k], nb, p.N, nullptr, dw[k], gw[k]);
                if (p.epi.sign_bits && m < p.M) p.epi.sign_bits[(p.epi.row0 + m) * p.epi.ld_sign_bits + (nb >> 5)] = sign_word(acc[k], nb, p.N);
                store_chunk(p, map_c, tma_store, box, acc[k], m0 + quarter * 32, nb, p.bn - c0, lane);
            }
        }
        if (tma_store && lane == 0) bulk_wait_all();
    } else if (warp < TMA_WARP) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        // Conversion: thread t of a group takes the float4 t + 128 it of the tile's 128 x 8, row it * 16 + t / 8; the swizzle
        // (bits 4-5 of the offset by bits 7-8) is the same for all of them.
        const int t = (threadIdx.x - EPI_WARPS * 32) % GROUP_THREADS, group = (warp - EPI_WARPS) / GROUP_WARPS;
        const uint32_t at = (uint32_t)((t >> 3) * 64 + ((((t & 7) >> 1) ^ ((t >> 4) & 3)) << 4) + (t & 1) * 8);
        const int64_t stages = blockIdx.x < tiles ? (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x * nk : 0;
        RawRing raw;
        Ring stage;
        raw.next(p.raw_slots, group);
        stage.next(p.stages, group);
        for (int64_t st = group; st < stages; st += GROUPS) {
            if (!warp_wait(&bars.raw_full[raw.bar()], raw.use(), bars, p)) break;
            float4 v[RAW_ITS];
            take_raw(v, raws + (size_t)raw.slot * RAW_BYTES, t);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.raw_empty[raw.bar()]);
            if (!warp_wait(&bars.empty[stage.i], stage.use ^ 1, bars, p)) break;
            uint8_t* dst = smem + (size_t)stage.i * stage_bytes + at;
#pragma unroll
            for (int it = 0; it < RAW_ITS; ++it) split4<KkSums::TRIM_A>(v[it], dst + it * 16 * 64, KK_PART);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.full[stage.i]);
            raw.next(p.raw_slots, GROUPS);
            stage.next(p.stages, GROUPS);
        }
    } else if (warp == TMA_WARP) {
        if (lane == 0) load_kk(p, bars, map_a, map_b, smem, raws, stage_bytes, PARTS * KK_PART, b_part, PARTS, nk, tiles);
    } else {
        const uint32_t idesc = make_idesc<KIND_BF16>(BM, p.bn, false);
        MmaState st;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x)
            for (int ks = 0; ks < nk && ok; ++ks) {
                const uint32_t sa = smem_u32(smem + (size_t)st.stage.i * stage_bytes), sb = sa + PARTS * KK_PART;
                ok = mma_stage<KkSums>(st, bars, p, tmem, idesc, ks + 1 == nk, make_desc(sa, 16, 512, 4), make_desc(sb, 16, 512, 4), KK_PART, b_part, 32);
            }
    }
    cta_end(bars, warp, tmem);
}

// ---------------------------------------------------------------- MN-major form (weight gradient)
__global__ void __launch_bounds__(THREADS, 1) gemm_split_mm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                                                                   const SplitParams p) {
    pdl_wait();               // (see chain_begin)
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) Shared bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bw = p.bn > 64 ? 128 : 64;                                    // columns of B that are converted
    const uint32_t b_part = (uint32_t)(bw / 64) * CHUNK, stage_bytes = PARTS * (MM_PART + b_part);
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* raws = smem + (size_t)p.stages * stage_bytes;
    const int64_t tile = blockIdx.x, m0 = (tile / p.n_tiles) * BM, n0 = (tile % p.n_tiles) * p.bn;
    const int64_t kb = (int64_t)blockIdx.z * p.k_per_split, ke = kb + p.k_per_split < p.K ? kb + p.k_per_split : p.K;
    const int nk = (int)((ke - kb + BK - 1) / BK);
    const uint32_t tmem = cta_begin(bars, GROUP_WARPS, warp);

    if (warp < EPI_WARPS) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 128;");       // as in the K-major form
        const int quarter = warp & 3, half = warp >> 2;
        const int span = p.bn > 64 ? 64 : 32, c_first = half * span;
        const int chunks = p.bn <= c_first ? 0 : (p.bn - c_first > 32 && span == 64) ? 2 : 1;
        EpiState st;
        float acc[2][32];
        const bool ok = sum_tile<MmSums>(st, bars, p, tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c_first, chunks, nk, lane, acc);
        if (ok && !all_finite(acc, p.bn - c_first)) *p.overflow = 1;
        const int64_t m = m0 + quarter * 32 + lane;
        if (ok && m < p.M) {
            float* row = p.C + (p.raw ? (int64_t)blockIdx.z * p.M * p.N : 0) + m * p.ldc;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (k >= chunks) break;
                const int c0 = c_first + k * 32;
                const int64_t nb = n0 + c0;
                float* dst = row + nb;
                if (p.vec_c && nb + 31 < p.N && c0 + 31 < p.bn) {
#pragma unroll
                    for (int q = 0; q < 32; q += 4)
                        *reinterpret_cast<float4*>(dst + q) = make_float4(acc[k][q], acc[k][q + 1], acc[k][q + 2], acc[k][q + 3]);
                } else {
#pragma unroll
                    for (int q = 0; q < 32; ++q)
                        if (nb + q < p.N && c0 + q < p.bn) dst[q] = acc[k][q];
                }
            }
        }
    } else if (warp < TMA_WARP) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        // Conversion: thread t of a group takes the float4 t + 128 it.  Of a tile of 128 columns that is k-row it * 4 + t / 32, of
        // one of 64 k-row it * 8 + t / 16; the swizzle goes by k-row mod 8.
        const int t = (threadIdx.x - EPI_WARPS * 32) % GROUP_THREADS, group = (warp - EPI_WARPS) / GROUP_WARPS;
        auto place = [](int row, int c4) { return (uint32_t)((c4 >> 4) * CHUNK + row * 128 + ((((c4 & 15) >> 1) ^ (row & 7)) << 4) + (c4 & 1) * 8); };
        const uint32_t at_a = place(t >> 5, t & 31), at_b = place(t >> 4, t & 15);
        RawRing raw;
        Ring stage;
        raw.next(p.raw_slots, 2 * group);
        stage.next(p.stages, group);
        float4 v[RAW_ITS];
        // Column sums of B: the rows of tiles take the stages of a group in turn, each thread its own columns of the raw tile.
        const int m_tile = (int)(tile / p.n_tiles);
        int turn = (int)p.m_tiles - m_tile;                            // 0 after m_tile stages
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        auto add_columns = [&](const auto& w, int its) {
#pragma unroll
            for (int it = 0; it < its; ++it) { add2(sum.x, sum.y, w[it].x, w[it].y); add2(sum.z, sum.w, w[it].z, w[it].w); }
        };
        for (int ks = group; ks < nk; ks += GROUPS) {
            if (!warp_wait(&bars.raw_full[raw.bar()], raw.use(), bars, p)) break;
            take_raw(v, raws + (size_t)raw.slot * RAW_BYTES, t);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.raw_empty[raw.bar()]);
            raw.next(p.raw_slots);
            if (!warp_wait(&bars.empty[stage.i], stage.use ^ 1, bars, p)) break;
            uint8_t* dst = smem + (size_t)stage.i * stage_bytes;
#pragma unroll
            for (int it = 0; it < RAW_ITS; ++it) split4<MmSums::TRIM_A>(v[it], dst + (at_a ^ (it & 1) * 64) + it * 4 * 128, MM_PART);
            if (!warp_wait(&bars.raw_full[raw.bar()], raw.use(), bars, p)) break;
            dst += PARTS * MM_PART;
            if (turn == (int)p.m_tiles) turn = 0;
            const bool sums = p.colsum_part && turn++ == 0;
            if (bw == 128) {
                take_raw(v, raws + (size_t)raw.slot * RAW_BYTES, t);
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.raw_empty[raw.bar()]);
                if (sums) add_columns(v, RAW_ITS);
#pragma unroll
                for (int it = 0; it < RAW_ITS; ++it) split4<0>(v[it], dst + (at_a ^ (it & 1) * 64) + it * 4 * 128, b_part);
            } else {
                float4 w[RAW_ITS / 2];
                take_raw(w, raws + (size_t)raw.slot * RAW_BYTES, t);
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars.raw_empty[raw.bar()]);
                if (sums) add_columns(w, RAW_ITS / 2);
#pragma unroll
                for (int it = 0; it < RAW_ITS / 2; ++it) split4<0>(w[it], dst + at_b + it * 8 * 128, b_part);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.full[stage.i]);
            raw.next(p.raw_slots);
            raw.next(p.raw_slots, 2 * (GROUPS - 1));
            stage.next(p.stages, GROUPS);
        }
        if (p.colsum_part) {
            // all raw tiles are used up (by both groups): their memory takes the threads' sums
            const int all = threadIdx.x - EPI_WARPS * 32;
            float* sums = reinterpret_cast<float*>(raws);
            asm volatile("bar.sync 1, %0;" ::"n"(CONV_WARPS * 32) : "memory");
            reinterpret_cast<float4*>(sums)[all] = sum;
            asm volatile("bar.sync 1, %0;" ::"n"(CONV_WARPS * 32) : "memory");
            if (all < p.bn && n0 + all < p.N) {
                double s = 0.0;
                for (int i = all; i < CONV_WARPS * 32 * 4; i += bw) s += (double)sums[i];
                p.colsum_part[((int64_t)blockIdx.z * p.m_tiles + m_tile) * p.N + n0 + all] = s;
            }
        }
    } else if (warp == TMA_WARP) {
        if (lane == 0) {
            RawRing raw;
            for (int u = 0; u < 2 * nk; ++u, raw.next(p.raw_slots)) {         // A, B, A, B, ...
                if (!raw_free(raw, bars, p)) break;
                const int32_t k = (int32_t)(kb + (int64_t)(u >> 1) * BK);
                mbar_expect_tx(&bars.raw_full[raw.bar()], u & 1 ? (uint32_t)bw * BK * 4 : (uint32_t)RAW_BYTES);
                if (p.drop_load && u == 0) continue;
                tma_load_2d(raws + (size_t)raw.slot * RAW_BYTES, u & 1 ? &map_b : &map_a, (int32_t)(u & 1 ? n0 : m0), k, &bars.raw_full[raw.bar()]);
            }
        }
    } else {
        const uint32_t idesc = make_idesc<KIND_BF16>(BM, p.bn, true);
        MmaState st;
        for (int ks = 0; ks < nk; ++ks) {
            const uint32_t sa = smem_u32(smem + (size_t)st.stage.i * stage_bytes), sb = sa + PARTS * MM_PART;
            if (!mma_stage<MmSums>(st, bars, p, tmem, idesc, ks + 1 == nk, make_desc(sa, CHUNK, 1024, 2), make_desc(sb, CHUNK, 1024, 2), MM_PART, b_part, 2048)) break;
        }
    }
    cta_end(bars, warp, tmem);
}

// ---------------------------------------------------------------- bf16 product of fp32 rows
// The K-major form with one part: a bf16 product whose fp32 operand comes without a bf16 copy (the features of an inference, mostly).
// Converted on the way in, it is read once; a pass that wrote the copy first read and wrote it besides.  All K terms go to one
// accumulator in the order of the bf16 kernel, so the bits are that kernel's on the copy.  700 K x 130 x 301: 377 us with the
// pass, 242 so.  Bound: the hand-overs between the roles, as above: DRAM 5.0 TB/s of the 6.5 a copy reaches, tensor pipe 13 % busy,
// issue slots 25 %; the epilogue spills 64 bytes a thread (96 registers: it has no register split).
__global__ void __launch_bounds__(THREADS, 1) gemm_cvt_kk_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                                                                 const __grid_constant__ CUtensorMap map_c, const SplitParams p, const int tma_store) {
    chain_begin();
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) Shared bars;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t stage_bytes = KK_PART + (uint32_t)((p.bn + 31) & ~31) * BK * 2;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* raws = smem + (size_t)p.stages * stage_bytes;
    uint8_t* boxes = raws + (size_t)p.raw_slots * RAW_BYTES;
    const int nk = (int)((p.K + BK - 1) / BK);
    const int64_t tiles = p.m_tiles;                                        // one column of tiles
    const uint32_t tmem = cta_begin(bars, GROUP_WARPS + 1, warp);

    if (warp < EPI_WARPS) {
        const int quarter = warp & 3, half = warp >> 2;                     // 32-column chunks half, half + 2, ...
        const bool masks = p.epi.drop != nullptr || p.epi.gate != nullptr || p.epi.gate_bits != nullptr;
        uint8_t* const box = boxes + (size_t)warp * 4096;
        uint32_t c = 0;
        for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++c) {
            const int64_t m0 = tile * BM + quarter * 32, m = m0 + lane;
            uint32_t dw[4], gw[4];
            if (masks) mask_words(p.epi, m0, p.M, p.N, half * 32, 64, p.bn, lane, dw, gw);
            if (!warp_wait(&bars.hi_full[c & 1], (c >> 1) & 1, bars, p)) break;
            tc_fence_after();
#pragma unroll
            for (int ci = 0; ci < 4; ++ci) {
                const int nb = half * 32 + ci * 64;
                if (nb >= p.N) break;
                uint32_t r[32];
                tc_ld32(tmem + (c & 1) * CVT_COLS + ((uint32_t)(quarter * 32) << 16) + (uint32_t)nb, r);
                tc_wait_ld();
                float v[32];
#pragma unroll
                for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
                chunk_epilogue(p.epi, v, nb, p.N, nullptr, masks ? dw[ci] : 0xFFFFFFFFu, masks ? gw[ci] : 0xFFFFFFFFu);
                if (p.epi.sign_bits && m < p.M) p.epi.sign_bits[(p.epi.row0 + m) * p.epi.ld_sign_bits + (nb >> 5)] = sign_word(v, nb, p.N);
                store_chunk(p, map_c, tma_store, box, v, m0, nb, p.bn - nb, lane);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.hi_empty[c & 1]);
        }
        if (tma_store && lane == 0) bulk_wait_all();
    } else if (warp < TMA_WARP) {
        const int t = (threadIdx.x - EPI_WARPS * 32) % GROUP_THREADS, group = (warp - EPI_WARPS) / GROUP_WARPS;
        const uint32_t at = (uint32_t)((t >> 3) * 64 + ((((t & 7) >> 1) ^ ((t >> 4) & 3)) << 4) + (t & 1) * 8);     // as in the K-major form
        const int64_t stages = blockIdx.x < tiles ? (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x * nk : 0;
        RawRing raw;
        Ring stage;
        raw.next(p.raw_slots, group);
        stage.next(p.stages, group);
        for (int64_t st = group; st < stages; st += GROUPS) {
            if (!warp_wait(&bars.raw_full[raw.bar()], raw.use(), bars, p)) break;
            float4 v[RAW_ITS];
            take_raw(v, raws + (size_t)raw.slot * RAW_BYTES, t);
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.raw_empty[raw.bar()]);
            if (!warp_wait(&bars.empty[stage.i], stage.use ^ 1, bars, p)) break;
            uint8_t* dst = smem + (size_t)stage.i * stage_bytes + at;
#pragma unroll
            for (int it = 0; it < RAW_ITS; ++it)
                *reinterpret_cast<uint2*>(dst + it * 16 * 64) = make_uint2(pack_bf16(v[it].x, v[it].y), pack_bf16(v[it].z, v[it].w));
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars.full[stage.i]);
            raw.next(p.raw_slots, GROUPS);
            stage.next(p.stages, GROUPS);
        }
    } else if (warp == TMA_WARP) {
        if (lane == 0) load_kk(p, bars, map_a, map_b, smem, raws, stage_bytes, KK_PART, stage_bytes - KK_PART, 1, nk, tiles);
    } else {
        const uint32_t idesc = make_idesc<KIND_BF16>(BM, p.bn, false);
        Ring stage;
        uint32_t c = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++c) {
            if (!warp_wait(&bars.hi_empty[c & 1], ((c >> 1) & 1) ^ 1, bars, p)) break;
            for (int ks = 0; ks < nk; ++ks, stage.next(p.stages)) {
                if (!warp_wait(&bars.full[stage.i], stage.use, bars, p)) { ok = false; break; }
                tc_fence_after();
                const uint32_t sa = smem_u32(smem + (size_t)stage.i * stage_bytes);
                const uint64_t da = make_desc(sa, 16, 512, 4), db = make_desc(sa + KK_PART, 16, 512, 4);
                if (elect_one()) {
                    tc_mma<KIND_BF16>(tmem + (c & 1) * CVT_COLS, da, db, idesc, ks ? 1u : 0u);
                    tc_mma<KIND_BF16>(tmem + (c & 1) * CVT_COLS, da + 2, db + 2, idesc, 1u);
                    tc_commit(&bars.empty[stage.i]);
                    if (ks + 1 == nk) tc_commit(&bars.hi_full[c & 1]);
                }
                __syncwarp();
            }
        }
    }
    cta_end(bars, warp, tmem);
}

// Packed planes of the weight matrix: plane q of dst (rows x kpad bf16) holds part q of trans ? src[k][n] : src[n][k], zeros
// outside N x K.
__global__ void pack_split_kernel(const float* __restrict__ src, int64_t ld, int trans, int N, int K, int rows, int kpad, int parts,
                                  uint16_t* __restrict__ dst) {
    chain_begin();
    const int64_t plane = (int64_t)rows * kpad, i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= plane) return;
    const int n = trans ? (int)(i % rows) : (int)(i / kpad), k = trans ? (int)(i / rows) : (int)(i % kpad);     // consecutive threads read consecutive words
    float v = 0.0f;
    if (n < N && k < K) v = trans ? __ldg(src + (int64_t)k * ld + n) : __ldg(src + (int64_t)n * ld + k);
#pragma unroll
    for (int q = 0; q < PARTS; ++q) {
        if (q >= parts) break;
        const uint32_t b = pack_bf16(v, 0.0f) & 0xFFFFu;
        dst[q * plane + (int64_t)n * kpad + k] = (uint16_t)b;
        v -= __uint_as_float(b << 16);
    }
}

}  // namespace

namespace mixgcn {

// Whether a product is faster here than on the FMA pipes, by what both take (us, from measurements; both sides in brackets, here
// first, calls back to back):
//  * here 12 for packing, launches and the tail, and 0.75 per stage and 1.2 per tile of the longest CTA: a wave that is nearly
//    empty counts in full.  20 K x 32 x 500 is two waves of sixteen stages (40 : 35, left there, and 5 K x 128 x 256, 24 : 27);
//    20 K x 64 x 500, as long here, 42 : 74; 52 K x 80 x 80 27 : 41; 876 K x 8 x 210 277 : 361; 876 K x 210 x 8 339 : 556;
//  * there 20 TFLOP/s and more, with columns padded to 32, and 2 TB/s;
//  * weight gradients here 16 and 0.85 per stage.  A stage takes 1.0, but the FMA kernel's narrow tiles do not reach 20 TFLOP/s
//    either, so the line lies about right: 64 x 16 x 200 K 58 : 40, 128 x 128 x 5 K 29 : 21, 128 x 128 x 10 K 30 : 28 and
//    64 x 64 x 20 K 25 : 27 are left there, 40 x 40 x 200 K 60 : 89, 80 x 80 x 52 K 33 : 47 and 64 x 47 x 400 K 102 : 162 taken
//    (33 x 63 x 200 K, 63 : 89, is not).
// Below 4 columns (and, untried, 32 rows of a weight gradient) padding takes it all.  The K-major form adds up one fp32 chain of
// K / 32 sums, which past 1024 terms of one sign is less accurate than the two levels of the FMA kernel (1.2e-7 : 5e-8 at 2048).
// (Which kernel a product takes depends on its rows: the same row may be rounded differently in a compacted, a chunked and a whole
// product.)
static bool split_pays(const mixgcn_ctx* ctx, int ta, int64_t M, int64_t N, int64_t K) {
    if (N < 4 || (ta ? M < 32 : K > 1024)) return false;
    auto ceil_div = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    const int64_t tiles = ceil_div(M, BM) * ceil_div(N, BN_MAX), nk = ceil_div(K, BK), sms = ctx->sm_count;
    const double ops_us = 2.0 * M * (ceil_div(N, 32) * 32) * K / 20e6, bytes_us = 4.0 * (M * K + K * N + M * N) / 2e6;
    const double fma_us = 2.0 + (ops_us > bytes_us ? ops_us : bytes_us);
    if (!ta) return 12.0 + ceil_div(tiles, sms) * (1.2 + 0.75 * nk) < fma_us;
    const int64_t least = nk < 8 ? nk : 8, stages = ceil_div(nk * tiles, sms);
    return 16.0 + 0.85 * (stages > least ? stages : least) < fma_us;
}

// slots of raw tiles that fit beside `fixed` bytes (one block per SM: 227 KB, less the barriers)
static int raw_slots(size_t fixed, int slot) {
    const int n = (int)((227 * 1024 - 512 - fixed) / (size_t)slot);
    return n < RAW_MAX ? n : RAW_MAX;
}

// fp32 products that pay on the tensor cores; MIXGCN_EUNSUPPORTED (nothing launched) for the others, which the FMA kernel takes.
// *overflow_flag: the device word that the FMA kernel launched behind has to look at.
mixgcn_status launch_gemm_split(mixgcn_ctx* ctx, int ta, int tb, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda,
                                const float* B, int64_t ldb, float* C, int64_t ldc, const mixgcn_epilogue* epi, int64_t epi_row0,
                                cudaStream_t s, bool* bits_done, const int32_t** overflow_flag, float* colsum_b, bool* colsum_done) {
    if (bits_done) *bits_done = false;
    if (colsum_done) *colsum_done = false;
    if (M <= 0 || N <= 0 || K <= 0 || (ta && tb) || M >= (1ll << 31) || N >= (1ll << 31) || K >= (1ll << 31)) return MIXGCN_EUNSUPPORTED;
    if (!aligned16(A) || (lda & 3) || (ta && (!aligned16(B) || (ldb & 3) || epi))) return MIXGCN_EUNSUPPORTED;
    if (!split_pays(ctx, ta, M, N, K)) return MIXGCN_EUNSUPPORTED;
    auto ceil_div = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    SplitParams p{};
    p.M = M; p.N = N; p.K = K; p.C = C; p.ldc = ldc;
    p.vec_c = aligned16(C) && (ldc & 3) == 0;
    p.n_tiles = ceil_div(N, BN_MAX);
    p.bn = (int)(p.n_tiles == 1 ? ceil_div(N, 16) * 16 : ceil_div(ceil_div(N, p.n_tiles), 32) * 32);
    p.n_tiles = ceil_div(N, p.bn);
    p.stages = p.bn > 64 ? 3 : 4;                      // as many as leave three raw slots and more
    p.m_tiles = ceil_div(M, BM);
    const int64_t tiles = p.m_tiles * p.n_tiles;
    if (tiles > 0x7FFFFFFFll) return MIXGCN_EUNSUPPORTED;
    p.epi = make_tc_epi(epi, epi_row0);
    p.status = ctx->d_status;
    p.wait_limit = ctx->debug_wait_limit > 0 ? (uint32_t)ctx->debug_wait_limit : WAIT_LIMIT_DEFAULT;
    p.drop_load = ctx->debug_drop_load;
    p.overflow = ctx->d_status + SPLIT_OVERFLOW_WORD;
    *overflow_flag = p.overflow;
    if (!ta) {
        const int bn32 = (p.bn + 31) & ~31, kpad = (int)(ceil_div(K, BK) * BK);
        const int rows = (int)p.n_tiles * bn32;
        p.plane_rows = rows;
        MIXGCN_TRY(ensure_workspace(ctx, (int64_t)PARTS * rows * kpad * 2));
        uint16_t* planes = reinterpret_cast<uint16_t*>(ctx->workspace);
        CUtensorMap map_a, map_b, map_c;
        if (!encode_2d(&map_a, A, 4, K, M, lda, BK, BM, CU_TENSOR_MAP_SWIZZLE_NONE)) return MIXGCN_EUNSUPPORTED;
        if (!encode_2d(&map_b, planes, 2, kpad, (int64_t)PARTS * rows, kpad, BK, bn32, CU_TENSOR_MAP_SWIZZLE_64B)) return MIXGCN_EUNSUPPORTED;
        map_c = map_a;
        const int tma_store = p.vec_c;
        if (tma_store && !encode_2d(&map_c, C, 4, N, M, ldc, 32, 32)) return MIXGCN_EUNSUPPORTED;
        const size_t fixed = (size_t)p.stages * PARTS * (KK_PART + bn32 * BK * 2) + (size_t)EPI_WARPS * 4096 + 1024;
        p.raw_slots = raw_slots(fixed, RAW_BYTES);
        const size_t smem = fixed + (size_t)p.raw_slots * RAW_BYTES;
        MIXGCN_CUDA(cudaFuncSetAttribute(gemm_split_kk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        MIXGCN_TRY(launch_clear(ctx, PH_GEMM, p.overflow, 1, nullptr, s));
        {
            LaunchScope scope(ctx, PH_GEMM, s);
            launch_chained(pack_split_kernel, dim3((unsigned)ceil_div((int64_t)rows * kpad, 256)), 256, 0, s, B, ldb, tb ? 0 : 1, (int)N, (int)K, rows, kpad, PARTS, planes);
        }
        LaunchScope scope(ctx, PH_GEMM, s);
        const unsigned grid = (unsigned)(tiles < ctx->sm_count ? tiles : ctx->sm_count);
        launch_chained(gemm_split_kk_kernel, dim3(grid), THREADS, smem, s, map_a, map_b, map_c, p, tma_store);
        MIXGCN_CUDA(cudaGetLastError());
        if (bits_done) *bits_done = p.epi.sign_bits != nullptr;
        return MIXGCN_OK;
    }
    // one CTA per SM: as many splits as fill the machine once, no shorter than eight stages
    // and none longer than 8,192 terms: the sums in registers are one fp32 chain
    int64_t splits = ctx->sm_count / tiles;
    if (splits < ceil_div(K, 8192)) splits = ceil_div(ceil_div(K, 8192) * tiles, ctx->sm_count) * ctx->sm_count / tiles;
    const int64_t most = ceil_div(K, 8 * BK);
    if (splits > most) splits = most;
    if (splits < 1) splits = 1;
    p.k_per_split = ceil_div(ceil_div(K, splits), BK) * BK;
    splits = ceil_div(K, p.k_per_split);
    p.raw = splits > 1;
    const int64_t part_bytes = splits > 1 ? (splits * M * N * (int64_t)sizeof(float) + 7) / 8 * 8 : 0;
    const int64_t sums_bytes = colsum_b ? splits * p.m_tiles * N * (int64_t)sizeof(double) : 0;
    if (part_bytes + sums_bytes) MIXGCN_TRY(ensure_workspace(ctx, part_bytes + sums_bytes));
    if (colsum_b) p.colsum_part = reinterpret_cast<double*>(reinterpret_cast<char*>(ctx->workspace) + part_bytes);
    if (splits > 1) {
        p.C = reinterpret_cast<float*>(ctx->workspace); p.ldc = N; p.vec_c = (N & 3) == 0;
    }
    const int bw = p.bn > 64 ? 128 : 64;
    CUtensorMap map_a, map_b;
    if (!encode_2d(&map_a, A, 4, M, K, lda, BM, BK, CU_TENSOR_MAP_SWIZZLE_NONE)) return MIXGCN_EUNSUPPORTED;
    if (!encode_2d(&map_b, B, 4, N, K, ldb, bw, BK, CU_TENSOR_MAP_SWIZZLE_NONE)) return MIXGCN_EUNSUPPORTED;
    const size_t fixed = (size_t)p.stages * PARTS * (BM + bw) / 64 * CHUNK + 1024;
    p.raw_slots = raw_slots(fixed, RAW_BYTES);
    const size_t smem = fixed + (size_t)p.raw_slots * RAW_BYTES;
    MIXGCN_CUDA(cudaFuncSetAttribute(gemm_split_mm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    MIXGCN_TRY(launch_clear(ctx, PH_GEMM, p.overflow, 1, nullptr, s));
    {
        LaunchScope scope(ctx, PH_GEMM, s);
        launch_chained(gemm_split_mm_kernel, dim3((unsigned)tiles, 1, (unsigned)splits), THREADS, smem, s, map_a, map_b, p);
    }
    MIXGCN_CUDA(cudaGetLastError());
    const ColSums sums = colsum_b ? ColSums{p.colsum_part, (int)(splits * p.m_tiles), colsum_b} : ColSums{};
    if (splits > 1) MIXGCN_TRY(launch_splitk_reduce(ctx, M, N, (int)splits, p.C, C, ldc, nullptr, s, sums));
    else if (colsum_b) MIXGCN_TRY(launch_colsum_splits(ctx, N, sums.splits, sums.part, sums.out, s));
    if (colsum_b && colsum_done) *colsum_done = true;
    return MIXGCN_OK;
}

// C = bf16(A) bf16(op(B)) for fp32 rows A without a bf16 copy, K-major, N up to 256 (one column of tiles: wider results read and
// convert A again for each); MIXGCN_EUNSUPPORTED (nothing launched) otherwise.
mixgcn_status launch_gemm_cvt(mixgcn_ctx* ctx, int tb, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B, int64_t ldb, float* C,
                              int64_t ldc, const mixgcn_epilogue* epi, int64_t epi_row0, cudaStream_t s, bool* bits_done) {
    if (bits_done) *bits_done = false;
    if (M <= 0 || N <= 0 || K <= 0 || N > (int64_t)CVT_COLS || M >= (1ll << 31) || K >= (1ll << 31) || !aligned16(A) || (lda & 3)) return MIXGCN_EUNSUPPORTED;
    // few tiles with many stages each: the bf16 kernel's longer stages win over the pass (4 K x 256 x 2048: 49 us here, 37 there)
    if (M <= (int64_t)BM * (ctx->sm_count - 1) && K > 512) return MIXGCN_EUNSUPPORTED;
    if (ctx->debug_drop_load == 1) return MIXGCN_EUNSUPPORTED;        // the hook is meant for the bf16 kernel then
    auto ceil_div = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    SplitParams p{};
    p.M = M; p.N = N; p.K = K; p.C = C; p.ldc = ldc;
    p.vec_c = aligned16(C) && (ldc & 3) == 0;
    p.n_tiles = 1; p.bn = (int)(ceil_div(N, 16) * 16); p.m_tiles = ceil_div(M, BM); p.stages = STAGES_MAX;
    p.epi = make_tc_epi(epi, epi_row0);
    p.status = ctx->d_status;
    p.wait_limit = ctx->debug_wait_limit > 0 ? (uint32_t)ctx->debug_wait_limit : WAIT_LIMIT_DEFAULT;
    p.drop_load = ctx->debug_drop_load;
    const int bn32 = (p.bn + 31) & ~31, kpad = (int)(ceil_div(K, BK) * BK);
    MIXGCN_TRY(ensure_workspace(ctx, (int64_t)bn32 * kpad * 2));
    uint16_t* packed = reinterpret_cast<uint16_t*>(ctx->workspace);
    CUtensorMap map_a, map_b, map_c;
    if (!encode_2d(&map_a, A, 4, K, M, lda, BK, BM, CU_TENSOR_MAP_SWIZZLE_NONE)) return MIXGCN_EUNSUPPORTED;
    if (!encode_2d(&map_b, packed, 2, kpad, bn32, kpad, BK, bn32, CU_TENSOR_MAP_SWIZZLE_64B)) return MIXGCN_EUNSUPPORTED;
    map_c = map_a;
    const int tma_store = p.vec_c;
    if (tma_store && !encode_2d(&map_c, C, 4, N, M, ldc, 32, 32)) return MIXGCN_EUNSUPPORTED;
    const size_t fixed = (size_t)p.stages * (KK_PART + bn32 * BK * 2) + (size_t)EPI_WARPS * 4096 + 1024;
    p.raw_slots = raw_slots(fixed, RAW_BYTES);
    const size_t smem = fixed + (size_t)p.raw_slots * RAW_BYTES;
    MIXGCN_CUDA(cudaFuncSetAttribute(gemm_cvt_kk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    {
        LaunchScope scope(ctx, PH_GEMM, s);
        launch_chained(pack_split_kernel, dim3((unsigned)ceil_div((int64_t)bn32 * kpad, 256)), 256, 0, s, B, ldb, tb ? 0 : 1, (int)N, (int)K, bn32, kpad, 1, packed);
    }
    LaunchScope scope(ctx, PH_GEMM, s);
    const unsigned grid = (unsigned)(p.m_tiles < ctx->sm_count ? p.m_tiles : ctx->sm_count);
    launch_chained(gemm_cvt_kk_kernel, dim3(grid), THREADS, smem, s, map_a, map_b, map_c, p, tma_store);
    MIXGCN_CUDA(cudaGetLastError());
    if (bits_done) *bits_done = p.epi.sign_bits != nullptr;
    return MIXGCN_OK;
}

}  // namespace mixgcn
