// The gather kernels of the aggregation over whole rows and their launches (see spmm.cu).  Compiled twice: with MIXGCN_SPMM_HUB 0 for
// matrices without tiles, with 1 for what the tiles of a graph's dense corner leave (spmm_hub.cu), where every kernel that has a row's sum
// adds the row's tiles to it -- in the same kernels that would cost calls without tiles 1 to 2 % (registers, a test per row).
#pragma once
#include <type_traits>

#include "hub_tiles.cuh"
#include "internal.cuh"

// Launch shapes the measurements settled on (workload with 30M nodes, width 128, and the wide / dense ones).
constexpr int SPMM_MINB = 4;          // CTAs per SM asked of the compiler for the narrow (VPL <= 2) group kernels
constexpr int SPMM_FOLD_WMAX = 128;   // widest aggregation the two folds below apply to
constexpr int SPMM_FOLD_SEG = 2;      // long-row segments at widths <= 128: 16 lanes x 2 float4 per unit (1 would be 32 lanes x 1)
constexpr int SPMM_FOLD_MED = 2;      // the same for rows of 13 entries up to the schedule's segment length (64..512)
constexpr int SPMM_SHORT_RB = 4;      // rows a warp of the short-row kernel takes at once
constexpr int SPMM_SHORT_MINB = 5;    // CTAs per SM asked of the compiler for it
constexpr int SPMM_SHORT_MAXE = 2;    // rows of at most this many entries go to the short-row kernel
constexpr int SPMM_U = 8;             // float4 loads a lane keeps in flight

constexpr bool HUB = MIXGCN_SPMM_HUB != 0;

namespace mixgcn {

struct SpmmParams {
    const SpmmRec* rec;    // schedule records, or null: unit idx is row idx of the CSR
    const int64_t* rowptr;
    const int32_t* col;
    const float* val;
    int64_t idx_begin, idx_end;
    int32_t w;             // columns handled by this launch (slice width)
    int32_t j0;            // first column of the slice (multiple of 4)
    int32_t w_total;       // full width (for the dense drop-mask index)
    const float* Y; int64_t ldy;
    float* Z; int64_t ldz;
    uint16_t* Z_lp; int64_t ldz_lp;   // nullable: bf16 copy of Z (after the epilogue) for a bf16 dense product that follows
    float* partial;        // non-null: unit idx writes its raw sums to partial[idx * ldp + ...]
    int64_t ldp;
    // row-sparse input (spmm_sparse_kernel): rows v of the input with in_mask[v] == 0 are exactly zero
    // and are skipped; a kept row v is read from Y row in_pos[v] (in_pos == null: row v itself)
    const uint8_t* in_mask;
    const int32_t* in_pos;
    uint8_t* out_mask;     // nullable: receives 1 for output rows that received a contribution, else 0
    // row filter (spmm_filtered_kernel): only output rows u with row_filter[u] != 0 are computed and written
    const uint8_t* row_filter;
    const int32_t* seg_perm;   // segment records carry the long row's index i; its row is seg_perm[i] (null: the record's row)
    // sampled aggregation Z = (A_hat Y) (.) M, Eq. 4: bit j of row u of the bitmap says whether output (u, j) is kept
    // The same bitmap serves a bit-packed gate (the bitmap mask buffer of Section 3.2.1 holding a ReLU mask): kept
    // outputs are then scaled by bits_scale and nothing is skipped (bits_skip = 0).
    const uint32_t* out_bits;  // [n x ld_bits] words, null: every output is kept
    int64_t ld_bits;
    float bits_scale;          // factor of the kept outputs (1 for the sampled aggregation, the gate's scale for a gate)
    int bits_skip;             // 1: lanes whose four columns of a row are all masked skip that row's gathers
    // epilogue
    const float* bias; int relu;
    const uint8_t* drop; float keep_scale;
    const float* gate; int64_t ld_gate; float gate_scale;
    const float* residual; int64_t ld_residual; float residual_scale;
    // loss epilogue (kernels instantiated with LOSS): labels, train mask, number of train nodes, per-row loss, arg-max
    const int32_t* loss_labels; const uint8_t* loss_mask; const unsigned long long* loss_count;
    float* loss_row; int32_t* loss_pred; int loss_zero_rows;
    // limits for the index tests of the bounds-checked debug build (unused otherwise)
    int32_t* status;
    int64_t n_cols;        // column ids lie in [0, n_cols) (they index in_mask / in_pos, or Y itself)
    int64_t y_rows;        // rows of Y
    int64_t n_out;         // output rows
    int64_t n_long;        // long rows of the schedule (a segment record's `row` is an ordinal among them)
    int64_t nnz;           // stored entries
    int64_t n_partial;     // partial-row slots
};
// ... and where tiles come on top
struct SpmmHubParams : SpmmParams {
    // tiles of the dense corner (hub_tiles.cu): the rank of every row (-1: in no row of tiles).  A row of rank h has partial rows
    // in the pieces piece_first[h / 256] .. piece_first[h / 256 + 1] - 1, which count row_scale[h] times.
    const int32_t* hub_rank; const int32_t* piece_first; const float* row_scale;
    const float* tile_sums; int64_t n_tile_sums;     // partial rows, ldp floats apart
};

// Narrow aggregations (w_total <= 64 columns): column lanes and float4 per lane, chosen so that few column slots of
// a lane group stay empty.  The choice goes by the call's full width, not the slice's: the lane split decides the order
// in which a unit's entries are added, and results do not depend on the slicing.
struct NarrowCfg { int cl, vpl; };
inline NarrowCfg narrow_cfg(int w_total) {
    const int w4 = (w_total + 3) >> 2;
    if (w4 > 16) return {0, 0};
    if (w4 <= 1) return {1, 1};
    if (w4 <= 2) return {2, 1};
    if (w4 <= 4) return {4, 1};
    if (w4 <= 6) return {2, 3};
    if (w4 <= 8) return {8, 1};
    if (w4 <= 12) return {4, 3};
    return {8, 2};
}
// One slice of an aggregation over the rows of schedule S: segments of the long rows (partial rows at `partial`), the other rows by
// bucket, the combination.  In spmm_hub.cu, for schedules of what tiles leave:
mixgcn_status launch_rows_hub(mixgcn_ctx* ctx, const SpmmHubParams& p, const SpmmSchedule& S, NarrowCfg narrow, bool loss, int phase, float* partial, cudaStream_t s);

}  // namespace mixgcn

namespace {

using namespace mixgcn;

using Params = std::conditional<HUB, SpmmHubParams, SpmmParams>::type;

// entry range and row of a unit: tested in the debug build before anything is addressed with them
__device__ __forceinline__ bool unit_ok(const Params& p, int64_t b, int64_t e, int64_t u) {
    return index_ok(b, p.nnz + 1, p.status, SITE_SPMM_RANGE) && index_ok(e, p.nnz + 1, p.status, SITE_SPMM_RANGE) &&
           index_ok(u, p.partial ? p.n_long : p.n_out, p.status, SITE_SPMM_ROW);   // a segment's record names its long row by ordinal
}

__device__ __forceinline__ float epilogue1(const Params& p, float y, int64_t u, int j) {
    if (p.residual) y = fmaf(p.residual_scale, p.residual[u * p.ld_residual + j], y);
    if (p.bias) y += p.bias[j];
    if (p.relu) y = fmaxf(y, 0.0f);
    if (p.drop) y = p.drop[u * p.w_total + j] ? y * p.keep_scale : 0.0f;
    if (p.gate) y = p.gate[u * p.ld_gate + j] > 0.0f ? y * p.gate_scale : 0.0f;
    return y;
}

// four fp32 -> four bf16 (round to nearest even), 8 bytes
__device__ __forceinline__ void store_lp4(uint16_t* dst, float x, float y, float z, float w) {
    uint32_t lo, hi;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(y), "f"(x));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(w), "f"(z));
    *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
}

__device__ __forceinline__ void store_row(const Params& p, int64_t u, int c4, float4 a) {
    const int j = p.j0 + c4 * 4;           // global column of a.x
    const int jend = p.j0 + p.w;           // one past the last valid column of the slice
    float r[4] = {a.x, a.y, a.z, a.w};
    if (!p.bias && !p.residual && a.x == 0.0f && a.y == 0.0f && a.z == 0.0f && a.w == 0.0f) {
        // ReLU, dropout and the gate all map 0 to 0: no mask or gate byte needs to be read (the empty
        // rows of a row-sparse aggregation take this path)
        if (p.Z) *reinterpret_cast<float4*>(p.Z + u * p.ldz + j) = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.Z_lp) *reinterpret_cast<uint2*>(p.Z_lp + u * p.ldz_lp + j) = make_uint2(0u, 0u);
        return;
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) r[t] = (j + t < jend) ? epilogue1(p, r[t], u, j + t) : 0.0f;
    if (p.out_bits) {
        const uint32_t nib = (__ldg(p.out_bits + u * p.ld_bits + (j >> 5)) >> (j & 31)) & 0xFu;   // j % 4 == 0: one word
#pragma unroll
        for (int t = 0; t < 4; ++t) r[t] = ((nib >> t) & 1u) ? r[t] * p.bits_scale : 0.0f;
    }
    if (p.Z) *reinterpret_cast<float4*>(p.Z + u * p.ldz + j) = make_float4(r[0], r[1], r[2], r[3]);   // null: bf16 copy only
    if (p.Z_lp) store_lp4(p.Z_lp + u * p.ldz_lp + j, r[0], r[1], r[2], r[3]);
}

// What stands between the sums and the stored row -- the general epilogue's code costs the gather loop registers
// under the cap, so the forms the epochs spend their time in have instances without it:
//   EPI_PLAIN  nothing (every forward aggregation of an aggregate-first layer, every partial row of a long-row segment)
//   EPI_BITS   a bit-packed gate only (the backward aggregation that produces a gated input gradient)
//   EPI_BIAS   bias, then ReLU if asked (the forward aggregation of an update-first layer)
//   EPI_GATE   an fp32 gate only, 16-byte aligned with a leading dimension that is a multiple of 4
//   EPI_LOSS   bias + soft-max cross-entropy (loss_epilogue)
//   EPI_ANY    everything store_row knows
enum { EPI_ANY = 0, EPI_LOSS = 1, EPI_PLAIN = 2, EPI_BITS = 3, EPI_BIAS = 4, EPI_GATE = 5 };
constexpr bool epi_is_lean(int epi) { return epi >= EPI_PLAIN; }

// store_row for the lean instances; pad columns of the last group are written as zeros, as store_row does.
template <int EPI>
__device__ __forceinline__ void store_lean(const Params& p, int64_t u, int c4, float4 y) {
    const int j = p.j0 + c4 * 4;
    const int left = p.j0 + p.w - j;             // valid columns of this group (>= 1)
    if constexpr (EPI == EPI_BIAS) {
        float4 b4;
        if (left >= 4) b4 = __ldg(reinterpret_cast<const float4*>(p.bias + j));
        else b4 = make_float4(__ldg(p.bias + j), left > 1 ? __ldg(p.bias + j + 1) : 0.0f, left > 2 ? __ldg(p.bias + j + 2) : 0.0f, 0.0f);
        y.x += b4.x; y.y += b4.y; y.z += b4.z; y.w += b4.w;
        if (p.relu) { y.x = fmaxf(y.x, 0.0f); y.y = fmaxf(y.y, 0.0f); y.z = fmaxf(y.z, 0.0f); y.w = fmaxf(y.w, 0.0f); }
    }
    if constexpr (EPI == EPI_GATE) {
        const float4 g4 = __ldg(reinterpret_cast<const float4*>(p.gate + u * p.ld_gate + j));   // inside the row: ld_gate % 4 == 0
        y.x = g4.x > 0.0f ? y.x * p.gate_scale : 0.0f; y.y = g4.y > 0.0f ? y.y * p.gate_scale : 0.0f;
        y.z = g4.z > 0.0f ? y.z * p.gate_scale : 0.0f; y.w = g4.w > 0.0f ? y.w * p.gate_scale : 0.0f;
    }
    if constexpr (EPI == EPI_BITS) {
        const uint32_t nib = (__ldg(p.out_bits + u * p.ld_bits + (j >> 5)) >> (j & 31)) & 0xFu;   // j % 4 == 0: one word
        y.x = (nib & 1u) ? y.x * p.bits_scale : 0.0f; y.y = (nib & 2u) ? y.y * p.bits_scale : 0.0f;
        y.z = (nib & 4u) ? y.z * p.bits_scale : 0.0f; y.w = (nib & 8u) ? y.w * p.bits_scale : 0.0f;
    }
    if (left < 4) { if (left < 2) y.y = 0.0f; if (left < 3) y.z = 0.0f; y.w = 0.0f; }
    if (p.Z) *reinterpret_cast<float4*>(p.Z + u * p.ldz + j) = y;
    if (p.Z_lp) store_lp4(p.Z_lp + u * p.ldz_lp + j, y.x, y.y, y.z, y.w);
}

// Which lean instance serves this launch (EPI_ANY: none does).
inline int pick_epi(const Params& p) {
    if (!HUB && p.out_bits && p.bits_skip) return EPI_ANY;                 // the sampled aggregation skips gathers: general instance
    if (p.partial) return EPI_PLAIN;                               // a partial row never has an epilogue
    if (p.drop || p.residual) return EPI_ANY;
    const bool bias = p.bias != nullptr || p.relu, gate = p.gate != nullptr, bits = p.out_bits != nullptr;
    if (!bias && !gate && !bits) return EPI_PLAIN;
    if (bits && !bias && !gate) return EPI_BITS;
    if (bias && !gate && !bits && p.bias && (reinterpret_cast<uintptr_t>(p.bias) & 15u) == 0) return EPI_BIAS;
    if (gate && !bias && !bits && (reinterpret_cast<uintptr_t>(p.gate) & 15u) == 0 && (p.ld_gate & 3) == 0) return EPI_GATE;
    return EPI_ANY;
}

__device__ __forceinline__ void fma4(float4& acc, float a, const float4& y) {
    acc.x = fmaf(a, y.x, acc.x); acc.y = fmaf(a, y.y, acc.y);
    acc.z = fmaf(a, y.z, acc.z); acc.w = fmaf(a, y.w, acc.w);
}

// Soft-max cross-entropy of output row u taken from the registers that hold the aggregated row (the whole
// row belongs to one group of LPR lanes, lane `lig` holding float4 groups lig + v * LPR): logits = sums + bias;
// arg-max with lowest-index ties -> pred; on a train row the loss term lse - logit[label] -> loss_row[u] and the
// gradient (softmax - e_label) / #T -> Z row u.  The logits themselves are never written.
template <int LPR, int VPL>
__device__ __forceinline__ void loss_epilogue(const Params& p, int64_t u, int lig, unsigned mask, const float4 (&acc)[VPL]) {
    const int C = p.w;                 // one slice: j0 == 0
    const int w4 = (C + 3) >> 2;
    float x[VPL][4];
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int j = (lig + v * LPR) * 4;
        const float a[4] = {acc[v].x, acc[v].y, acc[v].z, acc[v].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) x[v][e] = j + e < C ? (p.bias ? a[e] + __ldg(p.bias + j + e) : a[e]) : -INFINITY;
    }
    float mx = -INFINITY; int arg = 0x7FFFFFFF;
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = (lig + v * LPR) * 4 + e;
            if (c < C && (x[v][e] > mx || (x[v][e] == mx && c < arg))) { mx = x[v][e]; arg = c; }
        }
    if (arg == 0x7FFFFFFF) arg = lig * 4 < C ? lig * 4 : 0;       // nothing but -inf / NaN in this lane's columns
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) {
        const float omx = __shfl_xor_sync(mask, mx, o, LPR);
        const int oarg = __shfl_xor_sync(mask, arg, o, LPR);
        if (omx > mx || (omx == mx && oarg < arg)) { mx = omx; arg = oarg; }
    }
    if (p.loss_pred && lig == 0) p.loss_pred[u] = arg;
    const unsigned long long T = *p.loss_count;
    const bool train = __ldg(p.loss_mask + u) != 0 && T != 0;
    int y = 0; bool ok = false;
    if (train) {
        y = __ldg(p.loss_labels + u);
        ok = y >= 0 && y < C;
        if (!ok && lig == 0) atomicMax(p.status, DEV_BAD_LABEL);
    }
    if (!train || !ok) {
        if (p.loss_zero_rows || train) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c4 = lig + v * LPR;
                if (c4 < w4) *reinterpret_cast<float4*>(p.Z + u * p.ldz + c4 * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        return;
    }
    float s = 0.0f, py = 0.0f;        // the label's logit lives in lane (y/4) % LPR of the group
#pragma unroll
    for (int v = 0; v < VPL; ++v)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = (lig + v * LPR) * 4 + e;
            if (c == y) py = x[v][e];
            x[v][e] = c < C ? expf(x[v][e] - mx) : 0.0f;
            s += x[v][e];
        }
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(mask, s, o, LPR);
    const float lse = mx + logf(s), share = 1.0f / s;
    py = __shfl_sync(mask, py, (y >> 2) & (LPR - 1), LPR);
    if (lig == 0) p.loss_row[u] = lse - py;
    const float invT = (float)(1.0 / (double)T);
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int c4 = lig + v * LPR;
        if (c4 < w4) {
            float r[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = c4 * 4 + e;
                r[e] = c < C ? (x[v][e] * share - (c == y ? 1.0f : 0.0f)) * invT : 0.0f;
            }
            *reinterpret_cast<float4*>(p.Z + u * p.ldz + c4 * 4) = make_float4(r[0], r[1], r[2], r[3]);
        }
    }
}

// The sums of row u's tiles, times the row's scale, added to those of its other entries: column groups lig, lig + LPR, ... of w4.  The
// pieces are added up in fp64: they are few, and in fp32 their chain would be most of the error of a hub's row.
template <int LPR, int VPL>
__device__ __forceinline__ void add_tiles(const Params& p, int64_t u, int lig, int w4, float4 (&acc)[VPL]) {
#if MIXGCN_SPMM_HUB
    const int32_t h = __ldg(p.hub_rank + u);
    if (h < 0) return;
    const int rb = h / HUB_ROWS, q0 = __ldg(p.piece_first + rb), q1 = __ldg(p.piece_first + rb + 1);
    if (q0 == q1) return;
    const int64_t row = (int64_t)q0 * HUB_ROWS + h % HUB_ROWS;
    if (!index_ok(row, p.n_tile_sums, p.status, SITE_SPMM_SEG) || !index_ok(row + (int64_t)(q1 - q0 - 1) * HUB_ROWS, p.n_tile_sums, p.status, SITE_SPMM_SEG)) return;
    const double scale = __ldg(p.row_scale + h);
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        if (lig + v * LPR >= w4) continue;
        const float4* src = reinterpret_cast<const float4*>(p.tile_sums + row * p.ldp) + lig + v * LPR;
        double x = 0.0, y = 0.0, z = 0.0, w = 0.0;
#pragma unroll 1
        for (int q = q0; q < q1; ++q, src += HUB_ROWS * p.ldp / 4) {
            const float4 t = __ldg(src);
            x += t.x; y += t.y; z += t.z; w += t.w;
        }
        acc[v].x = (float)(acc[v].x + x * scale); acc[v].y = (float)(acc[v].y + y * scale);
        acc[v].z = (float)(acc[v].z + z * scale); acc[v].w = (float)(acc[v].w + w * scale);
    }
#endif
}

template <int LPR, int VPL>
struct Cfg {
    static constexpr int U0 = SPMM_U / VPL < 1 ? 1 : SPMM_U / VPL;
    static constexpr int U = U0 > LPR ? LPR : U0;   // gathered rows in flight per lane group
};

// A batch of entries (zeros past the unit's end) added to a row's sums where tiles took entries out of the rows: what is left is cut
// into fewer and longer chains than whole rows are, so the batch is added up by itself first (300 K nodes of mean degree 31, positive numbers:
// 1.2 -> 0.9 of the error without tiles; 128 columns 292 -> 302 us, 48 columns at 2.4 M nodes 2.48 -> 2.25 ms; a second level of
// sums in shared memory every 64 entries costs the same).
template <int U, int VPL>
__device__ __forceinline__ void add_batch(float4 (&acc)[VPL], const float (&a)[U], float4 (&y)[U][VPL]) {
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        y[0][v].x *= a[0]; y[0][v].y *= a[0]; y[0][v].z *= a[0]; y[0][v].w *= a[0];
#pragma unroll
        for (int t = 1; t < U; ++t) fma4(y[0][v], a[t], y[t][v]);
        acc[v].x += y[0][v].x; acc[v].y += y[0][v].y; acc[v].z += y[0][v].z; acc[v].w += y[0][v].w;
    }
}

// The launches of one aggregation call are independent of each other but for the combination of the segments: every kernel lets its
// successor start at once, and waits for its predecessor's completion only before it ends.

// Accumulate entries [b, e) into acc[] for the lane's column groups, ascending entry order.
// The (col, val) pair of the NEXT batch of LPR entries is requested before the current batch's gathers,
// so that the index load's latency is hidden behind them instead of preceding every batch.
template <int LPR, int VPL, bool FULL = false>     // FULL: the slice has exactly LPR * VPL column groups (no lane is idle)
__device__ __forceinline__ void row_segment(const Params& p, int64_t b, int64_t e, int lig, unsigned mask,
                                            int w4, float4 (&acc)[VPL], unsigned keep = 0xFFFFFFFFu) {
    const float* Yb = p.Y + p.j0;
    if constexpr (LPR <= 2) {
        // too few lanes to hold a batch of (col, val) pairs: every lane reads them itself (its group reads one address)
        constexpr int U = VPL <= 2 ? 4 : 2;
        for (int64_t i0 = b; i0 < e; i0 += U) {
            int ck[U]; float ak[U]; float4 y[U][VPL];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const bool in = i0 + t < e;
                ck[t] = in ? __ldg(p.col + i0 + t) : 0;
                ak[t] = in ? __ldg(p.val + i0 + t) : 0.0f;
            }
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const float4* yr = reinterpret_cast<const float4*>(Yb + (int64_t)ck[t] * p.ldy);
                const bool live = i0 + t < e && index_ok(ck[t], p.y_rows, p.status, SITE_SPMM_COL);
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    const int c4 = lig + v * LPR;
                    y[t][v] = (live && (FULL || c4 < w4) && ((keep >> v) & 1u)) ? __ldg(yr + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int t = 0; t < U; ++t)
                if (!HUB && i0 + t < e) {
#pragma unroll
                    for (int v = 0; v < VPL; ++v) fma4(acc[v], ak[t], y[t][v]);
                }
            if (HUB) add_batch(acc, ak, y);
        }
        return;
    }
    constexpr int U = Cfg<LPR, VPL>::U;
    int c = 0; float a = 0.0f;
    if (b + lig < e) { c = __ldg(p.col + b + lig); a = __ldg(p.val + b + lig); }
    for (int64_t i0 = b; i0 < e; i0 += LPR) {
        int c_next = 0; float a_next = 0.0f;
        if (i0 + LPR + lig < e) { c_next = __ldg(p.col + i0 + LPR + lig); a_next = __ldg(p.val + i0 + LPR + lig); }
        const int cnt = (int)((e - i0) < LPR ? (e - i0) : LPR);
        for (int k = 0; k < cnt; k += U) {
            int ck[U]; float ak[U]; float4 y[U][VPL];
#pragma unroll
            for (int t = 0; t < U; ++t) {
                ck[t] = __shfl_sync(mask, c, k + t, LPR);
                ak[t] = __shfl_sync(mask, a, k + t, LPR);
            }
#pragma unroll
            for (int t = 0; t < U; ++t) {
                const float4* yr = reinterpret_cast<const float4*>(Yb + (int64_t)ck[t] * p.ldy);
                const bool live = k + t < cnt && index_ok(ck[t], p.y_rows, p.status, SITE_SPMM_COL);
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    const int c4 = lig + v * LPR;
                    y[t][v] = (live && (FULL || c4 < w4) && ((keep >> v) & 1u)) ? __ldg(yr + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int t = 0; t < U; ++t)
                if (!HUB && k + t < cnt) {
#pragma unroll
                    for (int v = 0; v < VPL; ++v) fma4(acc[v], ak[t], y[t][v]);
                }
            if (HUB) add_batch(acc, ak, y);
        }
        c = c_next; a = a_next;
    }
}

// The same for a whole warp on one unit of a narrow aggregation: EG = 32 / CL lane groups take entries g, g + EG, ...
// (each lane reads its group's column id and value itself, the next step's ahead of this step's gathers; consecutive
// groups read consecutive entries), then a butterfly over the groups leaves the complete sums in every lane.  The
// serial chain of a unit is EG times shorter than with one group per unit, which is what bounded narrow and small
// aggregations: 4,096 nodes / 70 K entries, widths 64 and 8: 60 -> 5 us for the slowest launch.
template <int CL, int VPL>
__device__ __forceinline__ void warp_segment(const Params& p, int64_t b, int len, int lane, int w4, float4 (&acc)[VPL],
                                             unsigned keep = 0xFFFFFFFFu) {
    constexpr int EG = 32 / CL, U = VPL == 1 ? 4 : 2;
    const int cl = lane & (CL - 1), eg = lane / CL;
    const float* Yb = p.Y + p.j0;
    const int32_t* col = p.col + b;
    const float* val = p.val + b;
    int c[U]; float a[U];
#pragma unroll
    for (int t = 0; t < U; ++t) {
        const int i = t * EG + eg;
        c[t] = i < len ? __ldg(col + i) : 0;
        a[t] = i < len ? __ldg(val + i) : 0.0f;
    }
    for (int i0 = 0; i0 < len; i0 += EG * U) {
        int cn[U]; float an[U]; float4 y[U][VPL];
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const int i = i0 + EG * U + t * EG + eg;
            cn[t] = i < len ? __ldg(col + i) : 0;
            an[t] = i < len ? __ldg(val + i) : 0.0f;
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
            const float4* yr = reinterpret_cast<const float4*>(Yb + (int64_t)c[t] * p.ldy);
            const bool live = i0 + t * EG + eg < len && index_ok(c[t], p.y_rows, p.status, SITE_SPMM_COL);
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c4 = cl + v * CL;
                y[t][v] = (live && c4 < w4 && ((keep >> v) & 1u)) ? __ldg(yr + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
#pragma unroll
        for (int t = 0; t < U; ++t)
            if (!HUB && i0 + t * EG + eg < len) {
#pragma unroll
                for (int v = 0; v < VPL; ++v) fma4(acc[v], a[t], y[t][v]);
            }
        if (HUB) add_batch(acc, a, y);
#pragma unroll
        for (int t = 0; t < U; ++t) { c[t] = cn[t]; a[t] = an[t]; }
    }
#pragma unroll
    for (int o = CL; o < 32; o <<= 1)
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            acc[v].x += __shfl_xor_sync(0xFFFFFFFFu, acc[v].x, o); acc[v].y += __shfl_xor_sync(0xFFFFFFFFu, acc[v].y, o);
            acc[v].z += __shfl_xor_sync(0xFFFFFFFFu, acc[v].z, o); acc[v].w += __shfl_xor_sync(0xFFFFFFFFu, acc[v].w, o);
        }
}

// Which of a lane's column groups the output mask of a sampled aggregation keeps (Eq. 4: outputs the mask drops are
// never computed -- a lane whose four columns of this row are all masked skips its gathers of every neighbour).
template <int LPR, int VPL>
__device__ __forceinline__ unsigned kept_groups(const Params& p, int64_t u, int lig, int w4) {
    const int64_t row = p.seg_perm ? __ldg(p.seg_perm + u) : u;
    unsigned keep = 0u;
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int c4 = lig + v * LPR;
        if (c4 < w4) {
            const int j = p.j0 + c4 * 4;
            if ((__ldg(p.out_bits + row * p.ld_bits + (j >> 5)) >> (j & 31)) & 0xFu) keep |= 1u << v;
        }
    }
    return keep;
}

// FULL (plain and bit-gate instances): the slice has exactly LPR * VPL column groups, so no load is predicated on its column.
template <int LPR, int VPL, int EPI = EPI_ANY, bool FULL = false>
__global__ void __launch_bounds__(256, VPL <= 2 ? SPMM_MINB : VPL == 3 && LPR >= 8 && LPR <= 16 ? (EPI == EPI_ANY ? SPMM_MINB - 1 : SPMM_MINB) : 1) spmm_group_kernel(const Params p) {
    constexpr bool LOSS = EPI == EPI_LOSS, PLAIN = epi_is_lean(EPI);
    pdl_trigger();
    const int lig = threadIdx.x % LPR;
    const int64_t idx = p.idx_begin + ((int64_t)blockIdx.x * 256 + threadIdx.x) / LPR;
    if (idx >= p.idx_end) return;  // the whole group leaves together
    const unsigned mask = LPR == 32 ? 0xFFFFFFFFu : (((1u << LPR) - 1u) << ((threadIdx.x & 31) & ~(LPR - 1)));
    int64_t b, e, u;
    if (p.rec) {
        const int4 r = __ldg(reinterpret_cast<const int4*>(p.rec + idx));
        b = ((int64_t)(uint32_t)r.y << 32) | (uint32_t)r.x;
        e = b + r.z;
        u = r.w;
    } else {
        u = idx;
        b = __ldg(p.rowptr + u);
        e = __ldg(p.rowptr + u + 1);
    }
    if (!unit_ok(p, b, e, u)) return;
    const int w4 = (p.w + 3) >> 2;
    float4 acc[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    unsigned keep = 0xFFFFFFFFu;
    if (!PLAIN && p.out_bits && p.bits_skip) keep = kept_groups<LPR, VPL>(p, u, lig, w4);
    row_segment<LPR, VPL, FULL>(p, b, e, lig, mask, w4, acc, keep);
    if (p.partial) {
        float4* dst = reinterpret_cast<float4*>(p.partial + idx * p.ldp);
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int c4 = lig + v * LPR;
            if (c4 < w4) dst[c4] = acc[v];
        }
    } else if constexpr (LOSS) {
        add_tiles<LPR, VPL>(p, u, lig, w4, acc);
        loss_epilogue<LPR, VPL>(p, u, lig, mask, acc);
    } else {
        add_tiles<LPR, VPL>(p, u, lig, w4, acc);
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int c4 = lig + v * LPR;
            if (c4 < w4) {
                if constexpr (PLAIN) store_lean<EPI>(p, u, c4, acc[v]);
                else store_row(p, u, c4, acc[v]);
            }
        }
    }
    pdl_wait();
}

// Units of more than 12 entries (and every segment) of an aggregation of at most 64 columns: one warp per unit.
template <int CL, int VPL, int EPI = EPI_ANY>
__global__ void __launch_bounds__(256, SPMM_MINB) spmm_warp_kernel(const Params p) {
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t idx = p.idx_begin + (((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5);
    if (idx >= p.idx_end) return;
    const int4 r = __ldg(reinterpret_cast<const int4*>(p.rec + idx));
    const int64_t b = ((int64_t)(uint32_t)r.y << 32) | (uint32_t)r.x, u = r.w;
    if (!unit_ok(p, b, b + r.z, u)) return;
    const int w4 = (p.w + 3) >> 2, cl = lane & (CL - 1);
    float4 acc[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    unsigned keep = 0xFFFFFFFFu;
    if (!HUB && EPI == EPI_ANY && p.out_bits && p.bits_skip) keep = kept_groups<CL, VPL>(p, u, cl, w4);
    warp_segment<CL, VPL>(p, b, r.z, lane, w4, acc, keep);
    if (lane < CL) {
        if (!p.partial) add_tiles<CL, VPL>(p, u, cl, w4, acc);
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int c4 = cl + v * CL;
            if constexpr (EPI != EPI_LOSS) {
                if (c4 < w4) {
                    if (p.partial) reinterpret_cast<float4*>(p.partial + idx * p.ldp)[c4] = acc[v];
                    else if constexpr (epi_is_lean(EPI)) store_lean<EPI>(p, u, c4, acc[v]);
                    else store_row(p, u, c4, acc[v]);
                }
            } else if (p.partial && c4 < w4) {
                reinterpret_cast<float4*>(p.partial + idx * p.ldp)[c4] = acc[v];
            }
        }
        if constexpr (EPI == EPI_LOSS) {
            if (!p.partial) loss_epilogue<CL, VPL>(p, u, cl, CL == 32 ? 0xFFFFFFFFu : (1u << (CL & 31)) - 1u, acc);
        }
    }
    pdl_wait();
}

// Rows of at most MAXE entries, width <= 128: a warp takes RB schedule records at once.  Lanes read the
// records, column ids and values in one coalesced load each; every gathered row of Y is then a single
// 512-byte request of the whole warp (lane = float4 column), RB of them in flight; entries of a row are
// added in entry order, as everywhere else.
template <int RB, int MAXE, int EPI = EPI_ANY, int VPL = 1>      // VPL float4 per lane: widths up to 128 * VPL
__global__ void __launch_bounds__(256, VPL == 1 && !HUB ? SPMM_SHORT_MINB : SPMM_MINB) spmm_short_kernel(const Params p) {
    static_assert(RB * MAXE <= 32, "one lane per (row, entry)");
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t idx0 = p.idx_begin + (((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5) * RB;
    if (idx0 >= p.idx_end) return;
    int4 rc = make_int4(0, 0, 0, 0);
    if (lane < RB && idx0 + lane < p.idx_end) rc = __ldg(reinterpret_cast<const int4*>(p.rec + idx0 + lane));
    if constexpr (DEBUG_BOUNDS) {
        const int64_t b0 = ((int64_t)(uint32_t)rc.y << 32) | (uint32_t)rc.x;
        if (!unit_ok(p, b0, b0 + rc.z, rc.w)) { rc.z = 0; rc.w = -1; }      // a bad record: no entries, no store
    }
    // lane (k, e) = (lane % RB, lane / RB) fetches entry e of row k
    const int k_of = lane % RB, e_of = lane / RB;
    const uint32_t lo = (uint32_t)__shfl_sync(0xFFFFFFFFu, rc.x, k_of), hi = (uint32_t)__shfl_sync(0xFFFFFFFFu, rc.y, k_of);
    const int len_of = __shfl_sync(0xFFFFFFFFu, rc.z, k_of);
    int c = 0; float a = 0.0f;
    if (e_of < MAXE && e_of < len_of) {
        const int64_t at = (((int64_t)hi << 32) | lo) + e_of;
        c = __ldg(p.col + at); a = __ldg(p.val + at);
    }
    const int w4 = (p.w + 3) >> 2;
    const float* Yb = p.Y + p.j0;
    float4 acc[RB][VPL];
#pragma unroll
    for (int k = 0; k < RB; ++k)
#pragma unroll
        for (int v = 0; v < VPL; ++v) acc[k][v] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int e = 0; e < MAXE; ++e) {
        float4 y[RB][VPL]; float ak[RB];
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int ck = __shfl_sync(0xFFFFFFFFu, c, k + e * RB);
            ak[k] = __shfl_sync(0xFFFFFFFFu, a, k + e * RB);
            const int len_k = __shfl_sync(0xFFFFFFFFu, rc.z, k);
            const bool live = e < len_k && index_ok(ck, p.y_rows, p.status, SITE_SPMM_COL);
            const float4* yr = reinterpret_cast<const float4*>(Yb + (int64_t)ck * p.ldy);
#pragma unroll
            for (int v = 0; v < VPL; ++v)
                y[k][v] = (live && lane + 32 * v < w4) ? __ldg(yr + lane + 32 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < RB; ++k) {
            const int len_k = __shfl_sync(0xFFFFFFFFu, rc.z, k);
            if (e < len_k) {
#pragma unroll
                for (int v = 0; v < VPL; ++v) fma4(acc[k][v], ak[k], y[k][v]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < RB; ++k) {
        const int64_t u = __shfl_sync(0xFFFFFFFFu, rc.w, k);
        if (idx0 + k < p.idx_end && (!DEBUG_BOUNDS || u >= 0)) {
            add_tiles<32, VPL>(p, u, lane, w4, acc[k]);
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c4 = lane + 32 * v;
                if (c4 < w4) {
                    if constexpr (epi_is_lean(EPI)) store_lean<EPI>(p, u, c4, acc[k][v]);      // as in spmm_group_kernel
                    else store_row(p, u, c4, acc[k][v]);
                }
            }
        }
    }
    pdl_wait();
}

// Long rows: add the segments' partial rows, apply the epilogue, write Z.  The rows come longest first: the first
// n_heavy of them (more than SPMM_HEAVY entries, tens to hundreds of segments) take a block each, whose threads split
// (column group, share of the segments) and add the shares in order through shared memory; the others take a warp
// (or, below 128 columns, a group of lanes) each.  With one warp for every row the launch lasted as long as the longest
// hub row's chain of loads: 300 K nodes, width 256: 108 -> 20 us per launch.
#if MIXGCN_SPMM_HUB
// The partial rows of a long row: its segments [0, segs), then its tiles' pieces [segs, all).
struct RowParts {
    const int64_t* seg_pos;          // of the row's first segment
    int64_t segs, all;
    static constexpr int64_t first = 0;
    const float* pieces; float scale;      // partial row of its first piece, the others HUB_ROWS rows apart
};
__device__ __forceinline__ RowParts row_parts(const Params& p, const int64_t* seg_pos, int64_t s0, int64_t s1, int64_t u) {
    RowParts r{seg_pos + s0, s1 - s0, s1 - s0, nullptr, 1.0f};
    const int32_t h = __ldg(p.hub_rank + u);
    if (h < 0) return r;
    const int rb = h / HUB_ROWS, q = __ldg(p.piece_first + rb), end = __ldg(p.piece_first + rb + 1);
    const int64_t row = (int64_t)q * HUB_ROWS + h % HUB_ROWS;
    if (end <= q || !index_ok(row + (int64_t)(end - q - 1) * HUB_ROWS, p.n_tile_sums, p.status, SITE_SPMM_SEG)) return r;
    r.all += end - q;
    r.pieces = p.tile_sums + row * p.ldp;
    r.scale = __ldg(p.row_scale + h);
    return r;
}
__device__ __forceinline__ float4 sum_parts(const Params& p, const RowParts& r, int64_t q, int64_t q_end, int c4) {
    double x = 0.0, y = 0.0, z = 0.0, w = 0.0;          // (see add_tiles)
    for (; q < q_end; q += 4) {
        float4 t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q + k >= q_end) continue;
            if (q + k < r.segs) {
                const int64_t slot = __ldg(r.seg_pos + q + k);
                if (index_ok(slot, p.n_partial, p.status, SITE_SPMM_SEG)) t[k] = __ldg(reinterpret_cast<const float4*>(p.partial + slot * p.ldp) + c4);
            } else {
                t[k] = __ldg(reinterpret_cast<const float4*>(r.pieces + (q + k - r.segs) * HUB_ROWS * p.ldp) + c4);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (q + k < q_end) {
                const double f = q + k < r.segs ? 1.0 : r.scale;
                x += f * t[k].x; y += f * t[k].y; z += f * t[k].z; w += f * t[k].w;
            }
    }
    return make_float4((float)x, (float)y, (float)z, (float)w);
}
#else
// The partial rows of a long row: its segments [first, all).
struct RowParts { const int64_t* seg_pos; int64_t first, all; };
__device__ __forceinline__ RowParts row_parts(const Params&, const int64_t* seg_pos, int64_t s0, int64_t s1, int64_t) { return {seg_pos, s0, s1}; }
__device__ __forceinline__ float4 sum_parts(const Params& p, const RowParts& r, int64_t q, int64_t q_end, int c4) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (; q < q_end; q += 4) {
        float4 t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q + k < q_end) {
                const int64_t slot = __ldg(r.seg_pos + q + k);
                if (index_ok(slot, p.n_partial, p.status, SITE_SPMM_SEG)) t[k] = __ldg(reinterpret_cast<const float4*>(p.partial + slot * p.ldp) + c4);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (q + k < q_end) { s.x += t[k].x; s.y += t[k].y; s.z += t[k].z; s.w += t[k].w; }
    }
    return s;
}
#endif

template <bool LOSS = false>
__global__ void __launch_bounds__(256) spmm_combine_kernel(const Params p, int64_t n_long, int64_t n_heavy,
                                                           const int64_t* __restrict__ seg_off,
                                                           const int64_t* __restrict__ seg_pos,
                                                           const int32_t* __restrict__ perm) {
    __shared__ float4 red[256];
    pdl_wait();                                   // the partial rows are complete
    const int w4 = (p.w + 3) >> 2;
    const bool heavy = blockIdx.x < n_heavy;
    int gl = 32;                                  // lanes per light row
    if (!LOSS && !heavy) while (gl > 1 && gl / 2 >= w4) gl >>= 1;
    const int64_t i = heavy ? (int64_t)blockIdx.x : n_heavy + (((int64_t)blockIdx.x - n_heavy) * 256 + threadIdx.x) / gl;
    if (i >= n_long) return;
    const int64_t s0 = seg_off[i], s1 = seg_off[i + 1];
    const int64_t u = perm[i];
    if (!index_ok(s0, p.n_partial + 1, p.status, SITE_SPMM_SEG) || !index_ok(s1, p.n_partial + 1, p.status, SITE_SPMM_SEG) ||
        !index_ok(u, p.n_out, p.status, SITE_SPMM_ROW)) return;
    if (p.row_filter && !__ldg(p.row_filter + u)) return;
    const RowParts parts = row_parts(p, seg_pos, s0, s1, u);
    if (heavy) {
        if (p.out_mask && threadIdx.x == 0) p.out_mask[u] = 1;    // long rows are kept without looking (conservative)
        int cp = 1;
        while (cp < 64 && cp * 4 < p.w_total) cp <<= 1;      // column groups side by side (by the full width: the shares set the order of the sums)
        const int shares = 256 / cp, col = threadIdx.x % cp, share = threadIdx.x / cp;
        const int64_t per = (parts.all - parts.first + shares - 1) / shares;
        const int64_t q0 = parts.first + share * per < parts.all ? parts.first + share * per : parts.all, q1 = q0 + per < parts.all ? q0 + per : parts.all;
        float4 row[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
        for (int c0 = 0; c0 < w4; c0 += cp) {
            const int c4 = c0 + col;
            red[threadIdx.x] = c4 < w4 ? sum_parts(p, parts, q0, q1, c4) : make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();
            if (threadIdx.x < cp) {
                float4 s = red[threadIdx.x];
                for (int k = 1; k < shares; ++k) {
                    const float4 t = red[k * cp + threadIdx.x];
                    s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
                }
                if constexpr (LOSS) red[threadIdx.x] = s;        // one turn: at most 256 columns
                else if (c4 < w4) store_row(p, u, c4, s);
            }
            __syncthreads();
        }
        if constexpr (LOSS) {
            if (threadIdx.x < 32) {
#pragma unroll
                for (int v = 0; v < 2; ++v) if ((int)threadIdx.x + v * 32 < w4) row[v] = red[threadIdx.x + v * 32];
                loss_epilogue<32, 2>(p, u, (int)threadIdx.x, 0xFFFFFFFFu, row);
            }
        }
        return;
    }
    const int lane = threadIdx.x % gl;
    if (p.out_mask && lane == 0) p.out_mask[u] = 1;
    if constexpr (LOSS) {
        // the whole row (at most 64 float4) in registers, then the same epilogue as the other rows
        float4 row[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int c4 = lane + v * 32;
            row[v] = c4 < w4 ? sum_parts(p, parts, parts.first, parts.all, c4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        loss_epilogue<32, 2>(p, u, lane, 0xFFFFFFFFu, row);
    } else {
        for (int c4 = lane; c4 < w4; c4 += gl) store_row(p, u, c4, sum_parts(p, parts, parts.first, parts.all, c4));
    }
}

// Launch with or without leave to start before the predecessor on the stream has finished (see pdl_trigger).
template <typename... Args>
void launch_k(void (*kernel)(Args...), unsigned blocks, cudaStream_t s, bool early, typename std::common_type<Args>::type... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

void launch_combine(const Params& p, const SpmmSchedule& S, bool loss, bool early, cudaStream_t s) {
    const int w4 = (p.w + 3) >> 2;
    int gl = 32;
    if (!loss) while (gl > 1 && gl / 2 >= w4) gl >>= 1;
    const int64_t light = S.n_long - S.n_heavy;
    const unsigned blocks = (unsigned)(S.n_heavy + (light * gl + 255) / 256);
    if (loss) launch_k(spmm_combine_kernel<true>, blocks, s, early, p, S.n_long, S.n_heavy, S.seg_off, S.seg_pos, S.perm);
    else launch_k(spmm_combine_kernel<false>, blocks, s, early, p, S.n_long, S.n_heavy, S.seg_off, S.seg_pos, S.perm);
}

template <int LPR, int VPL, bool LOSS = false>
void launch_group(const Params& p, cudaStream_t s, bool early) {
    const int64_t units = p.idx_end - p.idx_begin;
    if (units <= 0) return;
    const int per_block = 256 / LPR;
    const int64_t blocks = (units + per_block - 1) / per_block;
    // nothing between the sums and the stored row (or a partial row, which never has an epilogue): the plain instance
    // (one float4 per lane: the lean instances gain nothing there and the assembler spills a register in them)
    constexpr bool lean = !LOSS && VPL >= 2;
    if constexpr (lean) {
        constexpr bool FULL = LPR >= 8 && VPL != 3;                      // (narrow groups: nothing to gain; three float4: spills)
        const bool full = FULL && ((p.w + 3) >> 2) == LPR * VPL;
        switch (pick_epi(p)) {
            case EPI_PLAIN:
                if (full) launch_k(spmm_group_kernel<LPR, VPL, EPI_PLAIN, FULL>, (unsigned)blocks, s, early, p);
                else launch_k(spmm_group_kernel<LPR, VPL, EPI_PLAIN>, (unsigned)blocks, s, early, p);
                return;
            case EPI_BITS:
                if (full) launch_k(spmm_group_kernel<LPR, VPL, EPI_BITS, FULL>, (unsigned)blocks, s, early, p);
                else launch_k(spmm_group_kernel<LPR, VPL, EPI_BITS>, (unsigned)blocks, s, early, p);
                return;
            case EPI_BIAS: launch_k(spmm_group_kernel<LPR, VPL, EPI_BIAS>, (unsigned)blocks, s, early, p); return;
            case EPI_GATE: launch_k(spmm_group_kernel<LPR, VPL, EPI_GATE>, (unsigned)blocks, s, early, p); return;
            default: break;
        }
    }
    launch_k(spmm_group_kernel<LPR, VPL, LOSS ? EPI_LOSS : EPI_ANY>, (unsigned)blocks, s, early, p);
}

template <int CL, int VPL>
void launch_narrow(const Params& p, bool warp_units, bool loss, cudaStream_t s, bool early) {
    const int64_t units = p.idx_end - p.idx_begin;
    if (units <= 0) return;
    if (!warp_units) {
        if (loss) launch_group<CL, VPL, true>(p, s, early);
        else launch_group<CL, VPL>(p, s, early);
        return;
    }
    const unsigned blocks = (unsigned)((units + 7) / 8);
    if (loss) { launch_k(spmm_warp_kernel<CL, VPL, EPI_LOSS>, blocks, s, early, p); return; }
    switch (pick_epi(p)) {
        case EPI_PLAIN: launch_k(spmm_warp_kernel<CL, VPL, EPI_PLAIN>, blocks, s, early, p); return;
        case EPI_BIAS: launch_k(spmm_warp_kernel<CL, VPL, EPI_BIAS>, blocks, s, early, p); return;
        default: launch_k(spmm_warp_kernel<CL, VPL, EPI_ANY>, blocks, s, early, p); return;
    }
}

void dispatch_narrow(const Params& p, NarrowCfg c, bool warp_units, bool loss, cudaStream_t s, bool early) {
#define MIXGCN_SPMM_CASE(L, V) if (c.cl == L && c.vpl == V) { launch_narrow<L, V>(p, warp_units, loss, s, early); return; }
    MIXGCN_SPMM_CASE(1, 1) MIXGCN_SPMM_CASE(2, 1) MIXGCN_SPMM_CASE(4, 1) MIXGCN_SPMM_CASE(2, 3) MIXGCN_SPMM_CASE(8, 1)
    MIXGCN_SPMM_CASE(4, 3) MIXGCN_SPMM_CASE(8, 2)
#undef MIXGCN_SPMM_CASE
}

// The same packing for an aggregation with the loss epilogue (65..256 columns, one slice: at most two float4 per lane
// before folding).  Returns 0 if the shape has no instance.
int dispatch_loss(const Params& p, int fold, cudaStream_t s, bool early) {
    const int w4 = (p.w + 3) >> 2;
    int lpr = 1;
    while (lpr < 32 && lpr < w4) lpr <<= 1;
    int vpl = (w4 + lpr - 1) / lpr;
    while (fold > 1 && (lpr / fold < 1 || vpl * fold > 8)) fold >>= 1;
    lpr /= fold; vpl *= fold;
#define MIXGCN_SPMM_CASE(L, V) if (lpr == L && vpl == V) { launch_group<L, V, true>(p, s, early); return fold; }
    MIXGCN_SPMM_CASE(32, 1) MIXGCN_SPMM_CASE(32, 2) MIXGCN_SPMM_CASE(16, 2) MIXGCN_SPMM_CASE(16, 4)
    MIXGCN_SPMM_CASE(8, 4) MIXGCN_SPMM_CASE(8, 8) MIXGCN_SPMM_CASE(4, 8)
#undef MIXGCN_SPMM_CASE
    return 0;
}

// Base configuration for a slice of w4 float4 columns, then packed `fold`-fold (fold in {1,2,4,8}):
// fewer lanes per row, more float4 per lane.  Returns the fold actually used.
int dispatch(const Params& p, int fold, cudaStream_t s, bool early) {
    const int w4 = (p.w + 3) >> 2;
    int lpr = 1;
    while (lpr < 32 && lpr < w4) lpr <<= 1;
    int vpl = (w4 + lpr - 1) / lpr;
    while (fold > 1 && (lpr / fold < 1 || vpl * fold > 8)) fold >>= 1;
    lpr /= fold; vpl *= fold;
    // Three float4 a lane where a power of two leaves a quarter of the slots and more empty: a load costs the pipe four cycles however
    // many of its lanes take part (132 columns: 233 K nodes of mean degree 500 5.00 -> 4.55 ms, 700 K of 22 0.89 -> 0.80; 76 columns: 3.25 -> 2.73, 0.52 -> 0.46).  Entries are added in the same order.
    if (w4 > 16 && w4 <= 24 && ((lpr == 16 && vpl == 2) || (lpr == 8 && vpl == 4))) { launch_group<8, 3>(p, s, early); return fold; }
    if (w4 > 32 && w4 <= 48 && ((lpr == 32 && vpl == 2) || (lpr == 16 && vpl == 4))) { launch_group<16, 3>(p, s, early); return fold; }
#define MIXGCN_SPMM_CASE(L, V) if (lpr == L && vpl == V) { launch_group<L, V>(p, s, early); return fold; }
    MIXGCN_SPMM_CASE(32, 1) MIXGCN_SPMM_CASE(32, 2) MIXGCN_SPMM_CASE(32, 3) MIXGCN_SPMM_CASE(32, 4)
    MIXGCN_SPMM_CASE(32, 5) MIXGCN_SPMM_CASE(32, 6) MIXGCN_SPMM_CASE(32, 7) MIXGCN_SPMM_CASE(32, 8)
    MIXGCN_SPMM_CASE(16, 1) MIXGCN_SPMM_CASE(16, 2) MIXGCN_SPMM_CASE(16, 4) MIXGCN_SPMM_CASE(16, 6) MIXGCN_SPMM_CASE(16, 8)
    MIXGCN_SPMM_CASE(8, 1) MIXGCN_SPMM_CASE(8, 2) MIXGCN_SPMM_CASE(8, 4) MIXGCN_SPMM_CASE(8, 8)
    MIXGCN_SPMM_CASE(4, 1) MIXGCN_SPMM_CASE(4, 2) MIXGCN_SPMM_CASE(4, 4) MIXGCN_SPMM_CASE(4, 8)
    MIXGCN_SPMM_CASE(2, 1) MIXGCN_SPMM_CASE(2, 2) MIXGCN_SPMM_CASE(2, 4) MIXGCN_SPMM_CASE(2, 8)
    MIXGCN_SPMM_CASE(1, 1) MIXGCN_SPMM_CASE(1, 2) MIXGCN_SPMM_CASE(1, 4) MIXGCN_SPMM_CASE(1, 8)
#undef MIXGCN_SPMM_CASE
    return 0;
}

template <int RB, int VPL>
void launch_short(const Params& p, int64_t units, cudaStream_t s, bool early) {
    constexpr int MAXE = SPMM_SHORT_MAXE;
    const int64_t warps = (units + RB - 1) / RB;
    const unsigned blocks = (unsigned)((warps + 7) / 8);
    switch (pick_epi(p)) {
        case EPI_PLAIN: launch_k(spmm_short_kernel<RB, MAXE, EPI_PLAIN, VPL>, blocks, s, early, p); return;
        case EPI_BITS: launch_k(spmm_short_kernel<RB, MAXE, EPI_BITS, VPL>, blocks, s, early, p); return;
        case EPI_BIAS: launch_k(spmm_short_kernel<RB, MAXE, EPI_BIAS, VPL>, blocks, s, early, p); return;
        case EPI_GATE: launch_k(spmm_short_kernel<RB, MAXE, EPI_GATE, VPL>, blocks, s, early, p); return;
        default: launch_k(spmm_short_kernel<RB, MAXE, EPI_ANY, VPL>, blocks, s, early, p); return;
    }
}

// Segments of the long rows, the other rows by bucket, then the combination of the segments.  The first launch
// waits for whatever precedes it on the stream; the others may start as soon as their predecessor's blocks all
// run (each ends only after its predecessor has ended, and the combination waits before it reads).
mixgcn_status launch_rows(mixgcn_ctx* ctx, Params p, const SpmmSchedule& S, NarrowCfg narrow, bool loss, int64_t row_limit, int phase, float* partial, cudaStream_t s) {
    bool early = false;
    if (S.total_segs > 0) {
        p.partial = partial;
        LaunchScope scope(ctx, phase, s);
        p.idx_begin = 0; p.idx_end = S.total_segs;
        if (!HUB && p.out_bits && p.bits_skip) p.seg_perm = S.perm;       // a segment's record names its long row by ordinal
        if (narrow.cl) dispatch_narrow(p, narrow, true, false, s, early);
        else dispatch(p, p.w <= SPMM_FOLD_WMAX ? SPMM_FOLD_SEG : 1, s, early);
        p.seg_perm = nullptr; p.partial = nullptr;
        early = true;
    }
    // ordinary rows, in perm order: [n_long, n_rows) -> records [total_segs, total_segs + n_rows - n_long)
    int64_t bound[5];
    bound[0] = S.n_long;
    for (int q = 0; q < 3; ++q) bound[q + 1] = S.rows_above[q] > S.n_long ? S.rows_above[q] : S.n_long;
    bound[4] = S.n_rows;
    if (!HUB && row_limit >= 0 && row_limit < S.n_rows) {
        // rows come longest first: only the first row_limit of them are wanted (the rest are empty)
        const int64_t lim = row_limit > S.n_long ? row_limit : S.n_long;
        for (int q = 1; q < 5; ++q) if (bound[q] > lim) bound[q] = lim;
    }
    if (narrow.cl) bound[2] = bound[3] = bound[1];     // narrow rows of up to 12 entries: one bucket, one group of lanes each
    int64_t begin = bound[0];
    int fold = 1;
    for (int q = 0; q < 4; ++q, fold <<= 1) {
        int64_t end = bound[q + 1];
        if (end <= begin) continue;
        p.idx_begin = S.total_segs + (begin - S.n_long);
        p.idx_end = S.total_segs + (end - S.n_long);
        LaunchScope scope(ctx, phase, s);
        const int64_t units = p.idx_end - p.idx_begin;
        if (narrow.cl) {
            dispatch_narrow(p, narrow, q == 0, loss, s, early);
        } else if (loss) {
            if (!dispatch_loss(p, q == 0 ? (p.w <= SPMM_FOLD_WMAX ? SPMM_FOLD_MED : 1) : fold, s, early)) MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "spmm: no loss-epilogue kernel for width %d", p.w);
        } else if (q == 3 && p.w <= 128 && SPMM_PACK_DEG[2] <= SPMM_SHORT_MAXE) {
            // rows of at most SPMM_PACK_DEG[2] entries: several rows per warp, whole-warp gathers
            launch_short<SPMM_SHORT_RB, 1>(p, units, s, early);
        } else if (q == 3 && p.w <= 256 && SPMM_PACK_DEG[2] <= SPMM_SHORT_MAXE) {
            // the same for widths up to 256: two float4 per lane, two rows per warp
            launch_short<SPMM_SHORT_RB / 2, 2>(p, units, s, early);
        } else {
            dispatch(p, q == 0 ? (p.w <= SPMM_FOLD_WMAX ? SPMM_FOLD_MED : 1) : fold, s, early);
        }
        early = true;
        begin = end;
    }
    if (S.total_segs > 0) {
        LaunchScope scope(ctx, phase, s);
        p.partial = partial;
        launch_combine(p, S, loss, early, s);
        p.partial = nullptr;
    }
    return MIXGCN_OK;
}

}  // namespace
