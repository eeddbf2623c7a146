// Neighbour aggregation Z = A_hat Y (Algorithm 2, aggregation line): deterministic, atomic-free,
// row-wise CSR SpMM.
//
//  - A group of LPR lanes owns one output row (or one segment of a long row); each lane owns VPL
//    float4 column groups, so a gathered row of Y is read with coalesced 16-byte loads.
//  - The work list is the graph's schedule: one 16-byte record (first entry, length, row) per
//    unit, longest first, so a unit starts after ONE dependent load instead of a chain through
//    the permutation and the row pointers.
//  - (col,val) of the unit are fetched LPR at a time (one coalesced load per group) and handed
//    round with warp shuffles; U gathered rows (U * VPL = 8 float4 per lane) are in flight before
//    the FMAs, with a predicated tail instead of a one-by-one remainder.
//  - Degree buckets: rows of up to 12 / 5 / 2 entries share a warp 2- / 4- / 8-fold (fewer lanes per
//    row, more float4 per lane), so short rows still keep eight loads per lane in flight.
//  - Narrow aggregations (up to 64 columns) have too few column lanes to keep a long unit's loads in
//    flight: there a whole warp takes one unit of more than 12 entries, its lane groups take every EG-th
//    entry, and a butterfly adds the groups' sums (spmm_warp_kernel).
//  - Rows longer than the schedule's segment length (64..512 entries, shorter for small graphs) are cut (at
//    column-block boundaries and at that length) into segments that run as independent units, in order of
//    their first column, and write partial rows to scratch: hub rows that gather the same rows of Y do so
//    close in time and share them through the L2.  A last kernel adds the segments of each row in a fixed
//    order and applies the epilogue.  Every sum has a fixed order: the result is bit-reproducible.
//  - The launches of one call overlap: each releases its successor as soon as its own blocks are all
//    running (programmatic dependent launch), so a bucket's last wave shares the machine with the next bucket.
//  - The epilogue (bias, ReLU, dropout mask, gate by another tensor's sign) is applied in
//    registers before the single write of Z.
#define MIXGCN_SPMM_HUB 0
#include "spmm_kernels.cuh"

using namespace mixgcn;

namespace {

// Row-sparse input: most rows of Y are exactly zero (gradients of a masked loss and what they
// propagate to).  A unit scans its column ids, tests the row mask (one byte per entry, L2-resident)
// and gathers only the kept rows, four at a time, in entry order -- the same sum as the dense kernel
// with its zero terms left out.  Values are read for kept entries only.
template <int LPR, int VPL>
__global__ void __launch_bounds__(256) spmm_sparse_kernel(const SpmmParams p) {
    const int lig = threadIdx.x % LPR;
    const int64_t idx = p.idx_begin + ((int64_t)blockIdx.x * 256 + threadIdx.x) / LPR;
    if (idx >= p.idx_end) return;
    const int group_base = (threadIdx.x & 31) & ~(LPR - 1);
    const unsigned mask = LPR == 32 ? 0xFFFFFFFFu : (((1u << LPR) - 1u) << group_base);
    const int4 rc = __ldg(reinterpret_cast<const int4*>(p.rec + idx));
    const int64_t b = ((int64_t)(uint32_t)rc.y << 32) | (uint32_t)rc.x, e = b + rc.z;
    const int64_t u = rc.w;
    if (!unit_ok(p, b, e, u)) return;
    const int w4 = (p.w + 3) >> 2;
    const float* Yb = p.Y + p.j0;
    float4 acc[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    bool any = false;
    for (int64_t i0 = b; i0 < e; i0 += LPR) {
        int r = -1; float a = 0.0f;
        if (i0 + lig < e) {
            const int c = __ldg(p.col + i0 + lig);
            if (index_ok(c, p.n_cols, p.status, SITE_SPMM_COL) && __ldg(p.in_mask + c)) {
                r = p.in_pos ? __ldg(p.in_pos + c) : c;
                a = __ldg(p.val + i0 + lig);
            }
        }
        unsigned hits = __ballot_sync(mask, r >= 0) & mask;
        any |= hits != 0;
        constexpr int HB = VPL >= 4 ? 1 : 4 / VPL;     // kept rows gathered per batch
        while (hits) {
            int src[HB], nh = 0;
#pragma unroll
            for (int t = 0; t < HB; ++t) {
                src[t] = 0;
                if (hits) { src[t] = __ffs(hits) - 1 - group_base; hits &= hits - 1; ++nh; }
            }
            int rk[HB]; float ak[HB]; float4 y[HB][VPL];
#pragma unroll
            for (int t = 0; t < HB; ++t) {
                rk[t] = __shfl_sync(mask, r, src[t], LPR);
                ak[t] = __shfl_sync(mask, a, src[t], LPR);
            }
#pragma unroll
            for (int t = 0; t < HB; ++t) {
                const float4* yr = reinterpret_cast<const float4*>(Yb + (int64_t)(rk[t] < 0 ? 0 : rk[t]) * p.ldy);
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    const int c4 = lig + v * LPR;
                    y[t][v] = (t < nh && c4 < w4 && index_ok(rk[t], p.y_rows, p.status, SITE_SPMM_POS)) ? __ldg(yr + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int t = 0; t < HB; ++t)
                if (t < nh) {
#pragma unroll
                    for (int v = 0; v < VPL; ++v) fma4(acc[v], ak[t], y[t][v]);
                }
        }
    }
    if (p.partial) {
        float4* dst = reinterpret_cast<float4*>(p.partial + idx * p.ldp);
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int c4 = lig + v * LPR;
            if (c4 < w4) dst[c4] = acc[v];
        }
        return;
    }
    if (p.out_mask && lig == 0 && p.j0 == 0) p.out_mask[u] = any ? 1 : 0;
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int c4 = lig + v * LPR;
        if (c4 < w4) store_row(p, u, c4, acc[v]);
    }
}

// Row-filtered output: only the rows u with row_filter[u] != 0 are wanted (the last layer of a
// training step needs its output on train nodes only).  A warp scans 32 schedule records, tests the
// filter byte of each record's row and computes the kept ones one after the other with all 32 lanes,
// entries in the same order as spmm_group_kernel (bitwise the same rows as a full call without tiles).
template <int VPL>
__global__ void __launch_bounds__(256) spmm_filtered_kernel(const SpmmParams p) {
    const int lane = threadIdx.x & 31;
    const int64_t idx0 = p.idx_begin + ((((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5) << 5);
    if (idx0 >= p.idx_end) return;
    int4 rc = make_int4(0, 0, 0, 0);
    bool live = false;
    if (idx0 + lane < p.idx_end) {
        rc = __ldg(reinterpret_cast<const int4*>(p.rec + idx0 + lane));
        const int64_t b0 = ((int64_t)(uint32_t)rc.y << 32) | (uint32_t)rc.x;
        if (unit_ok(p, b0, b0 + rc.z, rc.w)) {
            const int64_t row = p.seg_perm ? __ldg(p.seg_perm + rc.w) : rc.w;
            live = index_ok(row, p.n_out, p.status, SITE_SPMM_ROW) && __ldg(p.row_filter + row) != 0;
        }
    }
    unsigned bits = __ballot_sync(0xFFFFFFFFu, live);
    const int w4 = (p.w + 3) >> 2;
    while (bits) {
        const int src = __ffs(bits) - 1;
        bits &= bits - 1;
        const uint32_t lo = (uint32_t)__shfl_sync(0xFFFFFFFFu, rc.x, src), hi = (uint32_t)__shfl_sync(0xFFFFFFFFu, rc.y, src);
        const int len = __shfl_sync(0xFFFFFFFFu, rc.z, src);
        const int64_t u = __shfl_sync(0xFFFFFFFFu, rc.w, src);
        const int64_t b = ((int64_t)hi << 32) | lo, e = b + len;
        float4 acc[VPL];
#pragma unroll
        for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        row_segment<32, VPL>(p, b, e, lane, 0xFFFFFFFFu, w4, acc);
        if (p.partial) {
            float4* dst = reinterpret_cast<float4*>(p.partial + (idx0 + src) * p.ldp);
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c4 = lane + v * 32;
                if (c4 < w4) dst[c4] = acc[v];
            }
        } else {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c4 = lane + v * 32;
                if (c4 < w4) store_row(p, u, c4, acc[v]);
            }
        }
    }
}

// The same for narrow aggregations: entry order and lane split of the dense path (one group of CL lanes walks a row
// of at most 12 entries, the whole warp shares a longer unit), so the rows are again bitwise those of the full call without tiles.
template <int CL, int VPL>
__global__ void __launch_bounds__(256) spmm_filtered_narrow_kernel(const SpmmParams p) {
    constexpr int PACKED = SPMM_PACK_DEG[0];
    const int lane = threadIdx.x & 31, cl = lane & (CL - 1);
    const int64_t idx0 = p.idx_begin + ((((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5) << 5);
    if (idx0 >= p.idx_end) return;
    int4 rc = make_int4(0, 0, 0, 0);
    bool live = false;
    if (idx0 + lane < p.idx_end) {
        rc = __ldg(reinterpret_cast<const int4*>(p.rec + idx0 + lane));
        const int64_t b0 = ((int64_t)(uint32_t)rc.y << 32) | (uint32_t)rc.x;
        if (unit_ok(p, b0, b0 + rc.z, rc.w)) {
            const int64_t row = p.seg_perm ? __ldg(p.seg_perm + rc.w) : rc.w;
            live = index_ok(row, p.n_out, p.status, SITE_SPMM_ROW) && __ldg(p.row_filter + row) != 0;
        }
    }
    unsigned bits = __ballot_sync(0xFFFFFFFFu, live);
    const int w4 = (p.w + 3) >> 2;
    const unsigned gmask = CL == 32 ? 0xFFFFFFFFu : (((1u << (CL & 31)) - 1u) << (lane & ~(CL - 1)));
    while (bits) {
        const int src = __ffs(bits) - 1;
        bits &= bits - 1;
        const uint32_t lo = (uint32_t)__shfl_sync(0xFFFFFFFFu, rc.x, src), hi = (uint32_t)__shfl_sync(0xFFFFFFFFu, rc.y, src);
        const int len = __shfl_sync(0xFFFFFFFFu, rc.z, src);
        const int64_t u = __shfl_sync(0xFFFFFFFFu, rc.w, src);
        const int64_t b = ((int64_t)hi << 32) | lo;
        float4 acc[VPL];
#pragma unroll
        for (int v = 0; v < VPL; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.partial || len > PACKED) warp_segment<CL, VPL>(p, b, len, lane, w4, acc);
        else row_segment<CL, VPL>(p, b, b + len, cl, gmask, w4, acc);
        if (lane < CL) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const int c4 = cl + v * CL;
                if (c4 < w4) {
                    if (p.partial) reinterpret_cast<float4*>(p.partial + (idx0 + src) * p.ldp)[c4] = acc[v];
                    else store_row(p, u, c4, acc[v]);
                }
            }
        }
        __syncwarp();
    }
}

void dispatch_filtered_narrow(const SpmmParams& p, NarrowCfg c, cudaStream_t s) {
    const int64_t units = p.idx_end - p.idx_begin;
    if (units <= 0) return;
    const unsigned blocks = (unsigned)((units + 255) / 256);   // 8 warps x 32 records
#define MIXGCN_SPMM_CASE(L, V) if (c.cl == L && c.vpl == V) { spmm_filtered_narrow_kernel<L, V><<<blocks, 256, 0, s>>>(p); return; }
    MIXGCN_SPMM_CASE(1, 1) MIXGCN_SPMM_CASE(2, 1) MIXGCN_SPMM_CASE(4, 1) MIXGCN_SPMM_CASE(2, 3) MIXGCN_SPMM_CASE(8, 1)
    MIXGCN_SPMM_CASE(4, 3) MIXGCN_SPMM_CASE(8, 2)
#undef MIXGCN_SPMM_CASE
}

template <int LPR, int VPL>
void launch_sparse(const SpmmParams& p, cudaStream_t s) {
    const int64_t units = p.idx_end - p.idx_begin;
    if (units <= 0) return;
    const int per_block = 256 / LPR;
    spmm_sparse_kernel<LPR, VPL><<<(unsigned)((units + per_block - 1) / per_block), 256, 0, s>>>(p);
}

void dispatch_sparse(const SpmmParams& p, int fold, cudaStream_t s) {
    const int w4 = (p.w + 3) >> 2;
    int lpr = 1;
    while (lpr < 32 && lpr < w4) lpr <<= 1;
    int vpl = (w4 + lpr - 1) / lpr;
    while (fold > 1 && (lpr / fold < 1 || vpl * fold > 8)) fold >>= 1;
    lpr /= fold; vpl *= fold;
#define MIXGCN_SPMM_CASE(L, V) if (lpr == L && vpl == V) { launch_sparse<L, V>(p, s); return; }
    MIXGCN_SPMM_CASE(32, 1) MIXGCN_SPMM_CASE(32, 2) MIXGCN_SPMM_CASE(32, 3) MIXGCN_SPMM_CASE(32, 4)
    MIXGCN_SPMM_CASE(32, 5) MIXGCN_SPMM_CASE(32, 6) MIXGCN_SPMM_CASE(32, 7) MIXGCN_SPMM_CASE(32, 8)
    MIXGCN_SPMM_CASE(16, 1) MIXGCN_SPMM_CASE(16, 2) MIXGCN_SPMM_CASE(16, 4) MIXGCN_SPMM_CASE(16, 6) MIXGCN_SPMM_CASE(16, 8)
    MIXGCN_SPMM_CASE(8, 1) MIXGCN_SPMM_CASE(8, 2) MIXGCN_SPMM_CASE(8, 4) MIXGCN_SPMM_CASE(8, 8)
    MIXGCN_SPMM_CASE(4, 1) MIXGCN_SPMM_CASE(4, 2) MIXGCN_SPMM_CASE(4, 4) MIXGCN_SPMM_CASE(4, 8)
    MIXGCN_SPMM_CASE(2, 1) MIXGCN_SPMM_CASE(2, 2) MIXGCN_SPMM_CASE(2, 4) MIXGCN_SPMM_CASE(2, 8)
    MIXGCN_SPMM_CASE(1, 1) MIXGCN_SPMM_CASE(1, 2) MIXGCN_SPMM_CASE(1, 4) MIXGCN_SPMM_CASE(1, 8)
#undef MIXGCN_SPMM_CASE
}

void dispatch_filtered(const SpmmParams& p, cudaStream_t s) {
    const int64_t units = p.idx_end - p.idx_begin;
    if (units <= 0) return;
    const unsigned blocks = (unsigned)((units + 255) / 256);   // 8 warps x 32 records
    const int vpl = (((p.w + 3) >> 2) + 31) / 32;
    switch (vpl) {
#define MIXGCN_SPMM_CASE(V) case V: spmm_filtered_kernel<V><<<blocks, 256, 0, s>>>(p); break;
        MIXGCN_SPMM_CASE(1) MIXGCN_SPMM_CASE(2) MIXGCN_SPMM_CASE(3) MIXGCN_SPMM_CASE(4)
        MIXGCN_SPMM_CASE(5) MIXGCN_SPMM_CASE(6) MIXGCN_SPMM_CASE(7) MIXGCN_SPMM_CASE(8)
#undef MIXGCN_SPMM_CASE
        default: break;
    }
}

constexpr int MAX_SLICE = 1024;      // columns per launch at most: 8 float4 per lane
constexpr int DEFAULT_SLICE = 256;   // widths above this run as slices of this many columns (2 float4 per lane, four CTAs per SM)

// bytes of scratch of one slice of w columns where tiles run: partial rows of the other entries' segments, then what the tiles need
int64_t tiles_scratch(const HubTiles* t, int32_t w, int64_t ldp, int64_t* images_at) {
    return t->rem.full.total_segs * ldp * (int64_t)sizeof(float) + 1024 + hub_tiles_scratch(t, w, ldp, images_at);
}
// of the widest slice of a call of w columns
int64_t tiles_scratch(const HubTiles* t, int32_t w) {
    const int32_t cols = w < DEFAULT_SLICE ? w : DEFAULT_SLICE;
    int64_t images_at = 0;
    return tiles_scratch(t, cols, ((int64_t)cols + 3) / 4 * 4, &images_at);
}

}  // namespace

namespace mixgcn {

mixgcn_status reserve_tiles_scratch(mixgcn_ctx* ctx, const HubTiles* t, int32_t w) {
    if (!t || w <= 0 || !hub_tiles_pay(t, w)) return MIXGCN_OK;
    const mixgcn_status st = ensure_workspace_spmm(ctx, tiles_scratch(t, w));
    return st == MIXGCN_ENOMEM ? MIXGCN_OK : st;
}

// Aggregation of all rows (chunks <= 1) or of row chunk k of `chunks` (the pipeline's chunks), each
// with its own schedule: long rows as column-ordered segments, then rows longest first, short rows packed.
mixgcn_status launch_spmm(mixgcn_ctx* ctx, const mixgcn_graph* g, const CsrView& A, int chunks, int k,
                          int32_t w, const float* Y, int64_t ldy, float* Z, int64_t ldz,
                          const mixgcn_epilogue* epi, cudaStream_t s, const SpmmOpts& opts) {
    const SpmmRowSparse* sparse = opts.sparse;
    const LossFuse* lf = opts.loss;
    const uint8_t* row_filter = opts.row_filter;
    const int phase = opts.phase;
    const int64_t row_limit = opts.row_limit;
    if (w <= 0) return MIXGCN_OK;
    if (!Z && !opts.Z_lp) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: no output");
    if (sparse && row_filter) MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "spmm: a row filter cannot be combined with a row-sparse input");
    if (epi && epi->sign_bits && (row_filter || opts.row_limit >= 0 || lf || !Z))
        MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "spmm: the sign bitmap needs every row of a plain fp32 result");
    if (lf) {
        if (sparse || row_filter || chunks > 1 || opts.out_bits || opts.Z_lp || opts.row_limit >= 0 || !Z || w > 256 ||
            (epi && (epi->relu || epi->drop_mask || epi->gate || epi->residual)))
            MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "spmm: the loss epilogue takes a plain aggregation of at most 256 columns with a bias");
    }
    if (chunks > 1) {
        MIXGCN_TRY(ensure_chunk_schedules(g, A, chunks));
        if (k < 0 || k >= A.n_chunk) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: chunk %d of %d does not exist", k, chunks);
    }
    recording_uses(ctx, g->memory);
    // tiles of the dense corner, where the call asks for them, the graph has them and the call is a plain one over a whole orientation
    const HubTiles* tiles = nullptr;
    if (opts.tiles && chunks <= 1 && !sparse && !row_filter && row_limit < 0 && !opts.out_bits && (&A == &g->fwd || &A == &g->bwd)) {
        tiles = g->tiles[&A == &g->bwd].load(std::memory_order_acquire);
        if (tiles && !hub_tiles_pay(tiles, w)) tiles = nullptr;
    }
    if (tiles) {        // scratch of the widest slice; the gather kernels alone where there is no memory for it
        const mixgcn_status st = ensure_workspace_spmm(ctx, tiles_scratch(tiles, w));
        if (st == MIXGCN_ENOMEM) tiles = nullptr;
        else MIXGCN_TRY(st);
    }
    // (with tiles the order of a row's sums goes by the slices' width, so that they always have the default one)
    const int slice = tiles ? DEFAULT_SLICE : lf ? MAX_SLICE : ctx->spmm_slice_cols > 0 ? (ctx->spmm_slice_cols < MAX_SLICE ? ctx->spmm_slice_cols : MAX_SLICE) : DEFAULT_SLICE;
    const CsrView& V = tiles ? tiles->rem : A;       // with tiles: what they leave
    const SpmmSchedule& S = chunks > 1 ? A.chunk[k] : V.full;
    if (S.n_rows <= 0) return MIXGCN_OK;
    SpmmParams p{};
    p.rowptr = V.rowptr; p.col = V.col; p.val = V.val;
    p.Y = Y; p.ldy = ldy; p.Z = Z; p.ldz = ldz; p.w_total = w;
    p.Z_lp = opts.Z_lp; p.ldz_lp = opts.ldz_lp;
    p.out_bits = opts.out_bits; p.ld_bits = opts.ld_bits; p.bits_scale = 1.0f; p.bits_skip = 1;
    if (epi && epi->gate_bits) {
        // a bit-packed gate goes through the same bitmap path as the sampled aggregation's output mask
        if (opts.out_bits) MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "spmm: a sampled aggregation takes no bit-packed gate as well");
        p.out_bits = epi->gate_bits; p.ld_bits = epi->ld_gate_bits; p.bits_scale = epi->gate_scale; p.bits_skip = 0;
    }
    if (epi) {
        p.bias = epi->bias; p.relu = epi->relu; p.drop = epi->drop_mask; p.keep_scale = epi->keep_scale;
        p.gate = epi->gate_bits ? nullptr : epi->gate; p.ld_gate = epi->ld_gate; p.gate_scale = epi->gate_scale;
        p.residual = epi->residual; p.ld_residual = epi->ld_residual; p.residual_scale = epi->residual_scale;
    }
    p.status = ctx->d_status;
    p.n_out = g->n; p.n_cols = g->n; p.y_rows = opts.y_rows >= 0 ? opts.y_rows : g->n;
    p.nnz = opts.nnz >= 0 ? opts.nnz : tiles ? tiles->rem_nnz : g->nnz;
    p.n_long = S.n_long; p.n_partial = S.total_segs;
    p.rec = S.rec;
    if (sparse) { p.in_mask = sparse->in_mask; p.in_pos = sparse->in_pos; p.out_mask = sparse->out_mask; }
    p.row_filter = row_filter;
    if (lf) {
        p.loss_labels = lf->labels; p.loss_mask = lf->train_mask; p.loss_count = lf->count;
        p.loss_row = lf->row_loss; p.loss_pred = lf->pred; p.loss_zero_rows = lf->zero_rows;
    }
    const NarrowCfg narrow = narrow_cfg(w);
    for (int j0 = 0; j0 < w; j0 += slice) {
        p.j0 = j0;
        p.w = (w - j0) < slice ? (w - j0) : slice;
        if (sparse) {
            // same units, sparse-input kernel: long-row segments to scratch + combine, then every other row
            if (S.total_segs > 0) {
                const int64_t ldp = ((int64_t)p.w + 3) / 4 * 4;
                MIXGCN_TRY(ensure_workspace_spmm(ctx, S.total_segs * ldp * (int64_t)sizeof(float)));
                p.partial = reinterpret_cast<float*>(ctx->workspace_spmm); p.ldp = ldp;
                {
                    LaunchScope scope(ctx, PH_SPMM_SPARSE, s);
                    p.idx_begin = 0; p.idx_end = S.total_segs;
                    dispatch_sparse(p, 1, s);
                }
                {
                    LaunchScope scope(ctx, PH_SPMM_SPARSE, s);
                    launch_combine(p, S, false, false, s);
                }
                p.partial = nullptr;
            }
            {
                // ordinary rows by degree bucket, short rows packed 2/4/8 per warp as in the dense path
                int64_t bnd[5];
                bnd[0] = S.n_long;
                for (int q = 0; q < 3; ++q) bnd[q + 1] = S.rows_above[q] > S.n_long ? S.rows_above[q] : S.n_long;
                bnd[4] = S.n_rows;
                int64_t begin = bnd[0];
                int fold = 1;
                for (int q = 0; q < 4; ++q, fold <<= 1) {
                    const int64_t end = bnd[q + 1];
                    if (end <= begin) continue;
                    p.idx_begin = S.total_segs + (begin - S.n_long);
                    p.idx_end = S.total_segs + (end - S.n_long);
                    LaunchScope scope(ctx, PH_SPMM_SPARSE, s);
                    dispatch_sparse(p, fold, s);
                    begin = end;
                }
            }
            continue;
        }
        if (row_filter) {
            // kept rows only: segments of kept long rows, their combination, then every other kept row
            if (S.total_segs > 0) {
                const int64_t ldp = ((int64_t)p.w + 3) / 4 * 4;
                MIXGCN_TRY(ensure_workspace_spmm(ctx, S.total_segs * ldp * (int64_t)sizeof(float)));
                p.partial = reinterpret_cast<float*>(ctx->workspace_spmm); p.ldp = ldp;
                {
                    LaunchScope scope(ctx, PH_SPMM_SPARSE, s);
                    p.idx_begin = 0; p.idx_end = S.total_segs;
                    p.seg_perm = S.perm;
                    if (narrow.cl) dispatch_filtered_narrow(p, narrow, s);
                    else dispatch_filtered(p, s);
                    p.seg_perm = nullptr;
                }
                {
                    LaunchScope scope(ctx, PH_SPMM_SPARSE, s);
                    launch_combine(p, S, false, false, s);
                }
                p.partial = nullptr;
            }
            if (S.n_rows > S.n_long) {
                LaunchScope scope(ctx, PH_SPMM_SPARSE, s);
                p.idx_begin = S.total_segs; p.idx_end = S.total_segs + (S.n_rows - S.n_long);
                if (narrow.cl) dispatch_filtered_narrow(p, narrow, s);
                else dispatch_filtered(p, s);
            }
            continue;
        }
        // the segments' partial rows, then what the tiles need
        const int64_t ldp = ((int64_t)p.w + 3) / 4 * 4, seg_bytes = S.total_segs * ldp * (int64_t)sizeof(float);
        int64_t images_at = 0;
        const int64_t scratch = tiles ? tiles_scratch(tiles, p.w, ldp, &images_at) : seg_bytes;
        if (scratch > 0) MIXGCN_TRY(ensure_workspace_spmm(ctx, scratch));
        float* partial = reinterpret_cast<float*>(ctx->workspace_spmm);
        p.ldp = ldp;
        if (!tiles) { MIXGCN_TRY(launch_rows(ctx, p, S, narrow, lf != nullptr, row_limit, phase, partial, s)); continue; }
        // the tiles first: the launch behind waits for their sums
        uint8_t* base = reinterpret_cast<uint8_t*>(((uintptr_t)partial + seg_bytes + 1023) & ~(uintptr_t)1023);
        float* sums = reinterpret_cast<float*>(base);
        static_assert(DEFAULT_SLICE <= HUB_SLICE, "a slice is one product");
        MIXGCN_TRY(launch_hub_tiles(ctx, tiles, phase, p.w, p.Y + j0, ldy, p.y_rows, sums, ldp, base + images_at, s));
        SpmmHubParams hp{};
        static_cast<SpmmParams&>(hp) = p;
        hp.hub_rank = tiles->rank; hp.piece_first = tiles->piece_first; hp.row_scale = tiles->row_scale;
        hp.tile_sums = sums; hp.n_tile_sums = (int64_t)tiles->n_pieces * HUB_ROWS;
        MIXGCN_TRY(launch_rows_hub(ctx, hp, S, narrow, lf != nullptr, phase, partial, s));
    }
    MIXGCN_CUDA(cudaGetLastError());
    // sign bitmap of the result: one more pass over the rows this call wrote
    if (epi && epi->sign_bits)
        MIXGCN_TRY(launch_mask_pack(ctx, S.n_rows, w, Z + S.row0 * ldz, ldz, nullptr, epi->sign_bits + S.row0 * epi->ld_sign_bits,
                                    epi->ld_sign_bits, s));
    return MIXGCN_OK;
}

}  // namespace mixgcn

extern "C" mixgcn_status mixgcn_spmm(mixgcn_ctx* ctx, const mixgcn_graph* g, int transposed, int32_t w,
                                     const float* Y, int64_t ldy, float* Z, int64_t ldz,
                                     const mixgcn_epilogue* epi, void* stream) {
    return mixgcn_spmm_tiles(ctx, g, transposed, w, Y, ldy, Z, ldz, epi, g && g->tiles_in_spmm.load(std::memory_order_acquire), stream);
}

extern "C" mixgcn_status mixgcn_spmm_tiles(mixgcn_ctx* ctx, const mixgcn_graph* g, int transposed, int32_t w,
                                           const float* Y, int64_t ldy, float* Z, int64_t ldz,
                                           const mixgcn_epilogue* epi, int32_t tiles, void* stream) {
    if (!ctx || !g || !Y || !Z) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: null argument");
    if (w <= 0) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: w must be positive (got %d)", w);
    if (ldy < w || ldz < w || (ldy & 3) || (ldz & 3))
        MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: leading dimensions must be multiples of 4 and >= w (ldy=%lld ldz=%lld w=%d)",
                    (long long)ldy, (long long)ldz, w);
    if (!aligned16(Y) || !aligned16(Z)) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: Y and Z must be 16-byte aligned");
    if (Y == Z) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: Y and Z must not overlap");
    if (epi && epi->gate && epi->ld_gate < w) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: gate leading dimension < w");
    if (epi && epi->residual && (epi->ld_residual < w || epi->residual == Z)) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: residual needs ld_residual >= w and must not be the output");
    if (epi && ((epi->gate_bits && epi->ld_gate_bits < (w + 31) / 32) || (epi->sign_bits && epi->ld_sign_bits < (w + 31) / 32)))
        MIXGCN_FAIL(MIXGCN_EINVAL, "spmm: a bit-packed mask needs ld >= ceil(w / 32) words");
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    SpmmOpts opts; opts.tiles = tiles != 0;
    return launch_spmm(ctx, g, transposed ? g->bwd : g->fwd, 1, 0, w, Y, ldy, Z, ldz, epi, (cudaStream_t)stream, opts);
}

namespace {

// bits[u][j] = (X == null || X[u][j] > 0) && (bytes == null || bytes[u*w + j] != 0): one thread per 32-bit word
__global__ void mask_pack_kernel(int64_t n, int w, const float* __restrict__ X, int64_t ldx, const uint8_t* __restrict__ bytes,
                                 uint32_t* __restrict__ bits, int64_t ld_bits) {
    const int words = (w + 31) >> 5;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * words) return;
    const int64_t u = t / words; const int wd = (int)(t % words);
    uint32_t out = 0;
    for (int b = 0; b < 32; ++b) {
        const int j = wd * 32 + b;
        if (j >= w) break;
        bool on = true;
        if (X) on = X[u * ldx + j] > 0.0f;
        if (bytes) on = on && bytes[u * (int64_t)w + j] != 0;
        out |= (on ? 1u : 0u) << b;
    }
    bits[u * ld_bits + wd] = out;
}

}  // namespace

namespace mixgcn {
mixgcn_status launch_mask_pack(mixgcn_ctx* ctx, int64_t n, int32_t w, const float* X, int64_t ldx, const uint8_t* bytes,
                               uint32_t* bits, int64_t ld_bits, cudaStream_t s) {
    if (n <= 0 || w <= 0) return MIXGCN_OK;
    const int64_t total = n * ((w + 31) / 32);
    LaunchScope scope(ctx, PH_ELEM, s);
    mask_pack_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(n, w, X, ldx, bytes, bits, ld_bits);
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}
}  // namespace mixgcn

extern "C" mixgcn_status mixgcn_mask_pack(mixgcn_ctx* ctx, int64_t n, int32_t w, const float* X, int64_t ldx,
                                          const uint8_t* bytes, uint32_t* bits, int64_t ld_bits, void* stream) {
    if (!ctx || !bits || (!X && !bytes)) MIXGCN_FAIL(MIXGCN_EINVAL, "mask_pack: null argument");
    if (n <= 0 || w <= 0 || ld_bits < (w + 31) / 32 || (X && ldx < w)) MIXGCN_FAIL(MIXGCN_EINVAL, "mask_pack: need n, w > 0, ld_bits >= ceil(w/32), ldx >= w");
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    return launch_mask_pack(ctx, n, w, X, ldx, bytes, bits, ld_bits, (cudaStream_t)stream);
}

extern "C" mixgcn_status mixgcn_spmm_sampled(mixgcn_ctx* ctx, const mixgcn_graph* g, int transposed, int32_t w,
                                             const float* Y, int64_t ldy, float* Z, int64_t ldz, const uint32_t* mask_bits,
                                             int64_t ld_bits, const mixgcn_epilogue* epi, void* stream) {
    if (!ctx || !g || !Y || !Z || !mask_bits) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: null argument");
    if (w <= 0) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: w must be positive (got %d)", w);
    if (ldy < w || ldz < w || (ldy & 3) || (ldz & 3) || ld_bits < (w + 31) / 32)
        MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: leading dimensions must be multiples of 4 and >= w, ld_bits >= ceil(w/32)");
    if (!aligned16(Y) || !aligned16(Z)) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: Y and Z must be 16-byte aligned");
    if (Y == Z) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: Y and Z must not overlap");
    if (epi && epi->gate && epi->ld_gate < w) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: gate leading dimension < w");
    if (epi && epi->residual && (epi->ld_residual < w || epi->residual == Z)) MIXGCN_FAIL(MIXGCN_EINVAL, "spmm_sampled: residual needs ld_residual >= w and must not be the output");
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    SpmmOpts opts; opts.out_bits = mask_bits; opts.ld_bits = ld_bits;
    return launch_spmm(ctx, g, transposed ? g->bwd : g->fwd, 1, 0, w, Y, ldy, Z, ldz, epi, (cudaStream_t)stream, opts);
}
