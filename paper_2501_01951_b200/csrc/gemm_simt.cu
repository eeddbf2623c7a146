// Dense update products in plain fp32 on the CUDA cores (the strict-precision mode of the
// update line of Algorithm 2 and of its two backward products, where they are too small or not aligned for the
// tensor cores), plus the small streaming
// kernels around them (column sums for the bias gradient, the ReLU/dropout gate on a gradient).
//
// Long reductions (K = number of nodes in the weight-gradient product) are split over CTAs into partial
// tiles that a second kernel adds in a fixed order in fp64, and inside a CTA the fp32 accumulator is
// flushed into a second-level sum every 1024 terms, so rounding error does not grow with the node count.
#include "internal.cuh"

using namespace mixgcn;

namespace {

constexpr int BK = 16;              // k-step
constexpr int STAGES = 3;
constexpr int FLUSH_STEPS = 64;     // 64 * 16 = 1024 terms per first-level accumulator
constexpr int MIN_K_PER_SPLIT = 128;

struct Epi {
    const float* bias; int relu;
    const uint8_t* drop; float keep_scale;
    const float* gate; int64_t ld_gate; float gate_scale;
    const uint32_t* gate_bits; int64_t ld_gate_bits;   // bit-packed gate (replaces `gate`)
    uint32_t* sign_bits; int64_t ld_sign_bits;         // output: bit = (final y > 0)
    int64_t row0;
};

__device__ __forceinline__ float apply_epi(const Epi& e, float y, int64_t m, int64_t n, int64_t N) {
    if (e.bias) y += e.bias[n];
    if (e.relu) y = fmaxf(y, 0.0f);
    if (e.drop) y = e.drop[(e.row0 + m) * N + n] ? y * e.keep_scale : 0.0f;
    if (e.gate) y = e.gate[(e.row0 + m) * e.ld_gate + n] > 0.0f ? y * e.gate_scale : 0.0f;
    if (e.gate_bits) y = ((e.gate_bits[(e.row0 + m) * e.ld_gate_bits + (n >> 5)] >> (n & 31)) & 1u) ? y * e.gate_scale : 0.0f;
    return y;
}

struct GemmParams {
    int64_t M, N, K;
    const float* A; int64_t lda;
    const float* B; int64_t ldb;
    float* C; int64_t ldc;       // output, or partial workspace [splits][M][N] when splits > 1
    int64_t k_per_split; int splits;
    int64_t m_tiles, n_tiles;
    int vec_a, vec_b, vec_c;     // 16-byte vector access is legal (pointer and ld aligned)
    int vec_drop;                // mask bytes that can be copied at once (16 or 4; 0: the mask is read in the epilogue)
    int vec_gate;                // 16-byte access for four gate values at a multiple of four columns
    const int32_t* only_if;      // nullable: every CTA returns at once where this word is zero
    Epi epi;
};

// two fp32 lanes in one register pair: one instruction, two IEEE FMAs
typedef unsigned long long f32x2;
__device__ __forceinline__ void ffma2(f32x2& d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ f32x2 dup2(float a) { f32x2 r; asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a)); return r; }
__device__ __forceinline__ float2 split2(f32x2 v) { float2 f; asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v)); return f; }

__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {      // the first `bytes` of 16, zeros behind
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
// four consecutive floats, the first `valid` of them read (<= 0: none, `base` stands in for the address)
__device__ __forceinline__ void copy4(float* dst, const float* src, int64_t valid, int vec, const float* base) {
    const int v = valid >= 4 ? 4 : valid > 0 ? (int)valid : 0;
    if (vec) { cp_async16(dst, v ? src : base, v * 4); return; }
#pragma unroll
    for (int t = 0; t < 4; ++t) cp_async4(dst + t, t < v ? src + t : base, t < v ? 4 : 0);
}

// C = op(A) op(B) on the FMA pipes: a BM x BN tile per CTA, an 8 x 16 (smaller tiles 8 x 8) micro-tile per thread held as packed pairs (one
// fma.rn.f32x2 does two FMAs, so that the shared-memory loads and the operand copies find free issue slots beside a full
// FMA pipe), 16-deep k-steps through three cp.async stages.  Bound by the FMA rate (72 TFLOP/s measured with either
// form of the instruction): 170 K x 256 x 256 forward 33.7 -> 42 TFLOP/s, weight gradient 25.4 -> 48 TFLOP/s against one
// stage, register staging and scalar FMAs; with the large tile's operands read ahead 44 (50.8 at K = 1024), the weight gradient 50.
// Next to the FMAs stand the operands: a micro-tile's 96 bytes a thread and k take the load/store pipe three quarters of the FMAs' time.
//   A with K contiguous stays [m][k] in shared memory and is read two k at a time (row pitch 20 floats: the four rows a
//   warp reads side by side lie in different banks); A with M contiguous, and B, are [k][m] / [k][n].  B with K
//   contiguous (the small weight matrix of dP W^T) is turned round by word-wide copies.
// Long reductions: after 1024 terms the accumulators are added to C (the partial tile or C itself), which serves as the
// second-level sum.
// KG > 1: KG groups of threads share a tile, each taking every KG-th part of a k-step; their sums are added, in order, in the
// epilogue's shared memory.  Small products have few tiles: the tile's length is then the product's, and KG warps walk it
// in a KG-th of the time without the smaller micro-tile's extra shared-memory traffic.
template <int BM, int BN, int TN, int KG>
struct SimtCfg {
    static constexpr int GROUP = BM * BN / (8 * TN), NT = GROUP * KG;    // threads of a group, of the CTA
    static constexpr int MIN_CTAS = BM == 128 ? (BN == 128 ? 2 : 4) : (BN == 64 ? 6 : 10) / KG;
    static constexpr int a_floats(bool ta) { return ta ? BK * (BM + 4) : BM * (BK + 4); }
    static constexpr int B_FLOATS = BK * (BN + 4);
    // the k-steps' ring, which the epilogue uses again for half of the tile; the mask of the tile lies behind
    static constexpr int ring_bytes(bool ta) {
        const int ring = STAGES * (a_floats(ta) + B_FLOATS), half_tile = BM / 2 * (BN + 4);
        return (ring > half_tile ? ring : half_tile) * (int)sizeof(float);
    }
};
constexpr int FINE_KG = 4;

template <int BM, int BN, int TN, int KG, bool TA, bool TB>
__global__ void __launch_bounds__(SimtCfg<BM, BN, TN, KG>::NT, SimtCfg<BM, BN, TN, KG>::MIN_CTAS) gemm_simt_kernel(const GemmParams p) {
    if (p.splits == 1) pdl_trigger();        // (see chain_begin)
    pdl_wait();
    constexpr int TM = 8, NT = SimtCfg<BM, BN, TN, KG>::NT, H = TM / 4, TX = BN / TN, Q = TN / 4, QW = BN / Q;   // Q groups of four columns, QW columns apart
    constexpr int A_PITCH = TA ? BM + 4 : BK + 4, B_PITCH = BN + 4;
    using Cfg = SimtCfg<BM, BN, TN, KG>;
    constexpr int A_FLOATS = Cfg::a_floats(TA), B_FLOATS = Cfg::B_FLOATS;
    extern __shared__ __align__(16) float smem_f[];
    if (p.only_if && *p.only_if == 0) return;
    const int tid = threadIdx.x, lane = tid & 31;
    const int kg = tid / SimtCfg<BM, BN, TN, KG>::GROUP, warp = (tid % SimtCfg<BM, BN, TN, KG>::GROUP) >> 5;
    // a warp covers 4 x 8 micro-tiles (TX >= 8) or 8 x 4
    constexpr int WX = TX >= 8 ? 8 : TX, WY = 32 / WX, WARPS_X = TX / WX;
    const int tx = (warp % WARPS_X) * WX + lane % WX, ty = (warp / WARPS_X) * WY + lane / WX;
    const int64_t tile = blockIdx.x;
    const int64_t m0 = (tile / p.n_tiles) * BM, n0 = (tile % p.n_tiles) * BN;
    const int64_t kb = (int64_t)blockIdx.z * p.k_per_split;
    const int64_t ke = (kb + p.k_per_split < p.K) ? kb + p.k_per_split : p.K;
    const int steps = (int)((ke - kb + BK - 1) / BK);
    // rows of the micro-tile: i-th row is ty + i * (BM / TM) with A as [m][k], (i / 4) * (BM / H) + ty * 4 + i % 4 as [k][m];
    // columns: (j / 4) * QW + tx * 4 + j % 4
    auto row_of = [&](int i) { return TA ? (i >> 2) * (BM / H) + ty * 4 + (i & 3) : ty + i * (BM / TM); };

    auto load_a = [&](int ks) {
        float* As = smem_f + (ks % STAGES) * (A_FLOATS + B_FLOATS);
        const int64_t k0 = kb + (int64_t)ks * BK;
        auto one = [&](int i, int vec) {
            const int f = tid + i * NT;
            if (!TA) {
                const int r = f / 4, kq = (f % 4) * 4;
                const int64_t m = m0 + r, k = k0 + kq;
                copy4(As + r * A_PITCH + kq, p.A + m * p.lda + k, m < p.M ? ke - k : 0, vec, p.A);
            } else {
                const int kr = f / (BM / 4), mq = (f % (BM / 4)) * 4;
                const int64_t k = k0 + kr, m = m0 + mq;
                copy4(As + kr * A_PITCH + mq, p.A + k * p.lda + m, k < ke ? p.M - m : 0, vec, p.A);
            }
        };
        if (p.vec_a) {
#pragma unroll
            for (int i = 0; i < BM * BK / 4 / NT; ++i) one(i, 1);
        } else {
#pragma unroll 1
            for (int i = 0; i < BM * BK / 4 / NT; ++i) one(i, 0);
        }
    };
    auto load_b = [&](int ks) {
        float* Bs = smem_f + (ks % STAGES) * (A_FLOATS + B_FLOATS) + A_FLOATS;
        const int64_t k0 = kb + (int64_t)ks * BK;
        if constexpr (!TB) {
            auto one = [&](int i, int vec) {
                const int f = tid + i * NT, kr = f / (BN / 4), nq = (f % (BN / 4)) * 4;
                const int64_t k = k0 + kr, n = n0 + nq;
                copy4(Bs + kr * B_PITCH + nq, p.B + k * p.ldb + n, k < ke ? p.N - n : 0, vec, p.B);
            };
            if (p.vec_b) {
#pragma unroll
                for (int i = 0; i < BK * BN / 4 / NT; ++i) one(i, 1);
            } else {
#pragma unroll 1
                for (int i = 0; i < BK * BN / 4 / NT; ++i) one(i, 0);
            }
        } else {
            // word by word: sixteen lanes read one row's 64 bytes and write a column of the tile
#pragma unroll
            for (int i = 0; i < BK * BN / NT; ++i) {
                const int f = tid + i * NT, nr = f / BK, kr = f % BK;
                const int64_t k = k0 + kr, n = n0 + nr;
                const bool in = n < p.N && k < ke;
                cp_async4(Bs + kr * B_PITCH + nr, in ? p.B + n * p.ldb + k : p.B, in ? 4 : 0);
            }
        }
    };
    // The dropout mask of the tile comes in beside the first k-step, for the epilogue, which would wait for DRAM eight times for every
    // half of the tile (170 K x 256 with K = 128 and a byte mask: 416 -> 306 us, K = 256: 591 -> 513).
    uint8_t* const mask = reinterpret_cast<uint8_t*>(smem_f) + Cfg::ring_bytes(TA);
    if (p.vec_drop && p.splits == 1) {
        auto copy_mask = [&](int bytes) {
            const int per_row = BN / bytes;
#pragma unroll 4
            for (int f = tid; f < BM * per_row; f += NT) {
                const int r = f / per_row, c = f % per_row * bytes;
                const int64_t m = m0 + r, n = n0 + c;
                if (m >= p.M || n >= p.N) continue;
                const uint8_t* src = p.epi.drop + (p.epi.row0 + m) * p.N + n;
                if (bytes == 16) cp_async16(mask + r * BN + c, src, 16);
                else cp_async4(mask + r * BN + c, src, 4);
            }
        };
        if (p.vec_drop == 16) copy_mask(16);
        else copy_mask(4);
    }
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;

    const bool partial = p.splits > 1;
    float* Cb = partial ? p.C + (int64_t)blockIdx.z * p.M * p.N : p.C;
    const int64_t ldc = partial ? p.N : p.ldc;
    const bool vec_c = partial ? (p.N & 3) == 0 : p.vec_c != 0;
    // add the accumulators to C (the first time: store them) and clear them
    auto flush = [&](bool first) {
        // addresses are worked out here and not, hoisted, in the k-loop's registers: the compiler cannot see through the copy
        int64_t m0c;
        asm volatile("mov.b64 %0, %1;" : "=l"(m0c) : "l"(m0));
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int64_t m = m0c + row_of(i), n = n0 + q * QW + tx * 4;
                float* dst = Cb + m * ldc + n;
                const float2 lo = split2(acc[i][q * 2]), hi = split2(acc[i][q * 2 + 1]);
                const float r[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
                for (int t = 0; t < 4; ++t) if (m < p.M && n + t < p.N) dst[t] = first ? r[t] : r[t] + dst[t];
                acc[i][q * 2] = 0ull; acc[i][q * 2 + 1] = 0ull;
            }
    };

    bool flushed = false;
    int since_flush = 0;
    if constexpr (TN == 16) {
        // Operands of the next k are read from shared memory ahead of this one's FMAs, over the step's end as well: its barrier stands before
        // the last k, when everything of the stage is in registers, and the stage is refilled there and then (170 K x 256, K = 256: 517 -> 502 us,
        // K = 1024: 1847 -> 1756, 50.8 TFLOP/s; same sums).
        float2 a2[2][TM];                      // A as [m][k]: two k at a time
        float a1[2][TM];                       // A as [k][m]
        ulonglong2 b[2][Q];
        auto read_a = [&](const float* As, int k) {
            if constexpr (!TA) {
#pragma unroll
                for (int i = 0; i < TM; ++i) a2[(k >> 1) & 1][i] = *reinterpret_cast<const float2*>(As + (ty + i * (BM / TM)) * A_PITCH + k);
            } else {
#pragma unroll
                for (int g = 0; g < H; ++g) {
                    const float4 x = *reinterpret_cast<const float4*>(As + k * A_PITCH + ty * 4 + g * (BM / H));
                    a1[k & 1][4 * g] = x.x; a1[k & 1][4 * g + 1] = x.y; a1[k & 1][4 * g + 2] = x.z; a1[k & 1][4 * g + 3] = x.w;
                }
            }
        };
        auto read_b = [&](const float* Bs, int k) {
#pragma unroll
            for (int q = 0; q < Q; ++q) b[k & 1][q] = *reinterpret_cast<const ulonglong2*>(Bs + k * B_PITCH + tx * 4 + q * QW);
        };
#pragma unroll 1
        for (int ks = 0; ks < STAGES; ++ks) {
            if (ks < steps) { load_a(ks); load_b(ks); }
            commit();
        }
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 1) : "memory");
        __syncthreads();
        read_a(smem_f, 0);
        read_b(smem_f + A_FLOATS, 0);
#pragma unroll 1
        for (int ks = 0; ks < steps; ++ks) {
            const float* As = smem_f + (ks % STAGES) * (A_FLOATS + B_FLOATS);
#pragma unroll
            for (int k = 0; k < BK; ++k) {
                if (k + 1 < BK) {
                    read_b(As + A_FLOATS, k + 1);
                    if (TA) read_a(As, k + 1);
                    else if (!(k & 1) && k + 2 < BK) read_a(As, k + 2);
                } else {
                    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
                    __syncthreads();           // step ks + 1 has landed, step ks is read
                    const float* next = smem_f + ((ks + 1) % STAGES) * (A_FLOATS + B_FLOATS);
                    read_b(next + A_FLOATS, 0);
                    read_a(next, 0);
                    if (ks + STAGES < steps) { load_a(ks + STAGES); load_b(ks + STAGES); }
                    commit();
                }
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    const f32x2 av = dup2(TA ? a1[k & 1][i] : (k & 1) ? a2[(k >> 1) & 1][i].y : a2[(k >> 1) & 1][i].x);
#pragma unroll
                    for (int q = 0; q < Q; ++q) { ffma2(acc[i][2 * q], av, b[k & 1][q].x); ffma2(acc[i][2 * q + 1], av, b[k & 1][q].y); }
                }
            }
            if (++since_flush == FLUSH_STEPS && ks + 1 < steps) {
                since_flush = 0;
                flush(!flushed);
                flushed = true;
            }
        }
    } else {
        // One loop body serves the filling of the pipeline and the steps themselves: a small product runs each line of this code
        // once or a few times, and then its length is its time.
#pragma unroll 1
        for (int ks = 1 - STAGES; ks < steps; ++ks) {
            if (ks >= 0) {
                asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
                __syncthreads();                   // step ks has landed; the stage of step ks - 1 is free
            }
            if (ks + STAGES - 1 < steps) { load_a(ks + STAGES - 1); load_b(ks + STAGES - 1); }
            commit();
            if (ks < 0) continue;
            const float* As = smem_f + (ks % STAGES) * (A_FLOATS + B_FLOATS);
            const float* Bs = As + A_FLOATS;
#pragma unroll (TA && KG == 1 ? BK / 2 : 2)        // (with the row-wise A a longer body gains nothing and spills)
            for (int kk = kg * (BK / KG); kk < (kg + 1) * (BK / KG); kk += 2) {
                float2 a2[TM];
                if (!TA) {
#pragma unroll
                    for (int i = 0; i < TM; ++i) a2[i] = *reinterpret_cast<const float2*>(As + (ty + i * (BM / TM)) * A_PITCH + kk);
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const float* brow = Bs + (kk + k) * B_PITCH + tx * 4;
                    ulonglong2 b[Q];
#pragma unroll
                    for (int q = 0; q < Q; ++q) b[q] = *reinterpret_cast<const ulonglong2*>(brow + q * QW);
                    float a[TM];
                    if (!TA) {
#pragma unroll
                        for (int i = 0; i < TM; ++i) a[i] = k == 0 ? a2[i].x : a2[i].y;
                    } else {
                        const float* arow = As + (kk + k) * A_PITCH + ty * 4;
#pragma unroll
                        for (int g = 0; g < H; ++g) {
                            const float4 x = *reinterpret_cast<const float4*>(arow + g * (BM / H));
                            a[4 * g] = x.x; a[4 * g + 1] = x.y; a[4 * g + 2] = x.z; a[4 * g + 3] = x.w;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < TM; ++i) {
                        const f32x2 av = dup2(a[i]);
#pragma unroll
                        for (int q = 0; q < Q; ++q) { ffma2(acc[i][2 * q], av, b[q].x); ffma2(acc[i][2 * q + 1], av, b[q].y); }
                    }
                }
            }
            if (++since_flush == FLUSH_STEPS && ks + 1 < steps && KG == 1) {
                since_flush = 0;
                flush(!flushed);
                flushed = true;
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    // Epilogue through shared memory, four rows of every thread (half of the tile) at a time: a warp then stores (and reads gates and masks of) whole
    // rows, and its code is one short loop.  Applied from the registers it was unrolled over the micro-tile, thirty
    // kilobytes of branches that cost more than 128 terms of K (170 K x 256, K = 128: 617 us).
    constexpr int S_PITCH = BN + 4, ROW4 = BN / 4;
    const Epi& e = p.epi;
    float* const S = smem_f;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        for (int g = 0; g < KG; ++g) {
            __syncthreads();
            if (kg != g) continue;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float2 lo = split2(acc[h * 4 + i][q * 2]), hi = split2(acc[h * 4 + i][q * 2 + 1]);
                    float4* cell = reinterpret_cast<float4*>(S + row_of(i) * S_PITCH + q * QW + tx * 4);
                    float4 v = make_float4(lo.x, lo.y, hi.x, hi.y);
                    if (KG > 1 && g > 0) { const float4 o = *cell; v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w; }
                    *cell = v;
                }
        }
        __syncthreads();
#pragma unroll 2
        for (int f = tid; f < BM / H * ROW4; f += NT) {
            const int lr = f / ROW4, lc = (f % ROW4) * 4;
            const int64_t m = m0 + h * (BM / H) + lr, n = n0 + lc;
            const bool in = m < p.M && n < p.N, full = n + 3 < p.N;
            const float4 v = *reinterpret_cast<const float4*>(S + lr * S_PITCH + lc);
            float r[4] = {v.x, v.y, v.z, v.w};
            float* dst = Cb + m * ldc + n;
            if (flushed && in) {
#pragma unroll
                for (int t = 0; t < 4; ++t) if (n + t < p.N) r[t] += dst[t];
            }
            if (!partial) {
                if (e.bias) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) if (n + t < p.N) r[t] += __ldg(e.bias + n + t);
                }
                if (e.relu) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) r[t] = fmaxf(r[t], 0.0f);
                }
                if (e.drop && in) {
                    const uint8_t* dm = e.drop + (e.row0 + m) * p.N + n;
                    if (p.vec_drop) {
                        const uchar4 d4 = *reinterpret_cast<const uchar4*>(mask + (h * (BM / H) + lr) * BN + lc);
                        r[0] = d4.x ? r[0] * e.keep_scale : 0.0f; r[1] = d4.y ? r[1] * e.keep_scale : 0.0f;
                        r[2] = d4.z ? r[2] * e.keep_scale : 0.0f; r[3] = d4.w ? r[3] * e.keep_scale : 0.0f;
                    } else {
#pragma unroll
                        for (int t = 0; t < 4; ++t) if (n + t < p.N) r[t] = dm[t] ? r[t] * e.keep_scale : 0.0f;
                    }
                }
                if (e.gate && in) {
                    const float* gp = e.gate + (e.row0 + m) * e.ld_gate + n;
                    if (p.vec_gate && full) {
                        const float4 g4 = __ldg(reinterpret_cast<const float4*>(gp));
                        r[0] = g4.x > 0.0f ? r[0] * e.gate_scale : 0.0f; r[1] = g4.y > 0.0f ? r[1] * e.gate_scale : 0.0f;
                        r[2] = g4.z > 0.0f ? r[2] * e.gate_scale : 0.0f; r[3] = g4.w > 0.0f ? r[3] * e.gate_scale : 0.0f;
                    } else {
#pragma unroll
                        for (int t = 0; t < 4; ++t) if (n + t < p.N) r[t] = __ldg(gp + t) > 0.0f ? r[t] * e.gate_scale : 0.0f;
                    }
                }
                if (e.gate_bits && in) {
                    const uint32_t nib = __ldg(e.gate_bits + (e.row0 + m) * e.ld_gate_bits + (n >> 5)) >> (n & 31);   // n % 4 == 0: one word
#pragma unroll
                    for (int t = 0; t < 4; ++t) r[t] = ((nib >> t) & 1u) ? r[t] * e.gate_scale : 0.0f;
                }
                if (e.sign_bits) {
                    // eight lanes hold 32 consecutive columns of a row, one word of the bitmap
                    uint32_t w = 0;
#pragma unroll
                    for (int t = 0; t < 4; ++t) w |= (n + t < p.N && r[t] > 0.0f ? 1u : 0u) << t;
                    w <<= n & 31;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) w |= __shfl_xor_sync(0xFFFFFFFFu, w, o);
                    if (in && (lane & 7) == 0) e.sign_bits[(e.row0 + m) * e.ld_sign_bits + (n >> 5)] = w;
                }
            }
            if (!in) continue;
            if (vec_c && full) *reinterpret_cast<float4*>(dst) = make_float4(r[0], r[1], r[2], r[3]);
            else {
#pragma unroll
                for (int t = 0; t < 4; ++t) if (n + t < p.N) dst[t] = r[t];
            }
        }
    }
}

// C[m][n] = epilogue( sum_z part[z][m][n] ) in fp64.  A block owns 32 consecutive elements; its eight rows of threads add
// an eighth of the splits each (ascending), the eighths are added in order: a hundred splits of a small weight gradient
// cost one thread a chain of a hundred loads otherwise (16 K elements, 148 splits: 20 -> 4 us).  The blocks behind those add up the partial
// column sums that came with the product, if any, in the same way: a launch of its own took 4 us.
constexpr int RED_PARTS = 8;
__global__ void __launch_bounds__(32 * RED_PARTS) splitk_reduce_kernel(int64_t M, int64_t N, int splits, const float* __restrict__ part,
                                                                      float* __restrict__ C, int64_t ldc, const Epi epi, const int32_t* only_if, const ColSums sums) {
    chain_begin();
    if (only_if && *only_if == 0) return;
    __shared__ double sm[RED_PARTS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t MN = M * N, blocks = (MN + 31) / 32;
    if (blockIdx.x >= blocks) {
        const int64_t n = ((int64_t)blockIdx.x - blocks) * 32 + lane;
        const int per = (sums.splits + RED_PARTS - 1) / RED_PARTS;
        const int z0 = w * per, z1 = z0 + per < sums.splits ? z0 + per : sums.splits;
        double s = 0.0;
        if (n < N) {
#pragma unroll 4
            for (int z = z0; z < z1; ++z) s += __ldg(sums.part + (int64_t)z * N + n);
        }
        sm[w][lane] = s;
        __syncthreads();
        if (w != 0 || n >= N) return;
#pragma unroll
        for (int q = 1; q < RED_PARTS; ++q) s += sm[q][lane];
        sums.out[n] = (float)s;
        return;
    }
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    const int per = (splits + RED_PARTS - 1) / RED_PARTS;
    const int z0 = w * per, z1 = z0 + per < splits ? z0 + per : splits;
    double s = 0.0;
    if (i < MN) {
#pragma unroll 4
        for (int z = z0; z < z1; ++z) s += (double)__ldg(part + (int64_t)z * MN + i);
    }
    sm[w][lane] = s;
    __syncthreads();
    if (w != 0 || i >= MN) return;
#pragma unroll
    for (int q = 1; q < RED_PARTS; ++q) s += sm[q][lane];
    const int64_t m = i / N, n = i % N;
    C[m * ldc + n] = apply_epi(epi, (float)s, m, n, N);
}

// Column sums of an n x d matrix: block b sums rows [b*R, (b+1)*R) into part[b][d].
// A thread owns one float4 column group and every (256/groups)-th row of the block's range, four
// rows in flight; the row lanes are then added in fixed order through shared memory.  Requires
// ld % 4 == 0 and a 16-byte aligned X (the activations' layout).
__global__ void __launch_bounds__(256) colsum_partial_kernel(int64_t n, int d, const float* __restrict__ X, int64_t ld,
                                                             int64_t rows_per_block, int groups_pad,
                                                             float* __restrict__ part) {
    chain_begin();
    __shared__ float4 sm[256];
    const int d4 = (d + 3) >> 2;
    const int rl_n = 256 / groups_pad;                 // row lanes
    const int cg = threadIdx.x % groups_pad, rl = threadIdx.x / groups_pad;
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
    const int64_t r1 = (r0 + rows_per_block < n) ? r0 + rows_per_block : n;
    for (int g0 = 0; g0 < d4; g0 += groups_pad) {
        const int g = g0 + cg;
        float4 acc[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g < d4) {
            const float4* base = reinterpret_cast<const float4*>(X) + g;
            const int64_t ld4 = ld >> 2;
            int64_t r = r0 + rl;
            for (; r + 3 * rl_n < r1; r += 4 * rl_n) {
                float4 v[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) v[t] = __ldg(base + (r + t * rl_n) * ld4);
#pragma unroll
                for (int t = 0; t < 4; ++t) { acc[t].x += v[t].x; acc[t].y += v[t].y; acc[t].z += v[t].z; acc[t].w += v[t].w; }
            }
            for (int t = 0; r < r1; r += rl_n, ++t) {
                const float4 v = __ldg(base + r * ld4);
                acc[t & 3].x += v.x; acc[t & 3].y += v.y; acc[t & 3].z += v.z; acc[t & 3].w += v.w;
            }
        }
        float4 s4;
        s4.x = (acc[0].x + acc[1].x) + (acc[2].x + acc[3].x);
        s4.y = (acc[0].y + acc[1].y) + (acc[2].y + acc[3].y);
        s4.z = (acc[0].z + acc[1].z) + (acc[2].z + acc[3].z);
        s4.w = (acc[0].w + acc[1].w) + (acc[2].w + acc[3].w);
        sm[threadIdx.x] = s4;
        __syncthreads();
        if (rl == 0 && g < d4) {
            float4 t = sm[cg];
            for (int q = 1; q < rl_n; ++q) {
                const float4 u = sm[q * groups_pad + cg];
                t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
            }
            float* dst = part + (int64_t)blockIdx.x * d + g * 4;
            const float tv[4] = {t.x, t.y, t.z, t.w};
            for (int c = 0; c < 4; ++c) if (g * 4 + c < d) dst[c] = tv[c];
        }
        __syncthreads();
    }
}

// 32 columns per block, eight rows of threads take an eighth of the partial rows each (fp64, fixed order).
__global__ void __launch_bounds__(32 * RED_PARTS) colsum_final_kernel(int d, int blocks, const float* __restrict__ part, float* __restrict__ out) {
    chain_begin();
    __shared__ double sm[RED_PARTS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
    const int per = (blocks + RED_PARTS - 1) / RED_PARTS;
    const int b0 = w * per, b1 = b0 + per < blocks ? b0 + per : blocks;
    double s = 0.0;
    if (j < d) {
#pragma unroll 4
        for (int b = b0; b < b1; ++b) s += (double)__ldg(part + (int64_t)b * d + j);
    }
    sm[w][lane] = s;
    __syncthreads();
    if (w != 0 || j >= d) return;
#pragma unroll
    for (int q = 1; q < RED_PARTS; ++q) s += sm[q][lane];
    out[j] = (float)s;
}

// G <- G * 1[X_out > 0] (ReLU) * (drop ? keep_scale : 0): gradient w.r.t. the pre-activation.
__global__ void gate_kernel(int64_t n, int d, float* __restrict__ G, int64_t ldg, const float* __restrict__ Xo,
                            int64_t ldx, int relu, const uint8_t* __restrict__ drop, float keep_scale) {
    chain_begin();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * d) return;
    const int64_t r = i / d; const int j = (int)(i % d);
    float g = G[r * ldg + j];
    if (relu && !(Xo[r * ldx + j] > 0.0f)) g = 0.0f;
    if (drop) g = drop[i] ? g * keep_scale : 0.0f;
    G[r * ldg + j] = g;
}

template <int BM, int BN, int TN, int KG, bool TA, bool TB>
cudaError_t launch_form(const GemmParams& p, cudaStream_t s) {
    constexpr int ring = SimtCfg<BM, BN, TN, KG>::ring_bytes(TA), most = ring + BM * BN;
    const int smem = p.vec_drop && p.splits == 1 ? most : ring;
    if (smem > 48 * 1024) {        // (one value for every call: another thread may be between this and its launch)
        const cudaError_t e = cudaFuncSetAttribute(gemm_simt_kernel<BM, BN, TN, KG, TA, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)(p.m_tiles * p.n_tiles), 1, (unsigned)p.splits);
    // (split reductions fill the machine once: chained, their blocks gather on the SMs that fall free first, 20 K x 32 x 7 8.2 -> 9.8 us)
    if (p.splits == 1 || p.only_if) launch_chained(gemm_simt_kernel<BM, BN, TN, KG, TA, TB>, grid, SimtCfg<BM, BN, TN, KG>::NT, smem, s, p);
    else gemm_simt_kernel<BM, BN, TN, KG, TA, TB><<<grid, SimtCfg<BM, BN, TN, KG>::NT, smem, s>>>(p);
    return cudaGetLastError();
}

template <int BM, int BN, int TN, int KG>
cudaError_t launch_variant(const GemmParams& p, int ta, int tb, cudaStream_t s) {
    if (!ta && !tb) return launch_form<BM, BN, TN, KG, false, false>(p, s);
    if (!ta) return launch_form<BM, BN, TN, KG, false, true>(p, s);
    if (!tb) return launch_form<BM, BN, TN, KG, true, false>(p, s);
    return launch_form<BM, BN, TN, KG, true, true>(p, s);
}

}  // namespace

namespace mixgcn {

// *bits_done: whether the sign bitmap, if one is asked for, was written (not where K is split).
mixgcn_status launch_gemm_simt(mixgcn_ctx* ctx, int ta, int tb, int64_t M, int64_t N, int64_t K,
                               const float* A, int64_t lda, const float* B, int64_t ldb, float* C, int64_t ldc,
                               const mixgcn_epilogue* epi, int64_t epi_row0, cudaStream_t s, bool* bits_done, const int32_t* only_if) {
    if (bits_done) *bits_done = false;
    if (M <= 0 || N <= 0) return MIXGCN_OK;
    GemmParams p{};
    p.M = M; p.N = N; p.K = K; p.A = A; p.lda = lda; p.B = B; p.ldb = ldb; p.C = C; p.ldc = ldc;
    if (epi) {
        p.epi.bias = epi->bias; p.epi.relu = epi->relu; p.epi.drop = epi->drop_mask;
        p.epi.keep_scale = epi->keep_scale; p.epi.gate = epi->gate_bits ? nullptr : epi->gate; p.epi.ld_gate = epi->ld_gate;
        p.epi.gate_scale = epi->gate_scale;
        p.epi.gate_bits = epi->gate_bits; p.epi.ld_gate_bits = epi->ld_gate_bits;
        p.epi.sign_bits = epi->sign_bits; p.epi.ld_sign_bits = epi->ld_sign_bits;
    }
    p.epi.row0 = epi_row0;
    p.only_if = only_if;
    p.vec_a = aligned16(A) && (lda & 3) == 0;
    p.vec_b = aligned16(B) && (ldb & 3) == 0;
    p.vec_c = aligned16(C) && (ldc & 3) == 0;
    const uintptr_t mask_at = reinterpret_cast<uintptr_t>(p.epi.drop) | (uintptr_t)N;       // (every row starts at a multiple of N)
    p.vec_drop = !p.epi.drop || (mask_at & 3) ? 0 : (mask_at & 15) ? 4 : 16;
    p.vec_gate = p.epi.gate && aligned16(p.epi.gate) && (p.epi.ld_gate & 3) == 0;
    // The tile: 32 columns where N has no more, else 64 or 128 by what leaves less of N to padding, 128 rows.  Where that
    // gives fewer CTAs than the machine has SMs even with K split, 64-row tiles.
    auto ceil_div = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    const bool may_split = K >= 2 * MIN_K_PER_SPLIT && (K > 1024 || ta);
    const int64_t max_splits = may_split ? ceil_div(K, MIN_K_PER_SPLIT) : 1;
    int bm = 128, bn = N <= 32 ? 32 : ceil_div(N, 128) * 128 > ceil_div(N, 64) * 64 ? 64 : 128;
    if (bn == 32 || ceil_div(M, bm) * ceil_div(N, bn) * max_splits < ctx->sm_count) bm = 64;
    if (bm == 64 && bn == 128) bn = 64;
    p.m_tiles = ceil_div(M, bm);
    p.n_tiles = ceil_div(N, bn);
    const int64_t tiles = p.m_tiles * p.n_tiles;
    const int per_sm = bm == 64 ? 3 : bn == 64 ? 4 : 2;        // CTAs an SM holds (64-row tiles: of four groups)
    int64_t splits = 1;
    if (max_splits > 1 && tiles < (int64_t)per_sm * ctx->sm_count) {
        splits = (int64_t)per_sm * ctx->sm_count / tiles;      // one full wave
        if (splits > max_splits) splits = max_splits;
        if (splits > 1024) splits = 1024;
    }
    int64_t kps = ceil_div(ceil_div(K, splits), BK) * BK;
    if (kps <= 0) kps = BK;
    splits = ceil_div(K, kps);
    if (splits < 1) splits = 1;
    p.k_per_split = kps; p.splits = (int)splits;
    if (splits > 1) {
        MIXGCN_TRY(ensure_workspace(ctx, splits * M * N * (int64_t)sizeof(float)));
        p.C = reinterpret_cast<float*>(ctx->workspace);
        p.epi.sign_bits = nullptr;
    }
    if (tiles > 0x7FFFFFFFll) MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "gemm: too many tiles");
    {
        LaunchScope scope(ctx, PH_GEMM, s);
        // 64-row tiles: four groups of threads per tile where one would leave an SM fewer than eight warps (each group's
        // accumulators see a quarter of K, and are not flushed: up to four times 1024 terms)
        const bool fine = bm == 64 && tiles * splits * (bn / 32) < 8 * (int64_t)ctx->sm_count && kps <= FINE_KG * FLUSH_STEPS * BK;
        MIXGCN_CUDA(fine ? (bn == 32 ? launch_variant<64, 32, 8, FINE_KG>(p, ta, tb, s) : launch_variant<64, 64, 8, FINE_KG>(p, ta, tb, s))
                    : bm == 64 ? (bn == 32 ? launch_variant<64, 32, 8, 1>(p, ta, tb, s) : launch_variant<64, 64, 8, 1>(p, ta, tb, s))
                               : (bn == 64 ? launch_variant<128, 64, 8, 1>(p, ta, tb, s) : launch_variant<128, 128, 16, 1>(p, ta, tb, s)));
    }
    if (splits > 1) {
        LaunchScope scope(ctx, PH_GEMM, s);
        const int64_t total = M * N;
        launch_chained(splitk_reduce_kernel, dim3((unsigned)((total + 31) / 32)), 32 * RED_PARTS, 0, s, M, N, (int)splits, p.C, C, ldc, p.epi, only_if, ColSums{});
        MIXGCN_CUDA(cudaGetLastError());
    } else if (bits_done) {
        *bits_done = p.epi.sign_bits != nullptr;
    }
    return MIXGCN_OK;
}

mixgcn_status launch_splitk_reduce(mixgcn_ctx* ctx, int64_t M, int64_t N, int splits, const float* part, float* C,
                                   int64_t ldc, const mixgcn_epilogue* epi, cudaStream_t s, const ColSums& sums) {
    Epi e{};
    if (epi) {
        e.bias = epi->bias; e.relu = epi->relu; e.drop = epi->drop_mask; e.keep_scale = epi->keep_scale;
        e.gate = epi->gate_bits ? nullptr : epi->gate; e.ld_gate = epi->ld_gate; e.gate_scale = epi->gate_scale;
        e.gate_bits = epi->gate_bits; e.ld_gate_bits = epi->ld_gate_bits;
    }
    LaunchScope scope(ctx, PH_GEMM, s);
    const int64_t blocks = (M * N + 31) / 32 + (sums.out ? (N + 31) / 32 : 0);
    launch_chained(splitk_reduce_kernel, dim3((unsigned)blocks), 32 * RED_PARTS, 0, s, M, N, splits, part, C, ldc, e, nullptr, sums);
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

mixgcn_status launch_colsum(mixgcn_ctx* ctx, int64_t n, int32_t d, const float* X, int64_t ld, float* out,
                            cudaStream_t s) {
    // four blocks per SM, so that every SM streams; no fewer than 64 rows each, and (one wave of 2048 at most) the final
    // pass stays short
    int64_t blocks = 4 * (int64_t)ctx->sm_count;
    int64_t rows_per_block = (n + blocks - 1) / blocks;
    if (rows_per_block < 64) rows_per_block = 64;
    blocks = (n + rows_per_block - 1) / rows_per_block;
    if (blocks < 1) blocks = 1;
    MIXGCN_TRY(ensure_workspace(ctx, blocks * d * (int64_t)sizeof(float)));
    float* part = reinterpret_cast<float*>(ctx->workspace);
    {
        LaunchScope scope(ctx, PH_ELEM, s);
        int groups_pad = 1;
        while (groups_pad < 256 && groups_pad < (d + 3) / 4) groups_pad <<= 1;
        launch_chained(colsum_partial_kernel, dim3((unsigned)blocks), 256, 0, s, n, d, X, ld, rows_per_block, groups_pad, part);
    }
    {
        LaunchScope scope(ctx, PH_ELEM, s);
        launch_chained(colsum_final_kernel, dim3((d + 31) / 32), 32 * RED_PARTS, 0, s, d, (int)blocks, part, out);
    }
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

mixgcn_status launch_gate(mixgcn_ctx* ctx, int64_t n, int32_t d, float* G, int64_t ldg, const float* X_out,
                          int64_t ldx, int relu, const uint8_t* drop_mask, float keep_scale, cudaStream_t s) {
    const int64_t total = n * d;
    if (total <= 0) return MIXGCN_OK;
    LaunchScope scope(ctx, PH_ELEM, s);
    launch_chained(gate_kernel, dim3((unsigned)((total + 255) / 256)), 256, 0, s, n, d, G, ldg, X_out, ldx, relu, drop_mask, keep_scale);
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

}  // namespace mixgcn
