// The epilogue of a dense product in registers, shared by the tensor-core kernels: bias, ReLU, dropout mask, gate, sign bitmap
// and bf16 copy of 32 columns of one row at a time.
#pragma once
#include <cuda.h>

#include "internal.cuh"
#include "tc_ptx.cuh"

namespace mixgcn {
namespace tc {

// 2-D tensor map of fp32 (eb = 4) or bf16 (eb = 2) words, defined in gemm_tc.cu
bool encode_2d(CUtensorMap* map, const void* base, int eb, int64_t inner, int64_t outer, int64_t ld, int box_inner,
               int box_outer, CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B);

struct TcEpi {
    const float* bias; int relu;
    const uint8_t* drop; float keep_scale;
    const float* gate; int64_t ld_gate; float gate_scale;
    const uint32_t* gate_bits; int64_t ld_gate_bits;   // bit-packed gate (replaces `gate`): bit j & 31 of word j >> 5 of row i
    uint32_t* sign_bits; int64_t ld_sign_bits;         // output: bit = (final y > 0), written by the K-major kernels' epilogues
    int64_t row0;
};

inline TcEpi make_tc_epi(const mixgcn_epilogue* epi, int64_t row0) {
    TcEpi e{};
    if (epi) {
        e.bias = epi->bias; e.relu = epi->relu; e.drop = epi->drop_mask; e.keep_scale = epi->keep_scale;
        e.gate = epi->gate_bits ? nullptr : epi->gate; e.ld_gate = epi->ld_gate; e.gate_scale = epi->gate_scale;
        e.gate_bits = epi->gate_bits; e.ld_gate_bits = epi->ld_gate_bits;
        e.sign_bits = epi->sign_bits; e.ld_sign_bits = epi->ld_sign_bits;
    }
    e.row0 = row0;
    return e;
}

__device__ __forceinline__ float tc_apply_epi(const TcEpi& e, float y, int64_t m, int64_t n, int64_t N) {
    if (e.bias) y += e.bias[n];
    if (e.relu) y = fmaxf(y, 0.0f);
    if (e.drop) y = e.drop[(e.row0 + m) * N + n] ? y * e.keep_scale : 0.0f;
    if (e.gate) y = e.gate[(e.row0 + m) * e.ld_gate + n] > 0.0f ? y * e.gate_scale : 0.0f;
    if (e.gate_bits) y = ((e.gate_bits[(e.row0 + m) * e.ld_gate_bits + (n >> 5)] >> (n & 31)) & 1u) ? y * e.gate_scale : 0.0f;
    return y;
}

// bit q = (v[q] > 0) for the columns nb + q < N of one row's 32-column chunk
__device__ __forceinline__ uint32_t sign_word(const float (&v)[32], int64_t nb, int64_t N) {
    uint32_t w = 0;
#pragma unroll
    for (int q = 0; q < 32; ++q) w |= (v[q] > 0.0f ? 1u : 0u) << q;
    const int64_t left = N - nb;
    return left >= 32 ? w : (w & ((1u << (int)left) - 1u));
}

__device__ __forceinline__ bool aligned16_dev(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// 32 consecutive columns of one row as bf16 (round to nearest even); dst is 16-byte aligned when full.
__device__ __forceinline__ void store_lp_row(uint16_t* dst, const float (&v)[32], int valid) {
    if (valid >= 32) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            reinterpret_cast<uint4*>(dst)[q] = make_uint4(pack_bf16(v[8 * q], v[8 * q + 1]), pack_bf16(v[8 * q + 2], v[8 * q + 3]),
                                                           pack_bf16(v[8 * q + 4], v[8 * q + 5]), pack_bf16(v[8 * q + 6], v[8 * q + 7]));
    } else {
#pragma unroll
        for (int q = 0; q < 32; ++q)
            if (q < valid) dst[q] = (uint16_t)(pack_bf16(v[q], 0.0f) & 0xFFFFu);
    }
}

// ---- per-element masks of a tile's epilogue ----
// An epilogue thread owns a row of the accumulator and wants a dropout mask or gate as one word per 32 columns.  The words
// are made while the accumulator still is: bytes and fp32 gates are read with coalesced requests (a row's 32 columns by
// eight adjacent lanes), reduced to four bits per load, and brought to the row's lane by an 8 x 8 transpose of nibbles.
// (Applied to the staged output box instead, with a dependent byte load per element, a dropout product took three to four
// times as long: 180 K x 128 x 128: 136 us.)

// Lane (g, c) = (lane / 8, lane % 8) holds in nibble i the columns 4 c .. 4 c + 3 of row 4 i + g; returns the word of row `lane`.
__device__ __forceinline__ uint32_t row_word_from_nibbles(uint32_t x, int lane) {
    uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, 4);
    x = (lane & 4) ? (x & 0xFFFF0000u) | (y >> 16) : (x & 0x0000FFFFu) | (y << 16);
    y = __shfl_xor_sync(0xFFFFFFFFu, x, 2);
    x = (lane & 2) ? (x & 0xFF00FF00u) | ((y >> 8) & 0x00FF00FFu) : (x & 0x00FF00FFu) | ((y << 8) & 0xFF00FF00u);
    y = __shfl_xor_sync(0xFFFFFFFFu, x, 1);
    x = (lane & 1) ? (x & 0xF0F0F0F0u) | ((y >> 4) & 0x0F0F0F0Fu) : (x & 0x0F0F0F0Fu) | ((y << 4) & 0xF0F0F0F0u);
    return __shfl_sync(0xFFFFFFFFu, x, (lane & 3) * 8 + (lane >> 2));      // row 4 i + g now lies in lane (g, i)
}

// Words of the 32 rows from `row_first`, columns nb, nb + step, ... (CHUNKS blocks of 32), for this lane's row.
template <int CHUNKS>
__device__ __forceinline__ void mask_words(const TcEpi& e, int64_t row_first, int64_t M, int64_t N, int nb, int step, int nb_end, int lane,
                                           uint32_t (&dw)[CHUNKS], uint32_t (&gw)[CHUNKS]) {
    const int g = lane >> 3, c = lane & 7;
#pragma unroll
    for (int k = 0; k < CHUNKS; ++k) { dw[k] = 0xFFFFFFFFu; gw[k] = 0xFFFFFFFFu; }
    if (nb_end > N) nb_end = (int)N;
    if (e.drop) {
        if ((N & 3) == 0 && (reinterpret_cast<uintptr_t>(e.drop) & 3) == 0) {
            uint32_t x[CHUNKS][8];                       // every block's loads in flight together
#pragma unroll
            for (int k = 0; k < CHUNKS; ++k)
#pragma unroll
                for (int it = 0; it < 8; ++it) {
                    const int64_t row = row_first + it * 4 + g;
                    const int n = nb + k * step + c * 4;
                    x[k][it] = (row < M && n < nb_end) ? __ldg(reinterpret_cast<const uint32_t*>(e.drop + (e.row0 + row) * N + n)) : 0u;
                }
#pragma unroll
            for (int k = 0; k < CHUNKS; ++k) {
                if (nb + k * step >= nb_end) break;
                uint32_t nibbles = 0;
#pragma unroll
                for (int it = 0; it < 8; ++it) nibbles |= (((__vcmpne4(x[k][it], 0u) & 0x08040201u) * 0x01010101u) >> 24) << (4 * it);
                dw[k] = row_word_from_nibbles(nibbles, lane);
            }
        } else {
            // Rows that start at any byte: a lane's four bytes from the two aligned words they lie in (982 K x 63 x 91, fp32:
            // 605 us with one request and one vote per row, 396 so).  The second word only where it begins inside the mask.
            const uintptr_t end = reinterpret_cast<uintptr_t>(e.drop + (e.row0 + M) * N);
#pragma unroll
            for (int k = 0; k < CHUNKS; ++k) {
                const int left = nb_end - (nb + k * step);
                if (left <= 0) break;
                uint32_t x[8], y[8], shift[8];
#pragma unroll
                for (int it = 0; it < 8; ++it) {
                    const int64_t row = row_first + it * 4 + g;
                    const uintptr_t at = reinterpret_cast<uintptr_t>(e.drop + (e.row0 + row) * N + nb + k * step + c * 4), word = at & ~(uintptr_t)3;
                    const bool in = row < M && c * 4 < left;
                    shift[it] = (uint32_t)(at & 3) * 8;
                    x[it] = in ? __ldg(reinterpret_cast<const uint32_t*>(word)) : 0u;
                    y[it] = in && shift[it] && word + 4 < end ? __ldg(reinterpret_cast<const uint32_t*>(word + 4)) : 0u;
                }
                uint32_t nibbles = 0;
#pragma unroll
                for (int it = 0; it < 8; ++it)
                    nibbles |= (((__vcmpne4(__funnelshift_r(x[it], y[it], shift[it]), 0u) & 0x08040201u) * 0x01010101u) >> 24) << (4 * it);
                dw[k] = row_word_from_nibbles(nibbles, lane) & (left < 32 ? (1u << left) - 1u : 0xFFFFFFFFu);
            }
        }
    }
    if (e.gate_bits) {
#pragma unroll
        for (int k = 0; k < CHUNKS; ++k)
            if (nb + k * step < nb_end) gw[k] = row_first + lane < M ? __ldg(e.gate_bits + (e.row0 + row_first + lane) * e.ld_gate_bits + ((nb + k * step) >> 5)) : 0u;
    } else if (e.gate) {
        const bool vec = aligned16_dev(e.gate) && (e.ld_gate & 3) == 0;
#pragma unroll
        for (int k = 0; k < CHUNKS; ++k) {
            if (nb + k * step >= nb_end) break;
            float4 x[8];
#pragma unroll
            for (int it = 0; it < 8; ++it) {
                const int64_t row = row_first + it * 4 + g;
                const int n = nb + k * step + c * 4;
                x[it] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row < M && n < nb_end) {
                    const float* src = e.gate + (e.row0 + row) * e.ld_gate + n;
                    if (vec) x[it] = __ldg(reinterpret_cast<const float4*>(src));      // inside the row's allocation: ld_gate % 4 == 0
                    else {
                        x[it].x = __ldg(src);
                        if (n + 1 < nb_end) x[it].y = __ldg(src + 1);
                        if (n + 2 < nb_end) x[it].z = __ldg(src + 2);
                        if (n + 3 < nb_end) x[it].w = __ldg(src + 3);
                    }
                }
            }
            uint32_t nibbles = 0;
#pragma unroll
            for (int it = 0; it < 8; ++it)
                nibbles |= ((x[it].x > 0.0f ? 1u : 0u) | (x[it].y > 0.0f ? 2u : 0u) | (x[it].z > 0.0f ? 4u : 0u) | (x[it].w > 0.0f ? 8u : 0u)) << (4 * it);
            gw[k] = row_word_from_nibbles(nibbles, lane);
        }
    }
}

// Bias (from shared memory, or global where `bias_smem` is null), ReLU, dropout and gate on 32 columns of one row.
__device__ __forceinline__ void chunk_epilogue(const TcEpi& e, float (&v)[32], int nb, int64_t N, const float* bias_smem, uint32_t dw, uint32_t gw) {
    if (e.bias) {
        if (bias_smem || (aligned16_dev(e.bias) && nb + 31 < N)) {
            const float4* b4 = reinterpret_cast<const float4*>((bias_smem ? bias_smem : e.bias) + nb);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 b = bias_smem ? b4[q] : __ldg(b4 + q);
                v[4 * q] += b.x; v[4 * q + 1] += b.y; v[4 * q + 2] += b.z; v[4 * q + 3] += b.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 32; ++q)
                if (nb + q < N) v[q] += __ldg(e.bias + nb + q);
        }
    }
    if (e.relu) {
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = fmaxf(v[q], 0.0f);
    }
    if (e.drop) {
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = (dw >> q) & 1u ? v[q] * e.keep_scale : 0.0f;
    }
    if (e.gate_bits || e.gate) {
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = (gw >> q) & 1u ? v[q] * e.gate_scale : 0.0f;
    }
}

}  // namespace tc
}  // namespace mixgcn
