// Masked softmax cross-entropy with its gradient and arg-max (the loss line of Algorithm 2),
// and the Adam step (its weight-update line).  Both are streaming kernels; floating-point
// reductions run in a fixed order (per-warp shuffles, per-CTA partials, one final pass).
#include <stddef.h>

#include <atomic>

#include "internal.cuh"

using namespace mixgcn;

namespace {

constexpr int LOSS_WARPS = 8;

// number of non-zero bytes among four
__device__ __forceinline__ unsigned nonzero_bytes(uint32_t x) { return __popc(__vcmpne4(x, 0u)) >> 3; }

// Train nodes of the mask; integers, so the order of the atomics does not matter.  Sixteen mask bytes per load where the
// mask is aligned (2.4 M nodes: 6.5 -> 2.5 us).
__global__ void __launch_bounds__(256) count_mask_kernel(int64_t n, const uint8_t* __restrict__ mask, unsigned long long* count) {
    chain_begin();
    __shared__ unsigned int sm[8];
    unsigned int c = 0;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    const int64_t n16 = (reinterpret_cast<uintptr_t>(mask) & 15u) == 0 ? n >> 4 : 0;
    for (int64_t i = t0; i < n16; i += step) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(mask) + i);
        c += nonzero_bytes(v.x) + nonzero_bytes(v.y) + nonzero_bytes(v.z) + nonzero_bytes(v.w);
    }
    for (int64_t i = n16 * 16 + t0; i < n; i += step) c += mask[i] ? 1u : 0u;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xFFFFFFFFu, c, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int t = 0;
        for (int w = 0; w < 8; ++w) t += sm[w];
        if (t) atomicAdd(count, (unsigned long long)t);
    }
}

// The same in one block, which also clears what the loss kernels count up (`clear`: nullable): one launch instead of a
// clear or two and a count.
constexpr int64_t COUNT_ONE_BLOCK_MAX = 1 << 17;
__global__ void __launch_bounds__(1024) count_mask_small_kernel(int64_t n, const uint8_t* __restrict__ mask, unsigned long long* count,
                                                               unsigned int* done, unsigned long long* clear) {
    chain_begin();
    __shared__ unsigned int sm[32];
    unsigned int c = 0;
    const int64_t n16 = (reinterpret_cast<uintptr_t>(mask) & 15u) == 0 ? n >> 4 : 0;
    for (int64_t i = threadIdx.x; i < n16; i += 1024) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(mask) + i);
        c += nonzero_bytes(v.x) + nonzero_bytes(v.y) + nonzero_bytes(v.z) + nonzero_bytes(v.w);
    }
    for (int64_t i = n16 * 16 + threadIdx.x; i < n; i += 1024) c += mask[i] ? 1u : 0u;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xFFFFFFFFu, c, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x < 32) {
        c = sm[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xFFFFFFFFu, c, o);
        if (threadIdx.x == 0) {
            *count = c;
            *done = 0;
            if (clear) *clear = 0;
        }
    }
}

// A few words, in the chain of launches (a memset between two kernels takes 5 us from the one's end to the other's start).
__global__ void __launch_bounds__(32) clear_kernel(uint32_t* words, int n_words, int64_t* also) {
    chain_begin();
    if ((int)threadIdx.x < n_words) words[threadIdx.x] = 0;
    if (threadIdx.x == 0 && also) *also = 0;
}

// Sum of `blocks` partials by one block of `threads` threads, in a fixed order: thread t takes t, t + threads, ..., then a
// tree.  Valid in thread 0.
template <int THREADS>
__device__ __forceinline__ double sum_partials(const double* __restrict__ part, int blocks, double* sm) {
    double t = 0.0;
    for (int b = threadIdx.x; b < blocks; b += THREADS) t += part[b];
    sm[threadIdx.x] = t;
    __syncthreads();
    for (int half = THREADS / 2; half > 0; half >>= 1) {
        if (threadIdx.x < half) sm[threadIdx.x] += sm[threadIdx.x + half];
        __syncthreads();
    }
    return sm[0];
}

// One warp per row.  part[block] receives the block's sum of per-row losses.
__global__ void __launch_bounds__(LOSS_WARPS * 32) loss_rows_kernel(
    int64_t n, int C, const float* logits, int64_t ld, const int32_t* __restrict__ labels,
    const uint8_t* __restrict__ mask, const unsigned long long* __restrict__ count, float* dlogits,
    int32_t* __restrict__ pred, unsigned long long* n_correct, double* __restrict__ part, int32_t* status, bool zero_rows) {
    chain_begin();
    __shared__ double sm[LOSS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long T = *count;
    const float invT = T ? (float)(1.0 / (double)T) : 0.0f;
    double local = 0.0;
    unsigned int correct = 0;
    const int64_t stride = (int64_t)gridDim.x * LOSS_WARPS;
    for (int64_t v = (int64_t)blockIdx.x * LOSS_WARPS + warp; v < n; v += stride) {
        const float* row = logits + v * ld;
        // arg-max with lowest-index ties
        float mx = -INFINITY; int arg = 0x7FFFFFFF;
        for (int c = lane; c < C; c += 32) {
            const float x = row[c];
            if (x > mx || (x == mx && c < arg)) { mx = x; arg = c; }
        }
        if (arg == 0x7FFFFFFF) arg = lane < C ? lane : 0;  // all -inf or NaN in this lane's columns
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float omx = __shfl_xor_sync(0xFFFFFFFFu, mx, o);
            const int oarg = __shfl_xor_sync(0xFFFFFFFFu, arg, o);
            if (omx > mx || (omx == mx && oarg < arg)) { mx = omx; arg = oarg; }
        }
        if (pred && lane == 0) pred[v] = arg;
        const bool train = mask[v] != 0 && T != 0;
        int y = 0;
        bool ok = false;
        if (train) {
            y = labels[v];
            ok = y >= 0 && y < C;
            if (!ok && lane == 0) atomicMax(status, DEV_BAD_LABEL);
        }
        if (!train || !ok) {
            if (dlogits && (zero_rows || train)) for (int c = lane; c < C; c += 32) dlogits[v * ld + c] = 0.0f;
            continue;
        }
        float s = 0.0f;
        for (int c = lane; c < C; c += 32) s += expf(row[c] - mx);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        const float lse = mx + logf(s), share = 1.0f / s;
        const float py = row[y];
        if (lane == 0) { local += (double)(lse - py); if (arg == y) ++correct; }
        __syncwarp();  // dlogits may alias logits: every read of the row precedes the writes
        if (dlogits)
            for (int c = lane; c < C; c += 32) {
                const float g = (expf(row[c] - mx) * share - (c == y ? 1.0f : 0.0f)) * invT;
                dlogits[v * ld + c] = g;
            }
    }
    if (lane == 0) sm[warp] = local;
    if (n_correct && lane == 0 && correct) atomicAdd(n_correct, (unsigned long long)correct);
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < LOSS_WARPS; ++w) t += sm[w];
        part[blockIdx.x] = t;
    }
}

// Same computation for C <= 4 * LPR * VPL with the row held in registers: LPR lanes take a row (32 / LPR rows a warp), VPL
// float4-vectorised reads of the logits and writes of the gradient a lane (requires ld % 4 == 0 and 16-byte aligned pointers).
// The next rows' logits, mask bytes and labels are requested before the current ones are reduced.  Bound: instructions, so lanes are few and
// their columns many (a row's shuffles serve 32 / LPR rows at once), the arg-max is looked up behind the maximum, and the exponentials of
// the sum, over the sum, are the gradient's (as exp(x - log-sum-exp), with twice as many: 400 K x 47, 30 % in the mask, 71 us, now 47).
template <int LPR, int VPL>
__global__ void __launch_bounds__(LOSS_WARPS * 32) loss_rows_vec_kernel(
    int64_t n, int C, const float* logits, int64_t ld, const int32_t* __restrict__ labels,
    const uint8_t* __restrict__ mask, const unsigned long long* __restrict__ count, float* dlogits,
    int32_t* __restrict__ pred, unsigned long long* n_correct, double* __restrict__ part, int32_t* status, bool zero_rows) {
    chain_begin();
    constexpr int ROWS = 32 / LPR;
    __shared__ double sm[LOSS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lig = lane % LPR, sub = lane / LPR;
    const unsigned long long T = *count;
    const float invT = T ? (float)(1.0 / (double)T) : 0.0f;
    const int C4 = (C + 3) >> 2;
    double local = 0.0;
    unsigned int correct = 0;
    const int64_t stride = (int64_t)gridDim.x * LOSS_WARPS * ROWS;
    float4 nxt[VPL];
    uint8_t nxt_mask = 0; int nxt_y = 0;
    auto load_row = [&](int64_t v) {
        const float4* row4 = reinterpret_cast<const float4*>(logits + v * ld);
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            const int g = lig + LPR * q;
            nxt[q] = (v < n && g < C4) ? row4[g] : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
        if (v < n) { nxt_mask = mask[v]; nxt_y = labels[v]; }
    };
    int64_t v0 = ((int64_t)blockIdx.x * LOSS_WARPS + warp) * ROWS;
    load_row(v0 + sub);
    for (; v0 < n; v0 += stride) {                                 // (the whole warp together)
        const int64_t v = v0 + sub;
        const bool in = v < n;
        float x[VPL][4];
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            const int g = lig + LPR * q;
            x[q][0] = nxt[q].x; x[q][1] = nxt[q].y; x[q][2] = nxt[q].z; x[q][3] = nxt[q].w;
#pragma unroll
            for (int e = 0; e < 4; ++e) if (g * 4 + e >= C) x[q][e] = -INFINITY;   // pad columns are not data
        }
        const bool train = in && nxt_mask != 0 && T != 0;
        const int y = nxt_y;
        load_row(v + stride);
        float mx = -INFINITY;
#pragma unroll
        for (int q = 0; q < VPL; ++q) mx = fmaxf(mx, fmaxf(fmaxf(x[q][0], x[q][1]), fmaxf(x[q][2], x[q][3])));      // (no NaN among them)
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
        // the lowest column that attains it
        int arg = 0x7FFFFFFF;
#pragma unroll
        for (int q = VPL - 1; q >= 0; --q)
#pragma unroll
            for (int e = 3; e >= 0; --e) {
                const int c = (lig + LPR * q) * 4 + e;
                if (x[q][e] == mx && c < C) arg = c;
            }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) arg = min(arg, __shfl_xor_sync(0xFFFFFFFFu, arg, o));
        if (arg == 0x7FFFFFFF) arg = 0;                            // NaN everywhere
        if (pred && in && lig == 0) pred[v] = arg;
        const bool ok = train && y >= 0 && y < C;
        if (train && !ok && lig == 0) atomicMax(status, DEV_BAD_LABEL);
        if (!__any_sync(0xFFFFFFFFu, ok)) {
            if (dlogits && in && (zero_rows || train)) {
#pragma unroll
                for (int q = 0; q < VPL; ++q)
                    if (lig + LPR * q < C4) reinterpret_cast<float4*>(dlogits + v * ld)[lig + LPR * q] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            continue;
        }
        float s = 0.0f, py = 0.0f;
        // the label's logit lives in lane (y/4) % LPR of the row, slot (y/4) / LPR, element y % 4
#pragma unroll
        for (int q = 0; q < VPL; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = (lig + LPR * q) * 4 + e;
                if (c == y) py = x[q][e];
                x[q][e] = c < C ? expf(x[q][e] - mx) : 0.0f;
                s += x[q][e];
            }
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        py = __shfl_sync(0xFFFFFFFFu, py, (y >> 2) & (LPR - 1), LPR);
        if (ok && lig == 0) { local += (double)(mx + logf(s) - py); if (arg == y) ++correct; }
        if (!dlogits || !in || !(ok || zero_rows || train)) continue;
        const float share = 1.0f / s;
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            const int g = lig + LPR * q;
            if (g < C4) {
                float r[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) r[e] = ok && g * 4 + e < C ? (x[q][e] * share - (g * 4 + e == y ? 1.0f : 0.0f)) * invT : 0.0f;
                reinterpret_cast<float4*>(dlogits + v * ld)[g] = make_float4(r[0], r[1], r[2], r[3]);
            }
        }
    }
    // the rows of a warp in order, then its share of the block
#pragma unroll
    for (int o = LPR; o < 32; o <<= 1) {
        local += __shfl_down_sync(0xFFFFFFFFu, local, o);
        correct += __shfl_down_sync(0xFFFFFFFFu, correct, o);
    }
    if (lane == 0) sm[warp] = local;
    if (n_correct && lane == 0 && correct) atomicAdd(n_correct, (unsigned long long)correct);
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < LOSS_WARPS; ++w) t += sm[w];
        part[blockIdx.x] = t;
    }
}

// Train rows only: a warp scans 32 mask bytes, then handles the train rows among them one by one.
// Rows outside the mask are neither read nor written (pred receives -1 there).
__global__ void __launch_bounds__(LOSS_WARPS * 32) loss_rows_subset_kernel(
    int64_t n, int C, const float* logits, int64_t ld, const int32_t* __restrict__ labels,
    const uint8_t* __restrict__ mask, const unsigned long long* __restrict__ count, float* dlogits,
    int32_t* __restrict__ pred, unsigned long long* n_correct, double* __restrict__ part, int32_t* status) {
    chain_begin();
    __shared__ double sm[LOSS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long T = *count;
    const float invT = T ? (float)(1.0 / (double)T) : 0.0f;
    double local = 0.0;
    unsigned int correct = 0;
    const int64_t stride = (int64_t)gridDim.x * LOSS_WARPS * 32;
    for (int64_t v0 = ((int64_t)blockIdx.x * LOSS_WARPS + warp) * 32; v0 < n; v0 += stride) {
        const int64_t vl = v0 + lane;
        const bool mine = vl < n && mask[vl] != 0 && T != 0;
        if (pred && vl < n && !mine) pred[vl] = -1;
        unsigned live = __ballot_sync(0xFFFFFFFFu, mine);
        while (live) {
            const int64_t v = v0 + __ffs(live) - 1;
            live &= live - 1;
            const float* row = logits + v * ld;
            float mx = -INFINITY; int arg = 0x7FFFFFFF;
            for (int c = lane; c < C; c += 32) {
                const float x = row[c];
                if (x > mx || (x == mx && c < arg)) { mx = x; arg = c; }
            }
            if (arg == 0x7FFFFFFF) arg = lane < C ? lane : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float omx = __shfl_xor_sync(0xFFFFFFFFu, mx, o);
                const int oarg = __shfl_xor_sync(0xFFFFFFFFu, arg, o);
                if (omx > mx || (omx == mx && oarg < arg)) { mx = omx; arg = oarg; }
            }
            if (pred && lane == 0) pred[v] = arg;
            const int y = labels[v];
            if (y < 0 || y >= C) {
                if (lane == 0) atomicMax(status, DEV_BAD_LABEL);
                __syncwarp();
                if (dlogits) for (int c = lane; c < C; c += 32) dlogits[v * ld + c] = 0.0f;
                continue;
            }
            float s = 0.0f;
            for (int c = lane; c < C; c += 32) s += expf(row[c] - mx);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            const float lse = mx + logf(s), share = 1.0f / s;
            const float py = row[y];
            if (lane == 0) { local += (double)(lse - py); if (arg == y) ++correct; }
            __syncwarp();  // dlogits may alias logits: every read of the row precedes the writes
            if (dlogits)
                for (int c = lane; c < C; c += 32) dlogits[v * ld + c] = (expf(row[c] - mx) * share - (c == y ? 1.0f : 0.0f)) * invT;
            __syncwarp();
        }
    }
    if (lane == 0) sm[warp] = local;
    if (n_correct && lane == 0 && correct) atomicAdd(n_correct, (unsigned long long)correct);
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < LOSS_WARPS; ++w) t += sm[w];
        part[blockIdx.x] = t;
    }
}

// Launches the row pass: one partial sum a block in `part`.  False on a launch error.
bool launch_loss_rows(unsigned blocks, cudaStream_t s, int64_t n, int C, const float* logits, int64_t ld,
                      const int32_t* labels, const uint8_t* mask, const unsigned long long* count, float* dlogits,
                      int32_t* pred, unsigned long long* n_correct, double* part, int32_t* status, bool zero_rows = true) {
    // Rows in registers up to 512 columns, three or four float4 a lane; the lines lie where another float4 or twice the lanes are needed.  1 % : 8 : 30 : 60 of
    // the rows in the mask, us, against tiles of rows that bulk copies brought to shared memory (dense rows of 33 to 288 columns, four lanes
    // a row, train rows by whole warps; 8, 16 and 32 lanes with one float4 each for the others):
    //   400 K x 47 41 : 44 : 47 : 48 against 54 : 64 : 87 : 112, with a pitch of 52 47 : 50 : 52 : 52 against 62 : 66 : 76 : 85
    //   1 M x 20 54 : 64 : 73 : 73 against 67 : 79 : 95 : 103;  x 64 99 : 114 : 126 : 128 against 127 : 143 : 189 : 243
    //   1 M x 100 159 : 179 : 224 : 239 against 159 : 196 : 286 : 394;  x 172 239 : 243 : 265 : 300 against 262 : 255 : 350 : 460
    // (the bytes alone: 24, 26, 25, 80, 124 and 214 us.)
    const bool vec = (ld & 3) == 0 && aligned16(logits) && (!dlogits || aligned16(dlogits));
    auto rows_vec = [&](auto kernel) { launch_chained(kernel, dim3(blocks), LOSS_WARPS * 32, 0, s, n, C, logits, ld, labels, mask, count, dlogits, pred, n_correct, part, status, zero_rows); };
    const int C4 = (C + 3) >> 2;
    if (vec && C4 <= 4) rows_vec(loss_rows_vec_kernel<4, 1>);
    else if (vec && C4 <= 8) rows_vec(loss_rows_vec_kernel<4, 2>);
    else if (vec && C4 <= 12) rows_vec(loss_rows_vec_kernel<4, 3>);
    else if (vec && C4 <= 16) rows_vec(loss_rows_vec_kernel<4, 4>);
    else if (vec && C4 <= 24) rows_vec(loss_rows_vec_kernel<8, 3>);
    else if (vec && C4 <= 32) rows_vec(loss_rows_vec_kernel<8, 4>);
    else if (vec && C4 <= 48) rows_vec(loss_rows_vec_kernel<16, 3>);
    else if (vec && C4 <= 64) rows_vec(loss_rows_vec_kernel<16, 4>);
    else if (vec && C4 <= 96) rows_vec(loss_rows_vec_kernel<32, 3>);
    else if (vec && C4 <= 128) rows_vec(loss_rows_vec_kernel<32, 4>);
    else
        launch_chained(loss_rows_kernel, dim3(blocks), LOSS_WARPS * 32, 0, s, n, C, logits, ld, labels, mask, count, dlogits, pred, n_correct, part, status, zero_rows);
    return cudaGetLastError() == cudaSuccess;
}

// (one thread adding 2,368 partials took 17 us, and 65 us beside the traffic of a large call)
constexpr int LOSS_FINAL_THREADS = 256;
__device__ __forceinline__ void store_loss(double sum, unsigned long long T, float* loss, int32_t* status) {
    if (T == 0) { *loss = 0.0f; atomicMax(status, DEV_EMPTY_MASK); return; }
    *loss = (float)(sum / (double)T);
}

__global__ void __launch_bounds__(LOSS_FINAL_THREADS) loss_final_kernel(int blocks, const double* __restrict__ part,
                                                                       const unsigned long long* __restrict__ count, float* loss, int32_t* status) {
    chain_begin();
    __shared__ double sm[LOSS_FINAL_THREADS];
    const double t = sum_partials<LOSS_FINAL_THREADS>(part, blocks, sm);
    if (threadIdx.x == 0) store_loss(t, *count, loss, status);
}

// Final pass of the loss taken inside the aggregation: the per-row terms of the train rows are added in row
// order (block b owns rows [b * chunk, (b + 1) * chunk), its threads stride through them, fixed-order tree
// within the block), and the correct predictions are counted.  The block that finishes last adds the blocks' sums, in
// their order, and stores the loss.
constexpr int FUSE_REDUCE_THREADS = 256;
__global__ void __launch_bounds__(FUSE_REDUCE_THREADS) loss_rows_reduce_kernel(
    int64_t n, int C, int64_t chunk, const uint8_t* __restrict__ mask, const int32_t* __restrict__ labels,
    const float* __restrict__ row_loss, const int32_t* __restrict__ pred, double* part,
    unsigned long long* n_correct, unsigned int* done, const unsigned long long* __restrict__ count, float* loss, int32_t* status) {
    chain_begin();
    __shared__ bool last;
    __shared__ double sm[FUSE_REDUCE_THREADS];
    __shared__ unsigned int sc[FUSE_REDUCE_THREADS / 32];
    const int64_t r0 = (int64_t)blockIdx.x * chunk, r1 = r0 + chunk < n ? r0 + chunk : n;
    double local = 0.0;
    unsigned int correct = 0;
    for (int64_t v = r0 + threadIdx.x; v < r1; v += FUSE_REDUCE_THREADS) {
        if (!mask[v]) continue;
        const int y = labels[v];
        if (y < 0 || y >= C) continue;            // reported by the aggregation's epilogue; contributes nothing
        local += (double)row_loss[v];
        if (pred && pred[v] == y) ++correct;
    }
    sm[threadIdx.x] = local;
    for (int o = 16; o > 0; o >>= 1) correct += __shfl_down_sync(0xFFFFFFFFu, correct, o);
    if ((threadIdx.x & 31) == 0) sc[threadIdx.x >> 5] = correct;
    __syncthreads();
    for (int half = FUSE_REDUCE_THREADS / 2; half > 0; half >>= 1) {
        if (threadIdx.x < half) sm[threadIdx.x] += sm[threadIdx.x + half];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[blockIdx.x] = sm[0];
        unsigned int t = 0;
        for (int w = 0; w < FUSE_REDUCE_THREADS / 32; ++w) t += sc[w];
        if (n_correct && t) atomicAdd(n_correct, (unsigned long long)t);   // integer: order does not matter
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double total = sum_partials<FUSE_REDUCE_THREADS>(part, (int)gridDim.x, sm);
    if (threadIdx.x == 0) store_loss(total, *count, loss, status);
}

constexpr int ADAM_MAX_TENSORS = 16;
struct AdamBatch {
    float* p[ADAM_MAX_TENSORS];
    const float* g[ADAM_MAX_TENSORS];
    float* m[ADAM_MAX_TENSORS];
    float* v[ADAM_MAX_TENSORS];
    int64_t numel[ADAM_MAX_TENSORS];
    int count;
    float lr, beta1, beta2, eps, inv_c1, inv_c2;
};

__global__ void adam_kernel(const AdamBatch b) {
    chain_begin();
    const int t = blockIdx.y;
    if (t >= b.count) return;
    const int64_t nel = b.numel[t];
    float* __restrict__ p = b.p[t]; const float* __restrict__ g = b.g[t];
    float* __restrict__ m = b.m[t]; float* __restrict__ v = b.v[t];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nel; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b.beta1 * m[i] + (1.0f - b.beta1) * gi;
        const float vi = b.beta2 * v[i] + (1.0f - b.beta2) * gi * gi;
        m[i] = mi; v[i] = vi;
        const float mhat = mi * b.inv_c1, vhat = vi * b.inv_c2;
        p[i] = p[i] - b.lr * mhat / (sqrtf(vhat) + b.eps);
    }
}

}  // namespace

namespace mixgcn {

mixgcn_status launch_clear(mixgcn_ctx* ctx, int phase, void* words, int n_words, int64_t* also, cudaStream_t s) {
    LaunchScope scope(ctx, phase, s);
    launch_chained(clear_kernel, dim3(1), 32, 0, s, static_cast<uint32_t*>(words), n_words, also);
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

// *count = train nodes; the word behind it (blocks that have finished) and *n_correct (nullable) are cleared.
static mixgcn_status count_train_nodes(mixgcn_ctx* ctx, int64_t n, const uint8_t* train_mask, unsigned long long* count,
                                       int64_t* n_correct, cudaStream_t s) {
    if (n <= COUNT_ONE_BLOCK_MAX) {
        LaunchScope scope(ctx, PH_LOSS, s);
        launch_chained(count_mask_small_kernel, dim3(1), 1024, 0, s, n, train_mask, count, reinterpret_cast<unsigned int*>(count + 1),
                                                  reinterpret_cast<unsigned long long*>(n_correct));
    } else {
        MIXGCN_TRY(launch_clear(ctx, PH_LOSS, count, 4, n_correct, s));
        LaunchScope scope(ctx, PH_LOSS, s);
        int64_t cb = (n / 16 + 255) / 256;
        if (cb > (int64_t)ctx->sm_count * 8) cb = (int64_t)ctx->sm_count * 8;
        launch_chained(count_mask_kernel, dim3((unsigned)cb), 256, 0, s, n, train_mask, count);
    }
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

// Scratch of the fused loss (a block of its own): [count u64][done u32][pad][partials double[blocks]][row_loss float[n]].
// Counts the train nodes (the gradient's 1/#T is needed inside the kernel that takes the loss) and clears n_correct.
mixgcn_status loss_fuse_begin(mixgcn_ctx* ctx, int64_t n, const int32_t* labels, const uint8_t* train_mask, int32_t* pred,
                              int64_t* n_correct, cudaStream_t s, LossFuse* out) {
    const int64_t cap = (int64_t)ctx->sm_count * 16;
    int64_t blocks = (n + FUSE_REDUCE_THREADS * 2 - 1) / (FUSE_REDUCE_THREADS * 2);
    if (blocks > cap) blocks = cap;
    const int64_t off_rows = (16 + blocks * (int64_t)sizeof(double) + 255) & ~(int64_t)255;
    const int64_t need = off_rows + n * (int64_t)sizeof(float);
    MIXGCN_TRY(grow_block(ctx, &ctx->workspace_loss, &ctx->workspace_loss_bytes, need, "loss scratch"));
    char* base = reinterpret_cast<char*>(ctx->workspace_loss);
    unsigned long long* count = reinterpret_cast<unsigned long long*>(base);
    MIXGCN_TRY(count_train_nodes(ctx, n, train_mask, count, n_correct, s));
    out->labels = labels; out->train_mask = train_mask; out->count = count; out->pred = pred;
    out->part = reinterpret_cast<double*>(base + 16); out->n_part = (int)blocks;
    out->row_loss = reinterpret_cast<float*>(base + off_rows);
    out->zero_rows = ctx->loss_train_rows_only == 2 ? 0 : 1;
    return MIXGCN_OK;
}

mixgcn_status loss_fuse_end(mixgcn_ctx* ctx, int64_t n, int32_t C, const LossFuse& lf, float* loss, int64_t* n_correct, cudaStream_t s) {
    const int64_t chunk = (n + lf.n_part - 1) / lf.n_part;
    {
        LaunchScope scope(ctx, PH_LOSS, s);
        launch_chained(loss_rows_reduce_kernel, dim3((unsigned)lf.n_part), FUSE_REDUCE_THREADS, 0, s, n, C, chunk, lf.train_mask, lf.labels, lf.row_loss, lf.pred, lf.part,
                                                                                  reinterpret_cast<unsigned long long*>(n_correct),
                                                                                  const_cast<unsigned int*>(reinterpret_cast<const unsigned int*>(lf.count + 1)), lf.count, loss, ctx->d_status);
    }
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

}  // namespace mixgcn

extern "C" mixgcn_status mixgcn_loss_softmax_xent(mixgcn_ctx* ctx, int64_t n, int32_t C, const float* logits,
                                                  int64_t ld, const int32_t* labels, const uint8_t* train_mask,
                                                  float* loss, float* dlogits, int32_t* pred, int64_t* n_correct,
                                                  void* stream) {
    if (!ctx || !logits || !labels || !train_mask || !loss) MIXGCN_FAIL(MIXGCN_EINVAL, "loss: null argument");
    if (n <= 0 || C <= 0 || C > 4096) MIXGCN_FAIL(MIXGCN_EINVAL, "loss: need n > 0 and 1 <= C <= 4096 (n=%lld C=%d)", (long long)n, C);
    if (ld < C) MIXGCN_FAIL(MIXGCN_EINVAL, "loss: ld (%lld) < C (%d)", (long long)ld, C);
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    int64_t blocks = (n + LOSS_WARPS - 1) / LOSS_WARPS;
    const int64_t cap = (int64_t)ctx->sm_count * 16;
    if (blocks > cap) blocks = cap;
    // workspace: [count u64][pad][partials double[blocks]]
    MIXGCN_TRY(mixgcn::ensure_workspace(ctx, 16 + blocks * (int64_t)sizeof(double)));
    unsigned long long* count = reinterpret_cast<unsigned long long*>(ctx->workspace);
    double* part = reinterpret_cast<double*>(reinterpret_cast<char*>(ctx->workspace) + 16);
    MIXGCN_TRY(count_train_nodes(ctx, n, train_mask, count, n_correct, s));
    bool launched = true;
    {
        LaunchScope scope(ctx, PH_LOSS, s);
        if (ctx->loss_train_rows_only == 1)
            launch_chained(loss_rows_subset_kernel, dim3((unsigned)blocks), LOSS_WARPS * 32, 0, s, n, C, logits, ld, labels, train_mask, count, dlogits, pred,
                                                                              reinterpret_cast<unsigned long long*>(n_correct), part, ctx->d_status);
        else
            launched = launch_loss_rows((unsigned)blocks, s, n, C, logits, ld, labels, train_mask, count, dlogits, pred,
                                        reinterpret_cast<unsigned long long*>(n_correct), part, ctx->d_status,
                                        ctx->loss_train_rows_only != 2);
    }
    if (!launched) MIXGCN_FAIL(MIXGCN_ECUDA, "loss: kernel launch failed: %s", cudaGetErrorString(cudaGetLastError()));
    {
        LaunchScope scope(ctx, PH_LOSS, s);
        launch_chained(loss_final_kernel, dim3(1), LOSS_FINAL_THREADS, 0, s, (int)blocks, part, count, loss, ctx->d_status);
    }
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

extern "C" mixgcn_status mixgcn_adam_step(mixgcn_ctx* ctx, int32_t n_tensors, float* const* param,
                                          const float* const* grad, float* const* m, float* const* v,
                                          const int64_t* numel, int64_t t, float lr, float beta1, float beta2,
                                          float eps, void* stream) {
    if (!ctx || n_tensors < 0 || (n_tensors > 0 && (!param || !grad || !m || !v || !numel)))
        MIXGCN_FAIL(MIXGCN_EINVAL, "adam: null argument");
    if (t < 1) MIXGCN_FAIL(MIXGCN_EINVAL, "adam: step count t must be >= 1 (got %lld)", (long long)t);
    for (int i = 0; i < n_tensors; ++i) {
        if (numel[i] < 0 || (numel[i] > 0 && (!param[i] || !grad[i] || !m[i] || !v[i])))
            MIXGCN_FAIL(MIXGCN_EINVAL, "adam: tensor %d has a null pointer or negative size", i);
    }
    MIXGCN_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    const double c1 = 1.0 - pow((double)beta1, (double)t), c2 = 1.0 - pow((double)beta2, (double)t);
    for (int base = 0; base < n_tensors; base += ADAM_MAX_TENSORS) {
        AdamBatch b{};
        int64_t mx = 0;
        b.count = n_tensors - base < ADAM_MAX_TENSORS ? n_tensors - base : ADAM_MAX_TENSORS;
        for (int i = 0; i < b.count; ++i) {
            b.p[i] = param[base + i]; b.g[i] = grad[base + i]; b.m[i] = m[base + i]; b.v[i] = v[base + i];
            b.numel[i] = numel[base + i];
            if (b.numel[i] > mx) mx = b.numel[i];
        }
        if (mx == 0) continue;
        b.lr = lr; b.beta1 = beta1; b.beta2 = beta2; b.eps = eps;
        b.inv_c1 = (float)(1.0 / c1); b.inv_c2 = (float)(1.0 / c2);
        int64_t bx = (mx + 255) / 256; if (bx > 1024) bx = 1024;
        LaunchScope scope(ctx, PH_ADAM, s);
        launch_chained(adam_kernel, dim3((unsigned)bx, (unsigned)b.count), 256, 0, s, b);
    }
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}

// ------------------------------------------------------------------------------------------------
// Allocation-free variant of the loss.
//
// Some callers cannot take device memory from the CUDA allocator: a process that has handed the
// whole GPU to its own memory pool (so cudaMalloc fails), or a latency-critical loop that cannot
// afford the device-wide synchronisation cudaMalloc and cudaFree imply.  They cannot create a
// mixgcn_ctx either (its status word and workspace come from cudaMalloc).  For them the loss
// kernels above run here with their scratch in a fixed array that is part of the library image.
// ------------------------------------------------------------------------------------------------
namespace {

constexpr int NOALLOC_MAX_PARTIALS = 32768;   // one fp64 partial per block
constexpr int NOALLOC_ROWS_PER_BLOCK = 1024;  // => at most 33,554,432 rows
constexpr int NOALLOC_MAX_DEVICES = 64;

struct NoAllocScratch {
    unsigned long long count;      // train nodes, cleared at the start of every call
    int32_t status;                // 0 ok, 1 empty train mask, 2 label out of range, 3 bounded wait expired; cleared likewise
    int32_t pad;
    double part[NOALLOC_MAX_PARTIALS];
};

// Held by every GPU that loads the library, until the process exits (about 256 KB).
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

// In host code the array's name is only a handle for the runtime, not a device address; the real
// address is looked up once per device (with that device current) and cached here.  Host threads that
// make their first call on a device at the same time both store the same address: the entries are
// atomic so that this is well defined.
std::atomic<NoAllocScratch*> g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

}  // namespace

extern "C" mixgcn_status mixgcn_loss_softmax_xent_noalloc(int64_t n, int32_t C, const float* logits, int64_t ld,
                                                          const int32_t* labels, const uint8_t* train_mask,
                                                          float* loss, float* dlogits, int32_t* pred,
                                                          int64_t* n_correct, int32_t* status, void* stream) {
    if (!logits || !labels || !train_mask || !loss) MIXGCN_FAIL(MIXGCN_EINVAL, "loss_noalloc: null argument");
    if (n <= 0 || C <= 0 || C > 4096)
        MIXGCN_FAIL(MIXGCN_EINVAL, "loss_noalloc: need n > 0 and 1 <= C <= 4096 (n=%lld C=%d)", (long long)n, C);
    if (ld < C) MIXGCN_FAIL(MIXGCN_EINVAL, "loss_noalloc: ld (%lld) < C (%d)", (long long)ld, C);
    const int64_t max_rows = (int64_t)NOALLOC_MAX_PARTIALS * NOALLOC_ROWS_PER_BLOCK;
    if (n > max_rows)
        MIXGCN_FAIL(MIXGCN_EUNSUPPORTED,
                    "loss_noalloc: n = %lld exceeds the %lld rows the built-in scratch covers; use mixgcn_loss_softmax_xent",
                    (long long)n, (long long)max_rows);
    int device = -1;
    MIXGCN_CUDA(cudaGetDevice(&device));
    if (device < 0 || device >= NOALLOC_MAX_DEVICES) MIXGCN_FAIL(MIXGCN_EUNSUPPORTED, "loss_noalloc: device index %d not supported", device);
    if (!g_noalloc_ptr[device].load(std::memory_order_acquire)) {
        // first call on this device: resolve the device address of the scratch array
        void* p = nullptr;
        MIXGCN_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        if (!p) MIXGCN_FAIL(MIXGCN_ECUDA, "loss_noalloc: the scratch symbol has no device address");
        g_noalloc_ptr[device].store(reinterpret_cast<NoAllocScratch*>(p), std::memory_order_release);
    }
    NoAllocScratch* sc = g_noalloc_ptr[device].load(std::memory_order_acquire);
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t blocks = (n + NOALLOC_ROWS_PER_BLOCK - 1) / NOALLOC_ROWS_PER_BLOCK;
    // the array keeps the previous call's contents: clear the counter and the status word
    MIXGCN_CUDA(cudaMemsetAsync(sc, 0, offsetof(NoAllocScratch, part), s));
    if (n_correct) MIXGCN_CUDA(cudaMemsetAsync(n_correct, 0, sizeof(int64_t), s));
    int64_t cb = (n + 255) / 256;
    if (cb > 4096) cb = 4096;
    launch_chained(count_mask_kernel, dim3((unsigned)cb), 256, 0, s, n, train_mask, &sc->count);
    if (!launch_loss_rows((unsigned)blocks, s, n, C, logits, ld, labels, train_mask, &sc->count, dlogits, pred,
                          reinterpret_cast<unsigned long long*>(n_correct), sc->part, &sc->status))
        MIXGCN_FAIL(MIXGCN_ECUDA, "loss_noalloc: kernel launch failed: %s", cudaGetErrorString(cudaGetLastError()));
    launch_chained(loss_final_kernel, dim3(1), LOSS_FINAL_THREADS, 0, s, (int)blocks, sc->part, &sc->count, loss, &sc->status);
    if (status) MIXGCN_CUDA(cudaMemcpyAsync(status, &sc->status, sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    MIXGCN_CUDA(cudaGetLastError());
    return MIXGCN_OK;
}
