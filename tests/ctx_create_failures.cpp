// mixgcn_ctx_create against a CUDA runtime that fails at its k-th call, for every k: the call reports the failure, leaves no
// stream, event or memory behind, and the device's memory pool keeps freed memory only while a context exists.
// Built with the host compiler from api.cu and this file; no GPU.
#include <stdio.h>
#include <string.h>

#include <set>

#include "internal.cuh"

namespace {
int calls = 0, fail_at = -1;
uint64_t kept = 0;                        // the pool's release threshold
std::set<void*> live;
char arena[1 << 16];
int used = 0;

cudaError_t step() { return calls++ == fail_at ? cudaErrorUnknown : cudaSuccess; }
template <class T> cudaError_t make(T* out) {
    const cudaError_t e = step();
    if (e != cudaSuccess) return e;
    *out = reinterpret_cast<T>(arena + used++);
    live.insert((void*)*out);
    return cudaSuccess;
}
template <class T> cudaError_t drop(T x) { live.erase((void*)x); return cudaSuccess; }
}  // namespace

namespace mixgcn { void free_step_cache(mixgcn_ctx*) {} }

extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return step(); }
cudaError_t cudaSetDevice(int) { return step(); }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { memset(p, 0, sizeof(*p)); p->major = 10; p->multiProcessorCount = 148; return step(); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { const cudaError_t e = step(); if (e == cudaSuccess) *p = (cudaMemPool_t)arena; return e; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 30; return step(); }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* v) { const cudaError_t e = step(); if (e == cudaSuccess) kept = *(uint64_t*)v; return e; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t) { return make(p); }
cudaError_t cudaMemset(void*, int, size_t) { return step(); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return make(s); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return make(e); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return drop(s); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return drop(e); }
cudaError_t cudaFree(void* p) { return drop(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return drop(p); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
}

int main() {
    for (int k = 0;; ++k) {
        mixgcn_ctx* ctx = nullptr;
        calls = 0; fail_at = k;
        const mixgcn_status st = mixgcn_ctx_create(&ctx, 0);
        const bool reached = calls > k;
        fail_at = -1;
        if (!reached) {
            if (st != MIXGCN_OK || !ctx || !kept) { printf("creation failed without a failing call\n"); return 1; }
            mixgcn_ctx_destroy(ctx);
            if (!live.empty() || kept) { printf("destroy left %d objects, %llu bytes kept\n", (int)live.size(), (unsigned long long)kept); return 1; }
            printf("%d calls\n", k);
            return 0;
        }
        if (st == MIXGCN_OK || ctx) { printf("call %d failed and was not reported\n", k); return 1; }
        if (!live.empty() || kept) { printf("call %d failed: %d objects left, %llu bytes kept\n", k, (int)live.size(), (unsigned long long)kept); return 1; }
    }
}
