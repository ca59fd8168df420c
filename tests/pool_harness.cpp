// Test harness for a context's memory pool (make_pool and StreamBuf of
// paper_2605_19254_gb300/csrc/smf_internal.h), compiled for the host against a
// fake of the CUDA calls it makes: the first `fails` pool creations fail.  Prints
// the status of each allocation in turn, then that of eight threads' allocations,
// the pools made, the bytes their threshold keeps, and the buffers not freed.
#include <stdio.h>
#include <stdlib.h>

#include <atomic>
#include <thread>
#include <vector>

#include "smf_internal.h"

static std::atomic<int> g_fails, g_made, g_live;
static uint64_t g_keep;

extern "C" {
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps* p) {
    if (g_fails > 0) {
        g_fails--;
        return cudaErrorMemoryAllocation;
    }
    if (p->location.id != 3) return cudaErrorInvalidDevice;
    std::this_thread::yield();
    g_made++;
    *pool = (cudaMemPool_t)&g_made;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* v) {
    g_keep = *(uint64_t*)v;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) {
    if (pool != (cudaMemPool_t)&g_made) return cudaErrorInvalidValue;
    g_live++;
    *p = malloc(n);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
    g_live--;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
}

int main(int argc, char** argv) {
    g_fails = argc > 1 ? atoi(argv[1]) : 0;
    smf_ctx ctx{};
    ctx.device = 3;
    ctx.pool_keep = 12345;
    for (int i = 0; i < 3; i++) {
        smf::StreamBuf b;
        printf("%d ", (int)b.alloc(&ctx, 100, nullptr));
    }
    smf_ctx many{};
    many.device = 3;
    many.pool_keep = 12345;
    std::atomic<int> bad{0};
    std::vector<std::thread> th;
    for (int i = 0; i < 8; i++)
        th.emplace_back([&] {
            for (int k = 0; k < 100; k++) {
                smf::StreamBuf b;
                if (b.alloc(&many, 64, nullptr) != cudaSuccess || !b.p) bad++;
            }
        });
    for (auto& t : th) t.join();
    printf("%d %d %llu %d\n", bad.load(), g_made.load(), (unsigned long long)g_keep, g_live.load());
    return 0;
}
