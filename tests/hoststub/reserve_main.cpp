// The estimate workspace when an allocation fails (test only): after the failure, whichever
// allocation it was, a smaller call finds every array that it will use, and no error of
// the failed allocation is left for a later launch to report.
#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include <cuda_runtime.h>

#include "dpd.h"
#include "dpd_gram.cuh"
#include "dpd_handle.h"

static int g_left = -1;   // allocations until one fails (-1: none does)
static int g_pending = 0;
static cudaError_t alloc(void **p, size_t n)
{
    if (g_left >= 0 && g_left-- == 0) return (cudaError_t)(g_pending = cudaErrorMemoryAllocation);
    *p = std::malloc(n < 64 ? n : 64);   // never read: only whether it is there counts
    return cudaSuccess;
}
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocHost(void **p, size_t n) { return alloc(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return alloc(p, n); }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaGetLastError() { const int e = g_pending; g_pending = 0; return (cudaError_t)e; }
}

namespace {
#include "reserve_part.h"
}

static bool whole(const EstimateWorkspace &w)
{
    for (const void *p : {(const void *)w.probs, (const void *)w.partials, (const void *)w.S, (const void *)w.Clag,
                          (const void *)w.G, (const void *)w.g, (const void *)w.U, (const void *)w.wide, (const void *)w.h64,
                          (const void *)w.d, (const void *)w.tt, (const void *)w.info, (const void *)w.tab,
                          (const void *)w.norm_part, (const void *)w.ubasis, (const void *)w.ubasis64,
                          (const void *)w.mom_part, (const void *)w.y, (const void *)w.e, (const void *)w.h_G,
                          (const void *)w.h_U, (const void *)w.h_info, (const void *)w.h_norm})
        if (!p) return false;
    return true;
}

int main()
{
    int failures = 0;
    for (int fail = 0;; ++fail) {
        dpd_filter h{};
        h.K = 97;
        h.B = 6;
        h.T = 8;
        bool ok = reserve(&h, 3, 2, dpd::kPrecTF32x3, 1000) == DPD_OK && whole(h.est);
        g_left = fail;
        const dpd_status st = reserve(&h, 300, 7, dpd::kPrecTF32x3, 100000);
        const bool failed = st == DPD_ERR_ALLOC;
        g_left = -1;
        ok = ok && (failed || st == DPD_OK) && g_pending == 0;
        ok = ok && reserve(&h, 2, 2, dpd::kPrecTF32x3, 500) == DPD_OK && whole(h.est);
        std::printf("allocation %d: %s, %s\n", fail, failed ? "failed" : "all made", ok ? "ok" : "BAD");
        if (!ok) return 1;
        if (!failed) break;
        ++failures;
    }
    std::printf("failures %d\n", failures);
    return failures >= 18 ? 0 : 2;
}
