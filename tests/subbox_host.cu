// The shared-amplitude route of the sub-box sums (subbox_cells.cu) with a scratch pool whose n-th allocation fails:
// no GPU, no driver.  The route hands the request back with nothing held, so that the box-by-box route finds
// the memory that it would have found alone.  Exit status 0 when that holds for every n, up to the one
// whose allocations all succeed (the first launch ends the program).
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "api_internal.h"
#include "subbox_points.h"

static int g_fail_at = 0, g_calls = 0;

#ifndef __CUDA_ARCH__   // the device pass has its own
extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h = nullptr; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st *) { exit(g_calls == g_fail_at - 1 ? 0 : 3); }   // all had: it launches
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { abort(); }
cudaError_t __cudaGetKernel(cudaKernel_t *, const void *) { abort(); }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { abort(); }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *, const void *) { abort(); }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { abort(); }
}
#endif

namespace ds {
void count_launches(int) {}
}  // namespace ds
ProfScope::ProfScope(ds_ctx *, const char *, cudaStream_t) {}
ProfScope::~ProfScope() {}
Scratch::~Scratch() {}
void *Scratch::get(size_t bytes) {
    if (++g_calls >= g_fail_at) return failed = true, nullptr;
    ptrs.push_back((void *)4096);   // never touched
    total += bytes;
    return ptrs.back();
}

int main() {
    ds_ctx ctx;
    ctx.budget = (size_t)1 << 40;
    ds_model m;
    m.ctx = &ctx;
    m.nsite = 2;
    m.nmodels = 1;
    m.n[0] = m.n[1] = m.n[2] = 16;
    ds_opts o;
    memset(&o, 0, sizeof(o));
    o.mode = DS_DIFFUSE;
    o.subbox_n = 5;
    for (g_fail_at = 1;; ++g_fail_at) {
        g_calls = 0;
        Scratch ws(nullptr);
        const bool took = subbox_cells_run<float>(&m, SB_DISP, nullptr, nullptr, 4096, nullptr, 1000, &o, nullptr, 1.0, ws, nullptr);
        if (took || ws.failed || !ws.ptrs.empty() || ws.total != 0) {
            fprintf(stderr, "allocation %d fails: taken %d, failed %d, %zu held\n", g_fail_at, took, ws.failed, ws.ptrs.size());
            return 1;
        }
        if (g_calls < 1) return fprintf(stderr, "the route was not tried\n"), 2;
    }
}
