// The serving loop (serving.cu) against stand-ins for the CUDA runtime and for the functions that queue kernels:
// no GPU, no driver.  Each stand-in of a driver call that frees something checks that the context's
// lock is free, since a completion callback that waits for the lock may be what the driver waits for.
// Usage: serving_host CASE; exit status 0 when the case holds.
#include <atomic>
#include <chrono>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>

#include "api_internal.h"

static ds_ctx *g_ctx = nullptr;
static std::atomic<int> g_locked{0}, g_destroyed{0};
static ds_status g_plan = DS_OK;      // what planning a displacive request returns

static void lock_must_be_free() {
    bool ok = false;
    std::thread([&] {
        ok = g_ctx->mu.try_lock();
        if (ok) g_ctx->mu.unlock();
    }).join();
    if (!ok) ++g_locked;
}

#ifndef __CUDA_ARCH__   // the device pass has its own
extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h = nullptr; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
cudaError_t cudaDeviceGetStreamPriorityRange(int *a, int *b) { return *a = 0, *b = -1, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = (cudaEvent_t)malloc(1), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { lock_must_be_free(); ++g_destroyed; free(e); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { lock_must_be_free(); return *ms = 1.f, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t fn, void *arg) {
    std::thread([=] { fn(arg); }).detach();
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
#endif

Scratch::~Scratch() {}
void Scratch::release() {}
ds_status ds_fail(ds_ctx *, ds_status st, const char *, ...) { return st; }
ds_status check_request(ds_model *, const ds_qgrid *, const ds_opts *) { return DS_OK; }
ds_status grid_indices(ds_ctx *, const ds_model *, const ds_qgrid *, int g0[3], int cnt[3]) {
    for (int a = 0; a < 3; ++a) g0[a] = 0, cnt[a] = 1;
    return DS_OK;
}
size_t request_footprint(const ds_model *, const ds_qgrid *, const ds_opts *, int) { return 1; }
ds_status queue_corner_xmax(ds_model *, const ds_qgrid *, const ds_opts *, cudaStream_t, Scratch &, double *) { return g_plan; }
ds_status resolve_taylor_order(ds_model *, const ds_qgrid *, const ds_opts *, cudaStream_t, Scratch &, int *P, double *x, double *u) {
    *P = 2, *x = 0.1, *u = 0.1;
    return g_plan;
}
ds_status taylor_order_from_corners(ds_ctx *, const ds_opts *, const double *, int *P, double *x, double *u) {
    *P = 2, *x = 0.1, *u = 0.1;
    return DS_OK;
}
template <typename T>
ds_status enqueue_request(ds_model *, const ds_qgrid *, const ds_opts *, T *, cudaStream_t, Scratch &, ds_result_info *, const TaylorHint *) {
    return DS_OK;
}
template ds_status enqueue_request<float>(ds_model *, const ds_qgrid *, const ds_opts *, float *, cudaStream_t, Scratch &,
                                          ds_result_info *, const TaylorHint *);
template ds_status enqueue_request<double>(ds_model *, const ds_qgrid *, const ds_opts *, double *, cudaStream_t, Scratch &,
                                           ds_result_info *, const TaylorHint *);
void serving_shutdown(ds_ctx *);

#define EXPECT(c) do { if (!(c)) { fprintf(stderr, "line %d: %s\n", __LINE__, #c); ++bad; } } while (0)

int main(int argc, char **argv) {
    const char *which = argc > 1 ? argv[1] : "";
    int bad = 0;
    ds_ctx ctx;
    g_ctx = &ctx;
    ctx.budget = 1 << 20;
    ds_model model;
    model.ctx = &ctx;
    ds_qgrid q;
    ds_opts o;
    memset(&q, 0, sizeof(q));
    memset(&o, 0, sizeof(o));
    o.precision = DS_FP32;
    o.disorder = DS_DISP;
    o.taylor_order = -1;
    float out = 0.f;
    uint64_t t = 0, t2 = 0;
    if (!strcmp(which, "planning_fails") || !strcmp(which, "planning_fails_without_a_slot")) {
        EXPECT(ds_submit(&model, &q, &o, &out, &t) == DS_OK);       // starts the worker
        EXPECT(ds_wait(&ctx, t, 10.0, nullptr) == DS_OK);
        if (strstr(which, "slot")) {
            std::lock_guard<std::mutex> g(ctx.mu);
            ctx.plan_free.clear();
        }
        g_plan = DS_ERR_UNSUPPORTED;
        EXPECT(ds_submit(&model, &q, &o, &out, &t2) == DS_ERR_UNSUPPORTED);
        EXPECT(g_destroyed == 4);
        EXPECT(ctx.jobs.empty() && ctx.queue.empty());
    } else if (!strcmp(which, "two_waiters")) {
        o.taylor_order = 2;
        ds_serving_pause(&ctx, 1);
        EXPECT(ds_submit(&model, &q, &o, &out, &t) == DS_OK);
        ds_status st[2];
        std::thread w[2];
        for (int i = 0; i < 2; ++i) w[i] = std::thread([&, i] { st[i] = ds_wait(&ctx, t, 10.0, nullptr); });
        std::this_thread::sleep_for(std::chrono::milliseconds(300));   // both wait
        ds_serving_pause(&ctx, 0);
        for (int i = 0; i < 2; ++i) w[i].join();
        EXPECT((st[0] == DS_OK && st[1] == DS_ERR_ARG) || (st[0] == DS_ERR_ARG && st[1] == DS_OK));
        EXPECT(g_destroyed == 2);
    } else {
        return 2;
    }
    EXPECT(g_locked == 0);
    serving_shutdown(&ctx);
    return bad ? 1 : 0;
}
