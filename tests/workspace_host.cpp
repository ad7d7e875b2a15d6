// dsq_workspace_status (csrc/dsq_workspace.cu) on a CUDA runtime that is a fake.  Built
// and driven by test_workspace_host.py.
#include "../paper_1908_05033_b200/csrc/dsq_workspace.cu"

#include <chrono>
#include <cstring>
#include <thread>
#include <utility>

namespace {
struct Fake {
    int host_allocs, host_frees, kernels, copies, syncs;
    int fail_host_alloc, device_of_ws, capture_elsewhere, broken;
    int pdl, dependent;          // the hook; launches with the attribute
    int schedule, late, waited;  // device flags; the kernel runs in the stream's wait; us before it
} f;
int *g_late[2];
std::chrono::steady_clock::time_point g_launched;
thread_local cudaStreamCaptureMode g_mode = cudaStreamCaptureModeGlobal;
int g_word[64];

cudaError_t unsafe()
{
    if (!f.capture_elsewhere || g_mode == cudaStreamCaptureModeRelaxed) return cudaSuccess;
    f.broken = 1;
    return cudaErrorStreamCaptureUnsupported;
}
}  // namespace

dsq_plan *&dsq_recording_plan()
{
    static dsq_plan *none = nullptr;
    return none;
}

DsqLaunchHooks dsq_launch_hooks()
{
    DsqLaunchHooks h = {};
    h.pdl = f.pdl;
    return h;
}

extern "C" {
Fake *fake() { return &f; }
// the status read by a thread of its own
int status_of_new_thread(int *ws, int calls)
{
    int st = 0;
    std::thread([&] {
        for (int i = 0; i < calls; ++i) {
            const int r = dsq_workspace_status(ws, nullptr);
            if (r) st = r;
        }
    }).join();
    return st;
}

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m)
{
    std::swap(*m, g_mode);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t, unsigned)
{
    if (f.fail_host_alloc) return cudaErrorMemoryAllocation;
    const cudaError_t e = unsafe();
    if (e != cudaSuccess) return e;
    *p = g_word;
    ++f.host_allocs;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *) { ++f.host_frees; return unsafe(); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *)
{
    a->type = cudaMemoryTypeDevice;
    a->device = f.device_of_ws;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceFlags(unsigned *flags) { *flags = (unsigned)f.schedule; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *cfg, const void *k, void **args)
{
    ++f.kernels;
    f.dependent += cfg->numAttrs != 0;
    g_late[0] = *(int **)args[0];
    g_late[1] = *(int **)args[1];
    g_launched = std::chrono::steady_clock::now();
    if (!f.late) status_kernel(g_late[0], g_late[1]);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    ++f.copies;
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t)
{
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t)
{
    ++f.syncs;
    if (f.late) {
        const auto us = std::chrono::duration_cast<std::chrono::microseconds>(std::chrono::steady_clock::now() - g_launched);
        if (!f.waited || us.count() < f.waited) f.waited = (int)us.count();
        status_kernel(g_late[0], g_late[1]);
    }
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}
