// The workspace of the tensor-core kernels: its size, clearing it, reading its status.
#include <chrono>

#include "dsq_launch.h"

namespace {

// Hands a workspace's status word to the host and clears it.  Written straight into
// page-locked host memory: a copy to pageable memory is staged and took 3 us more of
// every call that reads the status (binary GEMM 3136x512x4608: 41 -> 38 us).  Launched
// dependently: it starts beside the kernel whose status it reads and waits for it.
constexpr int STATUS_PENDING = 1;        // (statuses are 0 or negative)
__global__ void status_kernel(int *ws, volatile int *host)
{
#ifdef __CUDA_ARCH__
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
    const int st = *(volatile int *)(ws + DSQ_WS_STATUS);
    if (st) ws[DSQ_WS_STATUS] = ws[DSQ_WS_DETAIL] = 0;
    *host = st;
}

// One page-locked word per thread that asks, given back when the thread ends.
struct StatusMailbox {
    int *word = nullptr;
    // (nullptr where there is none to be had)
    int *get()
    {
        if (word) return word;
        const DsqCaptureRelaxed relaxed;
        void *p = nullptr;
        if (cudaHostAlloc(&p, sizeof(int), cudaHostAllocPortable) == cudaSuccess) word = (int *)p;
        else cudaGetLastError();
        return word;
    }
    ~StatusMailbox()
    {
        if (!word) return;
        const DsqCaptureRelaxed relaxed;
        cudaFreeHost(word);
    }
};

// Whether a kernel of the current device may read `p`: memory of another device may only
// be copied from.
bool on_current_device(const void *p)
{
    int dev = -1;
    cudaPointerAttributes a;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaPointerGetAttributes(&a, p) == cudaSuccess)
        return a.type == cudaMemoryTypeDevice && a.device == dev;
    cudaGetLastError();
    return false;
}

// Whether CUDA's own waits spin on the current device (the default while cores are free).
bool waits_spin()
{
    unsigned flags = 0;
    if (cudaGetDeviceFlags(&flags) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    flags &= cudaDeviceScheduleMask;
    return flags != cudaDeviceScheduleYield && flags != cudaDeviceScheduleBlockingSync;
}

}  // namespace

extern "C" {

size_t dsq_workspace_bytes(void) { return DSQ_WS_BYTES; }

int dsq_workspace_init(void *ws, size_t ws_bytes, void *stream)
{
    if (!ws) return DSQ_ERR_NULL;
    if (!dsq_aligned16(ws)) return DSQ_ERR_ALIGN;
    if (ws_bytes < DSQ_WS_BYTES) return DSQ_ERR_SIZE;
    DSQ_CUDA_TRY(cudaMemsetAsync(ws, 0, DSQ_WS_BYTES, (cudaStream_t)stream));
    return DSQ_OK;
}

int dsq_workspace_status(void *ws, void *stream)
{
    if (!ws) return DSQ_ERR_NULL;
    cudaStream_t s = (cudaStream_t)stream;
    static thread_local StatusMailbox box;
    int *const word = box.get();
    if (word && on_current_device(ws)) {
        *(volatile int *)word = STATUS_PENDING;
        int *w = (int *)ws;
        void *argv[] = {(void *)&w, (void *)&word};
        const DsqGrid one = {(const void *)status_kernel, dim3(1), dim3(1), 0, dsq_launch_hooks().pdl, 0};
        const int st = dsq_launch_args(one, argv, s);
        if (st) return st;
        // The word is watched for a while first: the stream's own wait, entered when its work
        // is as good as done, returns sooner than one that was asleep for it.  Not in a program
        // that has CUDA's waits yield or block: it wants its cores back.
        const auto t0 = std::chrono::steady_clock::now();
        bool pending = waits_spin();
        while (pending && std::chrono::steady_clock::now() - t0 < std::chrono::microseconds(200))
            for (int i = 0; i < 64 && pending; ++i) pending = *(volatile int *)word == STATUS_PENDING;
        DSQ_CUDA_TRY(cudaStreamSynchronize(s));
        return *(volatile int *)word;
    }
    int host[2] = {0, 0};
    DSQ_CUDA_TRY(cudaMemcpyAsync(host, ws, sizeof(host), cudaMemcpyDeviceToHost, s));
    DSQ_CUDA_TRY(cudaStreamSynchronize(s));
    if (host[DSQ_WS_STATUS]) DSQ_CUDA_TRY(cudaMemsetAsync(ws, 0, sizeof(host), s));
    return host[DSQ_WS_STATUS];
}

}  // extern "C"
