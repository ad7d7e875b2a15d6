// The recorded call sequences (csrc/dsq_plan.cu) on a CUDA runtime that is a fake: it
// counts what is launched, made and given back, refuses what a capture in another thread
// would refuse, and fails on demand.  Built and driven by test_plan_host.py.
#include "../paper_1908_05033_b200/csrc/dsq_plan.cu"

#include <cstdlib>
#include <new>

namespace {
struct Fake {
    int launches, graph_launches;          // kernels launched singly, graphs launched
    int captured;                          // kernels launched into the private capture
    int streams, graphs, execs;            // alive
    int instantiate_calls, fail_instantiate, fail_stream;
    int capture_elsewhere, broken;         // another thread's capture, and whether it was broken
    int caller_capturing, mode_changes;
    int no_memory;                         // on the host, for the records
} f;
cudaStreamCaptureMode g_mode = cudaStreamCaptureModeGlobal;
cudaStream_t g_private = nullptr;          // the stream being captured
char g_objects[3];

cudaError_t unsafe()
{
    if (!f.capture_elsewhere || g_mode == cudaStreamCaptureModeRelaxed) return cudaSuccess;
    f.broken = 1;
    return cudaErrorStreamCaptureUnsupported;
}
void kernel(int) { }
}  // namespace

unsigned dsq_hooks_generation() { return 0; }

// (the records are over-aligned)
void *operator new(size_t n, std::align_val_t a)
{
    void *p = f.no_memory ? nullptr : std::aligned_alloc((size_t)a, (n + (size_t)a - 1) / (size_t)a * (size_t)a);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p, std::align_val_t) noexcept { std::free(p); }
void operator delete(void *p, size_t, std::align_val_t) noexcept { std::free(p); }

extern "C" {
Fake *fake() { return &f; }
int fake_mode() { return (int)g_mode; }
int record_launch() { return dsq_launch(kernel, dim3(1), dim3(1), 0, nullptr, 1, 0, 7); }

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m)
{
    std::swap(*m, g_mode);
    ++f.mode_changes;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = f.caller_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    if (f.fail_stream) return cudaErrorMemoryAllocation;
    const cudaError_t e = unsafe();
    if (e != cudaSuccess) return e;
    *s = reinterpret_cast<cudaStream_t>(&g_objects[0]);
    ++f.streams;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { --f.streams; return unsafe(); }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode)
{
    g_private = s;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    g_private = nullptr;
    *g = reinterpret_cast<cudaGraph_t>(&g_objects[1]);
    ++f.graphs;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    ++f.instantiate_calls;
    const cudaError_t r = unsafe();
    if (r != cudaSuccess) return r;
    if (f.fail_instantiate) return cudaErrorMemoryAllocation;
    *e = reinterpret_cast<cudaGraphExec_t>(&g_objects[2]);
    ++f.execs;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { --f.graphs; return unsafe(); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { --f.execs; return unsafe(); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { ++f.graph_launches; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **)
{
    ++(g_private && c->stream == g_private ? f.captured : f.launches);
    return cudaSuccess;
}
}
