// Every kernel launch of the library's entry points goes through dsq_launch():
// it launches on the caller's stream or, while the calling thread records a
// plan (dsq_plan.h), appends the finished launch - kernel, grid, attributes and
// a copy of every argument - to that plan.  Internal to the library.
#pragma once

#include <cuda_runtime.h>

#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "dsq_common.cuh"

#define DSQ_HIDDEN __attribute__((visibility("hidden")))

// current values of the process-wide hooks (csrc/dsq_hooks.h)
struct DsqLaunchHooks {
    int pdl;                    // programmatic dependent launch on / off
    unsigned long long wait_ns; // limit of the device-side waits
    int skip_b_round;           // test hook, -1 = off
    int window3;                // dsq_set_conv3_window
    int w8;                     // dsq_set_conv3_expanded_weights
};
DSQ_HIDDEN DsqLaunchHooks dsq_launch_hooks();
// a number that changes whenever a hook is set
DSQ_HIDDEN unsigned dsq_hooks_generation();

// how a kernel is launched
struct DsqGrid {
    const void *func;
    dim3 grid, block;
    size_t smem;
    int pdl;                  // programmatic dependent launch
    int cluster;              // CTAs per cluster (0 or 1: none)
};

// one recorded launch: the arguments lie one behind the other at the offsets
// `arg_at` of `args` (64-byte aligned: tensor maps)
struct DsqLaunchRec {
    static constexpr int MAX_ARGS = 20;
    DsqGrid g;
    int n_args;
    unsigned short arg_at[MAX_ARGS];
    alignas(64) unsigned char args[1024];
};

// While one lives, calls that a stream capture anywhere in the process would forbid
// (creating and destroying streams, graphs, page-locked memory) are open to this
// thread and leave that capture alone.  Only around calls that enqueue nothing on a
// stream of the caller's.
struct DsqCaptureRelaxed {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    bool changed;
    DsqCaptureRelaxed() : changed(cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess) {}
    ~DsqCaptureRelaxed()
    {
        if (changed) cudaThreadExchangeStreamCaptureMode(&mode);
    }
    DsqCaptureRelaxed(const DsqCaptureRelaxed &) = delete;
    DsqCaptureRelaxed &operator=(const DsqCaptureRelaxed &) = delete;
};

struct dsq_plan {
    std::vector<DsqLaunchRec> recs;
    unsigned hooks_generation = 0;      // of the process-wide hooks when recorded
    int device = -1;
    int status = DSQ_OK;                // first failure while recording
    // the launches as a CUDA graph (dsq_plan_run); guarded by the lock
    std::mutex lock;
    int64_t runs = 0, next_try = GRAPH_AFTER;
    cudaGraphExec_t graph = nullptr;
    static constexpr int GRAPH_AFTER = 3;
    ~dsq_plan()
    {
        if (!graph) return;
        const DsqCaptureRelaxed relaxed;
        cudaGraphExecDestroy(graph);
    }
};

// the plan the calling thread records into, or nullptr
DSQ_HIDDEN dsq_plan *&dsq_recording_plan();

// Whether a kernel launched now may read a layer's constants (packed weights, scales,
// biases) before griddepcontrol.wait.  Every kernel of the library waits for the
// kernels ahead of it before it lets the next one start (or is launched without that
// attribute and starts behind them), so when a kernel starts,
// everything but its immediate predecessor has completed and is visible.  Behind
// another launch of the same plan that predecessor is a layer of the network, which
// writes activations only; elsewhere it may be what wrote the constants.
inline int dsq_early_constants()
{
    const dsq_plan *plan = dsq_recording_plan();
    return plan && !plan->recs.empty();
}

inline int dsq_launch_args(const DsqGrid &g, void *const *argv, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g.grid;
    cfg.blockDim = g.block;
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (g.cluster > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = (unsigned)g.cluster;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        ++na;
    }
    if (g.pdl) {
        // the kernel waits for its predecessors itself (griddepcontrol.wait)
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = (unsigned)na;
    if (cudaLaunchKernelExC(&cfg, g.func, const_cast<void **>(argv)) != cudaSuccess) {
        cudaGetLastError();
        return DSQ_ERR_CUDA;
    }
    return DSQ_OK;
}

inline int dsq_record_args(dsq_plan *plan, const DsqGrid &g, int n, void *const *argv,
                           const size_t *size, const size_t *align)
{
    DsqLaunchRec r;
    r.g = g;
    r.n_args = n;
    size_t at = 0;
    for (int i = 0; i < n; ++i) {
        at = (at + align[i] - 1) / align[i] * align[i];
        if (i >= DsqLaunchRec::MAX_ARGS || at + size[i] > sizeof(r.args)) {
            plan->status = DSQ_ERR_UNSUPPORTED;
            return DSQ_ERR_UNSUPPORTED;
        }
        r.arg_at[i] = (unsigned short)at;
        std::memcpy(r.args + at, argv[i], size[i]);
        at += size[i];
    }
    try {
        plan->recs.push_back(r);
    } catch (const std::bad_alloc &) {        // (no entry point throws)
        plan->status = DSQ_ERR_SIZE;
        return DSQ_ERR_SIZE;
    }
    return DSQ_OK;
}

template <class T> struct DsqSame { typedef T type; };   // (no deduction from the arguments)

// arguments are converted to the kernel's parameter types; returns a dsq_status
template <class... P>
inline int dsq_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                      int pdl, int cluster,
                      typename DsqSame<std::remove_cv_t<P>>::type... a)
{
    const DsqGrid g = {(const void *)kernel, grid, block, smem, pdl, cluster};
    void *argv[] = {(void *)&a...};
    dsq_plan *plan = dsq_recording_plan();
    if (!plan) return dsq_launch_args(g, argv, s);
    const size_t size[] = {sizeof(a)...}, align[] = {alignof(decltype(a))...};
    return dsq_record_args(plan, g, (int)sizeof...(P), argv, size, align);
}
