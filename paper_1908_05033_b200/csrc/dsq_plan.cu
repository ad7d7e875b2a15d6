// Recorded call sequences (dsq_plan.h).
#include "dsq_plan.h"

#include "dsq_launch.h"
#include "dsq_tc_host.h"

namespace {

// A pass whose kernels are short waits for its launches (3 us each of host time,
// against 2 to 4 us of GPU time a layer at batch 1): from the third run on they go as
// one CUDA graph.  Making it takes the third run 0.3 ms of host time more (20 and 52
// launches: 0.36 and 0.46 ms, where the second took 0.09 and 0.19 and the fourth 0.03);
// plans that run once or twice do not pay for it, nor do passes that are being captured.
// Where it cannot be made the launches go one by one, and it is tried again after twice
// as many runs.
constexpr size_t MIN_GRAPH = 4;

int launch_all(const dsq_plan *plan, cudaStream_t s)
{
    void *argv[DsqLaunchRec::MAX_ARGS];
    for (const DsqLaunchRec &r : plan->recs) {
        for (int i = 0; i < r.n_args; ++i)
            argv[i] = const_cast<unsigned char *>(r.args) + r.arg_at[i];
        const int st = dsq_launch_args(r.g, argv, s);
        if (st) return st;
    }
    return DSQ_OK;
}

// nullptr where it cannot be made
cudaGraphExec_t make_graph(const dsq_plan *plan)
{
    const DsqCaptureRelaxed relaxed;
    cudaStream_t s = nullptr;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess &&
        cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        const int st = launch_all(plan, s);
        if (cudaStreamEndCapture(s, &g) != cudaSuccess || st ||
            cudaGraphInstantiate(&exec, g, 0) != cudaSuccess)
            exec = nullptr;
    }
    if (g) cudaGraphDestroy(g);
    if (s) cudaStreamDestroy(s);
    cudaGetLastError();
    return exec;
}

}  // namespace

dsq_plan *&dsq_recording_plan()
{
    static thread_local dsq_plan *plan = nullptr;
    return plan;
}

extern "C" {

int dsq_plan_begin(void)
{
    dsq_plan *&rec = dsq_recording_plan();
    if (rec) return DSQ_ERR_UNSUPPORTED;          // no nesting
    int dev = -1;
    DSQ_CUDA_TRY(cudaGetDevice(&dev));
    rec = new (std::nothrow) dsq_plan;
    if (!rec) return DSQ_ERR_SIZE;
    rec->hooks_generation = dsq_hooks_generation();
    rec->device = dev;
    rec->status = DSQ_OK;
    return DSQ_OK;
}

int dsq_plan_end(dsq_plan **out)
{
    dsq_plan *&rec = dsq_recording_plan();
    if (!rec || !out) return DSQ_ERR_NULL;
    *out = rec->status == DSQ_OK ? rec : nullptr;
    const int st = rec->status;
    if (st != DSQ_OK) delete rec;
    rec = nullptr;
    return st;
}

void dsq_plan_free(dsq_plan *plan) { delete plan; }

int dsq_plan_launches(const dsq_plan *plan) { return plan ? (int)plan->recs.size() : 0; }

int dsq_plan_valid(const dsq_plan *plan)
{
    int dev = -1;
    return plan && plan->hooks_generation == dsq_hooks_generation() &&
           cudaGetDevice(&dev) == cudaSuccess && dev == plan->device;
}

int dsq_plan_run(dsq_plan *plan, void *stream)
{
    if (!plan) return DSQ_ERR_NULL;
    cudaStream_t s = (cudaStream_t)stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (plan->recs.size() >= MIN_GRAPH && cudaStreamIsCapturing(s, &cap) == cudaSuccess &&
        cap == cudaStreamCaptureStatusNone) {
        std::lock_guard<std::mutex> guard(plan->lock);
        if (!plan->graph && ++plan->runs == plan->next_try) {
            plan->graph = make_graph(plan);
            plan->next_try *= 2;
        }
        if (plan->graph) {
            if (cudaGraphLaunch(plan->graph, s) == cudaSuccess) return DSQ_OK;
            cudaGetLastError();
            return DSQ_ERR_CUDA;
        }
    }
    cudaGetLastError();
    return launch_all(plan, s);
}

}  // extern "C"
