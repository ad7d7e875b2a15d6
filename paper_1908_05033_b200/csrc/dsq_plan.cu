// Recorded call sequences (dsq_plan.h).
#include "dsq_plan.h"

#include "dsq_launch.h"
#include "dsq_tc_host.h"

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

int dsq_plan_run(const dsq_plan *plan, void *stream)
{
    if (!plan) return DSQ_ERR_NULL;
    void *argv[DsqLaunchRec::MAX_ARGS];
    for (const DsqLaunchRec &r : plan->recs) {
        for (int i = 0; i < r.n_args; ++i)
            argv[i] = const_cast<unsigned char *>(r.args) + r.arg_at[i];
        const int st = dsq_launch_args(r.g, argv, (cudaStream_t)stream);
        if (st) return st;
    }
    return DSQ_OK;
}

}  // extern "C"
