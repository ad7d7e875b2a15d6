/*
 * dsq_plan.h - recorded call sequences.  Not part of the public interface: the
 * Python layer uses it so that a whole stack is one call.
 *
 * Between dsq_plan_begin() and dsq_plan_end() the calling thread's entry points
 * validate and choose as always, but their kernel launches are appended to a
 * plan instead of going to a stream.  dsq_plan_run() launches them in order.
 * A plan holds the device pointers it was recorded with; the caller keeps the
 * buffers alive.  Calls that enqueue anything but kernels (memsets, copies) are
 * not for recording, nor are calls that write what a later one takes as weights,
 * scales or biases (those may be read while the launch before is still running).
 *
 * The launches of an ended plan do not change: several threads may run it, each
 * on its own stream.  The third run makes a CUDA graph of them (under a lock, on a
 * stream of its own, whatever any thread is capturing) that later runs launch;
 * CUDA may take memory for it, the device's included, until the plan is freed.  A
 * run into a stream that is being captured launches one by one.
 */
#ifndef DSQ_PLAN_H_
#define DSQ_PLAN_H_

#ifdef __cplusplus
extern "C" {
#endif

typedef struct dsq_plan dsq_plan;

int dsq_plan_begin(void);
/* *out = the plan (NULL when a call in between could not be recorded) */
int dsq_plan_end(dsq_plan **out);
void dsq_plan_free(dsq_plan *plan);
int dsq_plan_launches(const dsq_plan *plan);
/* 1 while the plan may run: the process-wide hooks are as they were when it
 * was recorded and the current device is the plan's */
int dsq_plan_valid(const dsq_plan *plan);
int dsq_plan_run(dsq_plan *plan, void *stream);

#ifdef __cplusplus
}
#endif
#endif /* DSQ_PLAN_H_ */
