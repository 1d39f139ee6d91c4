// Build plan: every stage of the Hamiltonian build as one grouped launch over
// all target-group pairs, target groups and L2 sets of one or many staged
// Hamiltonians (k_plan.cu).
#pragma once

#include <vector>

#include "hb_api_internal.cuh"

namespace hb {
struct Plan;
}

// Plan over n contexts (same orbital space: equal n_words, n_to and label
// count) writing into outs[i].  Prepares the tensor-core operands when
// precision is HB_MIXED.  Returns HB_OK or an error with *err set.
int plan_create(hb_ctx *const *ctxs, int n, const hb_blocks *outs, int precision, hb::Plan **out, std::string *err,
                cudaStream_t s, int shard_r = 0, int shard_n = 1);
// Phase of the next plan_run of a sharded plan: 1 the contraction only, 2 the
// rest, 0 everything; and whether a plan is the shard (precision, r, n).
void plan_set_phase(hb::Plan *p, int phase);
bool plan_is_shard(const hb::Plan *p, int precision, int r, int n);
// Point the plan's tasks at new output blocks (re-uploads the task tables).
int plan_set_outputs(hb::Plan *p, const hb_blocks *outs, std::string *err, cudaStream_t s);
bool plan_outputs_equal(const hb::Plan *p, const hb_blocks *outs);
int plan_precision(const hb::Plan *p);
bool plan_split_on(const hb::Plan *p);      // the expansion on the tensor cores
// Error word of the context's last build, once: 0 after the call that returned it
// (whichever call of the interface that was), or while the build runs.
int plan_last_error(hb_ctx *ctx);
// The same of the build of p that the caller has just waited for.
int plan_error(hb::Plan *p);
// Before a launch of p on s: zero the words of an error that has been returned.
void plan_clear_error(hb::Plan *p, cudaStream_t s);
// Issue every stage on stream s.  timing: record the stage events (as graph
// event nodes when capture is set).  *launches: kernels launched.
int plan_run(hb::Plan *p, cudaStream_t s, bool timing, bool capture, int *launches, std::string *err);
// Order stream s behind the last build of each context (whatever stream, plan or
// batch it ran by); and record the end of a build of p on s as that of its
// contexts.  Neither does anything on a stream that is being captured.
void plan_wait_last(hb_ctx *const *ctxs, int n, cudaStream_t s);
void plan_mark_built(hb::Plan *p, cudaStream_t s);
// Around what makes tables of a context and its base on s: behind what was made
// of them before, and recorded for what reads them next.
void plan_wait_tables(hb_ctx *ctx, cudaStream_t s);
void plan_mark_tables(hb_ctx *ctx, cudaStream_t s);
// a whole build, replayed as a graph where the same one is repeated
int plan_launch(hb::Plan *p, cudaStream_t s, int *launches, std::string *err);
// After the stream has finished a timed run: per-stage times and counters.
void plan_stats(hb::Plan *p, hb_stats *st);
// Time the result-identical launch-shape candidates of every tunable stage
// (split tile arrangement, class-4 state tile and threads, gamma warp or block
// per key) on this plan's own tasks, keep the fastest, re-upload the tables.
int plan_autotune(hb::Plan *p, cudaStream_t s, std::string *err);
bool plan_tuned(const hb::Plan *p);
// The launch shapes in use, as text.
std::string plan_report(const hb::Plan *p);
void plan_destroy(hb::Plan *p);
