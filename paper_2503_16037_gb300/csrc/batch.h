// Solves of several scenes batched into one persistent launch (the serving
// loop's passes over K across requests).
//
// A scene whose solve fits the persistent kernel hands it to the batcher as a
// job.  The batcher's thread gathers the jobs that wait while a launch runs,
// and the next cooperative launch runs them side by side, each on its own
// blocks with its own barrier and its own convergence: a job's bits depend on
// its own plan only, so a result does not depend on what it was batched with.
#pragma once

#include <cuda_runtime.h>

#include "batcher.h"
#include "persist.h"

namespace tk {

// A solve is batched when another one can run beside it: its plan has one
// group per block and takes at most this share of the GPU's blocks.  With two
// or more groups per block a plan takes more than half of them (ps_plan takes
// as few blocks as its largest share allows), and its groups are divided
// among the warps differently, so nothing that is batched fits beside it.
constexpr double kBatchShare = 0.75;
inline bool batch_can_pair(int nl, int nb, int nsm) { return nl == 1 && nb <= kBatchShare * nsm; }

// How long a solve waits for one that can run beside it and whose request is
// on its way (from its start it takes the host about 150 us to hand over its
// solve).  The wait lies inside the time that the solve's own assembly takes
// on the GPU; 1,024 mixed requests on eight workers, the 16 x 16 x 16 ones'
// median service: 1.2 to 1.6 ms with it and without batching alike (2.2 ms
// with 1 ms waited whether company could come or not).
constexpr int kBatchGatherUs = 200;

// Hand one solve to the batcher and block until its batch has been launched:
// the batch waits for `ready` (recorded on the scene's stream once the job's
// inputs are there) and records `done` when it has finished (or has finished
// by then).  Not launched: the job cannot be batched, or its launch was
// refused; the caller runs it itself.  Failed: it was launched and its end is
// unknown (a CUDA error).
// expected: what batcher_expect returned for it (it is expected no longer).
enum BatchResult { BATCH_NOT_LAUNCHED = 0, BATCH_LAUNCHED = 1, BATCH_FAILED = 2 };
BatchResult batcher_run(SolveBatcher *b, const PsJob &job, size_t smem, cudaEvent_t ready, cudaEvent_t done,
                        int expected = 0);

}  // namespace tk
