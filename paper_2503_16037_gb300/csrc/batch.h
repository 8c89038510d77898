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

// A solve is batched when its plan leaves room for another one beside it:
// at most this share of the GPU's blocks.
constexpr double kBatchShare = 0.75;
// How long a solve that is alone waits for one that fits beside it.
constexpr int kBatchGatherUs = 1000;

// Hand one solve to the batcher and block until its batch has been launched:
// the batch waits for `ready` (recorded on the scene's stream once the job's
// inputs are there) and records `done` when it has finished.  False (nothing
// launched) when the job cannot be batched; the caller then runs it itself.
bool batcher_run(SolveBatcher *b, const PsJob &job, size_t smem, cudaEvent_t ready, cudaEvent_t done);

}  // namespace tk
