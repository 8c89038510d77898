// Host interface of the batcher of solves (the serving loop's batched passes
// over K), for host-only code; the job layout is in batch.h.
#pragma once

#include "tursca.h"

namespace tk {

class SolveBatcher;

// A batcher on the current device (its own stream and thread), or null.
SolveBatcher *batcher_create();
void batcher_destroy(SolveBatcher *b);

// launches, jobs run in them, and the largest launch (jobs)
void batcher_stats(SolveBatcher *b, long long *batches, long long *jobs, int *max_jobs);

// Route a scene's solves through b (null: its own launches); FP32 +
// refinement scenes only.
void scene_attach_batcher(tursca_scene *sc, SolveBatcher *b);

}  // namespace tk
