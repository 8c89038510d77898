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

// A request for this grid has been taken up, and other solves may wait a
// moment for its solve: the blocks it will take (0: it will not be batched).
// It stops being expected when its scene (scene_expected) hands the solve over
// or batcher_expect_end is called.
int batcher_expect(SolveBatcher *b, const tursca_grid_desc &d);
void batcher_expect_end(SolveBatcher *b, int blocks);
void scene_expected(tursca_scene *sc, int blocks);
// what is left of it after the request: the blocks still expected
int scene_expected_end(tursca_scene *sc);

}  // namespace tk
