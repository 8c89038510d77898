// The persistent solve (kernels_persist.cu): one cooperative launch solves
// (I - K) x = s from the source to the refined solution, for scenes whose
// values stay on the chip (shared memory) and in L2.
#pragma once

#include <cuda_runtime.h>

#include "kern.h"
#include "persist_plan.h"

namespace tk {

constexpr int kPsMaxJobs = 8;  // solves in one launch
constexpr int kPsRec = 4;      // steps whose coefficients are reported

// what the solve reports (device, read back by the host)
struct PsInfo {
    // iters: BiCGStab steps (two products each) and residuals (one each), so
    // 2 iters - refinements products; state 1: converged, 2: stopped at max_iter, 3: gave up
    int iters, refinements, state, pad;
    double rel, sn;
    // alpha, then beta, of the first kPsRec steps in the compute type, from
    // which the host estimates K's spectral radius (zero at launch; a residual
    // counts in iters and leaves its entry 0, so the first refinement's end shows)
    double rec[2 * kPsRec];
    template <typename T>
    __host__ __device__ T *coef() {
        return reinterpret_cast<T *>(rec);
    }
};
enum { PS_RUNNING = 0, PS_CONVERGED = 1, PS_MAX_ITER = 2, PS_GAVE_UP = 3 };

struct PsJob {
    GridC g;
    const int *tstart;
    const long long *voff;
    const int2 *tpos;    // per template entry: (zz, in-layer haloed offset) of the source (persist_plan.h)
    const int *run;
    const void *val, *s;
    double *x;           // haloed FP64 solution
    float *xh, *xl;      // its FP32 pair, haloed (FP32 scenes)
    void *pub[3];        // haloed exchange vectors (compute type)
    double *part;        // [3][kPsDots][nb] block sums
    unsigned *bar;       // barrier count, zero at launch
    int *status;
    PsInfo *info;
    double rtol;
    int max_iter;
    int block0, nb;      // the job's blocks in the launch
    int nl, tl, nchunk, wpg, it, kcap, near;
};

PsGeom ps_geom(const GridC &g);
// static shared memory of the kernel and its per-block reserve
size_t ps_fixed_smem();

// One launch over jobs of the same compute type and warps per group; the jobs' block0 and nb
// give their shares of the grid, smem the largest of their plans.
cudaError_t launch_persist(cudaStream_t st, const PsJob *jobs, int njobs, int blocks, size_t smem, bool fp64);

// Self-test of the bounded grid barrier: `blocks` blocks of one cooperative
// launch meet at a barrier that expects blocks + (arrive ? 0 : 1) arrivals.
// Returns 0 when the barrier completed, STATUS_TIMEOUT when it gave up (every
// block then returns), -1 on a CUDA error.  Synchronises the stream;
// allocates and frees 8 bytes of device memory.
int barrier_selftest(cudaStream_t st, int blocks, int arrive);

}  // namespace tk
