// The batcher of the serving loop's solves (batch.h): a thread that gathers
// the jobs handed to it and launches them together.
//
// Protocol.  A scene's solve records `ready` on its stream, hands the job
// over and blocks until the job is launched.  The thread waits for the
// previous launch to finish (the jobs that arrive meanwhile form the next
// one) and, while a request that can join the oldest job is on its way to its
// solve, up to kBatchGatherUs for it; takes the waiting jobs in order while
// their blocks fit the GPU side by side, makes its stream wait for every job's
// `ready`, launches them in one cooperative kernel, records every job's `done`
// and lets their callers go on: each makes its own stream wait for its `done`.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <deque>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "batch.h"

namespace tk {

class SolveBatcher {
  public:
    int device = 0, nsm = 0;
    cudaStream_t st = nullptr;
    cudaEvent_t last = nullptr;  // the last launch has finished
    std::mutex mu;
    std::condition_variable cv, cv_launched;
    struct Pending {
        const PsJob *job;
        size_t smem;
        cudaEvent_t ready, done;
        bool launched = false;
        BatchResult result = BATCH_NOT_LAUNCHED;
    };
    std::deque<Pending *> q;
    std::vector<int> coming;  // blocks of the solves that are on their way
    std::thread th;
    bool stop = false;
    long long batches = 0, jobs = 0;
    int max_jobs = 0;

    void loop();
    void arrived(int nb);  // a solve that was on its way is not any more
};

void SolveBatcher::loop() {
    cudaSetDevice(device);
    std::unique_lock<std::mutex> lk(mu);
    for (;;) {
        cv.wait(lk, [&] { return stop || !q.empty(); });
        if (q.empty()) return;  // stopping
        lk.unlock();
        bool ok = cudaEventSynchronize(last) == cudaSuccess;
        lk.lock();
        // company for the oldest job: here, or on its way
        cv.wait_for(lk, std::chrono::microseconds(kBatchGatherUs), [&] {
            const int room = nsm - q[0]->job->nb;
            for (size_t i = 1; i < q.size(); ++i)
                if (q[i]->job->nb <= room) return true;
            for (int nb : coming)
                if (nb <= room) return stop;
            return true;
        });
        std::vector<Pending *> take;
        int blocks = 0;
        size_t smem = 0;
        for (auto it = q.begin(); it != q.end() && (int)take.size() < kPsMaxJobs;) {
            if (blocks + (*it)->job->nb <= nsm) {
                blocks += (*it)->job->nb;
                smem = std::max(smem, (*it)->smem);
                take.push_back(*it);
                it = q.erase(it);
            } else {
                ++it;
            }
        }
        lk.unlock();
        std::vector<PsJob> h(take.size());
        int b0 = 0;
        for (size_t i = 0; i < take.size(); ++i) {
            h[i] = *take[i]->job;
            h[i].block0 = b0;
            b0 += h[i].nb;
        }
        const int n = (int)take.size();
        for (Pending *p : take) ok = ok && cudaStreamWaitEvent(st, p->ready, 0) == cudaSuccess;
        ok = ok && launch_persist(st, h.data(), n, blocks, smem, false) == cudaSuccess;
        if (!ok) cudaGetLastError();  // a launch error stays with this thread: the callers run their own launches
        BatchResult result = ok ? BATCH_LAUNCHED : BATCH_NOT_LAUNCHED;
        if (ok) {
            // From here on the solves run: a caller that was told otherwise
            // would run a second one on the same vectors and barrier word.
            // Where an event cannot be recorded, the launch is waited for here.
            for (Pending *p : take) ok = cudaEventRecord(p->done, st) == cudaSuccess && ok;
            ok = cudaEventRecord(last, st) == cudaSuccess && ok;
            if (!ok) {
                cudaGetLastError();
                if (cudaStreamSynchronize(st) != cudaSuccess) result = BATCH_FAILED;
            }
        }
        lk.lock();
        if (result == BATCH_LAUNCHED) {
            batches++;
            jobs += n;
            max_jobs = std::max(max_jobs, n);
        }
        for (Pending *p : take) {
            p->launched = true;
            p->result = result;
        }
        cv_launched.notify_all();
    }
}

SolveBatcher *batcher_create() {
    SolveBatcher *b = new (std::nothrow) SolveBatcher();
    if (!b) return nullptr;
    const bool ok = cudaGetDevice(&b->device) == cudaSuccess &&
                    cudaDeviceGetAttribute(&b->nsm, cudaDevAttrMultiProcessorCount, b->device) == cudaSuccess &&
                    cudaStreamCreateWithFlags(&b->st, cudaStreamNonBlocking) == cudaSuccess &&
                    cudaEventCreateWithFlags(&b->last, cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventRecord(b->last, b->st) == cudaSuccess;
    if (!ok) {
        batcher_destroy(b);
        return nullptr;
    }
    b->th = std::thread([b] { b->loop(); });
    return b;
}

void batcher_destroy(SolveBatcher *b) {
    if (!b) return;
    {
        std::lock_guard<std::mutex> lk(b->mu);
        b->stop = true;
        b->cv.notify_all();
    }
    if (b->th.joinable()) b->th.join();
    if (b->st) cudaStreamSynchronize(b->st);
    if (b->last) cudaEventDestroy(b->last);
    if (b->st) cudaStreamDestroy(b->st);
    delete b;
}

int batcher_expect(SolveBatcher *b, const tursca_grid_desc &d) {
    // (a plan with one group per block has as many blocks as the grid has groups)
    const long long ng = ((long long)d.nx * d.ny + kPsRows - 1) / kPsRows * (d.nz + 1);
    if (!b || d.precision == TURSCA_FP64 || ng > b->nsm || !batch_can_pair(1, (int)ng, b->nsm)) return 0;
    std::lock_guard<std::mutex> lk(b->mu);
    b->coming.push_back((int)ng);
    return (int)ng;
}

void SolveBatcher::arrived(int nb) {
    if (nb <= 0) return;
    const auto it = std::find(coming.begin(), coming.end(), nb);
    if (it != coming.end()) coming.erase(it);
    cv.notify_all();
}

void batcher_expect_end(SolveBatcher *b, int nb) {
    if (!b || nb <= 0) return;
    std::lock_guard<std::mutex> lk(b->mu);
    b->arrived(nb);
}

BatchResult batcher_run(SolveBatcher *b, const PsJob &job, size_t smem, cudaEvent_t ready, cudaEvent_t done,
                        int expected) {
    if (!b || !batch_can_pair(job.nl, job.nb, b->nsm)) {
        batcher_expect_end(b, expected);
        return BATCH_NOT_LAUNCHED;
    }
    SolveBatcher::Pending p;
    p.job = &job;
    p.smem = smem;
    p.ready = ready;
    p.done = done;
    std::unique_lock<std::mutex> lk(b->mu);
    if (b->stop) return BATCH_NOT_LAUNCHED;
    b->q.push_back(&p);
    b->arrived(expected);
    b->cv.notify_all();
    b->cv_launched.wait(lk, [&] { return p.launched; });
    return p.result;
}

void batcher_stats(SolveBatcher *b, long long *batches, long long *jobs, int *max_jobs) {
    std::lock_guard<std::mutex> lk(b->mu);
    if (batches) *batches = b->batches;
    if (jobs) *jobs = b->jobs;
    if (max_jobs) *max_jobs = b->max_jobs;
}

}  // namespace tk
