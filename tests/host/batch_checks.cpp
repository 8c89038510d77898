// Host checks of the batcher of solves (batch.cu) against a stand-in for the
// CUDA runtime and for the launch: which solves it takes, that a solve alone does
// not wait, that one waits a moment for company that is on its way, and what
// happens when an event cannot be recorded.
// Built and run by tests/test_host_batcher.py; returns the number of failures.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdio>
#include <string>
#include <thread>
#include <vector>

#include "batch.h"
#include "graph.h"

namespace {
constexpr int kSms = 152;
int failures = 0;
std::atomic<int> last_jobs{0}, launches{0}, record_fails{0}, syncs_after_launch{0};
std::atomic<bool> launch_pending{false}, sync_fails{false};
void check(bool ok, const char *what) {
    std::printf("%s: %s\n", ok ? "ok" : "FAIL", what);
    failures += !ok;
}
}  // namespace

// ---- the runtime: every stream is empty, every event has happened
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = kSms, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = (cudaStream_t)1, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    if (launch_pending) ++syncs_after_launch;
    launch_pending = false;
    return sync_fails ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = (cudaEvent_t)1, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) {
    if (record_fails > 0) return --record_fails, cudaErrorMemoryAllocation;
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }

namespace tk {
cudaError_t launch_persist(cudaStream_t, const PsJob *, int njobs, int, size_t, bool) {
    last_jobs = njobs;
    ++launches;
    launch_pending = true;
    return cudaSuccess;
}
}  // namespace tk

int main() {
    // the plans of the serving shapes and others: two solves that are both
    // batched and small enough for company fit side by side, the rest never do
    const int shapes[][4] = {{16, 16, 16, 2}, {24, 24, 16, 2}, {32, 32, 24, 2}, {48, 48, 32, 2}, {64, 64, 32, 2},
                             {20, 20, 20, 2}, {24, 24, 24, 2}, {32, 32, 16, 2}, {40, 40, 24, 2}, {8, 8, 8, 1},
                             {21, 19, 9, 2},  {13, 11, 7, 1},  {32, 32, 18, 2}, {28, 28, 28, 1}};
    tk::SolveBatcher *b = tk::batcher_create();
    if (!b) return 1;
    std::vector<tk::PsJob> taken, refused;
    for (const auto &s : shapes) {
        tg::Graph G;
        if (!tg::build_graph(G, s[0], s[1], s[2], 0.05, 0.05, 0.1, s[3], 512).empty()) return 1;
        const int H = s[3], nxp = G.nx + 2 * H, lp = nxp * (G.ny + 2 * H), nxy = G.nx * G.ny;
        std::vector<int> nt(G.nz + 1);
        for (int z = 0; z <= G.nz; ++z) nt[z] = G.tmpl_start[z + 1] - G.tmpl_start[z];
        const tk::PsPlan P = tk::ps_plan(tk::PsGeom{G.nx, G.ny, G.nz, nxy, (nxy + 127) / 128, H, nxp, lp, G.R}, nt, 4,
                                         kSms, 227 * 1024, 13 * 1024);
        if (P.nb == 0) continue;
        tk::PsJob J{};
        J.nb = P.nb;
        J.nl = P.nl;
        J.wpg = P.wpg;
        const bool ran = (int)tk::batcher_run(b, J, P.smem, nullptr, nullptr) != 0;
        std::printf("%dx%dx%d R%d: %d blocks, %d groups each, %d warps a group: %s\n", s[0], s[1], s[2], s[3], P.nb, P.nl,
                    P.wpg, ran ? "batched" : "on its own");
        (ran ? taken : refused).push_back(J);
    }
    int smallest = kSms;
    for (const tk::PsJob &J : taken) smallest = std::min(smallest, J.nb);
    bool pairs = true, apart = true, same = true;
    for (const tk::PsJob &J : taken) {
        pairs = pairs && J.nb + smallest <= kSms;
        same = same && J.wpg == taken[0].wpg;
    }
    for (const tk::PsJob &J : refused)
        for (const auto *v : {&taken, &refused})
            for (const tk::PsJob &K : *v) apart = apart && (J.nb + K.nb > kSms || J.wpg != K.wpg || J.nb > 0.75 * kSms);
    check(!taken.empty() && pairs && same, "every solve that is batched can have company");
    check(!refused.empty() && apart, "no other solve could");

    // a solve alone
    tk::PsJob J{};
    J.nb = 34;
    J.nl = 1;
    J.wpg = 16;
    double best = 1e9;
    for (int i = 0; i < 20; ++i) {
        const auto t0 = std::chrono::steady_clock::now();
        if ((int)tk::batcher_run(b, J, 0, nullptr, nullptr) != 1) return 1;
        best = std::min(best, std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count());
    }
    std::printf("a solve alone: %.0f us from hand-over to launch\n", best);
    check(best < 500.0, "a solve alone is launched at once");

    // company that is on its way and arrives
    tursca_grid_desc d{};
    d.nx = d.ny = d.nz = 16;
    d.precision = TURSCA_FP32_REFINE;
    bool together = false;
    for (int i = 0; i < 20 && !together; ++i) {  // (a thread may start too late now and then)
        const int expected = tk::batcher_expect(b, d);
        if (expected != 34) return 1;
        std::thread other([&] { tk::batcher_run(b, J, 0, nullptr, nullptr, expected); });
        tk::batcher_run(b, J, 0, nullptr, nullptr);
        other.join();
        together = last_jobs == 2;
    }
    check(together, "a solve waits for one that is on its way");

    // company that never arrives, and company that stops being expected
    for (int gone = 0; gone < 2; ++gone) {
        best = 1e9;
        for (int i = 0; i < 20; ++i) {
            const int expected = tk::batcher_expect(b, d);
            if (gone) tk::batcher_expect_end(b, expected);
            const auto t0 = std::chrono::steady_clock::now();
            tk::batcher_run(b, J, 0, nullptr, nullptr);
            best = std::min(best,
                            std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count());
            if (!gone) tk::batcher_expect_end(b, expected);
        }
        std::printf("company %s: %.0f us\n", gone ? "gone" : "late", best);
        check(best < (gone ? 150.0 : 900.0), "and not longer than it may");
    }
    d.nx = d.ny = 32;  // two groups per block: nothing fits beside it
    d.nz = 24;
    check(tk::batcher_expect(b, d) == 0, "no one waits for a solve that is not batched");
    // an event that cannot be recorded behind a launch: the caller must not
    // launch its own solve beside the one that runs
    for (int at = 1; at <= 2; ++at) {
        launches = syncs_after_launch = 0;
        launch_pending = false;
        record_fails = at;
        const int r = (int)tk::batcher_run(b, J, 0, nullptr, nullptr);
        check(launches == 1 && r != 0, "a solve that was launched is not reported as not launched");
        check(syncs_after_launch == 1, "its launch has ended before the caller goes on");
        record_fails = 0;
    }
    record_fails = 1;
    sync_fails = true;
    check((int)tk::batcher_run(b, J, 0, nullptr, nullptr) == 2, "one whose end is unknown is a failure");
    sync_fails = false;
    tk::batcher_destroy(b);
    return failures;
}
