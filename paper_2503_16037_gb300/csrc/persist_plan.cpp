// Plan of the persistent solve (persist_plan.h).
#include "persist_plan.h"

#include <algorithm>

namespace tk {

// Values the blocks stream on every product, beyond shared memory: up to
// kPsL2Bytes of them stay in L2 (measured on GB300, a set read with a fixed
// mapping of blocks to data: 11 to 16 TB/s up to 100 MB; 130 MB and more fall
// to 7 TB/s, HBM's rate), the rest is read from HBM past it (150 MB: 16.8 us
// with 80 MB kept and 70 MB marked evict-first, 21.8 us without).  Above
// kPsMaxBytes a product is bound by HBM either way and the passes, which
// need no exchange of halves, take over.
constexpr double kPsL2Bytes = 80e6, kPsMaxBytes = 200e6;

// Groups of each of nb blocks, in strip order: equal shares of slots (a
// group's finish costs about 12 slots), one group each at least.
static std::vector<int> equal_shares(const PsGeom &g, const std::vector<int> &nt, int nb) {
    const long long ng = (long long)g.gpl * (g.nz + 1);
    auto cost = [&](long long e) { return nt[ps_layer(g, ps_zz(g, (int)e))] + 12.0; };
    double total = 0.0, acc = 0.0;
    for (long long e = 0; e < ng; ++e) total += cost(e);
    std::vector<int> run(nb + 1, 0);
    long long e = 0;
    for (int b = 0; b < nb; ++b) {
        run[b] = (int)e;
        const double target = total * (b + 1) / nb;
        const long long most = ng - (nb - 1 - b);  // leave a group for every later block
        do {
            acc += cost(e);
            ++e;
        } while (e < most && acc + 0.5 * cost(e) <= target);
    }
    run[nb] = (int)ng;
    return run;
}

PsPlan ps_plan(const PsGeom &g, const std::vector<int> &nt, int es, int nsm, size_t smem_max, size_t fixed_smem) {
    PsPlan P;
    const int nz1 = g.nz + 1;
    const long long ng = (long long)g.gpl * nz1;
    if (nsm <= 0 || ng <= 0 || ng > (long long)kPsMaxGroups * nsm) return P;
    if ((long long)g.lp >= (1ll << 27) || (long long)g.lp * nz1 >= (1ll << 31)) return P;
    int ntmax = 0;
    for (int v : nt) ntmax = std::max(ntmax, v);
    // as few blocks as the largest share allows: 200 groups on 152 SMs are
    // two per block either way, and 100 blocks meet sooner than 152
    const int per = (int)((ng + nsm - 1) / nsm);
    const int nb = (int)((ng + per - 1) / per);
    auto slots = [&](long long e) { return nt[ps_layer(g, ps_zz(g, (int)e))]; };
    std::vector<int> run = equal_shares(g, nt, nb);
    int nl = 0, nchunk = 0, tl = 0;
    for (int q = 0; q < g.gpl; ++q) tl = std::max(tl, (ps_y1(g, q) - ps_y0(g, q) + 1 + 2 * g.H) * g.nxp);
    for (int b = 0; b < nb; ++b) {
        int ns, sq[kPsMaxSeg], sc[kPsMaxSeg], sz[kPsMaxSeg], cb[kPsMaxChunk], cl[kPsMaxChunk], gs[kPsMaxGroups];
        const int nc = ps_walk(g, run[b], run[b + 1], &ns, sq, sc, sz, cb, cl, gs);
        if (nc < 0) return P;
        nl = std::max(nl, run[b + 1] - run[b]);
        nchunk = std::max(nchunk, nc);
    }
    // Groups run side by side, each on its own warps, with no barrier between
    // them: 16 warps on one group of a small scene, two per group where a
    // block has six or more (measured on the 64 x 64 x 32 plume, 7 groups a
    // block: 6.4 us for the products of one pass; all 16 warps sharing every
    // group, with a barrier per pair of groups, 10.6 us).
    const int wpg = nl >= 6 ? 2 : kPsW / nl;
    const int it = (ps_padded(ntmax, wpg, es) / wpg + 7) / 8 * 8;
    if ((long long)(nchunk + 1) * tl >= (1 << 16)) return P;
    const PsLayout L = ps_layout(es, nl, tl, nchunk, wpg, it);
    if (L.k + fixed_smem >= smem_max) return P;
    const size_t row = (size_t)kPsRows * es;
    int kcap = (int)((smem_max - fixed_smem - L.k) / row);
    long long most = 0;
    double streamed = 0.0;
    for (int b = 0; b < nb; ++b) {
        const int er = ps_first_resident(run[b], run[b + 1], kcap, wpg, es, slots);
        long long kept = 0;
        for (int k = run[b]; k < run[b + 1]; ++k) {
            if (k < er)
                streamed += (double)slots(k) * row;
            else
                kept += ps_padded(slots(k), wpg, es);
        }
        most = std::max(most, kept);
    }
    if (streamed > kPsMaxBytes) return P;
    kcap = (int)std::min<long long>(kcap, most);
    P.nb = nb;
    P.nl = nl;
    P.tl = tl;
    P.nchunk = nchunk;
    P.wpg = wpg;
    P.it = it;
    P.kcap = kcap;
    P.near = streamed <= 1.1 * kPsL2Bytes ? 1 << 30 : (int)(kPsL2Bytes / nb / row);
    P.smem = L.k + (size_t)kcap * row;
    P.run = std::move(run);
    return P;
}

RunPlan run_plan(const PsGeom &g, const std::vector<int> &nt, int nsm, size_t tile_bytes) {
    RunPlan P;
    const long long ng = (long long)g.gpl * (g.nz + 1);
    if (nsm <= 0 || ng < nsm || ng >= (1ll << 30) || (long long)g.lp * (g.nz + 1) >= (1ll << 31)) return P;
    for (int q = 0; q < g.gpl; ++q) P.tl = std::max(P.tl, (ps_y1(g, q) - ps_y0(g, q) + 1 + 2 * g.H) * g.nxp);
    P.tl = (P.tl + 3) / 4 * 4;
    const int nc = (int)std::min<size_t>(kRunMaxChunk, tile_bytes / ((size_t)P.tl * sizeof(float)));
    if (nc < 2 * g.R + 2) return P;  // not even two groups at a time
    const std::vector<int> run = equal_shares(g, nt, nsm);
    P.first.push_back(0);
    for (int b = 0; b < nsm; ++b) {
        for (int e = run[b]; e < run[b + 1];) {
            int ns, sq[kPsMaxSeg], sc[kPsMaxSeg], sz[kPsMaxSeg], cb[kPsMaxChunk], cl[kPsMaxChunk], gs[kPsMaxGroups];
            // rounds of equal size: a short last round would stream with few warps
            const int left = run[b + 1] - e, rounds = (left + kRunGroups - 1) / kRunGroups;
            int n = (left + rounds - 1) / rounds, c = 0;
            for (; n > 0; --n) {
                c = ps_walk(g, e, e + n, &ns, sq, sc, sz, cb, cl, gs);
                if (c >= 0 && c <= nc) break;
            }
            if (n == 0) return RunPlan();
            P.round.insert(P.round.end(), {e, n, (int)P.chunk.size() / 2, c});
            for (int k = 0; k < c; ++k) P.chunk.insert(P.chunk.end(), {cb[k], cl[k]});
            for (int i = 0; i < kRunGroups; ++i)
                P.own.push_back(i < n ? sc[gs[i]] + ps_zz(g, e + i) - sz[gs[i]] : 0);
            e += n;
        }
        P.first.push_back((int)P.round.size() / 4);
        P.rmax = std::max(P.rmax, P.first[b + 1] - P.first[b]);
    }
    if (P.rmax > kRunMaxRounds || g.nz > kRunMaxNz) return RunPlan();
    double values = 0.0;
    for (int z = 0; z <= g.nz; ++z) values += (double)nt[z] * g.gpl * kPsRows * sizeof(float);
    P.near = (int)(P.round.size() / 4 * std::min(1.0, kPsL2Bytes / values)) / nsm;
    P.nc = nc;
    P.nb = nsm;
    return P;
}

}  // namespace tk
