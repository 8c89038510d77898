// Plan of the persistent solve (persist_plan.h).
#include "persist_plan.h"

#include <algorithm>

namespace tk {

// Values a block streams from L2 on every product, over all blocks: above
// this the lines would not stay in L2 (measured on GB300: a set read with a
// fixed mapping of blocks to data streams at 6 TB/s up to 100 MB and at
// 2.3 TB/s from 120 MB on), and a pass per launch is the better form.
constexpr double kPsL2Bytes = 88e6;

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
    // equal shares of slots (a group's finish costs about 12 slots), one group each at least
    auto slots = [&](long long e) { return nt[ps_layer(g, ps_zz(g, (int)e))]; };
    double total = 0.0, acc = 0.0;
    for (long long e = 0; e < ng; ++e) total += slots(e) + 12.0;
    std::vector<int> run(nb + 1, 0);
    long long e = 0;
    for (int b = 0; b < nb; ++b) {
        run[b] = (int)e;
        const double target = total * (b + 1) / nb;
        const long long most = ng - (nb - 1 - b);  // leave a group for every later block
        do {
            acc += slots(e) + 12.0;
            ++e;
        } while (e < most && acc + 0.5 * (slots(e) + 12.0) <= target);
    }
    run[nb] = (int)ng;
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
    if (streamed > kPsL2Bytes) return P;
    kcap = (int)std::min<long long>(kcap, most);
    P.nb = nb;
    P.nl = nl;
    P.tl = tl;
    P.nchunk = nchunk;
    P.wpg = wpg;
    P.it = it;
    P.kcap = kcap;
    P.smem = L.k + (size_t)kcap * row;
    P.run = std::move(run);
    return P;
}

}  // namespace tk
