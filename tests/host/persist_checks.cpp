// Host checks of the persistent solve's plan, for K and K^T of several grid
// shapes: every group is owned once, every slot of every row gathers, from the
// block's tile, the element that was copied from the slot's source, the tile
// and every table stay inside their limits, and shared memory fits.  Built and
// run by tests/test_host_persist_plan.py; returns the number of failing shapes.
#include <cstdio>
#include <string>
#include <vector>

#include "graph.h"
#include "persist_plan.h"

using namespace tg;

namespace {

long check(const Graph &G, int H, int nsm, int es, bool transposed, bool *planned) {
    const int nx = G.nx, ny = G.ny, nz = G.nz, nxp = nx + 2 * H, lp = nxp * (ny + 2 * H), nxy = nx * ny;
    tk::PsGeom g{nx, ny, nz, nxy, (nxy + 127) / 128, H, nxp, lp, G.R};
    Transposed Tt;
    transpose_templates(G, H, Tt);
    const std::vector<int> &ts = transposed ? Tt.tstart : G.tmpl_start;
    std::vector<int> nt(nz + 1);
    for (int z = 0; z <= nz; ++z) nt[z] = ts[z + 1] - ts[z];
    const size_t fixed = 13 * 1024, most = 227 * 1024;
    const tk::PsPlan P = tk::ps_plan(g, nt, es, nsm, most, fixed);
    *planned = P.nb > 0;
    if (P.nb == 0) return 0;
    long bad = 0;
    if (P.nb > nsm || P.run[0] != 0 || P.run[P.nb] != g.gpl * (nz + 1)) ++bad;
    const tk::PsLayout L = tk::ps_layout(es, P.nl, P.tl, P.nchunk, P.wpg, P.it);
    if (P.smem + fixed > most || P.smem != L.k + (size_t)P.kcap * 128 * es) ++bad;
    std::vector<int> seen(g.gpl * (nz + 1), 0);
    for (int b = 0; b < P.nb; ++b) {
        int ns, sq[tk::kPsMaxSeg], sc[tk::kPsMaxSeg], sz[tk::kPsMaxSeg], cb[tk::kPsMaxChunk], cl[tk::kPsMaxChunk],
            gs[tk::kPsMaxGroups];
        const int e0 = P.run[b], e1 = P.run[b + 1];
        const int nc = tk::ps_walk(g, e0, e1, &ns, sq, sc, sz, cb, cl, gs);
        if (e1 <= e0 || e1 - e0 > P.nl || nc < 0 || nc > P.nchunk) {
            ++bad;
            continue;
        }
        for (int c = 0; c < nc; ++c)  // copies inside the haloed vectors and the chunk
            if (cb[c] < 0 || cl[c] > P.tl || cb[c] + cl[c] > (nz + 1) * lp) ++bad;
        for (int e = e0; e < e1; ++e) {
            const int q = tk::ps_strip(g, e), zz = tk::ps_zz(g, e), z = tk::ps_layer(g, zz), s = gs[e - e0];
            seen[z * g.gpl + q]++;
            if (sq[s] != q || tk::ps_padded(nt[z], P.wpg, es) > P.wpg * P.it) ++bad;
            for (int r = 0; r < 128; ++r) {
                const unsigned hp = tk::ps_row_pos(g, q, r);
                const int ro = tk::ps_row_off(g, q, r), rr = q * 128 + r;
                if (((hp & tk::kPsValid) != 0) != (rr < nxy)) ++bad;
                const int y = rr / nx, x = rr - y * nx, rp = z * lp + (y + H) * nxp + x + H;
                if (rr < nxy && z * lp + (int)(hp & tk::kPsPos) != rp) ++bad;
                const int own = tk::ps_off(g, P.tl, sc[s], sz[s], zz, 0) + ro;
                if (own < 0 || own >= nc * P.tl || (rr < nxy && cb[own / P.tl] + own % P.tl != rp)) ++bad;
                for (int i = ts[z]; i < ts[z + 1]; ++i) {
                    int zs, flat;  // source layer, haloed offset from the row
                    if (transposed) {
                        zs = Tt.recv_layer[i];
                        flat = Tt.flat_h[i];
                    } else {
                        zs = G.tmpl[i].sz >= 0 ? G.tmpl[i].sz : nz;
                        flat = (zs - z) * lp + G.tmpl[i].sdy * nxp + G.tmpl[i].sdx;
                    }
                    const int zzs = zs == nz ? 0 : zs + 1, off = flat - (zs - z) * lp;
                    const int o = tk::ps_off(g, P.tl, sc[s], sz[s], zzs, off), j = o + ro;
                    if (o < 0 || o > 65535 || j < 0 || j >= nc * P.tl) {
                        ++bad;
                        continue;
                    }
                    const int c = j / P.tl, in = j % P.tl;
                    if (rr < nxy && (in >= cl[c] || cb[c] + in != rp + flat)) ++bad;
                }
            }
        }
    }
    for (int v : seen) bad += v != 1;
    return bad;
}

// the rounds of the streamed passes: the same checks
long check_rounds(const Graph &G, int H, int nsm, size_t tile_bytes, bool transposed, bool *planned) {
    const int nx = G.nx, ny = G.ny, nz = G.nz, nxp = nx + 2 * H, lp = nxp * (ny + 2 * H), nxy = nx * ny;
    tk::PsGeom g{nx, ny, nz, nxy, (nxy + 127) / 128, H, nxp, lp, G.R};
    Transposed Tt;
    transpose_templates(G, H, Tt);
    const std::vector<int> &ts = transposed ? Tt.tstart : G.tmpl_start;
    std::vector<int> nt(nz + 1);
    for (int z = 0; z <= nz; ++z) nt[z] = ts[z + 1] - ts[z];
    const tk::RunPlan P = tk::run_plan(g, nt, nsm, tile_bytes);
    *planned = P.nb > 0;
    if (P.nb == 0) return 0;
    long bad = 0;
    const int nr = (int)P.round.size() / 4;
    if ((int)P.first.size() != P.nb + 1 || P.first[0] != 0 || P.first[P.nb] != nr || P.tl % 4 ||
        (size_t)P.nc * P.tl * 4 > tile_bytes)
        ++bad;
    std::vector<int> seen(g.gpl * (nz + 1), 0);
    for (int r = 0; r < nr; ++r) {
        const int e0 = P.round[4 * r], n = P.round[4 * r + 1], c0 = P.round[4 * r + 2], nc = P.round[4 * r + 3];
        if (n < 1 || n > tk::kRunGroups || nc > P.nc) ++bad;
        for (int c = 0; c < nc; ++c) {
            const int b = P.chunk[2 * (c0 + c)], l = P.chunk[2 * (c0 + c) + 1];
            if (b < 0 || l > P.tl || b + l > (nz + 1) * lp || (nxp % 4 == 0 && (b % 4 || l % 4))) ++bad;
        }
        for (int i = 0; i < n; ++i) {
            const int e = e0 + i, q = tk::ps_strip(g, e), zz = tk::ps_zz(g, e), z = tk::ps_layer(g, zz);
            seen[z * g.gpl + q]++;
            const int own = P.own[r * tk::kRunGroups + i];
            for (int row = 0; row < 128; ++row) {
                const int ro = tk::ps_row_off(g, q, row), rr = q * 128 + row, y = rr / nx, x = rr - y * nx;
                const int rp = z * lp + (y + H) * nxp + x + H;
                for (int k = ts[z]; k < ts[z + 1]; ++k) {
                    const int zs = transposed ? Tt.recv_layer[k] : (G.tmpl[k].sz >= 0 ? G.tmpl[k].sz : nz);
                    const int flat = transposed ? Tt.flat_h[k]
                                                : (zs - z) * lp + G.tmpl[k].sdy * nxp + G.tmpl[k].sdx;
                    const int zzs = zs == nz ? 0 : zs + 1;
                    const int j = (own + zzs - zz) * P.tl + flat - (zs - z) * lp + H * nxp + H + ro;
                    const int c = j / P.tl, in = j % P.tl;
                    if (j < 0 || c >= nc) {
                        ++bad;
                        continue;
                    }
                    if (rr < nxy && (in >= P.chunk[2 * (c0 + c) + 1] || P.chunk[2 * (c0 + c)] + in != rp + flat)) ++bad;
                }
            }
        }
    }
    for (int v : seen) bad += v != 1;
    return bad;
}

}  // namespace

int main() {
    const int shapes[][4] = {{64, 64, 32, 2}, {45, 37, 29, 2}, {48, 48, 32, 2}, {21, 19, 9, 2}, {13, 11, 7, 1},
                             {9, 10, 2, 2},   {5, 5, 1, 1},    {200, 7, 3, 2},  {8, 8, 8, 1},   {16, 16, 16, 2},
                             {127, 33, 6, 2}, {96, 96, 32, 2}, {128, 128, 2, 2}, {130, 61, 12, 2}};
    int failing = 0;
    for (const auto &s : shapes) {
        Graph G;
        const std::string e = build_graph(G, s[0], s[1], s[2], 0.05, 0.05, 0.1, s[3], 512);
        if (!e.empty()) {
            std::printf("%dx%dx%d: %s\n", s[0], s[1], s[2], e.c_str());
            ++failing;
            continue;
        }
        for (int es : {4, 8})
            for (int t = 0; t < 2; ++t) {
                bool planned = false;
                const long bad = check(G, s[3], 152, es, t != 0, &planned);
                std::printf("%dx%dx%d R%d %s %d bytes: %s, %ld bad\n", s[0], s[1], s[2], s[3], t ? "K^T" : "K", es,
                            planned ? "planned" : "no plan", bad);
                failing += bad != 0;
            }
        for (int t = 0; t < 2; ++t)
            for (size_t bytes : {(size_t)46 * 1024, (size_t)20 * 1024}) {
                bool planned = false;
                const long bad = check_rounds(G, s[3], 152, bytes, t != 0, &planned);
                std::printf("%dx%dx%d R%d %s rounds: %s, %ld bad\n", s[0], s[1], s[2], s[3], t ? "K^T" : "K",
                            planned ? "planned" : "none", bad);
                failing += bad != 0;
            }
    }
    return failing;
}
