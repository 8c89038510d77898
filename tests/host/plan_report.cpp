// Which driver the automatic solve takes: for each shape and precision the
// persistent solve's plan of K and of K^T, else whether the FP32 passes run in
// rounds.  Built and run by tests/test_host_plan_choice.py.
#include <cstdio>
#include <vector>

#include "graph.h"
#include "persist_plan.h"

using namespace tg;

int main(int argc, char **argv) {
    for (int a = 1; a + 3 < argc; a += 4) {
        int s[4];
        for (int i = 0; i < 4; ++i) std::sscanf(argv[a + i], "%d", &s[i]);
        Graph G;
        if (!build_graph(G, s[0], s[1], s[2], 0.05, 0.05, 0.1, s[3], 512).empty()) return 1;
        const int H = s[3], nxp = G.nx + 2 * H, lp = nxp * (G.ny + 2 * H), nxy = G.nx * G.ny;
        const tk::PsGeom g{G.nx, G.ny, G.nz, nxy, (nxy + 127) / 128, H, nxp, lp, G.R};
        Transposed T;
        transpose_templates(G, H, T);
        std::printf("%dx%dx%d R%d:", s[0], s[1], s[2], s[3]);
        for (int t = 0; t < 2; ++t) {
            const std::vector<int> &ts = t ? T.tstart : G.tmpl_start;
            std::vector<int> nt(G.nz + 1);
            for (int z = 0; z <= G.nz; ++z) nt[z] = ts[z + 1] - ts[z];
            for (int es : {4, 8}) {
                const bool plan = tk::ps_plan(g, nt, es, 152, 227 * 1024, 13 * 1024).nb > 0;
                const bool rounds = es == 4 && !plan && tk::run_plan(g, nt, 152, 46 * 1024).nb > 0;
                std::printf(" %s/%d=%s", t ? "KT" : "K", 8 * es, plan ? "persistent" : rounds ? "rounds" : "passes");
            }
        }
        std::printf("\n");
    }
    return 0;
}
