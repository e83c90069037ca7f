// Reach of the restriction stencils (Sec. 4.2-4.3) in neighbour hops of the fine
// level, on the library's own host tables: for every coarse edge and each of its ends k,
// the fine points whose fluxes and divergences the restricted flux reads (R_F), the
// halves its Coriolis tendency reads (R_u) and the node its B reads, measured from the
// points that are live when k is covered (the fine node at k and M_k).  An edge counts by
// the node of the element that owns it.  Every owner is checked to be an end of its
// edge and a vertex of its triangles.  Prints the largest distance.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "grid.h"

using namespace sww;

int main(int argc, char** argv) {
    const int jmin = std::atoi(argv[1]), jmax = std::atoi(argv[2]);
    Hierarchy H;
    build_hierarchy(H, jmin, jmax, 4, 6.371e6, 7.292e-5);
    int worst = 0;
    for (int j = jmin; j < jmax; ++j) {
        const HostLevel &C = H.lv[j], &F = H.lv[j + 1];
        for (int64_t e = 0; e < F.E; ++e)
            if (F.en[0][e] != e % F.nelem && F.en[1][e] != e % F.nelem) worst = 99;
        for (int64_t t = 0; t < F.T; ++t) {
            const int v = int(t % F.nelem);
            if (F.tn[0][t] != v && F.tn[1][t] != v && F.tn[2][t] != v) worst = 99;
        }
        std::vector<int> dist(F.N, -1), seen;
        std::vector<std::vector<int>> edges(C.N);
        for (int64_t e = 0; e < C.E; ++e) edges[C.en[0][e]].push_back(int(e)), edges[C.en[1][e]].push_back(int(e));
        for (int64_t k = 0; k < C.N; ++k) {
            seen.clear();
            auto put = [&](int v, int d) {
                if (dist[v] < 0) dist[v] = d, seen.push_back(v);
            };
            put(C.c2f[k], 0);
            for (int q = 0; q < 12; ++q)
                if (C.mk_i[q][k] >= 0) put(C.mk_i[q][k], 0);
            for (size_t i = 0; i < seen.size(); ++i)
                if (dist[seen[i]] < 8)
                    for (int r = 0; r < F.deg[seen[i]]; ++r) put(F.ring_n[r][seen[i]], dist[seen[i]] + 1);
            auto at = [&](int v) { worst = std::max(worst, dist[v] < 0 ? 99 : dist[v]); };
            for (int e : edges[k]) {
                for (int s = 0; s < RF_F; ++s)
                    if (C.rf_fw[s][e] != 0.0) at(int(C.rf_fi[s][e] % F.nelem));
                for (int s = 0; s < RF_C; ++s)
                    if (C.rf_cw[s][e] != 0.0) at(C.rf_ci[s][e]);
                at(int(C.half[0][e] % F.nelem)), at(int(C.half[1][e] % F.nelem));
            }
            for (int v : seen) dist[v] = -1;
        }
    }
    std::printf("%d\n", worst);
    return 0;
}
