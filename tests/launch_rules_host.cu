// Evaluates the launch rules of crbm_launch.h on the host, used only by tests.  Reads "rule arguments" lines on
// stdin and prints each rule's choice.
#include <cstdio>
#include <cstring>

#include "crbm_launch.h"

static crbm::Geometry lattice(int L, int Lc) {
    crbm::Geometry g{};
    g.L = L;
    g.Lc = Lc;
    g.W = (L + 1) / 2;
    g.Wc = (Lc + 1) / 2;
    g.N = L * Lc;
    g.n_cells = g.W * g.Wc;
    g.canonical = 1;
    return g;
}

int main() {
    char rule[32];
    while (std::scanf("%31s", rule) == 1) {
        int L, Lc, words;
        if ((!std::strcmp(rule, "rows") || !std::strcmp(rule, "count")) && std::scanf("%d %d %d", &L, &Lc, &words) == 3) {
            const crbm::RowCut c = rule[0] == 'r' ? crbm::row_cut(lattice(L, Lc), words, 152) : crbm::count_cut(lattice(L, Lc), words, 152);
            std::printf("%d %d\n", c.seg, c.rows);
        } else if (!std::strcmp(rule, "bitplane") && std::scanf("%d %d %d", &L, &Lc, &words) == 3) {
            crbm::Geometry g = lattice(L, Lc);
            g.bitplane = 1;
            std::printf("%d\n", crbm::sweep_warps(g, words, 152, false));
        } else if (!std::strcmp(rule, "canonical")) {
            int correlations;
            if (std::scanf("%d %d %d %d", &L, &Lc, &words, &correlations) != 4) return 1;
            std::printf("%d\n", crbm::sweep_warps(lattice(L, Lc), words, 152, correlations != 0));
        } else if (!std::strcmp(rule, "batch")) {
            int warps, ctas, smem;
            if (std::scanf("%d %d %d", &warps, &ctas, &smem) != 3) return 1;
            std::printf("%d\n", crbm::batch_warps(warps, ctas, smem, 152));
        } else if (!std::strcmp(rule, "schedule")) {
            int sweeps, cells, per_sm, resident;
            if (std::scanf("%d %d %d %d %d", &sweeps, &words, &cells, &per_sm, &resident) != 5) return 1;
            const crbm::CanonSchedule c = crbm::canon_schedule(sweeps, words, cells, 152, per_sm, resident);
            std::printf("%d %d\n", c.all ? 1 : 0, c.chunk);
        } else {
            return 1;
        }
    }
    return 0;
}
