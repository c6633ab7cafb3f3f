// Prints the canonical SMEM sweep's shared-memory layout (crbm_internal.h), used only by tests.  Reads
// "L Lc paper n_seg mode" lines on stdin; prints "name first end" triples of the arrays in words, one line
// per layout.  With arguments (reserved bytes, static bytes): whether the tables are where the kernels look.
#include <cstdio>
#include <cstdlib>

#include "crbm_internal.h"

int main(int argc, char** argv) {
    if (argc == 3) {
        std::printf("%d\n", crbm::dynamic_smem_at_base(std::atoi(argv[1]), std::strtoul(argv[2], nullptr, 10)) ? 1 : 0);
        return 0;
    }
    crbm::Geometry g{};
    int mode;
    while (std::scanf("%d %d %d %d %d", &g.L, &g.Lc, &g.paper, &g.n_seg, &mode) == 5) {
        g.W = g.L / 2;
        g.Wc = g.Lc / 2;
        g.N = g.L * g.Lc;
        g.n_cells = g.W * g.Wc;
        const crbm::CanonSmem s = crbm::canon_smem(g, mode);
        const int rec = mode == crbm::kCanonRec ? g.n_cells * crbm::kCellRec * 4 : 0;
        const int expand = mode == crbm::kCanonPacked && !g.paper ? 1024 : 0;
        const int pw = g.paper && mode != crbm::kCanonPacked ? g.n_cells * 64 : 0;
        std::printf("w %d %d pw %d %d rec %d %d rows %d %d expand %d %d tab %d %d total 0 %d\n", s.w,
                    s.w + g.n_cells * (mode == crbm::kCanonPacked && !g.paper ? 16 : 32), s.pw, s.pw + pw, s.rec,
                    s.rec + rec, s.rows, s.rows + g.W * g.n_seg * 32, s.expand, s.expand + expand, crbm::kCanonTabWord,
                    crbm::kCanonTabWord + crbm::kCanonTabBytes / 4, s.total);
    }
    return 0;
}
