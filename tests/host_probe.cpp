// Asks libgpcn.so's host side (no GPU) what it would do; see test_host_rules.py.
//   tables NX NY NZ MODES DT DT ...   tables built for each dt in turn into one Tables, against fresh ones: 1 where equal
#include "gp_host.h"

#include <cstdio>
#include <cstdlib>
#include <cstring>

using namespace gpcn;

static bool same(const AxisTables &a, const AxisTables &b) {
    return a.off_cp == b.off_cp && a.off_ip == b.off_ip && a.min_window == b.min_window && a.t_const == b.t_const &&
           a.pcr_levels == b.pcr_levels && a.off_pcr == b.off_pcr && a.off_pcr_inv == b.off_pcr_inv && a.cp_max == b.cp_max;
}

int main(int argc, char **argv) {
    if (argc > 6 && !std::strcmp(argv[1], "tables")) {
        Geometry G;
        for (int q = 0; q < 3; ++q) {
            G.n[q] = std::atoi(argv[2 + q]);
            G.d[q] = 0.1;
            G.w[q] = 1.0;
        }
        G.g = 10.0;
        const int modes = std::atoi(argv[5]);
        Tables kept;
        for (int q = 6; q < argc; ++q) {
            G.dt = std::atof(argv[q]) * 0.01;
            std::vector<char> host, fresh_host;
            Tables fresh;
            append_tables(G, false, modes, host, kept, kPcrChosen);
            append_tables(G, false, modes, fresh_host, fresh, kPcrChosen);
            bool eq = host == fresh_host;
            int levels = 0;
            for (int mode = 0; mode < 2; ++mode)
                for (int ax = 0; ax < 3; ++ax) {
                    eq = eq && same(kept.ax[mode][ax], fresh.ax[mode][ax]);
                    levels += fresh.ax[mode][ax].pcr_levels > 0;
                }
            std::printf("%d %d\n", eq ? 1 : 0, levels);
        }
        return 0;
    }
    return 2;
}
