// Asks libgpcn.so's host side (no GPU) what it would do; see test_host_rules.py.
//   optin                             the calls a kernel's opt-in makes: per device, per growth, on failure, from threads
//   streams ASKED KIND SITES ...      the groups of a batched step, a line of item numbers each
//   choose LINES N FORM KIND LEVELS ELEM   whether the cyclic reduction is chosen, and its lines per block
//   tables NX NY NZ MODES DT DT ...   tables built for each dt in turn into one Tables, against fresh ones: 1 where equal
#include "gp_host.h"
#include "gp_optin.h"

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <thread>
#include <vector>

using namespace gpcn;

static bool same(const AxisTables &a, const AxisTables &b) {
    return a.off_cp == b.off_cp && a.off_ip == b.off_ip && a.min_window == b.min_window && a.t_const == b.t_const &&
           a.pcr_levels == b.pcr_levels && a.off_pcr == b.off_pcr && a.off_pcr_inv == b.off_pcr_inv && a.cp_max == b.cp_max;
}

// Bytes set on a device by a sequence of raises, as cudaFuncSetAttribute would see them.
static int optin() {
    SmemOptIn kept;
    int limit[3] = {0, 0, 0}, calls[3] = {0, 0, 0};
    auto raise = [&](int dev, int bytes) {
        return kept.raise(dev, bytes, [&](int b) {
            ++calls[dev];
            limit[dev] = b;
            return cudaSuccess;
        });
    };
    for (int dev : {0, 1, 0, 1, 2}) raise(dev, 60000);
    raise(1, 70000);
    raise(1, 50000);
    for (int dev = 0; dev < 3; ++dev) std::printf("%d %d\n", limit[dev], calls[dev]);
    // a failed set is not remembered
    SmemOptIn bad;
    int tries = 0;
    for (int q = 0; q < 2; ++q) bad.raise(0, 60000, [&](int) { ++tries; return cudaErrorInvalidValue; });
    const int beyond = (int)bad.raise(kOptInDevices, 1, [&](int) { ++tries; return cudaSuccess; });
    std::printf("%d %d\n", tries, beyond);
    // threads of different sizes: never lowered
    SmemOptIn shared;
    int high = 0, lowered = 0;
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&, t] {
            for (int q = 0; q < 1000; ++q)
                shared.raise(0, 50000 + (q * 37 + t * 911) % 50000, [&](int b) {  // under the lock
                    lowered += b < high;
                    high = b;
                    return cudaSuccess;
                });
        });
    for (auto &t : threads) t.join();
    std::printf("%d %d\n", high, lowered);
    return 0;
}

int main(int argc, char **argv) {
    if (argc > 1 && !std::strcmp(argv[1], "optin")) return optin();
    if (argc == 8 && !std::strcmp(argv[1], "choose")) {
        int tl = 0;
        const bool yes = choose_pcr(std::atoll(argv[2]), std::atoi(argv[3]), (Form)std::atoi(argv[4]), (Kind)std::atoi(argv[5]),
                                    std::atoi(argv[6]), std::atoi(argv[7]), &tl);
        std::printf("%d %d\n", yes ? 1 : 0, tl);
        return 0;
    }
    if (argc > 4 && !std::strcmp(argv[1], "streams")) {
        std::vector<StreamItem> items;
        for (int q = 3; q + 1 < argc; q += 2)
            items.push_back({(int)items.size(), std::atoi(argv[q]), (size_t)std::atoll(argv[q + 1])});
        for (const auto &g : stream_groups(items, std::atoi(argv[2]))) {
            for (int i : g) std::printf("%d ", i);
            std::printf("\n");
        }
        return 0;
    }
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
