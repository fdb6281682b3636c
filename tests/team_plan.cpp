// A batch's team plan over seeded unit costs, for test_team_plan.py:
// argv: units, kinds, seed, log10 of the largest b / a (negative: every unit a = 1, b that large).  Prints per kind "capacity ctas units planned", then the
// plan's time over that of sorting the units once.
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "fg_team_plan.cuh"

int main(int argc, char **argv) {
    if (argc != 5) return 2;
    const int units = std::atoi(argv[1]), nk = std::atoi(argv[2]);
    std::mt19937 rng((unsigned)std::atoi(argv[3]));
    const double spread = std::atof(argv[4]);
    const int capacity[] = {608, 912, 456, 1};
    std::vector<fg::UnitCost> cost(units);
    std::map<int, fg::KindPlan> kinds;
    for (int u = 0; u < units; u++) {
        cost[u].a = std::exp(4.0 * rng() / 4294967296.0 - 3.0);
        cost[u].b = cost[u].a * std::pow(10.0, spread * rng() / 4294967296.0);
        if (spread < 0) cost[u] = {1.0, std::pow(10.0, -spread)};
        kinds[u % nk].capacity = capacity[u % nk % 4];
        kinds[u % nk].queries.push_back(u);
    }
    const auto t0 = std::chrono::steady_clock::now();
    fg::plan_teams(kinds, cost);
    const auto t1 = std::chrono::steady_clock::now();
    for (auto &kv : kinds) {
        const fg::KindPlan &k = kv.second;
        std::vector<char> seen(units, 0);
        int planned = 0, ctas = 0;
        for (size_t c = 0; c < k.class_q.size(); c++) {
            ctas += k.class_size[c] * k.class_teams[c];
            if (k.class_teams[c] < 1 || k.class_teams[c] > (int)k.class_q[c].size()) return 3;
            for (size_t i = 0; i < k.class_q[c].size(); i++) {
                const int u = k.class_q[c][i];
                planned += !seen[u];
                seen[u] = 1;
                if (i && cost[u].ms(k.class_size[c]) > cost[k.class_q[c][i - 1]].ms(k.class_size[c])) return 4;
            }
        }
        if (ctas != k.ctas) return 5;
        std::printf("%d %d %d %d\n", k.capacity, ctas, (int)k.queries.size(), planned);
    }
    std::vector<double> key(units);
    for (int u = 0; u < units; u++) key[u] = cost[u].b;
    const auto t2 = std::chrono::steady_clock::now();
    std::sort(key.begin(), key.end());
    const auto t3 = std::chrono::steady_clock::now();
    std::printf("%f\n", std::chrono::duration<double>(t1 - t0).count() / std::chrono::duration<double>(t3 - t2).count());
    return 0;
}
