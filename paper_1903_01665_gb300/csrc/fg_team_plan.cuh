// The planner of a batch: how many CTAs each unit's team gets, and how many
// teams there are.  Host code without a CUDA call.
#pragma once

#include <algorithm>
#include <map>
#include <utility>
#include <vector>

namespace fg {

// A unit on a team of p CTAs takes about a + b / p ms.
struct UnitCost {
    double a = 0, b = 0;
    double ms(int p) const { return a + b / p; }
};

struct KindPlan {
    int kind = 0;
    std::vector<int> queries;                 // units of the batch of this kind
    std::vector<int> class_size;              // team size per class
    std::vector<std::vector<int>> class_q;    // units per class, largest work first
    std::vector<int> class_teams;             // teams per class
    int capacity = 1;                         // co-resident CTAs
    int ctas = 0;
};

// Team sizes: 1, 2, 3, 4, 6, 8, 12, 16, ...
inline int next_team(int p) { return p < 2 ? 2 : (p & (p - 1)) == 0 ? p + p / 2 : p / 3 * 4; }

// Plans the teams of every kind for a common makespan T ms: each unit gets the
// smallest team that finishes it in T, the units of one size
// share as many teams as their times fill, and T is the smallest (in steps of
// 6 %) at which all teams are resident together.  (Team sizes by edge count
// and CTAs by a guess of the work left the longest unit of a mixed batch on a
// fifth of the device while a third of it idled: 12 graphs, 15.6 ms.)
//
// The time of the plan counts in the call.  Only the loads per team size are
// formed at each T, T is doubled until the teams fit and then searched within
// the last doubling, and the units are put in classes and sorted once, at the
// end (grouping and sorting them at every step: 62 ms for 10,000 units of
// mixed cost in three kinds, 850 ms for 100,000; now 1 and 12).
inline void plan_teams(std::map<int, KindPlan> &kinds, const std::vector<UnitCost> &cost) {
    struct Sizes {
        KindPlan *kp;
        std::vector<int> size;       // 1, 2, 3, 4, 6, ..., capacity
        std::vector<int> at;         // per unit: its size's index at the last T that was tried
        std::vector<double> load;    // per size: ms of its units
        std::vector<int> units;      // per size: their number
    };
    std::vector<Sizes> all;
    double t0 = 1e-3;
    for (auto &kv : kinds) {
        Sizes s;
        s.kp = &kv.second;
        for (int p = 1; p < s.kp->capacity; p = next_team(p)) s.size.push_back(p);
        s.size.push_back(s.kp->capacity);
        s.at.assign(s.kp->queries.size(), 0);
        for (int u : s.kp->queries) t0 = std::max(t0, cost[u].ms(s.kp->capacity));
        all.push_back(std::move(s));
    }
    auto teams_of = [](int units, double load, double T) {
        const double want = 1.1 * load / T + 0.999;
        return want >= units ? units : std::max(1, (int)want);
    };
    // whether the teams of makespan T are resident together (or no kind can do with less)
    auto fits = [&](double T) {
        double used = 0;
        bool least = true;
        for (Sizes &s : all) {
            const int top = (int)s.size.size() - 1;
            s.load.assign(s.size.size(), 0.0);
            s.units.assign(s.size.size(), 0);
            for (size_t i = 0; i < s.at.size(); i++) {
                const UnitCost &c = cost[s.kp->queries[i]];
                int &k = s.at[i];   // near the size at the last T
                while (k < top && c.ms(s.size[k]) > T) k++;
                while (k > 0 && c.ms(s.size[k - 1]) <= T) k--;
                s.load[k] += c.ms(s.size[k]);
                s.units[k]++;
            }
            double ctas = 0;
            for (int k = 0; k <= top; k++)
                if (s.units[k]) ctas += (double)teams_of(s.units[k], s.load[k], T) * s.size[k];
            used += ctas / s.kp->capacity;
            least &= ctas <= 1;
        }
        return used <= 1.0 || least;
    };
    constexpr double kStep = 1.06;
    constexpr int kSteps = 12;   // to a doubling
    double T = t0;
    if (!fits(T)) {
        double low = T, high = T;
        do {
            low = high;
            for (int i = 0; i < kSteps; i++) high *= kStep;
        } while (!fits(high));
        T = low * kStep;
        while (!fits(T) && T < high) T *= kStep;
    }
    for (Sizes &s : all) {
        KindPlan &kp = *s.kp;
        kp.class_size.clear();
        kp.class_q.clear();
        kp.class_teams.clear();
        kp.ctas = 0;
        std::vector<std::vector<std::pair<double, int>>> members(s.size.size());
        for (size_t i = 0; i < s.at.size(); i++) {
            const int u = kp.queries[i];
            members[s.at[i]].push_back({-cost[u].ms(s.size[s.at[i]]), u});
        }
        for (size_t k = 0; k < s.size.size(); k++) {
            if (members[k].empty()) continue;
            std::sort(members[k].begin(), members[k].end());
            std::vector<int> v;
            v.reserve(members[k].size());
            for (const auto &x : members[k]) v.push_back(x.second);
            const int teams = teams_of((int)v.size(), s.load[k], T);
            kp.class_size.push_back(s.size[k]);
            kp.class_q.push_back(std::move(v));
            kp.class_teams.push_back(teams);
            kp.ctas += teams * s.size[k];
        }
    }
}

}  // namespace fg
