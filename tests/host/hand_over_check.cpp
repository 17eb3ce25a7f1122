// Host-only check of the hand-over rule between writing warps and the MMA warp: every order of steps and of waits that run out
// is walked through, with the warps as the kernels run them (one group of writers per hand-over, and column groups with writers
// of their own).  Every order has to end with all warps through all hand-overs, no barrier left half full and no arrival counted for
// another hand-over; on one barrier, or without waiting after a failure, the walk has to find an order that does not.
#include <cstdio>
#include <set>
#include <string>
#include <vector>

#include "hand_over.h"

struct Rule {
    int (*barrier)(int);
    bool (*waits)(bool);
};

struct Warp {           // groups: the column groups it writes (or, for the MMA warp, all of them, in order)
    signed char p = 0, g = 0, failed = 0, on = -1, gen = 0;      // on: the barrier it waits at, gen: its turn then
};
struct Bar {
    signed char count = 0, p = -1, gen = 0;
};
struct State {
    std::vector<Warp> w;       // the last one issues the MMAs
    std::vector<Bar> bar;
    signed char answers = 0;   // answer p comes before hand-over p: p = 0 the first products, later what hand-over p - 1 led to
    bool mixed = false;
    std::string key() const {
        std::string s((const char*)w.data(), w.size() * sizeof(Warp));
        s.append((const char*)bar.data(), bar.size() * sizeof(Bar));
        s.push_back(answers);
        s.push_back(mixed);
        return s;
    }
};

struct Walk {
    Rule rule;
    std::vector<std::vector<int>> groups;       // of every writer, then all groups for the MMA warp
    std::vector<int> needed;                    // arrivals that complete a group's hand-over
    int G, P;
    std::set<std::string> seen;
    int bad = 0;

    void arrive(State& s, int i, bool waits) {
        Warp& w = s.w[i];
        const int g = groups[i][w.g], b = rule.barrier(w.p) * G + g;
        Bar& q = s.bar[b];
        if (q.count == 0) q.p = w.p;
        else if (q.p != w.p) s.mixed = true;
        if (waits) { w.on = (signed char)b; w.gen = q.gen; }
        if (++q.count == needed[g]) { q.count = 0; ++q.gen; }
        if (!waits) next(s, i);
    }
    void next(State& s, int i) {
        Warp& w = s.w[i];
        if (++w.g == (int)groups[i].size()) { w.g = 0; ++w.p; }
    }
    void go(const State& s) {
        if (bad || !seen.insert(s.key()).second) return;
        const int M = (int)s.w.size() - 1;
        bool moved = false, done = true;
        if (s.mixed) { bad = 1; return; }
        for (int i = 0; i <= M; ++i) {
            const Warp& w = s.w[i];
            if (w.p == P) continue;
            done = false;
            if (w.on >= 0) {                                       // at a barrier: on when its turn is complete
                if (s.bar[w.on].gen != w.gen) {
                    State t = s;
                    t.w[i].on = -1;
                    next(t, i);
                    moved = true;
                    go(t);
                }
                continue;
            }
            const bool first = w.g == 0;
            if (!w.failed && (i == M || first)) {                  // a wait with a limit may run out here
                State t = s;
                t.w[i].failed = 1;
                moved = true;
                go(t);
            }
            if (i == M) {
                State t = s;
                if (first && !w.failed) {
                    if (t.answers == w.p) { t.answers = (signed char)(w.p + 1); moved = true; go(t); continue; }
                }
                moved = true;
                arrive(t, i, true);
                go(t);
            } else if (w.failed || !first || s.answers > w.p) {
                State t = s;
                moved = true;
                arrive(t, i, rule.waits(w.failed));
                go(t);
            }
        }
        if (done)
            for (const Bar& b : s.bar)
                if (b.count) bad = 2;
        if (!done && !moved) bad = 3;
    }
    int run(int writers_per_group, int group_count, int split, int phases) {
        G = group_count; P = phases; bad = 0;
        seen.clear(); groups.clear();
        needed.assign(G, writers_per_group + 1);
        for (int sel = 0; sel < split; ++sel)                      // writers of groups sel, sel + split, ...
            for (int q = 0; q < writers_per_group; ++q) {
                std::vector<int> mine;
                for (int g = sel; g < G; g += split) mine.push_back(g);
                groups.push_back(mine);
            }
        std::vector<int> all;
        for (int g = 0; g < G; ++g) all.push_back(g);
        groups.push_back(all);
        State s;
        s.w.resize(groups.size());
        s.bar.resize(2 * G);
        go(s);
        return bad;
    }
};

int main() {
    const int shapes[][4] = {{2, 1, 1, 5}, {3, 1, 1, 4}, {4, 1, 1, 3}, {1, 4, 2, 3}, {2, 2, 2, 3}};     // writers per group, groups, sets of writers, hand-overs
    Walk v;
    for (const auto& s : shapes) {
        v.rule = Rule{[](int p) { return uoe::hand_over_barrier(p); }, [](bool f) { return uoe::hand_over_waits(f); }};
        if (const int bad = v.run(s[0], s[1], s[2], s[3])) { std::printf("shape %d %d %d %d: %d\n", s[0], s[1], s[2], s[3], bad); return 1; }
        std::printf("%zu states\n", v.seen.size());
    }
    v.rule = Rule{[](int) { return 0; }, [](bool) { return false; }};
    if (!v.run(3, 1, 1, 4)) return 2;
    v.rule = Rule{[](int) { return 0; }, [](bool f) { return f; }};
    if (!v.run(3, 1, 1, 4)) return 3;
    v.rule = Rule{[](int p) { return p & 1; }, [](bool) { return false; }};
    if (!v.run(3, 1, 1, 4)) return 4;
    std::printf("ok\n");
    return 0;
}
