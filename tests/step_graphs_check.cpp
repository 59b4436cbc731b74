// Host check of step_graphs.h with integers in the place of graphs: when a step of the caller's loop is due to be replayed, that a key is
// recorded once, that a recording which fails is not tried again and not destroyed, and that all others are.
#include <cstdio>
#include <set>
#include <tuple>

#include "../paper_2503_05931_b200/csrc/step_graphs.h"

using namespace aed;

#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main()
{
    typedef std::tuple<int, int, int, bool> Key;
    StepGraphs<Key, int> graphs;
    const Key a(8, 1, 0, false), b(8, 2, 0, false), c(8, 1, 4, false), full(8, 1, 0, true);

    // a caller whose sizes come once each, or fewer times than a recording takes to pay, never records
    for (bool many : {false, true}) {
        const int before = steps_before_recording(many);
        CHECK(before >= 8);
        const Key one(many, 7, 0, false), other(many, 8, 0, false);
        for (int i = 0; i < before; ++i) CHECK(!graphs.due(one, before));
        for (int i = 0; i < 3; ++i) CHECK(graphs.due(one, before));
        CHECK(!graphs.due(other, before));
    }

    int recordings = 0;
    auto record = [&](StepGraphs<Key, int>::Entry &e) { e.exec = ++recordings; e.nodes = 10 * recordings; return true; };
    const auto *ga = graphs.get(a, record);
    CHECK(ga && ga->exec == 1 && ga->nodes == 10);
    const auto *gb = graphs.get(b, record), *gc = graphs.get(c, record);
    CHECK(gb && gb->exec == 2 && gc && gc->exec == 3);
    CHECK(graphs.get(a, record) == ga && graphs.get(b, record) == gb && recordings == 3);

    int tries = 0;
    auto refuse = [&](StepGraphs<Key, int>::Entry &e) { ++tries; e.exec = -1; return false; };
    CHECK(!graphs.get(full, refuse));
    CHECK(!graphs.get(full, refuse) && tries == 1);
    CHECK(!graphs.get(full, record) && recordings == 3);

    std::set<int> gone;
    graphs.clear([&](int e) { gone.insert(e); });
    CHECK((gone == std::set<int>{1, 2, 3}));
    CHECK(graphs.get(a, record)->exec == 4);
    printf("ok\n");
    return 0;
}
