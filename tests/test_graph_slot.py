"""The step graphs kept between calls (lbm_graph_slot.h), compiled for the host with a
fake of the graph: a slot never holds a graph of another length than it says, nor
one whose building failed, whatever fails in between; and the graphs of sampled
steps are built where a run replays them, not for calls of one step."""
import subprocess

from paper_2009_04352_gb300 import build

SOURCE = r"""
#include <cassert>
#include <set>
#include "lbm_graph_slot.h"

struct Graph { int steps; };
static std::set<Graph *> live;
static int made = 0;
static int destroy(Graph *g) { assert(live.erase(g) == 1); delete g; return 0; }

enum Fail { NONE, EARLY, LATE };   // no graph, or one that was made and then refused
static int ensure(lbm::GraphSlot<Graph *> &s, int steps, Fail fail = NONE)
{
    return lbm::slot_ensure(s, steps, destroy, [=](Graph **out) {
        ++made;
        if (fail == EARLY) return -2;
        live.insert(*out = new Graph{steps});
        return fail == LATE ? -2 : 0;
    });
}
static void check(const lbm::GraphSlot<Graph *> &s, int steps)
{
    assert(s.steps == steps);
    assert(steps ? s.exec && s.exec->steps == steps && live.count(s.exec) : !s.exec);
}

int main()
{
    for (Fail fail : {EARLY, LATE}) {
        // an interval of 10, then of 5 whose second graph cannot be built, then 10 again
        lbm::GraphSlot<Graph *> a{}, b{};
        assert(ensure(a, 10) == 0 && ensure(b, 10) == 0);
        assert(ensure(a, 5) == 0 && ensure(b, 5, fail) == -2);
        check(a, 5);
        check(b, 0);
        assert(live.size() == 1);
        assert(ensure(a, 10) == 0 && ensure(b, 10) == 0);
        check(a, 10);
        check(b, 10);
        // nothing is built for what is there
        const int before = made;
        assert(ensure(a, 10) == 0 && ensure(b, 10) == 0 && made == before);
        // a first build that fails leaves nothing that a retry would take
        lbm::GraphSlot<Graph *> c{};
        assert(ensure(c, 4, fail) == -2);
        check(c, 0);
        assert(ensure(c, 4) == 0);
        check(c, 4);
        for (auto *s : {&a, &b, &c}) lbm::slot_clear(*s, destroy);
        check(a, 0);
        assert(live.empty());
    }
    return 0;
}
"""

DUE = r"""
#include <cassert>
#include "lbm_graph_slot.h"

int main()
{
    for (int every = 1; every <= 40; ++every)
        for (long long step = 0; step <= 3 * every; ++step)
            for (int cur = 0; cur < 2; ++cur) {
                // phases in which the next samples fall, one plain or sampled step at a time
                bool phase[2] = {false, false};
                for (long long t = step; t <= step + 2 * every; ++t)
                    if (t % every == 0) phase[cur ^ ((t - step) & 1)] = true;
                for (int start = 0; start < 2; ++start) {
                    assert(!lbm::sampled_graph_due(1, every, step, cur, start));
                    const bool due = lbm::sampled_graph_due(2, every, step, cur, start);
                    assert(due == lbm::sampled_graph_due(1000, every, step, cur, start));
                    assert(due == (every > 1 && phase[start]));
                }
            }
    return 0;
}
"""


def _run(tmp_path, source):
    src, exe = tmp_path / "slot.cpp", tmp_path / "slot"
    src.write_text(source)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I" + build.CSRC, "-o", str(exe), str(src)], check=True)
    subprocess.run([str(exe)], check=True)


def test_slots_hold_what_they_say(tmp_path):
    _run(tmp_path, SOURCE)


def test_sampled_graphs_are_built_where_they_are_replayed(tmp_path):
    _run(tmp_path, DUE)
