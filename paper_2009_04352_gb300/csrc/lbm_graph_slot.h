// Step graphs kept between calls: an executable graph together with the number of
// steps it advances, so that a graph of another length is never taken for it, and
// when one is worth building. Host code without CUDA types.
#pragma once

namespace lbm {

template <typename Exec> struct GraphSlot {
    Exec exec;
    int steps;
};

template <typename Exec, typename Destroy> void slot_clear(GraphSlot<Exec> &s, Destroy destroy)
{
    if (s.exec) destroy(s.exec);
    s.exec = nullptr;
    s.steps = 0;
}

// Make the slot hold a graph of `steps` steps: build(&exec) returns 0, or an error
// after which the slot is empty.
template <typename Exec, typename Destroy, typename Build>
int slot_ensure(GraphSlot<Exec> &s, int steps, Destroy destroy, Build build)
{
    if (s.exec && s.steps == steps) return 0;
    slot_clear(s, destroy);
    Exec e = nullptr;
    const int rc = build(&e);
    if (rc != 0) {
        if (e) destroy(e);
        return rc;
    }
    s.exec = e;
    s.steps = steps;
    return 0;
}

// Whether a call of n steps (or one after it) may replay a sampled step's graph from
// phase `start`: sampling every `every` steps, at step `step` and phase `cur` now. An
// even interval samples in one phase only. Calls of one step never replay one, and
// callers that make nothing else need not pay for it.
inline bool sampled_graph_due(int n, int every, long long step, int cur, int start)
{
    if (n < 2 || every < 2) return false;
    const long long to_next = (every - step % every) % every;
    return every % 2 || start == (cur ^ (int)(to_next & 1));
}

}  // namespace lbm
