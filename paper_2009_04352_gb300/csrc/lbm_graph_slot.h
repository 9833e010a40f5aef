// An executable graph kept together with the number of steps it advances, so that
// a graph of another length is never taken for it. Host code without CUDA types.
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

}  // namespace lbm
