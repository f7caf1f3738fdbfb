// lc_rollout.h -- which graphs a rollout of the learned correction launches (host only).
#pragma once

namespace vk {

// Steps of the long rollout graph: within a graph the launches of consecutive steps overlap, between graphs
// they do not (128 x 256: 46.0 us a step in graphs of eight, 48.4 in graphs of one; 32 x 64: 42.0 and 44.4).
constexpr int ROLL_STEPS = 8;
// Steps that a state must have taken, this call's included, before the long graph is captured for it: the
// capture and instantiation cost 225 us more than a one-step graph's 50, which about 94 steps win back.  (A
// state with another reference density needs new graphs, so a program may start often and run briefly.)
constexpr long long ROLL_MANY_FROM = 96;

struct RolloutPlan { bool capture_one, capture_many; int many, ones; };

// A call of `steps` steps after `taken` ones with the present graphs: launches of each graph, and which of them
// have to be captured.  Neither is captured unless this call launches it.
inline RolloutPlan rollout_plan(int steps, long long taken, bool have_one, bool have_many)
{
    RolloutPlan p{false, false, 0, 0};
    if (have_many || taken + steps >= ROLL_MANY_FROM) p.many = steps / ROLL_STEPS;
    p.ones = steps - p.many * ROLL_STEPS;
    p.capture_one = p.ones > 0 && !have_one;
    p.capture_many = p.many > 0 && !have_many;
    return p;
}

}  // namespace vk
