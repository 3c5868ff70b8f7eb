// Coordinate descent over the launch shapes of a level (tune.cu), apart from how a shape is timed.
#pragma once

#include <vector>

#include "mhm_internal.h"

namespace mhm {

// From `start`, the shape the level runs untuned: each field in turn over its values, the other
// fields at the best so far, two sweeps.  The start is the first shape timed, so the result is
// never slower than it.  time(shape, &ms) returns false to give up; *best_ms gets the result's time.
template <class Time>
Tuning tune_descend(const Tuning& start, double* best_ms, Time&& time) {
    struct Field {
        int Tuning::*m;
        std::vector<int> values;
    };
    const std::vector<Field> fields = {{&Tuning::nbuf, {2, 3, 4}},          {&Tuning::pf_all, {0, 1}},
                                       {&Tuning::l2pf, {0, 2, 4, 8}},       {&Tuning::op_policy, {0, 1, 2}},
                                       {&Tuning::blocks_per_sm, {2, 3, 4}}, {&Tuning::chunk, {2048, 4096, 8192}}};
    Tuning best = start;
    if (!time(best, best_ms)) return best;
    for (int sweep = 0; sweep < 2; ++sweep)
        for (const Field& fd : fields)
            for (int v : fd.values) {
                if (best.*(fd.m) == v) continue;
                Tuning cand = best;
                cand.*(fd.m) = v;
                double ms = 0.0;
                if (!time(cand, &ms)) return best;
                if (ms < *best_ms) {
                    *best_ms = ms;
                    best = cand;
                }
            }
    return best;
}

}  // namespace mhm
