// Choice of a launch shape by timing (host code, no CUDA).
#pragma once
#include <stdint.h>

#include <tuple>
#include <utility>
#include <vector>

namespace lrr {

// Everything a candidate's shape and time depend on: the device, the problem's
// order and rank, its blocks (how many, most columns, longest columns, both
// rounded up to what a shape can tell apart, so that another partition of the
// same problem seldom has to be timed again) and whether the workspace holds
// the clusterless form's part.
struct TuneKey {
    int dev, prec;
    int64_t m, n, r;
    int t, max_pp, max_L;
    bool grid;
    bool operator<(const TuneKey& o) const {
        return std::tie(dev, prec, m, n, r, t, max_pp, max_L, grid) <
               std::tie(o.dev, o.prec, o.m, o.n, o.r, o.t, o.max_pp, o.max_L, o.grid);
    }
};

// The id of the candidate (id, shape) that runs fastest, the first of equals.
// time(shape, warm_up) runs a shape and returns its milliseconds, negative on
// failure.  Each runs once untimed before it counts: its first run loads the
// kernel and asks the runtime for its limits (60 us, as long as the whole run
// of a small problem), and the first candidate would pay for all.  A shape that
// has been timed already is not timed again: it would only win by noise.
template <typename Shape, typename Time>
bool pick_fastest(const std::vector<std::pair<int, Shape>>& candidates, Time time, int* best) {
    float least = 0.f;
    bool any = false;
    for (size_t i = 0; i < candidates.size(); ++i) {
        bool known = false;
        for (size_t j = 0; j < i; ++j) known |= candidates[j].second == candidates[i].second;
        if (known) continue;
        if (time(candidates[i].second, true) < 0.f) return false;
        const float ms = time(candidates[i].second, false);
        if (ms < 0.f) return false;
        if (!any || ms < least) {
            least = ms;
            *best = candidates[i].first;
        }
        any = true;
    }
    return any;
}

}  // namespace lrr
