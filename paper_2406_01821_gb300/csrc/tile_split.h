// Into how many set groups the tiles beyond the last whole wave of a launch are split (hard_eval.cu), free
// of CUDA: the library's launches and a CPU test use it.
#pragma once
#include <algorithm>
#include <cstdint>

namespace rs {

// `rest` tiles (fewer than `slots`, the CTAs that are resident at once) are split into g groups of P
// sets each; a CTA takes as long as `base` sets for its tile and its sets rounded up to its W warps. The
// g of 1 .. P / W (rounded up) with the least waves x time, the smallest of equals. For a number of waves
// the most groups that they hold are the best, or fewer of the same rounded size, so that only one g per
// number of waves is looked at, until more waves cannot gain: their staging alone, with an even share of
// the sets, would take longer. (Trying every g took 1.5 us of a call with 4096 sets, and grew with P.)
inline int64_t split_groups(int64_t rest, int64_t slots, int64_t P, int64_t W, int64_t base)
{
    if (rest <= 0 || P <= 0) return 1;
    const int64_t most = (P + W - 1) / W, share = P * rest / slots;
    int64_t best = INT64_MAX, groups = 1;
    for (int64_t k = 1;; ++k) {
        const int64_t hi = std::min(most, k * slots / rest);
        const int64_t sets = ((P + hi - 1) / hi + W - 1) / W * W;
        const int64_t g = (P + sets - 1) / sets;
        const int64_t cost = (rest * g + slots - 1) / slots * (base + sets);
        if (cost < best) { best = cost; groups = g; }
        if (hi == most || (k + 1) * base + share >= best) return groups;
    }
}

}  // namespace rs
