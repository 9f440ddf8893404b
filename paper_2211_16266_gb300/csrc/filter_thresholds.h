// Two FP32 decisions of the consistency filter as comparisons: the floats at which
// they turn, searched on the host, so that its kernel neither divides nor takes
// roots. CUDA-free (tests/test_host_filter_thresholds.py checks every float around
// each of them).
#pragma once

#include <cmath>
#include <limits>

namespace pmsp {

// The smallest float x for which `pred` holds, pred being monotone (false, then
// true), from a guess a few floats away.
template <class Pred>
inline float first_float(float x, Pred pred) {
    const float inf = std::numeric_limits<float>::infinity();
    while (!pred(x) && x < inf) x = std::nextafter(x, inf);
    for (float below = std::nextafter(x, -inf); pred(below); below = std::nextafter(x, -inf)) x = below;
    return x;
}

struct FilterThresholds {
    float wrap_hi, wrap_lo;  // a difference of columns du wraps by -W from wrap_hi on, by +W below wrap_lo
    float max_sq;            // a squared distance below it has a root below max_px
};

// The wrap of du by whole panoramas is du - W floor(du / W + 1/2); |du| < W, so the
// floor is -1, 0 or 1. The distance test is sqrt(s) < max_px, max_px > 0.
inline FilterThresholds filter_thresholds(int width, float max_px) {
    const float W = (float)width;
    auto turns = [&](float du) {
        volatile float q = du / W;
        volatile float h = q + 0.5f;
        return std::floor(h);
    };
    FilterThresholds t;
    t.wrap_hi = first_float(0.5f * W, [&](float du) { return turns(du) >= 1.0f; });
    t.wrap_lo = first_float(-0.5f * W, [&](float du) { return turns(du) >= 0.0f; });
    t.max_sq = first_float(max_px * max_px, [&](float s) { return s > 0.0f && std::sqrt(s) >= max_px; });
    return t;
}

}  // namespace pmsp
