// Which half-sweeps of a run go to the bounded kernel (sweep_bounded), and when.
// CUDA-free (tests/test_host_sweep_policy.py).
#pragma once

namespace pmsp {

// Whether a run may use the bounded kernel. It pays with 4 to 10 views (1920x960, 8
// iterations, 3 views of 7x7 35.3 against 35.1 ms), with samples left to drop, 5 x 5 or more
// (1414x706, 6 views, 3 iterations with noise, 9x9 at stride 3, 9 samples: 7.02 against
// 6.30 ms; 8 iterations without noise 14.69 against 14.62, at stride 2, 25 samples, 29.3
// against 33.6), and on a grid that keeps the GPU busy while lanes of a warp wait for one
// another (384x192, 288 tiles, 6 views: 4.6 against 4.8 ms pooled; 640x320, 800 tiles:
// 10.8 against 9.8). A candidate of few view-samples needs more tiles (4 views of 5x5, 2
// iterations: 514x258, 561 tiles, 1.335 against 1.320 ms; 640x320 1.889 against 1.882; 6
// iterations 4.655 against 4.780).
constexpr bool bounded_serves(int views, int side, long long tiles, int sms) {
    return views >= 4 && views <= 10 && side >= 5 && tiles >= (views * side * side < 125 ? 5ll : 3ll) * sms;
}

// Pixels whose incumbent costs less than this are close: the bound, which needs a cost
// low enough to be passed after part of the samples, then drops most refinement tests.
constexpr float CLOSE_COST = 0.07f;

// Close pixels, of the W x H / 2 that the half-sweep before ended with, from which on
// the next one goes to the bounded kernel: 85 %. The lanes of a warp hand their tests
// to one another until the last is decided, so a few pixels whose tests run to the end
// cost the others more than theirs are shortened. Against the pooled kernel alone, over 192
// forms from 514x258 to 1000x502 (4 to 10 views, 25 to 49 samples, noise of 0 to 2 DN,
// 1 to 8 iterations), and their slowest:
//   close below     0.15            0.10            0.07            0.05
//   50 %       1.014x 0.854x   1.023x 0.883x   1.028x 0.925x   1.032x 0.953x
//   70 %       1.025x 0.877x   1.032x 0.940x   1.036x 0.971x   1.036x 0.982x
//   85 %       1.035x 0.963x   1.036x 0.979x   1.036x 0.989x   1.036x 0.988x
// From 960x480 to 3840x1920 (88 forms) 1.053x, slowest 0.997x, with 50 % below 0.15
// 1.046x and 0.944x.
constexpr long long bounded_from(int W, int H) { return (long long)W * H * 17 / 40; }

}  // namespace pmsp
