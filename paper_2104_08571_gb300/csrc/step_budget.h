// How many steps one launch of a multi-step Euler kernel takes: about a
// millisecond of them, so that neither a queued call nor a request that arrives
// meanwhile waits long behind one launch.  Host code without CUDA.
#pragma once
#include <algorithm>

namespace ripple {

// Seconds of an FP64 first-order 2D step on the tiles of euler_tile64.cuh: 64^2
// 7.4, 128^2 8.7, 512^2 64, 1024^2 240 us.
inline double tile64_step_seconds(double cells) { return 4.5e-6 + 0.23e-9 * cells; }

// Steps of a launch on a field, of the `left` that remain.  FP32: about 64 M
// cell updates, 256 steps at most (64^2 4.0 us a step, 1024^2 11.2 us, FORCE
// 4096^2 115 us); FP64 steps take up to twenty times as long.
inline int walk_steps(bool f64, long long cells, long long left)
{
    const long long most = f64 ? (long long)(1e-3 / tile64_step_seconds((double)cells)) : (64LL << 20) / cells;
    return (int)std::min(left, std::max(1LL, std::min(256LL, most)));
}

// Seconds of a served problem's step in a round of its own (the solo solver and
// the packed walks): FP32 64^2 3.4, 512^2 5.9, 1024^2 11.2 us; FP64 64^2 12.8,
// 256^2 40, 512^2 124, 1024^2 400 us.
inline double solo_step_seconds(bool f64, double cells)
{
    return f64 ? 12.5e-6 + 0.38e-9 * cells : 3.5e-6 + 7.5e-12 * cells;
}

// Steps of such a round: at most kSoloMaxSteps, and at least eight, so that
// queueing a round stays small beside it.
constexpr long long kSoloMaxSteps = 1024;
inline long long solo_steps(bool f64, long long cells, long long left)
{
    const long long k = (long long)(1e-3 / solo_step_seconds(f64, (double)cells));
    return std::min(left, std::max(8LL, std::min(kSoloMaxSteps, k)));
}

}  // namespace ripple
