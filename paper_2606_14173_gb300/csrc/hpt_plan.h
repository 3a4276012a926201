// How a frame is cut into waves, and what the autotuner times.
#pragma once
#include <algorithm>
#include <cmath>

namespace hpt {

// Frames of less than one full wave per lane are cut into a wave per lane, so that the lanes fill each
// other's tails and gaps (one wave on one lane leaves the chip to a chain of some twenty kernels), down
// to waves of MIN_WAVE paths: 5.5 M paths 7.8 -> 6.9 ms, 12.6 M bake paths 4.35 -> 4.06 ms, 0.6 M paths
// 968 -> 893 us; between 64k and 1M paths the limit moved small frames by under 8 % either way.
constexpr long long MIN_WAVE = 1 << 16;

// paths per wave of a launch group of 'total' paths: the wave capacity, or less when that would leave
// lanes without a wave
inline int wave_paths(long long total, int spp_max, int lanes, int capacity)
{
    if (total >= (long long)lanes * capacity) return capacity;
    return (int)std::min<long long>(capacity, std::max<long long>({(total + lanes - 1) / lanes + 32ll * spp_max, MIN_WAVE, spp_max}));
}

// The autotuner's wave sizes, and the rows of a frame that it times: with enough paths for two full waves of the
// largest size on every lane, as far as the frame has them.  With one wave a lane a large frame is not what is
// timed: no lane takes a second wave while the others are in their tails (the 4K frame of 185k triangles: 8 M waves
// look as good as 16 M ones, 65.0 and 65.2 ms a band, and run 1 % slower over the whole frame; with two 129.6 and 127.7 ms,
// with three the same choice).
constexpr int TUNE_WAVES[] = {1 << 21, 1 << 22, 1 << 23, 1 << 24};
inline int tune_rows(int W, int H, int n_lambda, int spp, int max_lanes)
{
    const double per_row = (double)W * std::max(n_lambda, 1) * std::max(spp, 1);
    return (int)std::min<double>(H, std::max(1.0, std::ceil(2.0 * max_lanes * TUNE_WAVES[3] / per_row)));
}
// Whether waves of 'capacity' paths are what timing them would run.  A frame too small for them runs smaller
// ones, the same for every such capacity: their times say nothing about it.
inline bool tune_runs_full(long long total, int spp, int lanes, int capacity)
{
    return wave_paths(total, spp, lanes, capacity) == capacity;
}

}  // namespace hpt
