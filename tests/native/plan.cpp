// The cut of frames into waves and the autotuner's band (csrc/hpt_plan.h) compiled with the host compiler, for the tests.
#include "hpt_plan.h"

using namespace hpt;

extern "C" int waves(long long total, int spp, int lanes, int capacity) { return wave_paths(total, spp, lanes, capacity); }
extern "C" int rows(int W, int H, int nl, int spp, int lanes) { return tune_rows(W, H, nl, spp, lanes); }
extern "C" int full(long long total, int spp, int lanes, int capacity) { return tune_runs_full(total, spp, lanes, capacity); }
extern "C" int tune_wave(int i) { return TUNE_WAVES[i]; }
