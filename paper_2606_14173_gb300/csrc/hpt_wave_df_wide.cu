// Trace and accumulation kernels of wide scenes for the coherent arithmetic 'df'.
#include "hpt_wave_inst.cuh"

namespace hpt {
cudaError_t wave_trace_wide_df(bool st, const JobTable *jt, const WaveDesc &wd, const PathBufs &pb, SlotScratch *scr, int it,
                               int grid, cudaStream_t s)
{
    return WaveLaunch<df, true>::trace(st, jt, wd, pb, scr, it, grid, s);
}
cudaError_t wave_accum_wide_df(const JobTable *jt, const WaveDesc &wd, const PathBufs &pb, SlotScratch *scr, cudaStream_t s)
{
    return WaveLaunch<df, true>::accum(jt, wd, pb, scr, s);
}
cudaError_t wave_preload_wide_df() { return WaveLaunch<df, true>::preload(); }
}  // namespace hpt
