// Time-blocked history convolution (Section 2.3) for FP32 history.
#include "sbim_ahead.cuh"

namespace sbim {

cudaError_t ahead_f32(const StepArgs& a, int stage, bool halves, cudaStream_t st,
                     const BatchLaunch* batch, int tiles) {
  return ahead::run_stage<dev::StoreF32>(a, stage, halves, st, batch, tiles);
}

}  // namespace sbim
