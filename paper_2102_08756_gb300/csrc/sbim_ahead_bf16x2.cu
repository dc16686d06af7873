// Time-blocked history convolution (Section 2.3) for BF16 hi/lo history.
#include "sbim_ahead.cuh"

namespace sbim {

cudaError_t ahead_bf16x2(const StepArgs& a, int stage, bool halves, cudaStream_t st,
                     const BatchLaunch* batch, int tiles) {
  return ahead::run_stage<dev::StoreBF16<true>>(a, stage, halves, st, batch, tiles);
}

}  // namespace sbim
