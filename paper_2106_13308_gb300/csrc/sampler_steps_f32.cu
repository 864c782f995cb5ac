// Instantiations of the one-step-at-a-time sampler for FP32 weights.
#include "sampler_steps.cuh"

namespace vqmc {
template cudaError_t launch_sampler_steps_wt<float>(const SamplerArgs& a, cudaStream_t st);
}  // namespace vqmc
