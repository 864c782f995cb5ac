// Instantiations of the one-step-at-a-time sampler for BF16 weights.
#include "sampler_steps.cuh"

namespace vqmc {
template cudaError_t launch_sampler_steps_wt<bf16>(const SamplerArgs& a, cudaStream_t st);
}  // namespace vqmc
