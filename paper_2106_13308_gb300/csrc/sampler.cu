// Exact autoregressive sampling (Algorithm 1 of the paper, Sec. 2.3) from
// Philox4x32-10 uniforms (Sec. 4), and the dispatch between the sampler kernels:
// the blocked tensor-core sampler (sampler_tc.cu) for the BF16 models it covers,
// for every other model one of the CUDA-core samplers, in blocks of steps
// (sampler_impl.cuh, instantiated in sampler_bf16.cu and sampler_f32.cu) or step by
// step (sampler_steps.cuh, sampler_steps_bf16.cu and sampler_steps_f32.cu).
//
// uniforms_kernel writes the same stream the samplers draw internally:
// u_{b,i} = word (i mod 4) of Philox4x32-10(counter (i/4, b0 + b, iteration),
// key = seed), as (x >> 8) 2^-24, with b0 the context's sample offset (0
// unless the context draws one shard of a batch spread over several GPUs).
#include <algorithm>

#include "sampler.cuh"

namespace vqmc {
namespace {

__global__ void uniforms_kernel(int B, int n, uint32_t k0, uint32_t k1, uint32_t it0, uint32_t it1, uint32_t boff,
                                float* __restrict__ u) {
  const int groups = (n + 3) / 4;
  const long long tot = (long long)B * groups;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < tot;
       q += (long long)gridDim.x * blockDim.x) {
    const int b = (int)(q / groups), g = (int)(q % groups);
    const uint4 r = philox4x32_10(make_uint4((uint32_t)g, (uint32_t)b + boff, it0, it1), k0, k1);
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = 4 * g + e;
      if (i < n) u[(size_t)b * n + i] = to_unit(w[e]);
    }
  }
}

}  // namespace

cudaError_t launch_uniforms(int B, int n, uint64_t seed, uint64_t iteration, float* d_u, cudaStream_t st,
                            uint32_t boff) {
  if (B <= 0 || n <= 0) return cudaSuccess;
  const long long work = (long long)B * ((n + 3) / 4);
  const int grid = (int)((work + 255) / 256 < 4096 ? (work + 255) / 256 : 4096);
  uniforms_kernel<<<grid, 256, 0, st>>>(B, n, (uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)iteration,
                                        (uint32_t)(iteration >> 32), boff, d_u);
  return cudaGetLastError();
}

// The time of a launch is the rounds of resident CTAs times the time of one round,
// estimated in us for both samplers; the shorter one is taken.
//   Step by step: a cost per step by the kernel's shape (up to 64, 1024 and 2048
// hidden units; beyond, or wide) and by the units that complete at a step.
//   In blocks: a cost per block, which holds up to 16 steps but only the steps of 16
// units, and per step; two CTAs on an SM take 1.18 times as long as one.
// The constants are fits to both kernels at 64 samples (GB300, n = 1 to 8000, h = n
// / 100 to 100 n).  With the rounds they name the slower one, by more than 5% and
// 0.7 us, in 2.4% of 13,512 measured sizes up to 65,536 samples (h <= 8 n: 1.1%, the
// worst of them 1.3 times, a call of 5 us).  What the line is for (relu, blocks | steps, us): BF16, 64
// samples, n = h = 1000 276 | 1397; n = 300, h = 4800 1862 | 409; n = 100, h = 1600
// 312 | 179; FP32, n = 1000, h = 50, 8192 samples 965 | 793.
bool sampler_stepwise(int prec, int act, int n, int h, int B, bool wide, int sms) {
  const int hp = pad_up(h), es = prec == VQMC_PREC_BF16 ? 2 : 4;
  const bool sig = act == VQMC_ACT_SIGMOID, big = hp > 2048;
  const double r = (double)h / n, m = std::min(r, 1.0);
  struct Shape {
    double step, unit, more, sigmoid;  // us per step: + unit m + more (r - 1), times 1 + sigmoid m
    int held;                          // samples an SM holds
  };
  const Shape s = wide || big    ? Shape{0.85, 0.12, 0.023, 0.17, 4}
                  : hp <= 64     ? Shape{0.83, 0.73, 0.120, 0.40, 128}
                  : hp <= 1024   ? Shape{0.90, 0.78, 0.037, 0.44, hp * es <= 1664 ? 32 : 16}
                                 : Shape{1.02, 0.24, 0.040, 0.30, 16};
  auto rounds = [&](int held) { return (double)((B + (long long)held * sms - 1) / ((long long)held * sms)); };
  double step = s.step + s.unit * m + s.more * std::max(r - 1.0, 0.0);
  if (!wide && !big) step += 0.02 * std::max(r - 40.0, 0.0);  // most units take the general form of a step
  if (es == 4) step *= sig ? 0.95 : 0.9;
  const double steps_us = (3.0 + n * step) * (sig ? 1.0 + s.sigmoid * m : 1.0) * rounds(s.held);
  const double blocks = std::min((double)n, std::max(n, h) / 16.0 + 1.0);
  double us = 1.5 + 0.13 * n + blocks * ((wide || big ? 2.2 : 1.75) + 0.00088 * hp);
  if (r > 16.0) us += n * (sig ? 1.2 : 0.4);  // the groups that have no step of their own
  if (sig) us *= 1.08 + 0.4 * m;
  double rounds_b = rounds(8);
  if (!big) {  // two CTAs of 8 samples per SM
    const int pair = 16 * sms, rest = B % pair;
    rounds_b = 1.18 * (B / pair) + (rest > 8 * sms ? 1.18 : rest > 0 ? 1.0 : 0.0);
  }
  return steps_us < us * rounds_b;
}

cudaError_t launch_sampler(const vqmc_ctx* c, int B, const float* d_u, uint64_t iteration, int8_t* d_s,
                           float* d_logp, cudaStream_t st, const unsigned long long* it_dev) {
  if (B <= 0) return cudaSuccess;
  if (c->sampler == VQMC_SAMPLER_TENSOR_CORE)
    return launch_sampler_tc(c, B, d_u, iteration, d_s, d_logp, st, nullptr, nullptr, nullptr, it_dev);
  SamplerArgs a{};
  a.n = c->n;
  a.h = c->h;
  a.hp = c->hp;
  a.B = B;
  a.wt = c->wt_s;
  a.v = c->v_s;
  a.b1 = c->b1;
  a.b2 = c->b2;
  a.u = d_u;
  a.key0 = (uint32_t)c->cfg.seed;
  a.key1 = (uint32_t)(c->cfg.seed >> 32);
  a.it0 = (uint32_t)iteration;
  a.it1 = (uint32_t)(iteration >> 32);
  a.boff = c->sample_offset;
  a.it_dev = it_dev;
  a.s_out = d_s;
  a.logp = d_logp;
  a.err = c->err;
  a.act = c->act;
  a.wide = c->sampler_wide;
  if (sampler_stepwise(c->prec, c->act, c->n, c->h, B, a.wide, c->num_sms))
    return c->prec == VQMC_PREC_BF16 ? launch_sampler_steps_wt<bf16>(a, st) : launch_sampler_steps_wt<float>(a, st);
  return c->prec == VQMC_PREC_BF16 ? launch_sampler_wt<bf16>(a, st) : launch_sampler_wt<float>(a, st);
}

}  // namespace vqmc
