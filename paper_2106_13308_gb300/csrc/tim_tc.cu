// Off-diagonal local energy of the transverse-field Ising model for the BF16
// model, in one kernel: the flipped states' hidden activations, the output
// layer on the tcgen05 tensor cores, log pi and the sum over the flips.
//
// As in tim.cu, flipping spin i moves the hidden pre-activations by a rank-1
// term, a_k(x^(i)) = a_k(x) - 2 s_i W1_ki, and the outputs before spin i have
// the same terms in log pi(x^(i)) and log pi(x).  A tile is 128 rows of the
// expansion: each of its four groups of 32 rows (one per epilogue warp pair)
// holds, for `spw` samples, `seg` consecutive flips and the sample itself (the
// base row), so that
//     Delta_i = log pi(x^(i)) - log pi(x),   sum_i alpha_i exp(Delta_i / 2)
// are formed inside a warp.  With seg = 31 the flips of a tile start at
// output tile t0 = 31 j / 128 and the tiles before it are skipped; the four
// samples of a tile share the rows of W1 it reads.  seg = n and several
// samples per group below 31 spins.
//
// Persistent CTAs of 10 warps, two per SM up to 256 hidden units: warps 0-7
// build the tile's operand (128 rows x hp BF16, 128-byte swizzle) in shared
// memory, then read the accumulators (warp w: rows 32 (w % 4) .., columns
// 64 (w / 4) .. of each 128-column output tile); warp 8 streams W2 tiles
// (128 outputs x 64 units) with TMA; warp 9 issues the MMAs into two
// accumulators, so that one output tile's epilogue runs beside the next
// one's MMAs.  They wait with try_wait, which suspends: polling took a fifth of
// the epilogue's issue slots.  Every wait is bounded: after a failed one the CTA
// raises the timeout bit and runs on without waiting.
//
// What bounds it: the issue slots of the epilogue, an exponential and a logarithm for
// every output of the tiles that are not skipped (185 M at n = 500, B = 1024, of which
// the B n n / 2 = 128 M that do not cancel are wanted).  Measured there, h = 193
// (GB300), a training step: 1141 us with the rows and their spins written to
// memory and read back by the general GEMM, 432 us with this kernel (0.21 ms
// of it; 145 M warp instructions, 61% of the issue slots).
#include <algorithm>

#include "gemm.cuh"
#include "tc_ptx.cuh"

namespace vqmc {
namespace {

using namespace tc;

constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (kEpiWarps + 2);
constexpr int kRows = 128;                    // rows per tile, outputs per output tile
constexpr int kTileBytes = 128 * 64 * 2;      // one 128 x 64 BF16 tile
constexpr int kMaxStages = 6;
constexpr int kMaxSeg = 31;                   // flips of one sample in a tile
constexpr int kMaxHp = 640;                   // the operand (hp / 64 tiles) and three stages in shared memory
constexpr int kTmemCols = 256;                // two accumulators of 128 columns
constexpr uint32_t kIdesc = idesc_bf16(128, 128);
// after the operand and the ring: barriers | slot, abort | bias per warp | halves' sums
constexpr int kOffAux = 256;
constexpr int kOffBias = kOffAux + 16;
constexpr int kOffSum = kOffBias + kEpiWarps * 64 * 4;
constexpr int kMisc = kOffSum + 2 * kRows * 4;

struct TimArgs {
  int n, h, hp, B, seg, spw, stages;
  int sblocks;          // blocks of 4 spw samples
  long long tiles;      // sblocks x blocks of seg flips
  const int8_t* S;      // [B][n]
  const float* A;       // [B][hp] pre-activations of the samples
  const float* W1t;     // [n][h] master weights
  const float* b2;
  const float* alpha;
  double* part;         // [blocks of flips][B]
  uint32_t* err;
};

// log sigma(x) = min(x, 0) - ln 2 log2(1 + 2^(-|x| log2 e)) on the hardware's
// exp2 and log2; subnormals are flushed, which 1 + .. absorbs
__device__ __forceinline__ float log_sigmoid_fast(float x) {
  float e, l;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(fabsf(x) * -1.44269504f));
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(1.0f + e));
  return fmaf(l, -0.69314718f, fminf(x, 0.0f));
}

template <int ACT>
__device__ __forceinline__ float act1(float a) {
  if constexpr (ACT == VQMC_ACT_RELU) return fmaxf(a, 0.0f);
  else return 1.0f / (1.0f + expf(-a));
}

template <int ACT>
__global__ void __launch_bounds__(kThreads, 2)
    tim_fused_kernel(const __grid_constant__ CUtensorMap mapV, const TimArgs g) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  const int nkc = g.hp / 64;                                   // 64-unit chunks of the operand
  const uint32_t ring = base + (uint32_t)nkc * kTileBytes;
  unsigned char* misc = sm + (nkc + g.stages) * kTileBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(misc);
  uint64_t* empty = full + kMaxStages;
  uint64_t* accfull = empty + kMaxStages;
  uint64_t* accempty = accfull + 2;
  uint64_t* aready = accempty + 2;
  uint64_t* drain = aready + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + kOffAux);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* sums = reinterpret_cast<float*>(misc + kOffSum);      // [2][kRows]

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const int n = g.n, h = g.h;
  const int ntiles = (n + kRows - 1) / kRows;
  if (tid == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&accfull[s]), 1);
      mbar_init(smem_u32(&accempty[s]), 32 * kEpiWarps);
    }
    mbar_init(smem_u32(aready), 32 * kEpiWarps);
    mbar_init(smem_u32(drain), 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpiWarps + 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = (uint32_t)uniform((int)*tmem_slot);

  // Tiles in order of the flip block (heaviest first), sample blocks inside;
  // CTA c takes every gridDim-th tile, so that all CTAs work on flip blocks
  // of about the same number of output tiles.
  // K chunks of output tile t: units complete before its last output
  auto chunks = [&](int t) {
    int lo, hi;
    gemm_k_range(kOpOut, t * kRows, min(t * kRows + kRows, n), h, n, h, &lo, &hi);
    return (hi + 63) / 64;
  };

  if (warp == kEpiWarps) {
    // ------------------------------------------------------------ producer
    if (elect_one()) {
      int it = 0;
      bool ok = true;
      for (long long q = blockIdx.x; q < g.tiles && ok; q += gridDim.x) {
        const int j = (int)(q / g.sblocks);
        for (int t = j * g.seg / kRows; t < ntiles && ok; ++t) {
          const int nk = chunks(t);
          for (int c = 0; c < nk; ++c, ++it) {
            const int s = it % g.stages;
            if (it >= g.stages &&
                !wait_or_abort(smem_u32(&empty[s]), (uint32_t)((it / g.stages - 1) & 1), abort, g.err)) {
              ok = false;
              break;
            }
            mbar_expect_tx(smem_u32(&full[s]), kTileBytes);
            tma_load_2d(ring + (uint32_t)(s * kTileBytes), &mapV, 64 * c, t * kRows, smem_u32(&full[s]));
          }
        }
      }
      // no copy may still be landing when the CTA exits
      for (int p = it > g.stages ? it - g.stages : 0; p < it; ++p)
        mbar_wait(smem_u32(&full[p % g.stages]), (uint32_t)((p / g.stages) & 1), g.err);
    }
  } else if (warp == kEpiWarps + 1) {
    // ---------------------------------------------------------- MMA issuer
    if (elect_one()) {
      int it = 0, acc = 0, turn = 0;
      bool ok = true;
      for (long long q = blockIdx.x; q < g.tiles && ok; q += gridDim.x, ++turn) {
        const int j = (int)(q / g.sblocks);
        ok = wait_or_abort(smem_u32(aready), (uint32_t)(turn & 1), abort, g.err);
        fence_after();
        for (int t = j * g.seg / kRows; t < ntiles && ok; ++t, ++acc) {
          const int nk = chunks(t), buf = acc & 1;
          if (acc >= 2) {
            ok = wait_or_abort(smem_u32(&accempty[buf]), (uint32_t)((acc / 2 - 1) & 1), abort, g.err);
            fence_after();
          }
          for (int c = 0; c < nk && ok; ++c, ++it) {
            const int s = it % g.stages;
            ok = wait_or_abort(smem_u32(&full[s]), (uint32_t)((it / g.stages) & 1), abort, g.err);
            if (!ok) break;
            fence_after();
            const uint64_t da = smem_desc_sw128(base + (uint32_t)(c * kTileBytes));
            const uint64_t db = smem_desc_sw128(ring + (uint32_t)(s * kTileBytes));
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_bf16(tmem + (uint32_t)(128 * buf), da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), kIdesc,
                       (c > 0 || k > 0) ? 1u : 0u);
            mma_commit(smem_u32(&empty[s]));
          }
          if (ok && nk > 0) mma_commit(smem_u32(&accfull[buf]));
          else mbar_arrive(smem_u32(&accfull[buf]));
        }
      }
      // every MMA has completed before tensor memory is released
      mma_commit(smem_u32(drain));
      mbar_wait(smem_u32(drain), 0u, g.err);
    }
  } else {
    // ------------------------------------------- operand, log pi, the sums
    const int quad = warp & 3, half = warp >> 2;
    const int seg = g.seg, spw = g.spw, per = seg + 1;
    const int s_in = lane / per, idx = lane % per;  // this lane's row: sample and flip (seg: the base row)
    float* bias = reinterpret_cast<float*>(misc + kOffBias) + warp * 64;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(64 * half);
    int acc = 0;
    for (long long q = blockIdx.x; q < g.tiles; q += gridDim.x) {
      const int j = (int)(q / g.sblocks), sb = (int)(q - (long long)j * g.sblocks);
      // the operand: flip rows warp, warp + 8, .. of every sample; a lane owns
      // two adjacent units of each chunk.  The previous tile's MMAs have
      // completed (its last accumulator was waited for).
#pragma unroll 1
      for (int s = 0; s < spw; ++s) {
#pragma unroll 1
        for (int k0 = 0; k0 < g.hp; k0 += 256) {
          const int np = min(4, (g.hp - k0) / 64);  // chunks of this pass
          float2 a[4][4];
          int b[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            b[u] = (sb * 4 + u) * spw + s;
#pragma unroll
            for (int p = 0; p < 4; ++p)
              a[u][p] = (b[u] < g.B && p < np)
                            ? __ldg(reinterpret_cast<const float2*>(g.A + (size_t)b[u] * g.hp + k0 + 64 * p + 2 * lane))
                            : make_float2(0.0f, 0.0f);
          }
#pragma unroll 2
          for (int f = warp; f <= seg; f += kEpiWarps) {
            const int i = j * seg + f;
            const bool flip = f < seg && i < n;
            const float* wrow = g.W1t + (size_t)(flip ? i : 0) * h + k0 + 2 * lane;
            float2 w[4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              const int k = k0 + 64 * p + 2 * lane;
              w[p].x = k < h ? __bfloat162float(__float2bfloat16_rn(__ldg(wrow + 64 * p))) : 0.0f;
              w[p].y = k + 1 < h ? __bfloat162float(__float2bfloat16_rn(__ldg(wrow + 64 * p + 1))) : 0.0f;
            }
            // units past h: activation of the zero padding of A, times zero weights
            unsigned char* row = sm + (size_t)(k0 / 64) * kTileBytes + sw128_offset(s * per + f, 2 * lane);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float two_s = flip && b[u] < g.B ? 2.0f * (float)__ldg(g.S + (size_t)b[u] * n + i) : 0.0f;
#pragma unroll
              for (int p = 0; p < 4; ++p) {
                if (p >= np) break;
                *reinterpret_cast<__nv_bfloat162*>(row + p * kTileBytes + u * 4096) =
                    __floats2bfloat162_rn(act1<ACT>(a[u][p].x - two_s * w[p].x), act1<ACT>(a[u][p].y - two_s * w[p].y));
              }
            }
          }
        }
      }
      fence_proxy_async();
      fence_before();
      mbar_arrive(smem_u32(aready));

      const int bme = (sb * 4 + quad) * spw + s_in, ime = j * seg + idx;
      double delta = 0.0;  // Delta of this lane's row
#pragma unroll 1
      for (int t = j * seg / kRows; t < ntiles; ++t, ++acc) {
        const int c0 = t * kRows + 64 * half, buf = acc & 1;
        // b2 of the warp's columns (columns past the last output get a logit
        // of 1e30, whose log sigma is exactly 0) and the row's spins as sign bits
        __syncwarp();
        bias[lane] = c0 + lane < n ? __ldg(g.b2 + c0 + lane) : 1e30f;
        bias[lane + 32] = c0 + 32 + lane < n ? __ldg(g.b2 + c0 + 32 + lane) : 1e30f;
        uint32_t neg0 = 0, neg1 = 0;
#pragma unroll 1
        for (int s = 0; s < spw; ++s) {
          const int b = (sb * 4 + quad) * spw + s;
          const int8_t* src = g.S + (size_t)b * n + c0 + lane;
          const uint32_t m0 = __ballot_sync(0xffffffffu, b < g.B && c0 + lane < n && __ldg(src) < 0);
          const uint32_t m1 = __ballot_sync(0xffffffffu, b < g.B && c0 + 32 + lane < n && __ldg(src + 32) < 0);
          if (s == s_in) neg0 = m0, neg1 = m1;
        }
        if (idx < seg && ime < n) {  // the flipped spin
          neg0 ^= (uint32_t)(ime - c0) < 32u ? 1u << (ime - c0) : 0u;
          neg1 ^= (uint32_t)(ime - c0 - 32) < 32u ? 1u << (ime - c0 - 32) : 0u;
        }
        __syncwarp();
        wait_or_abort(smem_u32(&accfull[buf]), (uint32_t)((acc >> 1) & 1), abort, g.err);
        __syncwarp();
        fence_after();
        // warp-uniform: tcgen05.ld is executed by all lanes of a warp or none
        const bool live = !__any_sync(0xffffffffu, *abort != 0) && chunks(t) > 0;
        float rs = 0.0f;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float v[16];
          if (live) {
            tmem_ld16(trow + (uint32_t)(128 * buf + 16 * c), v);
          } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = 0.0f;
          }
          const uint32_t neg = ((c & 2) ? neg1 : neg0) >> (16 * (c & 1));
          const float4* bv = reinterpret_cast<const float4*>(bias + 16 * c);
#pragma unroll
          for (int e4 = 0; e4 < 4; ++e4) {
            const float4 bb = bv[e4];
            const float bq[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float z = v[4 * e4 + e] + bq[e];
              const float x = __int_as_float(__float_as_int(z) ^ (int)((neg << (31 - 4 * e4 - e)) & 0x80000000u));
              rs += log_sigmoid_fast(x);
            }
          }
        }
        fence_before();
        mbar_arrive(smem_u32(&accempty[buf]));
        // the two column halves of a row, less the base row
        float* sum = sums + (buf * 4 + quad) * 32;
        if (half == 1) sum[lane] = rs;
        asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory");
        if (half == 0) {
          const float p = rs + sum[lane];
          delta += (double)p - (double)__shfl_sync(0xffffffffu, p, min(s_in * per + seg, 31));
        }
      }
      if (half == 0) {  // the sum over the flips
        const bool mine = s_in < spw && idx < seg && ime < n && bme < g.B;
        const double term = mine ? (double)__ldg(g.alpha + ime) * exp(0.5 * delta) : 0.0;
#pragma unroll 1
        for (int s = 0; s < spw; ++s) {
          double x = s == s_in ? term : 0.0;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
          const int b = (sb * 4 + quad) * spw + s;
          if (lane == 0 && b < g.B) g.part[(size_t)j * g.B + b] = x;
        }
      }
    }
  }

  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == kEpiWarps + 1) {
    fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// E[b] -= the flip blocks' sums, in order
__global__ void tim_finish_kernel(int B, int blocks, const double* __restrict__ part, float* __restrict__ E) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  double acc = 0.0;
  for (int j = 0; j < blocks; ++j) acc += part[(size_t)j * B + b];
  E[b] = (float)((double)E[b] - acc);
}

int seg_of(int n) { return std::min(n, kMaxSeg); }
int blocks_of(int n) { return (n + seg_of(n) - 1) / seg_of(n); }

// Ring stages: as many as let two CTAs share an SM if that leaves at least
// two, else as many as fit one CTA (hp up to kMaxHp leaves three).
int stages_of(int hp) {
  const int a = hp / 64 * kTileBytes + kMisc + 1024;
  const int two = (113 * 1024 - a) / kTileBytes, one = (227 * 1024 - a) / kTileBytes;
  return std::min(kMaxStages, a < 113 * 1024 && two >= 2 ? two : one);
}

OncePerDevice g_smem;


// Estimated time in us of both forms of an energy call, without what they share (the
// model's constants, fitted on a GB300 to 5,662 sizes: n = 1 to 500, h = 10 to 640,
// 1 to 4096 samples).  Here: rounds of resident CTAs, each with the operand of one
// tile (a sigmoid costs three times a relu) and the average of its output tiles.
// tim.cu: rows through memory, on the whole chip even where this kernel has few tiles,
// and a fixed cost for its launches.
struct Times {
  double tile;       // us of one round
  long long blocks;  // of flips
  int spw, per_sm;
  double rows;       // us per row of the general form
};
Times times_of(int act, int n, int hp) {
  const int seg = seg_of(n), nt = (n + kRows - 1) / kRows, blocks = blocks_of(n);
  double tiles = 0.0;
  for (int j = 0; j < blocks; ++j) tiles += nt - j * seg / kRows;
  const bool sig = act == VQMC_ACT_SIGMOID;
  return {hp / 64 * (sig ? 3.25 : 1.12) + 5.3 * tiles / blocks, blocks, 32 / (seg + 1),
          hp / 64 * kTileBytes + kMisc + 1024 + 2 * kTileBytes <= 113 * 1024 ? 2 : 1,
          1e-6 * (hp * (sig ? 1.9 : 1.2) + 445.0 * nt - 0.84 * n)};
}
bool faster(const Times& t, int n, int B, int sms) {
  if (n <= 2) return false;  // 1 or 2 flips for the 32 rows of a warp
  const long long tiles = t.blocks * ((B + 4 * t.spw - 1) / (4 * t.spw)), round = (long long)t.per_sm * sms;
  const double here = 21.2 + 0.0087 * n + t.tile * (double)((tiles + round - 1) / round);
  return here <= 28.9 + 0.069 * n + t.rows * (double)B * (n + 1);
}

}  // namespace

// The operand of hp units has to fit shared memory beside the ring, and the call has
// to be faster here than through tim.cu's row workspace and the general GEMM.  The
// estimate names the slower form, by more than 5% and 1 us, at 147 of 5,662 measured
// sizes, by at most 23%.  What the line is for (us, here | there): n = 64, h = 640, sigmoid,
// 1024 samples 242 | 130; n = 8, h = 640, sigmoid, 128 samples 74 | 38; n = 500, h = 192,
// relu, 1024 samples 236 | 761.
bool tim_tc_applies(int prec, int act, int n, int hp, int B, int sms) {
  return prec == VQMC_PREC_BF16 && hp <= kMaxHp && faster(times_of(act, n, hp), n, B, sms);
}

int tim_general_batch(int prec, int act, int n, int hp, int Bmax, int sms) {
  if (prec != VQMC_PREC_BF16 || hp > kMaxHp) return Bmax;
  const Times t = times_of(act, n, hp);
  int B = Bmax;
  while (B > 0 && faster(t, n, B, sms)) --B;
  return B;
}

size_t tim_tc_part_bytes(int Bmax, int n) { return (size_t)blocks_of(n) * (size_t)Bmax * sizeof(double); }

cudaError_t launch_tim_tc(const vqmc_ctx* c, int B, const int8_t* d_s, float* d_e, cudaStream_t st, int* launches) {
  CUtensorMap mapV;
  if (!tc_encode_bf16(&mapV, c->v_s, sampler_rows(c->n), c->hp, c->hp, kRows)) return cudaErrorInvalidValue;
  TimArgs a{};
  a.n = c->n, a.h = c->h, a.hp = c->hp, a.B = B;
  a.seg = seg_of(c->n), a.spw = 32 / (a.seg + 1);
  a.stages = stages_of(c->hp);
  a.sblocks = (B + 4 * a.spw - 1) / (4 * a.spw);
  const int blocks = blocks_of(c->n);
  a.tiles = (long long)a.sblocks * blocks;
  a.S = d_s, a.A = c->tim_A, a.W1t = c->theta, a.b2 = c->b2, a.alpha = c->alpha;
  a.part = (double*)c->tim_part;
  a.err = c->err;
  const int smem = 1024 + (c->hp / 64 + a.stages) * kTileBytes + kMisc;
  const auto kernels = {tim_fused_kernel<VQMC_ACT_RELU>, tim_fused_kernel<VQMC_ACT_SIGMOID>};
  cudaError_t e = allow_smem(g_smem, kernels, 227 * 1024);
  if (e != cudaSuccess) return e;
  const long long resident = (long long)c->num_sms * (smem <= 113 * 1024 ? 2 : 1);
  const int grid = (int)std::min(a.tiles, resident);
  if (c->act == VQMC_ACT_RELU) tim_fused_kernel<VQMC_ACT_RELU><<<grid, kThreads, smem, st>>>(mapV, a);
  else tim_fused_kernel<VQMC_ACT_SIGMOID><<<grid, kThreads, smem, st>>>(mapV, a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  tim_finish_kernel<<<(B + 127) / 128, 128, 0, st>>>(B, blocks, a.part, d_e);
  if (launches) *launches += 2;
  return cudaGetLastError();
}

}  // namespace vqmc
