// CUDA-core (FFMA) implementation of the masked GEMMs with fused epilogues:
// the plain FP32 precision (FP32 operands, FP32 accumulation).  The BF16
// precision runs the same GEMMs on the tcgen05 tensor cores (gemm_tc.cu).
//
// 256 threads, TM x TN outputs per thread (rows m0 + TM ty + i, columns
// n0 + 64 q + 4 tx + j, j < 4), K in steps of 16 through a ring of stages filled
// by 16-byte cp.async copies.  A is K-contiguous and stays so in shared memory
// (rows of 16 floats, padded to 20); B comes from its [K][N] form, which every
// operand here has beside the other, so that neighbouring columns are pairs for
// the packed multiply-adds (fma.rn.f32x2: half the issue slots of scalar ones).
// Per four K values a thread reads TM + TN times 16 bytes for 2 TM TN packed
// multiply-adds.  Every output is one chain over K in order (a split K: one
// chain per part, the parts added in order).
//
// What bounds it: the FP32 pipe and, at 128 x 128, the registers that two CTAs
// per SM leave (128 a thread).  Measured (GB300) at n = 10000, h = 2000, 2048
// samples, where a GEMM's 2.05e10 multiply-adds take 509 us at the derived peak
// of 80 TFLOP/s, against 128 x 128 x 16 tiles transposed through registers with
// scalar multiply-adds: hidden 1830 -> 956 us, output 1313 -> 862, hidden adjoint
// 1746 -> 914, weight gradients 1270 -> 990.  (4-byte copies that transposed both
// operands on the way cost more than they saved below 128 x 128: hidden 1445 us.)
// Small models: the weight gradients of n = 20, h = 40, 1024 samples, one tile,
// 144 -> 12 us with the batch split.
#include <algorithm>

#include "f32x2.cuh"
#include "gemm.cuh"

namespace vqmc {
namespace {

constexpr int BK = 16, kThreads = 256;

template <int TM, int TN>
struct Tile {
  static constexpr int BM = 16 * TM, BN = 16 * TN;
  static constexpr int kStages = TM * TN >= 64 ? 3 : 4;
  // A rows TM ty + i of 20 floats, 4 floats more every TM rows: the two ty of
  // a warp on different banks
  static constexpr int kLdA = 20, kA = BM * kLdA + 16 * 4;
  static constexpr int kStage = kA + BK * BN;
  static constexpr int kSmem = kStages * kStage * 4;
};

__device__ __forceinline__ float sigmoidf_(float x) { return 1.0f / (1.0f + expf(-x)); }

// 16 bytes to shared memory, the first `bytes` of them from src, zeros beyond
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// four consecutive floats; one 16-byte access where the address allows it and
// all four are inside
__device__ __forceinline__ void store4(float* p, const float (&x)[4], int valid) {
  if (valid >= 4 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < valid) p[j] = x[j];
  }
}
// signs of four consecutive spins (the first `valid`; +1 beyond)
__device__ __forceinline__ void spins4(const int8_t* p, int valid, float (&s)[4]) {
  uint32_t w = 0x01010101u;
  if (valid >= 4 && (reinterpret_cast<uintptr_t>(p) & 3) == 0) {
    w = __ldg(reinterpret_cast<const uint32_t*>(p));
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j < valid && p[j] < 0) w |= 0x80u << (8 * j);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) s[j] = (w >> (8 * j + 7)) & 1u ? -1.0f : 1.0f;
}

template <int OP, int TM, int TN>
__global__ void __launch_bounds__(kThreads, 2) gemm_simt_kernel(const GemmArgs<float> g, int kpart) {
  using T = Tile<TM, TN>;
  constexpr int BM = T::BM, BN = T::BN, kStages = T::kStages;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  constexpr int op = OP;
  // Tiles in launch order, heaviest K range first where the masks make the
  // ranges uneven (as in gemm_tc.cu)
  int tm = blockIdx.y, tn = blockIdx.x;
  if (op == kOpHidden || op == kOpGA || op == kOpOut) {
    const int L = blockIdx.y * gridDim.x + blockIdx.x;
    tm = L % gridDim.y;
    tn = op == kOpGA ? L / (int)gridDim.y : (int)gridDim.x - 1 - L / (int)gridDim.y;
  }
  const int m0 = tm * BM, n0 = tn * BN;
  const int m1 = min(m0 + BM, g.M), n1 = min(n0 + BN, g.N);
  constexpr bool wgrad = op == kOpDV || op == kOpDW;
  // Columns of a thread: 4 tx .. + 3 of each 64, or, where it sums along the
  // row, 8 tx .. + 7 (eight neighbours summed in order, then a tree over tx: the
  // energies that enter the gradient keep the sums' order).  The 16-byte pieces
  // of a B row lie in shared memory in the order in which the threads read them.
  constexpr bool kRowSum = op == kOpOut || op == kOpEloc;
  auto column = [&](int q) { return kRowSum ? 8 * tx + 4 * q : 64 * q + 4 * tx; };
  if (wgrad && gemm_tile_masked(op, m0, m1, n0, n1, g.n, g.h)) {
    if (gridDim.z == 1)
      for (int q = tid; q < BM * BN; q += kThreads) {
        const int m = m0 + q / BN, nn = n0 + q % BN;
        if (m < g.M && nn < g.N) g.gout[(size_t)m * g.ldg + nn] = 0.0f;
      }
    return;
  }
  if (op == kOpOut && g.flip_rows) {
    // single-flip rows of the transverse field: a tile whose columns all
    // precede the flipped spin of each of its rows (one sample, no unflipped
    // row) contributes nothing the log-ratios read, so it is skipped
    const int ia = (int)((g.row0 + m0) % (g.n + 1));
    if (ia + m1 - 1 - m0 < g.n && n0 + BN <= ia) return;
  }
  int klo, khi;
  gemm_k_range(op, n0, n1, g.K, g.n, g.h, &klo, &khi);
  klo = klo / BK * BK;
  if (gridDim.z > 1) klo = blockIdx.z * kpart, khi = min(khi, klo + kpart);
  const int nk = khi > klo ? (khi - klo + BK - 1) / BK : 0;

  // A: a thread copies the 16 bytes tid % 4 of rows tid / 4, + 64, ...; B: 16
  // bytes of the stage's 16 rows of BN floats
  const int cr = tid >> 2, ck = 4 * (tid & 3);
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
  auto issue = [&](int it) {
    if (it < nk) {
      const int k0 = klo + it * BK;
      const uint32_t dst = base + (it % kStages) * T::kStage * 4;
      const int bytes = max(0, min(16, 4 * (khi - k0 - ck)));
#pragma unroll
      for (int r = 0; r < BM; r += 64) {
        const int m = m0 + cr + r;
        const bool in = m < g.M && bytes > 0;
        cp16(dst + 4 * ((cr + r) * T::kLdA + (cr + r) / TM * 4 + ck), g.A + (in ? (size_t)m * g.lda + k0 + ck : 0),
             in ? bytes : 0);
      }
#pragma unroll
      for (int q = 0; q < BK * BN / 4; q += kThreads) {
        const int r = (q + tid) / (BN / 4), c = (q + tid) % (BN / 4) * 4;
        const bool in = k0 + r < khi && n0 + c < g.ldb;  // ldb: N padded to a multiple of 64
        const int place = kRowSum ? c / 8 * 4 + (c & 4) * 16 : c;
        cp16(dst + 4 * (T::kA + r * BN + place), g.Bm + (in ? (size_t)(k0 + r) * g.ldb + n0 + c : 0), in ? 16 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  uint64_t acc2[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc2[i][j] = 0ull;
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) issue(s);
  for (int it = 0; it < nk; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // stage it has landed for all; stage it - 1 is free
    issue(it + kStages - 1);
    const float* as = sm + (it % kStages) * T::kStage + TM * ty * T::kLdA + 4 * ty;
    const float* bs = sm + (it % kStages) * T::kStage + T::kA + 4 * tx;
#pragma unroll
    for (int k4 = 0; k4 < BK; k4 += 4) {
      float4 a[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(as + i * T::kLdA + k4);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        uint64_t b[TN / 2];
#pragma unroll
        for (int q = 0; q < TN / 4; ++q) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(bs + (k4 + kk) * BN + 64 * q);
          b[2 * q] = v.x, b[2 * q + 1] = v.y;
        }
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const float av = kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w;
          const uint64_t ai = pack2(av, av);
#pragma unroll
          for (int j = 0; j < TN / 2; ++j) acc2[i][j] = fma2(ai, b[j], acc2[i][j]);
        }
      }
    }
  }

  // ---------------------------------------------------------------- epilogue
  // columns in groups of four: group q starts at n0 + column(q)
  const int mb = m0 + ty * TM;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) unpack2(acc2[i][j], acc[i][2 * j], acc[i][2 * j + 1]);
  if constexpr (wgrad) {
    const bool split = gridDim.z > 1;  // parts are stored as they are, the sum over them applies the mask
    float* out = split ? g.part + (size_t)blockIdx.z * g.M * g.N : g.gout;
    const int ld = split ? g.N : g.ldg;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if (mb + i >= g.M) continue;
      const int cd = count_deg_le(mb + i, g.n, g.h);  // kept: W2 columns below it, W1^T columns from it on
#pragma unroll
      for (int q = 0; q < TN / 4; ++q) {
        const int nn = n0 + 64 * q + 4 * tx;
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = split || (nn + j < cd) == (op == kOpDV) ? acc[i][4 * q + j] : 0.0f;
        store4(out + (size_t)(mb + i) * ld + nn, x, g.N - nn);
      }
    }
    return;
  }

  float rowsum[TM], colsum[TN];
#pragma unroll
  for (int i = 0; i < TM; ++i) rowsum[i] = 0.0f;
#pragma unroll
  for (int j = 0; j < TN; ++j) colsum[j] = 0.0f;
  // TM consecutive rows of column nn of the transposed output
  auto store_t = [&](int nn, const float (&x)[TM]) {
    if (nn >= g.N) return;
    float* o = g.out_t + (size_t)nn * g.ldt + mb;  // ldt: a multiple of 64
    if (mb + TM <= g.M) {
#pragma unroll
      for (int i = 0; i < TM; i += 4) *reinterpret_cast<float4*>(o + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
    } else {
#pragma unroll
      for (int i = 0; i < TM; ++i)
        if (mb + i < g.M) o[i] = x[i];
    }
  };
#pragma unroll
  for (int q = 0; q < TN / 4; ++q) {
    const int nn = n0 + column(q), valid = g.N - nn;
    if (valid <= 0) continue;
    float bias[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if constexpr (op == kOpHidden || op == kOpOut)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < valid) bias[j] = g.bias[nn + j];
    float t[4][TM];  // values for the transposed output
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int m = mb + i;
      float x[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      if (m < g.M) {
        if constexpr (op == kOpHidden) {
          float a[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            a[j] = acc[i][4 * q + j] + bias[j];
            x[j] = g.act == VQMC_ACT_RELU ? fmaxf(a[j], 0.0f) : sigmoidf_(a[j]);
          }
          if (g.pre) store4(g.pre + (size_t)m * g.ldpre + nn, a, valid);
          store4(g.out + (size_t)m * g.ldo + nn, x, valid);
        } else if constexpr (op == kOpOut) {
          // with e = exp(-|x|): log sigma(x) = min(x, 0) - log(1 + e) and
          // sigma(-x) = (x >= 0 ? e : 1) / (1 + e), on the hardware exp2 / log2
          // approximations and the approximate division
          float s[4];
          spins4(g.S8 + (size_t)m * g.lds8 + nn, valid, s);
          const float cm = g.coef ? g.coef[m] : 0.0f;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float z = s[j] * (acc[i][4 * q + j] + bias[j]), e = __expf(-fabsf(z));
            if (j < valid) rowsum[i] += fminf(z, 0.0f) - __logf(1.0f + e);
            if (g.coef && j < valid) {
              x[j] = cm * s[j] * __fdividef(z >= 0.0f ? e : 1.0f, 1.0f + e);
              colsum[4 * q + j] += x[j];
            }
          }
          if (g.coef) store4(g.out + (size_t)m * g.ldo + nn, x, valid);
        } else if constexpr (op == kOpGA) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < valid) {
              const float hv = g.aux[(size_t)m * g.ldaux + nn + j];
              x[j] = acc[i][4 * q + j] * (g.act == VQMC_ACT_RELU ? (hv > 0.0f ? 1.0f : 0.0f) : hv * (1.0f - hv));
              colsum[4 * q + j] += x[j];
            }
          store4(g.out + (size_t)m * g.ldo + nn, x, valid);
        } else {
          float s[4];
          spins4(g.S8 + (size_t)m * g.lds8 + nn, valid, s);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < valid) rowsum[i] = fmaf(0.5f * s[j], acc[i][4 * q + j], rowsum[i]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) t[j][i] = x[j];
    }
    if constexpr (op == kOpHidden || op == kOpOut || op == kOpGA)
      if (g.out_t && (op != kOpOut || g.coef))
#pragma unroll
        for (int j = 0; j < 4; ++j) store_t(nn + j, t[j]);
  }

  // row partials: reduce over the 16 tx lanes of each half-warp
  if (g.row_part && (op == kOpOut || op == kOpEloc)) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      float v = rowsum[i];
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      if (tx == 0 && mb + i < g.M) g.row_part[(size_t)tn * g.ldr + mb + i] = v;
    }
  }
  // column partials: reduce over the 16 ty rows in a fixed order
  if (g.col_part && ((op == kOpOut && g.coef) || op == kOpGA)) {
    __syncthreads();  // the operand stages are consumed
    float(*colbuf)[BN] = reinterpret_cast<float(*)[BN]>(sm);
#pragma unroll
    for (int j = 0; j < TN; ++j) colbuf[ty][column(j / 4) + j % 4] = colsum[j];
    __syncthreads();
    if (tid < BN) {
      float v = 0.0f;
#pragma unroll
      for (int q = 0; q < 16; ++q) v += colbuf[q][tid];
      if (n0 + tid < g.N) g.col_part[(size_t)tm * g.ldc + n0 + tid] = v;
    }
  }
}

// The parts of a split K, added in order; zero outside the mask.  One row per
// blockIdx.y.
__global__ void wgrad_sum_kernel(int op, int M, int N, int parts, const float* __restrict__ part, int n, int h,
                                 float* __restrict__ gout, int ldg) {
  const int m = blockIdx.y, nn = blockIdx.x * blockDim.x + threadIdx.x;
  if (nn >= N) return;
  float s = 0.0f;
  if ((nn < count_deg_le(m, n, h)) == (op == kOpDV)) {
    const float* p = part + (size_t)m * N + nn;
#pragma unroll 1
    for (int z = 0; z < parts; z += 8) {  // eight loads in flight: their latency bounds the sum
      float x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = z + q < parts ? p[(size_t)(z + q) * M * N] : 0.0f;
#pragma unroll
      for (int q = 0; q < 8; ++q) s += x[q];  // (a zero past the last part changes nothing: s is never -0)
    }
  }
  gout[(size_t)m * ldg + nn] = s;
}

long long tiles(int M, int N, int BM, int BN) { return (long long)((M + BM - 1) / BM) * ((N + BN - 1) / BN); }

template <int OP, int TM, int TN>
cudaError_t launch_op(const GemmArgs<float>& a, int parts, int kpart, cudaStream_t st) {
  using T = Tile<TM, TN>;
  auto kern = gemm_simt_kernel<OP, TM, TN>;
  static OncePerDevice smem;
  const cudaError_t e = allow_smem(smem, std::initializer_list<decltype(kern)>{kern}, T::kSmem);
  if (e != cudaSuccess) return e;
  const dim3 grid((a.N + T::BN - 1) / T::BN, (a.M + T::BM - 1) / T::BM, parts);
  kern<<<grid, kThreads, T::kSmem, st>>>(a, kpart);
  if (parts > 1)
    wgrad_sum_kernel<<<dim3((a.N + 127) / 128, a.M), 128, 0, st>>>(a.op, a.M, a.N, parts, a.part, a.n, a.h, a.gout,
                                                                   a.ldg);
  return cudaGetLastError();
}

template <int TM, int TN>
cudaError_t launch_tile(const GemmArgs<float>& a, int parts, int kpart, cudaStream_t st) {
  switch (a.op) {
    case kOpHidden: return launch_op<kOpHidden, TM, TN>(a, 1, 0, st);
    case kOpDV: return launch_op<kOpDV, TM, TN>(a, parts, kpart, st);
    case kOpGA: return launch_op<kOpGA, TM, TN>(a, 1, 0, st);
    case kOpDW: return launch_op<kOpDW, TM, TN>(a, parts, kpart, st);
  }
  if constexpr (TN == 8) {  // a row partial per 128 columns
    if (a.op == kOpOut) return launch_op<kOpOut, TM, TN>(a, 1, 0, st);
    if (a.op == kOpEloc) return launch_op<kOpEloc, TM, TN>(a, 1, 0, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// Tile by the number of CTAs it gives: 128 x 128 from three CTAs per SM on
// (below, the masks' uneven K ranges and the last wave cost more than its better
// operand reuse gains: 256 tiles of the hidden GEMM above took 1103 us, 512 of 64
// x 128 987), 64 x 128 from one and a half, else 64 x 64 (tim500's hidden GEMM,
// 64 tiles: 70 -> 22 us); the ops with row partials keep 128 columns (a partial
// per 128 columns).
int gemm_simt_rows(int op, int M, int N, int sms) {
  return tiles(M, N, 128, 128) >= 3ll * sms ? 128 : 64;
}

namespace {

// 64 x 128 tiles: the choice between them and 64 x 64
bool wide_tiles(int M, int N, int sms) { return 2 * tiles(M, N, 64, 128) >= 3ll * sms; }

constexpr long long kMaxParts = 64;

}  // namespace

// The weight gradients of few tiles split K, the batch: as many parts as give four
// CTAs per SM, at most 64 and of at least 64 samples each (n = 301, h = 203, 777
// samples: 20 tiles, 10 parts).  With at most 16, 32 or 128 parts the backward pass of
// 432 models (n and h up to 1000 and 700, 129 to 16,384 samples) took 4%, 0.8% and 0.2%
// longer in the mean, up to 1.7, 1.2 and 1.1 times as long.  Sizes and the device alone
// decide, so that the same call gives the same bits in every context; the parts take
// at most 16 KB for each of the four CTAs.
int gemm_simt_parts(int M, int N, int K, int sms, int* kpart) {
  *kpart = 0;
  if (gemm_simt_rows(kOpDV, M, N, sms) == 128 || wide_tiles(M, N, sms)) return 1;
  const long long want = std::min({4ll * sms / tiles(M, N, 64, 64), (long long)K / 64, kMaxParts});
  if (want <= 1) return 1;
  *kpart = ((K + (int)want - 1) / (int)want + BK - 1) / BK * BK;
  return (K + *kpart - 1) / *kpart;
}

size_t gemm_simt_part_floats(int M, int N, int Kmax, int sms) {
  int kpart;
  if (gemm_simt_parts(M, N, Kmax, sms, &kpart) <= 1) return 0;
  // rounding the parts up to steps of K only lowers their number
  return (size_t)std::min({4ll * sms / tiles(M, N, 64, 64), (long long)Kmax / 64, kMaxParts}) * M * N;
}

cudaError_t launch_gemm_simt_f32(const GemmArgs<float>& a, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return cudaSuccess;
  const int sms = a.sms > 0 ? a.sms : 1;
  if (gemm_simt_rows(a.op, a.M, a.N, sms) == 128) return launch_tile<8, 8>(a, 1, 0, st);
  if (a.op == kOpOut || a.op == kOpEloc || wide_tiles(a.M, a.N, sms)) return launch_tile<4, 8>(a, 1, 0, st);
  int parts = 1, kpart = 0;
  if (a.op == kOpDV || a.op == kOpDW) parts = gemm_simt_parts(a.M, a.N, a.K, sms, &kpart);
  return launch_tile<4, 4>(a, parts, kpart, st);
}

}  // namespace vqmc
