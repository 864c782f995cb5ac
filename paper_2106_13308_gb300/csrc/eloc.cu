// Local energy (Sec. 2.1, Sec. 2.4), FP64 batch statistics (Eq. (e:vmc),
// Eq. (eq:stochastic_variance)) and spin-layout conversions.
//
// Sparse local energy.  For a diagonal Hamiltonian l(s) = H_ss =
// sum_{i<j} J_ij s_i s_j + sum_i h_i s_i.  The spins are first packed
// bit-transposed, 32 samples per word: Sbits[w][i] bit l = [s_i of sample
// 32w + l is -1] (one warp per 32 x 32 tile, coalesced reads).  Then one CTA
// per (word, slice of rows) loads its n words into shared memory, so one
// 32-bit xor of two words gives the sign of s_i s_j for all 32 samples, the
// warps take the slice's CSR rows in turn and lane l accumulates sample l.
// Slices hold about equal numbers of edges; their partial energies are summed
// in slice order.  Integer weights accumulate in int32 (exact).
#include "common.cuh"

namespace vqmc {
namespace {

constexpr int kElocWarps = 8;

// Sbits[w][i] for a 32-site x 32-sample tile per warp.
__global__ void __launch_bounds__(256) pack_bits_kernel(int B, int n, const int8_t* __restrict__ S,
                                                        uint32_t* __restrict__ bits) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = (blockIdx.x * 8 + warp) * 32, w = blockIdx.y;
  if (i0 >= n) return;
  const int b = 32 * w + lane;
  // lane l: bit i = [s_{i0+i} of sample b is -1]
  uint32_t m = 0;
  if (b < B) {
    const int8_t* row = S + (size_t)b * n + i0;
    const int cnt = min(32, n - i0);
    if (cnt == 32 && (reinterpret_cast<uintptr_t>(row) & 15) == 0) {
      const uint4 q0 = __ldg(reinterpret_cast<const uint4*>(row)), q1 = __ldg(reinterpret_cast<const uint4*>(row) + 1);
      const uint32_t wv[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        // sign bits of the 4 bytes of word k (spins are +-1: bit 7 set iff -1)
        const uint32_t sg = (wv[k] >> 7) & 0x01010101u;
        m |= ((sg * 0x01020408u) >> 24 & 0xFu) << (4 * k);
      }
    } else {
      for (int i = 0; i < cnt; ++i) m |= (__ldg(row + i) < 0 ? 1u : 0u) << i;
    }
  }
  uint32_t out = 0;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const uint32_t t = __ballot_sync(0xffffffffu, (m >> i) & 1u);
    if (lane == i) out = t;
  }
  if (i0 + lane < n) bits[(size_t)w * n + i0 + lane] = out;
}

// Edges of slice q are split evenly among the warps; each warp reads 32
// edges at a time (row, column, weight) with coalesced loads and broadcasts
// them with shuffles, so no load waits on another.
template <typename W, typename A>
__global__ void __launch_bounds__(kElocWarps * 32) eloc_sparse_kernel(int B, int n, const uint32_t* __restrict__ Sbits,
                                                                      const int32_t* __restrict__ row_ptr,
                                                                      const int32_t* __restrict__ erow,
                                                                      const int32_t* __restrict__ col,
                                                                      const W* __restrict__ w,
                                                                      const W* __restrict__ field,
                                                                      const int32_t* __restrict__ slice,
                                                                      A* __restrict__ part, int ldp) {
  extern __shared__ uint32_t bits[];  // [n]
  __shared__ A red[kElocWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wd = blockIdx.x, q = blockIdx.y;
  const uint32_t* src = Sbits + (size_t)wd * n;
  for (int i = threadIdx.x; i < n; i += kElocWarps * 32) bits[i] = __ldg(src + i);
  __syncthreads();
  A e = 0;
  const int r0 = __ldg(slice + q), r1 = __ldg(slice + q + 1);
  if (field)
    for (int i = r0 + warp; i < r1; i += kElocWarps) {
      const A f = (A)__ldg(field + i);
      e += ((bits[i] >> lane) & 1u) ? -f : f;
    }
  const int pa = __ldg(row_ptr + r0), pb = __ldg(row_ptr + r1);
  const int per = (pb - pa + kElocWarps - 1) / kElocWarps;
  const int p0 = pa + warp * per, p1 = min(pb, p0 + per);
  for (int pc = p0; pc < p1; pc += 32) {
    const int p = pc + lane;
    const bool in = p < p1;
    const int ei = in ? __ldg(erow + p) : 0, ej = in ? __ldg(col + p) : 0;
    const A ew = in ? (A)__ldg(w + p) : (A)0;
    const int cnt = min(32, p1 - pc);
#pragma unroll 4
    for (int k = 0; k < cnt; ++k) {
      const int i = __shfl_sync(0xffffffffu, ei, k), j = __shfl_sync(0xffffffffu, ej, k);
      const A wt = __shfl_sync(0xffffffffu, ew, k);
      const uint32_t x = bits[i] ^ bits[j];
      e += ((x >> lane) & 1u) ? -wt : wt;
    }
  }
  red[warp][lane] = e;
  __syncthreads();
  const int b = 32 * wd + lane;
  if (warp == 0 && b < B) {
    A t = red[0][lane];
#pragma unroll
    for (int k = 1; k < kElocWarps; ++k) t += red[k][lane];
    part[(size_t)q * ldp + b] = t;
  }
}

// Bit-sliced variant for small integer weights (|J_ij| < 2^(PL - 5)): the
// lanes take different edges and each handles all 32 samples of the word at
// once.  With x = bit_i xor bit_j (bit set: s_i s_j = -1), the slice's part
// of E_b is W - 2 sum_e J_e x_{e,b}, W the slice's weight sum.  A lane adds
// J_e x_e into a two's-complement counter kept as bit planes (bit b of plane
// t: bit t of sample b's partial sum; each addition a ripple of full adders
// over the planes): PL planes for runs of 15 edges (15 (2^(PL-5) - 1) <
// 2^(PL-1)), each run then sign-extended into 32 planes.  The lanes' and then
// the warps' counters are added plane-wise in a fixed order, and lane b
// finally reads sample b's integer off the planes.  The result equals the
// plain kernel's bit for bit (both are W - 2 sum J x in int32).
__device__ __forceinline__ void add_planes32(uint32_t (&C)[32], const uint32_t (&a)[32]) {
  uint32_t c = 0;
#pragma unroll
  for (int t = 0; t < 32; ++t) {
    const uint32_t s = C[t] ^ a[t] ^ c;
    c = (C[t] & a[t]) | (c & (C[t] ^ a[t]));
    C[t] = s;
  }
}

template <int PL, bool STAGE>
__global__ void __launch_bounds__(kElocWarps * 32) eloc_sliced_kernel(int B, int n, const uint32_t* __restrict__ Sbits,
                                                                     const int32_t* __restrict__ row_ptr,
                                                                     const int32_t* __restrict__ erow,
                                                                     const int32_t* __restrict__ col,
                                                                     const int32_t* __restrict__ w,
                                                                     const int32_t* __restrict__ field,
                                                                     const int32_t* __restrict__ slice,
                                                                     int32_t* __restrict__ part, int ldp) {
  // STAGE: the word's n spin words in shared memory; otherwise read through
  // L1 (no shared memory, so that the CTAs fit beside a GEMM's)
  extern __shared__ uint32_t staged[];  // [n] if STAGE
  __shared__ uint32_t planes[kElocWarps][32];
  __shared__ int32_t fpart[kElocWarps][32];
  __shared__ int32_t wpart[kElocWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wd = blockIdx.x, q = blockIdx.y;
  const uint32_t* src = Sbits + (size_t)wd * n;
  if constexpr (STAGE) {
    for (int i = threadIdx.x; i < n; i += kElocWarps * 32) staged[i] = __ldg(src + i);
    __syncthreads();
  }
  auto bit_word = [&](int i) -> uint32_t {
    if constexpr (STAGE) return staged[i];
    else return __ldg(src + i);
  };
  const int r0 = __ldg(slice + q), r1 = __ldg(slice + q + 1);
  // the field: lane = sample, as in the plain kernel
  int32_t fe = 0;
  if (field)
    for (int i = r0 + warp; i < r1; i += kElocWarps) {
      const int32_t f = __ldg(field + i);
      fe += ((bit_word(i) >> lane) & 1u) ? -f : f;
    }
  const int pa = __ldg(row_ptr + r0), pb = __ldg(row_ptr + r1);
  uint32_t C[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) C[t] = 0u;
  int32_t ws = 0;
  for (int p = pa + (int)threadIdx.x; p < pb;) {
    uint32_t L[PL];
#pragma unroll
    for (int t = 0; t < PL; ++t) L[t] = 0u;
    for (int k = 0; k < 15 && p < pb; ++k, p += kElocWarps * 32) {
      const int32_t wt = __ldg(w + p);
      const uint32_t x = bit_word(__ldg(erow + p)) ^ bit_word(__ldg(col + p));
      ws += wt;
      uint32_t c = 0;
#pragma unroll
      for (int t = 0; t < PL; ++t) {
        const uint32_t a = ((uint32_t)wt >> t) & 1u ? x : 0u;  // plane t of wt x (two's complement)
        const uint32_t sum = L[t] ^ a ^ c;
        c = (L[t] & a) | (c & (L[t] ^ a));
        L[t] = sum;
      }
    }
    uint32_t a[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) a[t] = L[t < PL ? t : PL - 1];  // sign extension
    add_planes32(C, a);
  }
  // the warp's lanes, then the CTA's warps (fixed order)
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint32_t o[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) o[t] = __shfl_xor_sync(0xffffffffu, C[t], d);
    add_planes32(C, o);
    ws += __shfl_xor_sync(0xffffffffu, ws, d);
  }
  planes[warp][lane] = C[lane];
  fpart[warp][lane] = fe;
  if (lane == 0) wpart[warp] = ws;
  __syncthreads();
  if (warp == 0) {
    uint32_t T[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) T[t] = planes[0][t];
    int32_t wsum = wpart[0], f = fpart[0][lane];
    for (int k = 1; k < kElocWarps; ++k) {
      uint32_t o[32];
#pragma unroll
      for (int t = 0; t < 32; ++t) o[t] = planes[k][t];
      add_planes32(T, o);
      wsum += wpart[k];
      f += fpart[k][lane];
    }
    uint32_t v = 0;  // sample lane's sum of J x (two's complement)
#pragma unroll
    for (int t = 0; t < 32; ++t) v |= ((T[t] >> lane) & 1u) << t;
    const int b = 32 * wd + lane;
    if (b < B) part[(size_t)q * ldp + b] = (int32_t)((uint32_t)wsum - 2u * v) + f;
  }
}

// E_b = sum of the slices' partial energies, in slice order
template <typename A>
__global__ void eloc_sum_kernel(int B, int nslices, const A* __restrict__ part, int ldp, A* __restrict__ E) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  A t = part[b];
  for (int q = 1; q < nslices; ++q) t += part[(size_t)q * ldp + b];
  E[b] = t;
}

// E_b = sum over N-tiles of the GEMM's row partials (1/2 s^T J s) + h.s, added
// in the order of the spins.  The chain of n additions bounds it, so little
// else is in it: a CTA takes 32 samples, its warps turn the spins of up to
// kFinishCols columns into sign words (a ballot per sample and 32 columns, many
// loads in flight), and one warp adds +-h_i, a sample per lane.  (One thread per
// sample reading its spins as it adds took 37 us for 1024 samples of 500 spins.)
constexpr int kFinishCols = 2048, kFinishThreads = 512;
__global__ void __launch_bounds__(kFinishThreads)
    eloc_dense_finish_kernel(int B, int n, int ntiles, const float* __restrict__ part, int ld,
                             const int8_t* __restrict__ S, const float* __restrict__ field, float* __restrict__ E) {
  __shared__ uint32_t down[32][kFinishCols / 32 + 1];  // bit q of word w: spin 32 w + q is not +1
  __shared__ __align__(16) float h[kFinishCols];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b0 = blockIdx.x * 32, b = b0 + lane;
  float e = 0.0f;
  if (warp == 0 && b < B)
    for (int t = 0; t < ntiles; ++t) e += part[(size_t)t * ld + b];
  for (int c0 = 0; field && c0 < n; c0 += kFinishCols) {
    const int cols = min(kFinishCols, n - c0), words = (cols + 31) / 32;
    for (int i = tid; i < cols; i += kFinishThreads) h[i] = field[c0 + i];
    // warp w: words of samples w and w + 16 in turn
#pragma unroll 8
    for (int q = 0; q < 2 * words; ++q) {
      const int s = warp + 16 * (q & 1), i = 32 * (q >> 1) + lane;
      const bool in = i < cols & b0 + s < B;
      const int8_t v = S[in ? (size_t)(b0 + s) * n + c0 + i : 0];
      const uint32_t m = __ballot_sync(0xffffffffu, in & v <= 0);
      if (lane == 0) down[s][q >> 1] = m;
    }
    __syncthreads();
    if (warp == 0) {
      for (int w = 0; w < words; ++w) {
        const uint32_t m = down[lane][w];
        const int cnt = min(32, cols - 32 * w);
        if (cnt == 32) {
#pragma unroll
          for (int i = 0; i < 32; ++i) e += (m >> i) & 1u ? -h[32 * w + i] : h[32 * w + i];
        } else {
          for (int i = 0; i < cnt; ++i) e += (m >> i) & 1u ? -h[32 * w + i] : h[32 * w + i];
        }
      }
    }
    __syncthreads();
  }
  if (warp == 0 && b < B) E[b] = e;
}

// FP64 statistics of B energies in one CTA with a fixed reduction order.
// With ds set, one thread also starts the next Adam step (t += 1 and its bias
// corrections), which the gradient kernels after it read.  Float energies
// (this kernel); the coefficients (E_b - mean) / B multiply by 1 / B (exact
// for B a power of two; otherwise within one rounding of the quotient before
// the conversion to FP32).  Integer energies: stats_int_kernel below.
// FP64 runs at 1/64 of the FP32 rate and bounds this kernel, so that only the
// sums are FP64: the extremes are taken in FP32 and the quotients by one thread
// (computed by every thread, with FP64 extremes, 1024 energies took 19 us and 8192
// took 41; now 10 and 24).
__global__ void __launch_bounds__(1024) stats_kernel(int B, const float* __restrict__ E, double* __restrict__ out,
                                                     float* __restrict__ coef, uint32_t* __restrict__ err,
                                                     DevState* ds, float beta1, float beta2) {
  __shared__ double ws[32], quot[2];
  __shared__ float wmn[32], wmx[32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // sum over the CTA (thread 0 holds it), in a fixed order
  auto cta_sum = [&](double x) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    if (lane == 0) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
      x = ws[lane];
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    }
    return x;
  };
  double sum = 0.0;
  float mn = __int_as_float(0x7f800000), mx = -mn;
  for (int b = t; b < B; b += 1024) {
    const float x = E[b];
    sum += (double)x;
    mn = x < mn ? x : mn;
    mx = x > mx ? x : mx;
  }
  auto extremes = [&] {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const float a = __shfl_down_sync(0xffffffffu, mn, d), b = __shfl_down_sync(0xffffffffu, mx, d);
      mn = a < mn ? a : mn;
      mx = b > mx ? b : mx;
    }
  };
  extremes();
  if (lane == 0) wmn[warp] = mn, wmx[warp] = mx;
  sum = cta_sum(sum);
  if (t == 0) quot[0] = sum / (double)B, quot[1] = 1.0 / (double)B;
  if (warp == 0) {
    mn = wmn[lane], mx = wmx[lane];
    extremes();
  }
  __syncthreads();
  const double mean = quot[0], inv = quot[1];
  double ss = 0.0;
  for (int b = t; b < B; b += 1024) {
    const double d = (double)E[b] - mean;
    ss += d * d;
    if (coef) coef[b] = (float)(d * inv);
  }
  ss = cta_sum(ss);
  if (ds && t == 1023) {  // beside thread 0's quotients
    ds->adam_t += 1;
    adam_factors(ds, beta1, beta2);
  }
  if (t == 0) {
    const double var = ss / (double)B;
    out[0] = mean;
    out[1] = var;
    out[2] = (double)mn;
    out[3] = (double)mx;
    if (!isfinite(mean) || !isfinite(var)) atomicOr(err, kErrNonfinite);
  }
}

// Integer energies: the same statistics with integer arithmetic only
// (FP64 is slow on this part).  mean = S / B from S = sum E (int64); the
// variance (B Q - S^2) / B^2 from Q = sum E^2 (128-bit integers: exact before
// its one rounding); the coefficients (B E_b - S) / B^2 as an FP32 product,
// equal to the FP64 path's (E_b - mean) / B rounded to FP32 when B is a power
// of two (otherwise within about one rounding of it).
__global__ void __launch_bounds__(1024) stats_int_kernel(int B, const int32_t* __restrict__ E, double* __restrict__ out,
                                                         float* __restrict__ coef, uint32_t* __restrict__ err,
                                                         DevState* ds, float beta1, float beta2) {
  __shared__ long long ws[32];
  __shared__ unsigned long long wql[32];
  __shared__ long long wqh[32];
  __shared__ int32_t wmn[32], wmx[32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = (int)(blockDim.x >> 5);
  if (ds && t == 0) {
    ds->adam_t += 1;
    adam_factors(ds, beta1, beta2);
  }
  long long sum = 0;
  __int128 sq = 0;
  int32_t mn = 0x7fffffff, mx = -0x7fffffff - 1;
  for (int b = t; b < B; b += blockDim.x) {
    const long long x = E[b];
    sum += x;
    sq += (__int128)(x * x);
    mn = (int32_t)x < mn ? (int32_t)x : mn;
    mx = (int32_t)x > mx ? (int32_t)x : mx;
  }
  auto reduce_warp = [&]() {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      sum += __shfl_down_sync(0xffffffffu, sum, d);
      const unsigned long long lo = (unsigned long long)sq, olo = __shfl_down_sync(0xffffffffu, lo, d);
      const long long hi = (long long)(sq >> 64), ohi = __shfl_down_sync(0xffffffffu, hi, d);
      sq += (__int128)(((unsigned __int128)(unsigned long long)ohi << 64) | olo);
      const int32_t a = __shfl_down_sync(0xffffffffu, mn, d), c = __shfl_down_sync(0xffffffffu, mx, d);
      mn = a < mn ? a : mn;
      mx = c > mx ? c : mx;
    }
  };
  reduce_warp();
  if (lane == 0) ws[warp] = sum, wql[warp] = (unsigned long long)sq, wqh[warp] = (long long)(sq >> 64),
                 wmn[warp] = mn, wmx[warp] = mx;
  __syncthreads();
  if (warp == 0) {
    sum = lane < nw ? ws[lane] : 0;
    sq = lane < nw ? (__int128)(((unsigned __int128)(unsigned long long)wqh[lane] << 64) | wql[lane]) : 0;
    mn = lane < nw ? wmn[lane] : 0x7fffffff;
    mx = lane < nw ? wmx[lane] : -0x7fffffff - 1;
    reduce_warp();
    if (lane == 0) ws[0] = sum, wql[0] = (unsigned long long)sq, wqh[0] = (long long)(sq >> 64), wmn[0] = mn, wmx[0] = mx;
  }
  __syncthreads();
  const long long S = ws[0];
  const double mean = (double)S / (double)B;
  if (t == 0) {
    const __int128 Q = (__int128)(((unsigned __int128)(unsigned long long)wqh[0] << 64) | wql[0]);
    const __int128 num = (__int128)B * Q - (__int128)S * (__int128)S;  // B^2 var >= 0
    const double var = (double)num / ((double)B * (double)B);
    out[0] = mean;
    out[1] = var;
    out[2] = (double)wmn[0];
    out[3] = (double)wmx[0];
    if (!isfinite(mean) || !isfinite(var)) atomicOr(err, kErrNonfinite);
  }
  if (coef) {
    const float inv2 = (float)(1.0 / ((double)B * (double)B));
    for (int b = t; b < B; b += blockDim.x) coef[b] = (float)((long long)B * E[b] - S) * inv2;
  }
}

template <typename T>
__device__ __forceinline__ T spin_val(int8_t s);
template <>
__device__ __forceinline__ float spin_val<float>(int8_t s) { return s > 0 ? 1.0f : -1.0f; }
template <>
__device__ __forceinline__ bf16 spin_val<bf16>(int8_t s) { return __float2bfloat16_rn(s > 0 ? 1.0f : -1.0f); }

// the first cnt of 16 spins as T in 16-byte stores, zeros after the last: rows are
// padded to multiples of 64 and start on 16-byte boundaries
template <bool ALL, typename T>
__device__ __forceinline__ void store_spins16(T* p, const uint32_t (&w)[4], int cnt) {
  constexpr int kPer = 16 / sizeof(T);
#pragma unroll
  for (int v = 0; v < 16 / kPer; ++v) {
    if (!ALL && kPer * v >= cnt) break;
    __align__(16) T x[kPer];
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int q = kPer * v + e;
      x[e] = ALL || q < cnt ? spin_val<T>((int8_t)(w[q >> 2] >> (8 * (q & 3)))) : T(0.0f);
    }
    reinterpret_cast<uint4*>(p)[v] = *reinterpret_cast<const uint4*>(x);
  }
}
template <typename T>
__device__ __forceinline__ void store_spins(T* p, const uint32_t (&w)[4], int cnt) {
  if (cnt >= 16) store_spins16<true>(p, w, cnt);
  else store_spins16<false>(p, w, cnt);
}

// int8 [B][n] -> T [B][ldx] and T [n][ldt] (transposed through a 64 x 64 tile).
// Bound by its writes; a thread moves 16 spins with 16-byte accesses (one spin
// and 2-byte stores per thread took 13 us for 4096 x 1000 in BF16, this 9).  Rows
// that don't start on such a boundary are cut from aligned words, and every piece
// is stored whole (with single bytes for these and for the last piece of a row 8192 x
// 301 spins took 8.1 us, so 3.8).
constexpr int kCvt = 64, kCvtLd = kCvt + 4;
template <typename T>
__global__ void __launch_bounds__(256) spins_convert_kernel(int B, int n, const int8_t* __restrict__ S,
                                                            T* __restrict__ Sx, int ldx, T* __restrict__ St, int ldt) {
  __shared__ __align__(16) int8_t tile[kCvt][kCvtLd];  // [sample][spin]
  const int i0 = blockIdx.x * kCvt, b0 = blockIdx.y * kCvt;
  const int r = threadIdx.x >> 2, c = 16 * (threadIdx.x & 3);
  uint32_t w[4] = {0, 0, 0, 0};
  if (b0 + r < B && i0 + c < n) {
    const int8_t* src = S + (size_t)(b0 + r) * n + i0 + c;
    const int cnt = min(16, n - i0 - c);
    const uintptr_t at = reinterpret_cast<uintptr_t>(src), word = at & ~(uintptr_t)3;
    const uintptr_t first = reinterpret_cast<uintptr_t>(S), end = first + (size_t)B * n;
    if ((at & 15) == 0 && at + 16 <= end) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(src));
      w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
    } else if (word >= first && word + 20 <= end) {  // the five words lie inside the array
      uint32_t x[5];
#pragma unroll
      for (int q = 0; q < 5; ++q) x[q] = __ldg(reinterpret_cast<const uint32_t*>(word) + q);
#pragma unroll
      for (int q = 0; q < 4; ++q) w[q] = __funnelshift_r(x[q], x[q + 1], 8 * (int)(at & 3));
    } else {
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (q < cnt) w[q >> 2] |= (uint32_t)(uint8_t)src[q] << (8 * (q & 3));
    }
    if (Sx) store_spins(Sx + (size_t)(b0 + r) * ldx + i0 + c, w, cnt);
  }
  if (!St) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) *reinterpret_cast<uint32_t*>(&tile[r][c + 4 * q]) = w[q];
  __syncthreads();
  // spin r of the tile, samples c .. c + 15
  if (i0 + r < n && b0 + c < B) {
    uint32_t x[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 16; ++q) x[q >> 2] |= (uint32_t)(uint8_t)tile[c + q][r] << (8 * (q & 3));
    store_spins(St + (size_t)(i0 + r) * ldt + b0 + c, x, min(16, B - b0 - c));
  }
}

__global__ void tile_sum_kernel(int cnt, int ntiles, const float* __restrict__ part, int ld, float* __restrict__ out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= cnt) return;
  float s = 0.0f;
  for (int t = 0; t < ntiles; ++t) s += part[(size_t)t * ld + q];
  out[q] = s;
}

}  // namespace

template <int PL>
cudaError_t eloc_sliced(const vqmc_ctx* c, int B, void* d_e, cudaStream_t st, bool stage) {
  const size_t smem = stage ? (size_t)c->n * sizeof(uint32_t) : 0;
  auto k = stage ? eloc_sliced_kernel<PL, true> : eloc_sliced_kernel<PL, false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int ns = c->eloc_slices;
  int32_t* part = ns > 1 ? (int32_t*)c->eloc_part : (int32_t*)d_e;
  k<<<dim3((B + 31) / 32, ns), kElocWarps * 32, smem, st>>>(B, c->n, c->Sbits, c->row_ptr, c->erow, c->col,
                                                           (const int32_t*)c->w, (const int32_t*)c->field,
                                                           c->eloc_slice, part, c->Bmax);
  if (ns > 1) eloc_sum_kernel<int32_t><<<(B + 255) / 256, 256, 0, st>>>(B, ns, part, c->Bmax, (int32_t*)d_e);
  return cudaGetLastError();
}

template <typename W, typename A>
cudaError_t eloc_sparse(const vqmc_ctx* c, int B, void* d_e, cudaStream_t st) {
  const size_t smem = (size_t)c->n * sizeof(uint32_t);
  auto k = eloc_sparse_kernel<W, A>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int ns = c->eloc_slices;
  A* part = ns > 1 ? (A*)c->eloc_part : (A*)d_e;
  k<<<dim3((B + 31) / 32, ns), kElocWarps * 32, smem, st>>>(B, c->n, c->Sbits, c->row_ptr, c->erow, c->col,
                                                           (const W*)c->w, (const W*)c->field, c->eloc_slice, part,
                                                           c->Bmax);
  if (ns > 1) eloc_sum_kernel<A><<<(B + 255) / 256, 256, 0, st>>>(B, ns, part, c->Bmax, (A*)d_e);
  return cudaGetLastError();
}

cudaError_t launch_eloc_sparse(const vqmc_ctx* c, int B, const int8_t* d_s, void* d_e, cudaStream_t st,
                               bool packed, bool beside) {
  if (B <= 0) return cudaSuccess;
  if (!packed) pack_bits_kernel<<<dim3((c->n + 255) / 256, (B + 31) / 32), 256, 0, st>>>(B, c->n, d_s, c->Sbits);
  if (c->ham == VQMC_HAM_SPARSE_I32) {
    // weights of at most 8 bits (magnitude): the bit-sliced kernel
    // beside: the launch shares the GPU with a GEMM, so the spin words are
    // read through L1 instead of taking shared memory
    if (c->eloc_wbits <= 1) return eloc_sliced<6>(c, B, d_e, st, !beside);
    if (c->eloc_wbits <= 4) return eloc_sliced<9>(c, B, d_e, st, !beside);
    if (c->eloc_wbits <= 8) return eloc_sliced<13>(c, B, d_e, st, !beside);
    return eloc_sparse<int32_t, int32_t>(c, B, d_e, st);
  }
  return eloc_sparse<float, float>(c, B, d_e, st);
}

cudaError_t launch_eloc_dense_finish(const vqmc_ctx* c, int B, const int8_t* d_s, void* d_e, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  const int ntiles = (c->n + 127) / 128;
  eloc_dense_finish_kernel<<<(B + 31) / 32, kFinishThreads, 0, st>>>(B, c->n, ntiles, c->row_part, c->row_part_ld, d_s,
                                                            (const float*)c->field, (float*)d_e);
  return cudaGetLastError();
}

cudaError_t launch_stats(const vqmc_ctx* c, int B, const void* d_e, double* d_stats, float* d_coef,
                         cudaStream_t st, bool advance) {
  if (B <= 0) return cudaSuccess;
  DevState* ds = advance ? c->dstate : nullptr;
  const float b1 = c->cfg.beta1, b2 = c->cfg.beta2;
  if (c->ham == VQMC_HAM_SPARSE_I32)
    stats_int_kernel<<<1, 1024, 0, st>>>(B, (const int32_t*)d_e, d_stats, d_coef, c->err, ds, b1, b2);
  else
    stats_kernel<<<1, 1024, 0, st>>>(B, (const float*)d_e, d_stats, d_coef, c->err, ds, b1, b2);
  return cudaGetLastError();
}

cudaError_t launch_spins_to_operands(const vqmc_ctx* c, int B, const int8_t* d_s, void* Sx, void* St,
                                     cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  dim3 grid((c->n + kCvt - 1) / kCvt, (B + kCvt - 1) / kCvt);
  if (c->prec == VQMC_PREC_BF16)
    spins_convert_kernel<bf16><<<grid, 256, 0, st>>>(B, c->n, d_s, (bf16*)Sx, c->np, (bf16*)St, c->Bp);
  else
    spins_convert_kernel<float><<<grid, 256, 0, st>>>(B, c->n, d_s, (float*)Sx, c->np, (float*)St, c->Bp);
  return cudaGetLastError();
}

cudaError_t launch_row_sum(const vqmc_ctx* c, int B, int ntiles, float* out, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  tile_sum_kernel<<<(B + 255) / 256, 256, 0, st>>>(B, ntiles, c->row_part, c->row_part_ld, out);
  return cudaGetLastError();
}

cudaError_t launch_col_sum(const vqmc_ctx* c, int N, int mtiles, float* out, cudaStream_t st) {
  if (N <= 0) return cudaSuccess;
  tile_sum_kernel<<<(N + 255) / 256, 256, 0, st>>>(N, mtiles, c->col_part, c->col_part_ld, out);
  return cudaGetLastError();
}

}  // namespace vqmc
