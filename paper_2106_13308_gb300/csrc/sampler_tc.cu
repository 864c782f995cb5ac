// Blocked autoregressive sampler on the tcgen05 tensor cores, for the BF16
// model (BF16 weights, hidden activations rounded to BF16, FP32 accumulation).
//
// Algorithm 1 draws s_1 .. s_n in order; with the incremental forward pass
// (Sec. 2.3) the logit of step i is
//     z_i = b2_i + sum_{k : m(k) < i} W2_ik g1_k,
//     g1_k = act(b1_k + sum_{j <= m(k)} W1_kj s_j),
// and with sorted degrees a hidden unit is complete once s_{m(k)} is drawn.
// This kernel processes the n steps in blocks of D (64 or 128).  For block
// [i0, i0 + D):
//   * units complete before the block (m(k) < i0, a prefix of the units)
//     feed every output of the block through one tensor-core GEMM,
//         Z[i][s] = sum_k W2[i][k] g1[k][s]     (M = 128 outputs, N = 16
//     samples, K = that prefix), with g1 kept in shared memory in BF16;
//   * the few units completing inside the block (m(k) in [i0, i0 + D), at
//     most 32: the "recent" units) are carried by a small sequential solver
//     that draws the D spins: z_i = Z[i] + b2_i + sum_recent W2_ik g1_k, with
//     each recent pre-activation extended by W1_ki s_i after every draw;
//   * the block's spins then update every unit still incomplete by a second
//     tensor-core GEMM, A[k][s] += sum_j W1[k][j] s_j over the block's inputs
//     (M = 128 units, N = 16, K = D), into FP32 accumulators that stay in
//     tensor memory for the whole run (16 columns per 128 units).
// The masks need no special handling: masked weights are stored as zeros, so
// an update adds nothing to a complete unit and an incomplete unit (g1 = 0
// in shared memory until it completes) adds nothing to any logit.
//
// CTA = 16 samples, 10 warps: warps 0-3 own TMEM lanes 32w..32w+31 (read Z
// and the recent pre-activations); warps 0, 1, 6 and 7 are the solver (8
// lanes per sample, each lane owning every 8th step of a segment and partial
// sums of all the block's recent units) and then write the block's spins as
// the update GEMM's operand; while they solve, warps 2, 3, 8 and 9 (the
// helpers) merge the previous
// block's recent g1 into the Z operand, prepare the next block's schedule,
// logits and recent-unit weights, write out the previous block's spins and add
// up its log pi; one thread of warp 4 streams 128 x 64 BF16 weight tiles with
// TMA into a ring of six tiles, consumed in two slots of three; one of warp 5
// issues the MMAs.  Every wait is bounded; after a failed wait the CTA raises
// the timeout bit and runs on without waiting, so it still finishes.
//
// What bounds it: the chain of the solver's segments, about 550 cycles each,
// then the helpers (models of few units per block), and some 3,300 cycles from one
// block's last draw to the next one's first.  Measured (GB300, n = 10000, h =
// 2000, 1024 samples with log pi): 1264 -> 726 us; n = 500, h = 193: 138 -> 85
// us; n = 10000, h = 424: 804 -> 505 us.  What that took, the arithmetic unchanged:
// warp-uniform values for the warp index and the segment bounds and one elected
// thread per issuing warp; one copy of each piece of code; predicated stores in
// place of branches; log pi and the next block's schedule moved to the helpers.
#include <algorithm>
#include <type_traits>

#include "gemm.cuh"
#include "f32x2.cuh"
#include "sampler.cuh"
#include "tc_ptx.cuh"

namespace vqmc {
namespace {

using namespace tc;

constexpr int kS = 16;                     // samples per CTA (MMA N)
constexpr int kRmax = 32;                  // recent units per block
constexpr int kNStage = 6;                 // weight tiles in the ring
constexpr int kTileBytes = 128 * 64 * 2;   // one 128 x 64 BF16 tile
// The ring is consumed in slots of up to three tiles (48 KB): one
// full-barrier wait and one commit per slot.  A slot's tiles that are
// consecutive 64-column chunks of the same rows arrive in one copy: the copy
// engine's time goes by copies more than by bytes (a 32 KB box streams about
// twice as fast as two 16 KB boxes).
constexpr int kSlotTiles = 3;
constexpr int kNSlot = kNStage / kSlotTiles;
constexpr int kMaxHp = 2048;               // hidden units (padded) in TMEM
constexpr int kDmax = 128;
constexpr int kTmemCols = 512;             // A: 16 per 128 units (<= 256), Z at 256
constexpr int kZCol = 256;
constexpr int kThreads = 320;
// The solver: kLanes lanes per sample on warps 0, 1, 6 and 7 (one warp on
// each SM sub-partition).
constexpr int kLanes = 8;
constexpr int kSolverThreads = kS * kLanes;
// The helpers: warps 2, 3, 8 and 9, also one on each sub-partition (two on the
// sub-partitions of warps 6 and 7 slowed those: 14,300 against 12,000 cycles a
// block for the solver without them, and with few units per block the helpers'
// work was the longer one: n = 10000, h = 424 599 -> 505 us with four).
constexpr int kHelpers = 128;
// named barriers: 1 = helpers and solver, 2 = helpers (arrive) with the solver
// (sync)
constexpr int kBar1Threads = kHelpers + kSolverThreads;
constexpr int kBar2Threads = kHelpers + kSolverThreads;
constexpr int kZld = kS + 1;               // padded row of the Z buffer
constexpr uint32_t kIdesc = idesc_bf16(128, kS);

// shared memory map (offsets from a 1024-byte aligned base)
constexpr int kOffRing = 0;
constexpr int kOffH = kOffRing + kNStage * kTileBytes;         // g1, [hp/64] x (16 x 64) swizzled
constexpr int kOffS = kOffH + (kMaxHp / 64) * 2048;            // spins, [2][D/64] x (16 x 64) swizzled
// Per-step tables of the solver have kDrows = D + 4 rows (the rows past the
// block are zero) so that it reads up to 3 steps ahead without clamping.  In
// the recent-unit tables column kRmax is zero and stands for "no unit".
constexpr int kDrows = kDmax + 4;
constexpr int kLdW = kRmax + 8;                                // bf16 row of the recent-unit weight tables
constexpr int kLdP = kRmax + 4;                                // float row of the per-sample unit tables
constexpr int kOffHr = kOffS + 2 * (kDmax / 64) * 2048;        // g1 of the last block's recent units, 2 x (16 x 64)
constexpr int kOffZ = kOffHr + 2 * 2048;                       // Z + b2 [kDrows][kZld] float
constexpr int kOffLG = kOffZ + kDrows * kZld * 4;              // logit(u) [2][kDrows][16] float
constexpr int kOffP = kOffLG + 2 * kDrows * kS * 4;            // recent pre-activations at block start [32][16]
constexpr int kOffWr = kOffP + kRmax * kS * 4;                 // W1 of recent units [kDrows][kLdW] bf16
constexpr int kOffVr = kOffWr + kDrows * kLdW * 2;             // W2 of recent units [kDrows][kLdW] bf16
constexpr int kOffPS = kOffVr + kDrows * kLdW * 2;             // solver: g1 of the recent units [16][kLdP]
constexpr int kOffSB = kOffPS + kS * kLdP * 4;                 // drawn spins, bit e%32 of word [2][16][e/32]
constexpr int kBlkInts = kRmax + 4;                            // completion step of each recent unit, then klo, R, zvalid
constexpr int kOffCU = kOffSB + 2 * kS * (kDmax / 32) * 4;     // [2][kBlkInts] int
constexpr int kOffBar = kOffCU + 2 * kBlkInts * 4;              // mbarriers + slots
constexpr int kSmemBytes = 1024 + kOffBar + 128;
static_assert(kSmemBytes <= 232448, "shared memory budget");

struct TcArgs {
  int n, h, hp, B, D;
  const bf16* w;      // w_s [h][np]: row k = W1[k] (column j-1 = input j)
  int np;
  const bf16* v;      // v_s  [rows][hp]: row r = W2[r] (output r + 1)
  const float* b1;
  const float* b2;
  const float* u;     // [B][n] or null (internal Philox)
  uint32_t key0, key1, it0, it1;
  uint32_t boff;      // index of sample 0 in the Philox counter (a shard's first global sample)
  const unsigned long long* it_dev;  // if not null: the Philox iteration, read on the device
  int8_t* s_out;      // [B][n]
  float* logp;        // [B] or null
  uint32_t* err;
  // optional copies of the spins for the rest of the step (null when absent):
  // GEMM operands Sx [B][ldsx] and St [n][ldst] (BF16 +-1) and the packed
  // layout of the sparse energy, bit l of 32-bit word [w][i] = [s_i of
  // sample 32 w + l is -1], written as 16-bit halves
  bf16* sx;
  int ldsx;
  bf16* stt;
  int ldst;
  uint16_t* sbits;
};

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
// the two BF16 weights of a word, widened (exactly) to an FP32 pair
__device__ __forceinline__ uint64_t bf2(uint32_t w) { return pack2(bf_lo(w), bf_hi(w)); }

// *p = x where ok holds, as a predicated store (a branch around one costs the
// warp some 70 cycles)
__device__ __forceinline__ void store_if(bool ok, float* p, float x) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %0, 0;\n\t@p st.shared.f32 [%1], %2;\n\t}" ::"r"((int)ok),
               "r"(smem_u32(p)), "f"(x)
               : "memory");
}
__device__ __forceinline__ void store_if(bool ok, void* p, bf16 x) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %0, 0;\n\t@p st.shared.b16 [%1], %2;\n\t}" ::"r"((int)ok),
               "r"(smem_u32(p)), "h"(__bfloat16_as_ushort(x))
               : "memory");
}

template <int ACT>
__device__ __forceinline__ float g1f(float a) {
  if constexpr (ACT == VQMC_ACT_RELU) return fmaxf(a, 0.0f);
  else return 1.0f / (1.0f + expf(-a));
}

// The sequential part of a block: the draws of its D steps, carried for
// sample s by solver threads 8s .. 8s+7 (kLanes lanes of one warp of the
// solver warps 0, 1, 6 and 7).  With sorted degrees at most
// one hidden unit completes per step (h < n), and the logit of step e
// depends on the earlier spins only through the units completed before e:
//     z_e = (Z_e + b2) + sum_{recent r: t_r < e} W2_{e,r} g1_r,
// t_r the step whose spin is recent unit r's last input.  So the steps
// between two completions, (t_{r-1}, t_r], are conditionally independent
// given g1_0 .. g1_{r-1}: they form one segment, drawn in parallel.  Lane q
// of the sample's kLanes draws the steps e = q (mod kLanes) and keeps, for
// all 32 recent units, its own partial pre-activation sum over the spins it
// drew (lane 0 also holds the value at the start of the block).  When
// segment r ends, unit r's partials are added with log2(kLanes) shuffles,
// and g1_r = bf16(act(a_r)) enters
// the logits of the later segments.  The chain from one completion to the
// next is: the shuffle reduction, the activation and the rounding, one FMA
// with W2_{e,r} (the rest of the lane's next logit is summed before the
// reduction), the compare, and the lane's partial sum of unit r+1.  W2_{e,r}
// is zero for units not complete before step e and W1 for inputs after a
// unit's last one, so no masks are applied; g1 is zero (HH) until a unit
// completes.  HH holds each sample's recent g1 in shared memory (written by
// all the sample's lanes with the same value).
template <int ACT, bool LP>
__device__ __forceinline__ void solve(const float* Pr, const bf16* Vr, const bf16* Wr, const float* Zs,
                                      float* LG, const int* TC, uint32_t* SB, float* HH, unsigned char* Hr,
                                      int s_me, int q, int klo, int R, int steps) {
  float* hh = HH + s_me * kLdP;
  float P[kRmax];
#pragma unroll
  for (int k = 0; k < kRmax; ++k) P[k] = q == 0 ? Pr[k * kS + s_me] : 0.0f;
  static_assert(kLanes == 8 && kRmax == 32, "hh is zeroed as one float4 per lane");
  reinterpret_cast<float4*>(hh)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncwarp();
  uint32_t bits = 0;  // this lane's drawn spins: bit i for step 8 i + q
  // The segments run in four phases by r / 8 (a template parameter PH of the
  // helpers below): in segment r only units 0 .. r-1 are complete (g1 != 0
  // in hh) and only units r .. 31 still need partial sums, so the logit's dot
  // product reads the 8-unit chunks 0 .. PH, the weight-row update writes the
  // chunks PH .. 3 and the completing unit's partial sum is one of 16 (8 in
  // the last phase).  The
  // skipped terms are zeros (g1 of incomplete units) or sums never read
  // again, so the draws are those of the full loops.
  // Z_e + b2 + the terms of the recent units completed so far (hh, chunks 0 .. PH)
  auto zdot = [&](auto ph, int e) -> float {
    constexpr int PH = decltype(ph)::value;
    const uint4* vr = reinterpret_cast<const uint4*>(Vr + e * kLdW);
    const float4* hv = reinterpret_cast<const float4*>(hh);
    // four FP32 accumulators a0..a3 as the pairs (a0, a1), (a2, a3)
    uint64_t a01 = pack2(Zs[e * kZld + s_me], 0.0f), a23 = pack2(0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c <= PH; ++c) {
      const uint4 v = vr[c];
      const float4 x = hv[2 * c], y = hv[2 * c + 1];
      a01 = fma2(bf2(v.x), pack2(x.x, x.y), a01);
      a23 = fma2(bf2(v.y), pack2(x.z, x.w), a23);
      a01 = fma2(bf2(v.z), pack2(y.x, y.y), a01);
      a23 = fma2(bf2(v.w), pack2(y.z, y.w), a23);
    }
    float a0, a1, a2, a3;
    unpack2(a01, a0, a1);
    unpack2(a23, a2, a3);
    return (a0 + a1) + (a2 + a3);
  };
  // this lane's partial sums of the recent units of chunks PH .. 3 += sv * W1 of step row el
  auto wrow = [&](auto ph, int el, float sv) {
    constexpr int PH = decltype(ph)::value;
    const uint4* wr = reinterpret_cast<const uint4*>(Wr + el * kLdW);
    const uint64_t s2 = pack2(sv, sv);
#pragma unroll
    for (int c = PH; c < 4; ++c) {
      const uint4 w = wr[c];
      const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint64_t pp = pack2(P[8 * c + 2 * j], P[8 * c + 2 * j + 1]);
        pp = fma2(bf2(ww[j]), s2, pp);
        unpack2(pp, P[8 * c + 2 * j], P[8 * c + 2 * j + 1]);
      }
    }
  };
  // draw of step e from its logit, and the spin into this lane's partial sums
  auto draw = [&](auto ph, int e, float z) {
    const bool up = z > LG[e * kS + s_me];  // u < sigma(z)
    bits |= (uint32_t)up << (e / kLanes);
    if constexpr (LP) LG[e * kS + s_me] = up ? z : -z;
    wrow(ph, e, up ? 1.0f : -1.0f);
  };
  // the partial sum of unit k among this lane's units 8 PH .. 8 PH + 15
  // (8 PH .. 31 in the last phase): a binary select by k - 8 PH
  auto extract = [&](auto ph, int k) -> float {
    constexpr int PH = decltype(ph)::value;
    constexpr int kB = 8 * PH, kN = PH < 3 ? 16 : 8;
    const int i = k - kB;
    float l1[kN / 2], l2[kN / 4], l3[kN / 8];
#pragma unroll
    for (int t = 0; t < kN / 2; ++t) l1[t] = (i & 1) ? P[kB + 2 * t + 1] : P[kB + 2 * t];
#pragma unroll
    for (int t = 0; t < kN / 4; ++t) l2[t] = (i & 2) ? l1[2 * t + 1] : l1[2 * t];
#pragma unroll
    for (int t = 0; t < kN / 8; ++t) l3[t] = (i & 4) ? l2[2 * t + 1] : l2[2 * t];
    if constexpr (kN == 16) return (i & 8) ? l3[1] : l3[0];
    else return l3[0];
  };
  auto wt = [&](int e, int r) { return r < kRmax ? __bfloat162float(Wr[e * kLdW + r]) : 0.0f; };
  auto vt = [&](int e, int r) { return r >= 0 ? __bfloat162float(Vr[e * kLdW + r]) : 0.0f; };
  auto allsum = [&](float x) {
#pragma unroll
    for (int d = 1; d < kLanes; d <<= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    return x;
  };
  // Prepared for this lane's step e of the current segment r (when the
  // segment has at most kLanes steps, a lane has at most one): its logit
  // without the unit completed last (zp), that unit's weight on it (vn),
  // logit(u) (lgn), unit r's weight on its spin (wn) and the lane's partial
  // sum of unit r over the earlier segments (xr).  Everything else of a
  // segment runs beside the chain of the completions.
  // The segment body below is free of lane-dependent branches: a lane
  // without a step in the segment (e past its end) draws nothing (sv = 0)
  // and reads row min(e, kDrows - 1) of the tables, so that the compiler can
  // move the next segment's loads ahead of the completion chain.
  using Ph0 = std::integral_constant<int, 0>;
  float g_last = 0.0f;  // g1 of the unit that completed last
  int lo = 0;
  int e = q;
  int hi = R > 0 ? uniform(TC[0]) : steps - 1;  // last step of the current segment
  float zp = 0.0f, vn = 0.0f, lgn = 0.0f, wn = 0.0f, xr = 0.0f;
  if (e <= hi) zp = zdot(Ph0{}, e), lgn = LG[e * kS + s_me], wn = wt(e, 0);
  xr = extract(Ph0{}, 0);
  // segment r: steps [lo, hi], units 0 .. r-1 complete; true after the last (r = R)
  auto segment = [&](auto ph, int r) -> bool {
    const int nhi = r + 1 < R ? uniform(TC[r + 1]) : steps - 1;  // last step of segment r + 1
    hh[r > 0 ? r - 1 : 0] = g_last;                     // (unit 0's entry is still zero at r = 0)
    float x;
    if (hi - lo + 1 <= kLanes) {
      // ---- at most one step per lane: the chain, then the rest
      const bool own = e <= hi;
      const int el = min(e, kDrows - 1);
      const float z = fmaf(vn, g_last, zp);
      const bool up = z > lgn;
      const float sv = own ? (up ? 1.0f : -1.0f) : 0.0f;
      x = allsum(fmaf(wn, sv, xr));
      bits |= (uint32_t)(own && up) << ((uint32_t)e / kLanes);
      if constexpr (LP) store_if(own, LG + el * kS + s_me, up ? z : -z);
      wrow(ph, el, sv);
    } else {
      // ---- a long segment: every step of the lane with its full logit,
      // then unit r's partial sums
#pragma unroll 1
      for (int ee = lo + ((q - lo) & (kLanes - 1)); ee <= hi; ee += kLanes) draw(ph, ee, zdot(ph, ee));
      x = allsum(extract(ph, r < kRmax ? r : kRmax - 1));
    }
    if (r == R) return true;
    // prepare this lane's step of segment r + 1 (hh holds units 0 .. r-1);
    // a lane without one (e > nhi) keeps values that its sv = 0 ignores
    const int nlo = hi + 1;
    e = nlo + ((q - nlo) & (kLanes - 1));
    {
      const int el = min(e, kDrows - 1);
      zp = zdot(ph, el);
      vn = vt(el, r);
      lgn = LG[el * kS + s_me];
      wn = wt(el, r + 1);
    }
    xr = extract(ph, r + 1 < kRmax ? r + 1 : kRmax - 1);
    g_last = bf16r(g1f<ACT>(x));
    lo = nlo;
    hi = nhi;
    return false;
  };
  bool last = false;
  int r = 0;
#pragma unroll 1
  for (; r < 8 && !last; ++r) last = segment(Ph0{}, r);
#pragma unroll 1
  for (; r < 16 && !last; ++r) last = segment(std::integral_constant<int, 1>{}, r);
#pragma unroll 1
  for (; r < 24 && !last; ++r) last = segment(std::integral_constant<int, 2>{}, r);
#pragma unroll 1
  for (; !last; ++r) last = segment(std::integral_constant<int, 3>{}, r);  // r <= R <= 32
  // the sample's spins: step e is bit e % 32 of word e / 32 = bit 8 (i % 4) + q
  // of word i / 4, i = e / 8.  The lanes' bits are combined with shuffles;
  // lane q < 4 stores word q.
  static_assert(kLanes == 8 && kDmax == 128, "four words of four groups of 8 steps");
  uint32_t wd[kDmax / 32];
#pragma unroll
  for (int t = 0; t < kDmax / 32; ++t) {
    const uint32_t x = bits >> (4 * t);
    wd[t] = ((x & 1u) | (x & 2u) << 7 | (x & 4u) << 14 | (x & 8u) << 21) << q;
#pragma unroll
    for (int d = 1; d < kLanes; d <<= 1) wd[t] |= __shfl_xor_sync(0xffffffffu, wd[t], d);
  }
  if (q < kDmax / 32) SB[s_me * (kDmax / 32) + q] = q == 0 ? wd[0] : q == 1 ? wd[1] : q == 2 ? wd[2] : wd[3];
  // every recent unit is complete: its g1 goes to the staging operand Hr
  // (2 chunks of 64 units from chunk klo / 64), once the helpers have moved
  // the previous block's recent g1 out of it
  asm volatile("bar.sync 2, %0;" ::"n"(kBar2Threads) : "memory");
#pragma unroll
  for (int j = 0; j < kRmax / kLanes; ++j) {
    const int r = q + kLanes * j;
    const int k = klo + r;
    store_if(r < R, Hr + ((k >> 6) - (klo >> 6)) * 2048 + sw128_offset(s_me, k & 63), __float2bfloat16_rn(hh[r]));
  }
}

// The schedule of block b, computed alike by the producer, the MMA issuer
// and the compute warps.  Recent units of block b: [klo, khi).
struct Blk {
  int klo, khi;
  int crit0, crit1;  // update tiles needed before block b's solver (those of its recent units)
  int bulk0;         // further update tiles [bulk0, ntiles), overlapped with block b's solver
  int cor0, cor1;    // chunks of block b-1's recent units (Hr), added to Z of block b
  int np;            // chunks [0, np) of the Z GEMM of block b+1, run during block b's solver
  bool zinit;        // Z of block b was started during block b-1
  bool zvalid;       // Z of block b holds any term
};
__device__ __forceinline__ Blk blk_of(int b, int n, int h, int D, int ntiles, int nblk) {
  Blk r;
  r.klo = count_deg_le(b * D, n, h);
  r.khi = count_deg_le(b * D + D, n, h);
  const int kprev = b > 0 ? count_deg_le((b - 1) * D, n, h) : 0;
  if (b > 0 && r.khi > r.klo) r.crit0 = r.klo / 128, r.crit1 = (r.khi - 1) / 128 + 1;
  else r.crit0 = r.crit1 = r.klo / 128;
  r.bulk0 = (b > 0 && b + 1 < nblk) ? (r.crit1 > r.klo / 128 ? r.crit1 : r.klo / 128) : ntiles;
  if (b > 0 && r.klo > kprev) r.cor0 = kprev / 64, r.cor1 = (r.klo - 1) / 64 + 1;
  else r.cor0 = r.cor1 = 0;
  r.np = b + 1 < nblk ? (r.klo + 63) / 64 : 0;
  r.zinit = b > 0 && (kprev + 63) / 64 > 0;  // np of block b-1
  r.zvalid = r.zinit || r.cor1 > r.cor0;
  return r;
}

// The four phases of the weight tiles in a block: [i0, i1) of phase p.  Update
// phases count tiles as unit tile * nkd + K-chunk (nkd = D / 64 is 1 or 2: a
// shift by nkd - 1 divides by it, a mask of nkd - 1 gives the chunk).
constexpr int kPhCrit = 0, kPhCor = 1, kPhBulk = 2, kPhZ = 3;
__device__ __forceinline__ void phase_range(const Blk& B, int p, int nkd, int ntiles, int& i0, int& i1) {
  i0 = p == kPhCrit ? B.crit0 * nkd : p == kPhCor ? B.cor0 : p == kPhBulk ? B.bulk0 * nkd : 0;
  i1 = p == kPhCrit ? B.crit1 * nkd : p == kPhCor ? B.cor1 : p == kPhBulk ? ntiles * nkd : B.np;
}

template <int ACT, bool LP>
__global__ void __launch_bounds__(kThreads, 1)
    sampler_tc_kernel(const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapW,
                      const __grid_constant__ CUtensorMap mapV2, const __grid_constant__ CUtensorMap mapV3,
                      const __grid_constant__ CUtensorMap mapW2, const TcArgs g) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  unsigned char* Hs = sm + kOffH;
  unsigned char* Ss = sm + kOffS;
  unsigned char* Hr = sm + kOffHr;
  float* Zs = reinterpret_cast<float*>(sm + kOffZ);
  float* LG = reinterpret_cast<float*>(sm + kOffLG);
  float* Pr = reinterpret_cast<float*>(sm + kOffP);
  bf16* Wr = reinterpret_cast<bf16*>(sm + kOffWr);
  bf16* Vr = reinterpret_cast<bf16*>(sm + kOffVr);
  float* PreS = reinterpret_cast<float*>(sm + kOffPS);
  uint32_t* SB = reinterpret_cast<uint32_t*>(sm + kOffSB);
  int* CU = reinterpret_cast<int*>(sm + kOffCU);
  const unsigned long long it_all = g.it_dev ? *g.it_dev : ((unsigned long long)g.it1 << 32 | g.it0);
  const uint32_t it0 = (uint32_t)it_all, it1 = (uint32_t)(it_all >> 32);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kOffBar);
  uint64_t* empty = full + kNStage;
  uint64_t* zfull = empty + kNStage;
  uint64_t* ready = zfull + 1;
  uint64_t* merged = ready + 1;
  uint64_t* drain = merged + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const int n = g.n, h = g.h, D = g.D;
  const int nblk = (n + D - 1) / D;
  const int ntiles = (g.hp + 127) / 128;
  const int nkd = D / 64;
  const int b0 = blockIdx.x * kS;

  if (tid == 0) {
    for (int s = 0; s < kNStage; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    mbar_init(smem_u32(zfull), 1);
    mbar_init(smem_u32(ready), kSolverThreads);
    mbar_init(smem_u32(merged), kHelpers);
    mbar_init(smem_u32(drain), 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  // g1 of every unit is zero until the unit completes; spins start at zero
  // zero g1 (every unit is zero until it completes), the spins, and the
  // solver tables (their padding rows and "no unit" columns stay zero)
  for (int q = tid; q < (kOffSB - kOffH) / 16; q += kThreads) reinterpret_cast<uint4*>(Hs)[q] = make_uint4(0, 0, 0, 0);
  fence_proxy_async();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = (uint32_t)uniform((int)*tmem_slot);
  // A = b1 for every sample
  if (warp < 4) {
#pragma unroll 1
    for (int t = 0; t < ntiles; ++t) {
      const int k = 128 * t + 32 * warp + lane;
      const float x = k < h ? g.b1[k] : 0.0f;
      float v[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = x;
      tmem_st16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(16 * t), v);
    }
  }
  fence_before();
  __syncthreads();
  fence_after();

  if (warp == 4) {
    // ----------------------------------------------------------- producer
    // Tiles in the MMA issuer's order; per block b: the update tiles needed
    // before its solver (W1, block b-1's inputs), the tiles of block b-1's
    // recent units (W2, block b's rows), the remaining update tiles, then the
    // Z GEMM of block b+1 over the units complete before block b (W2, block
    // b+1's rows).
    if (elect_one()) {
      int it = 0;  // slots issued
      bool ok = true;
#pragma unroll 1
      for (int b = 0; b < nblk && ok; ++b) {
        const Blk B = blk_of(b, n, h, D, ntiles, nblk);
#pragma unroll 1
        for (int p = 0; p < 4 && ok; ++p) {
          // the tiles [i0, i1) of phase p, kSlotTiles per slot.  An update
          // phase's index i is unit tile i / nkd, K-chunk i % nkd of block
          // b-1's inputs; a Z phase's is the 64-unit chunk.  A run of tiles
          // with the same rows and consecutive chunks (at most `most`) is one
          // copy through the chunked map of its length.
          const bool upd = p == kPhCrit || p == kPhBulk;
          int i0, i1;
          phase_range(B, p, nkd, ntiles, i0, i1);
          const CUtensorMap* m1 = upd ? &mapW : &mapV;
          const CUtensorMap* m2 = upd ? &mapW2 : &mapV2;
          const int most = upd ? 2 : 3;
          const int sh = upd ? nkd - 1 : 31, msk = upd ? nkd - 1 : -1;
          const int y0 = upd ? 0 : (p == kPhZ ? b + 1 : b) * D, c0 = upd ? (b - 1) * nkd : 0;
#pragma unroll 1
          for (int i = i0; i < i1; i += kSlotTiles) {
            const int cnt = min(kSlotTiles, i1 - i);
            const int s = it % kNSlot;
            if (it >= kNSlot &&
                !test_or_abort(smem_u32(&empty[s]), (uint32_t)((it / kNSlot - 1) & 1), abort, g.err)) {
              ok = false;
              break;
            }
            const uint32_t bar = smem_u32(&full[s]);
            mbar_expect_tx(bar, (uint32_t)(cnt * kTileBytes));
#pragma unroll 1
            for (int j = 0; j < cnt;) {
              const int t = (i + j) >> sh, k = (i + j) & msk;
              // chunks that follow in the same rows: all of a Z phase's, up to the last of an update tile's
              const int run = min(min(most, cnt - j), upd ? nkd - k : kSlotTiles);
              const uint32_t dst = base + kOffRing + (s * kSlotTiles + j) * kTileBytes;
              if (run == 1) tma_load_2d(dst, m1, 64 * (c0 + k), y0 + 128 * t, bar);
              else tma_load_3d(dst, run == 2 ? m2 : &mapV3, 0, y0 + 128 * t, c0 + k, bar);
              j += run;
            }
            ++it;
          }
        }
      }
      // no copy may still be landing when the CTA exits (after a failure
      // some loaded tiles are never consumed)
      for (int p = it > kNSlot ? it - kNSlot : 0; p < it; ++p)
        mbar_wait(smem_u32(&full[p % kNSlot]), (uint32_t)((p / kNSlot) & 1), g.err);
    }
  } else if (warp == 5) {
    // --------------------------------------------------------- MMA issuer
    // Block b: after block b-1's solver, the update of block b's recent units
    // by block b-1's spins and the terms of block b-1's recent units in Z of
    // block b (commit -> zfull); then, while block b's solver runs, the rest
    // of the update and, once block b-1's recent g1 are in the operand, the Z
    // GEMM of block b+1 into the other Z buffer.
    if (elect_one()) {
      int it = 0;  // slots consumed
      bool ok = true, any = false;
#pragma unroll 1
      for (int b = 0; b < nblk; ++b) {
        const Blk B = blk_of(b, n, h, D, ntiles, nblk);
        if (b > 0 && ok) {
          ok = test_or_abort(smem_u32(ready), (uint32_t)((b - 1) & 1), abort, g.err);
          fence_after();
        }
#pragma unroll 1
        for (int p = 0; p < 4; ++p) {
          // the tiles [i0, i1) of phase p in the producer's slots: accumulator
          // column, B operand and first chunk's accumulation.  Each 128 x 64
          // weight tile against a 16 x 64 operand is 4 MMAs of K = 16; one
          // commit releases the slot.
          const bool upd = p == kPhCrit || p == kPhBulk;
          int i0, i1;
          phase_range(B, p, nkd, ntiles, i0, i1);
          const int sh = upd ? nkd - 1 : 31, msk = upd ? nkd - 1 : -1;
          const uint32_t dcol = tmem + (uint32_t)(upd ? 0 : kZCol + 16 * ((p == kPhZ ? b + 1 : b) & 1));
          const uint32_t bop = base + (uint32_t)(upd ? kOffS + ((b - 1) & 1) * (kDmax / 64) * 2048
                                                     : p == kPhZ ? kOffH : kOffHr - 2048 * i0);
          const bool acc0 = upd || (p == kPhCor && B.zinit);
          if (p == kPhZ && B.np > 0 && ok) {
            ok = test_or_abort(smem_u32(merged), (uint32_t)(b & 1), abort, g.err);
            fence_after();
          }
#pragma unroll 1
          for (int i = i0; i < i1 && ok; i += kSlotTiles) {
            const int cnt = min(kSlotTiles, i1 - i);
            const int s = it % kNSlot;
            if (!test_or_abort(smem_u32(&full[s]), (uint32_t)((it / kNSlot) & 1), abort, g.err)) {
              ok = false;
              break;
            }
            fence_after();
#pragma unroll
            for (int j = 0; j < kSlotTiles; ++j) {
              if (j >= cnt) break;
              const uint32_t dc = dcol + (uint32_t)(16 * ((i + j) >> sh));
              const uint64_t da = smem_desc_sw128(base + kOffRing + (s * kSlotTiles + j) * kTileBytes);
              const uint64_t db = smem_desc_sw128(bop + (uint32_t)(((i + j) & msk) * 2048));
              const uint32_t acc = (acc0 || i + j > i0) ? 1u : 0u;
#pragma unroll
              for (int k = 0; k < 4; ++k)
                mma_bf16(dc, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), kIdesc, k > 0 ? 1u : acc);
            }
            mma_commit(smem_u32(&empty[s]));
            ++it;
            any = true;
          }
          if (p == kPhCor) {
            if (ok && any) mma_commit(smem_u32(zfull));  // also covers the previous block's work
            else mbar_arrive(smem_u32(zfull));
          }
        }
      }
      // every MMA has completed before tensor memory is released
      mma_commit(smem_u32(drain));
      mbar_wait(smem_u32(drain), 0u, g.err);
    }
  } else {
    // ---------------- warps 0-3 and 6-9: tensor-memory reads, solver, helpers
    // Warps 0, 1, 6 and 7 are the solver, one warp on each SM sub-partition
    // (warp w runs on w % 4): the solver is issue-bound, and the producer and
    // MMA warps that share sub-partitions 0 and 1 with it issue little.
    // Warps 0-3 read tensor memory; the helpers meanwhile prepare the next
    // block's logits and write out the previous block's spins.
    const bool solver = warp <= 1 || warp == 6 || warp == 7;
    const int sid = (warp <= 1 ? warp : warp - 4) * 32 + lane;  // solver thread
    const int ht = warp < 4 ? tid - 64 : tid - 192;               // helper thread
    const int s_me = sid / kLanes, sub = sid % kLanes;
    float lp = 0.0f, bias = 0.0f;
    const uint32_t tq = tmem + ((uint32_t)(32 * warp) << 16);
    // logit(u) of block b's steps into LG buffer b & 1; threads t0, t0 + nt, ...
    auto logits = [&](int b, int t0, int nt) {
      float* L = LG + (b & 1) * kDrows * kS;
#pragma unroll 1
      for (int q = t0; q < kS * (D / 4); q += nt) {
        const int s = q % kS, t = b * D + 4 * (q / kS);
        const int bb = b0 + s;
        float* dst = L + (size_t)(4 * (q / kS)) * kS + s;
        float x[4];
        if (g.u) {
#pragma unroll
          for (int w = 0; w < 4; ++w) x[w] = (bb < g.B && t + w < n) ? __ldg(g.u + (size_t)bb * n + t + w) : 0.5f;
        } else {
          const uint4 r = philox4x32_10(make_uint4((uint32_t)(t >> 2), (uint32_t)bb + g.boff, it0, it1), g.key0, g.key1);
          x[0] = to_unit(r.x), x[1] = to_unit(r.y), x[2] = to_unit(r.z), x[3] = to_unit(r.w);
        }
#pragma unroll
        for (int w = 0; w < 4; ++w) dst[w * kS] = logit(x[w]);
      }
    };
    // spins of block b (bits in SB buffer b & 1) to the outputs; threads t0,
    // t0 + nt, ...  Runs of 16 steps of one sample (s_out, sx) and the 16
    // samples of one step (stt) go out as 16-byte stores where the whole run
    // is inside the output and aligned, else element by element.
    auto write_spins = [&](int b, int t0, int nt) {
      const uint32_t* sb = SB + (b & 1) * kS * (kDmax / 32);
      const int steps = min(D, n - b * D);
      const bf16 one = __float2bfloat16_rn(1.0f), mone = __float2bfloat16_rn(-1.0f);
      // two spins as BF16 (+1 = 0x3F80, -1 = 0xBF80); bit set in dn: spin -1
      auto bf_pair = [](uint32_t dn) { return 0x3F803F80u | (dn & 1u) << 15 | (dn >> 1 & 1u) << 31; };
#pragma unroll 1
      for (int q = t0; q < kS * (kDmax / 16); q += nt) {
        const int s = q / (kDmax / 16), e0 = 16 * (q % (kDmax / 16));
        const int bb = b0 + s;
        if (bb >= g.B || e0 >= steps) continue;
        const uint32_t up = (sb[s * (kDmax / 32) + (e0 >> 5)] >> (e0 & 16)) & 0xFFFFu;  // bit k: step e0 + k is +1
        const int cnt = min(16, steps - e0);
        int8_t* so = g.s_out + (size_t)bb * n + b * D + e0;
        if (cnt == 16 && (reinterpret_cast<uintptr_t>(so) & 15) == 0) {
          uint32_t w[4];
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            // the 4 bits spread to bit 0 of 4 bytes (the shifted copies do
            // not overlap), then +1 -> 0x01 and -1 -> 0xFF per byte
            const uint32_t m = ((up >> (4 * p)) & 0xFu) * 0x00204081u & 0x01010101u;
            w[p] = m | (m ^ 0x01010101u) * 0xFFu;
          }
          *reinterpret_cast<uint4*>(so) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll 1
          for (int k = 0; k < cnt; ++k) so[k] = (up >> k) & 1u ? (int8_t)1 : (int8_t)-1;
        }
        if (g.sx) {
          bf16* dx = g.sx + (size_t)bb * g.ldsx + b * D + e0;
          if (cnt == 16 && (reinterpret_cast<uintptr_t>(dx) & 15) == 0) {
            const uint32_t dn = ~up;
            uint4* d4 = reinterpret_cast<uint4*>(dx);
            d4[0] = make_uint4(bf_pair(dn), bf_pair(dn >> 2), bf_pair(dn >> 4), bf_pair(dn >> 6));
            d4[1] = make_uint4(bf_pair(dn >> 8), bf_pair(dn >> 10), bf_pair(dn >> 12), bf_pair(dn >> 14));
          } else {
#pragma unroll 1
            for (int k = 0; k < cnt; ++k) dx[k] = (up >> k) & 1u ? one : mone;
          }
        }
      }
      // the 16 samples of each step (stt, sbits): a warp transposes a word of
      // 32 steps with ballots (lane s < 16 holds sample s's word; ballot j
      // collects step j's spins) and lane j keeps step j's column
      const uint32_t valid = b0 + kS <= g.B ? 0xFFFFu : (1u << (g.B - b0)) - 1u;  // samples inside B
      if (g.stt || g.sbits)
#pragma unroll 1
        for (int w = uniform(t0 >> 5); w < (steps + 31) / 32; w += nt >> 5) {
          const int ln = t0 & 31;
          const uint32_t word = ln < kS ? sb[ln * (kDmax / 32) + w] : 0u;
          uint32_t up = 0;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const uint32_t col = __ballot_sync(0xffffffffu, (word >> j) & 1u);
            up = ln == j ? col : up;
          }
          const int e = 32 * w + ln;
          if (e >= steps) continue;
          const uint32_t dn = ~up & valid;  // bit s: sample b0 + s has spin -1 at step e
          if (g.stt) {
            bf16* dt = g.stt + (size_t)(b * D + e) * g.ldst + b0;
            if (b0 + kS <= g.B && (reinterpret_cast<uintptr_t>(dt) & 15) == 0) {
              uint4* d4 = reinterpret_cast<uint4*>(dt);
              d4[0] = make_uint4(bf_pair(dn), bf_pair(dn >> 2), bf_pair(dn >> 4), bf_pair(dn >> 6));
              d4[1] = make_uint4(bf_pair(dn >> 8), bf_pair(dn >> 10), bf_pair(dn >> 12), bf_pair(dn >> 14));
            } else {
#pragma unroll 1
              for (int s = 0; s < kS; ++s)
                if (b0 + s < g.B) dt[s] = (dn >> s) & 1u ? mone : one;
            }
          }
          if (g.sbits) g.sbits[((size_t)(b0 >> 5) * n + b * D + e) * 2 + ((b0 >> 4) & 1)] = (uint16_t)dn;
        }
    };
    // The recent units' weights of block bb (W2 rows of its steps, W1 of its
    // recent units), loaded by the helpers (thread t) into registers during the
    // previous block's solver and stored into Vr / Wr once the solver is done.
    // Vr: thread t owns step t, 5 aligned 16-byte pieces of W2 from unit klo &
    // ~7; Wr: pieces (unit q % 32, inputs 8 (q / 32) ..) for q = t + 128 j, so
    // that a warp's transposing stores hit 32 different units.
    uint4 gv[5], gw[4];
    auto gather_load = [&](int bb, int t) {
      const int klo = count_deg_le(bb * D, n, h), R = count_deg_le(bb * D + D, n, h) - klo;
      const int steps = min(D, n - bb * D), k8 = klo & ~7;
#pragma unroll
      for (int c = 0; c < 5; ++c)
        gv[c] = (t < steps && k8 + 8 * c < g.hp)
                    ? __ldg(reinterpret_cast<const uint4*>(g.v + (size_t)(bb * D + t) * g.hp + k8) + c)
                    : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int q = t + kHelpers * j, r = q & 31, c = q >> 5;
        gw[j] = (8 * c < steps && r < R)  // pieces past the last step stay in [0, np)
                    ? __ldg(reinterpret_cast<const uint4*>(g.w + (size_t)(klo + r) * g.np + (size_t)bb * D) + c)
                    : make_uint4(0, 0, 0, 0);
      }
    };
    auto gather_store = [&](int bb, int t) {
      const int klo = count_deg_le(bb * D, n, h);
      const int steps = min(D, n - bb * D), off = klo & 7;
      // Vr[e][r] = W2 of step e, unit klo + r (r < 32; zero for units past the
      // block's recent ones: they complete after the block, masked in W2)
      if (t < D) {
        uint32_t w[20];
#pragma unroll
        for (int c = 0; c < 5; ++c) w[4 * c] = gv[c].x, w[4 * c + 1] = gv[c].y, w[4 * c + 2] = gv[c].z, w[4 * c + 3] = gv[c].w;
        // the 32 weights from element off on: a shift by off / 2 words (bits 1
        // and 2 of off in turn), then by half a word
#pragma unroll
        for (int i = 0; i < 18; ++i) w[i] = (off & 4) ? w[i + 2] : w[i];
#pragma unroll
        for (int i = 0; i < 17; ++i) w[i] = (off & 2) ? w[i + 1] : w[i];
        uint32_t d[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) d[i] = __byte_perm(w[i], w[i + 1], (off & 1) ? 0x5432 : 0x3210);
        uint4* dst = reinterpret_cast<uint4*>(Vr + t * kLdW);
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[j] = make_uint4(d[4 * j], d[4 * j + 1], d[4 * j + 2], d[4 * j + 3]);
      }
      // Wr[e][r] = W1 of unit klo + r, input of step e (zero for r >= R)
      unsigned short* sw = reinterpret_cast<unsigned short*>(Wr);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int q = t + kHelpers * j, r = q & 31, c = q >> 5;
        if (8 * c >= D) continue;
        const uint32_t w[4] = {gw[j].x, gw[j].y, gw[j].z, gw[j].w};
#pragma unroll
        for (int tt = 0; tt < 8; ++tt) {
          const int e = 8 * c + tt;
          sw[e * kLdW + r] = e < steps ? (unsigned short)(w[tt >> 1] >> (16 * (tt & 1))) : (unsigned short)0;
        }
      }
    };
    // Turn b: the solver draws block b; the helpers prepare block b + 1 and write
    // out block b - 1 (so there is one turn before the first block and one
    // after the last).
#pragma unroll 1
    for (int b = -1; b <= nblk; ++b) {
      const bool draws = b >= 0 && b < nblk;
      const int* cu = CU + (b & 1) * kBlkInts;
      const int klo = uniform(cu[kRmax]), R = uniform(cu[kRmax + 1]), zvalid = uniform(cu[kRmax + 2]);
      const int steps = min(D, n - b * D);
      if (warp < 4 && draws) {
      // Z and the recent pre-activations from tensor memory
      wait_or_abort(smem_u32(zfull), (uint32_t)(b & 1), abort, g.err);
      __syncwarp();
      fence_after();
      // warp-uniform: tcgen05.ld is executed by all lanes of a warp or none
      const bool live = !__any_sync(0xffffffffu, *abort != 0);
      {
        float v[16];
        if (zvalid && live) {
          tmem_ld16(tq + kZCol + 16 * (b & 1), v);
        } else {
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = 0.0f;
        }
        const int e = 32 * warp + lane;
        if (e < D) {
#pragma unroll
          for (int q = 0; q < 16; ++q) Zs[e * kZld + q] = v[q] + bias;  // b2 folded in
        }
      }
      if (R > 0 && live) {
#pragma unroll 1
        for (int t = klo / 128; t <= (klo + R - 1) / 128; ++t) {
          float v[16];
          tmem_ld16(tq + (uint32_t)(16 * t), v);
          const int k = 128 * t + 32 * warp + lane;
#pragma unroll
          for (int q = 0; q < 16; ++q) store_if(k >= klo && k < klo + R, Pr + (k - klo) * kS + q, v[q]);
        }
      }
      fence_before();  // the tensor-memory reads precede the next MMAs into Z (after merged)
      }
      if (draws) asm volatile("bar.sync 1, %0;" ::"n"(kBar1Threads) : "memory");
      {  // b2 of the next block's step, ahead of its use
        const int i = (b + 1) * D + 32 * warp + lane;
        bias = warp < 4 && 32 * warp + lane < D && i < n ? __ldg(g.b2 + i) : 0.0f;
      }
      // (c) the D draws of the block (the solver warps), then the block's
      // spins as the update GEMM's operand; the helpers meanwhile
      if (solver) {
        uint32_t* sb = SB + (b & 1) * kS * (kDmax / 32);
        if (draws)
          solve<ACT, LP>(Pr, Vr, Wr, Zs, LG + (b & 1) * kDrows * kS, cu, sb, PreS, Hr, s_me, sub, klo, R, steps);
        asm volatile("bar.sync 1, %0;" ::"n"(kBar1Threads) : "memory");
        if (!draws) continue;
        // (d) 8 spins of one sample per 16-byte store (+1 = 0x3F80, -1 = 0xBF80)
        unsigned char* ss = Ss + (b & 1) * (kDmax / 64) * 2048;
#pragma unroll 1
        for (int q = sid; q < kS * (D / 8); q += kSolverThreads) {
          const int s = q / (D / 8), e = 8 * (q % (D / 8));
          const uint32_t bits = ~(sb[s * (kDmax / 32) + (e >> 5)] >> (e & 31));  // bit set: spin -1
          uint32_t w[4];
#pragma unroll
          for (int p = 0; p < 4; ++p)
            w[p] = 0x3F803F80u | ((bits >> (2 * p)) & 1u) << 15 | ((bits >> (2 * p + 1)) & 1u) << 31;
          *reinterpret_cast<uint4*>(ss + (e >> 6) * 2048 + sw128_offset(s, e & 63)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        fence_proxy_async();
        fence_before();
        mbar_arrive(smem_u32(ready));
      } else {
        // block b-1's recent g1 from the staging operand into the GEMM
        // operand (the block's Z GEMM has read Hr: zfull), then release Hr
        // to the solver and the operand to the next Z GEMM
        if (draws) {
          if (b > 0) {
            const int kprev = count_deg_le((b - 1) * D, n, h), cb = kprev >> 6;
#pragma unroll 1
            for (int q = ht; q < (klo - kprev) * kS; q += kHelpers) {
              const int k = kprev + q / kS, s = q % kS;
              const uint32_t o = sw128_offset(s, k & 63);
              bf16* src = reinterpret_cast<bf16*>(Hr + ((k >> 6) - cb) * 2048 + o);
              *reinterpret_cast<bf16*>(Hs + (k >> 6) * 2048 + o) = *src;
              *src = __float2bfloat16_rn(0.0f);  // Hr is zero outside the current recent units
            }
          }
          fence_proxy_async();
          fence_before();
          mbar_arrive(smem_u32(merged));
          asm volatile("bar.arrive 2, %0;" ::"n"(kBar2Threads) : "memory");
        }
        if (LP && b > 0) {
          // log pi of block b - 1: the solver left +-z in place of the logits
          // of u.  The entries that a thread reads are those that it fills
          // next for block b + 1.
          const float* L = LG + ((b - 1) & 1) * kDrows * kS;
#pragma unroll 1
          for (int q = ht; q < kS * (D / 4); q += kHelpers) {
            const int e = 4 * (q / kS), left = n - (b - 1) * D - e;
            // sum of log sigma(x) = min(x, 0) - log(1 + exp(-|x|)): one
            // logarithm of the four factors, kept as their product minus 1
            // (0 for steps past the last, x = 1e30)
            float lin = 0.0f, prod1 = 0.0f;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              const float x = w < left ? L[(e + w) * kS + q % kS] : 1e30f;
              lin += fminf(x, 0.0f);
              prod1 = fmaf(expf(-fabsf(x)), 1.0f + prod1, prod1);
            }
            lp += lin - log1pf(prod1);
          }
        }
        if (b + 1 < nblk) {
          // block b + 1's schedule, out of the way of its solver: TC[r], the
          // step whose spin is recent unit r's last input, and klo, R, zvalid
          if (warp == 2) {
            const Blk N = blk_of(b + 1, n, h, D, ntiles, nblk);
            int* cn = CU + ((b + 1) & 1) * kBlkInts;
            const int Rn = N.khi - N.klo;  // <= kRmax (checked by the host)
            cn[lane] = lane < Rn ? degree(N.klo + lane, n, h) - 1 - (b + 1) * D : D;
            const int x = lane == 0 ? N.klo : lane == 1 ? Rn : (int)N.zvalid;
            if (lane < 3) cn[kRmax + lane] = x;
          }
          logits(b + 1, ht, kHelpers);
          gather_load(b + 1, ht);
        }
        if (b > 0) write_spins(b - 1, ht, kHelpers);
        asm volatile("bar.sync 1, %0;" ::"n"(kBar1Threads) : "memory");
        if (b + 1 < nblk) gather_store(b + 1, ht);
      }
    }
    if (LP && !solver) {  // the partial sums of log pi of each sample's eight threads
      lp += __shfl_xor_sync(0xffffffffu, lp, 16);
      if (lane < kS) LG[(ht >> 5) * kS + lane] = lp;
      asm volatile("bar.sync 2, %0;" ::"n"(kHelpers) : "memory");
      if (warp == 2 && lane < kS && b0 + lane < g.B && !*abort)
        g.logp[b0 + lane] = (LG[lane] + LG[kS + lane]) + (LG[2 * kS + lane] + LG[3 * kS + lane]);
    }
  }

  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 5) {
    __syncwarp();
    fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

OncePerDevice g_smem;

// largest number of units completing inside one block of D steps
int max_recent(int n, int h, int D) {
  int r = 0;
  for (int b = 0; b * D < n; ++b) r = std::max(r, count_deg_le(b * D + D, n, h) - count_deg_le(b * D, n, h));
  return r;
}

}  // namespace

// Block size the tensor-core sampler would use for this model, or 0 when it
// does not apply (FP32 weights, more than 2048 hidden units, or more than
// 32 units completing within every block size).
int sampler_tc_block(const vqmc_ctx* c) {
  // h < n: distinct degrees, at most one unit completes per step
  if (c->prec != VQMC_PREC_BF16 || c->hp > kMaxHp || c->h >= c->n) return 0;
  for (int D : {128, 64})
    if (max_recent(c->n, c->h, D) <= kRmax) return D;
  return 0;
}

cudaError_t launch_sampler_tc(const vqmc_ctx* c, int B, const float* d_u, uint64_t iteration, int8_t* d_s,
                              float* d_logp, cudaStream_t st, void* sx, void* stt, uint32_t* sbits,
                              const unsigned long long* it_dev) {
  const int D = sampler_tc_block(c);
  if (D == 0 || !gemm_tc_available()) return cudaErrorNotSupported;
  if (B <= 0) return cudaSuccess;
  // v_s [sampler_rows(n)][hp] and w_s [h][np] (hp, np multiples of 64): one
  // 128 x 64 tile per copy, or 2 or 3 consecutive chunks of the same rows
  CUtensorMap mapV, mapW, mapV2, mapV3, mapW2;
  if (!tc_encode_bf16(&mapV, c->v_s, sampler_rows(c->n), c->hp, c->hp, 128) ||
      !tc_encode_bf16(&mapW, c->w_s, c->h, c->np, c->np, 128) ||
      !tc_encode_bf16_chunks(&mapV2, c->v_s, sampler_rows(c->n), c->hp, c->hp, 128, 2) ||
      !tc_encode_bf16_chunks(&mapV3, c->v_s, sampler_rows(c->n), c->hp, c->hp, 128, 3) ||
      !tc_encode_bf16_chunks(&mapW2, c->w_s, c->h, c->np, c->np, 128, 2))
    return cudaErrorInvalidValue;
  using Kernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, TcArgs);
  constexpr Kernel kernels[] = {sampler_tc_kernel<VQMC_ACT_RELU, false>, sampler_tc_kernel<VQMC_ACT_RELU, true>,
                                sampler_tc_kernel<VQMC_ACT_SIGMOID, false>, sampler_tc_kernel<VQMC_ACT_SIGMOID, true>};
  const cudaError_t e = allow_smem(g_smem, kernels, kSmemBytes);
  if (e != cudaSuccess) return e;
  TcArgs a;
  a.n = c->n;
  a.h = c->h;
  a.hp = c->hp;
  a.B = B;
  a.D = D;
  a.w = reinterpret_cast<const bf16*>(c->w_s);
  a.np = c->np;
  a.v = reinterpret_cast<const bf16*>(c->v_s);
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
  a.sx = reinterpret_cast<bf16*>(sx);
  a.ldsx = c->np;
  a.stt = reinterpret_cast<bf16*>(stt);
  a.ldst = c->Bp;
  a.sbits = reinterpret_cast<uint16_t*>(sbits);
  const Kernel kernel = kernels[(c->act == VQMC_ACT_RELU ? 0 : 2) + (d_logp != nullptr)];
  kernel<<<(B + kS - 1) / kS, kThreads, kSmemBytes, st>>>(mapV, mapW, mapV2, mapV3, mapW2, a);
  return cudaGetLastError();
}

}  // namespace vqmc
