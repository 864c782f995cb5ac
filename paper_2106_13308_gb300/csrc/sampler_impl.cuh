// Blocked autoregressive sampler on the CUDA cores, included by one
// translation unit per weight type (sampler_bf16.cu, sampler_f32.cu).
//
// Algorithm 1 with the incremental forward pass (Sec. 2.3): the logit of step
// e (0-based) is
//     z_e = b2_e + sum_{k complete} W2_ek g1_k,   g1_k = act(b1_k + sum_{j<m(k)} W1_kj s_j),
// and with sorted degrees the complete units are a prefix.  A CTA draws 8
// samples.  The hidden units go in groups of 16 in degree order; the steps
// whose newest complete unit lies in group g ("the group's steps") are taken
// in blocks of at most 16, each in three phases:
//   Z  the terms of every unit before group g in the block's logits, a small
//      GEMM (steps x samples over the complete units) on all warps;
//   solve  two warps draw the block's spins one after another, carrying the
//      pre-activations of group g's 16 units (the only ones that complete
//      inside the block), 8 lanes per sample; the other warps meanwhile stage
//      the next block's tables and write the previous block's outputs;
//   U  the block's spins into the pre-activations of the units after group g,
//      a second small GEMM on all warps.
// All pre-activations (g1 once complete) of the CTA's samples stay in shared
// memory; the weights are read once per CTA from L2.
//
// The order of every FP32 operation is fixed by h alone.  A
// pre-activation is summed over the inputs in order.  A logit is summed as
// GW*64 chains over the units k = c, c + GW*64, c + 2 GW*64, ... (c the
// class of a unit), the chains of classes 2l and 2l + 1 added, then for each
// run of 32 such pairs ("virtual warp") a binary tree over l that joins l
// with l ^ 16 first, then ^ 8, 4, 2, 1, and the GW results added to b2 in
// order.  GW is 1 up to hp = 64, 2 up to 2048 and 4 beyond.  Group g holds 8
// neighbouring pairs (one octet) of one virtual warp, so the solver finishes
// the tree from its 8 leaves and the partial sums of the other octets.
//
// What bounds it: up to about 1000 hidden units the chain from one draw to the next
// (about 220 cycles, on two of the CTA's eight warps) with the Z and U phases before
// and after a block's draws (at n = h = 1000 some 350 cycles a draw), beyond it the
// issue slots and shared-memory reads of these phases (2 bytes per multiply-add;
// at n = h = 2000 55% of the issue slots and 60% of the load/store pipe are busy);
// two CTAs on an SM overlap one's draws with the other's GEMMs.  Measured
// (GB300), against one step at a time with a reduction over the CTA's lanes for
// every draw: a sampling and energy pass at n = h = 1000, 1024 samples (BF16)
// 1457 -> 293 us; a training step at n = h = 2000, 8192 samples (BF16) 9194 ->
// 4013 us; the draws alone at n = 10000, h = 2000, 2048 samples (FP32) 7800 ->
// 5040 us (16 TFLOP/s).  Loops are rolled and branches uniform: peeled and with
// branches on lane values it ran at 2.7 cycles per instruction.  No per-step store in
// the solver (25 cycles each, 70 behind a divergent branch): the spins are written
// after a block.
//
// Where it is not the faster one (many units completing at a step, or a small model's
// large batch), sampler.cu takes the sampler of sampler_steps.cuh: the same bits.
#pragma once

#include <type_traits>

#include "f32x2.cuh"
#include "sampler.cuh"

namespace vqmc {

namespace {

constexpr int kSamples = 8;      // samples per CTA
constexpr int kSteps = 16;       // steps per block
constexpr int kGroup = 16;       // hidden units per group
constexpr int kLeaves = kGroup / 2;
constexpr int kTI = 4;           // steps per Z task
constexpr int kWarps = 8;
constexpr int kSolvers = 2;      // warps that draw, 4 samples each: the last ones
constexpr int kThreads = 32 * kWarps;
constexpr int kChunk = 64;       // units per chunk of the state

__device__ __forceinline__ float sum2(uint64_t v) {
  float lo, hi;
  unpack2(v, lo, hi);
  return lo + hi;
}
// 16 bytes from global to shared memory, asynchronously
__device__ __forceinline__ void cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {  // all but the last N groups have landed
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// 16 bytes to shared memory if in: one predicated store (a divergent branch
// around it costs about 70 cycles)
__device__ __forceinline__ void st16_if(uint32_t dst, uint64_t x, uint64_t y, bool in) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\t@q st.shared.v2.b64 [%0], {%1, %2};\n\t}" ::"r"(dst), "l"(x),
               "l"(y), "r"((int)in)
               : "memory");
}

// Weights as stored: those of one pair of units (2q, 2q + 1), and of four
// consecutive units (two pairs); widened to FP32 pairs (BF16 by a shift).
template <typename T>
struct Raw;
template <>
struct Raw<bf16> {
  using two = uint32_t;
  using four = unsigned long long;
  static __device__ __forceinline__ uint64_t f32(two x) {
    return pack2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
  }
  // zero if !in; volatile: issued where it stands (before the draws)
  static __device__ __forceinline__ four ld4(const bf16* p, bool in) {
    four v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\tmov.b64 %0, 0;\n\t@q ld.global.nc.b64 %0, [%1];\n\t}"
                 : "=l"(v)
                 : "l"(p), "r"((int)in));
    return v;
  }
  static __device__ __forceinline__ uint64_t lo(const four& x) { return f32((uint32_t)x); }
  static __device__ __forceinline__ uint64_t hi(const four& x) { return f32((uint32_t)(x >> 32)); }
};
template <>
struct Raw<float> {
  using two = uint64_t;
  using four = ulonglong2;
  static __device__ __forceinline__ uint64_t f32(two x) { return x; }
  static __device__ __forceinline__ four ld4(const float* p, bool in) {
    four v;
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\tmov.b64 %0, 0;\n\tmov.b64 %1, 0;\n\t"
        "@q ld.global.nc.v2.b64 {%0, %1}, [%2];\n\t}"
        : "=l"(v.x), "=l"(v.y)
        : "l"(p), "r"((int)in));
    return v;
  }
  static __device__ __forceinline__ uint64_t lo(const four& x) { return x.x; }
  static __device__ __forceinline__ uint64_t hi(const four& x) { return x.y; }
};

// The tables of one block that the solver reads, staged during the previous
// block's draws.
struct Leaf {       // one pair of the group's units at one step
  uint64_t v, w;    // W2 (this step's output) and W1 (this step's input)
};
struct LeafSum {    // one leaf of one sample at one step
  uint64_t pre;     // the pair's two chains over the units before the group
  uint64_t join;    // {the sum that joins the leaf on the tree's first level, on the second}
};
struct Tables {
  Leaf leaf[kSteps][kLeaves];
  float logit[kSteps][kSamples];        // logit(u)
  float b2[kSteps];
  int done[kSteps];                     // units of the group complete at the step
};
// What a block's draws leave for the outputs: bit t of bits[s]: spin of step
// e0 + t is +1; s_e z_e for log pi.
struct Drawn {
  float x[kSteps * kSamples];
  uint32_t bits[kSamples];
};

// Steps [e0, e1) of group grp.
struct Block {
  int e0, e1, grp, pad;
};

// count_deg_le and degree in 32 bits: n h < 2^31 for every model (h <= 5120; a sparse
// instance has n <= 51,200, a dense one n^2 FP32 couplings in device memory).
__device__ __forceinline__ int complete_before(int e, int n, int h) {  // units with m(k) <= e
  if (e < 1) return 0;
  if (n <= 1) return h;
  return min((int)(((unsigned)e * (unsigned)h + (unsigned)(n - 2)) / (unsigned)(n - 1)), h);
}
__device__ __forceinline__ Block next_block(int e0, int n, int h) {
  Block b;
  b.e0 = e0;
  b.grp = complete_before(e0, n, h) / kGroup;
  const int last = kGroup * b.grp + kGroup - 1;  // the group's last unit is complete from step degree(last) on
  const int e1 = last < h ? 1 + (int)((unsigned)last * (unsigned)(n - 1) / (unsigned)h) : n;
  b.e1 = min(min(e1, n), e0 + kSteps);
  b.pad = 0;
  return b;
}

template <typename WT, int GW, bool RELU>
struct BlockSampler {
  static constexpr int GL = GW * 32;  // pair classes
  static constexpr int RL = GW * 64;  // classes
  // a logit is ((zb + the group's tree) + post[0]) + ...
  struct Post {
    float zb, lg, post[GW == 4 ? 6 : 2];
  };

  // W2 reaches shared memory through a ring per warp (cp.async, no other warp
  // involved): a stage holds 4 rows x 64 units, one round of Z.
  static constexpr int kStageBytes = 256 * (int)sizeof(WT);
  static constexpr int kDepth = sizeof(WT) == 2 ? 4 : 2;
  static constexpr int kRingBytes = kDepth * kStageBytes;

  // shared memory (bytes).  State: chunks of 64 units x 8 samples,
  // [chunk][sample][64], the one past hp for a group that starts at hp; a
  // chunk of zeros stands for pairs that are not complete.
  static constexpr int kStateChunk = kSamples * kChunk;                   // floats
  static constexpr int kOffZ = 0;                                         // leaf records [16][8][8] (LeafSum)
  static constexpr int kOffR = kOffZ + kSteps * kSamples * kLeaves * 16;  // ring of each warp
  static constexpr int kOffT = kOffR + kWarps * kRingBytes;               // trees of the other virtual warps [GW][16][8]
  static constexpr int kOffS = kOffT + GW * kSteps * kSamples * 4;        // spins {s, s} [16][8]
  static constexpr int kOffP = kOffS + kSteps * kSamples * 8;             // what the solver adds to a tree [16][8] (Post)
  static constexpr int kOffTab = kOffP + kSteps * kSamples * (int)sizeof(Post);  // Tables [2]
  static constexpr int kOffDrawn = kOffTab + 2 * (int)sizeof(Tables);     // Drawn [2]
  static constexpr int kOffNext = kOffDrawn + 2 * (int)sizeof(Drawn);     // Block [2]
  static constexpr int kOffZero = kOffNext + 2 * (int)sizeof(Block);      // a zero chunk
  static constexpr int kOffA = kOffZero + 4 * kStateChunk;                // state
  static_assert(kOffTab % 16 == 0 && sizeof(Tables) % 16 == 0 && kOffNext % 16 == 0 && kOffA % 16 == 0, "alignment");
  static size_t smem_bytes(int hp) { return kOffA + (size_t)(hp / kChunk + 1) * kStateChunk * 4; }

  // hidden activation as the output layer sees it: rounded to bfloat16 in
  // the BF16 model (as the BF16 forward GEMM stores it), exact in FP32
  static __device__ __forceinline__ float g1(float a) {
    const float g = RELU ? fmaxf(a, 0.0f) : 1.0f / (1.0f + expf(-a));
    if constexpr (sizeof(WT) == 2) return __bfloat162float(__float2bfloat16_rn(g));
    else return g;
  }
  static __device__ __forceinline__ uint64_t g1_pair(uint64_t a) {
    float lo, hi;
    unpack2(a, lo, hi);
    return pack2(g1(lo), g1(hi));
  }

  // What a warp streams through its ring: the W2 rows of its first Z task of
  // the next block (of every further task by itself).
  struct Stream {
    const WT* p;     // this lane's source of the next stage
    int left;        // stages left
    uint32_t slot;   // byte offset of the next stage in the ring
  };
  static constexpr int kCol = 16 / (int)sizeof(WT);  // weights per lane and copy
  static constexpr int kZLanes = 64 / kCol;          // lanes per row of a stage
  static constexpr int kCopies = kStageBytes / 512;  // per lane and stage
  static __device__ __forceinline__ void issue(Stream& x, uint32_t ring, int hp, int lane) {
    if (x.left > 0) {
#pragma unroll
      for (int j = 0; j < kCopies; ++j) cp16(ring + x.slot + 16 * lane + 512 * j, x.p + j * (32 / kZLanes) * hp);
      x.p += RL, --x.left;
    }
    cp_commit();
    x.slot = (x.slot + kStageBytes) & (kRingBytes - 1);
  }
  static __device__ __forceinline__ int rounds(int vw, int pairs) {  // in which some lane's pair is complete
    return pairs > vw * 32 ? (pairs - vw * 32 + GL - 1) / GL : 0;
  }
  // starts the stream of Z task (vw, 4 steps from e); sampler_rows() leaves room past the last step
  static __device__ __forceinline__ void start(Stream& x, uint32_t ring, const WT* v, int hp, int e, int vw, int lane,
                                               int pairs) {
    x.p = v + (unsigned)((e + lane / kZLanes) * hp + 64 * vw + (lane % kZLanes) * kCol);
    x.left = rounds(vw, pairs), x.slot = 0;
#pragma unroll 1
    for (int d = 0; d < kDepth; ++d) issue(x, ring, hp, lane);
  }

  // Z task: virtual warp vw, 4 steps from block step t0.  Lane (i, g), i < 16,
  // sums the chains of pair classes i and i + 16 over the complete units (pairs
  // below `pairs`) for samples 4g .. 4g + 3: the tree's first level joins the
  // two on the lane itself.  32 accumulator pairs per lane, each weight pair
  // serving 4 FMAs and each state pair 4.
  static __device__ __forceinline__ void z_task(Stream& x, const unsigned char* ring, uint32_t ring_s, int hp,
                                                const float* A, const float* zero, int t0, int vw, int lane, int pairs,
                                                bool leaves, int octet, LeafSum* Z, float* T) {
    uint64_t acc[2][kTI][4];
#pragma unroll
    for (int i = 0; i < 2 * kTI * 4; ++i) acc[i / 16][i / 4 % 4][i % 4] = 0ull;
    const int nr = rounds(vw, pairs), i16 = lane & 15, sg = lane >> 4;
    int q = vw * 32 + i16;
    const float* a = A + vw * kStateChunk + 4 * sg * kChunk + 2 * i16;
#pragma unroll 1
    for (int r = 0; r < nr; ++r) {
      uint64_t xs[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint64_t* xp = reinterpret_cast<const uint64_t*>(q + 16 * h < pairs ? a + 32 * h : zero);
#pragma unroll
        for (int s = 0; s < 4; ++s) xs[h][s] = xp[s * kChunk / 2];
      }
      cp_wait<kDepth - 1>();
      __syncwarp();
      const typename Raw<WT>::two* w = reinterpret_cast<const typename Raw<WT>::two*>(ring + x.slot) + i16;
#pragma unroll
      for (int t = 0; t < kTI; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint64_t wf = Raw<WT>::f32(w[32 * t + 16 * h]);
#pragma unroll
          for (int s = 0; s < 4; ++s) acc[h][t][s] = fma2(wf, xs[h][s], acc[h][t][s]);
        }
      __syncwarp();
      issue(x, ring_s, hp, lane);
      q += GL;
      a += GW * kStateChunk;
    }
    if (leaves) {
      // the group's own octet keeps its pairs, each with the sums that join
      // it on the tree's first two levels
      const bool own = (i16 >> 3) == (octet & 1), upper = octet >= 2;
      const uint32_t rec =
          (uint32_t)__cvta_generic_to_shared(Z + (t0 * kSamples + 4 * sg) * kLeaves + (lane & 7));
#pragma unroll
      for (int t = 0; t < kTI; ++t)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const float v0 = sum2(acc[0][t][s]), v1 = sum2(acc[1][t][s]);
          const float d = __shfl_xor_sync(0xffffffffu, v0 + v1, 8);
          st16_if(rec + (t * kSamples + s) * kLeaves * 16, upper ? acc[1][t][s] : acc[0][t][s], pack2(upper ? v0 : v1, d),
                  own);
        }
    } else {
      // the rest of the tree: 16 values over 16 lanes, halving the values
      // held at every level; lane i ends with value i
      float v[kTI * 4];
#pragma unroll
      for (int i = 0; i < kTI * 4; ++i) v[i] = sum2(acc[0][i / 4][i % 4]) + sum2(acc[1][i / 4][i % 4]);
#pragma unroll
      for (int o = 8; o >= 1; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
          const float keep = up ? v[i + o] : v[i], send = up ? v[i] : v[i + o];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      T[(vw * kSteps + t0 + (i16 >> 2)) * kSamples + 4 * sg + (i16 & 3)] = v[0];
    }
  }

  // The draws of one block for 4 samples by one warp, 8 lanes per sample: lane
  // l of a sample holds leaf l of the group's octet.  The chain from one draw
  // to the next (the newest unit's pre-activation and act, its leaf's FMA, four
  // levels of sums, three shuffles, b2, the other virtual warps' trees, the
  // compare) is about 220 cycles; a spin has two values, so both logits of step
  // t + 1 are begun before spin t is known, and each iteration finishes the two
  // logits of step t beside the first half of step t + 1's.  Only the units
  // that complete with spin t differ between the two.  Nothing is stored per
  // step (a store costs about 25 cycles there, a divergent one 70).
  // A: the group's units of sample 0 in the state; multi: several units may
  // complete with one spin; over: the group's steps end with this block.
  static __device__ __forceinline__ void solve(const Tables& tb, Drawn& out, const LeafSum* Z, const float* T, Post* P,
                                               uint64_t* SP, float* A, int steps, int wg, int sw, int lane, bool multi,
                                               bool over) {
    const int s = 4 * sw + (lane >> 3), l = lane & 7;
    // what joins the group's tree to a logit: one (step, sample) per lane and turn
#pragma unroll
    for (int i = lane; i < 4 * kSteps; i += 32) {
      const int t = i >> 2, sq = 4 * sw + (i & 3);
      Post x{};
      x.zb = tb.b2[t], x.lg = tb.logit[t][sq];
      if constexpr (GW > 1) {
#pragma unroll
        for (int q = 0; q < GW; ++q) {
          const float y = T[(q * kSteps + t) * kSamples + sq];
          x.zb = q < wg ? x.zb + y : x.zb;
          if (q > 0) x.post[q - 1] = q > wg ? y : 0.0f;
        }
      }
      P[t * kSamples + sq] = x;
    }
    __syncwarp();
    uint64_t* row = reinterpret_cast<uint64_t*>(A + s * kChunk) + l;
    const LeafSum* zr = Z + s * kLeaves + l;
    float a0, a1, g0 = 0.0f, g1_ = 0.0f;  // this leaf's units: pre-activations, activations (zero until complete)
    unpack2(*row, a0, a1);
    const int first = uniform(tb.done[0]);
    int u = 0;  // units done so far
#pragma unroll 1
    for (; u < first; ++u) {
      const float f = g1(u & 1 ? a1 : a0);
      const bool mine = (u >> 1) == l;
      g0 = mine && !(u & 1) ? f : g0;
      g1_ = mine && (u & 1) ? f : g1_;
    }
    auto leaf_sum = [&](const ulonglong2& r, uint64_t v, float x0, float x1) {
      float c, d;
      unpack2(r.y, c, d);
      return (sum2(fma2(v, pack2(x0, x1), r.x)) + c) + d;
    };
    ulonglong2 vw = *reinterpret_cast<const ulonglong2*>(&tb.leaf[0][l]);
    // the candidates after spin t - 1 = -1 (m) and +1 (p)
    float ym = leaf_sum(*reinterpret_cast<const ulonglong2*>(zr), vw.x, g0, g1_), yp = ym;
    float m0 = g0, m1 = g1_, p0 = g0, p1 = g1_;
    uint64_t w = 0ull;  // W1 of spin t - 1
    bool up = true;
    uint32_t bits = 0;
    float xlo = 0.0f, xhi = 0.0f;  // s z of steps l and l + 8
    // one step; MULTI: several units may complete with one spin
    auto step = [&](int t, auto multi) {
      constexpr bool MULTI = decltype(multi)::value;
      const int tn = min(t + 1, steps - 1);
      const ulonglong2 rn = *reinterpret_cast<const ulonglong2*>(zr + tn * kSamples * kLeaves);
      const ulonglong2 vwn = *reinterpret_cast<const ulonglong2*>(&tb.leaf[tn][l]);
      const float4 pz = *reinterpret_cast<const float4*>(P + t * kSamples + s);
      int dn = tb.done[tn];
      if constexpr (MULTI || !RELU) dn = uniform(dn);
      // spin t - 1 is known: its pre-activations and activations
      const float sv = up ? 1.0f : -1.0f;
      unpack2(fma2(w, pack2(sv, sv), pack2(a0, a1)), a0, a1);
      w = vw.y;
      g0 = up ? p0 : m0, g1_ = up ? p1 : m1;
      m0 = p0 = g0, m1 = p1 = g1_;
      // the units that complete with spin t, for both of its values
      float w0, w1;
      unpack2(w, w0, w1);
      auto complete = [&](bool any) {
        const float xa = u & 1 ? a1 : a0, xw = u & 1 ? w1 : w0;
        const float fm = g1(xa - xw), fp = g1(xa + xw);
        const bool mine = any && (u >> 1) == l;
        const bool lo = mine && !(u & 1), hi = mine && (u & 1);
        m0 = lo ? fm : m0, p0 = lo ? fp : p0;
        m1 = hi ? fm : m1, p1 = hi ? fp : p1;
      };
      if constexpr (MULTI) {
#pragma unroll 1
        for (; u < dn; ++u) complete(true);
      } else if constexpr (RELU) {
        complete(u < dn);
      } else {
        if (u < dn) complete(true);
      }
      u = dn;
      // the two logits of step t
      float zm = ym + __shfl_xor_sync(0xffffffffu, ym, 4), zp = yp + __shfl_xor_sync(0xffffffffu, yp, 4);
      zm += __shfl_xor_sync(0xffffffffu, zm, 2), zp += __shfl_xor_sync(0xffffffffu, zp, 2);
      zm += __shfl_xor_sync(0xffffffffu, zm, 1), zp += __shfl_xor_sync(0xffffffffu, zp, 1);
      zm = pz.x + zm, zp = pz.x + zp;
      if constexpr (GW > 1) zm += pz.z, zp += pz.z;
      if constexpr (GW == 4) {
        const float q = P[t * kSamples + s].post[2];
        zm = (zm + pz.w) + q, zp = (zp + pz.w) + q;
      }
      ym = leaf_sum(rn, vwn.x, m0, m1);
      yp = leaf_sum(rn, vwn.x, p0, p1);
      vw = vwn;
      const float z = up ? zp : zm;
      up = z > pz.y;  // u < sigma(z)
      const float x = up ? z : -z;
      xlo = t == l ? x : xlo, xhi = t == l + 8 ? x : xhi;
      bits |= (up ? 1u : 0u) << t;
    };
    if (multi) {
#pragma unroll 1
      for (int t = 0; t < steps; ++t) step(t, std::true_type{});
    } else {
#pragma unroll 1
      for (int t = 0; t < steps; t += 2) {
        step(t, std::false_type{});
        if (t + 1 < steps) step(t + 1, std::false_type{});
      }
    }
    out.bits[s] = bits;
    out.x[l * kSamples + s] = xlo, out.x[(l + 8) * kSamples + s] = xhi;
#pragma unroll
    for (int t = l; t < kSteps; t += 8) {
      const float sn = (bits >> t) & 1u ? 1.0f : -1.0f;
      SP[t * kSamples + s] = pack2(sn, sn);
    }
    // the group's state back: g1 if its steps are over
    const float sv = up ? 1.0f : -1.0f;
    const uint64_t a = fma2(w, pack2(sv, sv), pack2(a0, a1));
    *row = over ? g1_pair(a) : a;
  }
};

// Fills the tables of block b; i: 0 .. 63
template <typename WT>
__device__ __forceinline__ void stage_tables(Tables* tb, const SamplerArgs& g, const Block& b, int b0, uint32_t it0,
                                             uint32_t it1, int i) {
  using R = Raw<WT>;
  const int steps = b.e1 - b.e0, k0 = kGroup * b.grp;
  const WT* wt = reinterpret_cast<const WT*>(g.wt);
  const WT* v = reinterpret_cast<const WT*>(g.v);
  const int t = i >> 2, c = i & 3;  // units 4c .. 4c + 3 of the group at step t
  typename R::four wv{}, ww{};
  if (t < steps && k0 + kGroup <= g.hp) {
    wv = __ldg(reinterpret_cast<const typename R::four*>(v + (size_t)(b.e0 + t) * g.hp + k0 + 4 * c));
    ww = __ldg(reinterpret_cast<const typename R::four*>(wt + (size_t)(b.e0 + 1 + t) * g.hp + k0 + 4 * c));
  }
  const int e = b.e0 + t, done = complete_before(e, g.n, g.h) - k0 - 4 * c;
  tb->leaf[t][2 * c] = Leaf{R::lo(wv), R::lo(ww)}, tb->leaf[t][2 * c + 1] = Leaf{R::hi(wv), R::hi(ww)};
  if (c == 0) tb->b2[t] = e < b.e1 ? __ldg(g.b2 + e) : 0.0f, tb->done[t] = done;
  // the uniforms: 4 steps of one sample per thread (a block touches at most 5 groups of 4 steps)
  const int s = i & 7, c4 = 4 * ((b.e0 >> 2) + (i >> 3));
  if (c4 < b.e1) {
    uint32_t xw[4] = {0, 0, 0, 0};
    if (!g.u) {
      const uint4 r = philox4x32_10(make_uint4((uint32_t)c4 >> 2, (uint32_t)(b0 + s) + g.boff, it0, it1), g.key0, g.key1);
      xw[0] = r.x, xw[1] = r.y, xw[2] = r.z, xw[3] = r.w;
    }
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      const int e4 = c4 + j;
      const uint32_t w = j & 2 ? (j & 1 ? xw[3] : xw[2]) : (j & 1 ? xw[1] : xw[0]);
      if (e4 < b.e0 || e4 >= b.e1) continue;
      const float u = !g.u ? to_unit(w) : b0 + s < g.B ? __ldg(g.u + (size_t)(b0 + s) * g.n + e4) : 0.5f;
      tb->logit[e4 - b.e0][s] = logit(u);
    }
  }
}

// The outputs of block b by one warp; lanes 0 .. 7 keep log pi of the samples.
__device__ __forceinline__ void write_block(const SamplerArgs& g, const Block& b, Drawn* d, int b0, int lane,
                                            float& lp) {
  const int steps = b.e1 - b.e0, s = lane >> 2;
  const uint32_t bits = d->bits[s];
  if (b0 + s < g.B) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int t = 4 * (lane & 3) + j;
      if (t < steps) g.s_out[(size_t)(b0 + s) * g.n + b.e0 + t] = (bits >> t) & 1u ? (int8_t)1 : (int8_t)-1;
    }
  }
  if (g.logp) {
#pragma unroll 1
    for (int q = lane; q < steps * kSamples; q += 32) d->x[q] = log_sigmoid(d->x[q]);
    __syncwarp();
    if (lane < kSamples)
#pragma unroll 1
      for (int t = 0; t < steps; ++t) lp += d->x[t * kSamples + lane];
  }
}

// The phases alternate every few thousand cycles, so the kernel's code is kept small:
// the activation is a template parameter, and loops are unrolled no further than
// their operands' latency asks for.
template <typename WT, int GW, bool RELU>
__global__ void __launch_bounds__(kThreads, 2) sampler_kernel(const SamplerArgs g) {
  using K = BlockSampler<WT, GW, RELU>;
  using R = Raw<WT>;
  extern __shared__ __align__(16) unsigned char smem[];
  LeafSum* Z = reinterpret_cast<LeafSum*>(smem + K::kOffZ);
  unsigned char* ring = smem + K::kOffR + uniform(threadIdx.x >> 5) * K::kRingBytes;
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
  float* T = reinterpret_cast<float*>(smem + K::kOffT);
  uint64_t* SP = reinterpret_cast<uint64_t*>(smem + K::kOffS);
  typename K::Post* P = reinterpret_cast<typename K::Post*>(smem + K::kOffP);
  Tables* tables = reinterpret_cast<Tables*>(smem + K::kOffTab);
  Drawn* drawn = reinterpret_cast<Drawn*>(smem + K::kOffDrawn);
  Block* next = reinterpret_cast<Block*>(smem + K::kOffNext);
  float* zero = reinterpret_cast<float*>(smem + K::kOffZero);
  float* A = reinterpret_cast<float*>(smem + K::kOffA);

  const int n = g.n, h = g.h, hp = g.hp;
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const int b0 = blockIdx.x * kSamples;
  const WT* wt = reinterpret_cast<const WT*>(g.wt);
  const WT* v = reinterpret_cast<const WT*>(g.v);
  const unsigned long long it = g.it_dev ? *g.it_dev : ((unsigned long long)g.it1 << 32 | g.it0);
  const uint32_t it0 = (uint32_t)it, it1 = (uint32_t)(it >> 32);

#pragma unroll 1
  for (int k = tid; k < hp + kChunk; k += kThreads) {
    const float x = k < h ? __ldg(g.b1 + k) : 0.0f;
#pragma unroll
    for (int s = 0; s < kSamples; ++s) A[(k / kChunk) * K::kStateChunk + s * kChunk + k % kChunk] = x;
  }
#pragma unroll 1
  for (int k = tid; k < K::kStateChunk; k += kThreads) zero[k] = 0.0f;
  for (int k = tid; k < kSteps * kSamples; k += kThreads) SP[k] = 0ull;
  __syncthreads();

  // The blocks go through a pipeline, so that each part stands once in the
  // code: turn i finds block i + 2, stages the tables of block i + 1, takes
  // block i through Z, the draws and U, and writes the outputs of block i - 1.
  Block b{0, 0, 0, 0}, nb{0, 0, 0, 0}, prev{0, 0, 0, 0};  // e0 == e1: none
  float lp = 0.0f;
  typename K::Stream st{};
#pragma unroll 1
  for (int turn = -2;; ++turn) {
    const int par = turn & 1, steps = b.e1 - b.e0;
    if (steps > 0) {
      // ----------------------------------------------------------- Z
      const int gs = b.grp % (4 * GW), pairs = kLeaves * b.grp;
#pragma unroll 1
      for (int task = warp; task < 4 * GW; task += kWarps) {
        const int vw = task >> 2, t0 = kTI * (task & 3);
        if (t0 >= steps) continue;
        if (GW > 2 && task != warp) {
          __syncwarp();
          K::start(st, ring_s, v, hp, b.e0 + t0, vw, lane, pairs);
        }
        K::z_task(st, ring, ring_s, hp, A, zero, t0, vw, lane, pairs, vw == gs >> 2, gs & 3, Z, T);
      }
    }
    __syncthreads();  // Z and T complete
    const bool more = nb.e1 > nb.e0;
    // requested before the draws: the weights of this warp's first round of U
    // (128 units, four consecutive ones per lane) and of its next Z task
    const bool u_todo = steps > 0 && more;
    const int k1 = kGroup * (b.grp + 1) + 128 * warp;
    const int ue = b.e0 + 1;  // W1 row of the block's first input
    constexpr int kAhead = sizeof(WT) == 2 ? kSteps : kSteps / 2;
    typename R::four w[kAhead];
    auto load = [&](int t, int k) {
      w[t % kAhead] = R::ld4(wt + (unsigned)((ue + t) * hp + k + 4 * lane), t < steps && k + 4 * lane < hp);
    };
    if (u_todo) {
#pragma unroll
      for (int t = 0; t < kAhead; ++t) load(t, k1);
      K::start(st, ring_s, v, hp, nb.e0 + kTI * (warp & 3), warp >> 2, lane,
               warp < 4 * GW && kTI * (warp & 3) < nb.e1 - nb.e0 ? kLeaves * nb.grp : 0);
    }
    if (warp >= kWarps - kSolvers) {
      if (steps > 0) {
        const int k0 = kGroup * b.grp, gs = b.grp % (4 * GW);
        K::solve(tables[par], drawn[par], Z, T, P, SP, A + k0 / kChunk * K::kStateChunk + k0 % kChunk, steps, gs >> 2,
                 warp - (kWarps - kSolvers), lane, h > n || (h == n && b.e0 == 0), nb.grp != b.grp);
      }
    } else if (warp == 2) {
      if (lane == 0) {
        Block x{0, 0, 0, 0};
        const int e = turn == -2 ? 0 : nb.e1;
        if (e < n && (turn == -2 || more)) x = next_block(e, n, h);
        next[par] = x;
      }
      if (prev.e1 > prev.e0) write_block(g, prev, drawn + (par ^ 1), b0, lane, lp);
    } else if (more && warp < 2) {
      stage_tables<WT>(tables + (par ^ 1), g, nb, b0, it0, it1, tid);
    }
    __syncthreads();  // the block's spins are drawn
    prev = b;
    b = nb;
    nb = next[par];
    nb = Block{uniform(nb.e0), uniform(nb.e1), uniform(nb.grp), 0};
    if (steps == 0 || !more) {
      if (turn >= 0 && steps == 0) break;  // the last block's outputs are written
      continue;
    }
    // ------------------------------------------------------------- U
#pragma unroll 1
    for (int k = k1; k < hp; k += 128 * kWarps) {
      const int kl = k + 4 * lane;
      const bool in = kl < hp;
      float* a = A + kl / kChunk * K::kStateChunk + kl % kChunk;
      uint64_t a0[kSamples], a1[kSamples];
#pragma unroll
      for (int s = 0; s < kSamples; ++s) {
        ulonglong2 x = make_ulonglong2(0ull, 0ull);
        if (in) x = *reinterpret_cast<const ulonglong2*>(a + s * kChunk);
        a0[s] = x.x, a1[s] = x.y;
      }
#pragma unroll
      for (int t = 0; t < kSteps; ++t) {
        if (t >= steps) break;
        const uint64_t u0 = R::lo(w[t % kAhead]), u1 = R::hi(w[t % kAhead]);
        const ulonglong2* sp = reinterpret_cast<const ulonglong2*>(SP + t * kSamples);
#pragma unroll
        for (int s = 0; s < kSamples; s += 2) {
          const ulonglong2 x = sp[s / 2];
          a0[s] = fma2(u0, x.x, a0[s]);
          a1[s] = fma2(u1, x.x, a1[s]);
          a0[s + 1] = fma2(u0, x.y, a0[s + 1]);
          a1[s + 1] = fma2(u1, x.y, a1[s + 1]);
        }
        // 16 rows in registers: the next round's; 8 (FP32): this round's second half
        if (kAhead == kSteps) load(t, k + 128 * kWarps);
        else if (t + kAhead < kSteps) load(t + kAhead, k);
      }
      if (kAhead < kSteps)
#pragma unroll
        for (int t = 0; t < kAhead; ++t) load(t, k + 128 * kWarps);
      if (in)
#pragma unroll
        for (int s = 0; s < kSamples; ++s)
          *reinterpret_cast<ulonglong2*>(a + s * kChunk) = make_ulonglong2(a0[s], a1[s]);
      if (kl < kGroup * b.grp && in)  // units of a group that has no steps of its own are complete now
#pragma unroll 1
        for (int i = 0; i < 2 * kSamples; ++i) {
          uint64_t* x = reinterpret_cast<uint64_t*>(a + (i >> 1) * kChunk) + (i & 1);
          *x = K::g1_pair(*x);
        }
    }
    // the next Z reads the units below group b.grp: group prev.grp (written
    // by the solver) and, if there are any, the groups completed just now
    if (b.grp > prev.grp + 1) __syncthreads();
  }
  if (warp == 2 && lane < kSamples && g.logp && b0 + lane < g.B) g.logp[b0 + lane] = lp;
}

template <typename WT, int GW>
cudaError_t launch_cfg(const SamplerArgs& a, cudaStream_t st) {
  const bool relu = a.act == VQMC_ACT_RELU;
  auto kern = relu ? sampler_kernel<WT, GW, true> : sampler_kernel<WT, GW, false>;
  const size_t smem = BlockSampler<WT, GW, true>::smem_bytes(a.hp);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(a.B + kSamples - 1) / kSamples, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

// The summation order (GW) by hp; `wide` asks for the order of hp > 2048 at any hp.
template <typename WT>
cudaError_t launch_sampler_wt(const SamplerArgs& a, cudaStream_t st) {
  if (!sampler_wt_supports<WT>(a.hp)) return cudaErrorNotSupported;
  if (a.wide || a.hp > 2048) return launch_cfg<WT, 4>(a, st);
  if (a.hp <= 64) return launch_cfg<WT, 1>(a, st);
  return launch_cfg<WT, 2>(a, st);
}

// Whether the CUDA-core samplers run models with hp padded hidden units: two
// stages of the step-at-a-time sampler's weight ring have to fit the shared
// memory.
template <typename WT>
bool sampler_wt_supports(int hp) {
  return hp <= (sizeof(WT) == 2 ? 5120 : 2816);
}

}  // namespace vqmc
