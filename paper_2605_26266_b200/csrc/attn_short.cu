// Corrected chunk attention for a few query rows over a long cache (small steps of a decoding reply, short chunks), and for
// problems that are small altogether.
//
// The tcgen05 kernel works on 256 query rows at a time; with 16 of them it spends its time on padding (scores,
// exponentials, and a dequantization into shared memory that 16 rows cannot pay for).  Here a CTA takes 16 rows of one
// (batch, head) and a range of the keys, each of its four warps takes every fourth step of 32 keys, and the packed codes
// go from global memory through registers straight into the B operands of mma.sync: the contraction over channels
// may run in any order, so a lane takes the D/4 channels whose codes it can load at once, and the output channels may be
// numbered in any order, so a lane takes D/8 consecutive ones of the values of its four keys.  Nothing is staged in shared
// memory but the query rows.
//
// Algorithm 1 as in the other kernels: rotated query in FP16, weights and values in BF16, FP32 sums, exact running maximum.
// Keys of at most two groups a head are not dequantized: their operand is the codes, and step, zero-point and the bias
// -(sigma/24) sum_j nu_j step_j^2 are applied to the sums in FP32 (code_steps).  With four groups that would be as many
// instructions as it saves: FP16 keys there, and the bias is one more MMA step (nu as a BF16 high and low part, step^2 is exact in
// BF16).  Ranges of one (batch, head) leave FP32 partial rows that a second kernel, or in small problems the cluster of their CTAs,
// merges in a fixed order.
//
// What bounds it: latency and instruction issue (two CTAs of four warps an SM, as registers allow), then HBM.  32 heads of 128 channels, 16
// rows, 16 384 tokens at 4 bits, group 128, where inputs change from call to call: 41.0 us with FP16 keys (36 warp instructions a
// key), 36.4 with products of codes, 35.4 with the rest as it is here (28 instructions): all query rows and the first keys loaded
// together, addresses from 32-bit slots, a current step's values on their way while its weights are computed, the merge's rows fetched with
// their maxima.  Two groups, on the same inputs again and again, 36.2 -> 32.1 us at 2 bits and 37.2 -> 34.2 at 4, four 35.9 -> 34.6 and
// 37.7 -> 36.2.  Three CTAs an SM: with spilled registers 25 % slower, with the query in shared memory and hardly any spills 4 to 9 %.  The four
// score tiles of a step one after the other instead of in turn: 7 %.
#include <cuda_fp16.h>

#include <cmath>
#include <type_traits>

#include "kvq_common.cuh"

namespace kvq {
namespace {

constexpr int kRows = 16;
constexpr int kWarps = 4;
constexpr int kStep = 32;            // keys a warp takes at a time
constexpr int kCtasPerSm = 2;      // up to 255 registers a thread, nothing spilled
constexpr int kCtasPerSm64 = 3;    // heads of 64 channels
constexpr float kLog2e = 1.4426950408889634f;

struct SParams {
  const uint16_t* q; const uint16_t* kc; const uint16_t* vc; uint16_t* out;
  int64_t q_sb, q_sh, q_st, kv_sb, kv_sh, kv_st, v_sb, v_sh, v_st, o_sb, o_sh, o_st;
  const uint8_t* codes[2]; const uint8_t* scale[2]; const uint16_t* zero[2];    // keys, values
  const int8_t* signs;
  int64_t capacity, cache_begin;
  int heads, rotate, correction;
  int m_tokens, n_cached, n_cur;
  int q_blocks, splits;
  int split_steps, split_rest;         // steps = splits * split_steps + split_rest
  float scale_log2, ax_coef;           // sigma * log2(e), -sigma / 24
  float q_limit;                       // products of codes: rotated query channels count as at most this, see launch_attn_short
  float* lse; float* cached_mass;
  float* partial;                      // splits > 1: one slot per CTA, see slot_floats
};

// Partial rows of a CTA: O[16][D] (not normalised), then m[16] (log2 units), l_cur[16], l_cached[16].
__host__ __device__ constexpr int slot_floats(int D) { return kRows * D + 64; }

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the first product of a chain
__device__ __forceinline__ void mma_f16_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
               : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
__device__ __forceinline__ uint32_t pack_f16_sat(float lo, float hi) {
  lo = fminf(fmaxf(lo, -65504.f), 65504.f);
  hi = fminf(fmaxf(hi, -65504.f), 65504.f);
  return (uint32_t)__half_as_ushort(__float2half_rn(lo)) | ((uint32_t)__half_as_ushort(__float2half_rn(hi)) << 16);
}
__device__ __forceinline__ uint32_t fma_f16x2(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t fma_bf16x2(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
// A zero-point within 2^96, so that its product with a step and a row's sum is a number also where it is none.
__device__ __forceinline__ uint32_t finite_bf16x2(uint32_t a) {
  uint32_t d;
  asm("{\n\t.reg .b32 t;\n\tmin.bf16x2 t, %1, %2;\n\tmax.bf16x2 %0, t, %3;\n\t}" : "=r"(d) : "r"(a), "r"(0x6F806F80u), "r"(0xEF80EF80u));
  return d;
}
// x shifted so that bit `from` lands on bit `to` (both known at compile time once unrolled)
__device__ __forceinline__ uint32_t move_bits(uint32_t x, int from, int to) { return from <= to ? x << (to - from) : x >> (from - to); }

// Shared memory of the CTAs of the cluster.
__device__ __forceinline__ uint32_t remote(uint32_t saddr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ float load_remote(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float4 load_remote4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// What a lane expands in one step where a head has four groups: of the keys 8 t + lane / 4 (t = 0 .. 3) the codes of its D/4 channels, of
// the values 2 (lane % 4) + {0, 1} + 8 t those of its D/8 channels; a lane's channels lie in one group, and of each key it has that one's
// step and zero-point.
template <int D, int BITS>
struct Keys {
  static constexpr int W = D / 4 * BITS / 32;
  uint32_t w[4][W], step[4], zero[4];                              // step byte, zero-point (BF16 bits)
};
template <int D, int BITS>
struct Values {
  static constexpr int B = D / 8 * BITS / 8;                       // bytes: 2, 4 or 8
  static constexpr int W = B < 4 ? 1 : B / 4;
  uint32_t w[8][W], step[8], zero[8];
};
// The same for at most two groups a head: products of keys are taken of the codes themselves, one group at a time, so a lane has D/4/G
// channels of each; steps and zero-points are those of keys 8 t + 2 (lane % 4) + {0, 1}, all in one load.
template <int D, int BITS, int GROUP>
struct CodeKeys {
  static constexpr int G = D / GROUP, C = GROUP / 4, W = C * BITS < 32 ? 1 : C * BITS / 32;      // channels and words of a group
  static constexpr int N = C * BITS < 32 ? C : 32 / BITS;                                         // codes of a word
  uint32_t w[4][G][W], step[4], zero[4][G];
};
template <int D, int BITS, int GROUP>
struct CodeValues {
  static constexpr int G = D / GROUP, B = D / 8 * BITS / 8, W = B < 4 ? 1 : B / 4;
  uint32_t w[8][W], step[4], zero[4][G];
};
// First slots of the two halves of a step (16 slots each never straddle the end of the slab, 32 may), in the slab of the head.
struct Step { uint32_t slot[2]; };
// The cache of one head.  32-bit slots (attn_short_supports), so that an address is one multiply-add.
struct Slab { const uint8_t* codes[2]; const uint8_t* scale[2]; const uint16_t* zero[2]; };

template <int BYTES, int W>
__device__ __forceinline__ void load_bytes(uint32_t (&w)[W], const void* src) {
  if constexpr (BYTES == 1) w[0] = load_coherent(static_cast<const uint8_t*>(src));
  else if constexpr (BYTES == 2) w[0] = load_coherent(static_cast<const uint16_t*>(src));
  else if constexpr (BYTES == 4) w[0] = load_coherent(static_cast<const uint32_t*>(src));
  else if constexpr (BYTES == 8) { const uint2 v = load_coherent(static_cast<const uint2*>(src)); w[0] = v.x; w[1] = v.y; }
  else { const uint4 v = load_coherent(static_cast<const uint4*>(src)); w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w; }
}
// Addresses: one per half of a step and array, the other keys at fixed offsets from it.
template <int D, int BITS, int GROUP>
__device__ __forceinline__ void load_keys(Keys<D, BITS>& r, const Slab& p, const Step& st, int g, int c) {
  constexpr int CB = D * BITS / 8, G = D / GROUP;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const uint8_t* src = p.codes[0] + (uint64_t)(st.slot[u] + g) * CB + c * (CB / 4);
    const uint64_t at = (uint64_t)(st.slot[u] + g) * G + c * (D / 4) / GROUP;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      load_bytes<CB / 4>(r.w[2 * u + t], src + 8 * t * CB);
      r.step[2 * u + t] = load_coherent(p.scale[0] + at + 8 * t * G);
      r.zero[2 * u + t] = load_coherent(p.zero[0] + at + 8 * t * G);
    }
  }
}
// Tokens past the window: step and zero-point 0, so that scores are finite (and masked later) and values exact zeros, whatever
// the bytes there are.  Done where the loads are used, not where they are issued: anything that touches a loaded register
// makes the warp wait for it, and with eight warps an SM little hides that.
template <int D, int BITS>
__device__ __forceinline__ void mask_keys(Keys<D, BITS>& r, int n_valid, int g) {
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if (8 * t + g >= n_valid) r.step[t] = r.zero[t] = 0u;
}
template <int D, int BITS>
__device__ __forceinline__ void mask_values(Values<D, BITS>& r, int n_valid, int c) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (2 * c + (i & 1) + 8 * (i >> 1) >= n_valid) r.step[i] = r.zero[i] = 0u;
}
template <int D, int BITS, int GROUP>
__device__ __forceinline__ void load_values(Values<D, BITS>& r, const Slab& p, const Step& st, int g, int c) {
  constexpr int CB = D * BITS / 8, G = D / GROUP;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const uint8_t* src = p.codes[1] + (uint64_t)(st.slot[u] + 2 * c) * CB + g * (CB / 8);
    const uint64_t at = (uint64_t)(st.slot[u] + 2 * c) * G + g * (D / 8) / GROUP;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int key = (i & 1) + 8 * (i >> 1);
      load_bytes<CB / 8>(r.w[4 * u + i], src + key * CB);
      r.step[4 * u + i] = load_coherent(p.scale[1] + at + key * G);
      r.zero[4 * u + i] = load_coherent(p.zero[1] + at + key * G);
    }
  }
}

template <int G>
__device__ __forceinline__ void load_constants(uint32_t& step, uint32_t (&zero)[G], const Slab& p, int which, uint32_t slot) {
  uint32_t s[1];
  load_bytes<2 * G>(s, p.scale[which] + (uint64_t)slot * G);
  step = s[0];
  load_bytes<4 * G>(zero, p.zero[which] + (uint64_t)slot * G);
}
template <int D, int BITS, int GROUP>
__device__ __forceinline__ void load_keys(CodeKeys<D, BITS, GROUP>& r, const Slab& p, const Step& st, int g, int c) {
  using K = CodeKeys<D, BITS, GROUP>;
  constexpr int CB = D * BITS / 8;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const uint8_t* src = p.codes[0] + (uint64_t)(st.slot[u] + g) * CB + c * (K::C * BITS / 8);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
#pragma unroll
      for (int gr = 0; gr < K::G; ++gr) load_bytes<K::C * BITS / 8>(r.w[2 * u + t][gr], src + 8 * t * CB + gr * (CB / K::G));
      load_constants<K::G>(r.step[2 * u + t], r.zero[2 * u + t], p, 0, st.slot[u] + 2 * c + 8 * t);
    }
  }
}
template <int D, int BITS, int GROUP>
__device__ __forceinline__ void load_values(CodeValues<D, BITS, GROUP>& r, const Slab& p, const Step& st, int g, int c) {
  using V = CodeValues<D, BITS, GROUP>;
  constexpr int CB = D * BITS / 8;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const uint8_t* src = p.codes[1] + (uint64_t)(st.slot[u] + 2 * c) * CB + g * V::B;
#pragma unroll
    for (int i = 0; i < 4; ++i) load_bytes<V::B>(r.w[4 * u + i], src + ((i & 1) + 8 * (i >> 1)) * CB);
#pragma unroll
    for (int t = 0; t < 2; ++t) load_constants<V::G>(r.step[2 * u + t], r.zero[2 * u + t], p, 1, st.slot[u] + 2 * c + 8 * t);
  }
}
// Steps and zero-points of a pair of keys, as they are loaded: key by key, its groups side by side.  Those of one group:
template <int G>
__device__ __forceinline__ float2 steps_of(uint32_t step, int gr) {
  const uint32_t bytes = G == 1 ? step : __byte_perm(step, 0u, gr == 0 ? 0x4420 : 0x4431);   // the group may be known at run time only
  uint32_t h;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h) : "h"((uint16_t)bytes));
  return __half22float2(*reinterpret_cast<__half2*>(&h));
}
template <int G>
__device__ __forceinline__ uint32_t zeros_of(const uint32_t (&zero)[G], int gr) {      // two BF16
  return G == 1 ? zero[0] : __byte_perm(zero[0], zero[G - 1], gr == 0 ? 0x5410 : 0x7632);
}
__device__ __forceinline__ float2 bf16x2_to_f32(uint32_t z) { return make_float2(__uint_as_float(z << 16), __uint_as_float(z & 0xFFFF0000u)); }
// 0 past the window, so that scores are finite and weights and values zeros whatever the bytes there are.
template <int G>
__device__ __forceinline__ void mask_pairs(uint32_t (&step)[4], uint32_t (&zero)[4][G], int n_valid, int c) {
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int left = n_valid - (8 * t + 2 * c);                    // valid keys of the pair
    if (left < 2) {
      step[t] &= left == 1 ? (G == 1 ? 0xFFu : 0xFFFFu) : 0u;
      zero[t][0] &= left == 1 ? (G == 1 ? 0xFFFFu : ~0u) : 0u;
      if (G == 2) zero[t][G - 1] = 0u;
    }
  }
}
// Where code i of a 16-bit half of a key's word is picked up as an FP16: shifted right by `shift` it starts at bit `bit` of the ten lowest,
// which hold two codes of 4 bits or five of 2, and the FP16's value is code * 2^(bit - 24), a subnormal and exact.
struct Place { int shift, bit; };
template <int BITS>
__host__ __device__ constexpr Place key_place(int i) {
  return BITS == 4 ? Place{i < 2 ? 0 : 8, 4 * (i & 1)} : Place{i < 5 ? 0 : 10, 2 * (i < 5 ? i : i - 5)};
}
// ANY_ZERO: groups whose constants are not exact (key_constant_exact, value_constant_exact) are expanded in FP32, as in the
// warp-level kernel, which served the calls this is set for before: heads of 64 channels, and chunks TMA cannot address.  A
// warp works in 16 bits, notes whether it met such a group, and then takes its steps once more in FP32.  Any branch inside a
// step costs every call: 16 rows over 8 192 tokens of 160 heads of 64 channels take 109 us without the second form, 115 us as
// here, 140 us with a branch at each step or an early exit.  Three CTAs an SM for 64 channels (two with the registers of the
// second form: 237 against 140 us for 32 such rows).
// CLUSTER: the splits of a unit are the CTAs of one cluster, which merge their rows themselves (a form of its own: its shared memory
// and registers cost the others 2 % of the smallest calls).
template <int D, int BITS, int GROUP, bool ANY_ZERO, bool CLUSTER>
__global__ void __launch_bounds__(kWarps * 32, D == 64 ? kCtasPerSm64 : kCtasPerSm) attn_short_kernel(const SParams p) {
  constexpr int LD = D + 8;                                        // padded rows of the query tiles
  constexpr int KS = D / 16;                                       // MMA steps over the channels
  constexpr int NT = D / 8;                                        // output tiles of 8 channels
  constexpr int G = D / GROUP;
  constexpr bool kCodes = G <= 2;                                  // products of the codes themselves
  using KeysT = typename std::conditional<kCodes, CodeKeys<D, BITS, GROUP>, Keys<D, BITS>>::type;
  using ValuesT = typename std::conditional<kCodes, CodeValues<D, BITS, GROUP>, Values<D, BITS>>::type;
  constexpr int kOStride = D + 4;
  // the query tiles are done with when the warps' outputs are exchanged
  __shared__ __align__(16) union {
    struct { uint16_t q[kRows * LD], qr[kRows * LD]; float nu[kRows * 4], sum[kRows * 2]; int shift[kRows]; } in;
    struct { float o[kWarps][kRows * kOStride]; } x;
  } sm;
  __shared__ float s_stat[kWarps][3][kRows];                       // m, l_cur, l_cached
  __shared__ __align__(16) float s_part[CLUSTER ? kRows * D + 3 * kRows : 4];      // this CTA's partial rows for the others of its cluster

  wait_for_previous_grid();                                        // the first kernel of a call: nothing global is touched before
  allow_next_grid();                                               // the merge kernel
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int unit = blockIdx.x / p.splits, split = blockIdx.x - unit * p.splits;
  const int bh = unit / p.q_blocks, b = bh / p.heads, h = bh - b * p.heads;
  const int row0 = (unit - bh * p.q_blocks) * kRows;

  // ---- this CTA's share of the steps: cached keys first, then the current chunk's; warp w takes every fourth ----
  const int n_cs = (p.n_cached + kStep - 1) / kStep;
  const int first = split * p.split_steps + split * p.split_rest / p.splits, last = (split + 1) * p.split_steps + (split + 1) * p.split_rest / p.splits;
  int st = first + warp;
  const int last_c = min(last, n_cs);
  Slab slab;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int64_t at = (int64_t)bh * p.capacity;
    slab.codes[i] = p.codes[i] + at * (D * BITS / 8); slab.scale[i] = p.scale[i] + at * G; slab.zero[i] = p.zero[i] + at * G;
  }
  auto step_of = [&](int i) {
    Step x;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t slot = (uint32_t)p.cache_begin + (uint32_t)i * kStep + 16 * u;
      x.slot[u] = slot - (slot >= (uint32_t)p.capacity ? (uint32_t)p.capacity : 0u);
    }
    return x;
  };
  KeysT keys;
  auto load_keys_of = [&](int i) { load_keys<D, BITS, GROUP>(keys, slab, step_of(i), g, c); };
  // ---- query rows: as they are, and rotated (FP16, in the order the expanded codes come in), per-group norms ----
  {
    constexpr int LPR = D / 8;                                     // lanes per row, 8 channels each
    const int ln = lane % LPR;
    constexpr int kAtOnce = kWarps * 32 / LPR;                     // rows
    uint4 raws[kRows / kAtOnce];                                   // all on their way together, and the first keys behind them
#pragma unroll
    for (int it = 0; it < kRows / kAtOnce; ++it) {
      const int row = row0 + it * kAtOnce + warp * (32 / LPR) + lane / LPR;
      raws[it] = make_uint4(0, 0, 0, 0);
      if (row < p.m_tokens) raws[it] = load_coherent(reinterpret_cast<const uint4*>(p.q + (int64_t)b * p.q_sb + (int64_t)h * p.q_sh + (int64_t)row * p.q_st) + ln);
    }
    if (st < last_c) load_keys_of(st);
#pragma unroll
    for (int it = 0; it < kRows / kAtOnce; ++it) {
      const int r = it * kAtOnce + warp * (32 / LPR) + lane / LPR;
      const uint4 raw = raws[it];
      *reinterpret_cast<uint4*>(sm.in.q + r * LD + ln * 8) = raw;
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
      float x[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = bf16_bits_to_f32(e & 1 ? w[e >> 1] >> 16 : w[e >> 1] & 0xFFFFu);
      if (p.rotate) {
        if (p.signs) {
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] *= (float)p.signs[ln * 8 + e];
        }
#pragma unroll
        for (int hh = 1; hh < 8; hh *= 2)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if ((i & hh) == 0) { const float u = x[i], v = x[i + hh]; x[i] = u + v; x[i + hh] = u - v; }
#pragma unroll
        for (int lm = 1; lm < LPR; lm *= 2)
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float o = __shfl_xor_sync(0xFFFFFFFFu, x[e], lm);
            x[e] = (ln & lm) ? (o - x[e]) : (x[e] + o);
          }
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] *= D == 64 ? 0.125f : 0.08838834764831845f;
      }
      float nu = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) nu += x[e] * x[e];
#pragma unroll
      for (int off = 1; off < GROUP / 8; off *= 2) nu += __shfl_xor_sync(0xFFFFFFFFu, nu, off);
      if (ln % (GROUP / 8) == 0) sm.in.nu[r * 4 + ln / (GROUP / 8)] = nu;
      // a word of N codes expands to the pairs (i, i + N / 2): that order, pair by pair
      if constexpr (kCodes) {
        // by groups, then lanes; times 2^shift, so that the row's largest value is at 2^14 (rows below 2^-10: 2^24), and 2^-bit of where
        // the channel's code lies
        constexpr int N = KeysT::N, C = KeysT::C;
        float top = 0.f, sum = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) { x[e] = fminf(fmaxf(x[e], -p.q_limit), p.q_limit); top = fmaxf(top, fabsf(x[e])); }
#pragma unroll
        for (int off = 1; off < LPR; off *= 2) top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, off));
        const int shift = min(24, 14 + 127 - (int)(__float_as_uint(top) >> 23));      // -100 at least, by q_limit
        const float scale = __uint_as_float((uint32_t)(127 + shift) << 23);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int ch = ln * 8 + e, i = ch % N;                   // N is 8 or 16, so i % (N / 2) is known at compile time up to where it matters
          const int bit = key_place<BITS>(N == 16 ? e : e & 3).bit;
          const __half hv = __float2half_rn(x[e] * scale * (1.0f / (1 << bit)));
          sum += __half2float(hv) * (float)(1 << bit);
          sm.in.qr[r * LD + ch / N * N + 2 * (i % (N / 2)) + i / (N / 2)] = __half_as_ushort(hv);
        }
#pragma unroll
        for (int off = 1; off < GROUP / 8; off *= 2) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
        if (ln % (GROUP / 8) == 0) sm.in.sum[r * 2 + ln / (GROUP / 8)] = sum * 0x1p-24f;
        if (ln == 0) sm.in.shift[r] = shift;
        static_assert(N == 8 || N == 16, "eight channels of a lane: whole words, or the same places in each half");
        static_assert(C % N == 0, "whole words");
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          constexpr int N = 32 / BITS;
          const int ch = ln * 8 + e, i = ch % N;
          sm.in.qr[r * LD + ch / N * N + 2 * (i % (N / 2)) + i / (N / 2)] = __half_as_ushort(__float2half_rn(fminf(fmaxf(x[e], -65504.f), 65504.f)));
        }
      }
    }
  }
  __syncthreads();
  uint32_t qf[KS][4];
  constexpr int KW = kCodes ? D / GROUP * CodeKeys<D, BITS, GROUP>::W : Keys<D, BITS>::W;      // words of a lane
  constexpr int N = kCodes ? CodeKeys<D, BITS, GROUP>::N : 32 / BITS, KPW = N / 4;              // codes and MMA steps of a word
  constexpr int KWG = kCodes ? KW / G : KW;                                                   // words of a group
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const int w = ks / KPW, col = ((w / KWG * 4 + c) * KWG + w % KWG) * N + 4 * (ks % KPW);
    const uint2 lo = *reinterpret_cast<const uint2*>(sm.in.qr + g * LD + col), hi = *reinterpret_cast<const uint2*>(sm.in.qr + (g + 8) * LD + col);
    qf[ks][0] = lo.x; qf[ks][1] = hi.x; qf[ks][2] = lo.y; qf[ks][3] = hi.y;
  }
  // At most two groups: scores are computed in units of 2^(24 - shift) of their row, s = sum over groups of step (sum_c q'_c code_c - zero
  // sum_c q'_c) + step^2 nu', in FP32 behind the products of q' and the codes themselves, so that expanding a key is an AND for two codes
  // and its constants are spent once per key.
  float row_unit[2], row_scale[2], row_sum[2][2], row_nu[2][2];    // of rows g, g + 8; of these by group
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = g + 8 * i, shift = kCodes ? sm.in.shift[r] : 24;
    row_unit[i] = __uint_as_float((uint32_t)(127 + shift - 24) << 23);
    row_scale[i] = p.scale_log2 * __uint_as_float((uint32_t)(127 + 24 - shift) << 23);
#pragma unroll
    for (int gr = 0; gr < 2; ++gr) {
      row_sum[i][gr] = kCodes && gr < G ? sm.in.sum[r * 2 + gr] : 0.f;
      row_nu[i][gr] = kCodes && gr < G && p.correction ? p.ax_coef * sm.in.nu[r * 4 + gr] * row_unit[i] : 0.f;
    }
  }
  // bias operand: columns 2 c, 2 c + 1 are the high and low part of lane c's group, with ANY_ZERO column 2 c + 8 is the rest
  // (the warp-level kernel applies the bias in FP32); one lane per group counts it
  uint32_t ax[4] = {0u, 0u, 0u, 0u};
  if (!kCodes && p.correction && c % (4 / G) == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float a = p.ax_coef * sm.in.nu[(g + 8 * i) * 4 + c / (4 / G)];
      const uint32_t hi = f32_to_bf16_bits(a);
      const float rest = a - bf16_bits_to_f32(hi);
      const uint32_t lo = f32_to_bf16_bits(rest);
      ax[i] = hi | (lo << 16);
      if (ANY_ZERO) ax[2 + i] = f32_to_bf16_bits(rest - bf16_bits_to_f32(lo));
    }
  }

  float acc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_cur[2] = {0.f, 0.f}, l_cac[2] = {0.f, 0.f};
  uint32_t pf[8];
  // online softmax over the 32 scores of a step (this lane: rows g, g + 8, keys 8 t + 2 c + {0, 1}); leaves the weights in their place
  // The maximum is kept as a raw score and subtracted before the scale: exact for the largest score however large it is (a key
  // masked with the lowest number), where the exact product of an FMA and a rounded maximum would differ.
  auto softmax_step = [&](float (&s)[4][4], int n_valid, float (&l)[2]) {
    if (n_valid < kStep) {
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (8 * t + 2 * c + (e & 1) >= n_valid) s[t][e] = -INFINITY;
    }
    float m_new[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      float mx = -INFINITY;
#pragma unroll
      for (int t = 0; t < 4; ++t) mx = fmaxf(mx, fmaxf(s[t][2 * r], s[t][2 * r + 1]));
      mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
      m_new[r] = fmaxf(m_run[r], mx);
    }
    if (__any_sync(0xFFFFFFFFu, m_new[0] > m_run[0] || m_new[1] > m_run[1])) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float f = ex2((m_run[r] - no_key_yet(m_new[r])) * row_scale[r]);
        l_cur[r] *= f; l_cac[r] *= f;
        m_run[r] = m_new[r];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          const float2 o = __fmul2_rn(make_float2(acc[j][2 * r], acc[j][2 * r + 1]), make_float2(f, f));
          acc[j][2 * r] = o.x; acc[j][2 * r + 1] = o.y;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float m = no_key_yet(m_run[r]);
      float2 sum;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float2 x = __fmul2_rn(__fadd2_rn(make_float2(s[t][2 * r], s[t][2 * r + 1]), make_float2(-m, -m)), make_float2(row_scale[r], row_scale[r]));
        const float2 e = make_float2(ex2(x.x), ex2(x.y));
        sum = t == 0 ? e : __fadd2_rn(sum, e);
        s[t][2 * r] = e.x; s[t][2 * r + 1] = e.y;
      }
      l[r] += sum.x + sum.y;
    }
  };

  auto pack_weights = [&](const float (&s)[4][4]) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
      for (int r = 0; r < 2; ++r) pf[2 * t + r] = pack_bf16(s[t][2 * r], s[t][2 * r + 1]);
  };

  // kFp32: (code - zero) * step in FP32, rounded once.  Otherwise in 16 bits; with ANY_ZERO false if some constants were not
  // exact (such steps are in the sums by then).
  auto cached_steps = [&](auto fp32, auto& keys) {
    constexpr bool kFp32 = decltype(fp32)::value;
    constexpr float kOff = BITS == 2 ? 4.f : 16.f;
    constexpr uint32_t kMask = (1u << BITS) - 1;
    bool exact = true;
#pragma unroll 1
    for (; st < last_c; st += kWarps) {
      Values<D, BITS> vals;                                        // on their way while the scores are computed
      load_values<D, BITS, GROUP>(vals, slab, step_of(st), g, c);
      float s[4][4];
      const int n_valid = p.n_cached - st * kStep;
      if (n_valid < kStep) mask_keys(keys, n_valid, g);
      // (OFF + code) * step - (OFF + zero) * step with OFF from the exponent bits OR-ed over the code, one FMA per pair
      uint32_t step2[4], off2[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float ds = e4m3_byte_to_f32(keys.step[t]), zs = bf16_bits_to_f32(keys.zero[t]);
        const float off = -(kOff + zs) * ds;
        step2[t] = pack_f16_sat(ds, ds); off2[t] = pack_f16_sat(off, off);
        if (ANY_ZERO && !kFp32) exact &= key_constant_exact<BITS>(zs);
        s[t][0] = s[t][1] = s[t][2] = s[t][3] = 0.f;
        if (p.correction) {
          const uint32_t b = pack_bf16(ds * ds, ds * ds);
          mma_bf16(s[t], ax[0], ax[1], ax[2], ax[3], b, ANY_ZERO ? b : 0u);
        }
      }
      // the four tiles in turn: a tile's products are one chain, and four chains hide each other's latency
#pragma unroll
      for (int wi = 0; wi < KW; ++wi)
#pragma unroll
        for (int j = 0; j < KPW; ++j)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            uint32_t bf[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              if constexpr (kFp32) {
                const float ds = e4m3_byte_to_f32(keys.step[t]), zs = bf16_bits_to_f32(keys.zero[t]);
                const uint32_t x = keys.w[t][wi] >> ((2 * j + i) * BITS);
                bf[i] = pack_f16_sat(((float)(x & kMask) - zs) * ds, ((float)((x >> 16) & kMask) - zs) * ds);
              } else {
                const uint32_t x = move_bits(keys.w[t][wi], (2 * j + i) * BITS, BITS == 2 ? 8 : 6);
                bf[i] = fma_f16x2(BITS == 2 ? (x & 0x03000300u) | 0x44004400u : (x & 0x03C003C0u) | 0x4C004C00u, step2[t], off2[t]);
              }
            }
            const uint32_t (&a)[4] = qf[wi * KPW + j];
            mma_f16(s[t], a[0], a[1], a[2], a[3], bf[0], bf[1]);
          }
      if (st + kWarps < last_c) load_keys_of(st + kWarps);
      softmax_step(s, n_valid, l_cac);
      pack_weights(s);
      if (n_valid < kStep) mask_values(vals, n_valid, c);
      // values, 16 keys at a time: keys 2 c, 2 c + 1 (and 8 more) side by side in the halves of a register, code i of both at once
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        uint32_t step2[2], off2[2];
        float ds[2][2], zs[2][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            ds[u][i] = e4m3_byte_to_f32(vals.step[4 * kk + 2 * u + i]);
            zs[u][i] = bf16_bits_to_f32(vals.zero[4 * kk + 2 * u + i]);
            if (ANY_ZERO && !kFp32) exact &= value_constant_exact<BITS>(zs[u][i]);
          }
          step2[u] = pack_bf16(ds[u][0], ds[u][1]);
          off2[u] = BITS == 2 ? pack_bf16(-(4.f + zs[u][0]) * ds[u][0], -(4.f + zs[u][1]) * ds[u][1]) : pack_bf16(16.f + zs[u][0], 16.f + zs[u][1]);
        }
        constexpr int kPer = 16 / BITS;                            // codes in half a word
#pragma unroll
        for (int hw = 0; hw < NT / kPer; ++hw) {
          uint32_t z[2];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            z[u] = __byte_perm(vals.w[4 * kk + 2 * u][hw / 2], vals.w[4 * kk + 2 * u + 1][hw / 2], hw & 1 ? 0x7632 : 0x5410);
#pragma unroll
          for (int i = 0; i < kPer; ++i) {
            uint32_t bf[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              if constexpr (kFp32) {
                const uint32_t x = z[u] >> (i * BITS);
                bf[u] = pack_bf16(((float)(x & kMask) - zs[u][0]) * ds[u][0], ((float)((x >> 16) & kMask) - zs[u][1]) * ds[u][1]);
              } else {
                const uint32_t x = move_bits(z[u], i * BITS, BITS == 2 ? 5 : 3);
                if constexpr (BITS == 2) bf[u] = fma_bf16x2((x & 0x00600060u) | 0x40804080u, step2[u], off2[u]);
                else bf[u] = mul_bf16x2(sub_bf16x2((x & 0x00780078u) | 0x41804180u, off2[u]), step2[u]);
              }
            }
            mma_bf16(acc[hw * kPer + i], pf[4 * kk], pf[4 * kk + 1], pf[4 * kk + 2], pf[4 * kk + 3], bf[0], bf[1]);
          }
        }
      }
    }
    return !ANY_ZERO || kFp32 || __all_sync(0xFFFFFFFFu, exact);
  };
  // The same for at most two groups a head, with products of the keys' codes.  (Weights times the steps of their values, rounded then, and
  // code - zero as the values' operand, 8 instructions of 10 a register, took 1 to 2 us of 34 less, but weights near 1 lose what they have
  // from lying at the top of their binade: errors up to 4 % larger.)
  auto code_steps = [&](auto fp32, auto& keys, auto& vals) {
    constexpr bool kFp32 = decltype(fp32)::value;
    constexpr uint32_t kMask = (1u << BITS) - 1;
    bool exact = true;
#pragma unroll 1
    for (; st < last_c; st += kWarps) {
      const Step here = step_of(st);
      load_values<D, BITS, GROUP>(vals, slab, here, g, c);         // on their way while the scores are computed
      float s[4][4], raw[4][4];                                    // FP32 form: keys themselves, one chain of products over both groups
      const int n_valid = p.n_cached - st * kStep;
#pragma unroll
      for (int gr = 0; gr < G; ++gr) {
        float key_step[4], key_zero[4];                            // of key 8 t + g, which the FP32 form expands with: the lane with c = g / 2 has it
        if constexpr (kFp32) {
          if (gr == 0 && n_valid < kStep) mask_pairs<G>(keys.step, keys.zero, n_valid, c);
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const uint32_t both = zeros_of<G>(keys.zero[t], gr);
            const float2 steps = steps_of<G>(keys.step[t], gr);
            const int from = (lane & ~3) | (g >> 1);
            const uint32_t zero = __shfl_sync(0xFFFFFFFFu, both, from);
            const float s0 = __shfl_sync(0xFFFFFFFFu, steps.x, from), s1 = __shfl_sync(0xFFFFFFFFu, steps.y, from);
            key_step[t] = g & 1 ? s1 : s0;
            key_zero[t] = __uint_as_float(g & 1 ? zero & 0xFFFF0000u : zero << 16);
          }
        }
        // the four tiles in turn: a tile's products are one chain, and four chains hide each other's latency
#pragma unroll
        for (int wi = 0; wi < KWG; ++wi) {
          uint32_t w[4];
#pragma unroll
          for (int t = 0; t < 4; ++t)                              // eight codes of 2 bits: four in each half
            w[t] = N * BITS < 32 ? __byte_perm(keys.w[t][gr][wi], 0u, 0x4140) : keys.w[t][gr][wi];
#pragma unroll
          for (int j = 0; j < KPW; ++j)
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              uint32_t bf[2];
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const Place at = key_place<BITS>(2 * j + i);
                if constexpr (kFp32) {                             // rounded to FP16
                  const uint32_t x = w[t] >> ((2 * j + i) * BITS);
                  bf[i] = pack_f16_sat(((float)(x & kMask) - key_zero[t]) * key_step[t], ((float)((x >> 16) & kMask) - key_zero[t]) * key_step[t]);
                } else {
                  bf[i] = (w[t] >> at.shift) & ((kMask | (kMask << 16)) << at.bit);
                }
              }
              const uint32_t (&a)[4] = qf[(gr * KWG + wi) * KPW + j];
              if (wi == 0 && j == 0 && (!kFp32 || gr == 0)) mma_f16_first(raw[t], a[0], a[1], a[2], a[3], bf[0], bf[1]);
              else mma_f16(raw[t], a[0], a[1], a[2], a[3], bf[0], bf[1]);
            }
        }
        if (!kFp32 && gr == 0 && n_valid < kStep) mask_pairs<G>(keys.step, keys.zero, n_valid, c);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const uint32_t zeros = zeros_of<G>(keys.zero[t], gr);
          // 128 channels: a key that was appended with an infinite channel takes all of the weight or none, as where FP16 keys saturate.  With
          // ANY_ZERO its scores are not numbers here, but such a zero-point is not exact either: the FP32 form follows, whose keys saturate
          const float2 step = steps_of<G>(keys.step[t], gr), zero = bf16x2_to_f32(D == 128 && !ANY_ZERO ? finite_bf16x2(zeros) : zeros);
          const float2 off = __fmul2_rn(step, make_float2(-zero.x, -zero.y)), sq = __fmul2_rn(step, step);
          if (ANY_ZERO && !kFp32) exact &= key_constant_exact<BITS>(zero.x) && key_constant_exact<BITS>(zero.y);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            // the bias last: beside the two sums that cancel it would lose bits
            const float2 x = make_float2(raw[t][2 * r], raw[t][2 * r + 1]);
            const float2 sum = make_float2(s[t][2 * r], s[t][2 * r + 1]), nu = make_float2(row_nu[r][gr], row_nu[r][gr]);
            float2 v;
            if constexpr (kFp32) {
              v = gr == 0 ? __fmul2_rn(sq, nu) : __ffma2_rn(sq, nu, sum);
              if (gr == G - 1) v = __ffma2_rn(x, make_float2(0x1p-24f, 0x1p-24f), v);
            } else {
              v = __ffma2_rn(sq, nu, __ffma2_rn(x, step, __fmul2_rn(off, make_float2(row_sum[r][gr], row_sum[r][gr]))));
              if (gr > 0) v = __fadd2_rn(v, sum);
            }
            s[t][2 * r] = v.x; s[t][2 * r + 1] = v.y;
          }
        }
      }
      if (st + kWarps < last_c) load_keys_of(st + kWarps);
      if (n_valid < kStep) mask_pairs<G>(vals.step, vals.zero, n_valid, c);
      softmax_step(s, n_valid, l_cac);
      pack_weights(s);
      // values, 16 keys at a time: keys 2 c, 2 c + 1 (and 8 more) side by side in the halves of a register, code i of both at once
      const int gr = g * (D / 8) / GROUP;                          // of this lane's channels
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        uint32_t step2[2], off2[2];
        float2 ds[2], zs[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t z = zeros_of<G>(vals.zero[2 * kk + u], gr);
          ds[u] = steps_of<G>(vals.step[2 * kk + u], gr);
          zs[u] = bf16x2_to_f32(z);
          if (ANY_ZERO && !kFp32) exact &= value_constant_exact<BITS>(zs[u].x) && value_constant_exact<BITS>(zs[u].y);
          step2[u] = pack_bf16(ds[u].x, ds[u].y);
          // 2 bits: -(4 + zero) * step, 4 bits: 16 + zero
          const float2 off = __fadd2_rn(zs[u], make_float2(BITS == 2 ? 4.f : 16.f, BITS == 2 ? 4.f : 16.f));
          off2[u] = BITS == 2 ? pack_bf16(-off.x * ds[u].x, -off.y * ds[u].y) : pack_bf16(off.x, off.y);
        }
        constexpr int kPer = 16 / BITS;                            // codes in half a word
#pragma unroll
        for (int hw = 0; hw < NT / kPer; ++hw) {
          uint32_t z[2];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            z[u] = __byte_perm(vals.w[4 * kk + 2 * u][hw / 2], vals.w[4 * kk + 2 * u + 1][hw / 2], hw & 1 ? 0x7632 : 0x5410);
#pragma unroll
          for (int i = 0; i < kPer; ++i) {
            uint32_t bf[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              if constexpr (kFp32) {
                const uint32_t x = z[u] >> (i * BITS);
                bf[u] = pack_bf16(((float)(x & kMask) - zs[u].x) * ds[u].x, ((float)((x >> 16) & kMask) - zs[u].y) * ds[u].y);
              } else {
                const uint32_t x = move_bits(z[u], i * BITS, BITS == 2 ? 5 : 3);
                if constexpr (BITS == 2) bf[u] = fma_bf16x2((x & 0x00600060u) | 0x40804080u, step2[u], off2[u]);
                else bf[u] = mul_bf16x2(sub_bf16x2((x & 0x00780078u) | 0x41804180u, off2[u]), step2[u]);
              }
            }
            mma_bf16(acc[hw * kPer + i], pf[4 * kk], pf[4 * kk + 1], pf[4 * kk + 2], pf[4 * kk + 3], bf[0], bf[1]);
          }
        }
      }
    }
    return !ANY_ZERO || kFp32 || __all_sync(0xFFFFFFFFu, exact);
  };
  auto cached = [&](auto fp32) { ValuesT vals; if constexpr (kCodes) return code_steps(fp32, keys, vals); else return cached_steps(fp32, keys); };
  if (!cached(std::false_type{})) {                                // the warp's steps once more
    st = first + warp;
    if (st < last_c) load_keys_of(st);
    if constexpr (kCodes) {                                        // with keys themselves: the query without the powers of two of the codes' places
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t up = (uint32_t)(15 + key_place<BITS>(2 * (ks % KPW) + (i >> 1)).bit) << 10;
          qf[ks][i] = fma_f16x2(qf[ks][i], up | (up << 16), 0u);
        }
    }
    m_run[0] = m_run[1] = -INFINITY;
    l_cur[0] = l_cur[1] = l_cac[0] = l_cac[1] = 0.f;
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    cached(std::true_type{});
  }
  // ---- current chunk: unrotated query, BF16 keys and values, no bias ----
  // 64 channels: keys of the next step and values of this one are on their way while scores and weights are computed; 128, which have no
  // registers for that: values while the weights are.
  uint4 kx[4][D / 32];
  auto load_current_keys = [&](int i) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int key = min((i - n_cs) * kStep + 8 * t + g, p.n_cur - 1);
      const uint4* src = reinterpret_cast<const uint4*>(p.kc + (int64_t)b * p.kv_sb + (int64_t)h * p.kv_sh + (int64_t)key * p.kv_st + c * (D / 4));
#pragma unroll
      for (int j = 0; j < D / 32; ++j) kx[t][j] = load_coherent(src + j);
    }
  };
  constexpr bool kAhead = D == 64;
  if (kAhead && st < last) load_current_keys(st);
#pragma unroll 1
  for (; st < last; st += kWarps) {
    const int k0 = (st - n_cs) * kStep, nv = p.n_cur - k0;
    uint4 vx[D / 64][8];                                           // of keys 2 c + {0, 1} + 8 u, 8 of the lane's channels at a time
    const uint16_t* vbase = p.vc + (int64_t)b * p.v_sb + (int64_t)h * p.v_sh + g * (D / 8);
    auto load_current_values = [&]() {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int key = 2 * c + (u & 1) + 8 * (u >> 1);
#pragma unroll
        for (int i = 0; i < D / 64; ++i)
          vx[i][u] = key < nv ? load_coherent(reinterpret_cast<const uint4*>(vbase + (int64_t)(k0 + key) * p.v_st) + i) : make_uint4(0, 0, 0, 0);
      }
    };
    if (kAhead) load_current_values();
    else load_current_keys(st);
    float s[4][4];
#pragma unroll
    for (int t = 0; t < 4; ++t) s[t][0] = s[t][1] = s[t][2] = s[t][3] = 0.f;
#pragma unroll
    for (int i = 0; i < D / 32; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int col = c * (D / 4) + 8 * i + 4 * j;
        const uint2 lo = *reinterpret_cast<const uint2*>(sm.in.q + g * LD + col), hi = *reinterpret_cast<const uint2*>(sm.in.q + (g + 8) * LD + col);
#pragma unroll
        for (int t = 0; t < 4; ++t) mma_bf16(s[t], lo.x, hi.x, lo.y, hi.y, j ? kx[t][i].z : kx[t][i].x, j ? kx[t][i].w : kx[t][i].y);
      }
    if (!kAhead) load_current_values();
    else if (st + kWarps < last) load_current_keys(st + kWarps);
    if constexpr (kCodes) {
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[t][e] *= row_unit[e >> 1];
    }
    softmax_step(s, nv, l_cur);
    pack_weights(s);
#pragma unroll
    for (int kk = 0; kk < 2; ++kk)
#pragma unroll
      for (int i = 0; i < D / 64; ++i) {
        const uint4 (&v)[8] = vx[i];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint32_t sel = e & 1 ? 0x7632 : 0x5410;
          auto word = [&](const uint4& x) { return (e >> 1) == 0 ? x.x : (e >> 1) == 1 ? x.y : (e >> 1) == 2 ? x.z : x.w; };
          mma_bf16(acc[8 * i + e], pf[4 * kk], pf[4 * kk + 1], pf[4 * kk + 2], pf[4 * kk + 3],
                   __byte_perm(word(v[4 * kk]), word(v[4 * kk + 1]), sel), __byte_perm(word(v[4 * kk + 2]), word(v[4 * kk + 3]), sel));
        }
      }
  }

  // ---- the four warps' partial rows ----
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    l_cur[r] += __shfl_xor_sync(0xFFFFFFFFu, l_cur[r], 1);
    l_cur[r] += __shfl_xor_sync(0xFFFFFFFFu, l_cur[r], 2);
    l_cac[r] += __shfl_xor_sync(0xFFFFFFFFu, l_cac[r], 1);
    l_cac[r] += __shfl_xor_sync(0xFFFFFFFFu, l_cac[r], 2);
    if (c == 0) { s_stat[warp][0][g + 8 * r] = m_run[r] * row_scale[r]; s_stat[warp][1][g + 8 * r] = l_cur[r]; s_stat[warp][2][g + 8 * r] = l_cac[r]; }
  }
  __syncthreads();                                                 // also: the query tiles are free
#pragma unroll
  for (int j = 0; j < NT; j += 4)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      *reinterpret_cast<float4*>(&sm.x.o[warp][(g + 8 * (e >> 1)) * kOStride + (2 * c + (e & 1)) * (D / 8) + j]) =
          make_float4(acc[j][e], acc[j + 1][e], acc[j + 2][e], acc[j + 3][e]);
  __syncthreads();
  constexpr int kPerRow = kWarps * 32 / kRows;                     // threads per row
  const int r = threadIdx.x / kPerRow, t8 = threadIdx.x % kPerRow, row = row0 + r;
  if (!CLUSTER && row >= p.m_tokens) return;
  float m = -INFINITY, f[kWarps], lc = 0.f, la = 0.f;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) m = fmaxf(m, s_stat[w][0][r]);
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {                               // a warp without keys has m = -inf: weight 0
    f[w] = ex2(s_stat[w][0][r] - no_key_yet(m));
    lc += f[w] * s_stat[w][1][r]; la += f[w] * s_stat[w][2][r];
  }
  const float l = lc + la, inv = 1.0f / l;
  float* slot = p.partial + (size_t)blockIdx.x * slot_floats(D);
  uint16_t* dst = p.out + (int64_t)b * p.o_sb + (int64_t)h * p.o_sh + (int64_t)row * p.o_st;
#pragma unroll
  for (int i = 0; i < D / 4; i += kPerRow) {
    const int ch = (i + t8) * 4;
    float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float4 v = *reinterpret_cast<const float4*>(&sm.x.o[w][r * kOStride + ch]);
      o[0] += f[w] * v.x; o[1] += f[w] * v.y; o[2] += f[w] * v.z; o[3] += f[w] * v.w;
    }
    if constexpr (CLUSTER) *reinterpret_cast<float4*>(s_part + r * D + ch) = make_float4(o[0], o[1], o[2], o[3]);
    else if (p.splits > 1) *reinterpret_cast<float4*>(slot + r * D + ch) = make_float4(o[0], o[1], o[2], o[3]);
    else *reinterpret_cast<uint2*>(dst + ch) = make_uint2(pack_bf16(o[0] * inv, o[1] * inv), pack_bf16(o[2] * inv, o[3] * inv));
  }
  if constexpr (CLUSTER) {
    // Every CTA has left its rows in its shared memory; CTA c combines rows c, c + splits, ... of all of them, in the order of the
    // splits, a thread four channels of a row.
    if (t8 == 0) { s_part[kRows * D + r] = m; s_part[kRows * D + kRows + r] = lc; s_part[kRows * D + 2 * kRows + r] = la; }
    __syncwarp();
    cluster_sync();
    constexpr int kThreadsPerRow = D / 4, kRowsAtOnce = kWarps * 32 / kThreadsPerRow;
    const int mine = threadIdx.x % kThreadsPerRow;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(s_part);
    for (int rr = split + threadIdx.x / kThreadsPerRow * p.splits; rr < kRows && row0 + rr < p.m_tokens; rr += kRowsAtOnce * p.splits) {
      float top = -INFINITY;
      for (int c2 = 0; c2 < p.splits; ++c2) top = fmaxf(top, load_remote(remote(base, c2) + (kRows * D + rr) * 4));
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
      float sc = 0.f, sa = 0.f;
#pragma unroll 4
      for (int c2 = 0; c2 < p.splits; ++c2) {
        const uint32_t at = remote(base, c2);
        const float w = ex2(load_remote(at + (kRows * D + rr) * 4) - no_key_yet(top));
        sc += w * load_remote(at + (kRows * D + kRows + rr) * 4); sa += w * load_remote(at + (kRows * D + 2 * kRows + rr) * 4);
        const float4 v = load_remote4(at + (rr * D + mine * 4) * 4);
        a.x += w * v.x; a.y += w * v.y; a.z += w * v.z; a.w += w * v.w;
      }
      const float ls = sc + sa, is = 1.0f / ls;
      *reinterpret_cast<uint2*>(p.out + (int64_t)b * p.o_sb + (int64_t)h * p.o_sh + (int64_t)(row0 + rr) * p.o_st + mine * 4) =
          make_uint2(pack_bf16(a.x * is, a.y * is), pack_bf16(a.z * is, a.w * is));
      if (mine == 0) {
        const int64_t idx = (int64_t)bh * p.m_tokens + row0 + rr;
        if (p.lse) p.lse[idx] = (top + log2f(ls)) * 0.6931471805599453f;
        if (p.cached_mass) p.cached_mass[idx] = sa * is;
      }
    }
    __syncwarp();
    cluster_sync();                                                // the others may still read this CTA's rows
  } else if (t8 == 0) {
    if (p.splits > 1) {
      float* stat = slot + kRows * D;
      stat[r] = m; stat[16 + r] = lc; stat[32 + r] = la;
    } else {
      const int64_t idx = (int64_t)bh * p.m_tokens + row;
      if (p.lse) p.lse[idx] = (m + log2f(l)) * 0.6931471805599453f;
      if (p.cached_mass) p.cached_mass[idx] = la * inv;
    }
  }
}

// Combines the partial rows of a unit's splits in a fixed order: a block per row, warp w taking every fourth split, its
// lanes the channels, so that the loads of a row are all in flight together.
template <int D>
__global__ void __launch_bounds__(kWarps * 32) attn_short_merge_kernel(const SParams p) {
  constexpr int E = D / 32;                                        // channels of a lane
  wait_for_previous_grid();                                        // the partial rows
  const int unit = blockIdx.x / kRows, r = blockIdx.x % kRows, bh = unit / p.q_blocks, b = bh / p.heads, h = bh - b * p.heads;
  const int row = (unit - bh * p.q_blocks) * kRows + r;
  if (row >= p.m_tokens) return;                                   // the whole block
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ float s_o[kWarps][D], s_l[kWarps][2];
  const float* slots = p.partial + (size_t)unit * p.splits * slot_floats(D);
  auto load_row = [&](int s, float (&v)[E], float& lc, float& la) {
    const float* sl = slots + (size_t)s * slot_floats(D);
    lc = sl[kRows * D + 16 + r]; la = sl[kRows * D + 32 + r];
    if constexpr (E == 4) { const float4 u = *reinterpret_cast<const float4*>(sl + r * D + lane * E); v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w; }
    else { const float2 u = *reinterpret_cast<const float2*>(sl + r * D + lane * E); v[0] = u.x; v[1] = u.y; }
  };
  auto maximum_of = [&](int s) { return slots[(size_t)s * slot_floats(D) + kRows * D + r]; };
  // the warp's first splits, mostly all, come in one trip to memory with the maxima
  constexpr int kFirst = 4;
  float v[kFirst][E], fm[kFirst], fc[kFirst], fa[kFirst];
#pragma unroll
  for (int i = 0; i < kFirst; ++i) {
    const int s = warp + kWarps * i;
    fm[i] = -INFINITY; fc[i] = fa[i] = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) v[i][e] = 0.f;
    if (s < p.splits) { fm[i] = maximum_of(s); load_row(s, v[i], fc[i], fa[i]); }
  }
  float m = -INFINITY;
  for (int s = lane; s < p.splits; s += 32) m = fmaxf(m, maximum_of(s));
#pragma unroll
  for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
  float o[E] = {}, lc = 0.f, la = 0.f;
#pragma unroll
  for (int i = 0; i < kFirst; ++i) {
    if (warp + kWarps * i >= p.splits) break;                      // the whole warp
    const float f = ex2(fm[i] - m);
    lc += f * fc[i]; la += f * fa[i];
#pragma unroll
    for (int e = 0; e < E; ++e) o[e] += f * v[i][e];
  }
#pragma unroll 4
  for (int s = warp + kWarps * kFirst; s < p.splits; s += kWarps) {
    float w[E], wc, wa;
    load_row(s, w, wc, wa);
    const float f = ex2(maximum_of(s) - m);
    lc += f * wc; la += f * wa;
#pragma unroll
    for (int e = 0; e < E; ++e) o[e] += f * w[e];
  }
#pragma unroll
  for (int e = 0; e < E; ++e) s_o[warp][lane * E + e] = o[e];
  if (lane == 0) { s_l[warp][0] = lc; s_l[warp][1] = la; }
  __syncthreads();
  lc = la = 0.f;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) { lc += s_l[w][0]; la += s_l[w][1]; }
  const float l = lc + la, inv = 1.0f / l;
  if (threadIdx.x < D) {
    float x = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) x += s_o[w][threadIdx.x];
    p.out[(int64_t)b * p.o_sb + (int64_t)h * p.o_sh + (int64_t)row * p.o_st + threadIdx.x] = (uint16_t)f32_to_bf16_bits(x * inv);
  }
  if (threadIdx.x == 0) {
    const int64_t idx = (int64_t)bh * p.m_tokens + row;
    if (p.lse) p.lse[idx] = (m + log2f(l)) * 0.6931471805599453f;
    if (p.cached_mass) p.cached_mass[idx] = la * inv;
  }
}

int64_t resident_ctas() {
  int sms = 0;
  if (device_sm_count(&sms) != KVQ_OK) sms = 148;                  // sizes only: the launch itself fails loudly
  return (int64_t)sms * kCtasPerSm;
}

// Units (batch*head, 16 rows) and into how many ranges the keys of each are cut: as many as let every CTA be resident at
// once, but no range below 2 steps a warp, nor more than the merge can have in flight.
struct Plan { int64_t q_blocks, units; int splits; bool clusters; };
Plan plan(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur) {
  Plan pl;
  pl.q_blocks = (m_tokens + kRows - 1) / kRows;
  pl.units = (int64_t)d->batch * d->heads * pl.q_blocks;
  const int64_t steps = (cache_len + kStep - 1) / kStep + (n_cur + kStep - 1) / kStep;
  int64_t s = resident_ctas() / pl.units;
  if (s > steps / (2 * kWarps)) s = steps / (2 * kWarps);
  if (s > 128) s = 128;
  pl.splits = (int)(s < 1 ? 1 : s);
  // The splits of a unit as one cluster (eight CTAs is what every device places) that merges its rows in shared memory: no
  // second launch and no trip through global memory.  Up to three fifths of the CTAs that run at once: clusters leave gaps in the
  // processors of a GPC, and with a full device some wait for others to end (64 heads of 64 x 16 rows over 16 384 keys 51 -> 65 us,
  // 48 heads of 128 over 2 048 14 -> 21 us).  Device time, us: 2 heads of 64 x 256 rows over 1 024 keys 8.5 -> 7.2, 1 to 32 heads of
  // 64 6 to 17 % less, of 128 3 to 7 %; eight CTAs at 128 channels -4 to +5 %, so not those.
  pl.clusters = pl.splits > 1 && pl.splits <= (d->head_dim == 64 ? 8 : 6) && pl.units * pl.splits * 5 <= resident_ctas() * 3;
  return pl;
}

template <int D, int BITS, int GROUP>
int launch(const SParams& p, const Plan& pl, bool any_zero, cudaStream_t st) {
  const dim3 grid((unsigned)(pl.units * pl.splits));
  if (pl.clusters && (D == 64 || !any_zero))
    return launch_after(true, pl.splits, grid, dim3(kWarps * 32), 0, st, attn_short_kernel<D, BITS, GROUP, D == 64, true>, p);
  const auto kern = D == 64 || any_zero ? attn_short_kernel<D, BITS, GROUP, true, false> : attn_short_kernel<D, BITS, GROUP, D == 64, false>;
  const int r = launch_after(true, 1, grid, dim3(kWarps * 32), 0, st, kern, p);
  if (r != KVQ_OK) return r;
  if (pl.splits > 1)
    return launch_after(true, 1, dim3((unsigned)(pl.units * kRows)), dim3(kWarps * 32), 0, st, attn_short_merge_kernel<D>, p);
  return KVQ_OK;
}

}  // namespace

bool attn_short_supports(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur, uint32_t flags) {
  if ((flags & KVQ_KERNEL_MASK) != KVQ_KERNEL_AUTO || (flags & KVQ_CORRECTION_EXACT) || (d->flags & KVQ_K_PER_CHANNEL) || m_tokens < 1 || d->capacity > INT32_MAX)
    return false;
  // Every 16 rows expand the codes again, 256 rows of the tcgen05 kernel once; but that kernel has a pre-pass, a larger
  // prologue and a larger merge.  Both kernels as they are, device time of a call among others on the same inputs (us here /
  // there, 128 channels, 2 bits, group 64): one block of rows is faster here (32 heads over 16 384 keys 32 / 58, over none 4.7 / 5.9).
  // The lines for two blocks (4 200 (head, 128-key tile) pairs), three (1 200) and four (400), as long as all CTAs run at once, were
  // drawn for FP16 keys and launches that did not overlap.  With both kernels as they are they meet near 2 500, 900 and 480: two blocks, 32
  // heads, 23 / 25 at 1 056, 36 / 38 at 2 112, 50 / 47 at 3 104, 63 / 58 at 4 128; three 19 / 20 at 544, 22 / 24 at 800, 27 / 25 at 1 056; four
  // 17 / 20 at 320, 21 / 20 at 480, 24 / 20 at 576.  Between there and the lines a call takes up to a tenth longer here.  64 channels, where the other kernel has more fixed cost to each tile, stay ahead further: two blocks 24 / 40 at 2 080, 41 / 62 at
  // 4 128, 100 / 136 at 10 400 of 160 heads.
  const int64_t blocks = (m_tokens + kRows - 1) / kRows;
  if (blocks == 1) return true;
  // Small problems, whatever the rows: all CTAs run at once and each has few steps, while the other kernel is a chain of three
  // launches with a prologue of microseconds each.  Counted in steps of 32 keys over all blocks of 16 rows (as above; 4 bits
  // alike): 64 channels 2 heads x 256 rows over 1 024 keys, 1 280 steps, 6.9 / 14.6; at 4 352 steps 11.6 / 18; at 5 120 12 /
  // 15; at 8 192 the other kernel's units of 256 rows decide, 14 / 27 with one (16 000 keys), 14 / 22 with two, 15.6 / 15.8 with sixteen (8
  // heads x 512 rows over 512 keys; 2 x 1 000 over 1 024 17 / 15, the worst met); at 10 240 18.6 / 17.1 (8 x 512 over 768), 18.3 / 17.0 (4 x 1 024
  // over 256), 15.8 / 20.1 (16 x 320 over 700).  128 channels at 1 040 steps 10 / 17, at 4 160 15 / 19, at 4 608 15 / 19 to 17.4 / 17.8, at 6 400 20.5 / 18.2
  // (16 heads x 128 rows) and 18.6 / 18.4 (16 x 96); over an empty cache, where the other kernel is one launch as well, 5.5 / 6.6 for 16 heads x
  // 128 rows and 7.7 / 6.7 for 32.  For 128 channels only up to the 128 rows of one query tile of the other kernel, half of which idles there.
  const int64_t bh = (int64_t)d->batch * d->heads;
  const int64_t steps = (cache_len + kStep - 1) / kStep + (n_cur + kStep - 1) / kStep;
  // 64 channels, more heads than processors, one tile of rows, current keys within half a tile, no cache: a CTA of the tcgen05 kernel
  // would take several units of half a tile each.  Two of some 28 000 random calls of all kernels ended in a launch failure, two of the
  // three of this form and none of the 17 with more keys; the cause was not found by reading, and 300 such calls with every role's
  // steps recorded ran through.  Two gaps found since, one-CTA exits that left commits unwaited for and allocations by a warp that might not be
  // whole, are closed; that they were the cause is not known.  Such calls do not run there: 172 heads x 111 rows over 5 keys 11 us here (148
  // heads x 111 rows, which do, 7).
  if (d->head_dim == 64 && cache_len == 0 && n_cur <= 64 && blocks <= 8 && bh > resident_ctas() / kCtasPerSm) return true;
  if (d->head_dim == 64) {
    if (bh * blocks <= resident_ctas() / kCtasPerSm * kCtasPerSm64 && bh * blocks * steps <= 8192) return true;
  } else if (blocks <= 8 && bh * blocks <= resident_ctas() && bh * blocks * steps <= 4608) {
    return true;
  }
  const int64_t pairs = bh * ((cache_len + 127) / 128 + (n_cur + 127) / 128);
  if (d->head_dim == 64) return (blocks == 2 && pairs <= 16384) || (blocks == 3 && pairs <= 1200) || (blocks == 4 && pairs <= 600);
  return bh * blocks <= resident_ctas() && ((blocks == 2 && pairs <= 4200) || (blocks == 3 && pairs <= 1200) || (blocks == 4 && pairs <= 400));
}

size_t attn_short_workspace_bytes(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur) {
  const Plan pl = plan(d, cache_len, m_tokens, n_cur);
  return pl.splits > 1 ? ((size_t)pl.units * pl.splits * slot_floats(d->head_dim) * sizeof(float) + 255) / 256 * 256 : 0;
}

int attn_short_kernel_launches(const kvq_cache_desc* d, int64_t cache_len, int64_t m_tokens, int64_t n_cur) {
  const Plan pl = plan(d, cache_len, m_tokens, n_cur);
  return pl.splits > 1 && !pl.clusters ? 2 : 1;
}

int launch_attn_short(const AttnArgs& a) {
  const kvq_cache_desc* d = a.desc;
  const Plan pl = plan(d, a.cache_len, a.m_tokens, a.n_cur);
  SParams p;
  p.q = static_cast<const uint16_t*>(a.q); p.kc = static_cast<const uint16_t*>(a.k_cur);
  p.vc = static_cast<const uint16_t*>(a.v_cur); p.out = static_cast<uint16_t*>(a.out);
  p.q_sb = a.qs.b; p.q_sh = a.qs.h; p.q_st = a.qs.t;
  p.kv_sb = a.kvs.b; p.kv_sh = a.kvs.h; p.kv_st = a.kvs.t;
  p.v_sb = a.vs.b; p.v_sh = a.vs.h; p.v_st = a.vs.t;
  p.o_sb = a.os.b; p.o_sh = a.os.h; p.o_st = a.os.t;
  p.codes[0] = static_cast<const uint8_t*>(d->k_codes); p.codes[1] = static_cast<const uint8_t*>(d->v_codes);
  p.scale[0] = static_cast<const uint8_t*>(d->k_scale); p.scale[1] = static_cast<const uint8_t*>(d->v_scale);
  p.zero[0] = static_cast<const uint16_t*>(d->k_zero); p.zero[1] = static_cast<const uint16_t*>(d->v_zero);
  p.signs = d->signs;
  p.capacity = d->capacity; p.cache_begin = a.cache_begin % d->capacity;
  p.heads = d->heads; p.rotate = (d->flags & KVQ_ROTATE_K) ? 1 : 0;
  p.correction = (a.flags & KVQ_CORRECTION_ON) ? 1 : 0;
  p.m_tokens = (int)a.m_tokens; p.n_cached = (int)a.cache_len; p.n_cur = (int)a.n_cur;
  p.q_blocks = (int)pl.q_blocks; p.splits = pl.splits;
  const int steps = (int)((a.cache_len + kStep - 1) / kStep + (a.n_cur + kStep - 1) / kStep);
  p.split_steps = steps / pl.splits; p.split_rest = steps % pl.splits;
  p.scale_log2 = a.softmax_scale * kLog2e;
  p.ax_coef = -a.softmax_scale / 24.0f;
  // Scores in log2 units have to stay below 2^128, and a row's scale with them, or the parts of a row cannot be merged.  With keys in FP16's
  // range they are below 2^23 times scale_log2 and this limit.  Ordinary scales leave queries room up to some 2^106; from scales of 2^87 on
  // channels are held where FP16 keys and queries held them.  (2^115 at most: the unit of a row, 2^(shift - 24), is a normal number.)
  p.q_limit = ldexpf(65504.f, min(99, max(0, 87 - ilogbf(p.scale_log2))));
  p.lse = a.lse; p.cached_mass = a.cached_mass;
  p.partial = static_cast<float*>(a.workspace);
  const bool any_zero = !attn_tcgen05_addressable(a);
#define KVQ_SHORT(D_, B_, G_) if (d->head_dim == D_ && d->bits == B_ && d->group == G_) return launch<D_, B_, G_>(p, pl, any_zero, a.stream);
  KVQ_SHORT(128, 2, 32) KVQ_SHORT(128, 2, 64) KVQ_SHORT(128, 2, 128) KVQ_SHORT(128, 4, 32) KVQ_SHORT(128, 4, 64) KVQ_SHORT(128, 4, 128)
  KVQ_SHORT(64, 2, 32) KVQ_SHORT(64, 2, 64) KVQ_SHORT(64, 4, 32) KVQ_SHORT(64, 4, 64)
#undef KVQ_SHORT
  return KVQ_ERR_UNSUPPORTED;
}

}  // namespace kvq
