// Quantize-append kernel: Hadamard rotation (keys), group-wise asymmetric round-to-nearest
// quantization (Eq. (1)), bit packing and coalesced append of one finished chunk's K and V.
//
// Four lanes own one token-head vector (lane lv holds channels [lv*EPL, (lv+1)*EPL), EPL = head_dim/4), so a warp
// works on eight consecutive tokens, each warp by itself: a lane's codes fill a whole store (32 to 128 bits), the stores
// of a warp are contiguous, and nothing is staged in shared memory.  The Walsh-Hadamard butterfly runs its first
// log2(EPL) stages inside a lane and the remaining two across lanes with shuffles; group minimum/maximum are shuffle
// reductions over the lanes of a group.  Every add, subtract, multiply and divide is a single IEEE binary32 operation
// (no contraction), so the stored codes, steps and zero-points are reproducible bit for bit.
//
// By its bytes the kernel would be HBM-bound on its BF16 input.  It was bound by instruction issue, because the
// bit-exact contract fixes the operations; with half the instructions (0.54 issued a cycle) its warps wait for their loads
// and their own chains.  A lane keeps its values as pairs (channel i, channel i + EPL/2) in
// the two halves of 64-bit registers and does everything but the last in-lane butterfly stage and the minimum/maximum
// with the packed instructions (add/mul/fma.rn.f32x2: two IEEE operations each), and adds the zero-point, clamps and packs
// the codes two at a time as 16-bit integers.  Measured at 24 heads x 4680 tokens, 128 channels, 2 bits, group 64
// (66 MB), the same inputs again and again: 36.9 us with one IEEE operation per instruction, persistent blocks and a staged tile;
// 23.6 us without either (19.6 us where launches overlap, see launch_after, and 18.0 us as here, with 32 bytes a load; 20.2 us, 3.27
// TB/s, where inputs change from call to call),
// 3 % more with eight lanes per vector (shorter lanes repeat the per-group work more often); two
// tokens in flight per lane and persistent warps with a prefetch: 26.6 us (fewer warps fit).
#include <math_constants.h>

#include "kvq_common.cuh"

namespace kvq {
namespace {

constexpr int kWarps = 4;
constexpr int kLanes = 4;          // lanes per token-head vector
constexpr int kTokPerWarp = 32 / kLanes;
constexpr int kCtasPerSm = 5;      // register budget: up to 96 a thread, nothing spilled

struct QParams {
  const uint16_t* k; const uint16_t* v;
  int64_t sb, sh, st;          // element strides of k and v
  int64_t n_tokens, cache_len, capacity;
  int heads, group, rotate, rotate_v;
  int in_32;                   // tokens of k and v start on 32-byte boundaries
  int skip_k;                  // per-channel keys: the keys are written by quantize_k_per_channel_kernel instead
  const int8_t* signs;
  uint8_t* codes[2]; uint8_t* scale[2]; uint16_t* zero[2];
};

// The EPL values of a lane as pairs: v[i] = (x[i], x[i + EPL/2]).
template <int EPL>
struct Pairs { float2 v[EPL / 2]; };

// y = c_d * H_d * x for a vector spread over four lanes (lane lv holds channels [lv*EPL, (lv+1)*EPL)):
// stages h = 1, 2, 4, ... in that order, one rounding per operation.  The first log2(EPL) stages stay in
// registers (the last of them, h = EPL/2, inside the pairs), the last two exchange with lanes lv^1 and lv^2.
template <int EPL>
__device__ __forceinline__ void hadamard(Pairs<EPL>& x, int lv, float c_d) {
  constexpr int HP = EPL / 2;
  const float2 minus = make_float2(-1.0f, -1.0f);
#pragma unroll
  for (int h = 1; h < HP; h *= 2) {
#pragma unroll
    for (int i = 0; i < HP; ++i) {
      if ((i & h) == 0) {
        const float2 a = x.v[i], b = x.v[i + h];
        x.v[i] = __fadd2_rn(a, b);
        x.v[i + h] = __ffma2_rn(b, minus, a);          // a - b, rounded once
      }
    }
  }
#pragma unroll
  for (int i = 0; i < HP; ++i) {
    const float a = x.v[i].x, b = x.v[i].y;
    x.v[i] = make_float2(__fadd_rn(a, b), __fsub_rn(a, b));
  }
#pragma unroll
  for (int lm = 1; lm < kLanes; lm *= 2) {
    const float sg = (lv & lm) ? -1.0f : 1.0f;       // upper partner: other - own; fma(+-1, own, other) rounds once
    const float2 sg2 = make_float2(sg, sg);
#pragma unroll
    for (int i = 0; i < HP; ++i) {
      const float2 o = make_float2(__shfl_xor_sync(0xFFFFFFFFu, x.v[i].x, lm), __shfl_xor_sync(0xFFFFFFFFu, x.v[i].y, lm));
      x.v[i] = __ffma2_rn(sg2, x.v[i], o);
    }
  }
#pragma unroll
  for (int i = 0; i < HP; ++i) x.v[i] = __fmul2_rn(x.v[i], make_float2(c_d, c_d));
}

// What a lane stores for its vector: its codes (32 to 128 bits) and its group's step and zero-point.
template <int EPL, int BITS>
struct Quantized { uint32_t w[EPL * BITS / 32]; uint32_t sbyte, zbits; };

// Quantizes the vector held by kLanes lanes.  The per-group work (range, step, zero-point) is shared by the GROUP/EPL
// lanes of a group.
template <int EPL, int BITS, int GROUP>
__device__ __forceinline__ Quantized<EPL, BITS> quantize(const Pairs<EPL>& x) {
  constexpr float L = (float)((1 << BITS) - 1);
  constexpr int HP = EPL / 2;
  constexpr int lanes_per_group = GROUP / EPL;

  float mn = fminf(x.v[0].x, x.v[0].y), mx = fmaxf(x.v[0].x, x.v[0].y);
  float seen = mx;                                    // NaN if any value is (a maximum that propagates it)
#pragma unroll
  for (int i = 1; i < HP; ++i) {                      // three-input minimum and maximum: one instruction per two elements
    asm("min.f32 %0, %1, %2, %3;" : "=f"(mn) : "f"(mn), "f"(x.v[i].x), "f"(x.v[i].y));
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(seen) : "f"(seen), "f"(x.v[i].x), "f"(x.v[i].y));
  }
  if (!__any_sync(0xFFFFFFFFu, !(seen == seen) || !(x.v[0].x == x.v[0].x) || !(x.v[0].y == x.v[0].y))) {
    mx = seen;
  } else {                                            // some value of the warp is NaN: the maximum of the others
    seen = CUDART_NAN_F;
#pragma unroll
    for (int i = 1; i < HP; ++i) mx = fmaxf(mx, fmaxf(x.v[i].x, x.v[i].y));
  }
#pragma unroll
  for (int off = 1; off < lanes_per_group; off *= 2) {
    mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, off));
    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
  }
  // Divisions.  x / b as q0 = x*r, rem = fma(-q0, b, x), q = fma(rem, r, q0) with r = RN(1/b) (Markstein's correction
  // of an approximate quotient by its exact remainder) is the correctly rounded quotient for every divisor used here
  // (3, 15 and the 126 positive E4M3 values: checked against IEEE division for all 2^23 significands of x) as long
  // as nothing overflows.  A quotient too small to be computed exactly needs no care: it is below 2^-40 and rounds to
  // the integer 0, or to the step floor 2^-9, either way.  Rounding to an integer is q + 1.5*2^23 (the FMA pipe instead
  // of the quarter-rate conversion unit), whose low mantissa bits are rint(q) while |q| < 2^22.  Vectors with magnitudes
  // or quotients beyond those bounds take IEEE division and rintf instead, the whole warp together.
  const float range = __fsub_rn(mx, mn);
  const float amax = fmaxf(fabsf(range), fmaxf(fabsf(mn), fabsf(mx)));
  auto fast_div = [](float a, float b, float r) {
    const float q0 = __fmul_rn(a, r);
    return __fmaf_rn(__fmaf_rn(-q0, b, a), r, q0);
  };
  const bool big = !(amax < 0x1p60f);
  float step = fast_div(range, L, (BITS == 2) ? __uint_as_float(0x3EAAAAABu) : __uint_as_float(0x3D888889u));
  if (big) step = __fdiv_rn(range, L);
  uint32_t sbyte = f32_to_e4m3_byte(step);
  if (sbyte == 0) sbyte = 1;                       // floor at the smallest subnormal 2^-9
  const float ds = e4m3_byte_to_f32(sbyte);
  const float rds = __frcp_rn(ds);
  const float reach = __fmul_rn(amax, rds);        // bound of |x / step|
  constexpr float kRound = 12582912.f;             // 1.5 * 2^23
  Quantized<EPL, BITS> out;
  out.sbyte = sbyte;
  constexpr int F = HP < 16 / BITS ? HP : 16 / BITS;   // codes in a 16-bit field
  constexpr int kAcc = HP / F;                         // words of two such fields
  uint32_t acc[kAcc];
  if (!__any_sync(0xFFFFFFFFu, big || !(reach < 0x1p13f) || !(seen == seen))) {
    // rint(x / step) is the low half of the bits of x / step + 1.5*2^23, a 16-bit integer here, as is the zero-point:
    // two values at a time, one byte permutation gathers the halves, one instruction adds the zero-point and clamps to
    // [0, L], one integer multiply-add puts the codes into the 16-bit fields of channels [.., EPL/2) and [EPL/2, ..).
    const float z = __fsub_rn(0.0f, __fsub_rn(__fadd_rn(fast_div(mn, ds, rds), kRound), kRound));
    out.zbits = f32_to_bf16_bits(z);
    const uint32_t zi = __float_as_uint(__fadd_rn(bf16_bits_to_f32(out.zbits), kRound));
    const uint32_t z2 = __byte_perm(zi, zi, 0x1010);
    const float2 r2 = make_float2(rds, rds), nds2 = make_float2(-ds, -ds), round2 = make_float2(kRound, kRound);
#pragma unroll
    for (int i = 0; i < HP; ++i) {
      const float2 q0 = __fmul2_rn(x.v[i], r2);
      const float2 q = __ffma2_rn(__ffma2_rn(q0, nds2, x.v[i]), r2, q0);
      const float2 n = __fadd2_rn(q, round2);
      const uint32_t n2 = __byte_perm(__float_as_uint(n.x), __float_as_uint(n.y), 0x5410);
      const uint32_t c2 = __viaddmin_s16x2_relu(n2, z2, BITS == 2 ? 0x00030003u : 0x000F000Fu);
      const int k = i / F, pos = (i % F) * BITS;
      acc[k] = pos == 0 ? c2 : c2 * (1u << pos) + acc[k];
    }
  } else {
    const bool slow = __any_sync(0xFFFFFFFFu, big || !(reach < 0x1p21f));
    const float z = __fsub_rn(0.0f, slow ? rintf(__fdiv_rn(mn, ds)) : __fsub_rn(__fadd_rn(fast_div(mn, ds, rds), kRound), kRound));
    out.zbits = f32_to_bf16_bits(z);
    const float zs = bf16_bits_to_f32(out.zbits);
    const float kz = __fsub_rn(kRound, zs);
    const bool low = __any_sync(0xFFFFFFFFu, zs != z);
    // the lower clamp first where it is needed: fminf / fmaxf return the other operand for a NaN
    auto code = [&](float v) {
      float c;
      if (slow) c = fmaxf(__fadd_rn(rintf(__fdiv_rn(v, ds)), zs), 0.0f);
      else { c = __fsub_rn(__fadd_rn(fast_div(v, ds, rds), kRound), kz); if (low) c = fmaxf(c, 0.0f); }
      return (uint32_t)fminf(c, L);
    };
#pragma unroll
    for (int k = 0; k < kAcc; ++k) acc[k] = 0;
#pragma unroll
    for (int i = 0; i < HP; ++i) {
      const int k = i / F, pos = (i % F) * BITS;
      acc[k] |= (code(x.v[i].x) | (code(x.v[i].y) << 16)) << pos;
    }
  }
  static_assert(F * BITS == 16, "full fields");
  if constexpr (kAcc == 1) out.w[0] = acc[0];
  else {
#pragma unroll
    for (int k = 0; k < kAcc; k += 2) {            // low fields: the first half of the lane's channels
      out.w[k / 2] = __byte_perm(acc[k], acc[k + 1], 0x5410);
      out.w[(kAcc + k) / 2] = __byte_perm(acc[k], acc[k + 1], 0x7632);
    }
  }
  return out;
}

template <int EPL>
struct RawVec { uint4 r[EPL / 8]; };      // EPL BF16 values of one lane

template <int EPL>
__device__ __forceinline__ void load_raw_vec(RawVec<EPL>& v, const uint16_t* p, int lv) {
#pragma unroll
  for (int i = 0; i < EPL / 8; ++i) v.r[i] = load_coherent(reinterpret_cast<const uint4*>(p) + lv * (EPL / 8) + i);
}
// The same with 32 bytes an instruction, from rows on 32-byte boundaries: a lane's channels are 64 bytes (32), so that an instruction of
// 16 bytes a lane meets every line of eight tokens and takes a quarter of it.  24 heads x 4680 tokens, 128 channels, the same again and
// again: 19.6 -> 18.0 us.
template <int EPL>
__device__ __forceinline__ void load_raw_vec_32(RawVec<EPL>& v, const uint16_t* p, int lv) {
#pragma unroll
  for (int i = 0; i < EPL / 8; i += 2) {
    uint4 &a = v.r[i], &b = v.r[i + 1];
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p + lv * EPL + i * 8) : "memory");
  }
}
template <int EPL>
__device__ __forceinline__ void decode_vec(const RawVec<EPL>& v, Pairs<EPL>& x) {
#pragma unroll
  for (int i = 0; i < EPL / 8; ++i) {
    const uint32_t w[4] = {v.r[i].x, v.r[i].y, v.r[i].z, v.r[i].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int c = 8 * i + 2 * e + j;                      // channel of the lane
        const float f = j ? __uint_as_float(w[e] & 0xFFFF0000u) : __uint_as_float(w[e] << 16);
        if (c < EPL / 2) x.v[c].x = f; else x.v[c - EPL / 2].y = f;
      }
    }
  }
}
template <int EPL>
__device__ __forceinline__ void apply_signs(Pairs<EPL>& x, const int8_t* signs) {
#pragma unroll
  for (int i = 0; i < EPL / 2; ++i)
    x.v[i] = __fmul2_rn(x.v[i], make_float2((float)signs[i], (float)signs[i + EPL / 2]));
}

// A warp takes eight consecutive tokens of one (batch, head), four lanes per token.  Blocks are not persistent: enough
// warps are resident to hide the loads, and the hardware deals the blocks out evenly.
template <int D, int BITS, int GROUP>
__global__ void __launch_bounds__(kWarps * 32, kCtasPerSm) quantize_append_kernel(QParams p) {
  constexpr int EPL = D / kLanes;
  constexpr int CB = D * BITS / 8;
  constexpr int G = D / GROUP;
  constexpr int lanes_per_group = GROUP / EPL;
  const int lane = threadIdx.x & 31, lv = lane & (kLanes - 1);
  const float c_d = (D == 64) ? 0.125f : __uint_as_float(0x3DB504F3u);
  const int bh = blockIdx.y, b = bh / p.heads, h = bh - b * p.heads;
  const int64_t t0 = ((int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5)) * kTokPerWarp;
  if (t0 >= p.n_tokens) return;                               // the whole warp
  const int64_t t = t0 + lane / kLanes;
  const bool valid = t < p.n_tokens;
  wait_for_previous_grid();                                   // whatever wrote the chunk or still reads the cache
  allow_next_grid();
  RawVec<EPL> raw[2];
  if (valid) {
    const int64_t off = (int64_t)b * p.sb + (int64_t)h * p.sh + t * p.st;
    if (p.in_32) {
      if (!p.skip_k) load_raw_vec_32<EPL>(raw[0], p.k + off, lv);
      load_raw_vec_32<EPL>(raw[1], p.v + off, lv);
    } else {
      if (!p.skip_k) load_raw_vec<EPL>(raw[0], p.k + off, lv);
      load_raw_vec<EPL>(raw[1], p.v + off, lv);
    }
  } else {                                                    // tokens past the end quantize zeros, never stored
#pragma unroll
    for (int w = 0; w < 2; ++w)
#pragma unroll
      for (int i = 0; i < EPL / 8; ++i) raw[w].r[i] = make_uint4(0, 0, 0, 0);
  }
  // slot of this token, modulo the capacity (p.cache_len is already reduced, and an append brings at most
  // `capacity` tokens, so one subtraction does)
  int64_t slot = p.cache_len + t;
  if (slot >= p.capacity) slot -= p.capacity;
  const int64_t at = (int64_t)bh * p.capacity + slot;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    if (w == 0 && p.skip_k) continue;
    Pairs<EPL> x;
    decode_vec<EPL>(raw[w], x);
    if (w == 0 ? p.rotate : p.rotate_v) {                     // values are stored rotated with KVQ_ROTATE_V only
      if (p.signs) apply_signs<EPL>(x, p.signs + lv * EPL);
      hadamard<EPL>(x, lv, c_d);
    }
    const Quantized<EPL, BITS> q = quantize<EPL, BITS, GROUP>(x);
    if (valid) {
      uint8_t* dst = p.codes[w] + at * CB + lv * (EPL * BITS / 8);
      if constexpr (EPL * BITS == 32) *reinterpret_cast<uint32_t*>(dst) = q.w[0];
      else if constexpr (EPL * BITS == 64) *reinterpret_cast<uint2*>(dst) = make_uint2(q.w[0], q.w[1]);
      else *reinterpret_cast<uint4*>(dst) = make_uint4(q.w[0], q.w[1], q.w[2], q.w[3]);
      if ((lv % lanes_per_group) == 0) {
        p.scale[w][at * G + lv / lanes_per_group] = (uint8_t)q.sbyte;
        p.zero[w][at * G + lv / lanes_per_group] = (uint16_t)q.zbits;
      }
    }
  }
}

// ---- per-channel keys (App. E) -----------------------------------------------------------------------
// One CTA per (batch*head, block of g = p.group tokens): the g x D block is rotated into shared memory (FP32), then
// thread c owns channel c: minimum and maximum over the block's tokens, step and zero-point with the arithmetic of
// Eq. (1) in plain IEEE operations (range / L, E4M3 rounding, -rint(min / step), rint(y / step) + zero, clamp),
// codes as bytes in shared memory; finally the codes of a token are packed 32 / BITS per word along the channels,
// the layout every other kernel reads.  An analysis option: nothing here is tuned.
template <int D, int BITS>
__global__ void __launch_bounds__(256) quantize_k_per_channel_kernel(QParams p) {
  constexpr int EPL = D / kLanes;
  constexpr int CB = D * BITS / 8;
  constexpr int LDY = D + 1;
  extern __shared__ __align__(16) uint8_t pc_smem[];
  const int g = p.group;
  float* y = reinterpret_cast<float*>(pc_smem);                       // [g][D + 1]
  uint8_t* codes = pc_smem + (size_t)g * LDY * sizeof(float);          // [g][D]
  const int bh = blockIdx.y, b = bh / p.heads, h = bh - b * p.heads;
  const int64_t t0 = (int64_t)blockIdx.x * g;                          // first token of the block within the chunk
  const int lane = threadIdx.x & 31, lv = lane & (kLanes - 1);
  const float c_d = (D == 64) ? 0.125f : __uint_as_float(0x3DB504F3u);
  for (int r = threadIdx.x / kLanes; r < g; r += 256 / kLanes) {       // kLanes lanes per token
    RawVec<EPL> raw;
    load_raw_vec<EPL>(raw, p.k + (int64_t)b * p.sb + (int64_t)h * p.sh + (t0 + r) * p.st, lv);
    Pairs<EPL> x;
    decode_vec<EPL>(raw, x);
    if (p.rotate) {
      if (p.signs) apply_signs<EPL>(x, p.signs + lv * EPL);
      hadamard<EPL>(x, lv, c_d);
    }
#pragma unroll
    for (int i = 0; i < EPL / 2; ++i) {
      y[r * LDY + lv * EPL + i] = x.v[i].x;
      y[r * LDY + lv * EPL + i + EPL / 2] = x.v[i].y;
    }
  }
  __syncthreads();
  int64_t slot0 = p.cache_len + t0;                                    // whole blocks never straddle the end of a ring
  slot0 %= p.capacity;
  if (threadIdx.x < D) {
    const int c = threadIdx.x;
    constexpr float L = (float)((1 << BITS) - 1);
    float mn = y[c], mx = y[c];
    for (int t = 1; t < g; ++t) { mn = fminf(mn, y[t * LDY + c]); mx = fmaxf(mx, y[t * LDY + c]); }
    const float step = __fdiv_rn(__fsub_rn(mx, mn), L);
    uint32_t sbyte = f32_to_e4m3_byte(step);
    if (sbyte == 0) sbyte = 1;                                         // floor at the smallest subnormal 2^-9
    const float ds = e4m3_byte_to_f32(sbyte);
    const float z = __fsub_rn(0.0f, rintf(__fdiv_rn(mn, ds)));
    const uint32_t zbits = f32_to_bf16_bits(z);
    const float zs = bf16_bits_to_f32(zbits);
    for (int t = 0; t < g; ++t) {
      const float cc = fminf(fmaxf(__fadd_rn(rintf(__fdiv_rn(y[t * LDY + c], ds)), zs), 0.0f), L);
      codes[t * D + c] = (uint8_t)cc;
    }
    const int64_t blk = (int64_t)bh * (p.capacity / g) + slot0 / g;
    p.scale[0][blk * D + c] = (uint8_t)sbyte;
    p.zero[0][blk * D + c] = (uint16_t)zbits;
  }
  __syncthreads();
  constexpr int kPer = 32 / BITS;                                      // codes per 32-bit word
  uint32_t* out = reinterpret_cast<uint32_t*>(p.codes[0] + ((int64_t)bh * p.capacity + slot0) * CB);
  for (int i = threadIdx.x; i < g * (CB / 4); i += 256) {
    const int t = i / (CB / 4), w = i - t * (CB / 4);
    uint32_t word = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) word |= (uint32_t)codes[t * D + w * kPer + j] << (j * BITS);
    out[i] = word;                                                     // tokens of a block are contiguous: out[t * CB/4 + w]
  }
}

template <int BITS>
__global__ void unpack_codes_kernel(const uint8_t* codes, uint8_t* out, int64_t capacity, int64_t begin,
                                    int64_t n, int D, int64_t total) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int c = (int)(i % D);
  const int64_t t = (i / D) % n;
  const int64_t bh = i / ((int64_t)D * n);
  const int CB = D * BITS / 8;
  int64_t slot = begin + t;                                   // begin is already reduced modulo the capacity
  if (slot >= capacity) slot -= capacity;
  const uint8_t byte = codes[(bh * capacity + slot) * CB + (c * BITS) / 8];
  out[i] = (byte >> ((c * BITS) % 8)) & ((1 << BITS) - 1);
}

}  // namespace

int launch_quantize_append(const kvq_cache_desc* d, int64_t cache_len, const void* k, const void* v,
                           kvq_strides kv, int64_t n_tokens, cudaStream_t st) {
  QParams p;
  p.k = static_cast<const uint16_t*>(k);
  p.v = static_cast<const uint16_t*>(v);
  p.sb = kv.b; p.sh = kv.h; p.st = kv.t;
  p.n_tokens = n_tokens; p.cache_len = cache_len % d->capacity; p.capacity = d->capacity;
  p.heads = d->heads; p.group = d->group; p.rotate = (d->flags & KVQ_ROTATE_K) ? 1 : 0;
  p.rotate_v = (d->flags & KVQ_ROTATE_V) ? 1 : 0;
  p.skip_k = (d->flags & KVQ_K_PER_CHANNEL) ? 1 : 0;
  p.signs = d->signs;
  p.in_32 = ((reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v)) % 32 == 0 && kv.b % 16 == 0 && kv.h % 16 == 0 && kv.t % 16 == 0) ? 1 : 0;
  p.codes[0] = static_cast<uint8_t*>(d->k_codes); p.codes[1] = static_cast<uint8_t*>(d->v_codes);
  p.scale[0] = static_cast<uint8_t*>(d->k_scale); p.scale[1] = static_cast<uint8_t*>(d->v_scale);
  p.zero[0] = static_cast<uint16_t*>(d->k_zero); p.zero[1] = static_cast<uint16_t*>(d->v_zero);
  const int64_t blocks = (n_tokens + kWarps * kTokPerWarp - 1) / (kWarps * kTokPerWarp);
  if (blocks > 0x7FFFFFFFLL) return KVQ_ERR_UNSUPPORTED;
  const dim3 grid((unsigned)blocks, (unsigned)(d->batch * d->heads)), block(kWarps * 32);
#define KVQ_QA(D_, B_, G_) if (d->head_dim == D_ && d->bits == B_ && d->group == G_) { err = launch_after(true, 1, grid, block, 0, st, quantize_append_kernel<D_, B_, G_>, p); launched = true; }
  bool launched = false;
  int err = KVQ_OK;
  KVQ_QA(128, 2, 32) KVQ_QA(128, 2, 64) KVQ_QA(128, 2, 128) KVQ_QA(128, 4, 32) KVQ_QA(128, 4, 64) KVQ_QA(128, 4, 128)
  KVQ_QA(64, 2, 32) KVQ_QA(64, 2, 64) KVQ_QA(64, 4, 32) KVQ_QA(64, 4, 64)
#undef KVQ_QA
  if (!launched) return KVQ_ERR_UNSUPPORTED;
  if (err != KVQ_OK) return err;
  if (p.skip_k) {                                     // per-channel keys: one CTA per block of `group` tokens
    const int64_t bh = (int64_t)d->batch * d->heads;
    if (bh > 65535) return KVQ_ERR_UNSUPPORTED;
    const dim3 pgrid((unsigned)(n_tokens / d->group), (unsigned)bh);
    const size_t smem = (size_t)d->group * (d->head_dim + 1) * sizeof(float) + (size_t)d->group * d->head_dim;
#define KVQ_PC(D_, B_) if (d->head_dim == D_ && d->bits == B_) { \
      KVQ_CUDA_TRY(cudaFuncSetAttribute(quantize_k_per_channel_kernel<D_, B_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
      quantize_k_per_channel_kernel<D_, B_><<<pgrid, 256, smem, st>>>(p); }
    KVQ_PC(128, 2) KVQ_PC(128, 4) KVQ_PC(64, 2) KVQ_PC(64, 4)
#undef KVQ_PC
    KVQ_CUDA_TRY(cudaGetLastError());
  }
  return KVQ_OK;
}

int launch_unpack_codes(const kvq_cache_desc* d, int which, int64_t begin, int64_t n, uint8_t* out,
                        cudaStream_t st) {
  const int64_t total = (int64_t)d->batch * d->heads * n * d->head_dim;
  if (total == 0) return KVQ_OK;
  const uint8_t* codes = static_cast<const uint8_t*>(which == 0 ? d->k_codes : d->v_codes);
  const int threads = 256;
  const int64_t blocks = (total + threads - 1) / threads;
  if (blocks > 0x7FFFFFFFLL) return KVQ_ERR_UNSUPPORTED;
  if (d->bits == 2)
    unpack_codes_kernel<2><<<(unsigned)blocks, threads, 0, st>>>(codes, out, d->capacity, begin % d->capacity, n, d->head_dim, total);
  else
    unpack_codes_kernel<4><<<(unsigned)blocks, threads, 0, st>>>(codes, out, d->capacity, begin % d->capacity, n, d->head_dim, total);
  KVQ_CUDA_TRY(cudaGetLastError());
  return KVQ_OK;
}

}  // namespace kvq
