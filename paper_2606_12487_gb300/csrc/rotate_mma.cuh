// rotate_mma.cuh -- the exact block-Hadamard rotation of rotate_row.cuh on the tensor
// cores and the packed fp32 pipe: the same sums, scales and codes, bit for bit.
//
// Numbers.  Every value x of a Hadamard block of 2^l elements is split into x = hi + lo with
// hi a multiple of 2^u and |lo| <= 2^(u - 1), u = 1 - l + k; both halves are binary16 numbers.
// A sum of such halves with signs is exact in fp32 while it stays below 2^24 of its unit:
//   hi: the block's sum of |x| is below 2^(24 + u) = 2^(25 - l + k)      (k is chosen so);
//   lo: 2^l 2^(u - 1) = 2^k is at most 2^24 units of 2^(k - 24), and every x is a multiple
//       of 2^(k - 24): always true for k = 0 (binary16 is a multiple of 2^-24).
// So each Hadamard sum is an exact fp32 pair, and fl(hi + lo), one addition, is the
// correctly rounded fp32 of the sum.
// For k > 0 (a block's sum of |x| of 2^(25 - l) or more) the few values below 2^(k - 14) that
// are finer than 2^(k - 24) are rounded to it first, and what that takes off (at most
// 2^(k - 25), a multiple of 2^-24) goes into a list of the unit: every sum of the block is then
// corrected by plus or minus each entry (unit_to_grid, unit_add_off; N(0, 3^2) in blocks of
// 4096 has one entry in 14 blocks).  Rows with a longer list, a sum of 2^22 or more,
// infinities or NaN are rotated in 64-bit integers (rotate_slow_row).
//
// Work split.  A warp takes a unit of 1024 consecutive elements, 32 a thread; 1, 2 or 4 warps
// share a block (G).  Element i of a unit, bits i9..i0:
//   * loads: lane (q = lane % 4, g = lane / 4) reads 8 consecutive halves (i2..i0) at
//     i4 i3 = q, i5 = g0, i9 i8 = g2 g1, four times (i7 i6);
//   * butterflies of bits 0, 1, 3, 4: one m16n8k16 MMA per half (hi, lo) and 128 elements
//     (a 16-point transform is the 16 x 16 matrix H; the fp16 registers are its B operand
//     as loaded), products and fp32 sums exact;
//   * bits 2, 6, 7 across the 8 MMAs' accumulators, packed fp32 pairs; bit 5 inside a pair;
//   * one exchange through shared memory (16 bytes = two sums' pairs, swizzled: no bank
//     conflicts either way) after which a thread holds bits 8 .. 11 of the block and 8, 4 or
//     2 consecutive elements (G = 1, 2, 4);
//   * bits 8 .. 11 on (hi, lo) pairs, one packed addition per element and level.
// Bits of l and above are left out (the MMA's matrix is the identity on them), so smaller
// blocks take the same code.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include "dptq_device.cuh"
#include "dptq_internal.h"
#include "rotate_row.cuh"

namespace dptq {

constexpr int kUnit = 1024;            // elements of one warp
constexpr int kUnitBytes = kUnit * 8;  // its (hi, lo) pairs in the exchange
constexpr int kOffMax = 63;             // entries of its list (unit_to_grid)
constexpr int kOffBytes = 4 * (1 + kOffMax);
constexpr int kStageBytes = kUnit * 2 + kOffBytes;  // its halves, waiting for their turn, and its list
constexpr uint32_t kRowSlow = 0x7FFFFFFFu;   // in place of a maximum: the row leaves the pair form

__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ void f2_bfly(uint64_t& a, uint64_t& b) {
  const uint64_t s = f2_add(a, b);
  b = f2_sub(a, b);
  a = s;
}

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__half2 v) { return *reinterpret_cast<const uint32_t*>(&v); }

// A operand of the 16-point transform for this lane: entry (row, k) is the product over
// the bit pairs of H_2 (bits below l) or I_2 (the others).  Row bits (g0, g1, g2, reg) and k
// bits stand for element bits 1, 3, 4, 0 and 0, 3, 4, 1.
__device__ __forceinline__ void mma_hadamard_a(int l, int lane, uint32_t (&a)[4]) {
  const uint32_t act = (l > 0 ? 1u : 0u) | (l > 1 ? 2u : 0u) | (l > 3 ? 4u : 0u) | (l > 4 ? 8u : 0u);
  const uint32_t g = lane >> 2, q = lane & 3;
  auto entry = [&](uint32_t rho, uint32_t k) -> uint32_t {   // both as bits (0, 1, 3, 4) of the element
    if ((rho ^ k) & ~act) return 0u;
    return (__popc(rho & k & act) & 1) ? 0xBC00u : 0x3C00u;   // -1, 1
  };
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    // register r: row g + 8 (r & 1), k = 2 q + 8 (r >> 1) and the next
    const uint32_t rho = (uint32_t)(r & 1) | ((g & 1) << 1) | ((g >> 1) << 2);
    const uint32_t kk = ((uint32_t)(r >> 1) << 1) | (q << 2);
    a[r] = entry(rho, kk) | (entry(rho, kk | 1u) << 16);
  }
}

// 16-byte granule of the exchange that holds elements i and i + 1 (i even) of a unit.
// Writers of a quarter warp differ in bits 1, 8, 9, readers in bits 3, 4, 5 (G = 1),
// 2, 3, 4 (G = 2) or 1, 2, 3 (G = 4): the low three bits of the granule differ in each.
// xch_granule(i ^ j) = xch_granule(i) ^ xch_granule(j), and its bits 3 and up are those of i / 2.
__host__ __device__ __forceinline__ constexpr int xch_granule(int i) {
  return (i >> 1) ^ ((i >> 4) & 1) ^ ((((i >> 8) ^ (i >> 5)) & 1) << 1) ^ (((i >> 9) & 1) << 2);
}

// 16 bytes at granule (base's) ^ g of a unit, g a constant: the low three bits by an exclusive
// or of the address (units are 128-byte aligned), the rest, which the base leaves zero, as
// an immediate offset.
__device__ __forceinline__ void xch_store(uint32_t base, int g, const float4& v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"((base ^ (16 * (g & 7))) + 16 * (g & ~7)), "f"(v.x),
               "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void xch_load(uint32_t base, int g, int off, uint64_t& a, uint64_t& b) {
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];"
               : "=l"(a), "=l"(b)
               : "r"((base ^ (16 * (g & 7))) + 16 * (g & ~7) + off)
               : "memory");
}

// The units of a row: whole blocks first, then the tail block in units of its own.
struct UnitMap {
  int nmain;   // units of whole blocks (a multiple of G)
  int units;   // with the tail's
};
__host__ __device__ __forceinline__ UnitMap unit_map(int K, int tail, int G) {
  const int main_len = K - tail;
  const int nm = (main_len + kUnit * G - 1) / (kUnit * G) * G;
  return UnitMap{nm, nm + (tail ? G : 0)};
}

// Correctly rounded fp32 of S / sqrt(2^l), S = hi + lo exactly (the value fixed_to_rotated
// gives for the same sum).
__device__ __forceinline__ float pair_to_rotated(float hi, float lo, int l, float c_hi, float c_lo) {
  const float sc = __int_as_float((127 - (l >> 1)) << 23);
  const float f = __fadd_rn(hi, lo);
  if ((l & 1) == 0) return __fmul_rn(f, sc);
  const float bv = __fsub_rn(f, hi);   // two-sum: rem = S - f exactly
  const float rem = __fadd_rn(__fsub_rn(hi, __fsub_rn(f, bv)), __fsub_rn(lo, bv));
  const float p = __fmul_rn(f, c_hi);
  const float err = __fmaf_rn(f, c_hi, -p);
  const float t = __fmaf_rn(f, c_lo, __fmaf_rn(rem, c_hi, err));
  return __fmul_rn(__fadd_rn(p, t), sc);
}

// ---------------------------------------------------------------- rotation of one unit
// First element of the lane's four runs of eight halves, 64 elements apart.
__device__ __forceinline__ int unit_lane_offset(int lane) {
  return (lane & 3) * 8 + ((lane >> 2) & 1) * 32 + (lane >> 3) * 256;
}
__device__ __forceinline__ void unit_load(const __half* row, int e0, int end, int lane, uint4 (&w)[4]) {
  const int o = e0 + unit_lane_offset(lane);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    w[j] = o + 64 * j < end ? __ldg(reinterpret_cast<const uint4*>(row + o + 64 * j)) : make_uint4(0u, 0u, 0u, 0u);
}
// The signs of a lane's eight halves at offset o (inside the row) applied to them.
__device__ __forceinline__ void run_signs(const int8_t* signs, int o, uint4& v) {
  const uint2 s = __ldg(reinterpret_cast<const uint2*>(signs + o));
  v.x ^= __byte_perm(s.x, 0u, 0x1404) & 0x80008000u;   // bytes 0, 1 to the sign bits
  v.y ^= __byte_perm(s.x, 0u, 0x3424) & 0x80008000u;
  v.z ^= __byte_perm(s.y, 0u, 0x1404) & 0x80008000u;
  v.w ^= __byte_perm(s.y, 0u, 0x3424) & 0x80008000u;
}
// Asynchronous copies of the lane's four runs to its own 16-byte places of `stg` (2048 bytes a
// warp, [run][lane]; zeros past the row): the next row waits there, not in registers.
__device__ __forceinline__ void unit_prefetch(const __half* row, int e0, int end, int lane, uint8_t* stg) {
  const int o = e0 + unit_lane_offset(lane);
  const uint32_t at = smem_u32(stg) + 16 * lane;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const bool in = o + 64 * j < end;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(at + 512 * j),
                 "l"(row + (in ? o + 64 * j : 0)), "r"(in ? 16 : 0)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// An upper bound of the unit's sum of |x| in units of 1/4, at least 2^24 when the sum is
// not known to be below 2^22 (also for infinities and NaN).  Eight binary16 additions in a
// row lose at most 7 2^-11 of their sum; the factor 1 + 2^-7 covers that and the fp32 steps.
constexpr uint32_t kL1Slow = 1u << 24;   // (in all 128 lanes of a group: 2^31)
template <class Run>
__device__ __forceinline__ uint32_t unit_l1(Run run) {
  __half2 s[2];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint4 v = run(j);
    const __half2 h[4] = {__habs2(as_half2(v.x)), __habs2(as_half2(v.y)), __habs2(as_half2(v.z)), __habs2(as_half2(v.w))};
    s[j >> 1] = (j & 1) ? __hadd2_rn(s[j >> 1], h[0]) : h[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) s[j >> 1] = __hadd2_rn(s[j >> 1], h[i]);
  }
  const float2 a = __half22float2(s[0]), b = __half22float2(s[1]);
  const float t = (a.x + a.y) + (b.x + b.y);
  uint32_t v = kL1Slow;
  if (t < 500000.f) v = (uint32_t)(int)(t * 4.04f) + 2u;   // 4 (1 + 2^-7) < 4.04
  return __reduce_add_sync(0xffffffffu, v);
}
// k of the block from the sum of its units' bounds.
__device__ __forceinline__ int split_k(uint32_t l1q, int l) {
  const int lg = 32 - __clz(l1q - 1);   // ceil(log2): l1q >= 2
  const int k = lg - (27 - l);
  return k > 0 ? k : 0;
}
// The unit's halves (in shared memory, [run][lane], each lane its own) rounded to multiples of
// 2^(k - 24) (k >= 1), what that took off, with the signs, into the unit's list: the count, then
// n 2^12 + i for n 2^-24 off element i of the group (|n| <= 2^(k - 1)).  A count above kOffMax: the
// list is too short.  A function of its own, in a small loop: few rows come here, and inlined it
// slowed the others down (2048 rows of K = 4096: 17.5 instead of 16.4 us).  Against a second
// pass over such rows in 64-bit integers, B = 4096, 4 bits: a fused launch of 32 tokens of
// N(0, 2.5^2), N = 4096, 25.8 -> 11.7 us (N(0, 1): 9.3 us); 2048 rows of K = 4096, N(0, 3^2),
// 95 -> 21 us, N(0, 1) with one value of 30000 in each, 166 -> 27 us (N(0, 1): 16 us).
static __device__ __noinline__ void unit_to_grid(uint8_t* halves, uint32_t* list, const int8_t* signs, int e0, int load_end,
                                                 int k, int wg, int lane) {
  const __half2 c = __half2half2(__ushort_as_half((unsigned short)((k - 14 + 15) << 10)));   // 2^(k - 14)
  int count = 0;
#pragma unroll 1
  for (int j = 0; j < 4; ++j) {
    uint4* const run = reinterpret_cast<uint4*>(halves + 512 * j + 16 * lane);
    const uint4 v = *run;
    uint32_t w[4] = {v.x, v.y, v.z, v.w}, d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2 m = __hmin2(__habs2(as_half2(w[i])), c);
      d[i] = as_u32(__hsub2_rn(m, __hsub2_rn(__hadd2_rn(m, c), c)));   // exact; 0 for |x| >= c
    }
    if (!__any_sync(0xffffffffu, ((d[0] | d[1] | d[2] | d[3]) & 0x7FFF7FFFu) != 0u)) continue;
    uint4 sv = v;
    const int o = e0 + unit_lane_offset(lane) + 64 * j;
    if (signs != nullptr && o < load_end) run_signs(signs, o, sv);
    const uint32_t sw[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = as_u32(__hsub2_rn(as_half2(w[i]), as_half2(d[i] ^ (w[i] & 0x80008000u))));   // exact
      const float2 t = __half22float2(as_half2(d[i] ^ (sw[i] & 0x80008000u)));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float e = h ? t.y : t.x;
        const uint32_t has = __ballot_sync(0xffffffffu, e != 0.f);
        const int at = count + __popc(has & ((1u << lane) - 1u));
        if (e != 0.f && at < kOffMax)
          list[1 + at] = (uint32_t)((int)(e * 16777216.f) * 4096 + wg * kUnit + o - e0 + 2 * i + h);
        count += __popc(has);
      }
    }
    *run = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if (lane == 0) list[0] = (uint32_t)count;
}

// Split, MMAs and the butterflies of bits 0 .. 7, then the unit's pairs into the exchange
// (`xu`: the unit's 8192 bytes).  FULL: l >= 8, every level applies; a level under a
// condition costs a register move for each of its additions.
template <bool FULL, class Run>
__device__ __forceinline__ void unit_phase1(Run run, const uint32_t (&am)[4], int l, int k, int lane, uint8_t* xu) {
  // C = T = 2^(10 + u): |x| + C for |x| <= T rounds to a multiple of 2^u; larger values
  // are multiples of 2^u already.
  const __half2 c = __half2half2(__ushort_as_half((unsigned short)((11 - l + k + 15) << 10)));
  uint64_t h[8][2], o[8][2];   // [instance 2 j + b2][bit 0]: pairs over bit 5
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint4 wv = run(j);
    const uint32_t w[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
    for (int b2 = 0; b2 < 2; ++b2) {
      uint32_t hi[2], lo[2];
#pragma unroll
      for (int b1 = 0; b1 < 2; ++b1) {
        const uint32_t x = w[2 * b2 + b1];
        const __half2 m = __hmin2(__habs2(as_half2(x)), c);
        const __half2 r = __hsub2_rn(__hadd2_rn(m, c), c);
        lo[b1] = as_u32(__hsub2_rn(m, r)) ^ (x & 0x80008000u);
        hi[b1] = as_u32(__hsub2_rn(as_half2(x), as_half2(lo[b1])));
      }
      float dh[4], dl[4];
      mma_16816(dh, am, hi[0], hi[1]);
      mma_16816(dl, am, lo[0], lo[1]);
      const int n = 2 * j + b2;
      h[n][0] = f2_pack(dh[0], dh[1]);
      h[n][1] = f2_pack(dh[2], dh[3]);
      o[n][0] = f2_pack(dl[0], dl[1]);
      o[n][1] = f2_pack(dl[2], dl[3]);
    }
  }
#pragma unroll
  for (int bit = 0; bit < 3; ++bit) {   // instance bits: element bits 2, 6, 7
    if (FULL || l > (bit == 0 ? 2 : 5 + bit)) {
#pragma unroll
      for (int n = 0; n < 8; ++n)
        if (!(n & (1 << bit))) {
#pragma unroll
          for (int b0 = 0; b0 < 2; ++b0) {
            f2_bfly(h[n][b0], h[n + (1 << bit)][b0]);
            f2_bfly(o[n][b0], o[n + (1 << bit)][b0]);
          }
        }
    }
  }
  // bit 5 and the stores: element bits 1 = g0, 3 = g1, 4 = g2, 8 = q0, 9 = q1
  const int g = lane >> 2, q = lane & 3;
  const uint32_t base = smem_u32(xu) + 16 * xch_granule(((g & 1) << 1) | ((g >> 1) << 3) | (q << 8));
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    float h00, h01, h10, h11, o00, o01, o10, o11;   // [bit 0][bit 5]
    f2_unpack(h[n][0], h00, h01);
    f2_unpack(h[n][1], h10, h11);
    f2_unpack(o[n][0], o00, o01);
    f2_unpack(o[n][1], o10, o11);
    float4 v0, v1;   // bit 5 = 0, 1: (hi, lo) of bit 0 = 0, then of bit 0 = 1
    if (FULL || l > 5) {
      v0 = make_float4(h00 + h01, o00 + o01, h10 + h11, o10 + o11);
      v1 = make_float4(h00 - h01, o00 - o01, h10 - h11, o10 - o11);
    } else {
      v0 = make_float4(h00, o00, h10, o10);
      v1 = make_float4(h01, o01, h11, o11);
    }
    const int i = ((n & 1) << 2) | ((n >> 1) << 6);
    xch_store(base, xch_granule(i), v0);
    xch_store(base, xch_granule(i | 32), v1);
  }
}

// Where a thread's 32 values sit after the exchange: 32 / R runs of R consecutive elements,
// run c at 256 c + low of the group's 1024 G elements.
template <int G>
struct RunLayout {
  static constexpr int R = G == 1 ? 8 : G == 2 ? 4 : 2;
  static constexpr int C = 32 / R;
  static __device__ __forceinline__ int low(int t) { return t * R; }   // t: thread of the group
};

// The exchange's reads and the butterflies of bits 8 .. 11.  v[c R + e]: (hi, lo) of element
// 256 c + low + e of the group.  FULL: every level applies (l = 8 + log2 of the runs).
template <int G, bool FULL>
__device__ __forceinline__ void unit_phase2(const uint8_t* xg, int t, int l, uint64_t (&v)[32]) {
  using RL = RunLayout<G>;
  const uint32_t base = smem_u32(xg) + 16 * xch_granule(RL::low(t));
#pragma unroll
  for (int c = 0; c < RL::C; ++c) {
#pragma unroll
    for (int e = 0; e < RL::R; e += 2) {
      xch_load(base, xch_granule(256 * (c & 3) + e), (c >> 2) * kUnitBytes, v[c * RL::R + e], v[c * RL::R + e + 1]);
    }
  }
#pragma unroll
  for (int bit = 0; (1 << bit) < RL::C; ++bit) {
    if (FULL || l > 8 + bit) {
#pragma unroll
      for (int x = 0; x < 32; ++x)
        if (!(x & (RL::R << bit))) f2_bfly(v[x], v[x + (RL::R << bit)]);
    }
  }
}

// The lists of the group's units (`stride` bytes apart) added to the thread's sums: an entry t at
// element i is +-t in the sums j of its block, minus for an odd number of common bits of i and j.
// |S| < 2^22, so with the pair first made (f, S - f), f = fl(S), |S - f| <= 1/8, the second part
// takes all corrections (multiples of 2^-24, below 1/2 together) exactly.
template <int G>
__device__ __forceinline__ void unit_add_off(const uint8_t* lists, int stride, int t, int l, uint64_t (&v)[32]) {
  using RL = RunLayout<G>;
#pragma unroll
  for (int x = 0; x < 32; ++x) {
    float h, o;
    f2_unpack(v[x], h, o);
    const float f = __fadd_rn(h, o), bv = __fsub_rn(f, h);   // two-sum: the remainder is exact
    v[x] = f2_pack(f, __fadd_rn(__fsub_rn(h, __fsub_rn(f, bv)), __fsub_rn(o, bv)));
  }
  // Value x is element j = low | 256 (x / R) + x % R (bits apart): its five bits of j one by one.
  const uint32_t low = (uint32_t)RL::low(t);
  constexpr uint32_t kBits[5] = {0xAAAAAAAAu, 0xCCCCCCCCu, 0xF0F0F0F0u, 0xFF00FF00u, 0xFFFF0000u};   // bit x: bit b of x
#pragma unroll 1
  for (int g = 0; g < G; ++g) {
    const uint32_t* const list = reinterpret_cast<const uint32_t*>(lists + g * stride);
    const int n = (int)list[0];
#pragma unroll 1
    for (int e = 1; e <= n; ++e) {
      const uint32_t i = list[e] & 4095u;
      const float d = (float)((int)list[e] >> 12) * 0x1p-24f;
      uint32_t odd = 0u - (__popc(i & low & ((1u << l) - 1u)) & 1u);   // bit x: minus
      uint32_t in = (((i ^ low) & RL::low(32 * G - 1)) >> l) == 0u ? ~0u : 0u;   // bit x: i and j in one block
#pragma unroll
      for (int b = 0; b < 5; ++b) {
        const int jb = (1 << b) < RL::R ? b : 8 + b - (RL::R == 8 ? 3 : RL::R == 4 ? 2 : 1);
        const uint32_t set = (i >> jb) & 1u ? kBits[b] : 0u;
        if (jb < l)
          odd ^= set;
        else
          in &= (i >> jb) & 1u ? kBits[b] : ~kBits[b];
      }
      if (in == 0u) continue;
      const uint32_t db = __float_as_uint(d);
#pragma unroll
      for (int x = 0; x < 32; ++x) {
        float f, rem;
        f2_unpack(v[x], f, rem);
        if (in & (1u << x)) rem = __fadd_rn(rem, __uint_as_float(db ^ ((odd << (31 - x)) & 0x80000000u)));
        v[x] = f2_pack(f, rem);
      }
    }
  }
}

// The same out of line, on sums that wait in the thread's own places of the exchange (`buf`: its
// first 16 bytes; 512 bytes from pair to pair).
template <int G>
__device__ __noinline__ void unit_add_off_at(const uint8_t* lists, int stride, int t, int l, ulonglong2* buf) {
  uint64_t v[32];
#pragma unroll
  for (int x = 0; x < 32; x += 2) {
    const ulonglong2 w = buf[16 * x];
    v[x] = w.x;
    v[x + 1] = w.y;
  }
  unit_add_off<G>(lists, stride, t, l, v);
#pragma unroll
  for (int x = 0; x < 32; x += 2) buf[16 * x] = make_ulonglong2(v[x], v[x + 1]);
}

// Largest |fl(S)| of the warp's values, as fp32 bits; part[g]: the lane's over values 8 g .. 8 g + 7.
__device__ __forceinline__ uint32_t warp_sum_max(const uint64_t (&v)[32], float (&part)[4]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    part[g] = 0.f;
#pragma unroll
    for (int e = 8 * g; e < 8 * g + 8; e += 2) {
      float h, o, h2, o2;
      f2_unpack(v[e], h, o);
      f2_unpack(v[e + 1], h2, o2);
      part[g] = fmaxf(part[g], fmaxf(fabsf(__fadd_rn(h, o)), fabsf(__fadd_rn(h2, o2))));
    }
  }
  return __reduce_max_sync(0xffffffffu,
                           __float_as_uint(fmaxf(fmaxf(part[0], part[1]), fmaxf(part[2], part[3]))));
}

// Largest |y| over the lane's values whose |fl(S)| is `wm`, 0 if it has none (odd l: 1 / sqrt 2
// and the sum's own remainder decide y's last bit).  Lanes look only at the eights that hold
// one.
__device__ __forceinline__ float largest_rotated(const uint64_t (&v)[32], const float (&part)[4], uint32_t wm, int l,
                                                 float c_hi, float c_lo) {
  float ym = 0.f;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    if (__float_as_uint(part[g]) == wm) {
      int left = 1;
#pragma unroll 1
      for (int it = 0; it < left; ++it) {   // the it-th such value
        float ch = 0.f, cl = 0.f;
        int c = 0;
#pragma unroll
        for (int e = 8 * g; e < 8 * g + 8; ++e) {
          float h, o;
          f2_unpack(v[e], h, o);
          if ((__float_as_uint(__fadd_rn(h, o)) & 0x7FFFFFFFu) == wm) {
            if (c == it) {
              ch = h;
              cl = o;
            }
            ++c;
          }
        }
        left = c;
        ym = fmaxf(ym, fabsf(pair_to_rotated(ch, cl, l, c_hi, c_lo)));
      }
    }
  }
  return ym;
}

// Codes of the thread's values as floats (whole numbers, no -0).  t = f r with f the fp32 of
// the sum and r = fl(factor / s) carries at most a few units of 2^-24 against the IEEE
// quotient of the correctly rounded y: |difference| <= |t| 2^-20.  Outside that distance from a
// half-integer both round to the same code; inside it (rare, margin 2^-17 at |t| <= 8 and
// 2^-13 at |t| <= 128) the quotient itself decides.  |t| never exceeds qmax (1 + 2^-22), so no
// code needs a clamp.
constexpr float kRoundBias = 12582912.0f;   // 1.5 * 2^23: x + bias rounds x to a whole number
__device__ __forceinline__ void pair_codes(const uint64_t (&v)[32], int e0, int l, float s, float r, float margin,
                                           float c_hi, float c_lo, float (&q)[8]) {
  const uint64_t nr = f2_pack(-r, -r), bias = f2_pack(kRoundBias, kRoundBias);
  float dm = 0.f;
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    float h0, o0, h1, o1;
    f2_unpack(v[e0 + e], h0, o0);
    f2_unpack(v[e0 + e + 1], h1, o1);
    const uint64_t f = f2_pack(__fadd_rn(h0, o0), __fadd_rn(h1, o1));
    const uint64_t qq = f2_sub(bias, f2_fma(f, nr, bias));   // rint(f r), +0 for zero
    float d0, d1;
    f2_unpack(f2_fma(f, nr, qq), d0, d1);                    // rint(f r) - f r
    dm = fmaxf(dm, fmaxf(fabsf(d0), fabsf(d1)));
    f2_unpack(qq, q[e], q[e + 1]);
  }
  if (__any_sync(0xffffffffu, dm > 0.5f - margin)) {
    uint32_t near = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float h, o;
      f2_unpack(v[e0 + e], h, o);
      if (fabsf(__fmaf_rn(__fadd_rn(h, o), -r, q[e])) > 0.5f - margin) near |= 1u << e;
    }
#pragma unroll 1
    while (near) {   // one value at a time, so that the division appears once
      const uint32_t bit = near & (0u - near);
      near ^= bit;
      float ch = 0.f, cl = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float h, o;
        f2_unpack(v[e0 + e], h, o);
        if (bit == (1u << e)) {
          ch = h;
          cl = o;
        }
      }
      const float c = __fadd_rn(rintf(__fdiv_rn(pair_to_rotated(ch, cl, l, c_hi, c_lo), s)), 0.f);
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (bit == (1u << e)) q[e] = c;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------- writers
// Destination of one row in mode MODE.
struct RowOut {
  uint8_t* p;          // row base (kRQPublic, kRQY) or the operand planes (kRQAct)
  size_t plane;        // kRQAct, 8 bits: bytes to the second plane
  size_t kb_stride;    // kRQAct: rows_out * 128
  int row, bits;       // (kRQY: `bits` is 1 if the rows start 16-byte aligned)
  // Address of element k, and from it to element k + 256.
  template <int MODE>
  __device__ __forceinline__ uint8_t* at(int k) const {
    if constexpr (MODE == kRQAct)
      return p + (size_t)(k >> 7) * kb_stride + (size_t)row * 128 + ((((k >> 4) & 7) ^ (row & 7)) << 4) + (k & 15);
    else
      return p + (MODE == kRQY ? 4 * k : bits == 4 ? k >> 1 : k);
  }
  template <int MODE>
  __device__ __forceinline__ size_t step256() const {
    return MODE == kRQAct ? 2 * kb_stride : MODE == kRQY ? 1024 : bits == 4 ? 128 : 256;
  }
};

// R (2, 4 or 8) consecutive codes from element k on (k a multiple of R, whole numbers); `p`
// the address of element k.
template <int MODE, int R>
__device__ __forceinline__ void store_codes_at(const RowOut& d, uint8_t* p, const float* q);
template <int MODE, int R>
__device__ __forceinline__ void store_codes(const RowOut& d, int k, const float* q) {
  store_codes_at<MODE, R>(d, d.at<MODE>(k), q);
}
template <int MODE, int R>
__device__ __forceinline__ void store_codes_at(const RowOut& d, uint8_t* p, const float* q) {
  if constexpr (MODE == kRQAct) {
    auto put = [&](uint8_t* at, const float* c) {
      if constexpr (R == 2) *reinterpret_cast<uint16_t*>(at) = (uint16_t)e4m3x2(c[0], c[1]);
      if constexpr (R == 4) *reinterpret_cast<uint32_t*>(at) = e4m3x2(c[0], c[1]) | (e4m3x2(c[2], c[3]) << 16);
      if constexpr (R == 8)
        *reinterpret_cast<uint2*>(at) = make_uint2(e4m3x2(c[0], c[1]) | (e4m3x2(c[2], c[3]) << 16),
                                                   e4m3x2(c[4], c[5]) | (e4m3x2(c[6], c[7]) << 16));
    };
    if (d.bits == 4) {
      put(p, q);
    } else {
      // c = hi + lo, hi = sign * 16 (|c| >> 4): |c| - 7.5 rounds to 16 (|c| >> 4) at a
      // spacing of 16 (adding 1.5 * 2^27), and c - sign * 7.5 to its signed value.
      float hi[R], lo[R];
      const uint64_t big = f2_pack(201326592.f, 201326592.f);
#pragma unroll
      for (int e = 0; e < R; e += 2) {
        const uint64_t c = f2_pack(q[e], q[e + 1]);
        const uint64_t h =
            f2_sub(f2_add(f2_sub(c, f2_pack(copysignf(7.5f, q[e]), copysignf(7.5f, q[e + 1]))), big), big);
        f2_unpack(h, hi[e], hi[e + 1]);
        f2_unpack(f2_sub(c, h), lo[e], lo[e + 1]);
      }
      put(p, hi);
      put(p + d.plane, lo);
    }
  } else if constexpr (MODE == kRQPublic) {
    // Several codes make one exact fp32 sum with a bias that keeps each field positive; the
    // fields are the low bits after adding 1.5 * 2^23, and flipping each top bit gives two's
    // complement.
    if (d.bits == 4) {
      auto four = [&](int e) {
        return __float_as_uint(__fadd_rn(
            __fmaf_rn(q[e + 3], 4096.f, __fmaf_rn(q[e + 2], 256.f, __fmaf_rn(q[e + 1], 16.f, q[e]))), kRoundBias + 34952.f));
      };
      if constexpr (R == 2) *p = (uint8_t)(__float_as_uint(__fadd_rn(__fmaf_rn(q[1], 16.f, q[0]), kRoundBias + 136.f)) ^ 0x88u);
      if constexpr (R == 4) *reinterpret_cast<uint16_t*>(p) = (uint16_t)(four(0) ^ 0x8888u);
      if constexpr (R == 8) *reinterpret_cast<uint32_t*>(p) = __byte_perm(four(0), four(4), 0x5410) ^ 0x88888888u;
    } else {
      auto two = [&](int e) {
        return __float_as_uint(__fadd_rn(__fmaf_rn(q[e + 1], 256.f, q[e]), kRoundBias + 32896.f));
      };
      auto word = [&](int e) { return __byte_perm(two(e), two(e + 2), 0x5410) ^ 0x80808080u; };
      if constexpr (R == 2) *reinterpret_cast<uint16_t*>(p) = (uint16_t)(two(0) ^ 0x8080u);
      if constexpr (R == 4) *reinterpret_cast<uint32_t*>(p) = word(0);
      if constexpr (R == 8) {   // rows start 4-byte aligned at least
        reinterpret_cast<uint32_t*>(p)[0] = word(0);
        reinterpret_cast<uint32_t*>(p)[1] = word(4);
      }
    }
  } else {   // kRQY: q holds the rotated values; rows start 16-byte aligned if `bits` says so
    if (d.bits) {
      if constexpr (R == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(q[0], q[1]);
      } else {
#pragma unroll
        for (int e = 0; e < R; e += 4) *reinterpret_cast<float4*>(p + 4 * e) = make_float4(q[e], q[e + 1], q[e + 2], q[e + 3]);
      }
    } else {
#pragma unroll
      for (int e = 0; e < R; ++e) reinterpret_cast<float*>(p)[e] = q[e];
    }
  }
}

// ---------------------------------------------------------------- rows outside the pair form
// Block-sized chunks of [k0, k1) of a row in 64-bit fixed point, by NT threads that meet at
// sync(): `ch` elements at a time through `sx` (ch values), two butterfly levels per pass.
// visit(k, S0, S1, l) sees elements k and k + 1 of every chunk.  Small code on purpose: it
// runs for few rows and must not cost the others registers.
template <class Sync, class Visit>
__device__ __forceinline__ void slow_sums(const RQArgs& a, int row, int k0, int k1, int ch, long long* sx, int tid, int NT,
                                          Sync sync, Visit visit) {
  const int tail_start = a.nfull << a.log2B;
#pragma unroll 1
  for (int c0 = k0; c0 < k1;) {
    const int end = c0 < tail_start ? min(k1, tail_start) : k1;
    const int l = c0 < tail_start ? a.log2B : a.log2T;
    const int len = min(ch, end - c0);
    sync();
#pragma unroll 1
    for (int i = tid; i < ch; i += NT) {
      long long f = 0;
      if (i < len) {
        f = half_to_fixed(__half_as_ushort(a.x[(size_t)row * a.K + c0 + i]));
        if (a.signs != nullptr && a.signs[c0 + i] < 0) f = -f;
      }
      sx[i] = f;
    }
#pragma unroll 1
    for (int b = 0; b < l; b += 2) {
      sync();
      const bool two = b + 1 < l;
#pragma unroll 1
      for (int t = tid; t < ch >> (two ? 2 : 1); t += NT) {
        long long* p = sx + (((t >> b) << (b + (two ? 2 : 1))) | (t & ((1 << b) - 1)));
        const int d = 1 << b;
        const long long s = p[0] + p[d], e = p[0] - p[d];
        if (!two) {
          p[0] = s;
          p[d] = e;
        } else {
          const long long s2 = p[2 * d] + p[3 * d], e2 = p[2 * d] - p[3 * d];
          p[0] = s + s2;
          p[d] = e + e2;
          p[2 * d] = s - s2;
          p[3 * d] = e - e2;
        }
      }
    }
    sync();
#pragma unroll 1
    for (int i = 2 * tid; i < len; i += 2 * NT) visit(c0 + i, sx[i], sx[i + 1], l);
    c0 += len;
  }
}

// A share [k0, k1) of a row in 64-bit fixed point, twice: the row maximum (`rowmax`: this
// thread's maximum in, the row's out), then the codes.
template <int MODE, class Sync, class RowMax>
__device__ __forceinline__ void rotate_slow_row(const RQArgs& a, int row, int k0, int k1, int ch, uint8_t* smem, int tid,
                                                int NT, Sync sync, const RowOut& dst, RowMax rowmax) {
  long long* sx = reinterpret_cast<long long*>(smem);
  float m = 0.f, amax = 0.f, s = 0.f;
  const float qmaxf = (float)((1 << (a.bits - 1)) - 1), qminf = -(float)(1 << (a.bits - 1));
#pragma unroll 1
  for (int pass = MODE == kRQY ? 1 : 0; pass < 2; ++pass) {
    slow_sums(a, row, k0, k1, ch, sx, tid, NT, sync, [&](int k, long long S0, long long S1, int l) {
      const float y0 = fixed_to_rotated(S0, l, a.c_hi, a.c_lo), y1 = fixed_to_rotated(S1, l, a.c_hi, a.c_lo);
      if (pass == 0) {
        m = fmaxf(m, fmaxf(fabsf(y0), fabsf(y1)));
        return;
      }
      float q[2] = {y0, y1};
      if (MODE != kRQY) {
        q[0] = amax > 0.f ? __fadd_rn(fminf(fmaxf(rintf(__fdiv_rn(y0, s)), qminf), qmaxf), 0.f) : 0.f;
        q[1] = amax > 0.f ? __fadd_rn(fminf(fmaxf(rintf(__fdiv_rn(y1, s)), qminf), qmaxf), 0.f) : 0.f;
      }
      store_codes<MODE, 2>(dst, k, q);
    });
    if (pass == 0) {
      amax = rowmax(m);
      s = __fdiv_rn(amax, qmaxf);
    }
  }
}

// ---------------------------------------------------------------- one unit, all steps
// The steps that the standalone kernel and the fused decode launch share.  Geometry of a
// warp's unit within its row:
template <int G>
struct UnitGeom {
  int e0, eg;            // first element of the unit, of its group
  int load_end, store_end;
  int l;                 // log2 of the unit's block
  int wg, tg;            // warp and thread within the group
  bool in;               // the unit exists (the same for a whole group)
  // `u`: the warp's unit in the row (groups start at multiples of G)
  __device__ __forceinline__ UnitGeom(const RQArgs& a, int u, int lane, int row_end) {
    const UnitMap um = unit_map(a.K, a.tail, G);
    const int tail_start = a.nfull << a.log2B;
    wg = u % G;
    tg = wg * 32 + lane;
    const int ug = u - wg;
    const bool main_unit = ug < um.nmain;
    in = ug < um.units;
    eg = main_unit ? ug * kUnit : in ? tail_start + (ug - um.nmain) * kUnit : row_end;
    e0 = eg + wg * kUnit;
    load_end = main_unit ? tail_start : a.K;
    store_end = main_unit && a.tail ? tail_start : row_end;
    l = main_unit ? a.log2B : a.log2T;
  }
  // First element of unit u (K past the last).
  static __device__ __forceinline__ int first(const RQArgs& a, int u) {
    const UnitMap um = unit_map(a.K, a.tail, G);
    return u < um.nmain ? min(u * kUnit, a.K) : u == um.nmain ? a.nfull << a.log2B : a.K;
  }
};

// From the lane's halves (raw(j): run j, signs(j, v): the signs applied to it, to_grid(k):
// unit_to_grid for them) to the thread's exact sums; false when the unit's block leaves the pair
// form (v is then meaningless).  l1s: a word per warp of the group; off: the unit's list, the
// group's OFF bytes apart; group_sync: the group's barrier; after_split(): called when the
// halves are no longer needed (the next row's loads).  APART: what few rows need is a call, for
// code that runs once a launch (the fused launch, M = 16, N = 512, K = 256: 7.57 -> 7.29 us) or
// spills more without (rotated fp32 rows, M = 4000, K = 28672: 271 -> 260 us).
template <int G, int OFF, bool APART, class Raw, class ToGrid, class Signs, class GroupSync, class After>
__device__ __forceinline__ bool unit_sums(const UnitGeom<G>& u, Raw raw, ToGrid to_grid, Signs signs, const uint32_t (&am)[4],
                                          int lane, uint8_t* xu, uint32_t* l1s, uint8_t* off, GroupSync group_sync,
                                          After after_split, uint64_t (&v)[32]) {
  constexpr int full_l = G == 1 ? 10 : G == 2 ? 11 : 12;
  uint32_t l1 = unit_l1(raw);
  if constexpr (G > 1) {
    if (lane == 0) l1s[u.wg] = l1;
    group_sync();
    l1 = 0;
#pragma unroll
    for (int i = 0; i < G; ++i) l1 += l1s[i];
  }
  bool ok = l1 < kL1Slow;
  const int k = ok ? split_k(l1, u.l) : 0;   // (the same in the whole group)
  if (__builtin_expect(k > 0, 0)) to_grid(k);
  auto run = [&](int j) {
    uint4 x = raw(j);
    signs(j, x);
    return x;
  };
  if (u.l >= 8)
    unit_phase1<true>(run, am, u.l, k, lane, xu);
  else
    unit_phase1<false>(run, am, u.l, k, lane, xu);
  after_split();
  group_sync();
  const uint8_t* xg = xu - u.wg * kUnitBytes;
  if (u.l == full_l)
    unit_phase2<G, true>(xg, u.tg, u.l, v);
  else
    unit_phase2<G, false>(xg, u.tg, u.l, v);
  if (__builtin_expect(k > 0, 0)) {
    const uint8_t* const lists = off - u.wg * OFF;
    uint32_t most = 0;   // entries of the group's longest list: every warp of it goes the same way
#pragma unroll
    for (int g = 0; g < G; ++g) most = max(most, *reinterpret_cast<const uint32_t*>(lists + g * OFF));
    if (most > (uint32_t)kOffMax) {
      ok = false;
    } else if (most > 0u) {
      if constexpr (APART) {
        group_sync();   // the group has read the exchange
        ulonglong2* const buf = reinterpret_cast<ulonglong2*>(xu) + lane;
#pragma unroll
        for (int x = 0; x < 32; x += 2) buf[16 * x] = make_ulonglong2(v[x], v[x + 1]);
        unit_add_off_at<G>(lists, OFF, u.tg, u.l, buf);
#pragma unroll
        for (int x = 0; x < 32; x += 2) {
          const ulonglong2 w = buf[16 * x];
          v[x] = w.x;
          v[x + 1] = w.y;
        }
      } else {
        unit_add_off<G>(lists, OFF, u.tg, u.l, v);
      }
    }
  }
  return ok;
}

// Largest |y| of the warp, as fp32 bits, or 0 if it is certainly not the largest of the
// warps that share `lead` (zero before the row's first warp).
__device__ __forceinline__ uint32_t unit_max(const uint64_t (&v)[32], int l, uint32_t* lead, int lane, float c_hi,
                                             float c_lo) {
  float part[4];
  const uint32_t wm = warp_sum_max(v, part);
  uint32_t m = __float_as_uint(__fmul_rn(__uint_as_float(wm), __int_as_float((127 - (l >> 1)) << 23)));
  if (l & 1) {
    // 2^-j fl(S) / sqrt 2, rounded twice, is within 2 units of y: only warps that are not
    // clearly below another form their largest y exactly.
    m = __float_as_uint(__fmul_rn(__uint_as_float(m), c_hi));
    uint32_t seen = 0u;
    if (lane == 0) seen = atomicMax(lead, m);
    seen = __shfl_sync(0xffffffffu, seen, 0);
    m = seen > m + 8u ? 0u
                      : __reduce_max_sync(0xffffffffu, __float_as_uint(largest_rotated(v, part, wm, l, c_hi, c_lo)));
  }
  return m;
}

// The thread's codes (kRQY: rotated values) to their places; s: the row's scale.
template <int MODE, int G>
__device__ __forceinline__ void unit_store(const RQArgs& a, const UnitGeom<G>& u, const uint64_t (&v)[32], float amax,
                                           float s, const RowOut& dst) {
  using RL = RunLayout<G>;
  const float p2 = __int_as_float((127 - (u.l >> 1)) << 23);   // 2^-(l / 2)
  const float r = __fmul_rn((u.l & 1) ? __fmul_rn(p2, a.c_hi) : p2, amax > 0.f ? __frcp_rn(s) : 0.f);
  const float margin = a.bits == 4 ? 0x1p-17f : 0x1p-13f;
  const int kb = u.eg + RL::low(u.tg);
  uint8_t* at = dst.at<MODE>(kb);
  const size_t step = dst.step256<MODE>();
#pragma unroll
  for (int e = 0; e < 32; e += 8) {
    float q[8];
    if constexpr (MODE == kRQY) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float h, o;
        f2_unpack(v[e + i], h, o);
        q[i] = pair_to_rotated(h, o, u.l, a.c_hi, a.c_lo);
      }
    } else {
      pair_codes(v, e, u.l, s, r, margin, a.c_hi, a.c_lo, q);
    }
#pragma unroll
    for (int c = 0; c < 8 / RL::R; ++c) {
      if (kb + 256 * (e / RL::R + c) < u.store_end) store_codes_at<MODE, RL::R>(dst, at, q + c * RL::R);
      at += step;
    }
  }
}

// ---------------------------------------------------------------- fused decode launch
// Token rows by the 8 converter warps of CTA `item` of the fused GEMM, into the operand
// planes, a unit per warp: `rpc` rows (8 / wpc at most, wpc warps each), or one row, or the
// half item % 2 of a row of more than 8 units (cpr = 2).  A row's maximum meets in `sh` (32
// words; 16 .. 23 zero before), and between the two CTAs of a row in its line of a.pmax in
// global memory (words 0, 1: 1 + the bits of each maximum, 0 = not yet written; words 4, 5
// the same for rows in 64-bit integers).
__device__ __forceinline__ uint32_t row_max_exchange(uint32_t* slots, int part, uint32_t mine, long long wait_cycles,
                                                     int* err) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(slots + part), "r"(mine + 1u) : "memory");
  const long long t0 = clock64();
  while (true) {
    uint32_t o;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(o) : "l"(slots + (part ^ 1)) : "memory");
    if (o != 0u) return max(mine, o - 1u);
    if (clock64() - t0 > wait_cycles) {   // bounded: the error word is set and the own maximum stands in
      atomicCAS(err, 0, (int)kDevTimeoutRowMax);
      return mine;
    }
    __nanosleep(20);
  }
}

template <int G, class Sync>
__device__ __forceinline__ void fused_rotate_rows(const RQArgs& a, int item, int cpr, int wpc, int rpc, uint8_t* smem,
                                                  uint32_t* sh, int wc, int lane, Sync sync, long long wait_cycles,
                                                  int* err) {
  uint32_t* const red = sh;            // [8] warp maxima
  uint32_t* const l1s = sh + 8;        // [8]
  uint32_t* const lead = sh + 16;      // [8], the row's first warp's
  uint32_t* const bc = sh + 24;
  const int tid = wc * 32 + lane;
  const int part = cpr > 1 ? item % cpr : 0;
  const int row0 = cpr > 1 ? item / cpr : item * rpc;
  const int slot = wc / wpc;           // the warp's row of the CTA's
  const int row = row0 + slot;
  const UnitGeom<G> u(a, part * wpc + wc - slot * wpc, lane, a.KB * 128);
  RowOut dst;
  dst.p = static_cast<uint8_t*>(a.out);
  dst.plane = (size_t)a.KB * a.rows_out * 128;
  dst.kb_stride = (size_t)a.rows_out * 128;
  dst.row = row;
  dst.bits = a.bits;
  // debug builds: the row is one of the planes' (site 4), its units lie inside it (site 5)
  // and its slots are one of the 64 lines (site 6)
  const bool act = slot < rpc && row < a.rows_in && u.in && DPTQ_CHECK(row >= 0 && row < a.rows_out, err, 4) &&
                   DPTQ_CHECK(u.load_end <= a.K && u.store_end <= a.KB * 128, err, 5);
  uint64_t v[32];
  uint32_t m = 0u;
  if (act) {
    uint32_t am[4];
    uint4 w[4];
    unit_load(a.x + (size_t)row * a.K, u.e0, u.load_end, lane, w);
    mma_hadamard_a(u.l, lane, am);
    const int o = u.e0 + unit_lane_offset(lane);
    const bool ok = unit_sums<G, kOffBytes, true>(
                                 u, [&](int j) { return w[j]; },
                                 [&](int k) {   // by way of the exchange, not yet in use
                                   uint8_t* const xu = smem + wc * kUnitBytes;
                                   uint4* const at = reinterpret_cast<uint4*>(xu) + lane;
#pragma unroll
                                   for (int j = 0; j < 4; ++j) at[32 * j] = w[j];
                                   unit_to_grid(xu, reinterpret_cast<uint32_t*>(smem + 8 * kUnitBytes + wc * kOffBytes),
                                                a.signs, u.e0, u.load_end, k, u.wg, lane);
#pragma unroll
                                   for (int j = 0; j < 4; ++j) w[j] = at[32 * j];
                                   __syncwarp();
                                 },
                                 [&](int j, uint4& x) {
                                   if (a.signs != nullptr && o + 64 * j < u.load_end) run_signs(a.signs, o + 64 * j, x);
                                 },
                                 am, lane, smem + wc * kUnitBytes, l1s + wc - u.wg,
                                 smem + 8 * kUnitBytes + wc * kOffBytes,
                                 [&] {
                                   if constexpr (G == 1)
                                     __syncwarp();
                                   else
                                     asm volatile("bar.sync %0, %1;" ::"r"(2 + wc / G), "n"(32 * G) : "memory");
                                 },
                                 [] {}, v);
    m = unit_max(v, u.l, lead + slot, lane, a.c_hi, a.c_lo);
    if (!ok) m = kRowSlow;
  }
  if (lane == 0) red[wc] = m;
  sync();
  // Maximum of the warps of row slot s (any s; the same in every thread).
  auto slot_max = [&](int s) { return __reduce_max_sync(0xffffffffu, (lane & 7) / wpc == s ? red[lane & 7] : 0u); };
  // Whether any row of the CTA leaves the pair form, before red is used again.
  const uint32_t any = __reduce_max_sync(0xffffffffu, red[lane & 7]);
  m = slot_max(slot);
  uint32_t* const slots = a.pmax + kRowMaxStride * row0;
  auto across = [&](uint32_t mine, int off) -> uint32_t {   // the row's maximum over its CTAs
    if (cpr == 1 || !DPTQ_CHECK(row0 < 64 && part < cpr && cpr <= 2, err, 6)) return mine;
    if (tid == 0) *bc = row_max_exchange(slots + off, part, mine, wait_cycles, err);
    sync();
    return *(volatile uint32_t*)bc;
  };
  if (cpr > 1) m = across(m, 0);   // (one row: slot 0 in every warp that counts)
  const float qmaxf = (float)((1 << (a.bits - 1)) - 1);
  if (act && m != kRowSlow) {
    const float amax = __uint_as_float(m);
    const float s = __fdiv_rn(amax, qmaxf);
    if (part == 0 && wc == slot * wpc && lane == 0) a.scales[row] = s;
    unit_store<kRQAct, G>(a, u, v, amax, s, dst);
  }
  if ((cpr > 1 ? m : any) != kRowSlow) return;
  // Rows in 64-bit integers, one after the other by all the warps.
  uint32_t slow = 0u;
  if (cpr > 1)
    slow = 1u;
  else
    for (int sl = 0; sl < rpc; ++sl) slow |= slot_max(sl) == kRowSlow ? 1u << sl : 0u;
  sync();   // red and the exchange are free
#pragma unroll 1
  for (; slow; slow &= slow - 1u) {
    const int r = row0 + __ffs(slow) - 1;
    dst.row = r;
    const int k0 = UnitGeom<G>::first(a, part * wpc), k1 = UnitGeom<G>::first(a, (part + 1) * wpc);
    rotate_slow_row<kRQAct>(a, r, k0, k1, kUnit * G, smem, tid, 256, sync, dst, [&](float mine) {
      const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(mine));
      sync();
      if (lane == 0) red[wc] = wm;
      sync();
      const float rm = __uint_as_float(across(__reduce_max_sync(0xffffffffu, red[lane & 7]), 4));
      if (part == 0 && tid == 0) a.scales[r] = rm > 0.f ? __fdiv_rn(rm, qmaxf) : 0.f;
      return rm;
    });
    if (part == cpr - 1) {
      const float zero[4] = {0.f, 0.f, 0.f, 0.f};
      for (int kz = a.K + 4 * tid; kz < a.KB * 128; kz += 4 * 256) store_codes<kRQAct, 4>(dst, kz, zero);
    }
  }
}

}  // namespace dptq
