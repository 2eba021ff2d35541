// kv_policy.cu -- two kernels next to the quantized linear layer:
//   * the group-wise symmetric 4-bit KV-cache quantizer (Section 4.2: KV cache quantized
//     group-wise with group size 128), and
//   * the sensitive-layer policy: Jump Ratio and historical-feature SNR per layer
//     (Section 3.1, Eqs. 8-11) thresholded into the 8-bit layer set (Section 3.3,
//     Eq. 20; Algorithm 1 step 2).
// Both are HBM-bound streams over their inputs; the per-group / per-token quantizer is
// the same exact quantizer as the activation path (rotate_row.cuh).
#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include "dptq_device.cuh"
#include "dptq_internal.h"
#include "rotate_mma.cuh"
#include "rotate_row.cuh"

namespace dptq {

// ------------------------------------------------------------------ KV4
// Any group size: one warp per (row, group) at a time.  Lane l holds columns 4l .. 4l + 3 of each
// 128-column block of the group (J = group / 128 blocks, at most 8): one 8-byte load per
// block, the group's absmax by shuffles, then four codes per block packed into 2 bytes
// (the warp stores 64 contiguous bytes per block).
constexpr int kKvWarps = 8;

// Groups of 128 (the paper's size): eight lanes a group, 16 values a lane in two runs of
// eight (16-byte loads, 128 contiguous bytes per eight lanes), four groups a warp at a time,
// kKvSets of them with all loads issued first.  The kernel is bound by instruction issue, so
// values are handled in pairs where the hardware has a packed form:
//   * max |x| on binary16 pairs, then three exchanges between the eight lanes;
//   * codes: |y / s| <= 7 (1 + 2^-22), so no code needs the clamp.  q = rint(y r) from one
//     fma with 1.5 * 2^23 (ties to even) and its remainder y r - q from another, two values
//     per instruction.  Where y r lies within 2^-15 of a half-integer, the IEEE quotient
//     y / s decides instead (|y r - y / s| and |fl(y / s) - y / s| are both below 2^-21, so
//     elsewhere the two agree);
//   * four codes make q0 + 16 q1 + 256 q2 + 4096 q3 + 8 (1 + 16 + 256 + 4096), exact in fp32,
//     read off the low bits after the same addition; flipping bit 3 of each nibble turns
//     q + 8 into two's complement.  A NaN (NaN or infinite input) takes the code -1.
// LLaMA-2-7B K cache of 8192 tokens (67 MB in, 19 MB out): 22.6 us with four values a lane and
// one value per instruction, 18.5 us now (4.6 TB/s).  One set in flight: 20.0 us, four: 20.7 us;
// a grid of all items instead of one resident wave: 20.4 us.
constexpr float kRoundMagic = 12582912.0f;   // 1.5 * 2^23
constexpr int kKvSets = 2;

__device__ __forceinline__ float kv4_sum4(const float* q) {   // four codes in the low 16 bits
  const float t = __fmaf_rn(q[3], 4096.f, __fmaf_rn(q[2], 256.f, __fmaf_rn(q[1], 16.f, q[0])));
  return __fadd_rn(t, kRoundMagic + 34952.f);   // 34952 = 8 * 0x1111
}

// ALIGNED4: codes start 4-byte aligned and a lane stores its word at once; otherwise (2-byte
// aligned) as two halves.
template <bool ALIGNED4>
__global__ void __launch_bounds__(kKvWarps * 32) kv4_quantize_g128_kernel(const KvArgs a) {
  const int lane = threadIdx.x & 31;
  const int sub = lane & 7, quad = lane >> 3;   // lane within the group, group of the four
  const long long ngroups = (long long)a.rows * (a.cols >> 7);   // groups are consecutive in memory
  const long long nitems = (ngroups + 4 * kKvSets - 1) / (4 * kKvSets);
  const long long nwarps = (long long)gridDim.x * kKvWarps;
  for (long long w = (long long)blockIdx.x * kKvWarps + (threadIdx.x >> 5); w < nitems; w += nwarps) {
    uint4 raw[kKvSets][2];
#pragma unroll
    for (int i = 0; i < kKvSets; ++i) {
      const long long g = 4 * (kKvSets * w + i) + quad;
      const uint4* src = reinterpret_cast<const uint4*>(a.kv + (size_t)g * 128) + sub;
#pragma unroll
      for (int j = 0; j < 2; ++j) raw[i][j] = g < ngroups ? __ldg(src + 8 * j) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < kKvSets; ++i) {
      const long long g = 4 * (kKvSets * w + i) + quad;
      const uint32_t x[8] = {raw[i][0].x, raw[i][0].y, raw[i][0].z, raw[i][0].w,
                             raw[i][1].x, raw[i][1].y, raw[i][1].z, raw[i][1].w};
      __half2 m = __habs2(as_half2(x[0]));   // (a NaN loses against a number)
#pragma unroll
      for (int k = 1; k < 8; ++k) m = __hmax2(m, __habs2(as_half2(x[k])));
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) m = __hmax2(m, as_half2(__shfl_xor_sync(0xffffffffu, as_u32(m), o)));
      const float amax = __half2float(__hmax(__low2half(m), __high2half(m)));
      const float s = __fdiv_rn(amax, 7.f);   // 0 for an all-zero group
      const float r = amax > 0.f ? __frcp_rn(s) : 0.f;
      const uint64_t r2 = f2_pack(-r, -r), bias = f2_pack(kRoundMagic, kRoundMagic);
      if (sub == 0 && g < ngroups) a.scales[g] = s;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        float y[8], q[8], dm = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&x[4 * j + k]));
          y[2 * k] = f.x;
          y[2 * k + 1] = f.y;
          const uint64_t f2 = f2_pack(f.x, f.y);
          const uint64_t qq = f2_sub(bias, f2_fma(f2, r2, bias));   // rint(y r), +0 for zero
          float d0, d1;
          f2_unpack(f2_fma(f2, r2, qq), d0, d1);
          dm = fmaxf(dm, fmaxf(fabsf(d0), fabsf(d1)));
          f2_unpack(qq, q[2 * k], q[2 * k + 1]);
        }
        if (__any_sync(0xffffffffu, dm >= 0.5f - 0x1p-15f)) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (fabsf(__fmaf_rn(y[k], -r, q[k])) >= 0.5f - 0x1p-15f) q[k] = rintf(__fdiv_rn(y[k], s));
        }
        float t0 = kv4_sum4(q), t1 = kv4_sum4(q + 4);
        if (isnan(t0 + t1)) {
#pragma unroll
          for (int k = 0; k < 8; ++k) q[k] = isnan(q[k]) ? -1.f : q[k];
          t0 = kv4_sum4(q);
          t1 = kv4_sum4(q + 4);
        }
        const uint32_t word = __byte_perm(__float_as_uint(t0), __float_as_uint(t1), 0x5410) ^ 0x88888888u;
        if (g < ngroups) {
          uint8_t* dst = a.codes + (size_t)g * 64 + 4 * (8 * j + sub);
          if constexpr (ALIGNED4) {
            *reinterpret_cast<uint32_t*>(dst) = word;
          } else {
            reinterpret_cast<uint16_t*>(dst)[0] = (uint16_t)word;
            reinterpret_cast<uint16_t*>(dst)[1] = (uint16_t)(word >> 16);
          }
        }
      }
    }
  }
}

__global__ void __launch_bounds__(kKvWarps * 32) kv4_quantize_kernel(const KvArgs a) {
  const int lane = threadIdx.x & 31;
  const int J = a.group >> 7;
  const int ng = a.cols / a.group;
  const long long ngroups = (long long)a.rows * ng;
  const long long nwarps = (long long)gridDim.x * kKvWarps;
  for (long long w = (long long)blockIdx.x * kKvWarps + (threadIdx.x >> 5); w < ngroups; w += nwarps) {
    const int row = (int)(w / ng);
    const int g = (int)(w - (long long)row * ng);
    const size_t base = (size_t)row * a.cols + (size_t)g * a.group;
    const __half* src = a.kv + base;
    uint2 raw[8];
    float amax = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < J) {
        raw[j] = __ldg(reinterpret_cast<const uint2*>(src + 128 * j + 4 * lane));
        const __half2 h0 = *reinterpret_cast<const __half2*>(&raw[j].x);
        const __half2 h1 = *reinterpret_cast<const __half2*>(&raw[j].y);
        amax = fmaxf(amax, fmaxf(fmaxf(fabsf(__low2float(h0)), fabsf(__high2float(h0))),
                                 fmaxf(fabsf(__low2float(h1)), fabsf(__high2float(h1)))));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    const float s = __fdiv_rn(amax, 7.f);
    const bool nz = amax > 0.f;
    const float r = nz ? __frcp_rn(s) : 0.f;
    if (lane == 0) a.scales[(size_t)row * ng + g] = nz ? s : 0.f;
    uint16_t* dst = reinterpret_cast<uint16_t*>(a.codes + base / 2);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < J) {
        const __half2 h0 = *reinterpret_cast<const __half2*>(&raw[j].x);
        const __half2 h1 = *reinterpret_cast<const __half2*>(&raw[j].y);
        const float y[4] = {__low2float(h0), __high2float(h0), __low2float(h1), __high2float(h1)};
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        if (nz) quant_code4(y, s, r, -8.f, 7.f, c);
        uint32_t packed = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) packed |= ((uint32_t)(int)c[e] & 0xFu) << (4 * e);
        dst[32 * j + lane] = (uint16_t)packed;   // columns 128 j + 4 lane .. + 3, low nibble first
      }
    }
  }
}

cudaError_t launch_kv4(const KvArgs& a, int num_sms, cudaStream_t s) {
  const long long ngroups = (long long)a.rows * (a.cols / a.group);
  const long long work = a.group == 128 ? (ngroups + 4 * kKvSets - 1) / (4 * kKvSets) : ngroups;   // warps' items
  long long blocks = (work + kKvWarps - 1) / kKvWarps;
  int per_sm = 8;
  const auto g128 = (reinterpret_cast<uintptr_t>(a.codes) & 3u) == 0 ? kv4_quantize_g128_kernel<true>
                                                                      : kv4_quantize_g128_kernel<false>;
  if (a.group == 128) {   // one wave of resident CTAs
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, g128, kKvWarps * 32, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
  }
  const long long cap = (long long)num_sms * per_sm;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  if (a.group == 128)
    g128<<<(unsigned)blocks, kKvWarps * 32, 0, s>>>(a);
  else
    kv4_quantize_kernel<<<(unsigned)blocks, kKvWarps * 32, 0, s>>>(a);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ policy
// Tokens of more than 4096 values: one CTA of 256 threads per (layer, token) at a time,
// with plain loads.  Thread t holds columns
// 4t + 1024 i of the token (float4 loads of x and dx).  Per element, in fp32:
//   |x|^2 and |dx|^2; u = fl(x + dx) as the quantizer's input (the fp32 sum);
//   the reconstruction error xhat - x = s c - dx - x = (s c - u) - (x + dx - u): the
//   first term by one fma, the second, the rounding residue of x + dx, exactly
//   (two-sum), so that no cancellation against |x| is lost.
// The three sums go per thread in fp32, across the CTA in fp64: through shared memory, one warp
// a sum, since the fp64 unit of this GPU is slow (a warp's addition takes about 16 clocks, and
// three butterflies in every warp took longer than the token's bytes).  For the same reason the
// tokens' JR and SNR terms are formed 32 at a time, one a lane, and added to the per-layer fp64
// sums; a second kernel averages them and applies the thresholds.
// 40 layers x 1000 tokens x 8192: 1176 -> 558 us (4.7 TB/s); 40 x 512 x 5120: 556 -> 229 us.
// One wave of CTAs (8 an SM: 96 instead of 86 us for 8 x 512 x 8192).
constexpr int kPolThreads = 256;

// Warp 0, converged: token i of the batch (i < nb, first item `item0`) has its sums in
// tok[i]; adds its terms to the per-layer outputs.
template <typename F>
__device__ __forceinline__ void pol_batch(const PolicyArgs& a, const F (*tok)[3], long long item0, int nb, int lane) {
  F jr = 0, snr = 0;
  int l = -1;
  if (lane < nb) {
    const F nx = tok[lane][0], nd = tok[lane][1], ne = tok[lane][2];
    const F eps = (F)a.eps;
    if constexpr (sizeof(F) == 8) {
      jr = sqrt(nd) / (sqrt(nx) + eps);
      snr = 10.0 * log10(nx / (ne + eps));
    } else {
      jr = __fdiv_rn(sqrtf(nd), __fadd_rn(sqrtf(nx), eps));
      snr = 10.f * log10f(__fdiv_rn(nx, __fadd_rn(ne, eps)));
    }
    l = (int)((item0 + lane) / a.T);
  }
  unsigned left = __ballot_sync(0xffffffffu, lane < nb);
  while (left) {   // one pass per layer present in the batch (the batch's items are consecutive)
    const int l0 = __shfl_sync(0xffffffffu, l, __ffs(left) - 1);
    const bool in = l == l0 && lane < nb;
    F vj = in ? jr : (F)0, vs = in ? snr : (F)0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      vj += __shfl_xor_sync(0xffffffffu, vj, o);
      vs += __shfl_xor_sync(0xffffffffu, vs, o);
    }
    if (lane == 0) {
      atomicAdd(a.jr + l0, (double)vj);
      atomicAdd(a.snr + l0, (double)vs);
    }
    left &= ~__ballot_sync(0xffffffffu, in);
  }
}

__global__ void __launch_bounds__(kPolThreads) policy_stats_kernel(const PolicyArgs a) {
  __shared__ float part[3][kPolThreads];   // every thread's |x|^2, |dx|^2, |err|^2
  __shared__ double tok[32][3];            // finished tokens' sums
  __shared__ float redf[kPolThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int qmax = (1 << (a.bits - 1)) - 1;
  const float qmaxf = (float)qmax, qminf = (float)(-(1 << (a.bits - 1)));
  const long long items = (long long)a.L * a.T;
  const long long t0 = items * blockIdx.x / gridDim.x;
  const int cnt = (int)(items * (blockIdx.x + 1) / gridDim.x - t0);
  for (int j = 0; j < cnt; ++j) {
    const long long it = t0 + j;
    const float* x = a.x + (size_t)it * a.d;
    const float* dx = a.dx + (size_t)it * a.d;
    // pass 1: norms and the quantizer's absmax
    float nx = 0.f, nd = 0.f, am = 0.f;
    for (int k = 4 * tid; k < a.d; k += 4 * kPolThreads) {
      const float4 xv = __ldg(reinterpret_cast<const float4*>(x + k));
      const float4 dv = __ldg(reinterpret_cast<const float4*>(dx + k));
      const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, ds[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        nx = __fmaf_rn(xs[e], xs[e], nx);
        nd = __fmaf_rn(ds[e], ds[e], nd);
        am = fmaxf(am, fabsf(__fadd_rn(xs[e], ds[e])));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
    __syncthreads();
    if ((tid & 31) == 0) redf[tid >> 5] = am;
    __syncthreads();
    float amax = redf[0];
#pragma unroll
    for (int w = 1; w < kPolThreads / 32; ++w) amax = fmaxf(amax, redf[w]);
    const float s = __fdiv_rn(amax, qmaxf);
    const bool nzs = amax > 0.f;
    const float r = nzs ? __frcp_rn(s) : 0.f;
    // pass 2 (the token's 8d bytes are still in L1/L2): the reconstruction error
    float ne = 0.f;
    auto err4 = [&](const float4 xv, const float4 dv) {
      const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, ds[4] = {dv.x, dv.y, dv.z, dv.w};
      float u[4], c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int e = 0; e < 4; ++e) u[e] = __fadd_rn(xs[e], ds[e]);
      if (nzs) quant_code4(u, s, r, qminf, qmaxf, c);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float bv = __fsub_rn(u[e], xs[e]);
        const float av = __fsub_rn(u[e], bv);
        const float res = __fadd_rn(__fsub_rn(xs[e], av), __fsub_rn(ds[e], bv));   // x + dx - u, exact
        const float err = __fsub_rn(__fmaf_rn(s, c[e], -u[e]), res);
        ne = __fmaf_rn(err, err, ne);
      }
    };
    for (int k = 4 * tid; k < a.d; k += 4 * kPolThreads)
      err4(__ldg(reinterpret_cast<const float4*>(x + k)), __ldg(reinterpret_cast<const float4*>(dx + k)));
    part[0][tid] = nx;   // (read before the two barriers of the next token)
    part[1][tid] = nd;
    part[2][tid] = ne;
    __syncthreads();
    if (warp < 3) {
      double v = 0.0;
#pragma unroll
      for (int i = 0; i < kPolThreads / 32; ++i) v += (double)part[warp][lane + 32 * i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) tok[j & 31][warp] = v;
    }
    if ((j & 31) == 31 || j == cnt - 1) {
      __syncthreads();
      if (warp == 0) pol_batch(a, tok, t0 + (j & ~31), (j & 31) + 1, lane);
    }
  }
}

// Tokens of up to 4096 values: the staged form.  Each CTA takes a contiguous range of
// (layer, token) items; bulk copies put whole tokens (x, then dx: 8d bytes) into a ring of
// kPolStages shared-memory stages, up to kPolStages tokens ahead.  Iteration j runs pass 2
// of token j - 1 (its quantizer is known) and pass 1 of token j on the same threads, then
// one barrier publishes the per-warp partials of both; the stage of token j - 1 is
// refilled right after that barrier.  The per-element arithmetic is that of the kernel
// above.  All sums are of non-negative terms and stay in fp32 up to the token (per thread
// 16 elements, then the warp's tree, then 8 warps: a relative error below 30 units of
// 2^-24).  Thread 0 records each finished token's three sums; every 32 tokens the lanes
// of warp 0 form the tokens' JR and SNR terms in parallel (fp32; the fp64 unit of this
// GPU is far slower) and add them per layer to the fp64 outputs, one atomic per layer.
// Two stages: three CTAs an SM, whose barriers then overlap (32 layers x 512 tokens x 4096:
// 97 us; three stages, two CTAs: 115 us; 384 or 512 threads a CTA: 114, 135 us).
constexpr int kPolStages = 2;
constexpr int kPolStagedThreads = 256;
constexpr int kPolMaxStagedD = 4096;

__global__ void __launch_bounds__(kPolStagedThreads) policy_stats_staged_kernel(const PolicyArgs a) {
  extern __shared__ __align__(128) uint8_t pol_smem[];
  __shared__ uint64_t full[kPolStages];
  __shared__ float part[2][4][kPolStagedThreads / 32];   // [iteration parity][amax, |x|^2, |dx|^2, |err|^2][warp]
  __shared__ float tok[32][3];                      // finished tokens' |x|^2, |dx|^2, |err|^2
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long n = (long long)a.L * a.T;
  const long long t0 = n * blockIdx.x / gridDim.x;
  const int cnt = (int)(n * (blockIdx.x + 1) / gridDim.x - t0);
  const uint32_t half_bytes = 4u * (uint32_t)a.d, stage_bytes = 8u * (uint32_t)a.d;
  const float qmaxf = (float)((1 << (a.bits - 1)) - 1), qminf = (float)(-(1 << (a.bits - 1)));
  if (tid == 0) {
    for (int i = 0; i < kPolStages; ++i) mbar_init(&full[i], 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const uint64_t pol = l2_policy_evict_first();
  auto issue = [&](int k) {   // token t0 + k into stage k % kPolStages (one thread)
    uint8_t* st = pol_smem + (size_t)(k % kPolStages) * stage_bytes;
    uint64_t* bar = &full[k % kPolStages];
    fence_proxy_async_smem();   // the stage's earlier generic reads come before the copy's writes
    mbar_arrive_expect_tx(bar, stage_bytes);
    bulk_g2s(st, a.x + (size_t)(t0 + k) * a.d, half_bytes, bar, pol);
    bulk_g2s(st + half_bytes, a.dx + (size_t)(t0 + k) * a.d, half_bytes, bar, pol);
  };
  int issued = 0;   // tokens whose copies were issued (meaningful in warp 0)
  if (warp == 0) {
    issued = cnt < kPolStages ? cnt : kPolStages;
    if (elect_one())
      for (int k = 0; k < issued; ++k) issue(k);
    __syncwarp();
  }
  float s = 0.f, r = 0.f;
  bool nzs = false;
  float tok_nx = 0.f, tok_nd = 0.f;   // thread 0: sums of token j - 1
  for (int j = 0; j <= cnt; ++j) {
    float am = 0.f, nx = 0.f, nd = 0.f, ne = 0.f;
    if (j >= 1) {   // pass 2 of token j - 1
      const float* xs = reinterpret_cast<const float*>(pol_smem + (size_t)((j - 1) % kPolStages) * stage_bytes);
      const float* ds = xs + a.d;
      const uint64_t nr2 = f2_pack(-r, -r), s2 = f2_pack(s, s), bias2 = f2_pack(12582912.f, 12582912.f), zero2 = 0u;
      const bool fin = fmaxf(s, r) < __int_as_float(0x7F800000);   // both finite
      uint64_t ne2 = 0u;
#pragma unroll
      for (int i = 0; i < kPolMaxStagedD / (4 * kPolStagedThreads); ++i) {
        const int k = 4 * (tid + kPolStagedThreads * i);
        if (k < a.d) {
          const ulonglong2 xp = *reinterpret_cast<const ulonglong2*>(xs + k), dp = *reinterpret_cast<const ulonglong2*>(ds + k);
          const uint64_t x2[2] = {xp.x, xp.y}, d2[2] = {dp.x, dp.y};
          uint64_t u2[2], c2[2];
          float dm = 0.f;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            u2[h] = f2_add(x2[h], d2[h]);
            c2[h] = f2_sub(bias2, f2_fma(u2[h], nr2, bias2));   // rint(u r), +0 for zero
            float m0, m1;
            f2_unpack(f2_fma(u2[h], nr2, c2[h]), m0, m1);
            dm = fmaxf(dm, fmaxf(fabsf(m0), fabsf(m1)));
          }
          if (__any_sync(__activemask(), dm >= 0.5f - 0x1p-15f) || !fin) {   // near a tie, or an infinite scale or reciprocal
            float u[4], c[4] = {0.f, 0.f, 0.f, 0.f};
            f2_unpack(u2[0], u[0], u[1]);
            f2_unpack(u2[1], u[2], u[3]);
            if (nzs) quant_code4(u, s, r, qminf, qmaxf, c);
            c2[0] = f2_pack(c[0], c[1]);
            c2[1] = f2_pack(c[2], c[3]);
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint64_t bv = f2_sub(u2[h], x2[h]);
            const uint64_t av = f2_sub(u2[h], bv);
            const uint64_t res = f2_add(f2_sub(x2[h], av), f2_sub(d2[h], bv));   // x + dx - u, exact
            const uint64_t err = f2_sub(f2_fma(s2, c2[h], f2_sub(zero2, u2[h])), res);
            ne2 = f2_fma(err, err, ne2);
          }
        }
      }
      float n0, n1;
      f2_unpack(ne2, n0, n1);
      ne = n0 + n1;
    }
    if (j < cnt) {   // pass 1 of token j
      const int st = j % kPolStages;
      if (mbar_wait_warp(&full[st], (uint32_t)(j / kPolStages) & 1u, &abort_flag, a.err, kDevTimeoutFull)) {
        const float* xs = reinterpret_cast<const float*>(pol_smem + (size_t)st * stage_bytes);
        const float* ds = xs + a.d;
        uint64_t nx2 = 0u, nd2 = 0u;   // two sums each, on packed pairs
#pragma unroll
        for (int i = 0; i < kPolMaxStagedD / (4 * kPolStagedThreads); ++i) {
          const int k = 4 * (tid + kPolStagedThreads * i);
          if (k < a.d) {
            const ulonglong2 xp = *reinterpret_cast<const ulonglong2*>(xs + k), dp = *reinterpret_cast<const ulonglong2*>(ds + k);
            const uint64_t x2[2] = {xp.x, xp.y}, d2[2] = {dp.x, dp.y};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              nx2 = f2_fma(x2[h], x2[h], nx2);
              nd2 = f2_fma(d2[h], d2[h], nd2);
              float u0, u1;
              f2_unpack(f2_add(x2[h], d2[h]), u0, u1);
              am = fmaxf(am, fmaxf(fabsf(u0), fabsf(u1)));
            }
          }
        }
        float n0, n1;
        f2_unpack(nx2, n0, n1);
        nx = n0 + n1;
        f2_unpack(nd2, n0, n1);
        nd = n0 + n1;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
      nx += __shfl_xor_sync(0xffffffffu, nx, o);
      nd += __shfl_xor_sync(0xffffffffu, nd, o);
      ne += __shfl_xor_sync(0xffffffffu, ne, o);
    }
    if (lane == 0) {
      part[j & 1][0][warp] = am;
      part[j & 1][1][warp] = nx;
      part[j & 1][2][warp] = nd;
      part[j & 1][3][warp] = ne;
    }
    __syncthreads();
    const bool aborted = __shfl_sync(0xffffffffu, *(volatile int*)&abort_flag, 0) != 0;
    if (warp == 0 && j >= 1 && j - 1 + kPolStages < cnt && !aborted) {   // refill the stage of token j - 1
      if (elect_one()) issue(j - 1 + kPolStages);
      __syncwarp();
      issued = j + kPolStages;
    }
    float amax = part[j & 1][0][0];
#pragma unroll
    for (int w = 1; w < kPolStagedThreads / 32; ++w) amax = fmaxf(amax, part[j & 1][0][w]);
    s = __fdiv_rn(amax, qmaxf);
    nzs = amax > 0.f;
    r = nzs ? __frcp_rn(s) : 0.f;
    if (warp == 0) {
      if (lane == 0) {
        float sx = 0.f, sd = 0.f, se = 0.f;
#pragma unroll
        for (int w = 0; w < kPolStagedThreads / 32; ++w) {
          sx += part[j & 1][1][w];
          sd += part[j & 1][2][w];
          se += part[j & 1][3][w];
        }
        if (j >= 1) {   // token j - 1 is complete
          tok[(j - 1) & 31][0] = tok_nx;
          tok[(j - 1) & 31][1] = tok_nd;
          tok[(j - 1) & 31][2] = se;
        }
        tok_nx = sx;
        tok_nd = sd;
      }
      __syncwarp();
      if (j >= 1 && (((j - 1) & 31) == 31 || j == cnt) && !aborted) {
        const int first = (j - 1) & ~31;
        pol_batch(a, tok, t0 + first, j - first, lane);
      }
      __syncwarp();
    }
  }
  if (abort_flag) {
    // A wait gave up (the outputs are incomplete; the error word says so): let the copies
    // already issued land before the CTA's shared memory is released (bounded, on the
    // tokens that may still be in flight).
    if (warp == 0) {
      volatile int no_abort = 0;
      const int lo = issued > kPolStages ? issued - kPolStages : 0;
      for (int k = lo; k < issued; ++k)
        mbar_wait_warp(&full[k % kPolStages], (uint32_t)(k / kPolStages) & 1u, &no_abort, a.err, kDevTimeoutDrain);
    }
  }
}

__global__ void policy_finish_kernel(const PolicyArgs a) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= a.L) return;
  const double jr = a.jr[l] / a.T, snr = a.snr[l] / a.T;
  a.jr[l] = jr;
  a.snr[l] = snr;
  a.bits_out[l] = (jr > a.tau_jr && snr < a.tau_snr) ? 8 : 4;
}

cudaError_t launch_policy(const PolicyArgs& a, int num_sms, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(a.jr, 0, sizeof(double) * a.L, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.snr, 0, sizeof(double) * a.L, s);
  if (e != cudaSuccess) return e;
  const long long items = (long long)a.L * a.T;
  if (a.d <= kPolMaxStagedD) {
    const int smem = kPolStages * 8 * a.d;
    e = ensure_max_dyn_smem(policy_stats_staged_kernel);
    int per_sm = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, policy_stats_staged_kernel, kPolStagedThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    long long blocks = (long long)num_sms * per_sm;
    if (blocks > items) blocks = items;
    policy_stats_staged_kernel<<<(unsigned)blocks, kPolStagedThreads, smem, s>>>(a);
  } else {
    long long blocks = items < (long long)num_sms * 4 ? items : (long long)num_sms * 4;   // one wave
    if (blocks < 1) blocks = 1;
    policy_stats_kernel<<<(unsigned)blocks, kPolThreads, 0, s>>>(a);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  policy_finish_kernel<<<(a.L + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace dptq
