// rotate_quant.cu -- standalone launches of the fused online block-Hadamard rotation +
// symmetric per-row quantization (Section 2, Eq. 4 then Eq. 2; Section 4.2): the
// tensor-core kernel for activations (rotate_mma.cuh), the per-row kernel in 64-bit integers
// (rotate_row.cuh; weights, Paley tails), and the converter of public codes into the
// GEMM's E4M3 planes.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include "dptq_device.cuh"
#include "dptq_internal.h"
#include "rotate_mma.cuh"
#include "rotate_row.cuh"

namespace dptq {

// Three CTAs per SM (at most 85 registers a thread; the body takes 79 or 80, without spilling):
// many-row launches (prefill) are bound by the latency of each row's chain of steps, so
// rows in flight per SM set their throughput.
template <int MODE>
__global__ void __launch_bounds__(kRQThreads, 3) rotate_quant_kernel(const RQArgs a) {
  extern __shared__ __align__(16) unsigned char rq_smem[];
  __shared__ float red[kRQThreads / 32];
  pdl_launch_dependents();
  pdl_wait();
  rotate_quant_row<MODE>(a, blockIdx.x, rq_smem, red, threadIdx.x, [] { __syncthreads(); });
}

// ---------------------------------------------------------------- tensor-core kernel
// Persistent: each CTA (or cluster of CTAs, for rows of more than 16 units) takes rows
// blockIdx.x / csize, + gridDim.x / csize, ...  A warp holds its unit's pairs in registers from
// the exchange to the codes; the next row's loads are issued before the exchange.
//
// Bound by the latency of its own chain of steps (35 warp instructions per 32 elements,
// half of the issue slots used: 14 to 16 warps of 128 registers an SM wait for one another
// once per row), not by HBM.  The kernel it replaced kept 64-bit integers (139 instructions).  Times, M =
// 2048, 4-bit operand planes, before -> now: K = 14336, B = 2048: 144.8 -> 57.0 us; K = 4096,
// B = 2048: 33.0 -> 17.2 us; M = 8192, K = 28672, B = 4096, 8 bits: 1907 -> 570 us; M = 64,
// same row, 4 bits: 33.8 -> 7.6 us.  At 128 registers the codes, and the planes of blocks over 2 or 4
// warps, spill nothing; planes of shorter blocks spill 16 bytes a thread, rotated fp32 rows 28 to 40.
template <int MODE, int G>
__global__ void __launch_bounds__(512, 1) rotate_mma_kernel(const RQArgs a, const int csize) {
  extern __shared__ __align__(128) uint8_t rm_smem[];
  constexpr int kBatch = 1024;       // rows between looks at the left-over ones (32 words)
  __shared__ uint32_t red[2][16];    // [row parity][warp]: fp32 bits of the largest |y|, or kRowSlow
  __shared__ uint32_t xmax[2][8];    // the same of the cluster's CTAs
  __shared__ uint32_t l1s[16];
  __shared__ uint32_t lead[2];       // [row parity]: largest |y| so far, nearly (odd log2 blocks)
  __shared__ uint32_t slow_rows[kBatch / 32];
  // A store into another CTA of the cluster needs that CTA to have started: every thread
  // arrives here, and waits while the first row's copies are on their way.
  if (csize > 1) cluster_arrive();
  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NT = blockDim.x, W = NT >> 5;
  const int rank = csize > 1 ? (int)(blockIdx.x % csize) : 0;   // one-dimensional clusters
  const int ncl = (int)gridDim.x / csize;
  const int K = a.K, K_pad = a.KB * 128;
  const UnitGeom<G> u(a, rank * W + warp, lane, MODE == kRQAct ? K_pad : K);
  uint8_t* const xu = rm_smem + warp * kUnitBytes;
  uint8_t* const stg = rm_smem + W * kUnitBytes + warp * kStageBytes;
  auto group_sync = [&] {
    if constexpr (G == 1)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / G), "n"(32 * G) : "memory");
  };
  // Maximum over the cluster's CTAs of `v` (the same in every thread of the CTA).
  int xpar = 0;
  auto cluster_max = [&](uint32_t v) -> uint32_t {
    if (csize == 1) return v;
    if (tid < csize) {
      const uint32_t at = smem_u32(&xmax[xpar][rank]);
      asm volatile(
          "{\n\t.reg .b32 r;\n\tmapa.shared::cluster.u32 r, %0, %1;\n\tst.shared::cluster.u32 [r], %2;\n\t}\n" ::"r"(at),
          "r"(tid), "r"(v)
          : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    uint32_t m = v;
    for (int i = 0; i < csize; ++i) m = max(m, xmax[xpar][i]);
    xpar ^= 1;
    return m;
  };
  uint32_t am[4];
  mma_hadamard_a(u.l, lane, am);
  const float qmaxf = (float)((1 << (a.bits - 1)) - 1);
  RowOut dst;
  dst.plane = (size_t)a.KB * a.rows_out * 128;
  dst.kb_stride = (size_t)a.rows_out * 128;
  dst.bits = MODE == kRQY ? (int)((reinterpret_cast<uintptr_t>(a.out) & 15u) == 0) : a.bits;
  auto row_out = [&](int r) {
    dst.row = r;
    dst.p = static_cast<uint8_t*>(a.out);
    if (MODE == kRQPublic) dst.p += (size_t)r * (a.bits == 4 ? K / 2 : K);
    if (MODE == kRQY) dst.p += (size_t)r * K * 4;
  };
  if (tid < 2) lead[tid] = 0u;
  if (tid < kBatch / 32) slow_rows[tid] = 0u;
  __syncthreads();

  // Batches of up to kBatch rows: all of them by the pairs, then the ones left over.
  int par = 0;
#pragma unroll 1
  for (int row0 = (int)blockIdx.x / csize; row0 < a.rows_out; row0 += kBatch * ncl) {
    bool any_slow = false;
    if (row0 < a.rows_in) unit_prefetch(a.x + (size_t)row0 * K, u.e0, u.load_end, lane, stg);
    // (the first batch: a cluster has at least one row, and its CTAs the same rows)
    if (csize > 1 && row0 == (int)blockIdx.x / csize) cluster_wait();
#pragma unroll 1
    for (int it = 0; it < kBatch; ++it, par ^= 1) {
      const int row = row0 + it * ncl;
      if (row >= a.rows_out) break;
      row_out(row);
      if (row >= a.rows_in) {   // padding row (operand planes): zero codes and scale
        if (MODE == kRQAct) {
          const float zero[4] = {0.f, 0.f, 0.f, 0.f};
          for (int k = 4 * (rank * NT + tid); k < K_pad; k += 4 * csize * NT) store_codes<kRQAct, 4>(dst, k, zero);
          if (rank == 0 && tid == 0 && a.scales != nullptr) a.scales[row] = 0.f;
        }
        continue;
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");   // the lane's own copies
      uint64_t v[32];
      const bool ok = unit_sums<G, kStageBytes, MODE == kRQY || (MODE == kRQAct && G == 1)>(
          u, [&](int j) { return *reinterpret_cast<const uint4*>(stg + 512 * j + 16 * lane); },
          [&](int k) {
            unit_to_grid(stg, reinterpret_cast<uint32_t*>(stg + kUnit * 2), a.signs, u.e0, u.load_end, k, u.wg, lane);
          },
          [&](int j, uint4& x) {
            const int o = u.e0 + unit_lane_offset(lane) + 64 * j;
            if (a.signs != nullptr && o < u.load_end) run_signs(a.signs, o, x);
          },
          am, lane, xu, l1s + warp - u.wg, stg + kUnit * 2, group_sync,
          [&] {
            if (it + 1 < kBatch && row + ncl < a.rows_in)
              unit_prefetch(a.x + (size_t)(row + ncl) * K, u.e0, u.load_end, lane, stg);
          },
          v);
      uint32_t m = MODE == kRQY ? 0u : unit_max(v, u.l, &lead[par], lane, a.c_hi, a.c_lo);
      if (!ok) m = kRowSlow;
      if (lane == 0) red[par][warp] = m;
      if (tid == 0) lead[par ^ 1] = 0u;
      __syncthreads();
      m = __reduce_max_sync(0xffffffffu, lane < W ? red[par][lane] : 0u);
      m = cluster_max(m);
      if (m == kRowSlow) {   // left for the loop below
        if (tid == 0) slow_rows[it >> 5] |= 1u << (it & 31);
        any_slow = true;
        continue;
      }
      const float amax = __uint_as_float(m);
      const float s = __fdiv_rn(amax, qmaxf);
      if (MODE != kRQY && rank == 0 && tid == 0 && a.scales != nullptr) a.scales[row] = s;
      unit_store<MODE, G>(a, u, v, amax, s, dst);
    }
    if (!any_slow) continue;
    const int k0 = UnitGeom<G>::first(a, rank * W), k1 = UnitGeom<G>::first(a, (rank + 1) * W);
#pragma unroll 1
    for (int it = 0; it < kBatch; ++it) {
      const int row = row0 + it * ncl;
      if (row >= a.rows_out) break;
      __syncthreads();
      if (!((slow_rows[it >> 5] >> (it & 31)) & 1u)) continue;
      row_out(row);
      rotate_slow_row<MODE>(a, row, k0, k1, kUnit * G, rm_smem, tid, NT, [] { __syncthreads(); }, dst, [&](float mine) {
        const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(mine));
        __syncthreads();
        if (lane == 0) red[0][warp] = wm;
        __syncthreads();
        const float rm = __uint_as_float(cluster_max(__reduce_max_sync(0xffffffffu, lane < W ? red[0][lane] : 0u)));
        if (rank == 0 && tid == 0 && a.scales != nullptr) a.scales[row] = rm > 0.f ? __fdiv_rn(rm, qmaxf) : 0.f;
        return rm;
      });
      if (MODE == kRQAct && rank == csize - 1) {
        const float zero[4] = {0.f, 0.f, 0.f, 0.f};
        for (int kz = K + 4 * tid; kz < K_pad; kz += 4 * NT) store_codes<kRQAct, 4>(dst, kz, zero);
      }
    }
    __syncthreads();
    if (tid < kBatch / 32) slow_rows[tid] = 0u;
    __syncthreads();
  }
}

int rotate_group(int K, int B, int tail) {
  const int b = K > tail ? B : tail;
  return b <= kUnit ? 1 : b / kUnit;
}

cudaError_t device_sms(int* sms) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

template <int MODE, int G>
cudaError_t launch_rotate_mma_g(const RQArgs& a, cudaStream_t s, bool pdl) {
  const int units = unit_map(a.K, a.tail, G).units;
  const int csize = ceil_div(units, 16);
  const int W = round_up(ceil_div(units, csize), G);
  // The exchange, or (64-bit integers) a block of 1024 G values; the coming row and the lists.
  const int smem = W * (kUnitBytes + kStageBytes);
  int sms = 0;
  cudaError_t e = device_sms(&sms);
  if (e == cudaSuccess) e = ensure_max_dyn_smem(rotate_mma_kernel<MODE, G>);
  if (e != cudaSuccess) return e;
  const int per_sm = std::max(1, 16 / W);   // 128 registers a thread: 16 warps an SM
  const int clusters = std::max(1, std::min(a.rows_out, sms * per_sm / csize));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * csize));
  cfg.blockDim = dim3((unsigned)(32 * W));
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pdl && pdl_allowed()) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (csize > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)csize;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = (unsigned)n;
  return cudaLaunchKernelEx(&cfg, rotate_mma_kernel<MODE, G>, a, csize);
}

template <int MODE>
cudaError_t launch_rotate_mma(const RQArgs& a, cudaStream_t s, bool pdl) {
  switch (rotate_group(a.K, a.B, a.tail)) {
    case 1: return launch_rotate_mma_g<MODE, 1>(a, s, pdl);
    case 2: return launch_rotate_mma_g<MODE, 2>(a, s, pdl);
    default: return launch_rotate_mma_g<MODE, 4>(a, s, pdl);
  }
}

size_t rotate_quant_smem(int K, int chunk) {
  (void)chunk;
  // the fp32 row, the int64 transpose chunk, and a Paley tail's character table (<= 256 B)
  return (size_t)K * sizeof(float) + (size_t)kChunkPadded * sizeof(long long) + 256;
}

cudaError_t launch_rotate_quant(RQMode mode, const RQArgs& a, cudaStream_t s, bool pdl) {
  // Activations take the tensor-core kernel; a Paley tail and the weight packer (16
  // consecutive codes a thread) the per-row kernel.
  if (a.tail_p <= 1 && rows_kernel_allowed()) {
    switch (mode) {
      case kRQPublic: return launch_rotate_mma<kRQPublic>(a, s, pdl);
      case kRQAct: return launch_rotate_mma<kRQAct>(a, s, pdl);
      case kRQY: return launch_rotate_mma<kRQY>(a, s, pdl);
      case kRQWeights: break;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.rows_out);
  cfg.blockDim = dim3(kRQThreads);
  cfg.dynamicSmemBytes = rotate_quant_smem(a.K, a.chunk);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = (pdl && pdl_allowed()) ? 1 : 0;
  auto launch = [&](void (*kernel)(const RQArgs)) {
    const cudaError_t e = ensure_max_dyn_smem(kernel);
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, kernel, a);
  };
  switch (mode) {
    case kRQPublic: return launch(rotate_quant_kernel<kRQPublic>);
    case kRQAct: return launch(rotate_quant_kernel<kRQAct>);
    case kRQY: return launch(rotate_quant_kernel<kRQY>);
    case kRQWeights: return launch(rotate_quant_kernel<kRQWeights>);
  }
  return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ public codes -> E4M3 planes
__global__ void __launch_bounds__(256) codes_to_act_kernel(const CodesArgs a) {
  const int nchunks = a.KB * 8;
  const long long total = (long long)a.M_pad * nchunks;
  const size_t plane_stride = (size_t)a.KB * a.M_pad * 128;
  for (long long idx = blockIdx.x * 256LL + threadIdx.x; idx < total; idx += (long long)gridDim.x * 256) {
    const int row = (int)(idx / nchunks);
    const int ch = (int)(idx - (long long)row * nchunks);
    const int kb = ch >> 3, j = ch & 7;
    const int k0 = ch * 16;
    uint32_t p0[4] = {0, 0, 0, 0}, p1[4] = {0, 0, 0, 0};
    if (row < a.M && k0 < a.K) {
      // K % 32 == 0, so a 16-code chunk is either fully inside K or fully padding.
      if (a.bits == 4) {
        const uint2 w = *reinterpret_cast<const uint2*>(a.codes + (size_t)row * (a.K / 2) + k0 / 2);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const uint32_t word = e < 8 ? w.x : w.y;
          int c = (int)((word >> (4 * (e & 7))) & 0xFu);
          c = c >= 8 ? c - 16 : c;
          p0[e >> 2] |= e4m3_small_int(c) << (8 * (e & 3));
        }
      } else {
        const uint4 w = *reinterpret_cast<const uint4*>(a.codes + (size_t)row * a.K + k0);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int c = (int)(int8_t)((ws[e >> 2] >> (8 * (e & 3))) & 0xFFu);
          p0[e >> 2] |= e4m3_hi_plane(c) << (8 * (e & 3));
          p1[e >> 2] |= e4m3_lo_plane(c) << (8 * (e & 3));
        }
      }
    }
    const size_t off = ((size_t)kb * a.M_pad + row) * 128 + ((j ^ (row & 7)) << 4);
    *reinterpret_cast<uint4*>(a.act + off) = make_uint4(p0[0], p0[1], p0[2], p0[3]);
    if (a.bits == 8) *reinterpret_cast<uint4*>(a.act + plane_stride + off) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
  }
}

cudaError_t launch_codes_to_act(const CodesArgs& a, cudaStream_t s) {
  const long long total = (long long)a.M_pad * a.KB * 8;
  long long blocks = (total + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  codes_to_act_kernel<<<(unsigned)blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace dptq
