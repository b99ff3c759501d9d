// Reclassification of weights and centroid offsets (Section 3.2 of the LCD paper), offline bookkeeping after a
// round of weight updates, for per-row codebooks sorted in ascending order:
//   a weight of cluster i with update dw moves to i - 1 when dw < -(C_i - C_{i-1}) / 2, to i + 1 when
//   dw > (C_{i+1} - C_i) / 2 (binary32: one subtraction, one halving; edge clusters have one side);
//   dC_j = sum over the weights that end up in j of (dw + (C_old - C_j)), counts alongside.
// One CTA per row; per-thread binary64 sums, combined in a fixed order: results are reproducible.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "common.h"
#include "device_util.h"

namespace lcd {

namespace {

constexpr int kRcThreads = 256;
constexpr int kRcMaxC = 16;

// AHEAD: the first step's loads are on their way before the thresholds are made.
template <int CMAX, bool AHEAD>
__global__ void __launch_bounds__(kRcThreads) reclassify_kernel(const uint8_t* __restrict__ idx, const uint16_t* __restrict__ codebook,
                                                                const float* __restrict__ delta_w, int64_t K, int64_t ldw, int C,
                                                                uint8_t* __restrict__ new_idx, double* __restrict__ delta_c,
                                                                int32_t* __restrict__ counts, const bool vec) {
  __shared__ float s_c[CMAX];
  __shared__ double2 s_step[CMAX];          // C_i - C_{i-1} and C_i - C_{i+1}: what a weight of cluster i that moves brings along
  __shared__ int s_total[3][4];             // packed counts of the CTA
  __shared__ float2 s_gap[CMAX];            // half-gaps (C_i - C_{i-1}) / 2 and (C_{i+1} - C_i) / 2, infinite at the edges
  const int64_t n = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint8_t* ir = idx + n * K;
  const float* dr = delta_w + n * ldw;
  uint8_t* outr = new_idx + n * K;
  // 16 weights per thread and step: one 16-byte index load, four 16-byte update loads, one 16-byte store
  uint4 iv = make_uint4(0u, 0u, 0u, 0u);
  float4 d[4];
  auto load = [&](int64_t k) {
    if (k >= K) return;
    iv = __ldg(reinterpret_cast<const uint4*>(ir + k));
#pragma unroll
    for (int q = 0; q < 4; ++q) d[q] = __ldg(reinterpret_cast<const float4*>(dr + k + 4 * q));
  };
  if (AHEAD && vec) load((int64_t)tid * 16);
  if (tid < 12) s_total[tid >> 2][tid & 3] = 0;
  if (tid < C) s_c[tid] = __half2float(__ushort_as_half(codebook[n * C + tid]));
  __syncthreads();
  if (tid < CMAX) {
    const float inf = __int_as_float(0x7f800000);
    s_gap[tid] = make_float2((tid > 0 && tid < C) ? __fmul_rn(__fsub_rn(s_c[tid], s_c[tid - 1]), 0.5f) : inf,
                             (tid < C - 1) ? __fmul_rn(__fsub_rn(s_c[tid + 1], s_c[tid]), 0.5f) : inf);
  }
  // Per thread and cluster, in the thread's own column of shared memory (indexed by the data-dependent cluster; a register
  // array would need one predicated copy of every operation per cluster): the binary64 sum of the arriving updates.  Members
  // and arrivals from either side are counted, the arrivals' centroid differences added at the end from the counts: up to
  // four clusters in bytes of three registers, emptied in time into a count per lane (4 bits of cluster and kind), up to
  // eight in shared memory.  With more the counts' space would halve the CTAs on an SM: there the differences are added
  // weight by weight and only the members are counted.  The load/store data pipe is what the kernel fills most (70 % busy, 55 %
  // of the warps resident at 42 registers): a weight takes six passes through it here (thirteen when a slot of sixteen bytes
  // held an error-free binary32 pair and the counts).  4096 x 4096, 4 / 8 / 16 clusters: 32.8 / 47 / 55 us (43 / 56 / 89 then).
  extern __shared__ double s_sum[];                                             // [CMAX][kRcThreads]
  constexpr bool kPacked = CMAX <= 4, kSteps = CMAX > 8;
  int* s_count = reinterpret_cast<int*>(s_sum + CMAX * kRcThreads);             // [1 or 3][CMAX][kRcThreads]: members, from left, from right
#pragma unroll
  for (int c = 0; c < CMAX; ++c) {
    s_sum[c * kRcThreads + tid] = 0.0;
    if (!kPacked) {
#pragma unroll
      for (int f = 0; f < (kSteps ? 1 : 3); ++f) s_count[(f * CMAX + c) * kRcThreads + tid] = 0;
    }
  }
  if (kSteps && tid < CMAX)
    s_step[tid] = make_double2((tid > 0 && tid < C) ? (double)s_c[tid] - (double)s_c[tid - 1] : 0.0,
                               (tid < C - 1) ? (double)s_c[tid] - (double)s_c[tid + 1] : 0.0);
  __syncthreads();
  uint32_t members = 0, from_left = 0, from_right = 0;
  // An index is reduced to the table size CMAX before it addresses shared memory, so a byte >= C (the caller's
  // error) cannot reach outside the slots: such a weight keeps its reduced index and is counted in no cluster.
  auto one = [&](int i, float dw) {
    const float2 gap = s_gap[i];
    const bool left = dw < -gap.x, right = !left && dw > gap.y;
    const int j = i - (left ? 1 : 0) + (right ? 1 : 0);
    double d = (double)dw;
    if (kSteps && (left || right)) {
      const double2 step = s_step[i];
      d += left ? step.x : step.y;
    }
    s_sum[j * kRcThreads + tid] += d;
    if (kPacked) {
      const uint32_t one_j = 1u << (8 * j);
      members += one_j;
      from_left += right ? one_j : 0u;
      from_right += left ? one_j : 0u;
    } else {
      int* at = s_count + j * kRcThreads + tid;
      atomicAdd(at, 1);
      if (!kSteps) {
        if (right) atomicAdd(at + CMAX * kRcThreads, 1);
        if (left) atomicAdd(at + 2 * CMAX * kRcThreads, 1);
      }
    }
    return (uint32_t)j;
  };
  int total = 0;      // packed: lane 4 f + c: this warp's members (f = 0) of cluster c, arrivals from the left, from the right
  auto empty = [&]() {
    if (kPacked) {
      const uint32_t w[3] = {members, from_left, from_right};
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        // bytes of the lanes' words, at most 255 each, summed in 16-bit fields
        const uint32_t even = __reduce_add_sync(0xffffffffu, w[f] & 0x00ff00ffu), odd = __reduce_add_sync(0xffffffffu, (w[f] >> 8) & 0x00ff00ffu);
        if ((lane >> 2) == f) total += (int)((((lane & 1) ? odd : even) >> ((lane & 2) ? 16 : 0)) & 0xffffu);
      }
      members = from_left = from_right = 0;
    }
  };
  int step = 0;
  if (vec) {
    for (int64_t k0 = 0; k0 < K; k0 += (int64_t)kRcThreads * 16) {
      if (kPacked && ++step == 16) { empty(); step = 1; }           // 240 weights since: no byte has overflowed
      const int64_t k = k0 + (int64_t)tid * 16;
      if (k >= K) continue;
      if (!AHEAD || k0 > 0) load(k);
      const uint32_t iw[4] = {iv.x, iv.y, iv.z, iv.w};
      uint32_t ow[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float dv[4] = {d[q].x, d[q].y, d[q].z, d[q].w};
        uint32_t o = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) o |= one((int)((iw[q] >> (8 * e)) & (uint32_t)(CMAX - 1)), dv[e]) << (8 * e);
        ow[q] = o;
      }
      *reinterpret_cast<uint4*>(outr + k) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
    }
  } else {
    // rows at any alignment: kRun weights' loads in flight together (one after the other, with the counts' emptying in between,
    // 5056 x 7606, 8 clusters, took 158 us, 92 so; 4802 x 6873, 4 clusters 134 and 72)
    constexpr int kRun = kPacked ? 4 : 8;          // (what the registers of the way above leave)
    for (int64_t k0 = 0; k0 < K; k0 += kRun * kRcThreads) {
      if (kPacked && (step += kRun) > 255) { empty(); step = kRun; }
      const int64_t k = k0 + tid;
      int i[kRun];
      float dw[kRun];
#pragma unroll
      for (int e = 0; e < kRun; ++e)
        if (k + e * kRcThreads < K) {
          i[e] = __ldg(ir + k + e * kRcThreads) & (CMAX - 1);
          dw[e] = __ldg(dr + k + e * kRcThreads);
        }
#pragma unroll
      for (int e = 0; e < kRun; ++e)
        if (k + e * kRcThreads < K) outr[k + e * kRcThreads] = (uint8_t)one(i[e], dw[e]);
    }
  }
  empty();
  if (kPacked && lane < 12) atomicAdd(&s_total[lane >> 2][lane & 3], total);
  // A warp folds the 256 columns of slots of every eighth cluster: each lane adds its eight columns, then a butterfly over
  // the lanes (a butterfly in every warp over its own columns costs as much as the row's weights).
  __syncthreads();
  for (int c = warp; c < C; c += kRcThreads / 32) {
    double sum = 0.0;
    int q = 0, fl = 0, fr = 0;
#pragma unroll
    for (int w = 0; w < kRcThreads / 32; ++w) {
      const int at = c * kRcThreads + w * 32 + lane;
      sum += s_sum[at];
      if (!kPacked) q += s_count[at];
      if (!kPacked && !kSteps) {
        fl += s_count[CMAX * kRcThreads + at];
        fr += s_count[2 * CMAX * kRcThreads + at];
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (!kPacked) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (!kPacked && !kSteps) {
        fl += __shfl_xor_sync(0xffffffffu, fl, o);
        fr += __shfl_xor_sync(0xffffffffu, fr, o);
      }
    }
    if (kPacked) {
      q = s_total[0][c & 3];
      fl = s_total[1][c & 3];
      fr = s_total[2][c & 3];
    }
    if (lane == 0) {
      if (c > 0) sum += (double)fl * ((double)s_c[c - 1] - (double)s_c[c]);
      if (c < C - 1) sum += (double)fr * ((double)s_c[c + 1] - (double)s_c[c]);
      delta_c[n * C + c] = sum;
      counts[n * C + c] = q;
    }
  }
}

template <int CMAX, bool AHEAD = false>
lcd_status launch_rows(const uint8_t* idx, const uint16_t* codebook, const float* delta_w, int64_t N, int64_t K, int64_t ldw, int C,
                       uint8_t* new_idx, double* delta_c, int32_t* counts, bool vec, cudaStream_t s) {
  auto kern = reclassify_kernel<CMAX, AHEAD>;
  constexpr int smem = CMAX * kRcThreads * (CMAX <= 4 ? 8 : CMAX <= 8 ? 20 : 12);
  if (smem > 40 * 1024) {             // (with the static tables more than the 48 KB that need no opt-in)
    static PerDeviceFlag attr_set;    // needs the opt-in, on every device
    int dev;
    if (attr_set.first(&dev)) {
      const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (ea != cudaSuccess) { set_cuda_error((int)ea); return LCD_ERR_CUDA; }
      attr_set.done(dev);
    }
  }
  kern<<<(unsigned)N, kRcThreads, smem, s>>>(idx, codebook, delta_w, K, ldw, C, new_idx, delta_c, counts, vec);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  return LCD_OK;
}

}  // namespace

lcd_status launch_reclassify(const uint8_t* idx, const uint16_t* codebook, const float* delta_w, int64_t N, int64_t K,
                             int64_t ldw, int C, uint8_t* new_idx, double* delta_c, int32_t* counts, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const bool vec = K % 16 == 0 && ldw % 4 == 0 && al16(idx) && al16(delta_w) && al16(new_idx);
  if (C <= 4) return launch_rows<4>(idx, codebook, delta_w, N, K, ldw, C, new_idx, delta_c, counts, vec, s);
  if (C <= 8) return launch_rows<8>(idx, codebook, delta_w, N, K, ldw, C, new_idx, delta_c, counts, vec, s);
  // Above eight clusters shared memory holds few CTAs an SM: the loads go ahead (4096 x 4096, 10 / 16 clusters 55.3 / 59.4 -> 51.0 /
  // 55.4 us, 777 x 8192, 10 clusters 24.6 -> 22.2), but on short rows, of which a part of the CTA takes one step, the registers for it
  // cost more (512 x 512 / 1024, 16 clusters 6.7 / 7.6 -> 7.2 / 8.2; 512 x 2048 8.2 either way), as they do with fewer clusters (8192
  // x 8192, 4 clusters 99.2 -> 102.5).
  if (K >= 2048) return launch_rows<kRcMaxC, true>(idx, codebook, delta_w, N, K, ldw, C, new_idx, delta_c, counts, vec, s);
  return launch_rows<kRcMaxC>(idx, codebook, delta_w, N, K, ldw, C, new_idx, delta_c, counts, vec, s);
}

}  // namespace lcd
