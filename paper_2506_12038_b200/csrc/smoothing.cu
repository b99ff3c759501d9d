// Adaptive smoothing search (Section 3.4 of the LCD paper), offline: for every candidate migration strength alpha
// the per-channel factors s_k = xmax_k^alpha / wmax_k^(1 - alpha) and the objective
// MSE(X, Q_INT8(X / s) * s) over a calibration batch; the candidate with the smallest error wins and its 1/s_k
// are written for the online input transformation.  The level decisions use the binary32 steps of the 8-bit
// quantiser (quantize8.cu); reconstruction and sums are binary64 in a fixed order, so results are reproducible.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "common.h"
#include "device_util.h"

namespace lcd {

namespace {

constexpr int kMaxAlphas = 64;
struct AlphaList {
  int count;
  float a[kMaxAlphas];
};

// For 32 columns a CTA: xmax_k = max over the batch of |x[t][k]|, then for every candidate s[g][k] (binary64 powers, one
// rounding to binary32; zero maxima leave the channel alone; clamp to [1e-5, 1e5]) and 1 / s[g][k], which the error kernel
// would otherwise divide out once per token.  CTA 0 clears the error kernel's arrival counter.  x and wmax are read with
// ordinary loads (no __restrict__): this kernel may be running while an earlier one still writes them.  It does not let the next
// one in early, which reads the factors with __ldg, for data that nobody writes while the reading kernel runs (an early
// start gains nothing; ordinary loads there cost 8 % of the search, __ldcg 15).
__global__ void __launch_bounds__(256) smoothing_factors_kernel(const __half* x, int64_t T, int64_t K, int64_t ldx,
                                                                const float* wmax, const AlphaList alphas,
                                                                float* __restrict__ s, float* __restrict__ inv, unsigned* __restrict__ arrived) {
  __shared__ float part[8][32];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  const int64_t k = (int64_t)blockIdx.x * 32 + lane;
  if (blockIdx.x == 0 && threadIdx.x == 0) *arrived = 0u;
  float m = 0.0f;
  if (k < K) {
#pragma unroll 8
    for (int64_t t = row; t < T; t += 8) m = fmaxf(m, fabsf(__half2float(x[t * ldx + k])));
  }
  part[row][lane] = m;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 8; ++r) m = fmaxf(m, part[r][lane]);
  if (k >= K) return;
  const double xm = (double)m, wm = (double)wmax[k];
  for (int g = row; g < alphas.count; g += 8) {
    const double al = (double)alphas.a[g];
    double v = 1.0;
    if (xm > 0.0 && wm > 0.0) v = pow(xm, al) / pow(wm, 1.0 - al);
    v = fmin(fmax(v, 1e-5), 1e5);
    s[(int64_t)g * K + k] = (float)v;
    inv[(int64_t)g * K + k] = __fdiv_rn(1.0f, (float)v);
  }
}

// partial[g][t] = sum_k (x - level * s_q * s)^2 of token t under candidate g, kTokens tokens a CTA (a factor is loaded and
// widened once for all of them); the CTA that arrives last averages, picks the first smallest candidate and writes its
// factors.  Per element and candidate two multiplications, rounding by one addition, one conversion and four binary64
// operations, 22 instructions in all with the pass that finds the tokens' maxima.  128 tokens, 4096 columns, 21 candidates: 11 M of
// them are 6.5 us of issue, of 22.1 for the whole search.  No pipe is full: the factors' kernel takes 6 (a chain of binary64 powers in
// less than a CTA an SM), this one's elements 11, with half of the issue slots and half of the warps' places used and the loads
// as the longest stall, starting, the last CTA's means and the copy of the winner's factors 5.  (24.1 with a clip, two
// minimum operations, and an integer addition more; 512 x 14336 x 33: 205 and 236.)
constexpr int kTokens = 4;
// PER_SM: CTAs that an SM must hold.  Four leave all the registers the compiler wants; a grid that does not fit four times
// into the SMs is faster with five (512 tokens x 14336 columns x 33 candidates 221 -> 205 us, six 208; 128 x 4096 x 21: 24.4, 22.1
// and 22.9), a smaller one is not.  Single columns a step (rows at odd addresses) take what they want (200 x 5003 x 11: 31.7 us).
template <bool VEC, int PER_SM>
__global__ void __launch_bounds__(256, PER_SM) smoothing_error_kernel(const __half* __restrict__ x, int64_t T, int64_t K, int64_t ldx, int G,
                                                              const float* __restrict__ s, const float* __restrict__ inv,
                                                              double* __restrict__ partial, unsigned* __restrict__ arrived,
                                                              double* __restrict__ mse, int32_t* __restrict__ best, float* __restrict__ inv_smooth) {
  constexpr int W = VEC ? 8 : 1;          // columns a thread takes at once
  __shared__ float s_f[kTokens][8];
  __shared__ double s_d[kTokens][8];
  __shared__ double s_mse[kMaxAlphas];
  __shared__ int s_best, s_last;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t t0 = (int64_t)blockIdx.x * kTokens;
  const int g = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_tok = (int)(T - t0 < kTokens ? T - t0 : kTokens);
  const __half* xr = x + t0 * ldx;
  const float *sg = s + (int64_t)g * K, *ig = inv + (int64_t)g * K;
  auto columns = [&](const float* p, int64_t k, float (&f)[W]) {
    if constexpr (VEC) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(p + k)), b = __ldg(reinterpret_cast<const float4*>(p + k) + 1);
      f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
    } else {
      f[0] = __ldg(p + k);
    }
  };
  auto activations = [&](int t, int64_t k, float (&f)[W]) {
    if constexpr (VEC) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(xr + t * ldx + k));
      const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 p = __half22float2(h[i]);
        f[2 * i] = p.x;
        f[2 * i + 1] = p.y;
      }
    } else {
      f[0] = __half2float(xr[t * ldx + k]);
    }
  };
  float amax[kTokens] = {};
  for (int64_t k = (int64_t)tid * W; k < K; k += 256 * W) {
    float iv[W];
    columns(ig, k, iv);
#pragma unroll
    for (int t = 0; t < kTokens; ++t)
      if (t < n_tok) {
        float xv[W];
        activations(t, k, xv);
#pragma unroll
        for (int i = 0; i < W; ++i) amax[t] = fmaxf(amax[t], fabsf(__fmul_rn(xv[i], iv[i])));
      }
  }
#pragma unroll
  for (int t = 0; t < kTokens; ++t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax[t] = fmaxf(amax[t], __shfl_xor_sync(0xffffffffu, amax[t], o));
    if (lane == 0) s_f[t][warp] = amax[t];
  }
  __syncthreads();
  float r[kTokens];
  double sq[kTokens], err[kTokens] = {};
  bool finite = true;
#pragma unroll
  for (int t = 0; t < kTokens; ++t) {
    float A = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) A = fmaxf(A, s_f[t][w]);
    finite = finite && A < 3e38f;
    r[t] = A > 0.0f ? __fdiv_rn(127.0f, A) : 0.0f;
    sq[t] = A > 0.0f ? (double)__fdiv_rn(A, 127.0f) : 1.0;
  }
  // |x / s| * (127 / A) is at most 127 and a rounding: clipping changes nothing where A is finite
  auto errors = [&](auto clip) {
    for (int64_t k = (int64_t)tid * W; k < K; k += 256 * W) {
      float iv[W], sv[W];
      columns(ig, k, iv);
      columns(sg, k, sv);
      double sd[W];
#pragma unroll
      for (int i = 0; i < W; ++i) sd[i] = (double)sv[i];
#pragma unroll
      for (int t = 0; t < kTokens; ++t)
        if (t < n_tok) {
          float xv[W];
          activations(t, k, xv);
#pragma unroll
          for (int i = 0; i < W; ++i) {
            // clipped first (the bounds are integers: the same level), then rounded half to even by one addition, which leaves
            // the level in the sum's low bits; under the exponent of 2^52 the sum's bits are the level and a constant, binary64
            const float v = __fmul_rn(__fmul_rn(xv[i], iv[i]), r[t]), u = decltype(clip)::value ? fminf(fmaxf(v, -128.0f), 127.0f) : v;
            const int bits = (int)__float_as_uint(__fadd_rn(u, 12582912.0f));                 // 0x4b400000 + level
            const double lev = __hiloint2double(0x43300000, bits) - (4503599627370496.0 + 1262485504.0);
            const double d = (double)xv[i] - lev * sq[t] * sd[i];
            err[t] += d * d;
          }
        }
    }
  };
  if (finite) errors(std::false_type()); else errors(std::true_type());
#pragma unroll
  for (int t = 0; t < kTokens; ++t) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) err[t] += __shfl_xor_sync(0xffffffffu, err[t], o);
    if (lane == 0) s_d[t][warp] = err[t];
  }
  __syncthreads();
  if (tid < n_tok) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += s_d[tid][w];
    __stcg(partial + (int64_t)g * T + t0 + tid, v);
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(arrived, 1u) == gridDim.x * gridDim.y - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // a warp per candidate: the lanes' tokens in order, then the lanes
  for (int c = warp; c < G; c += 8) {
    const double* p = partial + (int64_t)c * T;
    double v = 0.0;
#pragma unroll 4
    for (int64_t t = lane; t < T; t += 32) v += __ldcg(p + t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) {
      v /= (double)T * (double)K;
      s_mse[c] = v;
      mse[c] = v;
    }
  }
  __syncthreads();
  if (warp == 0) {          // the first of the smallest
    int b = lane < G ? lane : 0;
    if (lane + 32 < G && s_mse[lane + 32] < s_mse[b]) b = lane + 32;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const int other = __shfl_xor_sync(0xffffffffu, b, o);
      if (s_mse[other] < s_mse[b] || (s_mse[other] == s_mse[b] && other < b)) b = other;
    }
    if (lane == 0) {
      s_best = b;
      if (best) *best = b;
    }
  }
  __syncthreads();
  if (inv_smooth) {
    const float* from = inv + (int64_t)s_best * K;
#pragma unroll 8
    for (int64_t k = tid; k < K; k += 256) inv_smooth[k] = __ldg(from + k);
  }
}

size_t align256s(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

// factors | reciprocal factors | errors per candidate and token | arrival counter
size_t smoothing_search_workspace_bytes(int64_t T, int64_t K, int G) {
  return 2 * align256s((size_t)G * K * sizeof(float)) + align256s((size_t)G * T * sizeof(double)) + 256;
}

lcd_status launch_smoothing_search(const void* x, int64_t T, int64_t K, int64_t ldx, const float* wmax, const float* alphas_host,
                                   int G, void* workspace, double* mse, int32_t* best, float* inv_smooth, void* stream) {
  AlphaList al;
  al.count = G;
  for (int i = 0; i < kMaxAlphas; ++i) al.a[i] = i < G ? alphas_host[i] : 0.0f;
  uint8_t* base = static_cast<uint8_t*>(workspace);
  const size_t factors = align256s((size_t)G * K * sizeof(float));
  float* s = reinterpret_cast<float*>(base);
  float* inv = reinterpret_cast<float*>(base + factors);
  double* partial = reinterpret_cast<double*>(base + 2 * factors);
  unsigned* arrived = reinterpret_cast<unsigned*>(base + 2 * factors + align256s((size_t)G * T * sizeof(double)));
  const __half* xh = static_cast<const __half*>(x);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((K + 31) / 32));
  cfg.blockDim = dim3(256);
  cfg.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, smoothing_factors_kernel, xh, T, K, ldx, wmax, al, s, inv, arrived);
  if (e == cudaSuccess) {
    // rows of x start on 16 bytes (the rows of the factors do where K is a multiple of four)
    const bool vec = K % 8 == 0 && ldx % 8 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
    cfg.gridDim = dim3((unsigned)((T + kTokens - 1) / kTokens), (unsigned)G);
    const bool many = (uint64_t)cfg.gridDim.x * cfg.gridDim.y > 4ull * (uint64_t)current_sm_count();
    auto kern = !vec ? smoothing_error_kernel<false, 1> : many ? smoothing_error_kernel<true, 5> : smoothing_error_kernel<true, 4>;
    e = cudaLaunchKernelEx(&cfg, kern, xh, T, K, ldx, G, (const float*)s, (const float*)inv, partial, arrived, mse, best, inv_smooth);
  }
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  return LCD_OK;
}

}  // namespace lcd
