// Density-based centroid initialisation (DBCI, Section 3.1 of the LCD paper), offline, on a flat array of weights:
// sort; sigma from six nearest-rank percentiles; two seed clusters around the extreme weights; MinPts and eps from
// them; DBSCAN on the rest; lower medians.  On sorted one-dimensional data DBSCAN is local: a point's neighbours are its
// neighbours in the array, core points chain into one cluster while the gap to the core point before is at most eps, and
// another point needs the nearest core point on either side.  So two passes over the sorted array do it: one marks
// the core points and sums up every tile (first and last core point, gaps between), one writes the labels, with a scan
// over the tiles in either direction between them: what lies before a word of 32 points and the first core point after it
// are then known, and no point looks at another one, however many share its value (walking out to the core points takes up
// to MinPts steps a point: 400 K weights on eight values 107 ms, 0.2 so).  A tile without gaps or non-core points, nearly every
// one, is written without being read again, and where 4096 weights span less than eps two of them tell so: little more than the
// labels' 4 bytes a weight is moved.  45 M weights, after the sort: 100 us (bound by the labels, 45; 160 with a CTA a tile, a scan
// that reads its tiles one after the other and a pair of atomics for every 32 points).
// The sort is dbci_sort.cu's, or CUB's for arrays beyond what that takes.  All comparisons and the few scalar operations
// are binary64 on the binary32 data, so every decision has one right answer.
#include <cuda_runtime.h>

#include <cub/device/device_radix_sort.cuh>

#include "common.h"
#include "dbci_sort.h"
#include "device_util.h"

namespace lcd {

namespace {

// The kernels start while the one before them ends and wait for it here; what that one writes they read with ordinary loads.
__device__ __forceinline__ void wait_for_last_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

struct DbciParams {        // device-side scalars shared by the kernels; mirrored into lcd_dbci_result at the end
  double sigma, eps;
  long long L, R;          // left cluster = sorted [0, L), right cluster = [R, n)
  long long min_pts;
  int n_mid;               // clusters found among the middle points
  int n_noise;
};

// First index in [lo, hi) whose value is >= v (strict: > v), by a warp: 32 probes a step instead of one.  NEAR: the 32 values at
// the beginning (1) or at the end (-1) first: the weights near an extreme one are usually few.
template <bool STRICT, int NEAR = 0>
__device__ long long warp_bound(const float* x, long long lo, long long hi, double v) {
  const int lane = threadIdx.x & 31;
  if (NEAR != 0 && hi - lo > 32) {
    const long long a = NEAR > 0 ? lo : hi - 32;
    const bool before = STRICT ? (double)x[a + lane] <= v : (double)x[a + lane] < v;
    const int n = 32 - __clz(__ballot_sync(0xffffffffu, before));
    if (NEAR > 0) {
      if (n < 32) return a + n;
      lo = a + 32;
    } else {
      if (n > 0) return a + n;
      hi = a;
    }
  }
  while (lo < hi) {
    const long long step = (hi - lo + 31) / 32, at = lo + lane * step;
    bool before = false;
    if (at < hi) before = STRICT ? (double)x[at] <= v : (double)x[at] < v;
    // probes 0 .. n - 1 lie before the bound (the last that says so counts: NaNs sorted to the front compare false)
    const int n = 32 - __clz(__ballot_sync(0xffffffffu, before));
    if (n == 0) return lo;
    lo += (n - 1) * step + 1;
    const long long end = lo + step - 1;
    hi = end < hi ? end : hi;
  }
  return lo;
}

// All CTAs clear the clusters' first and last members (a list as long as the caller wants), two warps of CTA 0 do the rest.
__global__ void __launch_bounds__(256) dbci_params_kernel(const float* x, long long n, DbciParams* P,
                                                          int* first, int* last, int max_clusters) {
  wait_for_last_kernel();
  let_next_kernel_start();
  __shared__ long long found[2];
  __shared__ double sigma_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < max_clusters; i += gridDim.x * 256) { first[i] = 0x7fffffff; last[i] = -1; }
  if (blockIdx.x != 0) return;
  if (warp < 2) {
    const long long at = warp == 0 ? warp_bound<true>(x, 0, n, 0.0) : warp_bound<false>(x, 0, n, 0.0);
    if (lane == 0) found[warp] = at;
  }
  __syncthreads();
  if (warp == 0) {
    const long long first_pos = found[0], end_neg = found[1];     // positives: [first_pos, n); negatives: [0, end_neg)
    const long long n_pos = n - first_pos, n_neg = end_neg;
    // lanes 0, 2, 4: percentiles of the positive weights, lanes 1, 3, 5: of the magnitudes of the negative ones
    const double pct[3] = {0.6827, 0.9544, 0.9974};
    double value = 0.0;
    if (lane < 6) {
      const long long cnt = (lane & 1) ? n_neg : n_pos;
      if (cnt > 0) {
        long long k = (long long)ceil(pct[lane >> 1] * (double)cnt) - 1;
        k = k < 0 ? 0 : (k > cnt - 1 ? cnt - 1 : k);
        value = (lane & 1) ? -(double)x[end_neg - 1 - k] : (double)x[first_pos + k];
      }
    }
    double sum = 0.0;
    for (int i = 0; i < 6; ++i) sum += __shfl_sync(0xffffffffu, value, i);
    if (lane == 0) sigma_s = sum / 12.0;
  }
  __syncthreads();
  const double sigma = sigma_s;
  if (warp < 2) {
    const long long at = warp == 0 ? warp_bound<true, 1>(x, 0, n, (double)x[0] + sigma) : warp_bound<false, -1>(x, 0, n, (double)x[n - 1] - sigma);
    if (lane == 0) found[warp] = at;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long L = found[0];
    long long R = found[1];
    if (R < L) R = L;
    const long long min_pts = (n - R > 0) ? (L < n - R ? L : n - R) : L;
    P->sigma = sigma;
    P->eps = sigma / (double)min_pts;
    P->L = L;
    P->R = R;
    P->min_pts = min_pts;
    P->n_mid = 0;
    P->n_noise = 0;
  }
}

// ---- tiles ----------------------------------------------------------------------------------------------
// A tile is 4096 sorted points; warp w of a CTA has its points [512 w, 512 w + 512), 32 at a time.
constexpr int kTile = 4096, kTileWarps = 8, kWarpSteps = kTile / (32 * kTileWarps);

// The core points of a stretch: whether there are any, the values of the first and the last, and the gaps wider than eps
// between neighbouring ones.
struct Chain {
  float first, last;
  int any, gaps;
};
// The first core point of a tile, later the first one after it; whether there is one.
struct Next {
  float v;
  int any;
};
__device__ __forceinline__ bool gap_after(float before, float at, double eps) { return (double)at - (double)before > eps; }
__device__ __forceinline__ Chain join(const Chain& a, const Chain& b, double eps) {
  if (!a.any) return b;
  if (!b.any) return a;
  return {a.first, b.last, 1, a.gaps + b.gaps + (gap_after(a.last, b.first, eps) ? 1 : 0)};
}

// Where the neighbours of a tile's points may begin and end, places relative to the tile: the first neighbour of any of them lies
// in [lo0, lo1] (or is the point itself), the first point past the neighbours in [hi0, hi1].
struct Reach {
  int lo0, lo1, hi0, hi1;
};
// Whether each of N middle points is a core point: at least k points y of the middle with v - eps <= y <= v + eps (binary64).
// A binary32 y is >= a binary64 bound exactly if it is >= the bound rounded up to binary32, and likewise on the other side.
// Places are relative to the tile: at(i) is the point, [L, R) the middle, r[j] the places (all in the middle where `in` says so).
// The N searches take their steps together (one after the other, 16 a warp, they were most of a tile's 20 us), over at most
// `most` places.
template <int N, typename At>
__device__ __forceinline__ void are_core(const At& at, long long L, long long R, const Reach& reach, int most, const int (&r)[N], const float (&v)[N],
                                         const bool (&in)[N], double eps, long long k, unsigned (&word)[N]) {
  bool yes[N], open = false;
#pragma unroll
  for (int j = 0; j < N; ++j) yes[j] = in[j] && k <= 1;      // itself (and k = 0: an empty seed cluster, left by a NaN weight)
  if (k > 1) {
    float a[N], b[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      a[j] = __double2float_ru((double)v[j] - eps);
      b[j] = __double2float_rd((double)v[j] + eps);
      // k - 1 neighbours on one side, the usual case
      if (in[j]) yes[j] = (r[j] - (k - 1) >= L && at((int)(r[j] - (k - 1))) >= a[j]) || (r[j] + (k - 1) < R && at((int)(r[j] + (k - 1))) <= b[j]);
      open = open || (in[j] && !yes[j]);
    }
    if (__any_sync(0xffffffffu, open)) {
      int left[N], stop[N], right[N], end[N];                // first neighbour in [left, stop]; first point past them in [right, end]
#pragma unroll
      for (int j = 0; j < N; ++j) {
        left[j] = in[j] ? (int)(r[j] - (k - 1) > reach.lo0 ? r[j] - (k - 1) : reach.lo0) : r[j];
        stop[j] = in[j] ? min(r[j], reach.lo1) : r[j];
        right[j] = in[j] ? max(r[j], reach.hi0) : r[j];
        end[j] = in[j] ? (int)(r[j] + (k - 1) < reach.hi1 ? r[j] + (k - 1) : reach.hi1) : r[j];
      }
      for (int s = most > 0 ? 1 << (31 - __clz(most)) : 0; s > 0; s >>= 1) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
          if (left[j] + s <= stop[j] && at(left[j] + s - 1) < a[j]) left[j] += s;
          if (right[j] + s <= end[j] && at(right[j] + s - 1) <= b[j]) right[j] += s;
        }
      }
#pragma unroll
      for (int j = 0; j < N; ++j) yes[j] = in[j] && (yes[j] || right[j] - left[j] >= k);
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j) word[j] = __ballot_sync(0xffffffffu, yes[j]);
}

// The chain of a warp's 32 points: `word` their core flags, v the lane's value.
__device__ __forceinline__ Chain word_chain(unsigned word, float v, double eps) {
  if (word == 0) return {0.0f, 0.0f, 0, 0};
  const int lane = threadIdx.x & 31;
  const unsigned below = word & ((1u << lane) - 1u);
  const int before = below ? 31 - __clz(below) : lane;
  const float vb = __shfl_sync(0xffffffffu, v, before);
  const bool gap = ((word >> lane) & 1u) && below && (double)v - (double)vb > eps;
  return {__shfl_sync(0xffffffffu, v, __ffs(word) - 1), __shfl_sync(0xffffffffu, v, 31 - __clz(word)), 1,
          __popc(__ballot_sync(0xffffffffu, gap))};
}

// A CTA has up to kTileWarps tiles, n_ctas apart (the tiles that are not plain lie together, at the ends of the array), here and
// when the labels are written: a warp per tile looks whether the tile is plain, the CTA goes through the tiles that are not.
// Where the k - 1 points before and after a tile are few, all that are_core looks at is fetched at once.  Where they are many
// (few values, or a uniform distribution: the seed clusters are a large part of the array), the neighbours of the tile's first and
// last point are looked up: no other point has them beyond those, so a tile where these two reach over fewer than k points has no
// core point, nearly every one then, and in the others the searches are short (45 M weights clipped at 2.5 sigma, k = 2.6 M: 40 us;
// searches of every point over k points 1640, with their steps together 2460).
constexpr int kReach = 1024;
__global__ void __launch_bounds__(32 * kTileWarps) dbci_mark_kernel(const float* x, long long n, const DbciParams* P, int n_tiles, unsigned* core,
                                                                    Chain* chains, Next* next, unsigned char* plain) {
  __shared__ Chain part[kTileWarps];
  __shared__ int all[kTileWarps], is_plain[kTileWarps];
  __shared__ float window[kReach + kTile + kReach];
  __shared__ long long bound[4];             // of the tile's first and last point: first neighbour, first point past the neighbours
  wait_for_last_kernel();
  let_next_kernel_start();
  const long long L = P->L, R = P->R, k = P->min_pts;
  const double eps = P->eps;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // A whole tile at once: if its last value and the (k - 1)-th before its first lie within eps of each other, every point has
  // k - 1 neighbours on its left and no two neighbours a gap between them (subtraction and rounding are monotone).
  const int my_tile = blockIdx.x + warp * gridDim.x;
  if (my_tile < n_tiles) {
    const long long tile0 = (long long)my_tile * kTile;
    bool p = false;
    if (tile0 - (k - 1) >= L && tile0 + kTile <= R) {
      const float low = x[tile0 - (k - 1)], at = x[tile0], high = x[tile0 + kTile - 1];
      if (low >= __double2float_ru((double)high - eps) && !gap_after(low, high, eps)) {
        p = true;
        if (lane == 0) {
          chains[my_tile] = {at, high, 1, 0};
          next[my_tile] = {at, 1};
          plain[my_tile] = 1;
        }
      }
    }
    if (lane == 0) is_plain[warp] = p;
  }
  __syncthreads();
  for (int i = 0; i < kTileWarps; ++i) {
    const int tile = blockIdx.x + i * gridDim.x;
    if (tile >= n_tiles) break;
    if (is_plain[i]) continue;
    const long long tile0 = (long long)tile * kTile;
    const long long reach = k > 1 ? k - 1 : 0;
    const bool near = reach <= kReach;
    if (near) {
      const long long from = tile0 - reach > 0 ? tile0 - reach : 0, to = tile0 + kTile + reach < n ? tile0 + kTile + reach : n;
#pragma unroll 8
      for (long long g = from + threadIdx.x; g < to; g += 32 * kTileWarps) window[g - tile0 + kReach] = x[g];
      __syncthreads();
    }
    Reach all_of = {(int)(L - tile0), kTile, 0, (int)(R - tile0)};
    int most = (int)reach;
    bool none = false;
    if (!near) {
      const long long p0 = tile0 > L ? tile0 : L, p1 = (tile0 + kTile < R ? tile0 + kTile : R) - 1;
      none = p0 > p1;                             // no point of the middle
      if (!none) {
        if (warp < 4) {
          const long long p = (warp & 1) ? p1 : p0;
          const double v = (double)x[p];
          const long long at = warp < 2 ? warp_bound<false, -1>(x, p - reach > L ? p - reach : L, p, v - eps)
                                        : warp_bound<true, 1>(x, p, p + reach < R ? p + reach : R, v + eps);
          if (lane == 0) bound[warp] = at;
        }
        __syncthreads();
        all_of = {(int)(bound[0] - tile0), (int)(bound[1] - tile0), (int)(bound[2] - tile0), (int)(bound[3] - tile0)};
        most = max(all_of.lo1 - all_of.lo0, all_of.hi1 - all_of.hi0);
        none = bound[3] - bound[0] < k;
      }
    }
    Chain mine = {0.0f, 0.0f, 0, 0};
    bool every = true;
    auto words = [&](auto at) {
      constexpr int N = 4;
#pragma unroll 1
      for (int j0 = 0; j0 < kWarpSteps; j0 += N) {
        int r[N];
        float v[N];
        bool in[N];
        unsigned word[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
          r[j] = warp * (32 * kWarpSteps) + 32 * (j0 + j) + lane;
          v[j] = tile0 + r[j] < n ? at(r[j]) : 0.0f;
          in[j] = tile0 + r[j] >= L && tile0 + r[j] < R;
        }
        are_core<N>(at, L - tile0, R - tile0, all_of, most, r, v, in, eps, k, word);
#pragma unroll
        for (int j = 0; j < N; ++j) {
          if (lane == 0 && tile0 + r[j] < n) core[(tile0 + r[j]) >> 5] = word[j];
          every = every && word[j] == 0xffffffffu;
          mine = join(mine, word_chain(word[j], v[j], eps), eps);
        }
      }
    };
    if (none) {
      every = false;
      if (threadIdx.x < kTile / 32 && tile0 + 32 * threadIdx.x < n) core[(tile0 >> 5) + threadIdx.x] = 0u;
    } else if (near) {
      words([&](int i) { return window[i + kReach]; });
    } else {
      words([&](int i) { return x[tile0 + i]; });
    }
    if (lane == 0) {
      part[warp] = mine;
      all[warp] = every;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      Chain t = part[0];
      int e = all[0];
      for (int w = 1; w < kTileWarps; ++w) {
        t = join(t, part[w], eps);
        e = e && all[w];
      }
      chains[tile] = t;
      next[tile] = {t.first, t.any};
      plain[tile] = (unsigned char)(e && t.gaps == 0);
    }
    __syncthreads();
  }
}

// Exclusive scans over the tiles in place, by one CTA each, a warp a stretch of tiles, 32 at a time.  CTA 0: chains[t] becomes the
// chain of all tiles before t; the warps scan their stretches, then put what lies before a stretch in front.  CTA 1: next[t]
// becomes the first core point of all tiles after t.  The loads of kBatch steps are under way together.
constexpr int kBatch = 4;
__device__ __forceinline__ Chain shuffled_up(const Chain& c, int o) {
  return {__shfl_up_sync(0xffffffffu, c.first, o), __shfl_up_sync(0xffffffffu, c.last, o), __shfl_up_sync(0xffffffffu, c.any, o),
          __shfl_up_sync(0xffffffffu, c.gaps, o)};
}
__device__ __forceinline__ Chain scanned(Chain c, double eps) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Chain b = shuffled_up(c, o);
    if (lane >= o) c = join(b, c, eps);
  }
  return c;
}
__global__ void __launch_bounds__(1024) dbci_scan_kernel(DbciParams* P, Chain* chains, Next* next, int n_tiles) {
  __shared__ Chain part[32];
  __shared__ Next after_warp[32];
  wait_for_last_kernel();
  let_next_kernel_start();
  const double eps = P->eps;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int steps = (n_tiles + 1023) / 1024, t0 = warp * steps * 32;
  const Chain none = {0.0f, 0.0f, 0, 0};
  if (blockIdx.x == 1) {
    auto scan_back = [&](Next after, bool write) {
      for (int i0 = steps - 1; i0 >= 0; i0 -= kBatch) {
        Next c[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
          const int t = t0 + 32 * (i0 - b) + lane;
          c[b] = {0.0f, 0};
          if (i0 - b >= 0 && t < n_tiles) c[b] = next[t];
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
          const int t = t0 + 32 * (i0 - b) + lane;
          const unsigned any = __ballot_sync(0xffffffffu, c[b].any != 0), above = any & ~(0xffffffffu >> (31 - lane));
          const float v = __shfl_sync(0xffffffffu, c[b].v, above ? __ffs(above) - 1 : lane);
          const float v0 = __shfl_sync(0xffffffffu, c[b].v, any ? __ffs(any) - 1 : lane);
          if (write && i0 - b >= 0 && t < n_tiles) next[t] = above ? Next{v, 1} : after;
          if (any) after = {v0, 1};
        }
      }
      return after;
    };
    const Next mine = scan_back({0.0f, 0}, false);
    if (lane == 0) after_warp[warp] = mine;
    __syncthreads();
    Next after = {0.0f, 0};
    for (int w = 31; w > warp; --w)
      if (after_warp[w].any) after = after_warp[w];
    scan_back(after, true);
    return;
  }
  Chain run = none;
  for (int i0 = 0; i0 < steps; i0 += kBatch) {
    Chain c[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int t = t0 + 32 * (i0 + b) + lane;
      c[b] = i0 + b < steps && t < n_tiles ? chains[t] : none;
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int t = t0 + 32 * (i0 + b) + lane;
      const Chain up_to = scanned(c[b], eps);
      Chain before = shuffled_up(up_to, 1);
      if (lane == 0) before = none;
      if (i0 + b < steps && t < n_tiles) chains[t] = join(run, before, eps);
      run = join(run, {__shfl_sync(0xffffffffu, up_to.first, 31), __shfl_sync(0xffffffffu, up_to.last, 31), __shfl_sync(0xffffffffu, up_to.any, 31),
                       __shfl_sync(0xffffffffu, up_to.gaps, 31)}, eps);
    }
  }
  if (lane == 0) part[warp] = run;
  __syncthreads();
  if (warp == 0) {
    const Chain c = scanned(part[lane], eps);
    __syncwarp();
    part[lane] = c;
  }
  __syncthreads();
  if (threadIdx.x == 1023) P->n_mid = part[31].any ? part[31].gaps + 1 : 0;
  if (warp == 0) return;
  run = part[warp - 1];
  for (int i0 = 0; i0 < steps; i0 += kBatch) {
    Chain c[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int t = t0 + 32 * (i0 + b) + lane;
      c[b] = i0 + b < steps && t < n_tiles ? chains[t] : none;
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int t = t0 + 32 * (i0 + b) + lane;
      if (i0 + b < steps && t < n_tiles) chains[t] = join(run, c[b], eps);
    }
  }
}

// labels of all sorted points (0 left cluster, 1.. middle clusters in order, last = right cluster, -1 noise) and the
// first / last member of every cluster
__global__ void __launch_bounds__(32 * kTileWarps, 4) dbci_label_kernel(const float* x, long long n, DbciParams* P, int n_tiles, const unsigned* core,
                                                                        const Chain* chains, const Next* next, const unsigned char* plain,
                                                                        int* labels, int* first, int* last, int max_clusters) {
  __shared__ Chain part[kTileWarps], word_of[kTileWarps][kWarpSteps];
  __shared__ Next next_of[kTileWarps][kWarpSteps];          // the first core point after every word
  __shared__ int is_plain[kTileWarps];
  wait_for_last_kernel();
  let_next_kernel_start();
  const long long L = P->L, R = P->R;
  const double eps = P->eps;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_mid = P->n_mid;
  // The members of one cluster that a warp has met one after the other: sent when another cluster's come (thousands of words of
  // one cluster would queue for its two counters).
  int held = -1, held_first = 0, held_last = 0;
  auto send = [&]() {
    if (lane == 0 && held >= 0 && held < max_clusters) {
      atomicMin(first + held, held_first);
      atomicMax(last + held, held_last);
    }
    held = -1;
  };
  const int my_tile = blockIdx.x + warp * gridDim.x;
  if (my_tile < n_tiles) {
    const int p = plain[my_tile];
    if (lane == 0) is_plain[warp] = p;
    if (p) {
      // every point a core point of one cluster (a whole tile of the middle)
      const Chain before = chains[my_tile];
      const long long tile0 = (long long)my_tile * kTile;
      const int lab = !before.any ? 1 : before.gaps + 1 + (gap_after(before.last, x[tile0], eps) ? 1 : 0);
      if (labels) {
        int* to = labels + tile0;
        if ((reinterpret_cast<uintptr_t>(labels) & 15) == 0) {
          const int4 v = make_int4(lab, lab, lab, lab);
#pragma unroll 8
          for (int i = lane; i < kTile / 4; i += 32) __stcs(reinterpret_cast<int4*>(to) + i, v);
        } else {
#pragma unroll 8
          for (int i = lane; i < kTile; i += 32) to[i] = lab;
        }
      }
      held = lab;
      held_first = (int)tile0;
      held_last = (int)tile0 + kTile - 1;
      send();
    }
  }
  __syncthreads();
  for (int tile_i = 0; tile_i < kTileWarps; ++tile_i) {
    const int tile = blockIdx.x + tile_i * gridDim.x;
    if (tile >= n_tiles) break;
    if (is_plain[tile_i]) continue;
    const long long tile0 = (long long)tile * kTile;
    const Chain before = chains[tile];
    const Next after_tile = next[tile];
    const long long w0 = tile0 + warp * (32 * kWarpSteps);
    unsigned words[kWarpSteps];
    float vs[kWarpSteps];
    Chain mine = {0.0f, 0.0f, 0, 0};
#pragma unroll
    for (int i = 0; i < kWarpSteps; ++i) {
      const long long g = w0 + 32 * i + lane;
      words[i] = w0 + 32 * i < n ? core[(w0 >> 5) + i] : 0u;
      vs[i] = g < n ? x[g] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < kWarpSteps; ++i) {
      const Chain c = word_chain(words[i], vs[i], eps);
      if (lane == 0) word_of[warp][i] = c;
      mine = join(mine, c, eps);
    }
    __syncthreads();                      // the last tile's parts have been read
    if (lane == 0) part[warp] = mine;
    __syncthreads();
    Chain run = before;
    for (int w = 0; w < warp; ++w) run = join(run, part[w], eps);
    // of the warp's later words, of the later warps, of the later tiles
    Next after = after_tile;
    for (int w = kTileWarps - 1; w > warp; --w)
      if (part[w].any) after = {part[w].first, 1};
    int noise = 0;
#pragma unroll
    for (int i = kWarpSteps - 1; i >= 0; --i) {
      if (lane == 0) next_of[warp][i] = after;
      if (words[i]) after = {__shfl_sync(0xffffffffu, vs[i], __ffs(words[i]) - 1), 1};
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kWarpSteps; ++i) {
      const long long g0 = w0 + 32 * i, g = g0 + lane;
      const unsigned word = words[i], below = word & ((1u << lane) - 1u), above = word & ~(0xffffffffu >> (31 - lane));
      const float v = vs[i];
      const float vb = __shfl_sync(0xffffffffu, v, below ? 31 - __clz(below) : lane), va = __shfl_sync(0xffffffffu, v, above ? __ffs(above) - 1 : lane);
      const bool is = (word >> lane) & 1u;
      // the core point before this one: in this word, or the last of the run so far
      const bool starts = is && (below ? (double)v - (double)vb > eps : !run.any || gap_after(run.last, v, eps));
      const unsigned start_word = __ballot_sync(0xffffffffu, starts);
      const int started = run.any ? run.gaps + 1 : 0;              // clusters begun before this word
      const int upto = started + __popc(start_word & (0xffffffffu >> (31 - lane)));
      int lab = -2;                                                      // past the end of the array
      if (word == 0xffffffffu) {                                         // (all of the middle)
        lab = upto;
        if (labels) labels[g] = lab;
      } else if (g < n) {
        if (g < L) lab = 0;
        else if (g >= R) lab = n_mid + 1;
        else if (is) lab = upto;
        else {
          const Next after_word = next_of[warp][i];
          const bool has_left = below || run.any, has_right = above || after_word.any;
          const float left = below ? vb : run.last, right = above ? va : after_word.v;
          const double dl = has_left ? (double)v - (double)left : 1e300, dr = has_right ? (double)right - (double)v : 1e300;
          if (dl <= eps && dl <= dr) lab = upto;
          else if (dr <= eps) lab = upto + (!has_left || gap_after(left, right, eps) ? 1 : 0);
          else lab = -1;
        }
        if (labels) labels[g] = lab;
      }
      noise += __popc(__ballot_sync(0xffffffffu, lab == -1));
      const int lab0 = __shfl_sync(0xffffffffu, lab, 0);
      if (__all_sync(0xffffffffu, lab == lab0)) {
        if (lab0 != held) {
          send();
          held = lab0;
          held_first = (int)g0;
        }
        held_last = (int)g0 + 31;
      } else if (lab >= 0 && lab < max_clusters) {
        atomicMin(first + lab, (int)g);
        atomicMax(last + lab, (int)g);
      }
      run = join(run, word_of[warp][i], eps);
    }
    send();
    if (lane == 0 && noise) atomicAdd(&P->n_noise, noise);
    __syncwarp();                         // word_of has been read
  }
}

// lower medians of the clusters in ascending order; result scalars
__global__ void __launch_bounds__(256) dbci_centroid_kernel(const float* x, long long n, const DbciParams* P,
                                                            const int* first, const int* last, int max_clusters,
                                                            float* centroids, int max_centroids, lcd_dbci_result* out) {
  wait_for_last_kernel();
  let_next_kernel_start();
  __shared__ int counts[256];
  const int n_clusters = P->n_mid + 2, stop = n_clusters < max_clusters ? n_clusters : max_clusters;
  const int per = (stop + 255) / 256, c0 = threadIdx.x * per, c1 = min(c0 + per, stop);
  int mine = 0;
  for (int c = c0; c < c1; ++c) mine += last[c] >= first[c];           // the right cluster can be empty
  counts[threadIdx.x] = mine;
  __syncthreads();
  int w = 0, total = 0;                              // clusters of the threads before this one, of all
  for (int t = threadIdx.x & 31; t < 256; t += 32) {
    const int warp_sum = __reduce_add_sync(0xffffffffu, counts[t]);
    total += warp_sum;
    w += t < (int)(threadIdx.x & ~31u) ? warp_sum : 0;
  }
  const int lane = threadIdx.x & 31;
  for (int l = 0; l < 32; ++l) {
    const int c = __shfl_sync(0xffffffffu, mine, l);
    w += l < lane ? c : 0;
  }
  for (int c = c0; c < c1; ++c) {
    if (last[c] < first[c]) continue;
    if (w < max_centroids) centroids[w] = x[first[c] + (last[c] - first[c]) / 2];
    ++w;
  }
  if (threadIdx.x != 0) return;
  out->sigma = P->sigma;
  out->eps = P->eps;
  out->min_pts = P->min_pts;
  out->left = P->L;
  out->right = n - P->R;
  out->n_centroids = total;
  out->n_noise = P->n_noise;
  out->n_clusters_found = n_clusters;
}

size_t al256(size_t v) { return (v + 255) & ~(size_t)255; }

struct DbciLayout {
  size_t sorted, core, chains, next, plain, first, last, params, sort, total, sort_bytes;
  int tiles;
};
DbciLayout dbci_layout(int64_t n, int max_clusters) {
  DbciLayout l;
  const size_t tiles = ((size_t)n + kTile - 1) / kTile;
  l.tiles = (int)tiles;
  size_t off = 0;
  l.sorted = off; off += al256((size_t)n * sizeof(float));
  l.core = off; off += al256(((size_t)n + 31) / 32 * sizeof(unsigned));
  l.chains = off; off += al256(tiles * sizeof(Chain));
  l.next = off; off += al256(tiles * sizeof(Next));
  l.plain = off; off += al256(tiles);
  l.first = off; off += al256((size_t)max_clusters * sizeof(int));
  l.last = off; off += al256((size_t)max_clusters * sizeof(int));
  l.params = off; off += al256(sizeof(DbciParams));
  l.sort_bytes = 0;
  if (dbci_sort_takes(n)) l.sort_bytes = dbci_sort_workspace_bytes(n);
  else cub::DeviceRadixSort::SortKeys(nullptr, l.sort_bytes, (const float*)nullptr, (float*)nullptr, (int)n);
  l.sort = off; off += al256(l.sort_bytes);
  l.total = off;
  return l;
}

}  // namespace

size_t dbci_workspace_bytes(int64_t n, int max_centroids) { return dbci_layout(n, max_centroids + 2).total; }

lcd_status launch_dbci(const float* weights, int64_t n, void* workspace, float* centroids, int max_centroids,
                       int32_t* labels, float* sorted_out, lcd_dbci_result* result, void* stream) {
  const int max_clusters = max_centroids + 2;
  const DbciLayout l = dbci_layout(n, max_clusters);
  uint8_t* base = static_cast<uint8_t*>(workspace);
  // sorted where the caller wants it, unless that is where the input lies
  const bool apart = sorted_out && (sorted_out + n <= weights || weights + n <= sorted_out);
  float* x = apart ? sorted_out : reinterpret_cast<float*>(base + l.sorted);
  unsigned* core = reinterpret_cast<unsigned*>(base + l.core);
  Chain* chains = reinterpret_cast<Chain*>(base + l.chains);
  Next* next = reinterpret_cast<Next*>(base + l.next);
  unsigned char* plain = base + l.plain;
  int* first = reinterpret_cast<int*>(base + l.first);
  int* last = reinterpret_cast<int*>(base + l.last);
  DbciParams* P = reinterpret_cast<DbciParams*>(base + l.params);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  size_t tmp_bytes = l.sort_bytes;
  cudaError_t e = dbci_sort_takes(n) ? launch_dbci_sort(weights, n, x, base + l.sort, s)
                                     : cub::DeviceRadixSort::SortKeys(base + l.sort, tmp_bytes, weights, x, (int)n, 0, 32, s);
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  const unsigned fill = (unsigned)((max_clusters + 255) / 256);
  const long long count = n;
  const float* xc = x;
  e = launch_after(dbci_params_kernel, fill < 1024 ? fill : 1024, 256, 0, s, xc, count, P, first, last, max_clusters);
  // tiles of a CTA: as many as still give every SM eight CTAs
  int per = l.tiles / (8 * current_sm_count());
  per = per < 1 ? 1 : per > kTileWarps ? kTileWarps : per;
  const unsigned ctas = (unsigned)((l.tiles + per - 1) / per);
  if (e == cudaSuccess) e = launch_after(dbci_mark_kernel, ctas, 32 * kTileWarps, 0, s, xc, count, P, l.tiles, core, chains, next, plain);
  if (e == cudaSuccess) e = launch_after(dbci_scan_kernel, 2, 1024, 0, s, P, chains, next, l.tiles);
  if (e == cudaSuccess)
    e = launch_after(dbci_label_kernel, ctas, 32 * kTileWarps, 0, s, xc, count, P, l.tiles, core, chains, next, plain, labels, first, last, max_clusters);
  if (e == cudaSuccess) e = launch_after(dbci_centroid_kernel, 1, 256, 0, s, xc, count, P, first, last, max_clusters, centroids, max_centroids, result);
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  if (sorted_out && !apart) {
    e = cudaMemcpyAsync(sorted_out, x, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  return LCD_OK;
}

}  // namespace lcd
