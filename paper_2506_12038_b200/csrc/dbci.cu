// Density-based centroid initialisation (DBCI, Section 3.1 of the LCD paper), offline, on a flat array of weights:
// sort; sigma from six nearest-rank percentiles; two seed clusters around the extreme weights; MinPts and eps from
// them; DBSCAN on the rest; lower medians.  On sorted one-dimensional data DBSCAN is local: a point's neighbours are its
// neighbours in the array, core points chain into one cluster while the gap to the core point before is at most eps, and
// another point needs the nearest core point on either side.  So two passes over the sorted array do it: one marks
// the core points and sums up every tile (first and last core point, gaps between), one writes the labels, with a scan
// over the tiles in either direction between them: what lies before a word of 32 points and the first core point after it
// are then known, and no point looks at another one, however many share its value (walking out to the core points takes up
// to MinPts steps a point: 400 K weights on eight values 107 ms, 0.2 so).  A tile without gaps or non-core points, nearly every one, is written without being read
// again, and where 4096 weights span less than eps two of them tell so: little more than the labels' 4 bytes a weight is
// moved (45 M weights: 130 us after the sort; with a thread a point, two max-scans and a sum-scan over the whole
// array 2600).
// The sort is a CUB device primitive; everything else is written here.  All comparisons and the few scalar operations
// are binary64 on the binary32 data, so every decision has one right answer.
#include <cuda_runtime.h>

#include <cub/device/device_radix_sort.cuh>

#include "common.h"

namespace lcd {

namespace {

struct DbciParams {        // device-side scalars shared by the kernels; mirrored into lcd_dbci_result at the end
  double sigma, eps;
  long long L, R;          // left cluster = sorted [0, L), right cluster = [R, n)
  long long min_pts;
  int n_mid;               // clusters found among the middle points
  int n_noise;
};

// First index in [lo, hi) whose value is >= v (strict: > v), by a warp: 32 probes a step instead of one.
template <bool STRICT>
__device__ long long warp_bound(const float* x, long long lo, long long hi, double v) {
  const int lane = threadIdx.x & 31;
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
__global__ void __launch_bounds__(256) dbci_params_kernel(const float* __restrict__ x, long long n, DbciParams* __restrict__ P,
                                                          int* __restrict__ first, int* __restrict__ last, int max_clusters) {
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
    const long long at = warp == 0 ? warp_bound<true>(x, 0, n, (double)x[0] + sigma) : warp_bound<false>(x, 0, n, (double)x[n - 1] - sigma);
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

// Whether the middle point at g is a core point: at least k points y of the middle with v - eps <= y <= v + eps (binary64).
// A binary32 y is >= a binary64 bound exactly if it is >= the bound rounded up to binary32, and likewise on the other side.
__device__ __forceinline__ bool is_core(const float* __restrict__ x, long long L, long long R, long long g, float v, double eps, long long k) {
  if (k <= 1) return true;                                   // itself (and k = 0: an empty seed cluster, left by a NaN weight)
  const float a = __double2float_ru((double)v - eps), b = __double2float_rd((double)v + eps);
  const long long left = g - (k - 1), right = g + (k - 1);
  if (left >= L && x[left] >= a) return true;                // k - 1 neighbours on one side, the usual case
  if (right < R && x[right] <= b) return true;
  long long lo = left > L ? left : L, hi = g;                // first neighbour: in [lo, g]
  while (lo < hi) {
    const long long mid = (lo + hi) >> 1;
    if (x[mid] < a) lo = mid + 1; else hi = mid;
  }
  const long long first = lo;
  lo = g;
  hi = right < R ? right : R;                                // first point past the neighbours: in (g, hi]
  while (lo < hi) {
    const long long mid = (lo + hi) >> 1;
    if (x[mid] <= b) lo = mid + 1; else hi = mid;
  }
  return lo - first >= k;
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

__global__ void __launch_bounds__(32 * kTileWarps) dbci_mark_kernel(const float* __restrict__ x, long long n, const DbciParams* __restrict__ P,
                                                                    unsigned* __restrict__ core, Chain* __restrict__ chains,
                                                                    Next* __restrict__ next, unsigned char* __restrict__ plain) {
  __shared__ Chain part[kTileWarps];
  __shared__ int all[kTileWarps];
  const long long L = P->L, R = P->R, k = P->min_pts, tile0 = (long long)blockIdx.x * kTile;
  const double eps = P->eps;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // A whole tile at once: if its last value and the (k - 1)-th before its first lie within eps of each other, every point has
  // k - 1 neighbours on its left and no two neighbours a gap between them (subtraction and rounding are monotone).
  if (tile0 - (k - 1) >= L && tile0 + kTile <= R) {
    const float low = x[tile0 - (k - 1)], high = x[tile0 + kTile - 1];
    if (low >= __double2float_ru((double)high - eps) && !gap_after(low, high, eps)) {
      if (threadIdx.x < kTile / 32) core[(tile0 >> 5) + threadIdx.x] = 0xffffffffu;
      if (threadIdx.x == 0) {
        chains[blockIdx.x] = {x[tile0], high, 1, 0};
        next[blockIdx.x] = {x[tile0], 1};
        plain[blockIdx.x] = 1;
      }
      return;
    }
  }
  Chain mine = {0.0f, 0.0f, 0, 0};
  bool every = true;
  const long long w0 = tile0 + warp * (32 * kWarpSteps);
  float vs[kWarpSteps];
#pragma unroll
  for (int i = 0; i < kWarpSteps; ++i) {
    const long long g = w0 + 32 * i + lane;
    vs[i] = g < n ? x[g] : 0.0f;
  }
#pragma unroll
  for (int i = 0; i < kWarpSteps; ++i) {
    const long long g = w0 + 32 * i + lane;
    const bool c = g >= L && g < R && is_core(x, L, R, g, vs[i], eps, k);
    const unsigned word = __ballot_sync(0xffffffffu, c);
    if (lane == 0 && w0 + 32 * i < n) core[(w0 >> 5) + i] = word;
    every = every && word == 0xffffffffu;
    mine = join(mine, word_chain(word, vs[i], eps), eps);
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
    chains[blockIdx.x] = t;
    next[blockIdx.x] = {t.first, t.any};
    plain[blockIdx.x] = (unsigned char)(e && t.gaps == 0);
  }
}

// Exclusive scans over the tiles in place, by one CTA each.  CTA 0: chains[t] becomes the chain of all tiles before t; a thread
// joins its run of tiles, the threads' runs are scanned, then it walks its run again.  CTA 1: next[t] becomes the first core
// point of all tiles after t.
__global__ void __launch_bounds__(1024) dbci_scan_kernel(DbciParams* __restrict__ P, Chain* __restrict__ chains, Next* __restrict__ next, int n_tiles) {
  __shared__ Chain part[1024];
  __shared__ unsigned any_of[32];          // CTA 1: threads whose runs have core points, a word per warp
  const double eps = P->eps;
  const int per = (n_tiles + 1023) / 1024, t0 = min((int)threadIdx.x * per, n_tiles), t1 = min(t0 + per, n_tiles);
  if (blockIdx.x == 1) {
    Next after = {0.0f, 0};
    for (int t = t1 - 1; t >= t0; --t) {
      const Next c = next[t];
      if (c.any) after = c;
    }
    part[threadIdx.x].first = after.v;
    const unsigned any_word = __ballot_sync(0xffffffffu, after.any != 0);
    if ((threadIdx.x & 31) == 0) any_of[threadIdx.x >> 5] = any_word;
    __syncthreads();
    int w = threadIdx.x >> 5;
    unsigned word = any_of[w] & ~(0xffffffffu >> (31 - (threadIdx.x & 31)));        // the threads after this one
    while (word == 0 && ++w < 32) word = any_of[w];
    after = {word ? part[32 * w + __ffs(word) - 1].first : 0.0f, word != 0};
    for (int t = t1 - 1; t >= t0; --t) {
      const Next c = next[t];
      next[t] = after;
      if (c.any) after = c;
    }
    return;
  }
  Chain mine = {0.0f, 0.0f, 0, 0};
  for (int t = t0; t < t1; ++t) mine = join(mine, chains[t], eps);
  part[threadIdx.x] = mine;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    Chain v = part[threadIdx.x];
    if ((int)threadIdx.x >= o) v = join(part[threadIdx.x - o], v, eps);
    __syncthreads();
    part[threadIdx.x] = v;
    __syncthreads();
  }
  Chain run = {0.0f, 0.0f, 0, 0};
  if (threadIdx.x > 0) run = part[threadIdx.x - 1];
  for (int t = t0; t < t1; ++t) {
    const Chain c = chains[t];
    chains[t] = run;
    run = join(run, c, eps);
  }
  if (threadIdx.x == 1023) P->n_mid = part[1023].any ? part[1023].gaps + 1 : 0;
}

// labels of all sorted points (0 left cluster, 1.. middle clusters in order, last = right cluster, -1 noise) and the
// first / last member of every cluster
__global__ void __launch_bounds__(32 * kTileWarps, 4) dbci_label_kernel(const float* __restrict__ x, long long n, DbciParams* __restrict__ P,
                                                                     const unsigned* __restrict__ core, const Chain* __restrict__ chains,
                                                                     const Next* __restrict__ next, const unsigned char* __restrict__ plain, int* __restrict__ labels,
                                                                     int* __restrict__ first, int* __restrict__ last, int max_clusters) {
  __shared__ Chain part[kTileWarps];
  __shared__ Next next_of[kTileWarps][kWarpSteps];          // the first core point after every word
  const long long L = P->L, R = P->R, tile0 = (long long)blockIdx.x * kTile;
  const double eps = P->eps;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_mid = P->n_mid;
  const Chain before = chains[blockIdx.x];
  if (plain[blockIdx.x]) {
    // every point a core point of one cluster (a whole tile of the middle)
    const int lab = !before.any ? 1 : before.gaps + 1 + (gap_after(before.last, x[tile0], eps) ? 1 : 0);
    if (labels) {
      const int4 v = make_int4(lab, lab, lab, lab);
      if ((reinterpret_cast<uintptr_t>(labels) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < kTile / 4 / (32 * kTileWarps); ++i)
          __stcs(reinterpret_cast<int4*>(labels + tile0) + i * (32 * kTileWarps) + threadIdx.x, v);
      } else {
        for (int i = threadIdx.x; i < kTile; i += 32 * kTileWarps) labels[tile0 + i] = lab;
      }
    }
    if (threadIdx.x == 0 && lab < max_clusters) {
      atomicMin(first + lab, (int)tile0);
      atomicMax(last + lab, (int)tile0 + kTile - 1);
    }
    return;
  }
  const long long w0 = tile0 + warp * (32 * kWarpSteps);
  unsigned words[kWarpSteps];
  float vs[kWarpSteps];
  Chain mine = {0.0f, 0.0f, 0, 0};
#pragma unroll
  for (int i = 0; i < kWarpSteps; ++i) {
    const long long g = w0 + 32 * i + lane;
    words[i] = w0 + 32 * i < n ? core[(w0 >> 5) + i] : 0u;
    vs[i] = g < n ? x[g] : 0.0f;
    mine = join(mine, word_chain(words[i], vs[i], eps), eps);
  }
  if (lane == 0) part[warp] = mine;
  __syncthreads();
  Chain run = before;
  for (int w = 0; w < warp; ++w) run = join(run, part[w], eps);
  // of the warp's later words, of the later warps, of the later tiles
  Next after = next[blockIdx.x];
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
    if (g < n) {
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
    // First and last member of every cluster: a warp whose lanes agree sends one pair.
    const int lab0 = __shfl_sync(0xffffffffu, lab, 0);
    if (__all_sync(0xffffffffu, lab == lab0)) {
      if (lab0 >= 0 && lab0 < max_clusters) {
        if (lane == 0) atomicMin(first + lab0, (int)g);
        if (lane == 31) atomicMax(last + lab0, (int)g);
      }
    } else if (lab >= 0 && lab < max_clusters) {
      atomicMin(first + lab, (int)g);
      atomicMax(last + lab, (int)g);
    }
    run = join(run, word_chain(word, v, eps), eps);
  }
  if (lane == 0 && noise) atomicAdd(&P->n_noise, noise);
}

// lower medians of the clusters in ascending order; result scalars
__global__ void __launch_bounds__(256) dbci_centroid_kernel(const float* __restrict__ x, long long n, const DbciParams* __restrict__ P,
                                                            const int* __restrict__ first, const int* __restrict__ last, int max_clusters,
                                                            float* __restrict__ centroids, int max_centroids, lcd_dbci_result* __restrict__ out) {
  __shared__ int counts[256];
  const int n_clusters = P->n_mid + 2, stop = n_clusters < max_clusters ? n_clusters : max_clusters;
  const int per = (stop + 255) / 256, c0 = threadIdx.x * per, c1 = min(c0 + per, stop);
  int mine = 0;
  for (int c = c0; c < c1; ++c) mine += last[c] >= first[c];           // the right cluster can be empty
  counts[threadIdx.x] = mine;
  __syncthreads();
  int w = 0, total = 0;
  for (int t = 0; t < 256; ++t) {
    w += t < (int)threadIdx.x ? counts[t] : 0;
    total += counts[t];
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
  size_t sorted, core, chains, next, plain, first, last, params, cub, total, cub_bytes;
};
DbciLayout dbci_layout(int64_t n, int max_clusters) {
  DbciLayout l;
  const size_t tiles = ((size_t)n + kTile - 1) / kTile;
  size_t off = 0;
  l.sorted = off; off += al256((size_t)n * sizeof(float));
  l.core = off; off += al256(((size_t)n + 31) / 32 * sizeof(unsigned));
  l.chains = off; off += al256(tiles * sizeof(Chain));
  l.next = off; off += al256(tiles * sizeof(Next));
  l.plain = off; off += al256(tiles);
  l.first = off; off += al256((size_t)max_clusters * sizeof(int));
  l.last = off; off += al256((size_t)max_clusters * sizeof(int));
  l.params = off; off += al256(sizeof(DbciParams));
  l.cub_bytes = 0;
  cub::DeviceRadixSort::SortKeys(nullptr, l.cub_bytes, (const float*)nullptr, (float*)nullptr, (int)n);
  l.cub = off; off += al256(l.cub_bytes);
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
  const unsigned tiles = (unsigned)((n + kTile - 1) / kTile);
  size_t tmp_bytes = l.cub_bytes;
  cudaError_t e = cub::DeviceRadixSort::SortKeys(base + l.cub, tmp_bytes, weights, x, (int)n, 0, 32, s);
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  const unsigned fill = (unsigned)((max_clusters + 255) / 256);
  dbci_params_kernel<<<fill < 1024 ? fill : 1024, 256, 0, s>>>(x, n, P, first, last, max_clusters);
  dbci_mark_kernel<<<tiles, 32 * kTileWarps, 0, s>>>(x, n, P, core, chains, next, plain);
  dbci_scan_kernel<<<2, 1024, 0, s>>>(P, chains, next, (int)tiles);
  dbci_label_kernel<<<tiles, 32 * kTileWarps, 0, s>>>(x, n, P, core, chains, next, plain, labels, first, last, max_clusters);
  dbci_centroid_kernel<<<1, 256, 0, s>>>(x, n, P, first, last, max_clusters, centroids, max_centroids, result);
  if (sorted_out && !apart) {
    e = cudaMemcpyAsync(sorted_out, x, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  return LCD_OK;
}

}  // namespace lcd
