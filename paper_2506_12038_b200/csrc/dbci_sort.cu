// The sort of the density-based centroid initialisation: binary32 weights in ascending order, by two passes over the data
// after one that counts.  Weights of a layer are spread smoothly over their range or repeat few values, so a piecewise linear
// map of the (order-preserving) key, fitted to a sample, cuts them into buckets of about kTarget keys that fit the shared
// memory of a CTA:
//   plan      range and histogram of 16384 samples; every bin of 2048 is divided into equal parts, as many as its samples
//             ask for ("fine bins", about 3 K keys of 45 M each; one more at either end for what
//             lies at or beyond the sample's extremes, where clipped weights repeat one value);
//   count     exact counts of the fine bins;
//   map       one CTA: neighbouring fine bins become buckets of at most kCap keys, a larger fine bin a bucket of its own;
//   partition every key to its bucket's place in the output, in no order;
//   buckets   a CTA sorts a bucket where it lies: 16384 equal parts of its range, a place for every key by a counting pass
//             (the shared-memory atomic's result), then sixteen neighbours at a time through a sorting network, twice, the
//             second time half a step further, which puts parts of up to eight keys in order.  A larger bucket is right if
//             it holds one value alone, and that is checked;
//   general   nothing, unless one of these has found keys that it cannot take (narrow clumps or values repeated among others
//             in one fine bin): then a radix sort of the input in four stable passes by one cooperative launch.  Zeros of either
//             sign are equal and keep their order; if there are both, the same launch writes them again in that order.
// 45 M Gaussian weights: 620 us (plan 6, count 55, map 18, partition 240, buckets 285), CUB's radix sort 1070; 925 K: 52 and 110.
// Bytes are 0.9 GB, 140 us: what bounds the passes is shared memory at random addresses (three lookups or atomics and two stores
// a key in the partition, an atomic, a lookup and a store in the buckets, each three to four bank conflicts a warp) and, where the
// partition writes runs of six keys, the sectors that L2 takes.  Inputs that need the general sort: 1490 us after the count
// (CUB 1070).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "dbci_sort.h"
#include "device_util.h"

namespace lcd {

namespace {

constexpr int kSamples = 16384, kBins = 2048, kFineMax = 24576, kFineBudget = 14334;
static_assert(kFineBudget + 5 * kBins + 2 <= kFineMax, "shares of the budget are rounded up, every bin has four parts at least");
constexpr int kCap = 16384;                  // keys a CTA sorts
constexpr int kTarget = 12288;               // keys of a bucket of a large array
constexpr int kMaxBuckets = 8192;
constexpr int64_t kMostKeys = (int64_t)(kMaxBuckets / 2 - 1) * kTarget;

struct SortState {
  unsigned kmin, kmax;      // sample extremes
  int shift;                // bin of a key: (key - kmin) >> shift
  int n_fine, n_buckets;
  int large;                // there are fine bins of more than kCap keys
  int zeros;                // bit 0: there are positive zeros, bit 1: negative ones
  int general;              // the radix sort has to do it
  int n_uneven;             // buckets for sort_uneven_kernel
};

__device__ __forceinline__ unsigned key_of(unsigned raw) { return raw ^ ((unsigned)((int)raw >> 31) | 0x80000000u); }
__device__ __forceinline__ unsigned raw_of(unsigned key) { return key ^ (~(unsigned)((int)key >> 31) | 0x80000000u); }

// The same for zeros of either sign, which are equal.
__device__ __forceinline__ unsigned value_of(unsigned raw) { return raw == 0x80000000u ? 0u : raw; }

// Exclusive sum over the 32 * WARPS threads of a CTA; part: WARPS + 1 words (the last: the total).
template <int WARPS>
__device__ __forceinline__ unsigned block_exclusive(unsigned v, unsigned* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += u;
  }
  if (lane == 31) part[warp] = s;
  __syncthreads();
  if (warp == 0) {
    unsigned p = lane < WARPS ? part[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned u = __shfl_up_sync(0xffffffffu, p, o);
      if (lane >= o) p += u;
    }
    if (lane < WARPS) part[lane] = p;
    if (lane == WARPS - 1) part[WARPS] = p;
  }
  __syncthreads();
  return s - v + (warp ? part[warp - 1] : 0u);
}

__device__ __forceinline__ void wait_for_last_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A cluster of CTAs fetches the samples, a sector each (one SM alone takes 8 us for them), its first CTA does the rest.  Bins that
// the samples missed get four parts all the same: 64 K keys, more than a bucket in a part, would have had 24 samples.
constexpr int kPlanCtas = 8;
__global__ void __cluster_dims__(kPlanCtas, 1, 1) __launch_bounds__(1024) sort_plan_kernel(const unsigned* in, long long n, int budget, SortState* st,
                                                                                          unsigned* samples, unsigned* table, unsigned* fine) {
  constexpr int PER = kSamples / 1024;
  __shared__ unsigned hist[kBins], part[33], lo_s[32], hi_s[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  wait_for_last_kernel();
  let_next_kernel_start();
#pragma unroll
  for (int j = 0; j < PER / kPlanCtas; ++j) {
    // a place in the i-th of kSamples equal stretches of the input
    const unsigned long long i = (blockIdx.x * (PER / kPlanCtas) + j) * 1024 + tid, a = i * n / kSamples, b = (i + 1) * n / kSamples;
    unsigned h = (unsigned)i * 2654435761u;
    h ^= h >> 15;
    h *= 2246822519u;
    h ^= h >> 13;
    __stcg(samples + i, key_of(in[a + ((h * (b - a)) >> 32)]));
  }
  for (int i = blockIdx.x * 1024 + tid; i < kFineMax / 4; i += kPlanCtas * 1024) reinterpret_cast<uint4*>(fine)[i] = make_uint4(0u, 0u, 0u, 0u);
  cooperative_groups::this_cluster().sync();
  if (blockIdx.x != 0) return;
  unsigned k[PER], lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int j = 0; j < PER / 4; ++j) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(samples) + j * 1024 + tid);
    k[4 * j] = v.x; k[4 * j + 1] = v.y; k[4 * j + 2] = v.z; k[4 * j + 3] = v.w;
  }
  for (int i = tid; i < kBins; i += 1024) hist[i] = 0u;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    lo = min(lo, k[j]);
    hi = max(hi, k[j]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) { lo_s[warp] = lo; hi_s[warp] = hi; }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, lo_s[lane]);
  hi = __reduce_max_sync(0xffffffffu, hi_s[lane]);
  const int bits = 32 - __clz(hi - lo), shift = bits > 12 ? bits - 11 : 1;
#pragma unroll
  for (int j = 0; j < PER; ++j) atomicAdd(&hist[(k[j] - lo) >> shift], 1u);
  __syncthreads();
  unsigned s[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    s[h] = max(4u, (hist[2 * tid + h] * (unsigned)budget + kSamples - 1) / kSamples);      // (16384 x 14334 fits)
    s[h] = min(s[h], 1u << min(shift, 15));                                                 // one value each at least
  }
  const unsigned base = block_exclusive<32>(s[0] + s[1], part);
  // a table entry: first fine bin << 16 | parts of the bin
  reinterpret_cast<uint2*>(table)[tid] = make_uint2((base + 1u) << 16 | s[0], (base + 1u + s[0]) << 16 | s[1]);
  if (tid == 0) {
    st->kmin = lo;
    st->kmax = hi;
    st->shift = shift;
    st->n_fine = (int)part[32] + 2;
    st->n_buckets = 0;
    st->large = 0;
    st->zeros = 0;
    st->general = 0;
    st->n_uneven = 0;
  }
}

// The fine bin of a key: 0 and n_fine - 1 take what lies at or beyond the sample's extremes.
struct FineMap {
  unsigned kmin, kmax;
  int shift, last;
  __device__ explicit FineMap(const SortState* st) : kmin(st->kmin), kmax(st->kmax), shift(st->shift), last(st->n_fine - 1) {}
  __device__ __forceinline__ int of(unsigned k, const unsigned* table) const {
    const unsigned d = k - kmin;
    if (d - 1u >= kmax - kmin - 1u || kmax == kmin) return k <= kmin ? 0 : last;          // seldom
    const unsigned e = table[d >> shift];
    return (int)((e >> 16) + __umulhi(d << (32 - shift), e & 0xffffu));                   // (d below its bin) * parts >> shift
  }
};

constexpr int kCountThreads = 768, kCountItems = 8;
constexpr int kCountSmem = (kBins + kFineMax) * 4;
__global__ void __launch_bounds__(kCountThreads, 2) sort_count_kernel(const unsigned* __restrict__ in, long long n, SortState* st,
                                                                      const unsigned* table_g, unsigned* fine) {
  extern __shared__ unsigned sm[];
  wait_for_last_kernel();
  let_next_kernel_start();
  unsigned *table = sm, *cnt = sm + kBins;
  const int tid = threadIdx.x;
  const FineMap map(st);
  for (int i = tid; i < kBins; i += kCountThreads) table[i] = table_g[i];
  for (int i = tid; i <= map.last; i += kCountThreads) cnt[i] = 0u;
  __syncthreads();
  constexpr int TILE = kCountThreads * kCountItems;
  for (long long t0 = (long long)blockIdx.x * TILE; t0 < n; t0 += (long long)gridDim.x * TILE) {
    unsigned v[kCountItems];
    const int left = (int)min((long long)TILE, n - t0);
    const unsigned* p = in + t0 + tid;
    if (left == TILE) {
#pragma unroll
      for (int j = 0; j < kCountItems; ++j) v[j] = __ldcs(p + j * kCountThreads);
#pragma unroll
      for (int j = 0; j < kCountItems; ++j) atomicAdd(&cnt[map.of(key_of(v[j]), table)], 1u);
    } else {
      for (int j = tid; j < left; j += kCountThreads) atomicAdd(&cnt[map.of(key_of(in[t0 + j]), table)], 1u);
    }
  }
  __syncthreads();
  for (int i = tid; i <= map.last; i += kCountThreads) {
    const unsigned c = cnt[i];
    if (c) atomicAdd(fine + i, c);
  }
}

// A bucket is a run of fine bins that begin between the same two multiples of `target` in the sorted order; a fine bin that ends
// more than kCap keys after the first of the two begins another one.  So a bucket has at most kCap keys unless it is a fine bin of
// more, and there are at most two for every `target` keys.  Empty fine bins begin none.
// begins: a word for sixteen fine bins, a bit for each that begins a bucket under the number of buckets begun before, less one.
constexpr int kMapThreads = kFineMax / 32, kMapWarps = kMapThreads / 32;
__global__ void __launch_bounds__(kMapThreads) sort_map_kernel(long long n, int target, SortState* st, unsigned* fine, const unsigned* samples, const unsigned* table,
                                                               unsigned* __restrict__ begins,
                                                               unsigned* __restrict__ first, unsigned* __restrict__ cursor) {
  constexpr int PER = 32;
  __shared__ unsigned part[kMapWarps + 1];
  __shared__ unsigned tail[kMapWarps], is_large[kMapThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  wait_for_last_kernel();
  let_next_kernel_start();
  unsigned c[PER], sum = 0, last = 0;
#pragma unroll
  for (int j = 0; j < PER / 4; ++j) {
    const uint4 v = reinterpret_cast<const uint4*>(fine)[tid * (PER / 4) + j];
    c[4 * j] = v.x; c[4 * j + 1] = v.y; c[4 * j + 2] = v.z; c[4 * j + 3] = v.w;
  }
  unsigned large = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    sum += c[j];
    last = c[j] ? c[j] : last;
    large |= c[j] > (unsigned)kCap ? 1u << j : 0u;
  }
  is_large[tid] = large;
  unsigned at = block_exclusive<kMapWarps>(sum, part);
  // the last non-empty fine bin before this thread's
  unsigned before = last;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o && before == 0) before = u;
  }
  if (lane == 31) tail[warp] = before;
  before = __shfl_up_sync(0xffffffffu, before, 1);
  if (lane == 0) before = 0;
  __syncthreads();
  for (int w = warp - 1; w >= 0 && before == 0; --w) before = tail[w];
  const unsigned t = (unsigned)target, room = (unsigned)(kCap - target);
  // p: where a bin begins in the sorted order; next: the first multiple of t after the last bin's
  unsigned starts = 0, p = at, next = before ? ((at - before) / t + 1u) * t : 0u;
#pragma unroll
  for (int j = 0; j < PER; ++j)
    if (c[j]) {
      if (p >= next) {
        starts |= 1u << j;
        next += t;
        if (p >= next) next = (p / t + 1u) * t;
      } else if (p + c[j] > next + room) {
        starts |= 1u << j;
      }
      p += c[j];
    }
  __syncthreads();
  unsigned id = block_exclusive<kMapWarps>((unsigned)__popc(starts), part);
  const int total = (int)part[kMapWarps];
  reinterpret_cast<uint2*>(begins)[tid] = make_uint2((id - 1u) << 16 | (starts & 0xffffu), (id - 1u + (unsigned)__popc(starts & 0xffffu)) << 16 | starts >> 16);
  p = at;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if ((starts >> j) & 1u) {
      first[id] = p;
      cursor[id] = p;
      ++id;
    }
    p += c[j];
  }
  // Fine bins of more than kCap keys: two different samples in one, and the work of the next two kernels would be in vain.
  const bool any_large = __syncthreads_or(large != 0u);
  bool mixed = false;
  if (any_large) {
    const FineMap map(st);
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if ((large >> j) & 1u) __stcg(fine + tid * PER + j, 0u);
    __syncthreads();
    for (int i = tid; i < kSamples; i += kMapThreads) {
      const unsigned k = key_of(value_of(raw_of(samples[i])));
      const int f = map.of(k, table);
      if ((is_large[f >> 5] >> (f & 31)) & 1u) {
        const unsigned other = atomicCAS(fine + f, 0u, k);
        mixed = mixed || (other != 0u && other != k);
      }
    }
  }
  mixed = __syncthreads_or(mixed);
  if (tid == 0) {
    first[total] = (unsigned)n;
    st->n_buckets = total;
    st->large = any_large;
    st->general = mixed;
  }
}

// A tile of 1024 * ITEMS keys at a time: its keys are put in bucket order in shared memory (a key's rank in its bucket is the
// result of the atomic that counts it), one reservation per bucket in the output, and written out in runs, whose beginnings are
// bits of a map of the tile (a bucket's number beside every key would be a store and a load more).  The next tile's keys are
// asked for before the writes.
constexpr int kPartThreads = 1024;
template <int ITEMS>
constexpr int partition_smem() { return kBins * 4 + kFineMax / 4 + kMaxBuckets * 8 + kPartThreads * ITEMS * 4 + kPartThreads * ITEMS / 32 * 8; }
template <int ITEMS>
__global__ void __launch_bounds__(kPartThreads, 1) sort_partition_kernel(const unsigned* __restrict__ in, long long n, const SortState* st,
                                                                         const unsigned* table_g, const unsigned* begins_g,
                                                                         unsigned* cursor, unsigned* __restrict__ out) {
  constexpr int TILE = kPartThreads * ITEMS, kLong = 128;
  extern __shared__ __align__(16) unsigned sm[];
  __shared__ unsigned part[kPartThreads / 32 + 1];
  __shared__ uint2 long_runs[TILE / kLong];
  __shared__ int n_long;
  wait_for_last_kernel();
  let_next_kernel_start();
  if (st->general) return;
  unsigned* at = sm;                                      // [kMaxBuckets] counts, then first place in the tile
  unsigned* delta = at + kMaxBuckets;                     // [kMaxBuckets] of the tile's runs: place in the output - place in the tile
  unsigned* table = delta + kMaxBuckets;                  // [kBins]
  unsigned* begins = table + kBins;                       // [kFineMax / 16]
  unsigned* keys = begins + kFineMax / 16;                // [TILE]
  uint2* runs = reinterpret_cast<uint2*>(keys + TILE);    // [TILE / 32] of 32 places: the first one's run, a bit for each place that begins one
  const int tid = threadIdx.x;
  const FineMap map(st);
  const bool many = st->n_buckets > kMaxBuckets / 2;
  for (int i = tid; i < kBins; i += kPartThreads) table[i] = table_g[i];
  for (int i = tid; i <= map.last / 16; i += kPartThreads) begins[i] = begins_g[i];
  long long t0 = (long long)blockIdx.x * TILE;
  unsigned v[ITEMS];
  auto load = [&](long long t) {
    if (t >= n) return;
    const int left = (int)min((long long)TILE, n - t);
    const unsigned* p = in + t + tid;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      if (j * kPartThreads + tid < left) v[j] = __ldcs(p + j * kPartThreads);
  };
  load(t0);
  for (; t0 < n; t0 += (long long)gridDim.x * TILE) {
    const int left = (int)min((long long)TILE, n - t0);
    reinterpret_cast<uint4*>(at)[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (many) reinterpret_cast<uint4*>(at)[kPartThreads + tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (tid < TILE / 32) runs[tid] = make_uint2(0u, 0u);          // (the last tile's have been read)
    if (tid == 0) n_long = 0;
    unsigned place[ITEMS];                                // bucket << 16 | rank
    auto classify = [&](auto whole) {
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        if (decltype(whole)::value || j * kPartThreads + tid < left) {
          const int f = map.of(key_of(v[j]), table);
          const unsigned w = begins[f >> 4], b = (unsigned)(((int)w >> 16) + __popc(w << ((~f & 15) | 16)));
          place[j] = b << 16 | atomicAdd(&at[b], 1u);
        }
    };
    if (left == TILE) classify(std::true_type()); else classify(std::false_type());
    __syncthreads();
    // places in the output (neighbouring lanes ask for neighbouring buckets: an atomic's cost is its sectors), then places in the
    // tile, BPT neighbouring buckets a thread
    auto reserve = [&](auto bpt) {
      constexpr int BPT = decltype(bpt)::value;
      unsigned g[BPT], e = 0;
      bool had[BPT];
#pragma unroll
      for (int q = 0; q < BPT; ++q) {
        const unsigned c = at[q * kPartThreads + tid];
        had[q] = c != 0;
        if (c) g[q] = atomicAdd(cursor + q * kPartThreads + tid, c);
      }
      // (counts of at most TILE keys in the low half, buckets with keys in the upper one)
      uint4* mine = reinterpret_cast<uint4*>(at) + tid * (BPT / 4);
#pragma unroll
      for (int q = 0; q < BPT / 4; ++q) {
        const uint4 w = mine[q];
        e += w.x + w.y + w.z + w.w + (((w.x != 0) + (w.y != 0) + (w.z != 0) + (w.w != 0)) << 16);
      }
      e = block_exclusive<kPartThreads / 32>(e, part);
#pragma unroll
      for (int q = 0; q < BPT / 4; ++q) {
        uint4 w = mine[q];
        // a bucket's first place in the tile and its run's number; the words of 32 places whose first one it has
        auto place_run = [&](unsigned& w1) {
          const unsigned first = e & 0xffffu, run = e >> 16, c = w1;
          w1 = e;
          if (c) {
            atomicOr(&runs[first >> 5].y, 1u << (first & 31u));
            if (c >= kLong) long_runs[atomicAdd(&n_long, 1)] = make_uint2(first | c << 16, run);
            else
              for (unsigned word = (first + 31u) >> 5; 32u * word < first + c; ++word) runs[word].x = run;
            e += c + 0x10000u;
          }
        };
        place_run(w.x); place_run(w.y); place_run(w.z); place_run(w.w);
        mine[q] = w;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < BPT; ++q) {
        const unsigned w = at[q * kPartThreads + tid];
        if (had[q]) delta[w >> 16] = g[q] - (w & 0xffffu);
      }
      for (int i = tid >> 5; i < n_long; i += kPartThreads / 32) {        // a warp for each (sorted inputs have nothing else)
        const unsigned first = long_runs[i].x & 0xffffu, end = first + (long_runs[i].x >> 16);
        for (unsigned word = ((first + 31u) >> 5) + (tid & 31u); 32u * word < end; word += 32u) runs[word].x = long_runs[i].y;
      }
    };
    if (many) reserve(std::integral_constant<int, kMaxBuckets / kPartThreads>());
    else reserve(std::integral_constant<int, kMaxBuckets / 2 / kPartThreads>());
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      if (j * kPartThreads + tid < left) {
        keys[(at[place[j] >> 16] + place[j]) & 0xffffu] = v[j];
      }
    load(t0 + (long long)gridDim.x * TILE);
    __syncthreads();
    // a warp's 32 places lie in one word: the runs that begin after the first place, counted
#pragma unroll 4
    for (int i = tid; i < left; i += kPartThreads) {
      const uint2 w = runs[i >> 5];
      out[delta[w.x + (unsigned)__popc(w.y & (0xffffffffu >> (31 - (i & 31))) & ~1u)] + (unsigned)i] = keys[i];
    }
  }
}

// Batcher's merge exchange of sixteen: 63 comparisons in ten steps
__device__ __forceinline__ void network16(unsigned (&v)[16]) {
  auto order = [&](int a, int b) {
    const unsigned lo = min(v[a], v[b]);
    v[b] ^= v[a] ^ lo;
    v[a] = lo;
  };
  order(0, 1); order(2, 3); order(4, 5); order(6, 7); order(8, 9); order(10, 11); order(12, 13); order(14, 15);
  order(0, 2); order(1, 3); order(4, 6); order(5, 7); order(8, 10); order(9, 11); order(12, 14); order(13, 15);
  order(1, 2); order(5, 6); order(9, 10); order(13, 14);
  order(0, 4); order(1, 5); order(2, 6); order(3, 7); order(8, 12); order(9, 13); order(10, 14); order(11, 15);
  order(2, 4); order(3, 5); order(10, 12); order(11, 13);
  order(1, 2); order(3, 4); order(5, 6); order(9, 10); order(11, 12); order(13, 14);
  order(0, 8); order(1, 9); order(2, 10); order(3, 11); order(4, 12); order(5, 13); order(6, 14); order(7, 15);
  order(4, 8); order(5, 9); order(6, 10); order(7, 11);
  order(2, 4); order(3, 5); order(6, 8); order(7, 9); order(10, 12); order(11, 13);
  order(1, 2); order(3, 4); order(5, 6); order(7, 8); order(9, 10); order(11, 12); order(13, 14);
}

constexpr int kSortThreads = 512, kSortItems = kCap / kSortThreads, kParts = 16384;
constexpr int kSortSmem = (kCap + 16) * 4 + kParts * 2;
// Place i of the keys in shared memory: the 16-byte words of a group of sixteen keys in an order that depends on the group, so
// that threads that read neighbouring groups do not meet in a bank.
__device__ __forceinline__ unsigned spread(unsigned i) { return i ^ ((i >> 3) & 12u); }

// Sixteen neighbours at a time, twice, the second time half a step further: parts of up to eight keys are in order then, and no
// key leaves its part.
__device__ __forceinline__ void sort_small_parts(unsigned* keys, int cnt) {
  const int groups = (cnt + 15) / 16;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    for (int g = threadIdx.x; g < groups; g += kSortThreads) {
      unsigned v[16];
      const unsigned i0 = (unsigned)(g * 16 + half * 8);
      if (half && (int)i0 + 8 >= cnt) break;                // nothing behind the half group
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 w = *reinterpret_cast<const uint4*>(keys + spread(i0 + 4 * q));
        v[4 * q] = w.x; v[4 * q + 1] = w.y; v[4 * q + 2] = w.z; v[4 * q + 3] = w.w;
      }
      network16(v);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(keys + spread(i0 + 4 * q)) = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
    __syncthreads();
  }
}

// cnt keys at `from` by one warp: bitonic merges whose comparisons all put the smaller key first, so that the places behind the
// last key, up to a power of two, need not be there.
__device__ void sort_by_warp(unsigned* keys, unsigned from, unsigned cnt) {
  const unsigned lane = threadIdx.x & 31;
  unsigned size = 16, lo = 0xffffffffu, hi = 0u;
  for (unsigned i = lane; i < cnt; i += 32) {
    lo = min(lo, keys[spread(from + i)]);
    hi = max(hi, keys[spread(from + i)]);
  }
  if (__reduce_min_sync(0xffffffffu, lo) == __reduce_max_sync(0xffffffffu, hi)) return;        // one value
  while (size < cnt) size *= 2;
  auto order = [&](unsigned a, unsigned b) {
    if (b >= cnt) return;
    unsigned &p = keys[spread(from + a)], &q = keys[spread(from + b)];
    const unsigned u = p, v = q;
    if (u > v) {
      p = v;
      q = u;
    }
  };
  for (unsigned k = 2; k <= size; k *= 2) {
    for (unsigned t = lane; t < size / 2; t += 32) {
      const unsigned block = t & ~(k / 2 - 1), off = t & (k / 2 - 1);
      order(2 * block + off, 2 * block + k - 1 - off);
    }
    __syncwarp();
    for (unsigned j = k / 4; j > 0; j /= 2) {
      for (unsigned t = lane; t < size / 2; t += 32) {
        const unsigned a = 2 * t - (t & (j - 1));
        order(a, a + j);
      }
      __syncwarp();
    }
  }
}

// SINGLE: the whole array is one bucket, read from `in` (the call's first kernel: no __restrict__, its loads may not become
// non-coherent ones, as an earlier kernel may still be writing the weights while this one starts); otherwise the buckets of x,
// in place, the next one's keys on their way while one is sorted.
template <bool SINGLE>
__global__ void __launch_bounds__(kSortThreads, 2) sort_buckets_kernel(const unsigned* in, long long n, SortState* st,
                                                                       const unsigned* first, unsigned* x, uint2* uneven) {
  extern __shared__ __align__(16) unsigned sm[];
  __shared__ unsigned part[kSortThreads / 32 + 1], lo_s[kSortThreads / 32], hi_s[kSortThreads / 32], most_s[kSortThreads / 32];
  unsigned* keys = sm;                              // [kCap + 16]
  unsigned* bins = sm + kCap + 16;                  // [kParts / 2] two 16-bit counts a word, then two first places
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int nb = 1;
  wait_for_last_kernel();
  let_next_kernel_start();
  if (!SINGLE) {
    if (__syncthreads_or(tid == 0 && st->general)) return;        // (asked once: another CTA may be setting it)
    nb = st->n_buckets;
    if (st->large) {
      // Every CTA takes a stretch of the array and compares what lies in buckets of more than kCap keys with their first one.
      const unsigned a = (unsigned)(n * blockIdx.x / gridDim.x), e = (unsigned)(n * (blockIdx.x + 1) / gridDim.x);
      int l = 0, h = nb - 1;                        // the bucket of place a
      while (l < h) {
        const int m = (l + h + 1) >> 1;
        if (first[m] <= a) l = m; else h = m - 1;
      }
      bool same = true;
      for (; l < nb && first[l] < e; ++l) {
        const unsigned f0 = first[l], f1 = first[l + 1];
        if (f1 - f0 <= (unsigned)kCap) continue;
        const unsigned want = value_of(__ldcg(x + f0)), to = min(f1, e);
        unsigned ones = 0xffffffffu, any = 0u;
#pragma unroll 4
        for (unsigned i = max(f0, a) + tid; i < to; i += kSortThreads) {
          const unsigned v = __ldcg(x + i);
          ones &= v;
          any |= v;
          same = same && value_of(v) == want;
        }
        if (want == 0u && ones <= any) {                  // (some were read)
          const int zeros = (ones == 0u ? 1 : 0) | (any != 0u ? 2 : 0);
          if (~st->zeros & zeros) atomicOr(&st->zeros, zeros);
        }
      }
      if (!same) st->general = 1;
    }
  }
  unsigned k[kSortItems], at = 0;
  int cnt = (int)n;
  unsigned at_next = 0, end_next = 0;               // of the bucket to be loaded next
  auto look = [&](int b) {
    at_next = end_next = 0;
    if (!SINGLE && b < nb) {
      at_next = first[b];
      end_next = first[b + 1];
    }
  };
  auto reload = [&]() {
    const unsigned* src = SINGLE ? in : x + at;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
      if (j * kSortThreads + tid < cnt) k[j] = __ldcs(src + j * kSortThreads + tid);
  };
  auto load = [&]() {
    if (!SINGLE) {
      at = at_next;
      cnt = (int)(end_next - at_next);
      if (cnt == 1 && tid == 0) {                     // nothing to sort, but it may be the only zero of its sign
        const unsigned v = __ldcg(x + at);
        if (value_of(v) == 0u) atomicOr(&st->zeros, v == 0u ? 1 : 2);
      }
      if (cnt < 2 || cnt > kCap) cnt = 0;             // one key, or one value (see above)
    }
    reload();
  };
  look(blockIdx.x);
  load();
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    look(b + gridDim.x);
    if (cnt == 0) {
      load();
      continue;
    }
    unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int i = 0; i < kParts / 8 / kSortThreads; ++i) reinterpret_cast<uint4*>(bins)[i * kSortThreads + tid] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
      if (j * kSortThreads + tid < cnt) {
        k[j] = key_of(k[j]);
        lo = min(lo, k[j]);
        hi = max(hi, k[j]);
      }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { lo_s[warp] = lo; hi_s[warp] = hi; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lo_s[lane & (kSortThreads / 32 - 1)]);
    hi = __reduce_max_sync(0xffffffffu, hi_s[lane & (kSortThreads / 32 - 1)]);
    if (SINGLE && tid == 0) st->general = st->n_uneven = 0;
    if (lo <= 0x80000000u && hi >= 0x7fffffffu) {
      int zeros = 0;
#pragma unroll
      for (int j = 0; j < kSortItems; ++j)
        if (j * kSortThreads + tid < cnt && k[j] - 0x7fffffffu <= 1u) zeros |= k[j] == 0x80000000u ? 1 : 2;
      const int pos = __syncthreads_or(zeros & 1), neg = __syncthreads_or(zeros & 2);
      zeros = (pos ? 1 : 0) | (neg ? 2 : 0);
      if (tid == 0) { if (SINGLE) st->zeros = zeros; else atomicOr(&st->zeros, zeros); }
    } else if (SINGLE && tid == 0) {
      st->zeros = 0;
    }
    // The part of a key, monotone in the key: one value each if there are enough parts for the range, else equal stretches of
    // the range of the keys' values, over which they are spread smoothly (the bits of one binary order of magnitude have half the
    // density of the one below); or of their bits, where 512 of the keys say so (a tail of many orders of magnitude).
    const unsigned span = hi - lo;
    const bool exact = span < (unsigned)kParts;
    const unsigned up = exact ? 1u : 0u, factor = exact ? 0x80000000u : (unsigned)(((unsigned long long)kParts << 32) / ((unsigned long long)span + 1ull));
    const float low = __uint_as_float(raw_of(lo)), scale = (float)kParts / (__uint_as_float(raw_of(hi)) - low);
    auto by_bits = [&](unsigned key) { return __umulhi((key - lo) << up, factor); };
    auto by_value = [&](unsigned key) {
      return min(__float2uint_rz(__fmul_rn(__fsub_rn(__uint_as_float(raw_of(key)), low), scale)), (unsigned)kParts - 1u);
    };
    bool value = span >> 23 && scale > 0.0f && scale < 3e38f;          // a binary order of magnitude or more, finite
    if (value) {
      __shared__ unsigned coarse[128];
      if (tid < 128) coarse[tid] = 0u;
      __syncthreads();
      if (tid < cnt) {
        atomicAdd(&coarse[by_bits(k[0]) >> 8], 1u);
        atomicAdd(&coarse[64 + (by_value(k[0]) >> 8)], 1u);
      }
      __syncthreads();
      const unsigned most_bits = __reduce_max_sync(0xffffffffu, max(coarse[lane], coarse[lane + 32]));
      const unsigned most_value = __reduce_max_sync(0xffffffffu, max(coarse[lane + 64], coarse[lane + 96]));
      value = 2 * most_value <= 3 * most_bits;
    }
    unsigned rank[kSortItems / 2];
    unsigned most = 0;
    auto count = [&](auto part_of) {
#pragma unroll
      for (int j = 0; j < kSortItems; ++j) {
        unsigned r = 0;
        if (j * kSortThreads + tid < cnt) {
          const unsigned p = part_of(k[j]), s = (p & 1u) * 16u;
          r = (atomicAdd(&bins[p >> 1], 1u << s) >> s) & 0xffffu;
          most = max(most, r);
        }
        rank[j / 2] = (j & 1) ? rank[j / 2] | r << 16 : r;
      }
    };
    if (value) count(by_value); else count(by_bits);
    most = exact ? 0u : __reduce_max_sync(0xffffffffu, most);
    // (not hi_s: a warp without keys comes here while others still read that, no barrier lies between on the usual way)
    if (lane == 0) most_s[warp] = most;
    __syncthreads();
    most = __reduce_max_sync(0xffffffffu, most_s[lane & (kSortThreads / 32 - 1)]);
    const bool far = most >= 8, loose = most >= 1;       // parts of more than eight keys, of more than one
    {
      // first places: 32 parts a thread, read twice (their counts beside the keys and ranks would not fit the registers)
      constexpr int Q = kParts / 8 / kSortThreads;
      uint4* mine = reinterpret_cast<uint4*>(bins) + tid * Q;
      unsigned sum = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const uint4 v = mine[i];
        sum += v.x + v.y + v.z + v.w;                 // two sums of 16 bits: at most kCap together
      }
      unsigned e = block_exclusive<kSortThreads / 32>((sum & 0xffffu) + (sum >> 16), part);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        uint4 v = mine[i];
        auto place = [&](unsigned& w) {
          const unsigned a = w & 0xffffu, b = w >> 16;
          w = e | (e + a) << 16;
          e += a + b;
        };
        place(v.x); place(v.y); place(v.z); place(v.w);
        mine[i] = v;
      }
    }
    __syncthreads();
    auto scatter = [&](auto part_of) {
#pragma unroll
      for (int j = 0; j < kSortItems; ++j)
        if (j * kSortThreads + tid < cnt) {
          const unsigned p = part_of(k[j]);
          const unsigned to = ((bins[p >> 1] >> ((p & 1u) * 16u)) & 0xffffu) + ((rank[j / 2] >> ((j & 1) * 16)) & 0xffffu);
          keys[spread(to)] = k[j];
        }
    };
    if (value) scatter(by_value); else scatter(by_bits);
    const unsigned to0 = at;
    const int sorted = cnt;
    // the network's groups are whole: what lies behind the last key stays there
    if (tid < 24 && sorted + tid < (sorted + 15) / 16 * 16 + 8) keys[spread((unsigned)(sorted + tid))] = 0xffffffffu;
    if (!SINGLE) load();
    __syncthreads();
    if (loose) {
      for (bool again = false;; again = true) {
        // parts of more than eight keys; many in a part are often one value repeated, among others that are, in order as it is
        if (far && (again || most >= 64)) {
          bool bad = false;
          for (int i = tid + 1; i < sorted; i += kSortThreads) {
            const unsigned u = keys[spread(i - 1)], v = keys[spread(i)];
            bad = bad || (u > v && (u != 0x80000000u || v != 0x7fffffffu));          // (zeros of either sign are equal)
          }
          if (!__syncthreads_or(bad)) break;
          if (again) {
            if (tid == 0) uneven[atomicAdd(&st->n_uneven, 1)] = make_uint2(to0, (unsigned)sorted);
            break;
          }
        } else if (again) {
          break;
        }
        sort_small_parts(keys, sorted);
      }
    }
#pragma unroll 8
    for (int i = tid; i < sorted; i += kSortThreads) __stcg(x + to0 + i, raw_of(keys[spread(i)]));
  }
}

// A bucket that equal stretches of its range leave with too many keys in one of them (an infinity among ordinary weights, values
// repeated in the tail of others): a run of keys is counted in kCoarse equal stretches of its range, these are divided into parts, as
// many as their keys ask for, kParts in all, and the keys are placed by parts.  Up to eight keys of a part are left to the network, up
// to kWarpKeys to a warp, more are a run of their own, of at most a 256th of the range: a key is placed three times at most, and of
// 16384 keys at most 31 runs wait at any time.  (One bitonic sort of the bucket took 150 to 200 us: 925 K weights on 255 levels with
// 10 % of others 349 us the whole call, 213 so; 4 M weights, 300 of them infinite 319, 239.)
constexpr unsigned kWarpKeys = 512;
constexpr int kCoarse = 512;
static_assert(kCoarse == kSortThreads, "a thread has one coarse stretch");
__device__ __forceinline__ void sort_uneven_bucket(unsigned* x, int cnt, SortState* st, unsigned* keys, unsigned* bins) {
  __shared__ uint2 runs[kCap / kWarpKeys];          // first place, keys
  __shared__ unsigned full[kCap / 9];               // parts for a warp: first place << 16 | keys
  __shared__ int n_runs, n_full;
  __shared__ unsigned part[kSortThreads / 32 + 1], lo_s[kSortThreads / 32], hi_s[kSortThreads / 32];
  __shared__ unsigned table[kCoarse];               // keys of a coarse stretch, then its first part << 16 | its parts
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll 8
  for (int i = tid; i < cnt; i += kSortThreads) {
    const unsigned v = __ldcg(x + i);
    if (v == 0x80000000u) atomicOr(&st->zeros, 3);          // one value with positive zeros here: written again by the next kernel
    keys[spread(i)] = key_of(value_of(v));
  }
  if (tid < 24 && cnt + tid < (cnt + 15) / 16 * 16 + 8) keys[spread((unsigned)(cnt + tid))] = 0xffffffffu;
  if (tid == 0) {
    runs[0] = make_uint2(0u, (unsigned)cnt);
    n_runs = 1;
  }
  __syncthreads();
  while (n_runs > 0) {
    const uint2 run = runs[n_runs - 1];
    const unsigned from = run.x, c = run.y;
    unsigned k[kSortItems], lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
      if ((unsigned)(j * kSortThreads + tid) < c) {
        k[j] = keys[spread(from + j * kSortThreads + tid)];
        lo = min(lo, k[j]);
        hi = max(hi, k[j]);
      }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { lo_s[warp] = lo; hi_s[warp] = hi; }
    table[tid] = 0u;
#pragma unroll
    for (int i = 0; i < kParts / 2 / kSortThreads; ++i) bins[i * kSortThreads + tid] = 0u;
    __syncthreads();                                // (also: every thread has read the run)
    if (tid == 0) {
      --n_runs;
      n_full = 0;
    }
    lo = __reduce_min_sync(0xffffffffu, lo_s[lane & (kSortThreads / 32 - 1)]);
    hi = __reduce_max_sync(0xffffffffu, hi_s[lane & (kSortThreads / 32 - 1)]);
    const unsigned span = hi - lo;
    if (span == 0) {
      __syncthreads();
      continue;
    }
    const bool exact = span < (unsigned)kParts;     // a part for every value
    const int shift = exact ? 0 : 32 - __clz(span) - 9;
    if (!exact) {
#pragma unroll
      for (int j = 0; j < kSortItems; ++j)
        if ((unsigned)(j * kSortThreads + tid) < c) atomicAdd(&table[(k[j] - lo) >> shift], 1u);
      __syncthreads();
      const unsigned parts = min(1u + table[tid] * (unsigned)(kParts - kCoarse) / c, 1u << min(shift, 15));        // (16384 x 15872 fits)
      const unsigned first = block_exclusive<kSortThreads / 32>(parts, part);
      table[tid] = first << 16 | parts;
      __syncthreads();
    }
    auto part_of = [&](unsigned key) {
      const unsigned d = key - lo;
      if (exact) return d;
      const unsigned e = table[d >> shift];
      return (e >> 16) + __umulhi(d << (32 - shift), e & 0xffffu);
    };
    // the next place of a key's part; a warp whose keys are of one part (a value repeated: the bucket comes in the order of its parts)
    // asks once (11000 equal keys one by one take 20 us)
    auto next_of = [&](unsigned key, bool in) {
      const unsigned p = in ? part_of(key) : 0xffffffffu, s = (p & 1u) * 16u;
      const unsigned p0 = __shfl_sync(0xffffffffu, p, 0);
      unsigned v = 0;
      if (__all_sync(0xffffffffu, in && p == p0)) {
        if (lane == 0) v = atomicAdd(&bins[p >> 1], 32u << s);
        return ((__shfl_sync(0xffffffffu, v, 0) >> s) & 0xffffu) + lane;
      }
      if (in) v = atomicAdd(&bins[p >> 1], 1u << s);
      return (v >> s) & 0xffffu;
    };
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
      if ((unsigned)(j * kSortThreads + warp * 32) < c) next_of(k[j], (unsigned)(j * kSortThreads + tid) < c);
    __syncthreads();
    constexpr int Q = kParts / 8 / kSortThreads;
    uint4* mine = reinterpret_cast<uint4*>(bins) + tid * Q;
    unsigned sum = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const uint4 v = mine[i];
      sum += v.x + v.y + v.z + v.w;
    }
    unsigned e = block_exclusive<kSortThreads / 32>((sum & 0xffffu) + (sum >> 16), part);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      uint4 v = mine[i];
      auto place = [&](unsigned& w) {
        const unsigned first = w & 0xffffu, second = w >> 16;
        w = e | (e + first) << 16;
        e += first + second;
      };
      place(v.x); place(v.y); place(v.z); place(v.w);
      mine[i] = v;
    }
    __syncthreads();
    // every key takes its part's next place: the word of a part then says where it ends
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
      if ((unsigned)(j * kSortThreads + warp * 32) < c) {
        const bool in = (unsigned)(j * kSortThreads + tid) < c;
        const unsigned to = next_of(k[j], in);
        if (in) keys[spread(from + to)] = k[j];
      }
    __syncthreads();
    if (exact) continue;
    for (int w = tid; w < kParts / 2; w += kSortThreads) {
      const unsigned ends = bins[w], a = w ? bins[w - 1] >> 16 : 0u, b = ends & 0xffffu, z = ends >> 16;
      auto look = [&](unsigned first, unsigned end) {
        if (end - first > kWarpKeys) runs[atomicAdd(&n_runs, 1)] = make_uint2(from + first, end - first);
        else if (end - first > 8) full[atomicAdd(&n_full, 1)] = (from + first) << 16 | (end - first);
      };
      look(a, b);
      look(b, z);
    }
    __syncthreads();
    for (int i = warp; i < n_full; i += kSortThreads / 32) sort_by_warp(keys, full[i] >> 16, full[i] & 0xffffu);
    __syncthreads();
  }
  sort_small_parts(keys, cnt);
#pragma unroll 8
  for (int i = tid; i < cnt; i += kSortThreads) __stcg(x + i, raw_of(keys[spread(i)]));
  __syncthreads();
}

__global__ void __launch_bounds__(kSortThreads, 2) sort_uneven_kernel(SortState* st, const uint2* uneven, unsigned* x) {
  extern __shared__ __align__(16) unsigned sm[];
  wait_for_last_kernel();
  let_next_kernel_start();
  const int n = st->n_uneven;
  for (int i = blockIdx.x; i < n; i += gridDim.x) sort_uneven_bucket(x + uneven[i].x, (int)uneven[i].y, st, sm, sm + kCap + 16);
}

// ---- the general sort: four stable passes of eight bits ---------------------------------------------------
constexpr int kRadixThreads = 512, kRadixWarps = kRadixThreads / 32, kRadixRows = 16, kRadixTile = kRadixThreads * kRadixRows;
constexpr int kRadixGridMax = 512;
__device__ __forceinline__ unsigned digit_of(unsigned raw, int shift) { return (key_of(value_of(raw)) >> shift) & 255u; }

__global__ void __launch_bounds__(kRadixThreads, 2) sort_general_kernel(const unsigned* __restrict__ in, long long n, const SortState* __restrict__ st,
                                                                        unsigned* x, unsigned* tmp, unsigned* counts) {
  namespace cg = cooperative_groups;
  if (!st->general && st->zeros != 3) return;
  __shared__ unsigned keys[kRadixTile];
  __shared__ unsigned short warp_cnt[kRadixWarps][256];
  __shared__ unsigned run[256], delta[256], part[kRadixWarps + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = gridDim.x;
  const long long tiles = (n + kRadixTile - 1) / kRadixTile;
  const long long tile0 = tiles * blockIdx.x / G, tile1 = tiles * (blockIdx.x + 1) / G;
  const long long from = tile0 * kRadixTile, to = min(n, tile1 * kRadixTile);
  if (!st->general) {
    // Sorted but for the zeros, which belong in the order of the input: count them, find their place, write them again.
    const int full = (int)((to - from + kRadixThreads - 1) / kRadixThreads);
    int mine = 0;
#pragma unroll 8
    for (int j = 0; j < full; ++j) {
      const long long i = from + (long long)j * kRadixThreads + tid;
      if (i < to) mine += value_of(in[i]) == 0u;
    }
    mine = (int)__reduce_add_sync(0xffffffffu, (unsigned)mine);
    if (tid == 0) run[0] = 0u;
    __syncthreads();
    if (lane == 0) atomicAdd(&run[0], (unsigned)mine);
    __syncthreads();
    if (tid == 0) __stcg(counts + blockIdx.x, run[0]);
    cg::this_grid().sync();
    if (run[0] == 0u) return;
    unsigned place = 0;
    if (warp == 0) {
      for (int c = lane; c < (int)blockIdx.x; c += 32) place += __ldcg(counts + c);
      place = __reduce_add_sync(0xffffffffu, place);
      long long l = 0, h = n;                       // first place of x that does not lie before the zeros
      while (l < h) {
        const long long step = (h - l + 31) / 32, at = l + lane * step;
        const bool before = at < h && key_of(value_of(__ldcg(x + at))) < 0x80000000u;
        const int c = 32 - __clz(__ballot_sync(0xffffffffu, before));
        if (c == 0) break;
        l += (c - 1) * step + 1;
        h = min(h, l + step - 1);
      }
      if (lane == 0) run[1] = (unsigned)l + place;
    }
    __syncthreads();
    unsigned next = run[1];
    for (int j = 0; j < full; ++j) {
      const long long i = from + (long long)j * kRadixThreads + tid;
      const unsigned v = i < to ? in[i] : 1u;
      const bool zero = value_of(v) == 0u;
      if (!__syncthreads_or(zero)) continue;
      const unsigned e = block_exclusive<kRadixWarps>(zero ? 1u : 0u, part);
      if (zero) __stcg(x + next + e, v);
      next += part[kRadixWarps];
      __syncthreads();
    }
    return;
  }
  for (int pass = 0; pass < 4; ++pass) {
    const unsigned* src = pass == 0 ? in : (pass & 1) ? tmp : x;
    unsigned* dst = (pass & 1) ? x : tmp;
    const int shift = 8 * pass;
    if (tid < 256) run[tid] = 0u;
    __syncthreads();
    for (long long i0 = from; i0 < to; i0 += 8 * kRadixThreads) {
      unsigned v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (i0 + j * kRadixThreads + tid < to) v[j] = __ldcg(src + i0 + j * kRadixThreads + tid);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (i0 + j * kRadixThreads + tid < to) atomicAdd(&run[digit_of(v[j], shift)], 1u);
    }
    __syncthreads();
    if (tid < 256) __stcg(counts + blockIdx.x * 256 + tid, run[tid]);
    cg::this_grid().sync();
    // where this CTA's keys of every digit go: after all smaller digits, and after the CTAs before it
    unsigned mine = 0, all = 0;
    if (tid < 256) {
#pragma unroll 8
      for (int c = 0; c < G; ++c) {
        const unsigned v = __ldcg(counts + c * 256 + tid);
        all += v;
        mine += c < (int)blockIdx.x ? v : 0u;
      }
    }
    const unsigned smaller = block_exclusive<kRadixWarps>(all, part);
    if (tid < 256) run[tid] = smaller + mine;
    for (long long t = tile0; t < tile1; ++t) {
      const long long base = t * kRadixTile;
      const int left = (int)min((long long)kRadixTile, n - base);
      __syncthreads();
      for (int i = lane; i < 128; i += 32) reinterpret_cast<unsigned*>(warp_cnt[warp])[i] = 0u;
      __syncwarp();
      // a warp has 512 neighbouring keys, 32 at a time in order
      unsigned v[kRadixRows];
      unsigned rank[kRadixRows];
#pragma unroll
      for (int j = 0; j < kRadixRows; ++j) {
        const int i = warp * (32 * kRadixRows) + 32 * j + lane;
        v[j] = i < left ? __ldcg(src + base + i) : 0u;
      }
#pragma unroll
      for (int j = 0; j < kRadixRows; ++j) {
        const bool in_tile = warp * (32 * kRadixRows) + 32 * j + lane < left;
        const unsigned d = digit_of(v[j], shift);
        unsigned same = __ballot_sync(0xffffffffu, in_tile);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const unsigned w = __ballot_sync(0xffffffffu, (d >> b) & 1u);
          same &= ((d >> b) & 1u) ? w : ~w;
        }
        const unsigned before = in_tile ? warp_cnt[warp][d] : 0u, below = __popc(same & ((1u << lane) - 1u));
        rank[j] = before + below;
        __syncwarp();
        if (in_tile && below == 0) warp_cnt[warp][d] = (unsigned short)(before + __popc(same));
        __syncwarp();
      }
      __syncthreads();
      unsigned cnt = 0;
      if (tid < 256) {
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) {
          const unsigned c = warp_cnt[w][tid];
          warp_cnt[w][tid] = (unsigned short)cnt;
          cnt += c;
        }
      }
      const unsigned start = block_exclusive<kRadixWarps>(cnt, part);
      if (tid < 256) {
        delta[tid] = run[tid] - start;
        run[tid] += cnt;
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) warp_cnt[w][tid] = (unsigned short)(warp_cnt[w][tid] + start);
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < kRadixRows; ++j)
        if (warp * (32 * kRadixRows) + 32 * j + lane < left) keys[warp_cnt[warp][digit_of(v[j], shift)] + rank[j]] = v[j];
      __syncthreads();
      for (int i = tid; i < left; i += kRadixThreads) {
        const unsigned v1 = keys[i];
        __stcg(dst + delta[digit_of(v1, shift)] + i, v1);
      }
    }
    cg::this_grid().sync();
  }
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }
struct Layout {
  size_t state, samples, table, fine, begins, first, cursor, uneven, counts, tmp, total;
};
Layout layout(int64_t n) {
  Layout l;
  size_t off = 0;
  l.state = off; off += 256;
  l.samples = off; off += up256(kSamples * 4);
  l.table = off; off += up256(kBins * 4);
  l.fine = off; off += up256(kFineMax * 4);
  l.begins = off; off += up256(kFineMax / 4);
  l.first = off; off += up256((kMaxBuckets + 1) * 4);
  l.cursor = off; off += up256(kMaxBuckets * 4);
  l.uneven = off; off += up256(kMaxBuckets * 8);
  l.counts = off; off += up256(kRadixGridMax * 256 * 4);
  l.tmp = off; off += up256((size_t)n * 4);
  l.total = off;
  return l;
}

template <typename K>
cudaError_t opt_in(K kern, int smem, PerDeviceFlag& flag) {
  int dev;
  if (!flag.first(&dev)) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) flag.done(dev);
  return e;
}

}  // namespace

bool dbci_sort_takes(int64_t n) { return n <= kMostKeys; }
size_t dbci_sort_workspace_bytes(int64_t n) { return layout(n).total; }

cudaError_t launch_dbci_sort(const float* weights, int64_t n, float* sorted, void* workspace, cudaStream_t s) {
  const Layout l = layout(n);
  uint8_t* base = static_cast<uint8_t*>(workspace);
  SortState* st = reinterpret_cast<SortState*>(base + l.state);
  unsigned* samples = reinterpret_cast<unsigned*>(base + l.samples);
  unsigned* table = reinterpret_cast<unsigned*>(base + l.table);
  unsigned* fine = reinterpret_cast<unsigned*>(base + l.fine);
  unsigned* begins = reinterpret_cast<unsigned*>(base + l.begins);
  unsigned* first = reinterpret_cast<unsigned*>(base + l.first);
  unsigned* cursor = reinterpret_cast<unsigned*>(base + l.cursor);
  uint2* uneven = reinterpret_cast<uint2*>(base + l.uneven);
  unsigned* counts = reinterpret_cast<unsigned*>(base + l.counts);
  unsigned* tmp = reinterpret_cast<unsigned*>(base + l.tmp);
  const unsigned* in = reinterpret_cast<const unsigned*>(weights);
  unsigned* x = reinterpret_cast<unsigned*>(sorted);
  static PerDeviceFlag f_count, f_part_l, f_part_s, f_sort, f_single, f_uneven;
  const int sms = current_sm_count();
  cudaError_t e;
  if (n <= kCap) {
    if ((e = opt_in(sort_buckets_kernel<true>, kSortSmem, f_single)) != cudaSuccess) return e;
    e = launch_after(sort_buckets_kernel<true>, 1, kSortThreads, kSortSmem, s, in, (long long)n, st, (const unsigned*)first, x, uneven);
  } else {
    constexpr int L = 24, S = 4;
    if ((e = opt_in(sort_count_kernel, kCountSmem, f_count)) != cudaSuccess) return e;
    if ((e = opt_in(sort_partition_kernel<L>, partition_smem<L>(), f_part_l)) != cudaSuccess) return e;
    if ((e = opt_in(sort_partition_kernel<S>, partition_smem<S>(), f_part_s)) != cudaSuccess) return e;
    if ((e = opt_in(sort_buckets_kernel<false>, kSortSmem, f_sort)) != cudaSuccess) return e;
    // buckets for two CTAs on every SM, if they would not be too small
    const int64_t even = n / (2 * sms);
    const int target = (int)(even < 2048 ? 2048 : even > kTarget ? kTarget : even);
    const int64_t asked = 4 * n / target;
    const int budget = (int)(asked < kFineBudget ? asked : kFineBudget);
    if ((e = launch_after(sort_plan_kernel, kPlanCtas, 1024, 0, s, in, (long long)n, budget, st, samples, table, fine)) != cudaSuccess) return e;
    const int64_t count_tiles = (n + kCountThreads * kCountItems - 1) / (kCountThreads * kCountItems);
    e = launch_after(sort_count_kernel, (unsigned)(count_tiles < 2 * sms ? count_tiles : 2 * sms), kCountThreads, kCountSmem, s, in, (long long)n, st,
                     (const unsigned*)table, fine);
    if (e != cudaSuccess) return e;
    e = launch_after(sort_map_kernel, 1, kMapThreads, 0, s, (long long)n, target, st, fine, (const unsigned*)samples, (const unsigned*)table, begins, first, cursor);
    if (e != cudaSuccess) return e;
    const bool large = n >= (int64_t)kPartThreads * L * sms;
    const int64_t tile = kPartThreads * (large ? L : S), tiles = (n + tile - 1) / tile;
    const unsigned grid = (unsigned)(tiles < sms ? tiles : sms);
    e = launch_after(large ? sort_partition_kernel<L> : sort_partition_kernel<S>, grid, kPartThreads, large ? partition_smem<L>() : partition_smem<S>(), s,
                     in, (long long)n, (const SortState*)st, (const unsigned*)table, (const unsigned*)begins, cursor, x);
    if (e != cudaSuccess) return e;
    const int64_t most = 2 * (n / target) + 2;
    e = launch_after(sort_buckets_kernel<false>, (unsigned)(most < 2 * sms ? most : 2 * sms), kSortThreads, kSortSmem, s, in, (long long)n, st, (const unsigned*)first, x, uneven);
  }
  if (e != cudaSuccess) return e;
  if ((e = opt_in(sort_uneven_kernel, kSortSmem, f_uneven)) != cudaSuccess) return e;
  const int64_t uneven_most = n / 256 + 1;
  e = launch_after(sort_uneven_kernel, (unsigned)(n <= kCap ? 1 : uneven_most < 2 * sms ? uneven_most : 2 * sms), kSortThreads, kSortSmem, s, st, (const uint2*)uneven, x);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sort_general_kernel, kRadixThreads, 0)) != cudaSuccess) return e;
  const int64_t radix_tiles = (n + kRadixTile - 1) / kRadixTile;
  int64_t grid = (int64_t)per_sm * sms;
  grid = grid < kRadixGridMax ? grid : kRadixGridMax;
  grid = grid < radix_tiles ? grid : radix_tiles;
  long long n_arg = n;
  const SortState* st_arg = st;
  void* args[] = {(void*)&in, (void*)&n_arg, (void*)&st_arg, (void*)&x, (void*)&tmp, (void*)&counts};
  return cudaLaunchCooperativeKernel((const void*)sort_general_kernel, dim3((unsigned)grid), dim3(kRadixThreads), args, 0, s);
}

}  // namespace lcd
