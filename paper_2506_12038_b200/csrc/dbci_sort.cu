// The sort of the density-based centroid initialisation: binary32 weights in ascending order, by two passes over the data
// after one that counts.  Weights of a layer are spread smoothly over their range or repeat few values, so a piecewise linear
// map of the (order-preserving) key, fitted to a sample, cuts them into buckets of about kTarget keys that fit the shared
// memory of a CTA:
//   plan      range and histogram of 16384 samples; every bin of 2048 is divided into equal parts, as many as its samples
//             ask for ("fine bins", about 3 K keys of 45 M each; one more at either end for what
//             lies at or beyond the sample's extremes, where clipped weights repeat one value);
//   count     exact counts of the fine bins;
//   map       one CTA: neighbouring fine bins become buckets of at most kCap keys, a larger fine bin a segment of its own;
//   partition every key to its bucket's or segment's place in the output, in no order;
//   segments  nothing, unless there are some: those of one value stay as they are (weights in bf16, clipped or pruned ones), the
//             others (narrow clumps, a value repeated among others) are divided by their own ranges into buckets;
//   buckets   a CTA sorts a bucket where it lies: 16384 equal parts of its range, a place for every key by a counting pass
//             (the shared-memory atomic's result), then sixteen neighbours at a time through a sorting network, twice, the
//             second time half a step further, which puts parts of up to eight keys in order;
//   finish    nothing, unless a bucket's keys lie too close together in places (it is divided again by their density) or
//             there are zeros of either sign: they are equal and keep their order, so they are written again in the input's.
// 45 M Gaussian weights: 560 us (plan 6, count 55, map 15, partition 220, buckets 265), CUB's radix sort 1070; 925 K: 53 and 110.
// Bytes are 0.9 GB, 140 us: what bounds the passes is shared memory at random addresses (a key's three lookups or atomics, a store
// and two loads in the partition, an atomic, a lookup and a store in the buckets, each three to four bank conflicts a warp) and, where the
// partition writes runs of six keys, the sectors that L2 takes.
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
constexpr int kPartsOfChunk = 264;           // counters of a segment, for kCap of its keys: a part for 64 keys, two more and a margin
constexpr int kMaxBuckets = 8192;
constexpr int64_t kMostKeys = (int64_t)(kMaxBuckets / 2 - 1) * kTarget;

// A stretch of the array with more keys than a bucket holds, by chunks of kCap keys.
struct Segment {
  unsigned from, keys;
  unsigned chunk;           // its first one among those of its level
  unsigned lo, hi;          // no key lies outside
  unsigned pivot;           // a key of it, the one that repeats most where one does
  unsigned mixed;           // it has other keys
  unsigned equal, equal_to; // the pivot's places
};
constexpr int kLevels = 4;                   // 32 bits of a key, eight or more a level
constexpr int kPhases = 4 * kLevels + 3;     // of the kernels whose CTAs wait for one another
struct SortState {
  unsigned long long segments[kLevels];      // number << 32 | chunks
  unsigned ticket[kPhases], done[kPhases];
  int mixed[kLevels];       // some segment is
  unsigned kmin, kmax;      // sample extremes
  int shift;                // bin of a key: (key - kmin) >> shift
  int n_fine, n_buckets;
  int n_extra;              // buckets made from segments
  int zeros;                // bit 0: there are positive zeros, bit 1: negative ones
  int n_uneven;             // buckets to be divided again
};
constexpr size_t kStateBytes = 512;
static_assert(sizeof(SortState) <= kStateBytes, "space for the state");

__device__ __forceinline__ unsigned key_of(unsigned raw) { return raw ^ ((unsigned)((int)raw >> 31) | 0x80000000u); }
__device__ __forceinline__ unsigned raw_of(unsigned key) { return key ^ (~(unsigned)((int)key >> 31) | 0x80000000u); }

// The same for zeros of either sign, which are equal.
__device__ __forceinline__ unsigned value_of(unsigned raw) { return raw == 0x80000000u ? 0u : raw; }

// `items` pieces of work of one phase of a kernel, given out one by one to the CTAs that ask, then a wait until all are done.
// Nothing says that the CTAs of a launch run at the same time, so none waits for another one to come: what is not done was taken by
// a CTA that runs.  A CTA that has waited kPolls times (ten milliseconds or more) gets `false` and is to leave; the one that does the last
// piece never waits, goes on, and takes what the others leave.  What one phase writes the next ones read past L1 (__ldcg).
// ahead(i, slot): done by the first warp for a piece of work before its turn (slot: 0 and 1 in turn), the first one at once, the others
// where work(i, slot, look_ahead) calls look_ahead, once in every case.
constexpr int kPolls = 20000;
template <typename Ahead, typename Work>
__device__ __forceinline__ bool run_phase(SortState* st, int phase, unsigned items, Ahead ahead, Work work) {
  __shared__ unsigned given;
  if (items == 0) return true;
  const bool first_warp = threadIdx.x < 32, first = threadIdx.x == 0;
  unsigned mine = 0;
  if (first_warp) {
    if (first) mine = atomicAdd(&st->ticket[phase], 1u);
    mine = __shfl_sync(0xffffffffu, mine, 0);
    if (mine < items) ahead(mine, 0);
  }
  for (int slot = 0;; slot ^= 1) {
    __syncthreads();                      // the last piece's shared memory has been read
    if (first) given = mine;
    __syncthreads();
    const unsigned i = given;
    if (i >= items) break;
    if (first) mine = atomicAdd(&st->ticket[phase], 1u);          // (the next one, while this one is done)
    work(i, slot, [&]() {
      if (!first_warp) return;
      mine = __shfl_sync(0xffffffffu, mine, 0);
      if (mine < items) ahead(mine, slot ^ 1);
    });
    __syncthreads();
    if (first) {
      __threadfence();
      atomicAdd(&st->done[phase], 1u);
    }
  }
  bool all = false;
  if (first) {
    for (int t = 0; t < kPolls && !all; ++t) {
      unsigned done;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(done) : "l"(&st->done[phase]) : "memory");
      all = done >= items;
      if (!all) __nanosleep(100);
    }
  }
  return __syncthreads_or(all);
}
template <typename Work>
__device__ __forceinline__ bool run_phase(SortState* st, int phase, unsigned items, Work work) {
  return run_phase(st, phase, items, [](unsigned, int) {}, [&](unsigned i, int, auto look_ahead) {
    look_ahead();
    work(i);
  });
}

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
  if (tid < (int)(sizeof(SortState) / 4)) reinterpret_cast<unsigned*>(st)[tid] = 0u;
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
  // The keys of a fine bin.  bin: where to look for it, 0 or what an earlier fine bin left there.
  __device__ void bounds(int f, const unsigned* table, int& bin, unsigned& lo, unsigned& hi) const {
    lo = 0u;
    hi = 0xffffffffu;
    if (f == 0) hi = kmin;
    if (f == last) lo = kmax;
    if (f == 0 || f == last) return;
    if (bin == 0)
      for (int s = kBins / 2; s > 0; s /= 2)
        if ((int)(table[bin + s] >> 16) <= f) bin += s;
    while (bin + 1 < kBins && (int)(table[bin + 1] >> 16) <= f) ++bin;
    const unsigned parts = table[bin] & 0xffffu;
    const unsigned long long part = (unsigned)f - (table[bin] >> 16);
    lo = kmin + ((unsigned)bin << shift) + (unsigned)(((part << shift) + parts - 1) / parts);
    hi = kmin + ((unsigned)bin << shift) + (unsigned)((((part + 1) << shift) + parts - 1) / parts) - 1u;
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

// Segments are numbered in the order of their chunks.
__device__ __forceinline__ void add_segment(SortState* st, Segment* segments, int level, unsigned from, unsigned keys, unsigned lo, unsigned hi) {
  const unsigned long long at = atomicAdd(&st->segments[level], 1ull << 32 | (keys + kCap - 1) / kCap);
  Segment* s = segments + (at >> 32);
  s->from = from;
  s->keys = keys;
  s->chunk = (unsigned)at;
  s->lo = lo;
  s->hi = hi;
  s->mixed = 0;
}

// A bucket is a run of fine bins that begin between the same two multiples of `target` in the sorted order; a fine bin that ends
// more than kCap keys after the first of the two begins another one.  So a bucket has at most kCap keys unless it is a fine bin of
// more, and there are at most two for every `target` keys.  Empty fine bins begin none.
// begins: a word for sixteen fine bins, a bit for each that begins a bucket under the number of buckets begun before, less one.
constexpr int kMapThreads = kFineMax / 32, kMapWarps = kMapThreads / 32;
__global__ void __launch_bounds__(kMapThreads) sort_map_kernel(long long n, int target, SortState* st, const unsigned* fine, const unsigned* table, unsigned* __restrict__ begins,
                                                               unsigned* __restrict__ first, unsigned* __restrict__ cursor, Segment* segments) {
  constexpr int PER = 32;
  __shared__ unsigned part[kMapWarps + 1];
  __shared__ unsigned tail[kMapWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  wait_for_last_kernel();
  let_next_kernel_start();
  unsigned c[PER], sum = 0, last = 0;
#pragma unroll
  for (int j = 0; j < PER / 4; ++j) {
    const uint4 v = reinterpret_cast<const uint4*>(fine)[tid * (PER / 4) + j];
    c[4 * j] = v.x; c[4 * j + 1] = v.y; c[4 * j + 2] = v.z; c[4 * j + 3] = v.w;
  }
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    sum += c[j];
    last = c[j] ? c[j] : last;
  }
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
  unsigned large = 0;
  p = at;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if ((starts >> j) & 1u) {
      first[id] = p;
      cursor[id] = p;
      ++id;
    }
    large |= c[j] > (unsigned)kCap ? 1u << j : 0u;
    p += c[j];
  }
  int bin = 0;
  for (; large; large &= large - 1) {
    const int j = __ffs(large) - 1;
    unsigned lo, hi;
    FineMap(st).bounds(tid * PER + j, table, bin, lo, hi);
    if (hi == 0x7fffffffu) hi = 0x80000000u;          // (in a segment zeros of either sign count as positive ones)
    p = at;
    for (int i = 0; i < j; ++i) p += fine[tid * PER + i];
    add_segment(st, segments, 0, p, fine[tid * PER + j], lo, hi);
  }
  if (tid == 0) {
    first[total] = (unsigned)n;
    st->n_buckets = total;
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
                                                                         unsigned* cursor, unsigned* __restrict__ out, unsigned* counters) {
  constexpr int TILE = kPartThreads * ITEMS, kLong = 128;
  extern __shared__ __align__(16) unsigned sm[];
  __shared__ unsigned part[kPartThreads / 32 + 1];
  __shared__ uint2 long_runs[TILE / kLong];
  __shared__ int n_long;
  wait_for_last_kernel();
  let_next_kernel_start();
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
  if (st->segments[0] != 0) {                             // the next kernel's counters
    const unsigned all = (unsigned)st->segments[0] * kPartsOfChunk;
    for (unsigned i = blockIdx.x * kPartThreads + tid; i < all; i += gridDim.x * kPartThreads) counters[i] = 0u;
  }
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

__device__ __forceinline__ bool one_value(const unsigned* keys, unsigned from, unsigned cnt) {          // by a warp
  unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
  for (unsigned i = threadIdx.x & 31; i < cnt; i += 32) {
    const unsigned k = keys[spread(from + i)];
    lo = min(lo, k);
    hi = max(hi, k);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  return lo == hi;
}

// cnt keys at `from` by one warp: bitonic merges whose comparisons all put the smaller key first, so that the places behind the
// last key, up to a power of two, need not be there.
__device__ void sort_by_warp(unsigned* keys, unsigned from, unsigned cnt) {
  const unsigned lane = threadIdx.x & 31;
  if (cnt <= 32) {                        // a key a lane
    unsigned v = lane < cnt ? keys[spread(from + lane)] : 0xffffffffu;
#pragma unroll
    for (unsigned k = 2; k <= 32; k *= 2)
#pragma unroll
      for (unsigned j = k / 2; j > 0; j /= 2) {
        const unsigned o = __shfl_xor_sync(0xffffffffu, v, j == k / 2 ? k - 1 : j);
        v = (lane & j) ? max(v, o) : min(v, o);
      }
    if (lane < cnt) keys[spread(from + lane)] = v;
    __syncwarp();
    return;
  }
  unsigned size = 64;
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
                                                                       const unsigned* first, const uint2* extra, unsigned* x, uint2* uneven) {
  extern __shared__ __align__(16) unsigned sm[];
  __shared__ unsigned part[kSortThreads / 32 + 1], lo_s[kSortThreads / 32], hi_s[kSortThreads / 32], most_s[kSortThreads / 32];
  unsigned* keys = sm;                              // [kCap + 16]
  unsigned* bins = sm + kCap + 16;                  // [kParts / 2] two 16-bit counts a word, then two first places
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  wait_for_last_kernel();
  let_next_kernel_start();
  const int nf = SINGLE ? 1 : st->n_buckets, nb = SINGLE ? 1 : nf + st->n_extra;
  if (SINGLE) {
    if (tid < (int)(sizeof(SortState) / 4)) reinterpret_cast<unsigned*>(st)[tid] = 0u;
    __syncthreads();
  }
  unsigned k[kSortItems], at = 0;
  int cnt = (int)n;
  unsigned at_next = 0, end_next = 0;               // of the bucket to be loaded next
  auto look = [&](int b) {
    at_next = end_next = 0;
    if (!SINGLE && b < nf) {
      at_next = first[b];
      end_next = first[b + 1];
    } else if (!SINGLE && b < nb) {
      const uint2 e = extra[b - nf];
      at_next = e.x;
      end_next = e.x + e.y;
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
      if (cnt < 2 || cnt > kCap) cnt = 0;             // one key, or a segment
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
    if (lo <= 0x80000000u && hi >= 0x7fffffffu) {
      int zeros = 0;
#pragma unroll
      for (int j = 0; j < kSortItems; ++j)
        if (j * kSortThreads + tid < cnt && k[j] - 0x7fffffffu <= 1u) zeros |= k[j] == 0x80000000u ? 1 : 2;
      const int pos = __syncthreads_or(zeros & 1), neg = __syncthreads_or(zeros & 2);
      zeros = (pos ? 1 : 0) | (neg ? 2 : 0);
      if (tid == 0) atomicOr(&st->zeros, zeros);
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
      for (int round = 0;; ++round) {
        // parts of more than eight keys: up to three times where they are not many more (of 45 M Gaussian weights a few buckets have
        // such a part); many in a part are often one value repeated, among others that are, in order as it is
        if (far && (round > 0 || most >= 64)) {
          bool bad = false;
          for (int i = tid + 1; i < sorted; i += kSortThreads) {
            const unsigned u = keys[spread(i - 1)], v = keys[spread(i)];
            bad = bad || (u > v && (u != 0x80000000u || v != 0x7fffffffu));          // (zeros of either sign are equal)
          }
          if (!__syncthreads_or(bad)) break;
          if (round == 3 || (round == 1 && most >= 64)) {
            if (tid == 0) uneven[atomicAdd(&st->n_uneven, 1)] = make_uint2(to0, (unsigned)sorted);
            break;
          }
        } else if (round > 0) {
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
// to kWarpKeys to a warp, more are a run of their own, of at most a 1024th of the range: a key is placed three times at most, and of
// 16384 keys at most 31 runs wait at any time.  (One bitonic sort of the bucket took 150 to 200 us: 925 K weights on 255 levels with
// 10 % of others 349 us the whole call, 178 so; 4 M weights, 300 of them infinite 319, 228.)
constexpr unsigned kWarpKeys = 512;
constexpr int kCoarseLog = 11, kCoarse = 1 << kCoarseLog;
static_assert(kCoarse == 4 * kSortThreads, "a thread has four coarse stretches");
__device__ __forceinline__ void sort_uneven_bucket(unsigned* x, int cnt, SortState* st, unsigned* keys, unsigned* bins, unsigned* source) {
  __shared__ uint2 runs[kCap / kWarpKeys];          // first place, keys
  __shared__ unsigned full[kCap / 9];               // parts of more than eight keys: first place << 16 | keys
  __shared__ int n_runs, n_full;
  __shared__ unsigned part[kSortThreads / 32 + 1], lo_s, hi_s;
  __shared__ uint4 table4[kSortThreads];
  unsigned* table = reinterpret_cast<unsigned*>(table4);          // [kCoarse] keys of a coarse stretch, then its first part << 16 | its parts
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  bool negative = false;
#pragma unroll 8
  for (int i = tid; i < cnt; i += kSortThreads) {
    const unsigned v = __ldcg(x + i);
    negative = negative || v == 0x80000000u;
    source[i] = key_of(value_of(v));
  }
  if (negative) atomicOr(&st->zeros, 3);            // one value with positive zeros here: written again by the next phase
  if (tid < 24 && cnt + tid < (cnt + 15) / 16 * 16 + 8) keys[spread((unsigned)(cnt + tid))] = 0xffffffffu;
  unsigned from = 0, c = (unsigned)cnt;
  if (tid == 0) n_runs = 0;
  for (;;) {
    if (tid == 0) {
      lo_s = 0xffffffffu;
      hi_s = 0u;
      n_full = 0;
    }
    table4[tid] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = 0; i < kParts / 8 / kSortThreads; ++i) reinterpret_cast<uint4*>(bins)[i * kSortThreads + tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    unsigned lo = 0xffffffffu, hi = 0u;
#pragma unroll 4
    for (unsigned i = tid; i < c; i += kSortThreads) {
      const unsigned k = source[i];
      lo = min(lo, k);
      hi = max(hi, k);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      atomicMin(&lo_s, lo);
      atomicMax(&hi_s, hi);
    }
    __syncthreads();
    lo = lo_s;
    hi = hi_s;
    const unsigned span = hi - lo;
    const bool exact = span < (unsigned)kParts;     // a part for every value
    const int shift = exact ? 0 : 32 - __clz(span) - kCoarseLog;
    if (!exact) {
#pragma unroll 4
      for (unsigned i = tid; i < c; i += kSortThreads) atomicAdd(&table[(source[i] - lo) >> shift], 1u);
      __syncthreads();
      uint4 v = table4[tid];
      auto parts = [&](unsigned& w) { w = min(1u + w * (unsigned)(kParts - kCoarse) / c, 1u << min(shift, 15)); };        // (16384 x 14336 fits)
      parts(v.x); parts(v.y); parts(v.z); parts(v.w);
      unsigned first = block_exclusive<kSortThreads / 32>(v.x + v.y + v.z + v.w, part);
      auto entry = [&](unsigned& w) {
        const unsigned of = w;
        w |= first << 16;
        first += of;
      };
      entry(v.x); entry(v.y); entry(v.z); entry(v.w);
      table4[tid] = v;
      __syncthreads();
    }
    auto part_of = [&](unsigned key) {
      const unsigned d = key - lo;
      if (exact) return d;
      const unsigned e = table[d >> shift];
      return (e >> 16) + __umulhi(d << (32 - shift), e & 0xffffu);
    };
    // the next place of a key's part; a warp whose keys are of one part (a value repeated: the bucket comes in the order of its parts)
    // asks once
    auto next_of = [&](unsigned p, bool in) {
      const unsigned s = (p & 1u) * 16u, p0 = __shfl_sync(0xffffffffu, p, 0);
      const bool one = __all_sync(0xffffffffu, in && p == p0);
      unsigned v = 0;
      if (one ? lane == 0 : in) v = atomicAdd(&bins[p >> 1], (one ? 32u : 1u) << s);
      const unsigned v0 = __shfl_sync(0xffffffffu, v, 0);
      return one ? ((v0 >> s) & 0xffffu) + lane : (v >> s) & 0xffffu;
    };
#pragma unroll 2
    for (unsigned i = tid; i - lane < c; i += kSortThreads) next_of(i < c ? part_of(source[i]) : 0xffffffffu, i < c);
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
#pragma unroll 2
    for (unsigned i = tid; i - lane < c; i += kSortThreads) {
      const unsigned k = i < c ? source[i] : 0u, to = next_of(i < c ? part_of(k) : 0xffffffffu, i < c);
      if (i < c) keys[spread(from + to)] = k;
    }
    __syncthreads();
    if (!exact) {
      for (int w = tid; w < kParts / 2; w += kSortThreads) {
        const unsigned ends = bins[w], a = w ? bins[w - 1] >> 16 : 0u, b = ends & 0xffffu, z = ends >> 16;
        if (b - a > 8) full[atomicAdd(&n_full, 1)] = (from + a) << 16 | (b - a);
        if (z - b > 8) full[atomicAdd(&n_full, 1)] = (from + b) << 16 | (z - b);
      }
      __syncthreads();
      for (int i = warp; i < n_full; i += kSortThreads / 32) {
        const unsigned at = full[i] >> 16, of = full[i] & 0xffffu;
        if (one_value(keys, at, of)) continue;
        if (of <= kWarpKeys) sort_by_warp(keys, at, of);
        else if (lane == 0) runs[atomicAdd(&n_runs, 1)] = make_uint2(at, of);
      }
      __syncthreads();
    }
    if (n_runs == 0) break;
    from = runs[n_runs - 1].x;
    c = runs[n_runs - 1].y;
    for (unsigned i = tid; i < c; i += kSortThreads) source[i] = keys[spread(from + i)];
    __syncthreads();
    if (tid == 0) --n_runs;
  }
  sort_small_parts(keys, cnt);
#pragma unroll 8
  for (int i = tid; i < cnt; i += kSortThreads) __stcg(x + i, raw_of(keys[spread(i)]));
  __syncthreads();
}

// After the buckets: those left to be divided again, then the order of the zeros where there are some of either sign.  They are
// equal and belong in the order of the input: by chunks their number and their signs (a bit each), then their place in the sorted
// array, where they are written again.
constexpr int kSignWords = kCap / 32;
constexpr int kFinishSmem = kSortSmem + kCap * 4;
__global__ void __launch_bounds__(kSortThreads, 1) sort_finish_kernel(const unsigned* in, long long n, SortState* st, const uint2* uneven, unsigned* counts,
                                                                      unsigned* all_signs, unsigned* x) {
  extern __shared__ __align__(16) unsigned sm[];
  __shared__ unsigned of_warp[kSortThreads / 32], begin_s;
  wait_for_last_kernel();
  let_next_kernel_start();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!run_phase(st, 4 * kLevels, (unsigned)st->n_uneven, [&](unsigned i) { sort_uneven_bucket(x + uneven[i].x, (int)uneven[i].y, st, sm, sm + kCap + 16, sm + kSortSmem / 4); })) return;
  if (__ldcg(&st->zeros) != 3) return;
  constexpr int kRows = kCap / kSortThreads;
  static_assert(kRows == 32 && kSignWords == kSortThreads, "a lane keeps a row's word, a thread writes one");
  const unsigned chunks = (unsigned)((n + kCap - 1) / kCap);
  if (!run_phase(st, 4 * kLevels + 1, chunks, [&](unsigned chunk) {
        sm[tid] = 0u;
        // a warp has 32 rows of 32 neighbouring weights
        const long long i0 = (long long)chunk * kCap + warp * (32 * kRows) + lane;
        unsigned zeros = 0, negative = 0;              // zeros of the lane's row; the lane's own negative ones, a bit a row
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
          const unsigned v = i0 + 32 * j < n ? __ldcg(in + i0 + 32 * j) : 1u;
          const unsigned row = __ballot_sync(0xffffffffu, value_of(v) == 0u);
          if (lane == j) zeros = row;
          negative |= v == 0x80000000u ? 1u << j : 0u;
        }
        const unsigned mine = __reduce_add_sync(0xffffffffu, (unsigned)__popc(zeros));
        if (lane == 0) of_warp[warp] = mine;
        __syncthreads();
        const unsigned of = lane < kSortThreads / 32 ? of_warp[lane] : 0u;
        unsigned at = __reduce_add_sync(0xffffffffu, lane < warp ? of : 0u);
        const unsigned all = __reduce_add_sync(0xffffffffu, of);
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
          const unsigned row = __shfl_sync(0xffffffffu, zeros, j);
          if ((negative >> j) & 1u) {
            const unsigned i = at + (unsigned)__popc(row & ((1u << lane) - 1u));
            atomicOr(&sm[i >> 5], 1u << (i & 31u));
          }
          at += (unsigned)__popc(row);
        }
        __syncthreads();
        if (32u * tid < all) __stcg(all_signs + (size_t)chunk * kSignWords + tid, sm[tid]);
        if (tid == 0) __stcg(counts + chunk, all);
      }))
    return;
  if (warp == 0) {
    long long l = 0, h = n;                       // the first place of x that does not lie before the zeros
    while (l < h) {
      const long long step = (h - l + 31) / 32, at = l + lane * step;
      const bool before = at < h && key_of(value_of(__ldcg(x + at))) < 0x80000000u;
      const int c = 32 - __clz(__ballot_sync(0xffffffffu, before));
      if (c == 0) break;
      l += (c - 1) * step + 1;
      h = min(h, l + step - 1);
    }
    if (lane == 0) begin_s = (unsigned)l;
  }
  run_phase(st, 4 * kLevels + 2, chunks, [&](unsigned chunk) {
    const unsigned all = __ldcg(counts + chunk);
    if (all == 0u) return;
    unsigned before = 0;
    for (unsigned i = tid; i < chunk; i += kSortThreads) before += __ldcg(counts + i);
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) of_warp[warp] = before;
    if (32u * tid < all) sm[tid] = __ldcg(all_signs + (size_t)chunk * kSignWords + tid);
    __syncthreads();
    unsigned* to = x + (begin_s + __reduce_add_sync(0xffffffffu, lane < kSortThreads / 32 ? of_warp[lane] : 0u));
#pragma unroll 4
    for (unsigned i = tid; i < all; i += kSortThreads) __stcg(to + i, (sm[i >> 5] >> (i & 31u)) << 31);
  });
}

// ---- segments: more keys in one fine bin than a bucket holds ---------------------------------------------------
// A value repeated so often, by itself or among others, or a narrow clump.  Level by level: the segment's range is divided into 256 to
// 2048 equal parts, and the pivot, the median of 32 of its keys, has a part of its own between the smaller and the larger keys of the
// part it lies in.  A segment without other keys is left as it is.  Parts of one value each are written from their counts; otherwise
// the other keys are partitioned (and the pivot's written), parts of few keys become buckets together, and a part of more keys than
// a bucket holds is a segment of the next level, whose range has eight bits less at least.
// 45 M weights, the whole call: 255 levels with 10 % of other weights 992 us, eight clumps of 0.1 % width 1440 (a radix
// sort of the whole array in four passes 1785 and 2037; CUB's 1270 and, with the marking of before, 2775); eight levels: 76 us here.
constexpr int kSegThreads = 512, kSegTile = 8192, kSegItems = kSegTile / kSegThreads, kSegPartsLog = 11;
constexpr int kSegPer = 5, kSegSlots = kSegThreads * kSegPer;       // parts of a thread; of a segment: at most 2048 and two more
constexpr int kSegSmem = (2 * kSegSlots + 4 + kSegTile) * 4;
static_assert((1 << kSegPartsLog) + 2 <= kSegSlots && kCap % kSegTile == 0 && kCap / 64 + 2 <= kPartsOfChunk && kCap >= 64 << 8, "sizes of a segment's parts");

__global__ void __launch_bounds__(kSegThreads, 2) sort_segments_kernel(SortState* st, Segment* all_segments, int per_level, unsigned* all_counters,
                                                                       uint2* extra, unsigned* x, unsigned* tmp) {
  extern __shared__ __align__(16) unsigned sm[];
  unsigned *count = sm, *delta = sm + kSegSlots + 4, *keys = delta + kSegSlots;          // [kSegSlots + 1], [kSegSlots], [kSegTile]
  __shared__ unsigned part[kSegThreads / 32 + 1], tail[kSegThreads / 32], numbers[2];
  __shared__ Segment fetched[2];
  wait_for_last_kernel();
  let_next_kernel_start();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int level = 0; level < kLevels; ++level) {
    const unsigned long long number = __ldcg(&st->segments[level]);
    const unsigned n_segments = (unsigned)(number >> 32), n_chunks = (unsigned)number;
    if (n_segments == 0) return;
    Segment* segments = all_segments + level * per_level;
    auto fetch = [&](unsigned i, int slot) {
      if (lane == 0) numbers[slot] = i;
      if (lane < (int)(sizeof(Segment) / 4)) reinterpret_cast<unsigned*>(&fetched[slot])[lane] = __ldcg(reinterpret_cast<const unsigned*>(segments + i) + lane);
      __syncwarp();
    };
    // the segment of a chunk: the last one whose first chunk does not come after it
    auto find = [&](unsigned chunk, int slot) {
      unsigned l = 0, h = n_segments;           // in [l, h)
      while (h - l > 1) {
        const unsigned step = (h - l + 31) / 32, at = l + lane * step;
        const bool not_after = at < h && __ldcg(&segments[at].chunk) <= chunk;
        l += (unsigned)(__popc(__ballot_sync(0xffffffffu, not_after)) - 1) * step;
        h = min(h, l + step);
      }
      fetch(l, slot);
    };
    // a chunk's places in the array
    auto places = [&](const Segment& seg, unsigned chunk, unsigned& begin, unsigned& end) {
      begin = seg.from + (chunk - seg.chunk) * kCap;
      end = min(begin + kCap, seg.from + seg.keys);
    };
    // equal parts of 2^shift keys each, of one value if it is 0; part_of: the number of a key's part, with the pivot's
    auto shift_of = [&](const Segment& seg) { return max(32 - __clz(seg.hi - seg.lo) - min(31 - __clz(seg.keys / 64), kSegPartsLog), 0); };
    auto key_at = [&](const unsigned* p) { return key_of(value_of(__ldcg(p))); };
    auto part_of = [&](const Segment& seg, unsigned key, int shift) { return ((key - seg.lo) >> shift) + (key > seg.pivot ? 2u : key == seg.pivot ? 1u : 0u); };
    auto parts_of = [&](const Segment& seg, int shift) { return (int)((seg.hi - seg.lo) >> shift) + 3; };

    bool go = run_phase(
        st, 4 * level, n_chunks,
        [&](unsigned chunk, int slot) {
          find(chunk, slot);
          Segment& seg = fetched[slot];
          const unsigned k = key_at(x + seg.from + (unsigned)((unsigned long long)(seg.keys - 1) * lane / 31));
          int less = 0, equal = 0;
#pragma unroll
          for (int l = 0; l < 32; ++l) {
            const unsigned other = __shfl_sync(0xffffffffu, k, l);
            less += other < k;
            equal += other == k;
          }
          const unsigned middle = __ballot_sync(0xffffffffu, less <= 16 && less + equal > 16);
          const unsigned pivot = __shfl_sync(0xffffffffu, k, __ffs(middle) - 1);
          if (lane == 0) {
            seg.pivot = pivot;
            if (chunk == seg.chunk) __stcg(&segments[numbers[slot]].pivot, pivot);
          }
        },
        [&](unsigned chunk, int slot, auto look_ahead) {
          constexpr int kBatch = 16;                // (more would not stay in registers)
          const Segment& seg = fetched[slot];
          unsigned begin, end, v[kBatch];
          places(seg, chunk, begin, end);
          auto load = [&]() {
#pragma unroll
            for (int j = 0; j < kBatch; ++j)
              if (begin + j * kSegThreads + tid < end) v[j] = __ldcg(x + begin + j * kSegThreads + tid);
          };
          load();
          for (int d = tid; d < kSegSlots; d += kSegThreads) count[d] = 0u;
          look_ahead();
          __syncthreads();
          const unsigned pivot = seg.pivot, keys_of = end - begin;
          const int shift = shift_of(seg);
          unsigned others = 0, signs = 0;
          for (;;) {
#pragma unroll
            for (int j = 0; j < kBatch; ++j)
              if (begin + j * kSegThreads + tid < end) {
                const unsigned k = key_of(value_of(v[j]));
                signs |= k != 0x80000000u ? 0u : v[j] == 0u ? 1u : 2u;
                if (k != pivot) {
                  ++others;
                  atomicAdd(&count[part_of(seg, k, shift)], 1u);
                }
              }
            begin += kBatch * kSegThreads;
            if (begin >= end) break;
            load();
          }
          signs = __reduce_or_sync(0xffffffffu, signs);
          others = __reduce_add_sync(0xffffffffu, others);
          if (lane == 0 && signs) atomicOr(&st->zeros, (int)signs);
          unsigned& of_pivot = count[part_of(seg, pivot, shift)];
          if (lane == 0 && others) atomicSub(&of_pivot, others);
          if (tid == 0) atomicAdd(&of_pivot, keys_of);
          const bool mixed = __syncthreads_or(others != 0);
          unsigned* counters = all_counters + seg.chunk * kPartsOfChunk;
          if (!mixed) {
            if (tid == 0) atomicAdd(counters + part_of(seg, pivot, shift), keys_of);
            return;
          }
          for (int d = tid; d < kSegSlots; d += kSegThreads) {
            const unsigned c = count[d];
            if (c) atomicAdd(counters + d, c);
          }
          if (tid == 0) {
            segments[numbers[slot]].mixed = 1u;
            st->mixed[level] = 1;
          }
        });
    if (!go || __ldcg(&st->mixed[level]) == 0) return;

    // Where the parts begin.  Parts of up to half a bucket that begin between the same multiples of half a bucket form one together.
    go = run_phase(st, 4 * level + 1, n_segments, [&](unsigned i) {
      constexpr unsigned kHalf = kCap / 2;
      if (warp == 0) fetch(i, 0);
      __syncthreads();
      const Segment seg = fetched[0];
      if (!seg.mixed) return;
      const int shift = shift_of(seg), parts = parts_of(seg, shift), of_pivot = (int)part_of(seg, seg.pivot, shift);
      unsigned* counters = all_counters + seg.chunk * kPartsOfChunk;
      unsigned c[kSegPer], sum = 0, last = 0;            // last: keys of the last part that has any (the pivot's: more than any)
#pragma unroll
      for (int q = 0; q < kSegPer; ++q) {
        const int d = tid * kSegPer + q;
        c[q] = d < parts ? __ldcg(counters + d) : 0u;
        sum += c[q];
        if (c[q]) last = d == of_pivot ? 0xffffffffu : c[q];
      }
      const unsigned at = block_exclusive<kSegThreads / 32>(sum, part);
      unsigned p = at;
#pragma unroll
      for (int q = 0; q < kSegPer; ++q) {
        const int d = tid * kSegPer + q;
        if (d < parts) __stcg(counters + d, seg.from + p);
        if (d == of_pivot) {
          __stcg(&segments[i].equal, seg.from + p);
          __stcg(&segments[i].equal_to, seg.from + p + c[q]);
        }
        p += c[q];
      }
      if (shift == 0) return;
      unsigned before = last;                   // the same of the threads before
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
      unsigned starts = 0;
      p = at;
#pragma unroll
      for (int q = 0; q < kSegPer; ++q)
        if (c[q]) {
          const bool is_pivot = tid * kSegPer + q == of_pivot;
          if (before == 0 || before > kHalf || c[q] > kHalf || is_pivot || (p - before) / kHalf != p / kHalf) starts |= 1u << q;
          before = is_pivot ? 0xffffffffu : c[q];
          p += c[q];
        }
      unsigned to = block_exclusive<kSegThreads / 32>((unsigned)__popc(starts), part);
      const unsigned total = part[kSegThreads / 32];
      p = at;
#pragma unroll
      for (int q = 0; q < kSegPer; ++q) {
        if ((starts >> q) & 1u) {
          count[to] = p;
          delta[to++] = (unsigned)(tid * kSegPer + q);
        }
        p += c[q];
      }
      if (tid == 0) count[total] = seg.keys;
      __syncthreads();
      for (unsigned b = tid; b < total; b += kSegThreads) {
        const unsigned from = seg.from + count[b], of = count[b + 1] - count[b];
        const int d = (int)delta[b];
        if (d == of_pivot) continue;
        if (of > (unsigned)kCap) {              // (never at the last level, whose parts are of one value)
          unsigned lo = seg.lo + ((unsigned)(d < of_pivot ? d : d - 2) << shift), hi = lo + min((1u << shift) - 1u, seg.hi - lo);
          if (d == of_pivot - 1) hi = seg.pivot - 1u;
          if (d == of_pivot + 1) lo = seg.pivot + 1u;
          add_segment(st, all_segments + (level + 1) * per_level, level + 1, from, of, lo, hi);
        } else {
          extra[atomicAdd(&st->n_extra, 1)] = make_uint2(from, of);
        }
      }
    });
    if (!go) return;

    go = run_phase(st, 4 * level + 2, n_chunks, find, [&](unsigned chunk, int slot, auto look_ahead) {
      const Segment seg = fetched[slot];
      look_ahead();
      if (!seg.mixed) return;
      unsigned begin, end;
      places(seg, chunk, begin, end);
      const int shift = shift_of(seg), parts = parts_of(seg, shift);
      const unsigned pivot = seg.pivot;
      unsigned* counters = all_counters + seg.chunk * kPartsOfChunk;
      if (shift == 0) {                         // written from the parts' beginnings
        const int of_pivot = (int)part_of(seg, pivot, 0);
        for (int d = tid; d < parts; d += kSegThreads) count[d] = __ldcg(counters + d);
        __syncthreads();
#pragma unroll 4
        for (unsigned i = begin + tid; i < end; i += kSegThreads) {
          int d = 0;
#pragma unroll
          for (int s = 1 << kSegPartsLog; s > 0; s /= 2)
            if (d + s < parts && count[d + s] <= i) d += s;
          __stcg(x + i, raw_of(d == of_pivot ? pivot : seg.lo + (unsigned)(d < of_pivot ? d : d - 2)));
        }
        // zeros have become positive: if there are others, all are written again at the end
        if (tid == 0 && seg.lo <= 0x80000000u && seg.hi >= 0x80000000u && (__ldcg(&st->zeros) & 2)) atomicOr(&st->zeros, 3);
        return;
      }
      for (; begin < end; begin += kSegTile) {
        const int left = (int)min((unsigned)kSegTile, end - begin);
        unsigned v[kSegItems], rank[kSegItems / 2];          // ranks of 16 bits
#pragma unroll
        for (int j = 0; j < kSegItems; ++j)
          v[j] = j * kSegThreads + tid < left ? key_at(x + begin + j * kSegThreads + tid) : pivot;
        for (int d = tid; d < kSegSlots; d += kSegThreads) count[d] = 0u;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSegItems; ++j) {
          const unsigned r = v[j] != pivot ? atomicAdd(&count[part_of(seg, v[j], shift)], 1u) : 0u;
          rank[j / 2] = (j & 1) ? rank[j / 2] | r << 16 : r;
        }
        __syncthreads();
        unsigned c[kSegPer], g[kSegPer], sum = 0;
#pragma unroll
        for (int q = 0; q < kSegPer; ++q) {
          c[q] = count[tid * kSegPer + q];
          g[q] = c[q] ? atomicAdd(counters + tid * kSegPer + q, c[q]) : 0u;
          sum += c[q];
        }
        unsigned e = block_exclusive<kSegThreads / 32>(sum, part);
        const int others = (int)part[kSegThreads / 32];
#pragma unroll
        for (int q = 0; q < kSegPer; ++q) {
          count[tid * kSegPer + q] = e;
          delta[tid * kSegPer + q] = g[q] - e;
          e += c[q];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSegItems; ++j)
          if (v[j] != pivot) keys[count[part_of(seg, v[j], shift)] + ((rank[j / 2] >> ((j & 1) * 16)) & 0xffffu)] = v[j];
        __syncthreads();
#pragma unroll 4
        for (int i = tid; i < others; i += kSegThreads) {
          const unsigned k = keys[i];
          __stcg(tmp + (delta[part_of(seg, k, shift)] + (unsigned)i), raw_of(k));
        }
      }
      if (tid == 0 && seg.lo <= 0x80000000u && seg.hi >= 0x80000000u && (__ldcg(&st->zeros) & 2)) atomicOr(&st->zeros, 3);
    });
    if (!go) return;

    // back into the array, and the next level's counters cleared
    const unsigned next_chunks = level + 1 < kLevels ? (unsigned)__ldcg(&st->segments[level + 1]) : 0u;
    go = run_phase(st, 4 * level + 3, n_chunks, find, [&](unsigned chunk, int slot, auto look_ahead) {
      const Segment seg = fetched[slot];
      look_ahead();
      for (unsigned c = chunk; c < next_chunks; c += n_chunks)
        if (tid < kPartsOfChunk) __stcg(all_counters + c * kPartsOfChunk + tid, 0u);
      if (!seg.mixed || shift_of(seg) == 0) return;
      unsigned begin, end;
      places(seg, chunk, begin, end);
      const unsigned pivot = raw_of(seg.pivot);
#pragma unroll 16
      for (unsigned i = begin + tid; i < end; i += kSegThreads) __stcg(x + i, i >= seg.equal && i < seg.equal_to ? pivot : __ldcg(tmp + i));
    });
    if (!go) return;
  }
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }
// Segments of a level: more than kCap keys each.  Their chunks: at most two for every kCap keys.  Buckets made from a segment: a part of
// more than half a bucket, or what begins between two multiples of half a bucket; twice where the pivot lies between.
int64_t most_segments(int64_t n) { return n / kCap + 1; }
int64_t most_extra(int64_t n) { return kLevels * 7 * (n / kCap + 1); }
struct Layout {
  size_t state, samples, table, fine, begins, first, cursor, uneven, segments, counters, extra, tmp, total;
};
Layout layout(int64_t n) {
  Layout l;
  size_t off = 0;
  l.state = off; off += kStateBytes;
  l.samples = off; off += up256(kSamples * 4);
  l.table = off; off += up256(kBins * 4);
  l.fine = off; off += up256(kFineMax * 4);
  l.begins = off; off += up256(kFineMax / 4);
  l.first = off; off += up256((kMaxBuckets + 1) * 4);
  l.cursor = off; off += up256(kMaxBuckets * 4);
  l.uneven = off; off += up256((kMaxBuckets + most_extra(n)) * sizeof(uint2));
  l.segments = off; off += up256(kLevels * most_segments(n) * sizeof(Segment));
  l.counters = off; off += up256(2 * most_segments(n) * kPartsOfChunk * 4);
  l.extra = off; off += up256(most_extra(n) * sizeof(uint2));
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
  Segment* segments = reinterpret_cast<Segment*>(base + l.segments);
  unsigned* counters = reinterpret_cast<unsigned*>(base + l.counters);
  uint2* extra = reinterpret_cast<uint2*>(base + l.extra);
  unsigned* tmp = reinterpret_cast<unsigned*>(base + l.tmp);
  const unsigned* in = reinterpret_cast<const unsigned*>(weights);
  unsigned* x = reinterpret_cast<unsigned*>(sorted);
  static PerDeviceFlag f_count, f_part_l, f_part_s, f_sort, f_single, f_segments, f_finish;
  const int sms = current_sm_count();
  cudaError_t e;
  if (n <= kCap) {
    if ((e = opt_in(sort_buckets_kernel<true>, kSortSmem, f_single)) != cudaSuccess) return e;
    e = launch_after(sort_buckets_kernel<true>, 1, kSortThreads, kSortSmem, s, in, (long long)n, st, (const unsigned*)first, (const uint2*)extra, x, uneven);
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
    e = launch_after(sort_map_kernel, 1, kMapThreads, 0, s, (long long)n, target, st, (const unsigned*)fine, (const unsigned*)table, begins, first, cursor, segments);
    if (e != cudaSuccess) return e;
    const bool large = n >= (int64_t)kPartThreads * L * sms;
    const int64_t tile = kPartThreads * (large ? L : S), tiles = (n + tile - 1) / tile;
    const unsigned grid = (unsigned)(tiles < sms ? tiles : sms);
    e = launch_after(large ? sort_partition_kernel<L> : sort_partition_kernel<S>, grid, kPartThreads, large ? partition_smem<L>() : partition_smem<S>(), s,
                     in, (long long)n, (const SortState*)st, (const unsigned*)table, (const unsigned*)begins, cursor, x, counters);
    if (e != cudaSuccess) return e;
    if ((e = opt_in(sort_segments_kernel, kSegSmem, f_segments)) != cudaSuccess) return e;
    const int64_t chunks = 2 * most_segments(n);
    e = launch_after(sort_segments_kernel, (unsigned)(chunks < 2 * sms ? chunks : 2 * sms), kSegThreads, kSegSmem, s, st, segments, (int)most_segments(n), counters,
                     extra, x, tmp);
    if (e != cudaSuccess) return e;
    const int64_t most = 2 * (n / target) + 2;
    e = launch_after(sort_buckets_kernel<false>, (unsigned)(most < 2 * sms ? most : 2 * sms), kSortThreads, kSortSmem, s, in, (long long)n, st, (const unsigned*)first, (const uint2*)extra, x, uneven);
  }
  if (e != cudaSuccess) return e;
  if ((e = opt_in(sort_finish_kernel, kFinishSmem, f_finish)) != cudaSuccess) return e;
  const int64_t pieces = n / 256 + 1;                    // buckets of an array of that size, and more
  return launch_after(sort_finish_kernel, (unsigned)(n <= kCap ? 1 : pieces < sms ? pieces : sms), kSortThreads, kFinishSmem, s, in, (long long)n, st,
                      (const uint2*)uneven, counters, tmp, x);
}

}  // namespace lcd
