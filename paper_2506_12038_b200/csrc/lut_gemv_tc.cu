// Lookup and accumulation on the tcgen05 tensor cores (LCD_ALGO_TC_LUT, and LCD_ALGO_DENSE_TC up to a few hundred tokens).
//
// Section 4.2 of the LCD paper with per-row tables: a row's codebook is two byte tables in registers (16-bit fixed
// point: signed high byte, unsigned low byte), one PRMT looks four weights up, and the looked-up bytes go straight
// from registers into tensor memory (tcgen05.st) as the A operand of tcgen05.mma kind::i8; the tokens' levels are the
// B operand in shared memory.  Exact int32 sums, y = s_q * 2^e_n * (256 * sumH + sumL).
//
// What bounds it.  Per unit of 128 rows x 256 columns an SM has to read 4 KB x bits of indices (8 KB at 2 bit: 350
// clocks at its share of the memory bandwidth) and to look 32768 weights up: 10 (2 bit), 11 (3 bit) or 28 (4 bit)
// half-rate integer instructions per 16 weights = 320, 350 or 900 clocks.  Measured on B200: storing the 64 KB of
// looked-up bytes takes 128 clocks in the form used here, the 16 MMAs of a unit 170 / 270 / 520 / 1040 clocks at
// 16 / 32 / 64 / 128 tokens when they are issued under elect.sync (10.4 clocks each at 16 tokens; the same instruction
// issued under `lane == 0` takes 46, because its operands then pass through per-thread registers).  With A in shared
// memory an MMA takes 40 clocks at any width up to 32 tokens and competes with the decoders' stores for its bandwidth:
// that is why the lookups are written to tensor memory.
//
// Work.  A tile is 128 rows x NT tokens; the column units of all tiles of all problems of a launch form one sequence
// (problem, row tile, token tile, column unit), cut evenly over the CTAs, at most one per SM.  A CTA walks its piece from
// the end to the beginning.  A tile that is cut between CTAs is finished by the CTA with the tile's last columns, which
// reaches it last, with all its decoder warps; the others reach their part first and leave it in their slot of the
// scratch (one int32 per output where rows and pieces are short enough for the sum of both planes, see tc_plan_width).  A CTA
// therefore only ever waits for CTAs of smaller number, which were launched before it, and normally finds their part there.
//
// Where there are few tiles and many tokens, that one CTA reads megabits while the others have nothing to do: then the CTAs
// of a tile are a cluster (resident together, so they may wait for one another), every one stores its part of the tokens
// that are not its own and, after the cluster's barrier, finishes its own from the other CTAs' parts (4096 x 11008, 2 bit,
// 48 tokens, transformation to y: 16.9 us with one finisher, 15.1 so, parts of one number both; 512 x 14336 at 16 tokens
// 13.2 and 11.0; 2048 x 11008 at 32 tokens 16.7 and 13.6).  With few tokens the one finisher is as fast; the launcher's
// estimate decides (tc_plan_width).
//
// Layout.  An item of the index area (16 rows x 256 columns, lane 4g + t of a tile holds row g, column quarter t) is
// loaded as it lies; the 16x128b form of tcgen05.st wants exactly that distribution: lane 4g + t writes word t of
// every 4-word block of rows g and g + 8 (measured with 16 warps storing: 64 clocks per 2 KB, 16x256b takes 127,
// 32x32b, which wants a row per lane, 36).  Blocks 2j, 2j + 1 of a 128-column k-block are the K = 32 step j of the MMA:
// byte 16e + 4t + b of it holds column 32t + 8j + 4e + b (3 and 4 bit) or 32t + 16(j >> 1) + 8e + 2b + (j & 1) (2 bit:
// the order in which the selectors list the fields of a word), and the levels are placed alike.
//
// Warps: 0-15 decoders (tensor-memory quadrant = warp & 3, 16-row half (warp >> 2) & 1, even / odd units warp >> 3),
// 16-19 epilogue, 20-23 token levels (kActReady: epilogue as well), 24 index copies, 25 MMA issue, 26 copies of ready
// levels.  Every wait is bounded; on expiry the status word is set, all roles run out, drain what they issued and
// release tensor memory.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>

#include "common.h"
#include "device_util.h"
#include "selectors.cuh"

namespace lcd {

namespace {

constexpr int kTcRows = 128;                  // MMA M: weight rows per tile
constexpr uint32_t kTcACols = 128;            // tensor-memory columns of a unit's A operand: 64 words high plane + 64 low plane
constexpr int kTcDecoders = 16, kTcFirstEpi = 16, kTcFirstToken = 20, kTcTokenWarps = 4;
constexpr int kTcCopyWarp = 24, kTcMmaWarp = 25, kTcLevelWarp = 26;
constexpr int kTcThreads = 32 * 27;
constexpr int kTcWordUnits = 32;              // column units whose sum of both planes fits one int32: 32752 * 8 * 8192 < 2^31
constexpr int kTcExactUnits = 32;             // column units up to which either plane's sums of 4-bit levels fit 24 bits: 255 * 8 * 8192 < 2^24
constexpr int kTcMaxParts = 17;               // CTAs that share a tile, its finisher not counted (see tc_plan_width)
constexpr unsigned long long kTcWaitNs = 2000000000ull;

// Stored 4-bit levels and stored 8-bit levels (natural order, placed by the token warps), or signed bytes already in the
// operand order (written so by the kernel before; tensor copies bring them)
constexpr int kActPacked4 = 0, kActBytes = 1, kActReady = 2;

// Units in flight: A in tensor memory, B in shared memory.  Accumulators take the rest of the 512 columns: two buffers of
// (high, low) x NT columns up to 32 tokens, one above.
__host__ __device__ constexpr int tc_slots(int nt) { return nt == 128 ? 2 : 3; }
__host__ __device__ constexpr int tc_acc_bufs(int nt) { return nt <= 32 ? 2 : 1; }
// Ring slots of one unit each (even: a slot then always belongs to the same decoder group, whose parity waits rely on
// that).  About 64 KB in flight per SM, what a share of the memory bandwidth times a microsecond of latency needs.
__host__ __device__ constexpr int tc_ring(int bits) { return bits == 2 ? 8 : bits == 3 ? 6 : 4; }
// Token warps that share a unit's levels (its tokens)
__host__ __device__ constexpr int tc_token_share(int nt, int act) { return act != kActReady && nt * (act == kActBytes ? 2 : 1) > 32 ? 2 : 1; }

struct TcProblem {
  const uint16_t* codebook;
  const uint8_t* act;        // packed 4-bit levels [M][K_pad/2] or signed bytes [M][K_pad]
  const float* act_scale;    // [M]
  float* y;
  long long ldy;
  int N, M, n_rp, n_kt, n_mt, n_tiles;
  unsigned unit0;            // number of units of the problems before this one
};
struct TcBatch {
  int count;
  unsigned per, extra;       // units of the launch: grid * per + extra
  float ctas_per_unit;       // about grid / units
  int share;                 // SHARE: CTAs per tile
  int words;                 // 1: parts are sums of both planes, 2: the planes apart
  int clean;                 // leave the scratch zero-filled
  unsigned long long nonce;  // marks a part as left by this launch; the reader puts zero back
  int* parts;                // scratch [grid][words][NT][128 rows] int32
  unsigned long long* flags; // scratch [grid]
  TcProblem p[LCD_MAX_BATCH];
};
// Index areas as tensors [16-row group][column unit][item]: one copy brings the eight items of a unit.  Levels (kActReady)
// as [token][column].
struct alignas(64) TcMaps {
  CUtensorMap items[LCD_MAX_BATCH];
  CUtensorMap levels[LCD_MAX_BATCH];
};

__device__ __forceinline__ uint32_t tc_prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
__device__ __forceinline__ unsigned long long tc_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool tc_elect() {
  uint32_t p;
  asm volatile("{\n.reg .pred P;\nelect.sync _|P, 0xffffffff;\nselp.u32 %0, 1, 0, P;\n}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ bool tc_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait.  On expiry the abort flag is raised and every wait of the CTA from then on gives up at its first check:
// the roles run to their end on whatever data is there (the output is invalid, the caller learns it from the status
// word), so that they need not test the outcome of a wait.  The copying roles do test it: a second expect_tx on a
// barrier whose first copies have not landed is not allowed.
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (tc_try(bar, parity)) return true;
  const unsigned long long t0 = tc_timer();
#pragma unroll 1
  for (uint32_t it = 1; !tc_try(bar, parity); ++it) {
    if ((it & 63u) == 0) {
      if (*abort_flag) return false;
      if (tc_timer() - t0 > kTcWaitNs) { *abort_flag = 1; return false; }
    }
  }
  return true;
}
__device__ __forceinline__ void tc_drain(uint32_t bar, uint32_t parity) {
  const unsigned long long t0 = tc_timer();
  for (uint32_t it = 1; !tc_try(bar, parity); ++it)
    if ((it & 63u) == 0 && tc_timer() - t0 > kTcWaitNs) return;
}
__device__ __forceinline__ void tc_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tc_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
// kind::i8, A from tensor memory, B from shared memory (K-major, 128-byte swizzle)
__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// 16 rows x 32 words (eight 4-word blocks): lane 4g + t supplies word t of rows g (v[2n]) and g + 8 (v[2n + 1]) of block n
__device__ __forceinline__ void tc_st_16x128_x8(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tc_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_ld4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr) : "memory");
}
// The loaded registers are operands: nothing that reads them can be scheduled before the wait.
__device__ __forceinline__ void tc_wait_ld8(uint32_t (&a)[8], uint32_t (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
               :: "memory");
}
__device__ __forceinline__ void tc_wait_ld4(uint32_t (&a)[4], uint32_t (&b)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]) :: "memory");
}
// kind::i8 instruction descriptor: int32 accumulate, B signed, A signed (high plane) or unsigned (low plane)
__host__ __device__ constexpr uint32_t tc_idesc(int nt, bool a_signed) {
  return (2u << 4) | ((a_signed ? 1u : 0u) << 7) | (1u << 10) | ((uint32_t)(nt >> 3) << 17) |
         ((uint32_t)(kTcRows >> 4) << 24);
}
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t addr) {
  uint64_t d = (uint64_t)((addr & 0x3ffffu) >> 4);
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// CTA c of G owns the units [floor(c T / G), floor((c + 1) T / G)) = c * per + c * extra / G with T = G * per + extra; the
// CTA that owns unit u (an estimate, put right by a step or two).
__device__ __forceinline__ uint32_t unit_begin(uint32_t c, const TcBatch& B) { return c * B.per + c * B.extra / gridDim.x; }
__device__ __forceinline__ uint32_t unit_owner(uint32_t u, const TcBatch& B) {
  uint32_t c = min((uint32_t)((float)u * B.ctas_per_unit), gridDim.x - 1);
  while (c + 1 < gridDim.x && unit_begin(c + 1, B) <= u) ++c;
  while (c > 0 && unit_begin(c, B) > u) --c;
  return c;
}

// A CTA's segments: the parts of tiles in its piece of the sequence, from the last to the first.  A segment is the column
// units kb, kb - 1, .., ka of one tile.
struct Segments {
  int p, tile, kb, ka;
  uint32_t left;      // units not yet in a segment handed out
  __device__ __forceinline__ void take() {
    const uint32_t len = left < (uint32_t)kb + 1u ? left : (uint32_t)kb + 1u;
    ka = kb + 1 - (int)len;
    left -= len;
  }
  // [u0, u1), not empty
  __device__ __forceinline__ void first(uint32_t u0, uint32_t u1, const TcBatch& B) {
    p = 0;
    for (int i = 1; i < B.count; ++i)
      if (u1 - 1 >= B.p[i].unit0) p = i;
    const uint32_t n_kt = (uint32_t)B.p[p].n_kt, local = u1 - 1 - B.p[p].unit0;
    tile = (int)(local / n_kt);
    kb = (int)(local - (uint32_t)tile * n_kt);
    left = u1 - u0;
    take();
  }
  __device__ __forceinline__ bool next(const TcBatch& B) {
    if (left == 0) return false;
    if (--tile < 0) {
      --p;
      tile = B.p[p].n_tiles - 1;
    }
    kb = B.p[p].n_kt - 1;
    take();
    return true;
  }
  __device__ __forceinline__ int row_tile(const TcProblem& P) const { return P.n_mt == 1 ? tile : tile / P.n_mt; }
};

// Tokens of a tile that each of its `share` CTAs finishes (a multiple of eight, what the epilogue stores at a time).
__device__ __forceinline__ int share_tokens(int n_tok, int share) { return ((n_tok + 7) / 8 + share - 1) / share * 8; }

// Byte tables of one row: entry i is byte i & 3 of word i >> 2.  2 bit: one word (used twice by the lookup).
template <int BITS>
struct RowTables {
  static constexpr int W = BITS == 4 ? 4 : BITS == 3 ? 2 : 1;
  uint32_t hi[W], lo[W];
  // cb: the row's 2^BITS fp16 centroids in shared memory
  __device__ __forceinline__ void load(uint32_t cb) {
    uint32_t c[1 << (BITS - 1)];
    if constexpr (BITS == 2) {
      asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(c[0]), "=r"(c[1]) : "r"(cb));
    } else {
#pragma unroll
      for (int i = 0; i < (1 << (BITS - 3)); ++i)
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(c[4 * i]), "=r"(c[4 * i + 1]), "=r"(c[4 * i + 2]), "=r"(c[4 * i + 3]) : "r"(cb + 16u * i));
    }
    float mx = 0.0f;
#pragma unroll
    for (int i = 0; i < (1 << (BITS - 1)); ++i) {
      mx = fmaxf(mx, fabsf(__half2float(__ushort_as_half((unsigned short)(c[i] & 0xffffu)))));
      mx = fmaxf(mx, fabsf(__half2float(__ushort_as_half((unsigned short)(c[i] >> 16)))));
    }
    int ex = (int)((__float_as_uint(mx) >> 23) & 0xffu) - 126;
    ex = ex < -30 ? -30 : ex;
    const float up = __uint_as_float((uint32_t)(15 - ex + 127) << 23);
#pragma unroll
    for (int i = 0; i < W; ++i) hi[i] = lo[i] = 0u;
#pragma unroll
    for (int i = 0; i < (1 << BITS); ++i) {
      const int f = __float2int_rn(__half2float(__ushort_as_half((unsigned short)(c[i >> 1] >> (16 * (i & 1))))) * up);
      hi[i >> 2] |= ((uint32_t)(f >> 8) & 0xffu) << (8 * (i & 3));
      lo[i >> 2] |= ((uint32_t)f & 0xffu) << (8 * (i & 3));
    }
  }
};
// Four weights' bytes: selector nibbles sel (entry number, low three bits), pick (4 bit: byte choice by bit three).
template <int BITS>
__device__ __forceinline__ uint32_t tc_look(const uint32_t (&t)[RowTables<BITS>::W], uint32_t sel, uint32_t pick) {
  if constexpr (BITS == 2) return tc_prmt(t[0], t[0], sel);
  else if constexpr (BITS == 3) return tc_prmt(t[0], t[1], sel);
  else return tc_prmt(tc_prmt(t[0], t[1], sel), tc_prmt(t[2], t[3], sel), pick);
}
// 2^(e-15) of a row (see RowTables)
template <int BITS>
__device__ __forceinline__ float tc_row_scale(const uint16_t* cb) {
  float mx = 0.0f;
#pragma unroll
  for (int i = 0; i < (1 << BITS); ++i) mx = fmaxf(mx, fabsf(__half2float(__ushort_as_half(__ldg(cb + i)))));
  int ex = (int)((__float_as_uint(mx) >> 23) & 0xffu) - 126;
  ex = ex < -30 ? -30 : ex;
  return __uint_as_float((uint32_t)(ex - 15 + 127) << 23);
}

// Offsets in shared memory: 0 rings, 1 bytes of a ring slot, 2 barriers, 3 end
template <int BITS, int NT>
__host__ __device__ constexpr int tc_smem_layout(int what) {
  constexpr int kB = tc_slots(NT) * NT * 256, kRingSlot = 8 * 512 * BITS + (256 << BITS), kRing = tc_ring(BITS) * kRingSlot;
  constexpr int kBars = 3 * tc_slots(NT) + 2 * tc_ring(BITS) + 4 + 2;
  return what == 0 ? kB : what == 1 ? kRingSlot : what == 2 ? kB + kRing : kB + kRing + 8 * kBars + 16;
}

// SHARE: the CTAs of a tile are a cluster and finish it together (its own instances: 0.2 us of a launch otherwise).
template <int BITS, int NT, int ACT, bool SHARE>
__global__ void __launch_bounds__(kTcThreads, 1)
lut_gemv_tc_kernel(const __grid_constant__ TcMaps maps, const __grid_constant__ TcBatch B, int* status) {
  extern __shared__ uint8_t tc_smem_raw[];
  constexpr int ITEM = 512 * BITS, HALF = 256 * BITS, R = tc_ring(BITS), S = tc_slots(NT), NBUF = tc_acc_bufs(NT);
  constexpr int kBSlot = NT * 256, kRingSlot = tc_smem_layout<BITS, NT>(1), kCbRow = 2 << BITS;
  constexpr uint32_t kAccCol0 = S * kTcACols;
  constexpr int kEpiHalves = ACT == kActReady ? 2 : 1;          // epilogue warps per tensor-memory quadrant
  static_assert(kAccCol0 + NBUF * 2 * NT <= 512, "tensor memory");
  static_assert(kTcMaxParts <= 32 && kTcMaxParts * 2 * 4 * kTcRows * 4 <= tc_smem_layout<BITS, NT>(2), "room for four tokens of all parts");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const uint32_t raw_addr = (uint32_t)__cvta_generic_to_shared(tc_smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  uint8_t* gen_base = tc_smem_raw + (base - raw_addr);
  const uint32_t ring_base = base + tc_smem_layout<BITS, NT>(0);
  const uint32_t bar_base = base + tc_smem_layout<BITS, NT>(2);
  auto full = [&](uint32_t s) { return bar_base + 8u * s; };                       // a unit's A and B operands are in place
  // A unit's MMAs have finished: barrier (unit mod 2 S), phase unit / 2 S.  Unit i may be filled when unit i - S is done.
  // The roles that fill take turns at the units (decoders two, token warps up to four), so that a waiter knows only of
  // earlier units; with one barrier per slot its parity wait for unit i - S would pass while unit i - 2 S still held it.
  auto done = [&](uint32_t e) { return bar_base + 8u * (S + e); };
  auto ring_full = [&](uint32_t s) { return bar_base + 8u * (3 * S + s); };
  auto ring_empty = [&](uint32_t s) { return bar_base + 8u * (3 * S + R + s); };
  auto acc_full = [&](uint32_t b) { return bar_base + 8u * (3 * S + 2 * R + b); };
  auto acc_empty = [&](uint32_t b) { return bar_base + 8u * (3 * S + 2 * R + 2 + b); };
  const uint32_t drain_bar = bar_base + 8u * (3 * S + 2 * R + 4), part_bar = drain_bar + 8u;
  uint8_t* gen_misc = gen_base + tc_smem_layout<BITS, NT>(2) + 8 * (3 * S + 2 * R + 6);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(gen_misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gen_misc + 4);
  int* parts_stored = reinterpret_cast<int*>(gen_misc + 8);        // epilogue warps that have stored the CTA's part

  if (threadIdx.x == 0) {
    auto init = [](uint32_t bar, uint32_t count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
    };
    for (int s = 0; s < S; ++s) {
      init(full(s), kTcDecoders / 2 + tc_token_share(NT, ACT));
      init(done(s), 1);
      init(done(S + s), 1);
    }
    for (int s = 0; s < R; ++s) {
      init(ring_full(s), 1);
      init(ring_empty(s), kTcDecoders / 2);
    }
    for (int b = 0; b < 2; ++b) {
      init(acc_full(b), 1);
      init(acc_empty(b), 4 * kEpiHalves);
    }
    init(drain_bar, 1);
    init(part_bar, 1);
    *abort_flag = 0;
    *parts_stored = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kTcMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(tmem_holder)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  const uint32_t u0 = unit_begin(blockIdx.x, B), u1 = unit_begin(blockIdx.x + 1, B);      // not empty
  Segments sg;
  sg.first(u0, u1, B);

  // The piece's first tile, reached last, has columns in other CTAs: the decoder warps finish it.  The other parts come by bulk
  // copies into the shared memory that rings and levels have left (with plain loads, 32 KB in flight per SM, this took
  // 12 us for 100 tokens and three parts), tokens in rounds of as many as fit.
  auto finish = [&](uint32_t acc) {
    const TcProblem& P = B.p[sg.p];
    {
      const uint32_t last = u1 - u0 - 1, tile0 = P.unit0 + (uint32_t)sg.tile * (uint32_t)P.n_kt, quad = warp & 3;
      const int share = SHARE ? B.share : 0, rank = SHARE ? (int)(blockIdx.x % (uint32_t)share) : 0;
      const int parts = SHARE ? share - 1 : (int)(blockIdx.x - unit_owner(tile0, B));      // at most kTcMaxParts (the launcher's grid)
      auto part_block = [&](int i) { return SHARE ? blockIdx.x - rank + (i < rank ? i : i + 1) : blockIdx.x - 1 - i; };
      const int rt = sg.row_tile(P), m0 = (sg.tile - rt * P.n_mt) * NT, all_tok = min(NT, P.M - m0);
      // this CTA's tokens
      const int own = SHARE ? share_tokens(all_tok, share) : NT, first_tok = rank * own, n_tok = min(all_tok, first_tok + own);
      const int row = 32 * (int)quad + lane, out = rt * kTcRows + row, words = B.words;
      const float row_scale = tc_row_scale<BITS>(P.codebook + (size_t)min(out, P.n_rp * 16 - 1) * (1 << BITS));
      const int fit = (tc_smem_layout<BITS, NT>(2) / (parts * words * kTcRows * 4)) & ~3, step = fit < NT ? fit : NT;
      const size_t part_ints = (size_t)words * NT * kTcRows;
      asm volatile("griddepcontrol.wait;" ::: "memory");     // scales, scratch and y belong to earlier kernels until here
      tc_wait(done(last % (2 * S)), (last / (2 * S)) & 1u, abort_flag);
      __syncwarp();
      tc_fence_after();
      const uint32_t t_hi = tmem_base + ((32 * quad) << 16) + kAccCol0 + acc * (2 * NT);
      uint32_t round = 0;
#pragma unroll 1
      for (int c0 = first_tok; c0 < n_tok; c0 += step, ++round) {
        const int n_now = min(step, n_tok - c0);
        if (warp == 0) {
          if (lane == 0) tc_expect(part_bar, (uint32_t)(parts * words * n_now * kTcRows * 4));
          __syncwarp();
          if (lane < parts) {          // a lane per part: its copy starts as soon as it is there
            const int* src = B.parts + (size_t)part_block(lane) * part_ints + c0 * kTcRows;
            if (!SHARE && round == 0) {
              unsigned long long* flag = B.flags + (blockIdx.x - 1 - lane);
              const unsigned long long t0 = tc_timer();
              unsigned long long seen = 0;
#pragma unroll 1
              for (uint32_t it = 1;; ++it) {
                asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(seen) : "l"(flag) : "memory");
                if (seen == B.nonce) break;
                if ((it & 63u) == 0 && (*abort_flag || tc_timer() - t0 > kTcWaitNs)) { *abort_flag = 1; break; }
              }
              *flag = 0ull;
            }
            asm volatile("fence.proxy.async;" ::: "memory");       // written by ordinary stores, read by copies
            for (int w = 0; w < words; ++w)
              tc_bulk(base + (uint32_t)((lane * words + w) * step * kTcRows * 4), src + w * NT * kTcRows,
                      (uint32_t)(n_now * kTcRows * 4), part_bar);
          }
          __syncwarp();
        }
        const int* buf = reinterpret_cast<const int*>(gen_base) + row;
        bool landed = false;
#pragma unroll 1
        for (int c = 4 * (warp >> 2); c < n_now; c += 16) {
          uint32_t hi[4], lo[4];
          tc_ld4(t_hi + c0 + c, hi);
          tc_ld4(t_hi + NT + c0 + c, lo);
          const int m = m0 + c0 + c;
          const float sc = m + (lane & 3) < P.M ? ld_global(P.act_scale + m + (lane & 3)) : 0.0f;
          if (!landed) tc_wait(part_bar, round & 1u, abort_flag);
          landed = true;
          __syncwarp();
          tc_wait_ld4(hi, lo);
          if (words == 1) {
            long long sum[4];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              sum[j] = ACT == kActPacked4 ? (long long)((int)hi[j] >> 4) * 256 + ((int)lo[j] >> 4) : (long long)(int)hi[j] * 256 + (int)lo[j];
            for (int p = 0; p < parts; ++p)
#pragma unroll
              for (int j = 0; j < 4; ++j) sum[j] += buf[(p * step + c + j) * kTcRows];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float s = __shfl_sync(0xffffffffu, sc, j) * row_scale;
              if (c + j < n_now && out < P.N) P.y[(size_t)(m + j) * P.ldy + out] = __ll2float_rn(sum[j]) * s;
            }
          } else {
            for (int p = 0; p < parts; ++p)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                hi[j] += (uint32_t)buf[(2 * p * step + c + j) * kTcRows];
                lo[j] += (uint32_t)buf[((2 * p + 1) * step + c + j) * kTcRows];
              }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float s = __shfl_sync(0xffffffffu, sc, j) * (ACT == kActPacked4 ? row_scale * 0.0625f : row_scale);
              if (c + j < n_now && out < P.N) P.y[(size_t)(m + j) * P.ldy + out] = ((float)(int)hi[j] * 256.0f + (float)(int)lo[j]) * s;
            }
          }
          if (B.clean)
            for (int p = 0; p < parts; ++p) {
              int* at = B.parts + (size_t)part_block(p) * part_ints + (c0 + c) * kTcRows + row;
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (c + j < n_now) {
                  __stcg(at + j * kTcRows, 0);
                  if (words == 2) __stcg(at + (NT + j) * kTcRows, 0);
                }
            }
        }
        if (!landed) tc_wait(part_bar, round & 1u, abort_flag);      // (the copies land before the CTA may exit)
        asm volatile("bar.sync 2, 512;" ::: "memory");               // the buffer has been read
      }
      if (*abort_flag && round > 0) tc_drain(part_bar, (round - 1) & 1u);
    }
  };

  if (warp == kTcCopyWarp) {
    // ------------------------------------------------------------------ index copies
    // One tensor copy per unit (eight copies of an item each, issued by eight lanes, took 980 clocks per unit and bound
    // the kernel; row groups past the matrix arrive as zeros).  The first two units of a segment, one per decoder group,
    // also bring the tile's codebooks.
    if (tc_elect()) {
      bool ok = true;
      uint32_t rs = 0, parity = 1, n = 0;          // parity of the wait for a slot: the use before, passes at once at first
      do {
        const TcProblem& P = B.p[sg.p];
        const CUtensorMap* map = &maps.items[sg.p];
        const int rp0 = sg.row_tile(P) * (kTcRows / 16);
        const uint32_t cb_bytes = (uint32_t)min(8, P.n_rp - rp0) * 16 * kCbRow;
        const uint16_t* cb = P.codebook + (size_t)rp0 * 16 * (1 << BITS);
        for (int kt = sg.kb; kt >= sg.ka; --kt, ++n) {
          ok = tc_wait(ring_empty(rs), parity, abort_flag);
          if (!ok) break;
          const uint32_t dst = ring_base + rs * kRingSlot;
          const bool with_cb = sg.kb - kt < 2;
          tc_expect(ring_full(rs), 8u * ITEM + (with_cb ? cb_bytes : 0u));
          asm volatile(
              "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
              ::"r"(dst), "l"(map), "r"(0), "r"(kt), "r"(rp0), "r"(ring_full(rs)) : "memory");
          if (with_cb) tc_bulk(dst + 8 * ITEM, cb, cb_bytes, ring_full(rs));
          if (++rs == (uint32_t)R) { rs = 0; parity ^= 1u; }
        }
      } while (ok && sg.next(B));
      // after an expired wait: copies still in flight must land before the CTA's shared memory is released
      if (*abort_flag)
        for (uint32_t k = 1; k <= (uint32_t)R && k <= n; ++k) tc_drain(ring_full((n - k) % R), ((n - k) / R) & 1u);
    }
    __syncwarp();
  } else if (warp == kTcLevelWarp) {
    // ------------------------------------------------------------------ copies of ready levels
    if (ACT == kActReady && tc_elect()) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      bool ok = true;
      uint32_t slot = 0, i = 0;
      do {
        const TcProblem& P = B.p[sg.p];
        const CUtensorMap* map = &maps.levels[sg.p];
        const int m0 = (sg.tile - sg.row_tile(P) * P.n_mt) * NT;
        for (int kt = sg.kb; kt >= sg.ka; --kt, ++i) {
          const uint32_t js = i + S;               // unit i - S is js - 2 S
          ok = tc_wait(done(js % (2 * S)), (js / (2 * S) + 1) & 1u, abort_flag);
          if (!ok) break;
          tc_expect(full(slot), kBSlot);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                ::"r"(base + slot * kBSlot + h * (NT * 128)), "l"(map), "r"(kt * 256 + h * 128), "r"(m0), "r"(full(slot)) : "memory");
          if (++slot == S) slot = 0;
        }
      } while (ok && sg.next(B));
      if (*abort_flag)
        for (uint32_t k = 1; k <= (uint32_t)S && k <= i; ++k) tc_drain(full((i - k) % S), ((i - k) / S) & 1u);
    }
    __syncwarp();
  } else if (warp == kTcMmaWarp) {
    // ------------------------------------------------------------------ MMA issue
    // One wait and one commit per unit: with stages of half a unit and separate commits for the two operands this
    // thread, not the decoders, bound the kernel (a commit takes it about 70 clocks, the eight MMAs of a k-block 90).
    if (tc_elect()) {
      constexpr uint32_t idesc_hi = tc_idesc(NT, true), idesc_lo = tc_idesc(NT, false);
      const uint64_t b_desc0 = tc_smem_desc(base);
      uint32_t n_seg = 0, slot = 0, parity = 0, d = 0;         // d: unit mod 2 S
      do {
        const uint32_t buf = n_seg % NBUF;
        tc_wait(acc_empty(buf), ((n_seg / NBUF) & 1u) ^ 1u, abort_flag);
        tc_fence_after();
        const uint32_t d_hi = tmem_base + kAccCol0 + buf * (2 * NT);
        uint32_t accumulate = 0;
        for (int kt = sg.kb; kt >= sg.ka; --kt) {
          tc_wait(full(slot), parity, abort_flag);
          tc_fence_after();
          const uint32_t a = tmem_base + slot * kTcACols;
          const uint64_t bu = b_desc0 + (uint64_t)(slot * (kBSlot >> 4));
#pragma unroll
          for (int j = 0; j < 8; ++j) {           // k-block j >> 2, 32 columns per step
            const uint64_t b = bu + (uint64_t)((j >> 2) * (NT * 128 >> 4) + 2 * (j & 3));
            tc_mma(d_hi, a + 8 * j, b, idesc_hi, j == 0 ? accumulate : 1u);
            tc_mma(d_hi + NT, a + 64 + 8 * j, b, idesc_lo, j == 0 ? accumulate : 1u);
          }
          accumulate = 1u;
          tc_commit(done(d));
          if (++d == 2 * S) d = 0;
          if (++slot == S) { slot = 0; parity ^= 1u; }
        }
        tc_commit(acc_full(buf));
        ++n_seg;
      } while (sg.next(B));
      tc_commit(drain_bar);
      tc_drain(drain_bar, 0);
    }
    __syncwarp();
  } else if (warp < kTcDecoders) {
    // ------------------------------------------------------------------ decoders
    const uint32_t quad = warp & 3, half = (warp >> 2) & 1, grp = warp >> 3;
    const uint32_t rp_local = 2 * quad + half;
    const uint32_t a_base = tmem_base + ((32 * quad + 16 * half) << 16);
    const uint32_t cb_off = 8 * ITEM + (16 * rp_local + (lane >> 2)) * kCbRow;
    RowTables<BITS> tab[2];          // rows g and g + 8 of the warp's 16
    // own units grp, grp + 2, ..: ring slots and operand slots advance by two; skip: units until the next own one
    uint32_t rs = grp, r_parity = 0, slot = grp, prev = grp + S, p_parity = 1, skip = grp, n_seg = 0;
    while (true) {
      int kt = sg.kb - (int)skip;
      bool fresh = true;
      for (; kt >= sg.ka; kt -= 2) {
        tc_wait(ring_full(rs), r_parity, abort_flag);
        __syncwarp();
        const uint32_t src = ring_base + rs * kRingSlot;
        if (fresh) {
          tab[0].load(src + cb_off);
          tab[1].load(src + cb_off + 8 * kCbRow);
          fresh = false;
        }
        uint32_t raw[2][2][BITS];          // [row][k-block][word]
        const uint32_t it = src + rp_local * ITEM;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t tile = it + u * HALF;
          if constexpr (BITS == 2) {
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(raw[u][0][0]), "=r"(raw[u][0][1]), "=r"(raw[u][1][0]), "=r"(raw[u][1][1]) : "r"(tile + 16 * lane));
          } else if constexpr (BITS == 3) {
#pragma unroll
            for (int b = 0; b < 3; ++b)
              asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];"
                           : "=r"(raw[u][0][b]), "=r"(raw[u][1][b]) : "r"(tile + 256 * b + 8 * lane));
          } else {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(raw[u][h][0]), "=r"(raw[u][h][1]), "=r"(raw[u][h][2]), "=r"(raw[u][h][3]) : "r"(tile + 512 * h + 16 * lane));
          }
        }
        const uint32_t a_col = a_base + slot * kTcACols;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t sel[2][8], pick[2][8];         // [row][2 * block + word]
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if constexpr (BITS == 2) {
#pragma unroll
              for (int w = 0; w < 2; ++w) selectors_2bit(raw[u][h][w], sel[u] + 4 * w);
            } else if constexpr (BITS == 3) {
              selectors_3bit(raw[u][h][0], raw[u][h][1], raw[u][h][2], sel[u]);
            } else {
#pragma unroll
              for (int w = 0; w < 4; ++w) selectors_4bit(raw[u][h][w], sel[u] + 2 * w, pick[u] + 2 * w);
            }
          }
          uint32_t v[16], w[16];
          auto look_up = [&](uint32_t (&out)[16], bool high) {
#pragma unroll
            for (int n = 0; n < 8; ++n)
#pragma unroll
              for (int u = 0; u < 2; ++u)
                out[2 * n + u] = tc_look<BITS>(high ? tab[u].hi : tab[u].lo, sel[u][n], BITS == 4 ? pick[u][n] : 0u);
          };
          // the first lookups come before the wait for the slot
          look_up(v, true);
          if (BITS < 4) look_up(w, false);
          if (h == 0) {
            __syncwarp();
            if (lane == 0) tc_arrive(ring_empty(rs));
            tc_wait(done(prev), p_parity, abort_flag);
            __syncwarp();
            tc_fence_after();
          }
          tc_st_16x128_x8(a_col + 32 * h, v);
          if (BITS == 4) look_up(w, false);
          tc_st_16x128_x8(a_col + 64 + 32 * h, w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) tc_arrive(full(slot));
        rs += 2;
        if (rs >= (uint32_t)R) { rs -= R; r_parity ^= 1u; }
        slot += 2;
        if (slot >= S) slot -= S;
        prev += 2;
        if (prev >= 2 * S) { prev -= 2 * S; p_parity ^= 1u; }
      }
      skip = (uint32_t)(sg.ka - 1 - kt);
      if (sg.left == 0) break;
      sg.next(B);
      ++n_seg;
    }
    if (!SHARE && sg.ka > 0 && sg.kb == B.p[sg.p].n_kt - 1) finish(n_seg % NBUF);
  } else if (warp < kTcFirstToken || (ACT == kActReady && warp < kTcCopyWarp)) {
    // ------------------------------------------------------------------ epilogue
    asm volatile("griddepcontrol.wait;" ::: "memory");     // scales, scratch and y belong to earlier kernels until here
    const uint32_t quad = warp & 3, t_quad = tmem_base + ((32 * quad) << 16) + kAccCol0;
    const int half = (warp - kTcFirstEpi) >> 2, row = 32 * (int)quad + lane, words = B.words;
    uint32_t n_seg = 0;
    do {
      const TcProblem& P = B.p[sg.p];
      const bool owner = sg.kb == P.n_kt - 1;
      if (!SHARE && owner && sg.ka > 0) break;       // the last one: finished by the decoder warps
      const bool whole_tile = !SHARE && owner;
      const uint32_t buf = n_seg % NBUF;
      const int rt = sg.row_tile(P), m0 = (sg.tile - rt * P.n_mt) * NT, n_tok = min(NT, P.M - m0), out = rt * kTcRows + row;
      // a shared tile: this CTA finishes these tokens itself
      const int skip0 = SHARE ? (int)(blockIdx.x % (uint32_t)B.share) * share_tokens(n_tok, B.share) : 0;
      const int skip1 = SHARE ? skip0 + share_tokens(n_tok, B.share) : 0;
      float row_scale = 0.0f;
      if (whole_tile) row_scale = tc_row_scale<BITS>(P.codebook + (size_t)min(out, P.n_rp * 16 - 1) * (1 << BITS)) * (ACT == kActPacked4 ? 0.0625f : 1.0f);
      int* part = B.parts + (size_t)blockIdx.x * words * NT * kTcRows + row;
      auto scales = [&](int c) {
        const int m = m0 + 8 * c + (lane & 7);
        return whole_tile && m < P.M ? ld_global(P.act_scale + m) : 0.0f;
      };
      float sc = scales(half);
      tc_wait(acc_full(buf), (n_seg / NBUF) & 1u, abort_flag);
      __syncwarp();
      tc_fence_after();
      const uint32_t t_hi = t_quad + buf * (2 * NT);
      // eight tokens at a time, the next eight on their way from tensor memory
      uint32_t hi[8], lo[8];
      tc_ld8(t_hi + 8 * half, hi);
      tc_ld8(t_hi + NT + 8 * half, lo);
#pragma unroll 1
      for (int c = half; 8 * c < n_tok; c += kEpiHalves) {
        tc_wait_ld8(hi, lo);
        uint32_t h[8], l[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) { h[j] = hi[j]; l[j] = lo[j]; }
        const float sc_now = sc;
        if (8 * (c + kEpiHalves) < n_tok) {
          tc_ld8(t_hi + 8 * (c + kEpiHalves), hi);
          tc_ld8(t_hi + NT + 8 * (c + kEpiHalves), lo);
          sc = scales(c + kEpiHalves);
        }
        // (uniform) all eight tokens are inside: no test per token; these warps compete with the decoders for issue slots
        const bool whole = 8 * c + 8 <= n_tok;
        if (whole_tile) {
          float* y = P.y + (size_t)(m0 + 8 * c) * P.ldy + out;
          float v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float s = __shfl_sync(0xffffffffu, sc_now, j) * row_scale;
            v[j] = ((float)(int)h[j] * 256.0f + (float)(int)l[j]) * s;
          }
          if (out < P.N) {
            if (whole) {
#pragma unroll
              for (int j = 0; j < 8; ++j) y[(size_t)j * P.ldy] = v[j];
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (8 * c + j < n_tok) y[(size_t)j * P.ldy] = v[j];
            }
          }
        } else if (!SHARE || 8 * c < skip0 || 8 * c >= skip1) {
          int* at = part + 8 * c * kTcRows;
          if (words == 1) {
            // (packed levels are held as 16 q: all sums are multiples of 16)
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j] = ACT == kActPacked4 ? (uint32_t)((int)h[j] * 16 + ((int)l[j] >> 4)) : h[j] * 256u + l[j];
          }
          if (whole) {
#pragma unroll
            for (int j = 0; j < 8; ++j) __stcg(at + j * kTcRows, (int)h[j]);
            if (words == 2) {
#pragma unroll
              for (int j = 0; j < 8; ++j) __stcg(at + (NT + j) * kTcRows, (int)l[j]);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (8 * c + j < n_tok) {
                __stcg(at + j * kTcRows, (int)h[j]);
                if (words == 2) __stcg(at + (NT + j) * kTcRows, (int)l[j]);
              }
          }
        }
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");     // (n_tok <= 8 * half: the first loads are still out)
      tc_fence_before();
      if (!whole_tile) __threadfence();
      __syncwarp();
      if (lane == 0) {
        tc_arrive(acc_empty(buf));
        // the last of the warps says that the part is there (one flag: a reader's look at one takes it a microsecond)
        if (!whole_tile && !SHARE && atomicAdd(parts_stored, 1) == 4 * kEpiHalves - 1) {
          __threadfence();
          asm volatile("st.release.gpu.global.b64 [%0], %1;" ::"l"(B.flags + blockIdx.x), "l"(B.nonce) : "memory");
        }
      }
      ++n_seg;
    } while (sg.next(B));
  } else if (ACT != kActReady) {
    // ------------------------------------------------------------------ token levels
    // The four warps take turns at the units (or, where a warp has too few registers for a unit's levels, pairs of
    // warps do, each for half of the tokens).  Loads run one own unit ahead: latency over four (two) units' time.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    constexpr int kVec = ACT == kActPacked4 ? 1 : 2;
    constexpr int kShare = tc_token_share(NT, ACT), kTurns = kTcTokenWarps / kShare;
    constexpr int NIT = NT / (4 * kShare);                 // four tokens per warp and step
    const uint32_t tg = warp % kTurns;
    const int part = (warp - kTcFirstToken) / kTurns;
    uint4 cur[NIT][kVec];
    const int h = (lane >> 2) & 1, t = lane & 3;           // k-block and column quarter of this lane
    auto token_of = [&](int it) { return part * (NT / kShare) + 4 * it + (lane >> 3); };
    auto load = [&](const TcProblem& P, int kt) {
      // a token's 256 columns: eight lanes x 32 columns (16 bytes of packed levels, 32 of bytes)
      const size_t row = (size_t)P.n_kt * (ACT == kActBytes ? 256 : 128);
#pragma unroll
      for (int it = 0; it < NIT; ++it) {
        const int tok = token_of(it);
        if (tok < P.M) {
          const uint4* src = reinterpret_cast<const uint4*>(P.act + (size_t)tok * row + (size_t)kt * (ACT == kActBytes ? 256 : 128)) +
                             (lane & 7) * kVec;
#pragma unroll
          for (int v = 0; v < kVec; ++v) cur[it][v] = ld_global(src + v);
        }
      }
    };
    uint32_t i = 0;
    // the load of the next own unit: (problem, kt) kTurns units further on in the walk
    Segments ahead = sg;
    int a_kt = sg.kb;
    bool a_more = true;
    auto step = [&](uint32_t n) {
      a_kt -= (int)n;
      while (a_more && a_kt < ahead.ka) {
        const int over = ahead.ka - 1 - a_kt;              // units into the segment that follows
        a_more = ahead.next(B);
        a_kt = ahead.kb - over;
      }
    };
    step(tg);
    if (a_more) load(B.p[ahead.p], a_kt);
    do {
      const TcProblem& P = B.p[sg.p];
      for (int kt = sg.kb; kt >= sg.ka; --kt, ++i) {
        if (i % kTurns != tg) continue;
        const uint32_t slot = i % S, js = i + S;           // unit i - S is js - 2 S
        tc_wait(done(js % (2 * S)), (js / (2 * S) + 1) & 1u, abort_flag);
        uint8_t* dst = gen_base + slot * kBSlot + h * (NT * 128);
        // the eight columns of group jj of this lane's quarter as two words, of token row n
        auto put = [&](int n, int jj, uint32_t first, uint32_t second) {
          uint8_t* at = dst + (n >> 3) * 1024 + (n & 7) * 128 + 4 * t;
          // 16-byte chunk of a step's word e: 2 * step + e.  2 bit: step 2 * (jj >> 1) holds the even columns, the next
          // one the odd ones, both as word jj & 1; else step jj holds the first four columns and the last four.
          const int c0 = BITS == 2 ? 4 * (jj >> 1) + (jj & 1) : 2 * jj, c1 = BITS == 2 ? c0 + 2 : c0 + 1;
          *reinterpret_cast<uint32_t*>(at + 16 * (c0 ^ (n & 7))) = first;
          *reinterpret_cast<uint32_t*>(at + 16 * (c1 ^ (n & 7))) = second;
        };
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
          const int tok = token_of(it);
          if (tok < P.M) {
            if constexpr (ACT == kActPacked4) {
              const uint32_t w[4] = {cur[it][0].x, cur[it][0].y, cur[it][0].z, cur[it][0].w};
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) {
                // 16 * (a - 8) as signed bytes: the nibble in the upper half of its byte, the sign bit flipped
                const uint32_t even = ((w[jj] << 4) & 0xf0f0f0f0u) ^ 0x80808080u, odd = (w[jj] & 0xf0f0f0f0u) ^ 0x80808080u;
                if (BITS == 2) put(tok, jj, even, odd);
                else put(tok, jj, tc_prmt(even, odd, 0x5140u), tc_prmt(even, odd, 0x7362u));
              }
            } else {
              const uint32_t w[8] = {cur[it][0].x, cur[it][0].y, cur[it][0].z, cur[it][0].w,
                                     cur[it][kVec - 1].x, cur[it][kVec - 1].y, cur[it][kVec - 1].z, cur[it][kVec - 1].w};
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) {
                if (BITS == 2) put(tok, jj, tc_prmt(w[2 * jj], w[2 * jj + 1], 0x6420u), tc_prmt(w[2 * jj], w[2 * jj + 1], 0x7531u));
                else put(tok, jj, w[2 * jj], w[2 * jj + 1]);
              }
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) tc_arrive(full(slot));
        step(kTurns);
        if (a_more) load(B.p[ahead.p], a_kt);
      }
    } while (sg.next(B));
  }

  if constexpr (SHARE) {
    // every CTA of the cluster has stored its part (its warps have left their roles: all their waits are bounded)
    __threadfence();
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (warp < kTcDecoders) finish(0);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kTcMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag && status) atomicExch(status, (int)LCD_ERR_TIMEOUT);
}

// Levels as signed bytes in the operand order (see the top of this file): one thread per token, 128-column k-block and
// group jj of eight columns in each of its four quarters.  BYTES: from 8-bit levels, else from packed 4-bit ones.
template <int BITS, bool BYTES>
__global__ void __launch_bounds__(256) ready_levels_kernel(const uint8_t* __restrict__ act, int64_t n, uint8_t* __restrict__ out) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (i >= n) return;
  const int jj = (int)(i & 3);
  const int64_t blk = i >> 2;
  uint32_t first[4], second[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (BYTES) {
      const uint2 w = __ldcg(reinterpret_cast<const uint2*>(act + blk * 128 + 32 * t + 8 * jj));
      first[t] = BITS == 2 ? tc_prmt(w.x, w.y, 0x6420u) : w.x;
      second[t] = BITS == 2 ? tc_prmt(w.x, w.y, 0x7531u) : w.y;
    } else {
      const uint32_t w = __ldcg(reinterpret_cast<const uint32_t*>(act + blk * 64 + 16 * t + 4 * jj));
      const uint32_t e = ((w & 0x0f0f0f0fu) + 0x78787878u) ^ 0x80808080u, o = (((w >> 4) & 0x0f0f0f0fu) + 0x78787878u) ^ 0x80808080u;
      first[t] = BITS == 2 ? e : tc_prmt(e, o, 0x5140u);
      second[t] = BITS == 2 ? o : tc_prmt(e, o, 0x7362u);
    }
  }
  const int c0 = BITS == 2 ? 4 * (jj >> 1) + (jj & 1) : 2 * jj, c1 = BITS == 2 ? c0 + 2 : c0 + 1;
  uint4* dst = reinterpret_cast<uint4*>(out + blk * 128);
  dst[c0] = make_uint4(first[0], first[1], first[2], first[3]);
  dst[c1] = make_uint4(second[0], second[1], second[2], second[3]);
}

int tc_sm_count() { return current_sm_count(); }

// Shape of a launch.
constexpr int kTcMaxShare = 8;                // CTAs of a portable cluster

// Clusters of `size` CTAs with an SM each that are resident together (the graphics processing clusters' sizes decide).
int tc_max_clusters(int size);

struct TcPlan {
  int act, nt, words, grid, share;
  unsigned long long units;
  size_t parts_bytes, flags_bytes;
  double us;                 // estimated duration
};
// One token width: the grid with the shortest estimate.  Measured on B200 (microseconds): a unit 0.33 / 0.35 / 0.68 at
// up to 32 / 64 / 128 tokens, 2 bit (3 bit 5 % more; 4 bit 0.68 / 0.68 / 0.88: its lookups; 128 tokens take 0.57 in a launch
// of a few units per SM, 0.83 in one of a millisecond, as the dense kernel's stages lengthen too); 3 before the
// first unit and after the last store; a tile's drain 0.016 a token; a cut tile 2.5 for the hand-over, and 512 bytes a token
// and part at 20 GB/s per SM to read the parts back; a tile shared in a cluster 3.6, each CTA reading its tokens only.
// Against the dense kernel this chooses right to a few percent (2 bit, one call from x to y, tensor memory / dense): 13B
// layer 127 / 224 at 256 tokens, 254 / 299 at 512, 500 / 544 at 1024, 1060 / 975 at 2048; 7B layer 57 / 179 at 128, 320 /
// 348 at 1024, 684 / 637 at 2048; layer of 1024 columns 79 / 100 at 2048.  Candidates: all SMs (least work per CTA, most
// tiles cut), and, where the rows are of one length, one CTA per tile (none cut), two to four with the last one finishing,
// two to eight as a cluster that finishes together.
TcPlan tc_plan_width(const Problem* probs, int count, int nt) {
  TcPlan q = {};
  q.act = probs[0].dense_levels ? kActReady : probs[0].act_bits == 8 ? kActBytes : kActPacked4;
  q.nt = nt;
  int64_t max_kt = 1, min_kt = 1 << 30, max_m = 1;
  unsigned long long tiles = 0;
  for (int i = 0; i < count; ++i) {
    const Problem& p = probs[i];
    const int64_t kt = p.K_pad / kTileK;
    const unsigned long long t = (unsigned long long)((p.N_pad + kTcRows - 1) / kTcRows) * ((p.M + nt - 1) / nt);
    tiles += t;
    q.units += t * kt;
    max_kt = kt > max_kt ? kt : max_kt;
    min_kt = kt < min_kt ? kt : min_kt;
    max_m = p.M > max_m ? p.M : max_m;
  }
  // Pieces of at least a sixteenth of the longest row: a tile then lies in at most kTcMaxParts + 1 pieces (the finisher has
  // a lane and room in shared memory for each).
  const unsigned long long piece = (unsigned long long)(max_kt + 15) / 16, n_sm = (unsigned long long)tc_sm_count();
  unsigned long long most = n_sm < q.units ? n_sm : q.units;
  if (most > q.units / piece) most = q.units / piece;
  const double unit_us = probs[0].bits == 4 ? (nt == 128 ? 0.88 : 0.68) : (nt <= 32 ? 0.33 : nt == 64 ? 0.35 : 0.68) * (probs[0].bits == 3 ? 1.05 : 1.0);
  const double tokens = (double)(max_m < nt ? max_m : nt);
  const bool long_rows = max_kt > kTcExactUnits;
  const double part_bytes = probs[0].act_bits == 4 && long_rows ? 768 : 512;      // (two planes: 5120 x 13824 at 100 tokens 25.8 -> 24.9 us)
  auto consider = [&](unsigned long long grid, int share, double parts, double fixed, double read_tokens, double drains) {
    const double us = fixed + (double)((q.units + grid - 1) / grid) * unit_us + drains * tokens * 0.016 + parts * read_tokens * part_bytes / 20000;
    if (q.grid == 0 || us < q.us) {
      q.us = us;
      q.grid = (int)grid;
      q.share = share;
    }
  };
  const double drains = nt > 32 ? 1.0 + (double)tiles / most : 1.0;        // tiles drained one after the other
  consider(most, 0, (double)most / tiles + 0.5, 5.5, tokens, drains);
  if (min_kt == max_kt)
    for (int s = 1; s <= kTcMaxShare && s <= min_kt && tiles * s <= n_sm; ++s) {
      if (s == 1) consider(tiles, 0, 0.0, 3.0, 0.0, 1.0);
      else if (s <= 4 && tiles * s <= most) consider(tiles * s, 0, s - 1, 5.5, tokens, nt > 32 ? 1.0 + 1.0 / s : 1.0);
      if (s > 1 && tiles <= (unsigned long long)tc_max_clusters(s)) consider(tiles * s, s, s - 1, 6.6, (double)(((int64_t)tokens + 8 * s - 1) / (8 * s) * 8), 1.0);
    }
  // One number a part where the planes' sums fit 24 bits (255 * 8 * 8192 < 2^24): rounding their sum is then the same as rounding
  // them apart, what whole tiles and the dense kernel do, and y does not depend on which tiles were cut.  On longer rows the
  // planes stay apart (4096 x 11008, 2 bit, lookup alone at 48 / 16 tokens 12.5 / 10.5 us, 11.8 / 9.9 as one number).
  q.words = probs[0].act_bits == 4 && !long_rows && (q.units + q.grid - 1) / q.grid <= kTcWordUnits ? 1 : 2;
  q.parts_bytes = (size_t)q.grid * q.words * q.nt * kTcRows * sizeof(int);
  q.flags_bytes = (size_t)round_up_u64((uint64_t)q.grid * sizeof(unsigned long long), 256);
  return q;
}
TcPlan tc_plan(const Problem* probs, int count) {
  int64_t m = 1;
  for (int i = 0; i < count; ++i) m = probs[i].M > m ? probs[i].M : m;
  if (!probs[0].dense_levels) return tc_plan_width(probs, count, m <= 16 ? 16 : 32);
  TcPlan best = tc_plan_width(probs, count, 32);
  for (int nt = 64; nt <= 128 && m > nt / 2; nt *= 2) {
    const TcPlan q = tc_plan_width(probs, count, nt);
    if (q.us < best.us) best = q;
  }
  return best;
}

// Different for every launch of every process: parts left by an earlier launch, or whatever else a workspace holds at
// first, cannot pass for this launch's (the counter through a 64-bit mixing function, splitmix64's).
unsigned long long tc_nonce() {
  static std::atomic<unsigned long long> counter{(unsigned long long)reinterpret_cast<uintptr_t>(&counter)};
  unsigned long long z = counter.fetch_add(0x9E3779B97F4A7C15ull, std::memory_order_relaxed);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return (z ^ (z >> 31)) | 1ull;
}

template <typename... Params, typename... Args>
lcd_status tc_launch(void (*kern)(Params...), unsigned grid, unsigned cluster, unsigned block, size_t smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
  if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
  return LCD_OK;
}

// Weights are streamed before griddepcontrol.wait; levels, scales, scratch and y are touched after it.
template <int BITS, int NT, int ACT, bool SHARE>
lcd_status tc_launch_instance(const TcMaps& maps, const TcBatch& batch, int grid, int32_t* status, cudaStream_t stream) {
  auto kern = lut_gemv_tc_kernel<BITS, NT, ACT, SHARE>;
  constexpr size_t smem = 1024 + (size_t)tc_smem_layout<BITS, NT>(3);
  static_assert(smem <= 227 * 1024, "shared memory of one CTA");
  static PerDeviceFlag attr_set;   // per template instance and device
  int dev;
  if (attr_set.first(&dev)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) { set_cuda_error((int)e); return LCD_ERR_CUDA; }
    attr_set.done(dev);
  }
  return tc_launch(kern, (unsigned)grid, (unsigned)(SHARE ? batch.share : 1), kTcThreads, smem, stream, maps, batch, status);
}
template <int BITS, int NT, int ACT>
lcd_status tc_launch_t(const TcMaps& maps, const TcBatch& batch, int grid, int32_t* status, cudaStream_t stream) {
  return batch.share > 0 ? tc_launch_instance<BITS, NT, ACT, true>(maps, batch, grid, status, stream)
                         : tc_launch_instance<BITS, NT, ACT, false>(maps, batch, grid, status, stream);
}

int tc_max_clusters(int size) {
  static std::atomic<int> known[64][kTcMaxShare + 1];         // + 1; a property of the device
  int dev = 0;
  const bool have = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
  if (have) {
    const int v = known[dev][size].load(std::memory_order_relaxed);
    if (v > 0) return v - 1;
  }
  auto kern = lut_gemv_tc_kernel<2, 16, kActPacked4, true>;                  // (every instance takes an SM to itself)
  constexpr size_t smem = 1024 + (size_t)tc_smem_layout<2, 16>(3);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)size);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)size;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (!have || cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;                    // (no device: no shares)
  }
  known[dev][size].store(n + 1, std::memory_order_relaxed);
  return n;
}

template <int BITS>
lcd_status tc_launch_bits(const TcMaps& maps, const TcBatch& batch, const TcPlan& q, int32_t* status, cudaStream_t stream) {
  if (q.act == kActReady)
    return q.nt == 32   ? tc_launch_t<BITS, 32, kActReady>(maps, batch, q.grid, status, stream)
           : q.nt == 64 ? tc_launch_t<BITS, 64, kActReady>(maps, batch, q.grid, status, stream)
                        : tc_launch_t<BITS, 128, kActReady>(maps, batch, q.grid, status, stream);
  if (q.act == kActBytes)
    return q.nt == 16 ? tc_launch_t<BITS, 16, kActBytes>(maps, batch, q.grid, status, stream)
                      : tc_launch_t<BITS, 32, kActBytes>(maps, batch, q.grid, status, stream);
  return q.nt == 16 ? tc_launch_t<BITS, 16, kActPacked4>(maps, batch, q.grid, status, stream)
                    : tc_launch_t<BITS, 32, kActPacked4>(maps, batch, q.grid, status, stream);
}

}  // namespace

// The exact int32 sums hold |byte x 16 q| <= 255 * 128 per column: rows of at most 65536 columns.
bool lut_gemv_tc_supported(const Problem* probs, int count) {
  unsigned long long units = 0;
  for (int i = 0; i < count; ++i) {
    const Problem& p = probs[i];
    if (p.bits != probs[0].bits || p.act_bits != probs[0].act_bits || p.dense_levels != probs[0].dense_levels) return false;
    if (p.K_pad > 65536 || p.M < 1 || (p.act_bits != 4 && p.act_bits != 8)) return false;
    if (!p.dense_levels && p.M > 32) return false;
    units += (unsigned long long)((p.N_pad + kTcRows - 1) / kTcRows) * ((p.M + 15) / 16) * (p.K_pad / kTileK);
  }
  return units < (1ull << 30);
}

// Enough for any plan of these shapes: who asks does not say which levels there will be.
size_t lut_gemv_tc_workspace_bytes(const Problem* probs, int count) {
  int64_t m = 1;
  for (int i = 0; i < count; ++i) m = probs[i].M > m ? probs[i].M : m;
  const size_t n_sm = (size_t)tc_sm_count(), nt = m <= 16 ? 16 : m <= 32 ? 32 : m <= 64 ? 64 : 128;
  return n_sm * 2 * nt * kTcRows * sizeof(int) + (size_t)round_up_u64(n_sm * sizeof(unsigned long long), 256);
}

double lut_gemv_tc_estimate_us(const Problem* probs, int count) { return tc_plan(probs, count).us; }

lcd_status launch_ready_levels(const Problem& p, void* out, void* stream) {
  const int64_t n = p.M * (p.K_pad / 32);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  uint8_t* o = static_cast<uint8_t*>(out);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // (4-bit indices: the order of 3-bit ones)
  if (p.bits == 2)
    return p.act_bits == 8 ? tc_launch(ready_levels_kernel<2, true>, blocks, 1, 256, 0, s, p.act_idx, n, o)
                           : tc_launch(ready_levels_kernel<2, false>, blocks, 1, 256, 0, s, p.act_idx, n, o);
  return p.act_bits == 8 ? tc_launch(ready_levels_kernel<3, true>, blocks, 1, 256, 0, s, p.act_idx, n, o)
                         : tc_launch(ready_levels_kernel<3, false>, blocks, 1, 256, 0, s, p.act_idx, n, o);
}

lcd_status launch_lut_gemv_tc(const Problem* probs, int count, void* workspace, size_t workspace_bytes,
                              int32_t* status_word, void* stream) {
  if (count < 1 || count > LCD_MAX_BATCH) return LCD_ERR_INVALID_ARG;
  if (!lut_gemv_tc_supported(probs, count)) return LCD_ERR_UNSUPPORTED;
  const TcPlan q = tc_plan(probs, count);
  if (workspace == nullptr || workspace_bytes < q.parts_bytes + q.flags_bytes) return LCD_ERR_BUFFER_TOO_SMALL;
  const int bits = probs[0].bits;
  EncodeTiledFn encode = encode_tiled();
  if (!encode) return LCD_ERR_CUDA;
  TcMaps maps;
  TcBatch batch;
  batch.count = count;
  unsigned long long total = 0;
  int64_t max_m = 0;
  for (int i = 0; i < count; ++i) {
    const Problem& p = probs[i];
    TcProblem& g = batch.p[i];
    max_m = p.M > max_m ? p.M : max_m;
    g.codebook = p.codebook;
    g.act = p.act_idx;
    g.act_scale = p.act_scale;
    g.y = p.y;
    g.ldy = p.ldy;
    g.N = (int)p.N;
    g.M = (int)p.M;
    g.n_rp = (int)(p.N_pad / kPairRows);
    g.n_kt = (int)(p.K_pad / kTileK);
    g.n_mt = (int)((p.M + q.nt - 1) / q.nt);
    g.n_tiles = g.n_mt * (int)((p.N_pad + kTcRows - 1) / kTcRows);
    g.unit0 = (unsigned)total;
    total += (unsigned long long)g.n_tiles * (unsigned long long)g.n_kt;
    const cuuint32_t one[3] = {1, 1, 1};
    const cuuint64_t dims[3] = {(cuuint64_t)(64 * bits), (cuuint64_t)g.n_kt, (cuuint64_t)g.n_rp};     // items of 64 x bits 8-byte words
    const cuuint64_t strides[2] = {(cuuint64_t)(512 * bits), (cuuint64_t)g.n_kt * (512 * bits)};
    const cuuint32_t box[3] = {(cuuint32_t)(64 * bits), 1, 8};
    if (encode(&maps.items[i], CU_TENSOR_MAP_DATA_TYPE_INT64, 3, const_cast<uint8_t*>(p.tiles), dims, strides, box, one,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return LCD_ERR_CUDA;
    if (q.act == kActReady) {
      const cuuint64_t ldims[2] = {(cuuint64_t)p.K_pad, (cuuint64_t)p.M}, lstrides[1] = {(cuuint64_t)p.K_pad};
      const cuuint32_t lbox[2] = {128, (cuuint32_t)q.nt};
      if (encode(&maps.levels[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(p.act_idx), ldims, lstrides, lbox, one,
                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return LCD_ERR_CUDA;
    } else {
      maps.levels[i] = maps.items[i];
    }
  }
  for (int i = count; i < LCD_MAX_BATCH; ++i) {
    batch.p[i] = batch.p[0];
    maps.items[i] = maps.items[0];
    maps.levels[i] = maps.levels[0];
  }
  batch.per = (unsigned)(total / q.grid);
  batch.extra = (unsigned)(total % q.grid);
  batch.ctas_per_unit = (float)((double)q.grid / (double)total);
  batch.share = q.share;
  batch.words = q.words;
  batch.clean = max_m <= 32;       // few tokens: the scratch, zero-filled by the caller, is left zero-filled
  batch.nonce = tc_nonce();
  batch.parts = static_cast<int*>(workspace);
  batch.flags = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(workspace) + q.parts_bytes);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return bits == 2   ? tc_launch_bits<2>(maps, batch, q, status_word, s)
         : bits == 3 ? tc_launch_bits<3>(maps, batch, q, status_word, s)
                     : tc_launch_bits<4>(maps, batch, q, status_word, s);
}

}  // namespace lcd
