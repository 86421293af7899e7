// Dirty-query attention on the tensor cores (Section 3.3, Region-Level Sparse
// Attention): the queries of the active tokens attend over every token's keys
// and values.  In the self-attention K/V come from the (layer, timestep) cache
// whose dirty rows the QKV GEMM has just refreshed; in the text cross-
// attention they are the per-layer text keys / values.
//
// One work unit = one or two tiles of 128 queries of one head over the keys
// (or a share of them), in blocks of 80 keys; one persistent CTA per SM.  Two
// streams, each with its own S / P and O in tensor memory, its own issuing
// warp and its own four softmax warps, share every K and V block (two tiles:
// a stream each) or take the blocks in turn (one tile; their results are
// merged when the unit ends).
//   warp 0        Q and K: TMA, and cp.async for the last 8 head dims
//   warps 1, 3    a stream's S = Q K^T (M = 128, N = 80, 5 K-steps of 16) and
//                 O += P V (M = 128, N = 80, 5 K-steps of 16 keys; P read from
//                 TMEM as the A operand, V from shared memory, MN-major);
//                 warp 1 owns the tensor memory
//   warp 2        V, as K
//   warps 4-7     softmax of stream 0, one thread per query row
//   warps 8-11    softmax of stream 1
// Operands come through 3-D tensor maps (head_dim, head, row) as a 64-wide
// 128B-swizzled tile plus a tail; the head_dim extent is the true 72, and the
// pad to 80 is zero and adds nothing to Q K^T.  A stream's S has two buffers,
// and its P replaces the S that it came from, so that S of the next block is
// there when the softmax of this one ends.  The softmax (base 2) takes a max
// in a stream's first block only: later blocks use the same reference unless
// their exponentials grow past 2^64 of it (then the reference is raised, O
// rescaled and the block done again).
//
// What bounds it (80 keys, both streams): the tensor pipe and the shared
// memory that feeds it 1180 cycles without any softmax (920 of MMA, the rest
// TMA writes), the softmax 1250 without any MMA (640 of exponentials at 32 per
// cycle and SM; two warps a scheduler), together 1430.  Measured, earlier form
// (two CTAs an SM, 64-key blocks, one tile each, K and V tails through TMA,
// a max per block) -> this one: 831 x 4096 (with the combine kernel it needed)
// 36.4 -> 27.4 us, 4096 x 4096 116.6 -> 82.9, 3248 x 16384 326 -> 229 (1.07
// PFLOP/s), 132 x 1024 13.7 -> 10.3.
//
// Pairs left over by the last whole wave can have their keys shared by up to
// nine units.  Each leaves its unnormalised O with the rows' reference and sum
// in a workspace (as column planes, so that accesses are whole 512-byte runs),
// and the CTA that finishes last merges them.
#include <cuda.h>
#include <math.h>

#include <mutex>
#include <unordered_map>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"
#include "tma_host.h"

namespace rc {

namespace {

using namespace rc::tc;

constexpr int BQ = 128, BKV = 80, THREADS = 384;
// TMEM columns: two S buffers of each stream (P goes over the first half of
// its S), then O (80 each)
constexpr int TMEM_COLS = 512;
constexpr uint32_t TM_O = 4 * BKV, TM_O_STEP = 80;
static_assert(TM_O + 2 * TM_O_STEP <= TMEM_COLS, "two streams fit the tensor memory");
__device__ __forceinline__ uint32_t tm_s(int x, int b) { return uint32_t(BKV * (2 * x + b)); }
// floats per row of a workspace slot: a piece's DH columns, its row max and
// sum (as column planes: DH / 4 planes of 128 float4, then 128 (max, sum))
constexpr int PART_STRIDE = 76;
static_assert(72 + 2 <= PART_STRIDE, "a slot holds DH + 2 floats per row");
// A block's sum of exponentials past which its reference is raised.
constexpr float RAISE_SUM = 18446744073709551616.f;  // 2^64

// Packed f32x2 arithmetic (two lanes of f32 per 64-bit register pair).
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// The softmax's steps on columns in registers, in the order they are written.
__device__ __forceinline__ void scale_pair(uint32_t& a, uint32_t& b, uint64_t scale,
                                           uint64_t shift) {
  asm volatile(
      "{\n\t.reg .b64 t;\n\tmov.b64 t, {%0, %1};\n\t"
      "fma.rn.f32x2 t, t, %2, %3;\n\tmov.b64 {%0, %1}, t;\n\t}"
      : "+r"(a), "+r"(b)
      : "l"(scale), "l"(shift));
}
__device__ __forceinline__ void exp_in_place(uint32_t& a) {
  asm volatile("ex2.approx.ftz.f32 %0, %0;" : "+r"(a));
}
__device__ __forceinline__ void sum_pair(uint64_t& s, uint32_t a, uint32_t b) {
  asm volatile("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %2};\n\tadd.rn.f32x2 %0, %0, t;\n\t}"
               : "+l"(s)
               : "r"(a), "r"(b));
}
__device__ __forceinline__ uint32_t pack_pair(uint32_t lo, uint32_t hi) {
  uint32_t d;
  asm volatile("cvt.rn.bf16x2.f32 %0, %2, %1;"
               : "=r"(d)
               : "f"(__uint_as_float(lo)), "f"(__uint_as_float(hi)));
  return d;
}

// The reference a row's exponents are taken against: its max, or 0 when every
// score so far is -inf (whose exponentials are then 0, not NaN).
__device__ __forceinline__ float finite_max(float m) { return m == -INFINITY ? 0.f : m; }

template <int DH>
struct ACfg {
  static_assert(DH == 64 || DH == 72, "head_dim 64 or 72");
  static constexpr bool TAIL = DH > 64;          // head dims 64..79 (72..79 read as zero)
  static constexpr int DHP = TAIL ? 80 : 64;     // padded head dim of the PV accumulator
  // shared-memory operand tiles: a 64-wide 128B-swizzled part, a 16-wide
  // 32B-swizzled tail
  static constexpr int Q128 = BQ * 128, Q32 = TAIL ? BQ * 32 : 0;
  static constexpr int K128 = BKV * 128, K32 = TAIL ? BKV * 32 : 0;
  // K: 64-wide SW128 tile + 16-wide SW32 tail (the S MMA reads them as two
  // K-major operands); V: one SW128 atom per 64 head-dim columns, so that P V
  // is a single MMA of N = DHP per 16 keys (MN-major B spanning the atoms).
  // Of the second atom only 32 bytes a row are used, so four stages share one
  // A unit of one tile gives its blocks to the streams in turn, and a stream
  // waits only for its own: with rings of even depth a stage then keeps its
  // stream within a unit, so that a parity wait never meets a fill two ahead
  // of the last one it saw.  (From one unit to the next q_full and o_free
  // follow every K and V of the unit before.)
  static constexpr int K_STAGES = 6;
  static constexpr int V_STAGES = 8;
  static_assert(K_STAGES % 2 == 0 && V_STAGES % 2 == 0, "a stage belongs to one stream of a unit");
  static constexpr int Q_BYTES = Q128 + Q32;
  static constexpr int K_STRIDE = (K128 + K32 + 1023) & ~1023;  // bytes between K stages
  static constexpr int V_TAILS = TAIL ? (V_STAGES + 3) / 4 : 0;
  static constexpr size_t SMEM = size_t(2) * Q_BYTES + K_STAGES * K_STRIDE +
                                 size_t(V_STAGES + V_TAILS) * K128 + 1024;
  static_assert(Q_BYTES % 1024 == 0 && K128 % 1024 == 0, "128B-swizzled tiles start on 1024 bytes");
  // byte offset of V stage s and of its tail (32 s mod 128 into the rows of
  // a shared atom) from the start of the V ring
  __host__ __device__ static constexpr int v_main(int s) { return s * K128; }
  __host__ __device__ static constexpr int v_tails(int s) {
    return (V_STAGES + (s >> 2)) * K128 + 32 * (s & 3);
  }
  // kind::f16, D f32, A/B bf16; S: both K-major; PV: B (V) MN-major (bit 16)
  static constexpr uint32_t IDESC_S = (1u << 4) | (1u << 7) | (1u << 10) |
                                      (uint32_t(BKV >> 3) << 17) | (uint32_t(BQ >> 4) << 24);
  static constexpr uint32_t IDESC_PV = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) |
                                       (uint32_t(DHP >> 3) << 17) | (uint32_t(BQ >> 4) << 24);
};

// Query tile qt of a launch: its item, first compact row and live rows.
struct TileLoc {
  int item, row0, rows;
};
__device__ __forceinline__ TileLoc locate_tile(const RowMap& rm, int n_items, int D, int qt) {
  if (!rm.meta) return TileLoc{0, qt * BQ, min(BQ, D - qt * BQ)};
  int i = 0;
  while (i + 1 < n_items && __ldg(rm.meta + META_TILE + i + 1) <= qt) ++i;
  const int j = qt - __ldg(rm.meta + META_TILE + i);
  return TileLoc{i, __ldg(rm.meta + META_OFF + i) + j * BQ,
                 min(BQ, __ldg(rm.meta + META_CNT + i) - j * BQ)};
}

// Query tiles of a launch: 128-row tiles of each item's rows.
__device__ __forceinline__ int query_tiles(const RowMap& rm, int n_items, int D) {
  return rm.meta ? __ldg(rm.meta + META_TILE + n_items) : (D + BQ - 1) / BQ;
}

// A query group: one tile of 128 rows of an item, or two.  A pair = one query
// group of one head (heads outermost).  Whole waves of pairs are one unit
// each; the R pairs left over may have their keys shared by `split` units
// each, in one wave.
//
// The plan of a launch, tabulated by the host for 1 .. PLAN_TABLE query groups
// of one and of two tiles: the estimated duration and the split that gives it.
// The device picks the cheaper (a batch's items fill their groups unevenly,
// and only it knows their counts); larger launches take two tiles and no split.
constexpr int PLAN_TABLE = 160, MAX_SPLIT = 9;
struct PlanTable {
  uint16_t cost[2][PLAN_TABLE];
  uint8_t split[2][PLAN_TABLE];
};
// Estimated duration in units of 10 ns, fitted to launches of 39 .. 4096
// queries over 131 .. 16384 keys with every split: a block of 80 keys takes
// 0.45 us for one tile and 0.74 us for two, a wave UNIT more, and the merge of
// shared pairs, by the last of their units, MERGE + MERGE_SHARE per share.
// (4096 keys, the best / the next plan in us: 201 queries one tile split in
// four 15.3 / two tiles 21.2; 831 one tile whole 27.4 / two tiles split in two
// 30.2; 4096 two tiles whole 82.9 / one tile 94.6; 3248 queries over 16384
// keys two tiles, the rest split in two 229 / whole 291.)
constexpr int BLOCK1 = 45, BLOCK2 = 74, UNIT = 60;
constexpr int MERGE1 = 400, MERGE2 = 480, MERGE_SHARE1 = 30, MERGE_SHARE2 = 90;
constexpr int SLOTS_PER_SM = 2;    // workspace slots: two tiles of a shared unit
constexpr int CAPTURE_KEYS = 448;  // keys of a launch that captures probabilities, at most
int plan_cost(int pairs, int nkb, int grid, int tiles, int split) {
  const int block = tiles == 2 ? BLOCK2 : BLOCK1;
  if (split == 1) return (pairs + grid - 1) / grid * (nkb * block + UNIT);
  return pairs / grid * (nkb * block + UNIT) + (nkb + split - 1) / split * block + UNIT +
         (tiles == 2 ? MERGE2 + MERGE_SHARE2 * split : MERGE1 + MERGE_SHARE1 * split);
}
int pick_split(int pairs, int nkb, int grid, int tiles, int most, int* cost) {
  int best = 1;
  *cost = plan_cost(pairs, nkb, grid, tiles, 1);
  const int rest = pairs % grid;
  for (int s = 2; s <= most && s <= nkb && rest > 0 && rest * s <= grid; ++s) {
    const int c = plan_cost(pairs, nkb, grid, tiles, s);
    if (c < *cost) {
      *cost = c;
      best = s;
    }
  }
  return best;
}

__device__ __forceinline__ int query_groups(const RowMap& rm, int n_items, int D, int rows) {
  if (!rm.meta) return (D + rows - 1) / rows;
  int g = 0;
  for (int i = 0; i < n_items; ++i) g += (__ldg(rm.meta + META_CNT + i) + rows - 1) / rows;
  return g;
}
__device__ __forceinline__ TileLoc locate_group(const RowMap& rm, int n_items, int D, int rows,
                                                int g) {
  if (!rm.meta) return TileLoc{0, g * rows, min(rows, D - g * rows)};
  int i = 0, c = __ldg(rm.meta + META_CNT);
  while (i + 1 < n_items && g >= (c + rows - 1) / rows) {
    g -= (c + rows - 1) / rows;
    c = __ldg(rm.meta + META_CNT + ++i);
  }
  return TileLoc{i, __ldg(rm.meta + META_OFF + i) + g * rows, min(rows, c - g * rows)};
}

// The units of one CTA, handed out round robin.
struct AttnUnits {
  int groups, rows, split, whole, units, nkb;
  __device__ void init(const PlanTable& pt, const RowMap& rm, int n_items, int D, int heads, int Nk,
                       int grid) {
    nkb = (Nk + BKV - 1) / BKV;
    const int tiles = query_tiles(rm, n_items, D);
    rows = 2 * BQ;
    split = 1;
    groups = query_groups(rm, n_items, D, rows);
    if (tiles >= 1 && tiles <= PLAN_TABLE) {
      const bool one = pt.cost[0][tiles - 1] < pt.cost[1][groups - 1];
      split = one ? pt.split[0][tiles - 1] : pt.split[1][groups - 1];
      if (one) {
        rows = BQ;
        groups = tiles;
      }
    }
    const int pairs = groups * heads;
    whole = split == 1 ? pairs : pairs / grid * grid;
    units = whole + (pairs - whole) * split;
  }
};
struct AttnUnit {
  int pair, g, h, kb0, kb1;
  int share;  // index among the shared units, -1 for a whole pair
  __device__ void set(const AttnUnits& un, int u) {
    int q = 0, n = 1;
    pair = u;
    share = -1;
    if (u >= un.whole) {
      share = u - un.whole;
      n = un.split;
      pair = un.whole + share / n;
      q = share - share / n * n;
    }
    h = pair / un.groups;
    g = pair - h * un.groups;
    kb0 = un.nkb * q / n;
    kb1 = un.nkb * (q + 1) / n;
  }
};

// The last 8 of 72 head dims of a key block: 16 bytes a row, through cp.async
// (a TMA box takes as long for a row of 16 bytes as for one of 128: with
// 16-wide boxes for the tails 112 rows of K and V took 1043 cycles to load,
// with a 64-wide one for V 1210, without them 610).  Byte offset of 16-byte chunk j
// of row r in the K tail (32-byte rows, 32B swizzle) and in V's second atoms
// (128-byte rows, 128B swizzle; stage s has chunks 2 (s mod 4) and the next).
__device__ __forceinline__ int k_tail(int r, int j) { return r * 32 + 16 * (j ^ ((r >> 2) & 1)); }
__device__ __forceinline__ int v_tail(int r, int j) { return r * 128 + 16 * (j ^ (r & 7)); }
template <bool V>
__device__ __forceinline__ void load_tail(uint8_t* dst, int chunk, const bf16* src, int ld,
                                          int row0, int rows, int lane) {
#pragma unroll
  for (int q = 0; q < (BKV + 31) / 32; ++q) {
    const int r = q * 32 + lane;
    if (r < BKV) {
      // rows past the end are filled with zeros, as the TMA does
      const bool in = row0 + r < rows;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                       saddr(dst + (V ? v_tail(r, chunk) : k_tail(r, chunk)))),
                   "l"(src + size_t(in ? row0 + r : 0) * ld), "r"(in ? 16 : 0)
                   : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// The tails of all but the last PENDING of the blocks issued so far (g) have
// landed: made visible to the tensor core, and their stages' barriers told
// (told counts the blocks).
template <int PENDING>
__device__ __forceinline__ void tell_tails(int g, int& told, uint32_t full, int stages, int lane) {
  asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
  if (told >= g - PENDING) return;
  fence_proxy_async_smem();
  __syncwarp();
  for (; told < g - PENDING; ++told)
    if (lane == 0) mbar_arrive(full + 8 * (told % stages));
}

template <int DH, bool CAP>
__global__ void __launch_bounds__(THREADS, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmQt,
               const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
               const bf16* __restrict__ Kp, const bf16* __restrict__ Vp, int ldkv, int kv_rows,
               const __grid_constant__ AttnItems ai, const __grid_constant__ PlanTable pt,
               int Nk, bf16* __restrict__ O, int ldo,
               int heads, RowMap rm, float scale_log2, unsigned* err, float* __restrict__ part,
               unsigned* __restrict__ ticket, const __grid_constant__ AttnCapture cap) {
  using C = ACfg<DH>;
  constexpr int KS = C::K_STAGES, VS = C::V_STAGES;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sQ = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                           ~uintptr_t(1023));
  uint8_t* sK = sQ + 2 * C::Q_BYTES;
  uint8_t* sV = sK + KS * C::K_STRIDE;
  constexpr int BARS = 2 + 2 * KS + 2 * VS + 12 + 3;
  __shared__ uint64_t bars[BARS];
  __shared__ float2 s_ml[2][2][BQ];  // (max, sum) of the streams' rows, units alternating
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, s_last;
  volatile int* abort_flag = &s_abort;
  const uint32_t q_full = saddr(bars), q_empty = q_full + 8;
  const uint32_t k_full = q_empty + 8, k_empty = k_full + 8 * KS;          // [KS]
  const uint32_t v_full = k_empty + 8 * KS, v_empty = v_full + 8 * VS;      // [VS]
  const uint32_t s_full = v_empty + 8 * VS;                                 // [stream][buffer]
  const uint32_t p_ready = s_full + 32, pv_done = p_ready + 32;             // [stream][buffer]
  const uint32_t o_full = pv_done + 32, o_free = o_full + 8;
  const uint32_t meet = o_free + 8;  // the softmax warps of both streams

  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < BARS; ++i) mbar_init(q_full + 8 * i, 1);
    for (int i = 0; i < KS; ++i) mbar_init(k_empty + 8 * i, 2);
    for (int i = 0; i < VS; ++i) mbar_init(v_empty + 8 * i, 2);
    mbar_init(q_empty, 2);
    mbar_init(o_full, 2);
    if (C::TAIL) {  // the TMA's arrival and that of the tail's warp
      for (int i = 0; i < KS; ++i) mbar_init(k_full + 8 * i, 2);
      for (int i = 0; i < VS; ++i) mbar_init(v_full + 8 * i, 2);
    }
    for (int i = 0; i < 4; ++i) mbar_init(p_ready + 8 * i, 4);
    mbar_init(o_free, 8);
    mbar_init(meet, 8);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(saddr(&tmem_slot), TMEM_COLS);
  if (warp == 0 && elect_one()) {
    const CUtensorMap* maps[4] = {&tmQ, &tmK, &tmV, &tmQt};
#pragma unroll
    for (int i = 0; i < (C::TAIL ? 4 : 3); ++i)
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(maps[i])) : "memory");
  }
  if (C::TAIL) {
    // head dims 72 .. 79 of every K and V stage: zero, and never written again
    const uint4 z = make_uint4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < KS * BKV; i += THREADS) {
      const int r = i % BKV;
      *reinterpret_cast<uint4*>(sK + (i / BKV) * C::K_STRIDE + C::K128 + k_tail(r, 1)) = z;
    }
    for (int i = threadIdx.x; i < VS * BKV; i += THREADS) {
      const int r = i % BKV;
      const int s = i / BKV;
      *reinterpret_cast<uint4*>(sV + C::v_tails(s & ~3) + v_tail(r, 2 * (s & 3) + 1)) = z;
    }
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // the live row count (and, for several items, the row table) was written
  // two or more launches earlier: read before the programmatic-dependency
  // wait (every kernel of the library waits for its predecessor before
  // letting its successor start); Q and the fresh K / V rows come from the
  // predecessor
  const int D = live_count(rm.count, rm.bound, err);
  AttnUnits un;
  un.init(pt, rm, ai.n, D, heads, Nk, int(gridDim.x));
  const int u0 = blockIdx.x, du = gridDim.x;
  // the roles wait for the predecessor where they first need it: what comes
  // before (the first unit's place, and fetching the code that finds it) runs
  // beside the predecessor's end

  if (warp == 0) {
    // ------------------------------------------------------------ Q and K
    const bool leader = elect_one();
    int g = 0, uc = 0, told = 0;
    AttnUnit w;
    for (int u = u0; u < un.units; u += du, ++uc) {
      w.set(un, u);
      const TileLoc tl = locate_group(rm, ai.n, D, un.rows, w.g);
      const int krow = ai.krow[tl.item], tiles = tl.rows > BQ ? 2 : 1;
      if (!mbar_sleep_warp(q_empty, (uc & 1) ^ 1, abort_flag)) goto timeout;
      if (leader) mbar_expect_tx(q_full, tiles * C::Q_BYTES);
      if (uc == 0) {
        pdl_wait();
        pdl_trigger();
      }
      if (leader) {
        for (int x = 0; x < tiles; ++x) {
          uint8_t* q = sQ + x * C::Q_BYTES;
          tma_load_3d(saddr(q), &tmQ, q_full, 0, w.h, tl.row0 + x * BQ);
          if (C::TAIL) tma_load_3d(saddr(q + C::Q128), &tmQt, q_full, 64, w.h, tl.row0 + x * BQ);
        }
      }
      for (int kb = w.kb0; kb < w.kb1; ++kb, ++g) {
        const int s = g % KS;
        if (!mbar_sleep_warp(k_empty + 8 * s, ((g / KS) & 1) ^ 1, abort_flag)) goto timeout;
        uint8_t* b = sK + s * C::K_STRIDE;
        if (leader) {
          mbar_expect_tx(k_full + 8 * s, C::K128);
          tma_load_3d(saddr(b), &tmK, k_full + 8 * s, 0, w.h, krow + kb * BKV);
        }
        if (C::TAIL) {
          load_tail<false>(b + C::K128, 0, Kp + w.h * DH + 64, ldkv, krow + kb * BKV, kv_rows, lane);
          tell_tails<1>(g + 1, told, k_full, KS, lane);
        }
      }
      // (the next unit's Q waits for this one's last S, which waits for these)
      if (C::TAIL) tell_tails<0>(g, told, k_full, KS, lane);
    }
    if (uc == 0) pdl_wait();  // (no kernel ends before its predecessor has)
  } else if (warp == 1 || warp == 3) {
    // ------------------------------------------- S = Q K^T and O += P V of a stream
    // S runs up to two of the stream's blocks ahead (two buffers); a buffer
    // takes its next S once the P V of the P in it is done.  A block of a
    // unit with one tile is one stream's alone, which then frees its K and V
    // for both
    if (elect_one()) {
      const int x = warp >> 1;
      const uint64_t dq = sw128_desc(saddr(sQ)), dqt = sw32_kmajor_desc(saddr(sQ + C::Q128));
      const uint64_t dk = sw128_desc(saddr(sK)), dkt = sw32_kmajor_desc(saddr(sK + C::K128));
      const uint32_t bs = s_full + 16 * x, bp = p_ready + 16 * x, bd = pv_done + 16 * x;
      const uint32_t to = tmem + TM_O + TM_O_STEP * uint32_t(x);
      int g0 = 0, uc = 0, ns = 0, np = 0;  // blocks of earlier units; units; S, P V so far
      AttnUnit w;
      for (int u = u0; u < un.units; u += du, ++uc) {
        w.set(un, u);
        const int n = w.kb1 - w.kb0;
        const bool two = locate_group(rm, ai.n, D, un.rows, w.g).rows > BQ;
        const int i0 = two ? 0 : x, di = two ? 1 : 2;
        const uint64_t qo = two ? uint64_t(x * (C::Q_BYTES >> 4)) : 0;
        if (!mbar_sleep(q_full, uc & 1, abort_flag)) goto timeout;
        int is = i0;  // next block to compute S of
        for (int i = i0; i < n; i += di) {
          for (; is < n && is < i + 2 * di; is += di, ++ns) {
            const int g = g0 + is, s = g % KS, b = ns & 1;
            if (!mbar_sleep(k_full + 8 * s, (g / KS) & 1, abort_flag) ||
                !mbar_sleep(bd + 8 * b, ((ns >> 1) & 1) ^ 1, abort_flag))
              goto timeout;
            tc_fence_after();
            const uint64_t so = uint64_t(s * (C::K_STRIDE >> 4));
            const uint32_t sd = tmem + tm_s(x, b);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              umma_bf16(sd, dq + qo + 2 * kk, dk + so + 2 * kk, C::IDESC_S, kk > 0 ? 1u : 0u);
            if (C::TAIL) umma_bf16(sd, dqt + qo, dkt + so, C::IDESC_S, 1u);
            umma_commit(bs + 8 * b);
            umma_commit(k_empty + 8 * s);
            if (!two) umma_commit(k_empty + 8 * s);
            if (is + di >= n) umma_commit(q_empty);  // the unit's last S of this stream
          }
          const int g = g0 + i, s = g % VS, b = np & 1;
          // O of the previous unit has been read
          if (i == i0 && !mbar_sleep(o_free, (uc & 1) ^ 1, abort_flag)) goto timeout;
          if (!mbar_sleep(v_full + 8 * s, (g / VS) & 1, abort_flag) ||
              !mbar_sleep(bp + 8 * b, (np >> 1) & 1, abort_flag))
            goto timeout;
          ++np;
          tc_fence_after();
          // keys past the last valid one are left out in steps of 16 (their
          // values may belong to something else)
          const int valid = Nk - (w.kb0 + i) * BKV;
          const uint64_t vd = sw128_mnmajor_desc_lbo(
              saddr(sV) + uint32_t(C::v_main(s)),
              C::TAIL ? uint32_t(C::v_tails(s) - C::v_main(s)) : uint32_t(C::K128));
          const uint32_t tp = tmem + tm_s(x, b);
#pragma unroll
          for (int kk = 0; kk < BKV / 16; ++kk)
            if (kk == 0 || 16 * kk < valid)
              umma_bf16_ta(to, tp + 8 * kk, vd + 128 * kk, C::IDESC_PV,
                           (i > i0 || kk > 0) ? 1u : 0u);
          umma_commit(bd + 8 * b);
          umma_commit(v_empty + 8 * s);
          if (!two) umma_commit(v_empty + 8 * s);
        }
        if (i0 >= n) {
          // no block in this unit: o_full counts each stream once a unit, so
          // this one is told only when the unit before has been read
          umma_commit(q_empty);
          if (!mbar_sleep(o_free, (uc & 1) ^ 1, abort_flag)) goto timeout;
        }
        umma_commit(o_full);
        g0 += n;
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ V
    const bool leader = elect_one();
    int g = 0, told = 0;
    AttnUnit w;
    for (int u = u0; u < un.units; u += du) {
      w.set(un, u);
      const int vrow = ai.vrow[locate_group(rm, ai.n, D, un.rows, w.g).item];
      for (int kb = w.kb0; kb < w.kb1; ++kb, ++g) {
        const int s = g % VS;
        if (!mbar_sleep_warp(v_empty + 8 * s, ((g / VS) & 1) ^ 1, abort_flag)) goto timeout;
        if (g == 0) pdl_wait();
        if (leader) {
          mbar_expect_tx(v_full + 8 * s, C::K128);
          tma_load_3d(saddr(sV + C::v_main(s)), &tmV, v_full + 8 * s, 0, w.h, vrow + kb * BKV);
        }
        if (C::TAIL) {
          load_tail<true>(sV + C::v_tails(s & ~3), 2 * (s & 3), Vp + w.h * DH + 64, ldkv, vrow + kb * BKV, kv_rows, lane);
          tell_tails<1>(g + 1, told, v_full, VS, lane);
        }
      }
    }
    if (C::TAIL) tell_tails<0>(g, told, v_full, VS, lane);
  } else {
    // ------------------------------------------------------------ softmax
    const int sp = warp & 3, x = (warp - 4) >> 2, row = sp * 32 + lane;
    const uint32_t lane_off = uint32_t(sp * 32) << 16;
    const uint32_t to = tmem + TM_O + TM_O_STEP * uint32_t(x) + lane_off;
    int cnt = 0, uc = 0;  // blocks of this stream, units so far
    uint32_t met = 0;
    // one arrival per warp
    auto arrive = [&](uint32_t bar) {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    };
    // all eight softmax warps (a bounded wait, like every other)
    auto join = [&]() {
      arrive(meet);
      const bool ok = mbar_sleep_warp(meet, met, abort_flag);
      met ^= 1;
      return ok;
    };
    AttnUnit w;
    for (int u = u0; u < un.units; u += du, ++uc) {
      w.set(un, u);
      const int n = w.kb1 - w.kb0;
      const TileLoc tl = locate_group(rm, ai.n, D, un.rows, w.g);
      const bool two = tl.rows > BQ;
      if (uc == 0) pdl_wait();  // (before any global write)
      float m = -INFINITY, l = 0.f;
      float cap_s[8];  // scaled scores of the captured key columns
#pragma unroll
      for (int q = 0; q < 8; ++q) cap_s[q] = -INFINITY;
      for (int i = two ? 0 : x; i < n; i += two ? 1 : 2, ++cnt) {
        const int b = cnt & 1;
        const uint32_t ts = tmem + tm_s(x, b) + lane_off;
        const int key0 = (w.kb0 + i) * BKV, valid = Nk - key0;
        if (!mbar_sleep_warp(s_full + 8 * (2 * x + b), (cnt >> 1) & 1, abort_flag)) goto timeout;
        tc_fence_after();
        // p = 2^(s * scale - m) against a reference m (scaled base-2 units;
        // scale = log2 e / sqrt(dh)), the max of the stream's first block.
        // The result does not depend on the reference as long as nothing
        // overflows, so later blocks take no max: only when a block's sum is
        // past 2^64 (warp-uniform: the TMEM accesses are warp-wide) is the
        // reference raised and the block, still in its buffer, done again
        uint32_t r[BKV];
        float bl, alpha = 1.f;
        // (a row whose scores were all -inf so far has no reference yet)
        bool take_max = __any_sync(0xffffffffu, m == -INFINITY);
        for (;;) {
#pragma unroll
          for (int c = 0; c < BKV / 16; ++c) tmem_ld16_nowait(ts + 16u * c, r + 16 * c);
          if (CAP) {  // (warp-uniform) the captured columns that fall in this block
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (q < cap.n && cap.id[q] >= key0 && cap.id[q] < key0 + BKV)
                cap_s[q] = __uint_as_float(tmem_ld1_nowait(ts + uint32_t(cap.id[q] - key0)));
          }
          tmem_wait_ld();
          if (valid < BKV) {  // the last, partial key block (warp-uniform)
#pragma unroll
            for (int c = 0; c < BKV; ++c)
              if (c >= valid) r[c] = __float_as_uint(-INFINITY);
          }
          if (take_max) {
            float f8[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) f8[q] = __uint_as_float(r[q]);
#pragma unroll
            for (int c = 8; c < BKV; ++c) f8[c & 7] = fmaxf(f8[c & 7], __uint_as_float(r[c]));
            const float mx = fmaxf(fmaxf(fmaxf(f8[0], f8[1]), fmaxf(f8[2], f8[3])),
                                   fmaxf(fmaxf(f8[4], f8[5]), fmaxf(f8[6], f8[7]))) *
                             scale_log2;
            const float mn = fmaxf(m, mx);
            alpha = m == -INFINITY ? 0.f : ex2_ftz(m - mn);
            m = mn;
          }
          const float mr = finite_max(m);
          const uint64_t sc2 = f32x2(scale_log2, scale_log2), nm2 = f32x2(-mr, -mr);
          uint64_t sum2[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) sum2[q] = f32x2(0.f, 0.f);
          // software-pipelined by hand (the asm statements keep their order):
          // the scaling runs PIPE columns ahead of the exponentials and the
          // sums and packing PIPE columns behind, so that a single warp keeps
          // the special-function unit busy
          constexpr int PIPE = 16;
#pragma unroll
          for (int c = -PIPE; c < BKV + PIPE; c += 2) {
            if (c + PIPE < BKV) scale_pair(r[c + PIPE], r[c + PIPE + 1], sc2, nm2);
            if (c >= 0 && c < BKV) {
              exp_in_place(r[c]);
              exp_in_place(r[c + 1]);
            }
            if (c >= PIPE) {
              const int d = c - PIPE;
              sum_pair(sum2[(d >> 1) & 3], r[d], r[d + 1]);
              r[d >> 1] = pack_pair(r[d], r[d + 1]);
            }
          }
          float s0, s1, s2, s3, s4, s5, s6, s7;
          unpack_f32x2(sum2[0], s0, s1);
          unpack_f32x2(sum2[1], s2, s3);
          unpack_f32x2(sum2[2], s4, s5);
          unpack_f32x2(sum2[3], s6, s7);
          bl = ((s0 + s1) + (s2 + s3)) + ((s4 + s5) + (s6 + s7));
          if (!__any_sync(0xffffffffu, bl > RAISE_SUM) || take_max) break;
          take_max = true;
        }
        if (CAP) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (q < cap.n && cap.id[q] >= key0 && cap.id[q] < key0 + BKV) cap_s[q] *= scale_log2;
        }
        if (take_max && i != (two ? 0 : x)) {
          // O to the raised reference, once P V of the stream's previous block
          // has completed
          l *= alpha;
          if (!mbar_sleep_warp(pv_done + 8 * (2 * x + ((cnt - 1) & 1)), ((cnt - 1) >> 1) & 1,
                               abort_flag))
            goto timeout;
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < C::DHP / 16; ++c) {
            uint32_t o16[16];
            tmem_ld16_nowait(to + 16u * c, o16);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) o16[e] = __float_as_uint(__uint_as_float(o16[e]) * alpha);
            tmem_st16(to + 16u * c, o16);
          }
        }
        l += bl;
        // P row (80 keys as 40 bf16 pairs) over S: the A operand of P V
#pragma unroll
        for (int c = 0; c < BKV / 32; ++c) tmem_st16(ts + 16u * c, r + 16 * c);
        if (BKV % 32) tmem_st8(ts + uint32_t(BKV / 32 * 16), r + BKV / 32 * 16);
        tmem_wait_st();
        tc_fence_before();
        arrive(p_ready + 8 * (2 * x + b));
      }
      // ---- end of the unit.  Two tiles: a thread has its row's whole O.
      // One tile: the two streams' rows are merged, stream 0's thread taking
      // a row's first columns, stream 1's the rest
      float M = m, L = l, w0 = 1.f, w1 = 0.f;
      if (!two) {
        s_ml[uc & 1][x][row] = make_float2(m, l);
        if (!join()) goto timeout;
        const float2 ml = s_ml[uc & 1][x ^ 1][row];
        // (a stream without a block has m = -inf, l = 0 and no O)
        M = finite_max(fmaxf(m, ml.x));
        const float wm = ex2_ftz(m - M), wo = ex2_ftz(ml.x - M);
        L = l * wm + ml.y * wo;
        w0 = x ? wo : wm;
        w1 = x ? wm : wo;
      }
      if (!mbar_sleep_warp(o_full, uc & 1, abort_flag)) goto timeout;
      tc_fence_after();
      const int trow = (two ? x * BQ : 0) + row;  // row within the group
      const bool live = trow < tl.rows;
      bf16* orow = O + size_t(tl.row0 + trow) * ldo + w.h * DH;
      const float inv = L > 0.f ? 1.f / L : 0.f;
      constexpr int H0 = C::TAIL ? 40 : 32;  // columns of the first half; the second has 32
      const uint32_t tb = tmem + TM_O + lane_off + (two ? TM_O_STEP * uint32_t(x) : 0u);
      const bool shared = w.share >= 0;
      const size_t slot = (size_t(max(w.share, 0)) * 2 + (two ? x : 0)) * (BQ * PART_STRIDE);
      const int hf0 = two ? 0 : x, hf1 = two ? 2 : x + 1;
      for (int hf = hf0; hf < hf1; ++hf) {
        const int col0 = hf ? H0 : 0, ncol = hf ? DH - H0 : H0;
#pragma unroll
        for (int c = 0; c < H0; c += 8) {
          if (c >= ncol) break;
          uint32_t a[8], b[8];
          float o[8];
          tmem_ld8_nowait(tb + uint32_t(col0 + c), a);
          if (!two && n > 1) tmem_ld8_nowait(tb + TM_O_STEP + uint32_t(col0 + c), b);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            o[e] = __uint_as_float(a[e]) * w0;
            if (!two && n > 1) o[e] = fmaf(__uint_as_float(b[e]), w1, o[e]);
          }
          if (shared) {  // a share of the pair's keys: its planes to the workspace
            float4* mine = reinterpret_cast<float4*>(part + slot) + ((col0 + c) / 4) * BQ + row;
            __stcg(mine, make_float4(o[0], o[1], o[2], o[3]));
            __stcg(mine + BQ, make_float4(o[4], o[5], o[6], o[7]));
          } else if (live) {
            *reinterpret_cast<uint4*>(orow + col0 + c) =
                make_uint4(pack_bf16x2(o[0] * inv, o[1] * inv), pack_bf16x2(o[2] * inv, o[3] * inv),
                           pack_bf16x2(o[4] * inv, o[5] * inv), pack_bf16x2(o[6] * inv, o[7] * inv));
          }
        }
      }
      tc_fence_before();
      arrive(o_free);
      if (CAP && live) {  // the localisation scores of the listed keys (one share)
        const int tok = rm.tok ? __ldg(rm.tok + tl.row0 + trow) : tl.row0 + trow;
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < cap.n && (two || ((cap.id[q] / BKV) & 1) == x))  // this stream's block held it
            atomicAdd(cap.out + size_t(tok) * cap.ldo + cap.id[q],
                      cap.w * ex2_ftz(cap_s[q] - M) * inv);
      }
      if (shared) {
        // the last of the pair's units merges them all
        if (two || x == 0)
          __stcg(reinterpret_cast<float2*>(part + slot + DH * BQ) + row, make_float2(M, L));
        __threadfence();
        if (!join()) goto timeout;
        if (threadIdx.x == 128) {
          unsigned* tk = ticket + (w.pair - un.whole);
          const unsigned t = atomicAdd(tk, 1u);
          s_last = t == unsigned(un.split) - 1u;
          if (s_last) *tk = 0u;  // for the next launch
          __threadfence();
        }
        if (!join()) goto timeout;
        if (!s_last) continue;
        const float* base = part + (size_t(w.pair - un.whole) * un.split * 2 + (two ? x : 0)) *
                                       (BQ * PART_STRIDE);
        auto piece = [&](int q) { return base + size_t(q) * (2 * BQ * PART_STRIDE); };
        float Mt = -INFINITY;
#pragma unroll 4
        for (int q = 0; q < un.split; ++q)
          Mt = fmaxf(Mt, __ldcg(reinterpret_cast<const float2*>(piece(q) + DH * BQ) + row).x);
        Mt = finite_max(Mt);
        for (int hf = hf0; hf < hf1; ++hf) {
          // a half row's columns of two shares in flight at a time
          const int col0 = hf ? H0 : 0, ncol = hf ? DH - H0 : H0;
          float o[H0], Lt = 0.f;
#pragma unroll
          for (int c = 0; c < H0; ++c) o[c] = 0.f;
#pragma unroll 2
          for (int q = 0; q < un.split; ++q) {
            const float2 mq = __ldcg(reinterpret_cast<const float2*>(piece(q) + DH * BQ) + row);
            const float4* b = reinterpret_cast<const float4*>(piece(q)) + (col0 / 4) * BQ + row;
            float4 v[H0 / 4];
#pragma unroll
            for (int c4 = 0; c4 < H0 / 4; ++c4)
              if (4 * c4 < ncol) v[c4] = __ldcg(b + c4 * BQ);
            const float wq = ex2_ftz(mq.x - Mt);
            Lt += wq * mq.y;
#pragma unroll
            for (int c4 = 0; c4 < H0 / 4; ++c4)
              if (4 * c4 < ncol) {
                o[4 * c4] = fmaf(wq, v[c4].x, o[4 * c4]);
                o[4 * c4 + 1] = fmaf(wq, v[c4].y, o[4 * c4 + 1]);
                o[4 * c4 + 2] = fmaf(wq, v[c4].z, o[4 * c4 + 2]);
                o[4 * c4 + 3] = fmaf(wq, v[c4].w, o[4 * c4 + 3]);
              }
          }
          const float inv_t = Lt > 0.f ? 1.f / Lt : 0.f;
#pragma unroll
          for (int c = 0; c < H0; c += 8)
            if (c < ncol && live)
              *reinterpret_cast<uint4*>(orow + col0 + c) = make_uint4(
                  pack_bf16x2(o[c] * inv_t, o[c + 1] * inv_t),
                  pack_bf16x2(o[c + 2] * inv_t, o[c + 3] * inv_t),
                  pack_bf16x2(o[c + 4] * inv_t, o[c + 5] * inv_t),
                  pack_bf16x2(o[c + 6] * inv_t, o[c + 7] * inv_t));
        }
      }
    }
  }
  goto done;
timeout:
  *abort_flag = 1;
  atomicOr(err, DEVERR_TIMEOUT);
done:
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ------------------------------------------------- short keys (text cross-attention)
// All Nk <= 128 keys of a (query tile, head) in one pass, one CTA per pair:
// S = Q K^T (M = 128, N = 128) in TMEM, an exact softmax per row (no running
// max, no rescaling), P (bf16) written over S, O = P V (N = DHP, 8 MMAs of 16
// keys, P read from TMEM as the A operand), O normalised and stored.  The
// text cross-attention of a block has 120 keys: two dependent blocks of the
// general kernel.
constexpr int XK = 128;  // keys per pass
template <int DH>
struct XCfg {
  using C = ACfg<DH>;
  static constexpr int K128 = XK * 128, K32 = C::TAIL ? XK * 32 : 0;
  static constexpr int V_ATOM = XK * 128;  // one MN-major SW128 atom of 64 head-dim columns
  static constexpr int V_BYTES = C::TAIL ? 2 * V_ATOM : V_ATOM;
  static constexpr int BYTES = C::Q_BYTES + K128 + K32 + V_BYTES;
  // rounded up so that at most two CTAs share an SM (2 x 256 TMEM columns)
  static constexpr size_t SMEM = 100 * 1024;
  static_assert(size_t(BYTES) + 1024 + 64 <= SMEM, "cross-attention tiles exceed the request");
  static constexpr uint32_t IDESC_S = (1u << 4) | (1u << 7) | (1u << 10) |
                                      (uint32_t(XK >> 3) << 17) | (uint32_t(BQ >> 4) << 24);
};

template <int DH, bool CAP>
__global__ void __launch_bounds__(128, 2)
xattn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmQt,
                const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmKt,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ AttnItems ai,
                int Nk, bf16* __restrict__ O, int ldo, int heads, RowMap rm, float scale_log2,
                unsigned* err, const __grid_constant__ AttnCapture cap) {
  using C = ACfg<DH>;
  using X = XCfg<DH>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* sQ = smem;
  uint8_t* sK = sQ + C::Q_BYTES;
  uint8_t* sV = sK + X::K128 + X::K32;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + X::V_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t load_bar = saddr(bars), mma_bar = saddr(bars + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(load_bar, 1);
    mbar_init(mma_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmQ)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmK)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmV)) : "memory");
  }
  if (warp == 0) tmem_alloc(saddr(tmem_slot), 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tS = tmem_base, tO = tmem_base + XK;  // P is written over S

  pdl_wait();
  pdl_trigger();
  const int D = live_count(rm.count, rm.bound, err);
  const int qtiles = query_tiles(rm, ai.n, D);
  const int qt = int(blockIdx.x) / heads, h = int(blockIdx.x) - (int(blockIdx.x) / heads) * heads;
  bool ok = qt < qtiles;
  TileLoc tl{0, 0, 0};
  if (ok) tl = locate_tile(rm, ai.n, D, qt);
  const int row = warp * 32 + lane;
  const uint32_t lane_off = uint32_t(warp * 32) << 16;
  if (ok && threadIdx.x == 0) {
    // ---- loads: Q (128 rows of the tile), K and V (128 keys of the item)
    const int krow = ai.krow[tl.item], vrow = ai.vrow[tl.item];
    mbar_expect_tx(load_bar, X::BYTES);
    tma_load_3d(saddr(sQ), &tmQ, load_bar, 0, h, tl.row0);
    if (C::TAIL) tma_load_3d(saddr(sQ + C::Q128), &tmQt, load_bar, 64, h, tl.row0);
    tma_load_3d(saddr(sK), &tmK, load_bar, 0, h, krow);
    if (C::TAIL) tma_load_3d(saddr(sK + X::K128), &tmKt, load_bar, 64, h, krow);
    tma_load_3d(saddr(sV), &tmV, load_bar, 0, h, vrow);
    if (C::TAIL) tma_load_3d(saddr(sV + X::V_ATOM), &tmV, load_bar, 64, h, vrow);
    // ---- S = Q K^T over the 80 (72 + zero) head dims
    if (mbar_sleep(load_bar, 0, abort_flag)) {
      tc_fence_after();
      const uint64_t dq = sw128_desc(saddr(sQ)), dk = sw128_desc(saddr(sK));
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        umma_bf16(tS, dq + 2 * kk, dk + 2 * kk, X::IDESC_S, kk > 0 ? 1u : 0u);
      if (C::TAIL)
        umma_bf16(tS, sw32_kmajor_desc(saddr(sQ + C::Q128)), sw32_kmajor_desc(saddr(sK + X::K128)),
                  X::IDESC_S, 1u);
      umma_commit(mma_bar);
    } else {
      *abort_flag = 1;
    }
  }
  // ---- exact softmax of this thread's row
  if (ok) ok = mbar_sleep_warp(mma_bar, 0, abort_flag);
  float l = 0.f;
  if (ok) {
    tc_fence_after();
    uint32_t r[XK];
#pragma unroll
    for (int i = 0; i < XK / 16; ++i) tmem_ld16_nowait(tS + lane_off + 16u * i, r + 16 * i);
    tmem_wait_ld();
#pragma unroll
    for (int c = 0; c < XK; ++c)
      if (c >= Nk) r[c] = __float_as_uint(-INFINITY);
    float mx8[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) mx8[q] = __uint_as_float(r[q]);
#pragma unroll
    for (int c = 8; c < XK; ++c) mx8[c & 7] = fmaxf(mx8[c & 7], __uint_as_float(r[c]));
    const float m = fmaxf(fmaxf(fmaxf(mx8[0], mx8[1]), fmaxf(mx8[2], mx8[3])),
                          fmaxf(fmaxf(mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]))) * scale_log2;
    const uint64_t sc2 = f32x2(scale_log2, scale_log2), nm2 = f32x2(-m, -m);
    uint64_t sum2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) sum2[q] = f32x2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < XK; c += 2) {
      float a, b;
      unpack_f32x2(fma_f32x2(f32x2(__uint_as_float(r[c]), __uint_as_float(r[c + 1])), sc2, nm2),
                   a, b);
      a = ex2_ftz(a);
      b = ex2_ftz(b);
      r[c] = __float_as_uint(a);
      r[c + 1] = __float_as_uint(b);
      sum2[(c >> 1) & 3] = add_f32x2(sum2[(c >> 1) & 3], f32x2(a, b));
    }
    float s0, s1, s2, s3, s4, s5, s6, s7;
    unpack_f32x2(sum2[0], s0, s1);
    unpack_f32x2(sum2[1], s2, s3);
    unpack_f32x2(sum2[2], s4, s5);
    unpack_f32x2(sum2[3], s6, s7);
    l = ((s0 + s1) + (s2 + s3)) + ((s4 + s5) + (s6 + s7));
    if (CAP && cap.n && row < tl.rows) {  // the localisation scores of the listed keys
      const int qrow = tl.row0 + row;
      const int tok = rm.tok ? __ldg(rm.tok + qrow) : qrow;
      const float inv_l = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < cap.n) {
          float pq = 0.f;
#pragma unroll
          for (int c = 0; c < XK; ++c)
            if (c == cap.id[q]) pq = __uint_as_float(r[c]);
          atomicAdd(cap.out + size_t(tok) * cap.ldo + cap.id[q], cap.w * pq * inv_l);
        }
    }
    // P (bf16 pairs) over the first 64 columns of S: the A operand of P V
#pragma unroll
    for (int h2 = 0; h2 < XK / 32; ++h2) {
      uint32_t w[16];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        w[c] = pack_bf16x2(__uint_as_float(r[32 * h2 + 2 * c]),
                           __uint_as_float(r[32 * h2 + 2 * c + 1]));
      tmem_st16(tS + lane_off + 16u * h2, w);
    }
    tmem_wait_st();
  }
  tc_fence_before();
  __syncthreads();  // every row's P is in TMEM
  if (ok && threadIdx.x == 0) {
    tc_fence_after();
    const uint64_t dv = C::TAIL ? sw128_mnmajor_desc_lbo(saddr(sV), X::V_ATOM)
                                : sw128_mnmajor_desc(saddr(sV));
#pragma unroll
    for (int kk = 0; kk < XK / 16; ++kk)
      umma_bf16_ta(tO, tS + 8 * kk, dv + 128 * kk, C::IDESC_PV, kk > 0 ? 1u : 0u);
    umma_commit(mma_bar);
  }
  if (ok) ok = mbar_sleep_warp(mma_bar, 1, abort_flag);
  if (ok) {
    tc_fence_after();
    uint32_t o[C::DHP];
#pragma unroll
    for (int i = 0; i < C::DHP / 16; ++i) tmem_ld16_nowait(tO + lane_off + 16u * i, o + 16 * i);
    tmem_wait_ld();
    if (row < tl.rows) {
      const float inv = l > 0.f ? 1.f / l : 0.f;
      uint4* dst = reinterpret_cast<uint4*>(O + size_t(tl.row0 + row) * ldo + h * DH);
#pragma unroll
      for (int c8 = 0; c8 < DH / 8; ++c8) {
        uint4 w;
        w.x = pack_bf16x2(__uint_as_float(o[8 * c8 + 0]) * inv, __uint_as_float(o[8 * c8 + 1]) * inv);
        w.y = pack_bf16x2(__uint_as_float(o[8 * c8 + 2]) * inv, __uint_as_float(o[8 * c8 + 3]) * inv);
        w.z = pack_bf16x2(__uint_as_float(o[8 * c8 + 4]) * inv, __uint_as_float(o[8 * c8 + 5]) * inv);
        w.w = pack_bf16x2(__uint_as_float(o[8 * c8 + 6]) * inv, __uint_as_float(o[8 * c8 + 7]) * inv);
        dst[c8] = w;
      }
    }
  }
  if (qt < qtiles && (!ok || *abort_flag)) {
    if (threadIdx.x == 0) atomicOr(err, DEVERR_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 256);
  }
}

// ------------------------------------ cross-attention with the query folded in
// The text keys and W_xq are fixed for a turn, so the query projection can be
// folded into the keys once per turn: q'_h K_h^T = (xb W_xq,h^T + b_h) K_h^T =
// xb G_h^T + kb_h, G_h = K_h W_xq,h, kb_h = K_h b_h (a reassociation of the
// same products).  The cross-query GEMM then disappears from the block.

// A unit is one (query tile, head): S = xb_tile G_h^T accumulated over d in
// 64-column k-blocks (TMA ring, M = 128, N = 128), then the softmax of
// (S + kb) / sqrt(dh) per row, P over S in TMEM, O = P V, O / l stored.  One
// warp loads the keys and V (from before the dependency wait on), one the
// rows, one issues the MMAs with the next stage tested ahead.  Persistent, at
// most one CTA an SM: the units go round robin, S alternates between two
// regions, and the P V of a unit is issued two thirds into the next unit's
// S, so the softmax and the stores run under the MMAs.  (A CTA a unit of the
// row bound, the ones past the live rows leaving at once, kept the next
// kernel from starting until all had come and gone: 1024 px step 2640 us, 2594
// now; eight 512 px sessions 3694 us, 3505 now.)
constexpr int XF_STAGES = 6;
constexpr int XF_THREADS = 224;  // rows, MMA, 4 softmax warps, keys and V
template <int DH>
struct XFCfg {
  using C = ACfg<DH>;
  static constexpr int STAGE_A = BQ * 128, STAGE_G = XK * 128;
  static constexpr int STAGE = STAGE_A + STAGE_G;
  static constexpr int V_ATOM = XK * 128;
  static constexpr int V_BYTES = C::TAIL ? 2 * V_ATOM : V_ATOM;
  static constexpr size_t SMEM = size_t(XF_STAGES) * STAGE + V_BYTES + 1024 + 256;
  static constexpr uint32_t IDESC_S = (1u << 4) | (1u << 7) | (1u << 10) |
                                      (uint32_t(XK >> 3) << 17) | (uint32_t(BQ >> 4) << 24);
};

template <int DH, bool CAP>
__global__ void __launch_bounds__(XF_THREADS, 1)
xfused_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmG,
                 const __grid_constant__ CUtensorMap tmV, const float* __restrict__ kb,
                 const __grid_constant__ XqItems xi, int Nk, int d, bf16* __restrict__ O,
                 int ldo, int heads, RowMap rm, float scale_log2, unsigned* err,
                 const __grid_constant__ AttnCapture cap) {
  using C = ACfg<DH>;
  using X = XFCfg<DH>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* sV = smem + XF_STAGES * X::STAGE;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sV + X::V_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * XF_STAGES + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t full0 = saddr(bars), empty0 = saddr(bars + XF_STAGES);
  const uint32_t v_full = saddr(bars + 2 * XF_STAGES), p_ready = v_full + 8, o_full = v_full + 16,
                 s_full = v_full + 24;  // two, by S region
  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < XF_STAGES; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    mbar_init(v_full, 1);
    mbar_init(p_ready, 128);
    mbar_init(o_full, 1);
    mbar_init(s_full, 1);
    mbar_init(s_full + 8, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Before the programmatic-dependency wait this kernel reads only what was
  // written two or more launches earlier (every kernel of the library waits
  // for its predecessor before letting its successor start): the live row
  // count and the turn's folded keys, key biases and text values.  Only the
  // bf16 rows of x come from the predecessor.
  const int D = live_count(rm.count, rm.bound, err);
  const int units = query_tiles(rm, xi.n, D) * heads;
  // CTAs past the live units leave before taking tensor memory (but no kernel
  // ends before its predecessor has)
  if (int(blockIdx.x) >= units) {
    pdl_wait();
    return;
  }
  if (warp == 1) tmem_alloc(saddr(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // S0 | S1 | O; P is written over its S
  const uint32_t tO = tmem_base + 2 * XK;
  const int nkb = d / 64, at_pv = 2 * nkb / 3;
  bool ok = true;
  if (warp == 0) {
    // ------------------------------------------------------------ TMA: rows
    if (elect_one()) {
      int st = 0;
      uint32_t ph = 1;
      bool waited = false;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int row0 = locate_tile(rm, xi.n, D, u / heads).row0;
        for (int k = 0; k < nkb; ++k) {
          if (!mbar_wait(empty0 + 8 * st, ph, abort_flag)) {
            ok = false;
            break;
          }
          // (the keys may arrive before this expectation: the phase still
          // needs this arrival)
          mbar_expect_tx(full0 + 8 * st, X::STAGE);
          if (!waited) {  // (everything up to the first load runs beside the predecessor's end)
            waited = true;
            pdl_wait();
            pdl_trigger();
          }
          tma_load_3d(saddr(smem + st * X::STAGE), &tmA, full0 + 8 * st, 0, k, row0);
          if (++st == XF_STAGES) { st = 0; ph ^= 1; }
        }
      }
      if (!ok) *abort_flag = 1;
    }
  } else if (warp == 6) {
    // ------------------------------------------------------------ TMA: keys, V
    if (elect_one()) {
      int st = 0;
      uint32_t ph = 1;
      int n = 0;  // units so far
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++n) {
        const int qt = u / heads, h = u - qt * heads, item = locate_tile(rm, xi.n, D, qt).item;
        const int grow = xi.grow[item] + h * XK;
        // V once the ring is filled, or (the one buffer) at the end of a
        // later unit, when the previous P V has read it
        const int at_v = n ? nkb - 1 : (nkb < XF_STAGES ? nkb : XF_STAGES) - 1;
        for (int k = 0; k < nkb; ++k) {
          if (!mbar_wait(empty0 + 8 * st, ph, abort_flag)) {
            ok = false;
            break;
          }
          tma_load_3d(saddr(smem + st * X::STAGE + X::STAGE_A), &tmG, full0 + 8 * st, 0, k, grow);
          if (++st == XF_STAGES) { st = 0; ph ^= 1; }
          if (k == at_v) {
            if (n && !mbar_wait(o_full, (n - 1) & 1, abort_flag)) {
              ok = false;
              break;
            }
            mbar_expect_tx(v_full, X::V_BYTES);
            tma_load_3d(saddr(sV), &tmV, v_full, 0, h, xi.vrow[item]);
            if (C::TAIL) tma_load_3d(saddr(sV + X::V_ATOM), &tmV, v_full, 64, h, xi.vrow[item]);
          }
        }
      }
      if (!ok) *abort_flag = 1;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA
    if (elect_one()) {
      const uint64_t da = sw128_desc(saddr(smem)), dg = sw128_desc(saddr(smem + X::STAGE_A));
      const uint64_t dv = C::TAIL ? sw128_mnmajor_desc_lbo(saddr(sV), X::V_ATOM)
                                  : sw128_mnmajor_desc(saddr(sV));
      // P V of the n-th unit once every row's P is in TMEM (and the previous
      // O read) and V has landed
      auto pv = [&](int n) -> bool {
        if (!mbar_wait(p_ready, n & 1, abort_flag) || !mbar_wait(v_full, n & 1, abort_flag))
          return false;
        tc_fence_after();
        const uint32_t tP = tmem_base + uint32_t(n & 1) * XK;
#pragma unroll
        for (int kk = 0; kk < XK / 16; ++kk)
          umma_bf16_ta(tO, tP + 8 * kk, dv + 128 * kk, C::IDESC_PV, kk > 0 ? 1u : 0u);
        umma_commit(o_full);
        return true;
      };
      bool ready = false;
      int st = 0, n = 0;
      uint32_t ph = 0;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++n) {
        // the S region: its last reader was the P V of two units ago
        if (n >= 2 && !mbar_wait(o_full, n & 1, abort_flag)) ok = false;
        const uint32_t tS = tmem_base + uint32_t(n & 1) * XK;
        for (int k = 0; k < nkb && ok; ++k) {
          if (!ready && !mbar_wait(full0 + 8 * st, ph, abort_flag)) {
            ok = false;
            break;
          }
          const uint64_t so = uint64_t((st * X::STAGE) >> 4);
          const uint32_t eb = empty0 + 8 * st;
          if (++st == XF_STAGES) { st = 0; ph ^= 1; }
          ready = mbar_test(full0 + 8 * st, ph);  // (beside this stage's MMAs)
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            umma_bf16(tS, da + so + 2 * kk, dg + so + 2 * kk, X::IDESC_S,
                      (k > 0 || kk > 0) ? 1u : 0u);
          umma_commit(eb);
          if (n && k == at_pv) ok = pv(n - 1);
        }
        if (ok) umma_commit(s_full + 8 * (n & 1));
      }
      if (!(ok && pv(n - 1))) *abort_flag = 1;
    }
  } else {
    // ------------------------------------------------------------ softmax
    const int sp = warp & 3;
    const int row = sp * 32 + lane;
    const uint32_t lane_off = uint32_t(sp * 32) << 16;
    pdl_wait();  // (before any global write: the predecessor reads O's buffer)
    int n = 0;
    for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++n) {
      const int qt = u / heads, h = u - qt * heads;
      const TileLoc tl = locate_tile(rm, xi.n, D, qt);
      const float4* b4 =
          reinterpret_cast<const float4*>(kb + size_t(xi.grow[tl.item]) + size_t(h) * XK);
      const uint32_t tS = tmem_base + uint32_t(n & 1) * XK + lane_off;
      // (the key biases are fetched into L1 beside the product)
      const float4 warm = __ldg(b4 + lane);
      asm volatile("" ::"f"(warm.x));
      ok = mbar_sleep_warp(s_full + 8 * (n & 1), (n >> 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint32_t r[XK];
#pragma unroll
      for (int i = 0; i < XK / 16; ++i) tmem_ld16_nowait(tS + 16u * i, r + 16 * i);
      tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < XK / 4; ++c) {
        const float4 t = __ldg(b4 + c);
        const float a[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          r[4 * c + e] = 4 * c + e < Nk
                             ? __float_as_uint(__uint_as_float(r[4 * c + e]) + a[e])
                             : __float_as_uint(-INFINITY);
      }
      float mx8[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) mx8[q] = __uint_as_float(r[q]);
#pragma unroll
      for (int c = 8; c < XK; ++c) mx8[c & 7] = fmaxf(mx8[c & 7], __uint_as_float(r[c]));
      const float m = fmaxf(fmaxf(fmaxf(mx8[0], mx8[1]), fmaxf(mx8[2], mx8[3])),
                            fmaxf(fmaxf(mx8[4], mx8[5]), fmaxf(mx8[6], mx8[7]))) * scale_log2;
      const uint64_t sc2 = f32x2(scale_log2, scale_log2), nm2 = f32x2(-m, -m);
      uint64_t sum2[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) sum2[q] = f32x2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < XK; c += 2) {
        float a, b;
        unpack_f32x2(fma_f32x2(f32x2(__uint_as_float(r[c]), __uint_as_float(r[c + 1])), sc2, nm2),
                     a, b);
        a = ex2_ftz(a);
        b = ex2_ftz(b);
        r[c] = __float_as_uint(a);
        r[c + 1] = __float_as_uint(b);
        sum2[(c >> 1) & 3] = add_f32x2(sum2[(c >> 1) & 3], f32x2(a, b));
      }
      float s0, s1, s2, s3, s4, s5, s6, s7;
      unpack_f32x2(sum2[0], s0, s1);
      unpack_f32x2(sum2[1], s2, s3);
      unpack_f32x2(sum2[2], s4, s5);
      unpack_f32x2(sum2[3], s6, s7);
      const float l = ((s0 + s1) + (s2 + s3)) + ((s4 + s5) + (s6 + s7));
      if (CAP && cap.n && row < tl.rows) {  // the localisation scores of the listed keys
        const int qrow = tl.row0 + row;
        const int tok = rm.tok ? __ldg(rm.tok + qrow) : qrow;
        const float inv_l = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < cap.n) {
            float pq = 0.f;
#pragma unroll
            for (int c = 0; c < XK; ++c)
              if (c == cap.id[q]) pq = __uint_as_float(r[c]);
            atomicAdd(cap.out + size_t(tok) * cap.ldo + cap.id[q], cap.w * pq * inv_l);
          }
      }
#pragma unroll
      for (int h2 = 0; h2 < XK / 32; ++h2) {
        uint32_t w[16];
#pragma unroll
        for (int c = 0; c < 16; ++c)
          w[c] = pack_bf16x2(__uint_as_float(r[32 * h2 + 2 * c]),
                             __uint_as_float(r[32 * h2 + 2 * c + 1]));
        tmem_st16(tS + 16u * h2, w);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(p_ready);
      ok = mbar_sleep_warp(o_full, n & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint32_t o[C::DHP];
#pragma unroll
      for (int i = 0; i < C::DHP / 16; ++i) tmem_ld16_nowait(tO + lane_off + 16u * i, o + 16 * i);
      tmem_wait_ld();
      if (row < tl.rows) {
        const float inv = l > 0.f ? 1.f / l : 0.f;
        uint4* dst = reinterpret_cast<uint4*>(O + size_t(tl.row0 + row) * ldo + h * DH);
#pragma unroll
        for (int c8 = 0; c8 < DH / 8; ++c8) {
          uint4 w;
          w.x = pack_bf16x2(__uint_as_float(o[8 * c8 + 0]) * inv, __uint_as_float(o[8 * c8 + 1]) * inv);
          w.y = pack_bf16x2(__uint_as_float(o[8 * c8 + 2]) * inv, __uint_as_float(o[8 * c8 + 3]) * inv);
          w.z = pack_bf16x2(__uint_as_float(o[8 * c8 + 4]) * inv, __uint_as_float(o[8 * c8 + 5]) * inv);
          w.w = pack_bf16x2(__uint_as_float(o[8 * c8 + 6]) * inv, __uint_as_float(o[8 * c8 + 7]) * inv);
          dst[c8] = w;
        }
      }
    }
    if (!ok) *abort_flag = 1;
  }
  if ((!ok || *abort_flag) && threadIdx.x == 64) atomicOr(err, DEVERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ------------------------------------------------------------------- host
struct HeadMapKey {
  const void* p;
  int rows, ld, heads, dh;
  bool operator==(const HeadMapKey& o) const {
    return p == o.p && rows == o.rows && ld == o.ld && heads == o.heads && dh == o.dh;
  }
};
struct HeadMapHash {
  size_t operator()(const HeadMapKey& k) const {
    return std::hash<const void*>()(k.p) ^ (size_t(k.rows) * 1000003u) ^ (size_t(k.ld) * 7919u) ^
           (size_t(k.heads) * 131u) ^ size_t(k.dh);
  }
};

// (head_dim, head, row) view of a row-major [rows][ld] bf16 matrix whose row
// holds `heads` blocks of dh; boxes of box_w x 1 x box_rows (box_w 64 with the
// 128-byte swizzle, 16 with the 32-byte swizzle); reads outside the view
// (head_dim >= dh, row >= rows) return zero.
cudaError_t head_map(const bf16* p, int rows, int ld, int heads, int dh, int box_w, int box_rows,
                     CUtensorMap* out) {
  static std::mutex mu;
  static std::unordered_map<HeadMapKey, CUtensorMap, HeadMapHash> cache;
  HeadMapKey key{p, rows, ld, heads, (dh * 1024 + box_rows) * 256 + box_w};
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end()) {
      *out = it->second;
      return cudaSuccess;
    }
  }
  auto fn = tma_encode_fn();
  if (!fn) return cudaErrorNotSupported;
  cuuint64_t dims[3] = {cuuint64_t(dh), cuuint64_t(heads), cuuint64_t(rows)};
  cuuint64_t strides[2] = {cuuint64_t(dh) * sizeof(bf16), cuuint64_t(ld) * sizeof(bf16)};
  cuuint32_t box[3] = {cuuint32_t(box_w), 1, cuuint32_t(box_rows)};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(p), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  box_w == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(mu);
  if (cache.size() > 4096) cache.clear();
  cache.emplace(key, *out);
  return cudaSuccess;
}

int device_sms_attn() {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!sms[dev]) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaFuncSetAttribute(attn_tc_kernel<72, false>, smem, int(ACfg<72>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(attn_tc_kernel<72, true>, smem, int(ACfg<72>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(attn_tc_kernel<64, false>, smem, int(ACfg<64>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(attn_tc_kernel<64, true>, smem, int(ACfg<64>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(xattn_tc_kernel<72, false>, smem, int(XCfg<72>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(xattn_tc_kernel<72, true>, smem, int(XCfg<72>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(xattn_tc_kernel<64, false>, smem, int(XCfg<64>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(xattn_tc_kernel<64, true>, smem, int(XCfg<64>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(xfused_tc_kernel<72, false>, smem, int(XFCfg<72>::SMEM)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(xfused_tc_kernel<72, true>, smem, int(XFCfg<72>::SMEM)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(xfused_tc_kernel<64, false>, smem, int(XFCfg<64>::SMEM)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(xfused_tc_kernel<64, true>, smem, int(XFCfg<64>::SMEM)) !=
            cudaSuccess)
      return 0;
    sms[dev] = v;
  }
  return sms[dev];
}

// The plans of a (heads, keys) shape, cached.  With a capture every key sits in
// one unit, of one tile or two by the same estimate (always two, as for launches
// past the table, left 1024 tokens on 64 SMs: the scores of 28 blocks from 200
// text tokens and 8 of them listed 582 us, 474 now).
PlanTable plan_table(int heads, int Nk, int grid, bool capture) {
  static std::mutex mu;
  static std::unordered_map<uint64_t, PlanTable> cache;
  const uint64_t key = (uint64_t(capture ? 1 : 0) << 63) | (uint64_t(heads) << 40) |
                       (uint64_t(grid) << 32) | uint64_t(unsigned(Nk));
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  PlanTable t{};
  for (int tiles = 1; tiles <= 2; ++tiles)
    for (int i = 0; i < PLAN_TABLE; ++i) {
      int cost;
      t.split[tiles - 1][i] = uint8_t(pick_split((i + 1) * heads, (Nk + BKV - 1) / BKV, grid,
                                                 tiles, capture ? 1 : MAX_SPLIT, &cost));
      t.cost[tiles - 1][i] = uint16_t(cost < 65535 ? cost : 65535);
    }
  if (cache.size() > 1024) cache.clear();
  cache.emplace(key, t);
  return t;
}

}  // namespace

size_t attention_split_floats() {
  const int sms = device_sms_attn();
  return size_t(SLOTS_PER_SM) * (sms > 0 ? sms : 160) * BQ * PART_STRIDE;
}
size_t attention_tickets() {
  const int sms = device_sms_attn();
  return size_t(SLOTS_PER_SM) * (sms > 0 ? sms : 160);
}

cudaError_t launch_attention(const bf16* Q, int ldq, const bf16* K, const bf16* V, int ldkv,
                             int kv_rows, const AttnItems& ai, int Nk, bf16* O, int ldo, int heads,
                             int dh, const RowMap& rm, unsigned* err, const AttnScratch& as,
                             cudaStream_t st, const AttnCapture* capture) {
  if (rm.bound <= 0) return cudaSuccess;
  if (dh != 72 && dh != 64) return cudaErrorInvalidValue;
  if (ai.n < 1 || ai.n > MAX_ITEMS || (ai.n > 1 && !rm.meta)) return cudaErrorInvalidValue;
  for (int i = 0; i < ai.n; ++i)
    if (ai.krow[i] < 0 || ai.vrow[i] < 0 || ai.krow[i] > kv_rows - Nk || ai.vrow[i] > kv_rows - Nk)
      return cudaErrorInvalidValue;
  const int sms = device_sms_attn();
  if (!sms) return cudaErrorInvalidDevice;
  // 64-wide 128B-swizzled maps, and a 16-wide 32B-swizzled one for Q's tail
  CUtensorMap tq, tqt, tk, tv;
  RC_TRY(head_map(Q, rm.bound, ldq, heads, dh, 64, BQ, &tq));
  RC_TRY(head_map(K, kv_rows, ldkv, heads, dh, 64, BKV, &tk));
  RC_TRY(head_map(V, kv_rows, ldkv, heads, dh, 64, BKV, &tv));
  RC_TRY(head_map(Q, rm.bound, ldq, heads, dh, 16, BQ, &tqt));
  const float scale_log2 = float(1.4426950408889634 / sqrt(double(dh)));
  AttnCapture cap{};
  if (capture && capture->n > 0) {
    if (capture->n > 8 || !capture->out || Nk > CAPTURE_KEYS) return cudaErrorInvalidValue;
    for (int q = 0; q < capture->n; ++q)
      if (capture->id[q] < 0 || capture->id[q] >= Nk || capture->id[q] >= capture->ldo)
        return cudaErrorInvalidValue;
    cap = *capture;
  }
  if (Nk <= XK) {
    // short key sets (the text cross-attention): one pass per (query tile,
    // head), a CTA each; tiles beyond the live count exit at once
    CUtensorMap xk, xkt, xv;
    RC_TRY(head_map(K, kv_rows, ldkv, heads, dh, 64, XK, &xk));
    RC_TRY(head_map(K, kv_rows, ldkv, heads, dh, 16, XK, &xkt));
    RC_TRY(head_map(V, kv_rows, ldkv, heads, dh, 64, XK, &xv));
    const long long xgrid = ((long long)(rm.bound + BQ - 1) / BQ + ai.n - 1) * heads;
    if (xgrid >= (1ll << 31)) return cudaErrorInvalidValue;
    auto xk_fn = dh == 72 ? (cap.n ? xattn_tc_kernel<72, true> : xattn_tc_kernel<72, false>)
                          : (cap.n ? xattn_tc_kernel<64, true> : xattn_tc_kernel<64, false>);
    RC_TRY(launch_k(xk_fn, dim3(unsigned(xgrid)), dim3(128),
                    dh == 72 ? XCfg<72>::SMEM : XCfg<64>::SMEM, st, tq, tqt, xk, xkt, xv, ai, Nk,
                    O, ldo, heads, rm, scale_log2, err, cap));
    count_launches(1);
    return cudaSuccess;
  }
  const PlanTable plan = plan_table(heads, Nk, sms, cap.n > 0);
  if (as.part_floats < size_t(SLOTS_PER_SM) * sms * BQ * PART_STRIDE || !as.ticket)
    return cudaErrorInvalidValue;
  {
    const unsigned long long tiles = (rm.bound + BQ - 1) / BQ + ai.n - 1;
    if (tiles * heads * MAX_SPLIT >= (1ull << 31)) return cudaErrorInvalidValue;
  }
  auto fn = dh == 72 ? (cap.n ? attn_tc_kernel<72, true> : attn_tc_kernel<72, false>)
                     : (cap.n ? attn_tc_kernel<64, true> : attn_tc_kernel<64, false>);
  RC_TRY(launch_k(fn, dim3(sms), dim3(THREADS), dh == 72 ? ACfg<72>::SMEM : ACfg<64>::SMEM, st, tq,
                  tqt, tk, tv, K, V, ldkv, kv_rows, ai, plan, Nk, O, ldo, heads, rm, scale_log2,
                  err, as.part, as.ticket, cap));
  count_launches(1);
  return cudaSuccess;
}

cudaError_t launch_xattn_fused(const bf16* xb, int ldx, const bf16* G, const float* kb, int g_rows,
                               const bf16* V, int ldv, int v_rows, const XqItems& xi, int Nk,
                               bf16* O, int ldo, int heads, int dh, const RowMap& rm,
                               unsigned* err, cudaStream_t st, const AttnCapture* capture) {
  if (rm.bound <= 0) return cudaSuccess;
  const int d = heads * dh;
  if ((dh != 72 && dh != 64) || Nk < 1 || Nk > XK || d % 64 || ldx % 8 || ldv % 8)
    return cudaErrorInvalidValue;
  if (xi.n < 1 || xi.n > MAX_ITEMS || (xi.n > 1 && !rm.meta)) return cudaErrorInvalidValue;
  for (int i = 0; i < xi.n; ++i)
    if (xi.grow[i] < 0 || xi.grow[i] + heads * XK > g_rows || xi.vrow[i] < 0 ||
        xi.vrow[i] > v_rows - Nk)
      return cudaErrorInvalidValue;
  const int sms = device_sms_attn();
  if (!sms) return cudaErrorInvalidDevice;
  AttnCapture cap{};
  if (capture && capture->n > 0) {
    if (capture->n > 8 || !capture->out) return cudaErrorInvalidValue;
    for (int q = 0; q < capture->n; ++q)
      if (capture->id[q] < 0 || capture->id[q] >= Nk || capture->id[q] >= capture->ldo)
        return cudaErrorInvalidValue;
    cap = *capture;
  }
  // xb and G as (64 columns, column block, row) views, V as the head view
  CUtensorMap ta, tg, tv;
  RC_TRY(head_map(xb, rm.bound, ldx, d / 64, 64, 64, BQ, &ta));
  RC_TRY(head_map(G, g_rows, d, d / 64, 64, 64, XK, &tg));
  RC_TRY(head_map(V, v_rows, ldv, heads, dh, 64, XK, &tv));
  const float scale_log2 = float(1.4426950408889634 / sqrt(double(dh)));
  const long long grid = ((long long)(rm.bound + BQ - 1) / BQ + xi.n - 1) * heads;
  if (grid >= (1ll << 31)) return cudaErrorInvalidValue;
  auto fn = dh == 72 ? (cap.n ? xfused_tc_kernel<72, true> : xfused_tc_kernel<72, false>)
                     : (cap.n ? xfused_tc_kernel<64, true> : xfused_tc_kernel<64, false>);
  RC_TRY(launch_k(fn, dim3(unsigned(grid < sms ? grid : sms)), dim3(XF_THREADS),
                  dh == 72 ? XFCfg<72>::SMEM : XFCfg<64>::SMEM, st, ta, tg, tv, kb, xi, Nk, d, O, ldo, heads, rm, scale_log2, err, cap));
  count_launches(1);
  return cudaSuccess;
}

}  // namespace rc
