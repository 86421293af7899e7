// Tensor-core GEMM of the region-sparse block on sm_103a: tcgen05.mma with
// TMEM accumulators, operands staged by TMA (128-byte swizzle), persistent
// warp-specialised CTAs, and the block's epilogues fused (bias, tanh-GELU,
// gated residual, QKV with K/V rows written straight into the cache rows of
// the dirty tokens -- Section 3.4, Kernel Fusing -- and the merged hidden
// state written into the cache's H rows).
//
// C[M][n] = A[M][k] W[n][k]^T, A and W K-major bf16, f32 accumulation.
// M (the dirty-token count) may live on the device: every CTA reads it and
// derives the same schedule.  The tile is 128 x BN with BN in {64, 128, 192,
// 256}, chosen per launch from M by a cost model (the main loop streams
// (128 + BN) x 64 bf16 operands per k-block from L2 at a fixed per-SM rate,
// and only the last tile's epilogue is exposed), so that ragged row counts
// still spread over the GPU.  Whole tiles go out in waves.  The gated
// residual (x += gate (C + b)) is written as vector reductions into x, so
// pieces of a tile simply add up: for it a small last wave is instead cut
// into equal k-block ranges (stream-K).  Its casting variant (x += ..., then
// xb = bf16(x), read-modify-write) and the other epilogues see whole tiles.
//
// CTA = 15 warps: warp 0 issues TMA loads (A), warp 14 those of W, warp 1
// owns TMEM and issues the MMAs (one elected thread), warps 2..13 drain the
// accumulator (one TMEM lane = one output row per thread; three warps per
// TMEM lane quarter take every third 32-column chunk).  The epilogue is
// latency-bound (a CTA holds one tile at small row counts), so its width is
// worth more than a deeper ring, and every epilogue is its own kernel: a
// launch runs its code once per CTA, so instructions that it does not need
// cost fetches (at 831 rows warps of the one-kernel form waited 2-4 cycles
// per instruction for the next one).  Against that form, with two issuing
// threads, schedules chosen on the device, bf16 tiles re-staged through shared
// memory and W waiting for the previous kernel: a 28-block step at 831 rows
// 2980 -> 2718 us, at 1512 rows of 8 items 4312 -> 3950, two blocks at 132 /
// 4096 rows 177 -> 158 / 661 -> 604 us.  Two TMEM accumulators of up to 256 columns let the epilogue
// of one tile overlap the main loop of the next.
#include <cuda.h>

#include <mutex>
#include <unordered_map>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"
#include "tma_host.h"

namespace rc {

namespace {

using namespace rc::tc;

constexpr int BM = 128, BK = 64;
// TMA warp (A, or A and W for CTA pairs), MMA warp, 12 epilogue warps, a
// second TMA warp that loads W for unpaired CTAs (each TMA request takes long
// enough to issue that one thread issuing both operands bounds the main
// loop, and W does not wait for the previous kernel)
constexpr int THREADS = 480;
constexpr int W_WARP = 14;
constexpr int STAGE_A = BM * BK * 2;   // bytes
constexpr int MIN_KB_PER_CTA = 4;
// most equal parts of the k range of one tile (codes BN / 64 + 8 S are bytes)
constexpr int MAX_SPLIT = 8;
constexpr int STAGING_WARP = 32 * 128;  // epilogue staging: 32 rows of 128 B per warp
constexpr int STAGING_BYTES = 12 * STAGING_WARP;

// Operand ring: stages of A (16 KB) + B (BN x 128 B), as many as fit.
constexpr int RING_BYTES = 168 * 1024;
constexpr int MAX_STAGES = 9;
constexpr int TMEM_COLS = 512;  // two accumulators of up to 256 columns
// per-tile column vectors of the epilogue: bias and gate of up to 256 columns
constexpr int VEC_BYTES = 2 * 256 * 4;
constexpr size_t SMEM_BYTES = size_t(RING_BYTES) + STAGING_BYTES + VEC_BYTES + 1024 + 256;
// Instruction descriptor, kind::f16: D f32, A and B bf16, both K-major,
// M >> 4 at bit 24; N >> 3 goes to bit 17 at run time.
constexpr uint32_t IDESC_BASE = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(BM >> 4) << 24);
// the same for the M = 256 MMA of a CTA pair
constexpr uint32_t IDESC_PAIR = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(256 >> 4) << 24);
// The tile width and split chosen on the host for 1 .. BN_TABLE row tiles
// (BN / 64 + 8 S), passed by value; larger row counts take the last entry's
// width in whole tiles.
constexpr int BN_TABLE = 128;
struct BnTable {
  uint8_t w64[BN_TABLE];
};
// W tensor maps by box height 32, 64, 96, 128, 192, 256 rows (a CTA of a
// pair loads half a tile width)
constexpr int N_BMAPS = 6;
struct BMaps {
  CUtensorMap m[N_BMAPS];
};
__host__ __device__ constexpr int bmap_index(int rows) {
  return rows == 32 ? 0 : rows == 64 ? 1 : rows == 96 ? 2 : rows == 128 ? 3 : rows == 192 ? 4 : 5;
}

// ---------------------------------------------------------------- epilogue
__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c),
               "f"(d)
               : "memory");
}
// 32 bytes (one sector) per thread.
__device__ __forceinline__ void st_v8(void* p, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void ld_v8(const float* p, float* v) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
                 "=f"(v[6]), "=f"(v[7])
               : "l"(p)
               : "memory");
}

// The mode a schedule is planned for: a gated residual held to whole tiles
// plans like any other 4-byte epilogue whose tiles are not split.
__host__ __device__ inline int sched_mode(const GemmEpi& ep) {
  return ep.mode == EPI_GATE_RES && ep.whole_tiles ? int(EPI_F32) : ep.mode;
}

template <int MODE>
__device__ __forceinline__ bool gated(const GemmEpi& ep) {
  return (MODE == EPI_GATE_RES || MODE == EPI_GATE_RES_CAST) && ep.gate_tab;
}

// The column vectors of one tile (columns col0 .. col0 + BN - 1) in shared
// memory, written by the 384 epilogue threads before the accumulator is
// ready: sv[c] = bias (0 when absent, or when this piece of a split gated
// residual does not start at k = 0: the update is a sum over pieces, so the
// bias goes with one of them), sv[256 + c] = gate (table part, plus the
// item's timestep part when the launch has one item).
template <int MODE>
__device__ __forceinline__ void stage_vectors(const GemmEpi& ep, int col0, int BN, bool with_bias,
                                              float* sv, int etid) {
  const float* tb0 = (ep.its.n == 1 && ep.gate_off >= 0) ? ep.its.tb[0] : nullptr;
  if (etid < BN) {
    const int col = col0 + etid;
    sv[etid] = (ep.bias && with_bias) ? __ldg(ep.bias + col) : 0.f;
    if (gated<MODE>(ep))
      sv[256 + etid] = __ldg(ep.gate_tab + col) + (tb0 ? __ldg(tb0 + ep.gate_off + col) : 0.f);
  }
}

// Epilogue values of columns c0 .. c0+31 of one output row (cl = c0 within
// the tile): bias, tanh-GELU, gate, from the staged vectors (plus the row's
// item gate when the launch has several items; with one item it is folded
// into the staged gate).
template <int MODE>
__device__ __forceinline__ void epilogue_values(const GemmEpi& ep, int c0, int cl, int item,
                                                float* v, const float* sv) {
  const float4* b4 = reinterpret_cast<const float4*>(sv + cl);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 b = b4[i];
    v[4 * i] += b.x; v[4 * i + 1] += b.y; v[4 * i + 2] += b.z; v[4 * i + 3] += b.w;
  }
  if (MODE == EPI_GELU_BF16) {
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = gelu_tanh(v[i]);
  } else if (gated<MODE>(ep)) {
    const float* tb = ep.gate_off >= 0 && ep.its.n > 1 ? ep.its.tb[item] : nullptr;
    const float4* g4 = reinterpret_cast<const float4*>(sv + 256 + cl);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float4 g = g4[i];
      if (tb) {
        const float4 e = __ldg(reinterpret_cast<const float4*>(tb + ep.gate_off + c0) + i);
        g.x += e.x; g.y += e.y; g.z += e.z; g.w += e.w;
      }
      v[4 * i] *= g.x; v[4 * i + 1] *= g.y; v[4 * i + 2] *= g.z; v[4 * i + 3] *= g.w;
    }
  }
}

// Named barrier of the 12 epilogue warps.
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 384;" ::: "memory"); }

// Columns c0 .. c0 + 31 of output row r as bf16: two sectors of the row's own
// (the lanes' rows may lie anywhere: QKV scatters K and V to the cache rows
// of the rows' tokens).
__device__ __forceinline__ void store_bf16(bf16* p, const float* v) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t u[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) u[i] = pack_bf16x2(v[16 * h + 2 * i], v[16 * h + 2 * i + 1]);
    st_v8(p + 16 * h, u);
  }
}

// One warp's 32 x 32 chunk (lane = row, v = its 32 columns) in f32: stored to
// dst, or (ADD, the gated residual) as vector reductions into it.  Each lane
// parks its row in the warp's 4 KB staging area, then eight lanes take one
// whole 128-byte row piece: rows are n apart, so a lane's own 16-byte pieces
// would be half sectors of 32 different rows (a caller's 4096 x 4608 x 1152
// into f32 45.5 us that way, 34.3 this way; 9000 x 8192 x 128 147 and 72).
// (bf16 outputs go straight from registers, see store_bf16: their pieces of 32
// bytes are whole sectors.)
// Staging is XOR-swizzled in 16-byte units so that both the row-per-lane
// writes and the piece-per-lane-group reads are free of bank conflicts.
template <bool ADD>
__device__ __forceinline__ void write_chunk(uint8_t* stg, int lane, const float* v, float* dst) {
  const uint32_t s0 = saddr(stg);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(
                     s0 + lane * 128 + 16 * (j ^ (lane & 7))),
                 "f"(v[4 * j]), "f"(v[4 * j + 1]), "f"(v[4 * j + 2]), "f"(v[4 * j + 3])
                 : "memory");
  __syncwarp();
  const int j = lane & 7;
#pragma unroll
  for (int pass = 0; pass < 8; ++pass) {
    const int row = pass * 4 + (lane >> 3);
    float* d = reinterpret_cast<float*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst), row));
    const float4 x = *reinterpret_cast<const float4*>(stg + row * 128 + 16 * (j ^ (row & 7)));
    if (!d) continue;
    if (ADD) red_add_v4(d + 4 * j, x.x, x.y, x.z, x.w);
    else reinterpret_cast<float4*>(d)[j] = x;
  }
  __syncwarp();  // the staging area is rewritten by the next chunk
}

// One warp's 32 x 32 chunk: lane = output row r (token tok, item item), v its
// accumulator columns c0 .. c0 + 31 (cl within the tile).  x0: the row's
// residual columns, loaded before the accumulator was ready (CAST).
template <int MODE>
__device__ __forceinline__ void finish_chunk(const GemmEpi& ep, int r, int M, int tok, int item,
                                             int c0, int cl, float* v, const float* sv,
                                             uint8_t* stg, int lane, const float* x0) {
  epilogue_values<MODE>(ep, c0, cl, item, v, sv);
  if (MODE == EPI_GATE_RES) {
    write_chunk<true>(stg, lane, v, r < M ? ep.xf + size_t(r) * ep.ld_xf + c0 : nullptr);
    return;
  }
  if (MODE == EPI_F32) {  // (a caller's matrix: 16-byte aligned)
    write_chunk<false>(stg, lane, v, r < M ? ep.out_f + size_t(r) * ep.ld_out + c0 : nullptr);
    return;
  }
  if (r >= M) return;
  if (MODE == EPI_GATE_RES_CAST) {
    float* x = ep.xf + size_t(r) * ep.ld_xf + c0;
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] += x0[i];
#pragma unroll
    for (int q = 0; q < 4; ++q) st_v8(x + 8 * q, reinterpret_cast<const uint32_t*>(v + 8 * q));
    store_bf16(ep.out_bf + size_t(r) * ep.ld_out + c0, v);
  } else if (MODE == EPI_QKV) {
    const int part = c0 / ep.dsplit, cc = c0 - part * ep.dsplit;
    if (part == 0) {
      store_bf16(ep.out_bf + size_t(r) * ep.ld_out + cc, v);
    } else if (tok < 0 || tok >= ep.n_tokens || item < 0 || item >= ep.its.n) {
      atomicOr(ep.err, DEVERR_INDEX);
    } else {
      store_bf16(ep.its.slice[item] + (part == 1 ? ep.k_off : ep.v_off) +
                     size_t(tok) * ep.dsplit + cc,
                 v);
    }
  } else {
    store_bf16(ep.out_bf + size_t(r) * ep.ld_out + c0, v);
  }
}

// Schedule, identical in every thread.  Tiles t = nn * mt + m (m fastest, so
// CTAs in flight share weight tiles in L2) go whole to CTA t mod G in waves.
// The (non-casting) gated residual, whose pieces add up, may instead cut
// its k range: into S equal parts when tiles x S fit one wave (one piece per
// CTA), or, when the last wave would leave more than half the CTAs idle, by
// laying the R remainder tiles end to end by k-block and cutting them into
// Gr equal ranges (stream-K, at least MIN_KB_PER_CTA k-blocks each).
//
// Pairs (two CTAs of a cluster sharing one M = 256 MMA): the same, with a
// "tile" of two row tiles (2p, 2p + 1) and G the number of pairs.
struct Sched {
  int BN, stages, mt, nt, tiles, kbt, G, whole, Gr, S;
  bool pair;
  // every CTA holds at most one work item: its epilogue starts only once
  // all of its MMAs have read the ring, so the ring may run on over the
  // epilogue staging buffers that follow it
  bool alias;
  long long Wr;
  // S > 0: split-S (requires tiles * S <= grid); S == 0: waves (+ stream-K)
  __host__ __device__ void plan(int M, int bn, int n, int k, int grid, bool additive, int s,
                                bool pr) {
    BN = bn;
    pair = pr;
    stages = stages_for(bn, pr);
    const int mt_rows = (M + BM - 1) / BM;
    mt = pair ? (mt_rows + 1) / 2 : mt_rows;
    nt = n / BN;
    tiles = mt * nt;
    kbt = k / BK;
    G = pair ? grid / 2 : grid;
    S = s;
    alias = false;
    if (S > 0) {
      whole = 0;
      Wr = 0;
      Gr = 0;
      alias = true;  // one piece per CTA
      stages = stages_for(bn, pr, true);
      return;
    }
    const int R = tiles % G;
    const bool split = additive && R > 0 && 2 * R <= G && kbt >= 2 * MIN_KB_PER_CTA;
    whole = split ? tiles - R : tiles;
    Wr = split ? (long long)R * kbt : 0;
    long long g = Wr / MIN_KB_PER_CTA;
    if (g < 1) g = 1;
    Gr = split ? int(g < G ? g : G) : 0;
    alias = whole <= G && Gr == 0;
    stages = stages_for(bn, pr, alias);
  }
  // bytes of one stage in one CTA: A (128 x 64) and B (BN x 64, half of it
  // in each CTA of a pair)
  __host__ __device__ static int stage_bytes(int bn, bool pr) {
    return STAGE_A + (pr ? bn * BK : bn * BK * 2);
  }
  __host__ __device__ static int stages_for(int bn, bool pr, bool alias = false) {
    const int s = (RING_BYTES + (alias ? STAGING_BYTES : 0)) / stage_bytes(bn, pr);
    return s < MAX_STAGES ? s : MAX_STAGES;
  }
  // Estimated duration (SM cycles): k-blocks on the busiest CTA x per-k-block
  // time plus its exposed epilogues; a stream-K CTA holds two pieces.  Rates
  // measured on the five matrices of a 1152-wide block at 39 to 4096 rows:
  // single CTAs take 220 / 365 / 435 / 540 cycles a k-block at BN 64 / 128 /
  // 192 / 256, pairs 280 / 356 / 430 / 570 (operands at ~60 B/clk per SM, but
  // no less than the MMA issue time); an epilogue drains ~20 B/clk per SM
  // (15 where the output is reduced in place), and half of one shows on
  // every further wave.
  __host__ __device__ float cost(int out_bytes, bool additive) const {
    const float ckb =
        pair ? fmaxf(float(stage_bytes(BN, pair)) * (1.f / 60.f), 2.f * float(BN) + 25.f)
             : 125.f + 1.65f * float(BN);
    const float cep = float(BM * BN * out_bytes) * (additive ? 1.f / 15.f : 1.f / 20.f);
    if (S > 0) return float((kbt + S - 1) / S) * ckb + cep;
    const int waves = (whole + G - 1) / G;
    float c = float(waves) * (float(kbt) * ckb + 0.5f * cep) + (waves > 0 ? 0.5f * cep : 0.f);
    if (Gr > 0) c += float((Wr + Gr - 1) / Gr) * ckb + 2.f * cep;
    return c;
  }
  // Picks BN (n % BN == 0) and, for the additive gated residual, a split,
  // with the lowest estimate; ties go to wider tiles and fewer pieces.
  // Returns BN / 64 + 8 S.
  __host__ __device__ static int pick(int M, int n, int k, int grid, int mode, bool pr) {
    Sched s;
    const bool additive = mode == EPI_GATE_RES;
    const int out_bytes = mode == EPI_GATE_RES_CAST ? 10
                          : (mode == EPI_F32 || mode == EPI_GATE_RES) ? 4 : 2;
    const int cand[4] = {256, 192, 128, 64};
    float best = 3.4e38f;
    int code = 1;
    for (int i = 0; i < 4; ++i) {
      if (n % cand[i]) continue;
      for (int sp = 0; sp <= (additive ? MAX_SPLIT : 0); ++sp) {
        if (sp == 1) continue;
        s.plan(M, cand[i], n, k, grid, additive, sp, pr);
        if (sp > 0 && (s.tiles * sp > s.G || s.kbt < sp * MIN_KB_PER_CTA)) continue;
        const float c = s.cost(out_bytes, additive);
        if (c < best * 0.999f) {
          best = c;
          code = cand[i] / 64 + 8 * sp;
        }
      }
    }
    return code;
  }
  // table: the host's pick for 1 .. BN_TABLE row tiles
  __device__ void init(int M, int n, int k, int grid, int mode, const uint8_t* table, bool pr) {
    const int m_tiles = (M + BM - 1) / BM;
    const int code = int(table[m_tiles < 1 ? 0 : m_tiles <= BN_TABLE ? m_tiles - 1 : BN_TABLE - 1]);
    plan(M, 64 * (code & 7), n, k, grid, mode == EPI_GATE_RES,
         m_tiles <= BN_TABLE ? code >> 3 : 0, pr);
  }
  __device__ long long bound(int c) const { return Wr * c / Gr; }
};

// The segments (tile, k-blocks [kb0, kb1)) of one CTA, in order.
struct Segs {
  const Sched* sc;
  int t_next;
  long long cur, end;
  __device__ void init(const Sched& s, int c) {
    sc = &s;
    t_next = c;
    cur = c < s.Gr ? s.bound(c) : 0;
    end = c < s.Gr ? s.bound(c + 1) : 0;
    if (s.S > 0) {  // split-S: CTA c < tiles * S holds piece c / tiles of tile c % tiles
      cur = 0;
      end = c < s.tiles * s.S ? 1 : 0;
    }
  }
  __device__ bool next(int& t, int& kb0, int& kb1) {
    if (sc->S > 0) {
      if (cur >= end) return false;
      ++cur;
      const int p = t_next / sc->tiles;
      t = t_next - p * sc->tiles;
      kb0 = p * sc->kbt / sc->S;
      kb1 = (p + 1) * sc->kbt / sc->S;
      return true;
    }
    if (t_next < sc->whole) {
      t = t_next;
      t_next += sc->G;
      kb0 = 0;
      kb1 = sc->kbt;
      return true;
    }
    if (cur >= end) return false;
    const int tr = int(cur / sc->kbt);
    kb0 = int(cur - (long long)tr * sc->kbt);
    kb1 = int(min((long long)sc->kbt, kb0 + (end - cur)));
    cur += kb1 - kb0;
    t = sc->whole + tr;
    return true;
  }
};

// PAIR: launched in clusters of two CTAs that share every MMA (cta_group::2,
// M = 256): each CTA loads its own 128 rows of A and half of the W tile, and
// the even CTA's MMA thread multiplies the pair's operands into both CTAs'
// tensor memory.  Per k-block a CTA then holds (and pulls from L2)
// 16 KB + BN x 64 B instead of 16 KB + BN x 128 B, so the ring keeps more
// k-blocks in flight -- the main loop is bound by k-blocks in flight per SM
// over the load latency.
template <int MODE, bool PAIR>
__global__ void __launch_bounds__(THREADS, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ BMaps tmB,
               int Mbound, const int* __restrict__ dcount, int n, int k,
               const __grid_constant__ GemmEpi ep, const __grid_constant__ BnTable bt) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // 1024-aligned operand ring, epilogue staging, then barriers
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  // the staging buffers follow the ring; a CTA with one work item lets its
  // ring run on over them (see Sched::alias)
  uint8_t* sStg = smem + RING_BYTES;
  float* sVec = reinterpret_cast<float*>(sStg + STAGING_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sStg + STAGING_BYTES + VEC_BYTES);
  // bars: full[MAX_STAGES], empty[MAX_STAGES], tfull[2], tempty[2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_STAGES + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t full0 = saddr(bars), empty0 = saddr(bars + MAX_STAGES);
  const uint32_t tfull0 = saddr(bars + 2 * MAX_STAGES), tempty0 = saddr(bars + 2 * MAX_STAGES + 2);

  // rank 0 of a pair issues the MMAs; its barriers count the pair's loads
  // (full), and both CTAs' epilogue warps (tempty: one arrival per warp)
  const uint32_t rank = PAIR ? cluster_ctarank() : 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, PAIR ? 24 : 12);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (PAIR)
      tmem_alloc_pair(saddr(tmem_slot), TMEM_COLS);
    else
      tmem_alloc(saddr(tmem_slot), TMEM_COLS);
  }
  if (warp == 0 && elect_one())
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the peer's barriers are initialised before any of its loads, commits or
  // arrivals can reach them
  if (PAIR) cluster_sync();

  // everything above is private set-up.  The live row count was written two
  // or more launches earlier (a step's dirty count before its first block;
  // every kernel of the library waits for its predecessor before letting its
  // successor start), so it and the schedule come before the programmatic-
  // dependency wait; the operand rows and the residual are read after it, by
  // the warps that need them.  W is not the predecessor's either where the
  // caller says so (ep.early_w)
  const int M = live_count(dcount, Mbound, ep.err);
  Sched sc;
  sc.init(M, n, k, int(gridDim.x), sched_mode(ep), bt.w64, PAIR);
  const int BN = sc.BN, STAGES = sc.stages;
  const int STAGE = Sched::stage_bytes(BN, PAIR);
  // schedule position: the pair (its row tiles 2p + rank) or the CTA
  const int pos = PAIR ? int(blockIdx.x) >> 1 : int(blockIdx.x);

  if (warp == 0) {
    // ------------------------------------------------------- TMA producer
    if (elect_one()) {
      // W as one box of BN rows, or BN / 2 rows per CTA of a pair (maps for
      // the heights that divide n)
      const int brows = PAIR ? BN / 2 : BN;
      const CUtensorMap* tmW = &tmB.m[bmap_index(brows)];
      int stage = 0;
      uint32_t phase = 0;
      Segs sg;
      sg.init(sc, pos);
      int t, kb0, kb1;
      bool waited = false;
      while (sg.next(t, kb0, kb1)) {
        const int mq = t % sc.mt, nn = t / sc.mt;
        const int m = PAIR ? 2 * mq + int(rank) : mq;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag)) goto timeout;
          uint8_t* st = smem + stage * STAGE;
          // (for a pair both CTAs' bytes land on rank 0's barrier)
          if (rank == 0) mbar_expect_tx(full0 + 8 * stage, PAIR ? 2 * STAGE : STAGE);
          if (!waited) {  // (everything up to the first load runs beside the predecessor's end)
            waited = true;
            pdl_wait();
            pdl_trigger();
          }
          if (PAIR) {
            const uint32_t fb = mapa_shared(full0 + 8 * stage, 0);
            tma_load_2d_pair(saddr(st), &tmA, fb, kb * BK, m * BM);
            tma_load_2d_pair(saddr(st + STAGE_A), tmW, fb, kb * BK, nn * BN + int(rank) * brows);
          } else {
            // W comes from the W warp on the same barrier (which may see
            // its bytes before this expectation: the phase still needs this
            // arrival)
            tma_load_2d(saddr(st), &tmA, full0 + 8 * stage, kb * BK, m * BM);
          }
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (!waited) pdl_wait();  // (no kernel ends before its predecessor has)
    }
  } else if (warp == W_WARP) {
    // ------------------------------------------------------- TMA: W (unpaired)
    if (!PAIR && elect_one()) {
      const CUtensorMap* tmW = &tmB.m[bmap_index(BN)];
      if (!ep.early_w) pdl_wait();
      int stage = 0;
      uint32_t phase = 0;
      Segs sg;
      sg.init(sc, pos);
      int t, kb0, kb1;
      while (sg.next(t, kb0, kb1)) {
        const int nn = t / sc.mt;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag)) goto timeout;
          tma_load_2d(saddr(smem + stage * STAGE + STAGE_A), tmW, full0 + 8 * stage, kb * BK,
                      nn * BN);
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------- MMA issuer
    if (rank == 0 && elect_one()) {
      const uint32_t idesc = (PAIR ? IDESC_PAIR : IDESC_BASE) | (uint32_t(BN >> 3) << 17);
      const uint64_t da = sw128_desc(saddr(smem)), db = sw128_desc(saddr(smem + STAGE_A));
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ready = false;  // the current stage was seen full already
      Segs sg;
      sg.init(sc, pos);
      int t, kb0, kb1;
      while (sg.next(t, kb0, kb1)) {
        if (!mbar_wait(tempty0 + 8 * acc, acc_phase ^ 1, abort_flag)) goto timeout;
        tc_fence_after();
        const uint32_t dtm = tmem_base + uint32_t(acc * 256);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!ready && !mbar_wait(full0 + 8 * stage, phase, abort_flag)) goto timeout;
          // stage descriptors differ only in the start address field
          // (address >> 4; no carry out of its 14 bits below 256 KB)
          const uint64_t so = uint64_t((stage * STAGE) >> 4);
          const uint32_t eb = empty0 + 8 * stage;
          if (++stage == STAGES) { stage = 0; phase ^= 1; }
          // the next stage is tested before this one's MMAs are issued, so
          // that the test's latency (54 cycles) runs beside them
          ready = mbar_test(full0 + 8 * stage, phase);
          tc_fence_after();
          if (PAIR) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              umma_bf16_pair(dtm, da + so + 2 * kk, db + so + 2 * kk, idesc,
                             (kb > kb0 || kk > 0) ? 1u : 0u);
            umma_commit_pair(eb);  // frees the stage in both CTAs
          } else {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              umma_bf16(dtm, da + so + 2 * kk, db + so + 2 * kk, idesc,
                        (kb > kb0 || kk > 0) ? 1u : 0u);
            umma_commit(eb);
          }
        }
        if (PAIR)
          umma_commit_pair(tfull0 + 8 * acc);
        else
          umma_commit(tfull0 + 8 * acc);
        if (++acc == 2) { acc = 0; acc_phase ^= 1; }
      }
    }
  } else {
    // ------------------------------------------------------- epilogue (warps 2..13)
    const int sp = warp & 3;  // TMEM lane sub-partition this warp may access
    int acc = 0;
    uint32_t acc_phase = 0;
    Segs sg;
    sg.init(sc, pos);
    int t, kb0, kb1;
    // the accumulator is drained once every epilogue warp of the pair (or
    // CTA) has arrived on rank 0's barrier
    const uint32_t tempty_r0 = PAIR ? mapa_shared(tempty0, 0) : tempty0;
    // every epilogue warp passes the same number of epi_sync barriers, also
    // after a failed wait (it then skips the rest of the work), so that no
    // warp is ever left waiting at one
    bool ok = true;
    pdl_wait();
    while (sg.next(t, kb0, kb1)) {
      const int mq = t % sc.mt, nn = t / sc.mt;
      const int m = PAIR ? 2 * mq + int(rank) : mq;
      // everything that does not depend on the accumulator first, while the
      // main loop runs: the row's token / item, the tile's column vectors,
      // the first chunk's residual
      const int row = sp * 32 + lane;
      const int r = m * BM + row;
      int tok = 0, item = 0;
      if (r < M) {
        if (MODE == EPI_QKV) tok = ep.tok ? __ldg(ep.tok + r) : r;
        if (ep.item) item = __ldg(ep.item + r);
      }
      constexpr int XN = MODE == EPI_GATE_RES_CAST ? 32 : 1;
      float x0[XN];
      auto load_x = [&](int ch) {
        if (MODE == EPI_GATE_RES_CAST && r < M)
#pragma unroll
          for (int q = 0; q < XN / 8; ++q)
            ld_v8(ep.xf + size_t(r) * ep.ld_xf + nn * BN + ch * 32 + 8 * q, x0 + 8 * q);
      };
      const int ch0 = (warp - 2) >> 2;
      if (ch0 < BN / 32) load_x(ch0);
      epi_sync();  // the previous tile's readers of sVec are done
      stage_vectors<MODE>(ep, nn * BN, BN, kb0 == 0, sVec, int(threadIdx.x) - 64);
      epi_sync();
      if (ok && !mbar_sleep_warp(tfull0 + 8 * acc, acc_phase, abort_flag)) ok = false;
      if (ok) {
        tc_fence_after();
        const uint32_t tbase = tmem_base + uint32_t(acc * 256) + (uint32_t(sp * 32) << 16);
#pragma unroll 1
        for (int ch = ch0; ch < BN / 32; ch += 3) {
          float v[32];
          tmem_ld32(tbase + uint32_t(ch * 32), v);
          if (ch != ch0) load_x(ch);
          finish_chunk<MODE>(ep, r, M, tok, item, nn * BN + ch * 32, ch * 32, v, sVec,
                             sStg + (warp - 2) * STAGING_WARP, lane, x0);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR)
            mbar_arrive_cluster(tempty_r0 + 8 * acc);
          else
            mbar_arrive(tempty0 + 8 * acc);
        }
      }
      if (++acc == 2) { acc = 0; acc_phase ^= 1; }
    }
    if (!ok) goto timeout;
  }
  goto done;
timeout:
  *abort_flag = 1;
  atomicOr(ep.err, DEVERR_TIMEOUT);
done:
  tc_fence_before();
  __syncthreads();
  // no CTA leaves (or frees its tensor memory) while its peer may still
  // load, commit or arrive into it
  if (PAIR) cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if (PAIR)
      tmem_dealloc_pair(tmem_base, TMEM_COLS);
    else
      tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

using GemmKernel = decltype(&gemm_tc_kernel<EPI_F32, false>);
template <bool PAIR>
GemmKernel gemm_kernel(int mode) {
  switch (mode) {
    case EPI_F32: return gemm_tc_kernel<EPI_F32, PAIR>;
    case EPI_BIAS_BF16: return gemm_tc_kernel<EPI_BIAS_BF16, PAIR>;
    case EPI_GELU_BF16: return gemm_tc_kernel<EPI_GELU_BF16, PAIR>;
    case EPI_GATE_RES: return gemm_tc_kernel<EPI_GATE_RES, PAIR>;
    case EPI_QKV: return gemm_tc_kernel<EPI_QKV, PAIR>;
    default: return gemm_tc_kernel<EPI_GATE_RES_CAST, PAIR>;
  }
}
constexpr int GEMM_MODES = 6;

// ------------------------------------------------------------------- host
struct MapKey {
  const void* p;
  uint64_t rows, cols, ld;
  int box_rows;
  bool operator==(const MapKey& o) const {
    return p == o.p && rows == o.rows && cols == o.cols && ld == o.ld && box_rows == o.box_rows;
  }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    return std::hash<const void*>()(k.p) ^ (k.rows * 1000003ull) ^ (k.cols * 7919ull) ^
           (k.ld * 131ull) ^ size_t(k.box_rows);
  }
};

// 2-D bf16 row-major [rows][cols] (row stride ld elements), box BK x box_rows,
// 128-byte swizzle; out-of-range rows read as zero.
cudaError_t tensor_map(const bf16* p, int rows, int cols, int ld, int box_rows, CUtensorMap* out) {
  static std::mutex mu;
  static std::unordered_map<MapKey, CUtensorMap, MapKeyHash> cache;
  MapKey key{p, uint64_t(rows), uint64_t(cols), uint64_t(ld), box_rows};
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
  cuuint64_t dims[2] = {cuuint64_t(cols), cuuint64_t(rows)};
  cuuint64_t strides[1] = {cuuint64_t(ld) * sizeof(bf16)};
  cuuint32_t box[2] = {cuuint32_t(BK), cuuint32_t(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(p), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(mu);
  if (cache.size() > 4096) cache.clear();
  cache.emplace(key, *out);
  return cudaSuccess;
}

// Tile-width table of a GEMM shape, cached (the cost model runs up to 4 x 8
// plans per row-tile count).
BnTable bn_table(int n, int k, int grid, int mode, int mt_bound, bool pair) {
  static std::mutex mu;
  static std::unordered_map<uint64_t, BnTable> cache;
  const int mtb = mt_bound < BN_TABLE ? mt_bound : BN_TABLE;
  // bits: mode 0-2, pair 3, grid 4-11, mtb 12-19, k 20-41, n 42-63
  // (mode < 8, grid < 256, n, k < 2^22: checked by the launcher)
  const uint64_t full_key = uint64_t(mode & 7) | (uint64_t(pair ? 1 : 0) << 3) |
                            (uint64_t(grid & 255) << 4) | (uint64_t(mtb) << 12) |
                            (uint64_t(k & 0x3FFFFF) << 20) | (uint64_t(n) << 42);
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(full_key);
    if (it != cache.end()) return it->second;
  }
  BnTable bt{};
  for (int mt = 1; mt <= BN_TABLE; ++mt)
    bt.w64[mt - 1] =
        mt <= mtb ? uint8_t(Sched::pick(mt * BM, n, k, grid, mode, pair)) : bt.w64[mt - 2];
  std::lock_guard<std::mutex> lock(mu);
  if (cache.size() > 4096) cache.clear();
  cache.emplace(full_key, bt);
  return bt;
}

// Launch shape of the current device: CTA pairs (clusters of two, one CTA
// per SM) when every SM can hold one, else one CTA per SM unpaired.
// grid 0: no device.
struct GemmShape {
  int grid;
  bool pair;
};
constexpr int PAIR_MIN_ROWS = 2048;
int device_sms() {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!sms[dev] && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) !=
                       cudaSuccess)
    return 0;
  return sms[dev];
}
GemmShape device_shape() {
  static GemmShape shp[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return GemmShape{0, false};
  if (!shp[dev].grid) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        v >= 256)
      return GemmShape{0, false};
    for (int mode = 0; mode < GEMM_MODES; ++mode)
      if (cudaFuncSetAttribute(gemm_kernel<false>(mode), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(SMEM_BYTES)) != cudaSuccess ||
          cudaFuncSetAttribute(gemm_kernel<true>(mode), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               int(SMEM_BYTES)) != cudaSuccess)
        return GemmShape{0, false};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(v & ~1);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, gemm_kernel<true>(EPI_F32), &cfg) != cudaSuccess) {
      cudaGetLastError();
      nc = 0;
    }
    shp[dev] = nc > 0 && 2 * nc == (v & ~1) ? GemmShape{2 * nc, true} : GemmShape{v, false};
  }
  return shp[dev];
}

}  // namespace

cudaError_t launch_gemm(const bf16* A, int lda, const bf16* W, int Mbound, const int* dcount,
                        int n, int k, const GemmEpi& ep, cudaStream_t st) {
  if (Mbound <= 0) return cudaSuccess;
  if (n % 64 || k % BK || n >= (1 << 22) || k >= (1 << 22) || ep.mode < 0 ||
      ep.mode >= GEMM_MODES)
    return cudaErrorInvalidValue;
  const GemmShape shp = device_shape();
  if (!shp.grid) return cudaErrorInvalidDevice;
  cudaError_t e;
  CUtensorMap ta;
  BMaps tb;
  if ((e = tensor_map(A, Mbound, k, lda, BM, &ta)) != cudaSuccess) return e;
  // one W map per box height that divides n (the kernel picks the one its
  // tile width needs); the others repeat the 32-row map and are never used
  const int heights[N_BMAPS] = {32, 64, 96, 128, 192, 256};
  for (int i = 0; i < N_BMAPS; ++i) {
    const int h = n % heights[i] == 0 ? heights[i] : 32;
    if ((e = tensor_map(W, n, k, k, h, &tb.m[i])) != cudaSuccess) return e;
  }
  // pairs pay for their coupling and the cluster launch only with many row
  // tiles per CTA: measured faster at 4096 rows (QKV 37 -> 36, fc1 52 -> 48,
  // fc2 56 -> 47 us) and slower at 831 (cross-q 14.3 -> 16.4 us).  The row
  // count must be known here: a device-side count keeps CTAs unpaired.
  const bool pair = shp.pair && !dcount && Mbound >= PAIR_MIN_ROWS;
  const int grid = pair ? shp.grid : device_sms();
  const BnTable bt = bn_table(n, k, grid, sched_mode(ep), (Mbound + BM - 1) / BM, pair);
  if (pair)
    RC_TRY(launch_k_cluster(gemm_kernel<true>(ep.mode), dim3(shp.grid), dim3(THREADS), SMEM_BYTES, 2,
                            st, ta, tb, Mbound, dcount, n, k, ep, bt));
  else
    RC_TRY(launch_k(gemm_kernel<false>(ep.mode), dim3(grid), dim3(THREADS), SMEM_BYTES, st, ta, tb,
                    Mbound, dcount, n, k, ep, bt));
  count_launches(1);
  return cudaSuccess;
}

}  // namespace rc
