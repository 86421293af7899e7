// What an editing turn starts with (sm_103a): the text keys / values of every
// block from the new prompt, the cross-query projection folded into the keys,
// and the localisation scores of Section 3.2 from the cached states.  Every
// block's share is independent of the others', so each of the three runs as
// one launch over all blocks of the model instead of one (or two) per block.
#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"
#include "tma_host.h"

namespace rc {

namespace {

using namespace rc::tc;

constexpr int TM = 128;            // MMA rows: text keys, or image tokens
constexpr int TK = 64;             // k-block (one 128-byte swizzle row of bf16)
constexpr int A_TILE = TM * 128;   // bytes of a 128 x 64 bf16 tile
constexpr uint32_t idesc(int n, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn_major ? 1u << 16 : 0u) |
         (uint32_t(n >> 3) << 17) | (uint32_t(TM >> 4) << 24);
}

// Layers whose tensor maps one launch takes by value (kernel parameters are
// limited to 32 KB; deeper models take several launches).
constexpr int LAYERS_PER_LAUNCH = 32;
struct LayerMaps {
  CUtensorMap m[LAYERS_PER_LAUNCH];
  const float* bias[LAYERS_PER_LAUNCH];
};

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int x, int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y,
                                             int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(src), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Columns 0 .. 127 of this thread's TMEM lane, plus bias (null: none), as
// bf16 into two 128-byte-swizzled 128 x 64 tiles (row = the lane).
__device__ __forceinline__ void drain_tile(uint32_t taddr, uint8_t* tiles, int row,
                                           const float* bias) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float v[32];
    tmem_ld32(taddr + 32u * q, v);
    if (bias) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 b = __ldg(reinterpret_cast<const float4*>(bias + 32 * q) + i);
        v[4 * i] += b.x; v[4 * i + 1] += b.y; v[4 * i + 2] += b.z; v[4 * i + 3] += b.w;
      }
    }
    uint8_t* t = tiles + (q >> 1) * A_TILE + row * 128;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 4 * (q & 1) + i;
      *reinterpret_cast<uint4*>(t + 16 * (j ^ (row & 7))) =
          make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                     pack_bf16x2(v[8 * i + 4], v[8 * i + 5]),
                     pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
    }
  }
}

// ------------------------------------------------- text keys / values
// text[l] = ctx W_xkv,l^T + b_l for every layer, one CTA per (128 columns,
// layer).  Bound by the weights (5.3 MB a layer): two CTAs an SM, each with
// three 32 KB k-blocks in flight.  The output tile reuses the ring once the
// last MMA has read it.  28 layers of hidden 1152: 36 us (4.2 TB/s of weights)
// where one GEMM launch per layer took 28 x 10.8 us.
constexpr int KV_STAGES = 3, KV_THREADS = 192, KV_STAGE = 2 * A_TILE;
constexpr size_t KV_SMEM = size_t(KV_STAGES) * KV_STAGE + 1024;

__global__ void __launch_bounds__(KV_THREADS, 2)
text_kv_kernel(const __grid_constant__ CUtensorMap tmC, const __grid_constant__ LayerMaps lm,
               const __grid_constant__ CUtensorMap tmT, int layer0, int d, unsigned* err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  __shared__ uint64_t bars[2 * KV_STAGES + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;
  const uint32_t full0 = saddr(bars), empty0 = full0 + 8 * KV_STAGES, done = empty0 + 8 * KV_STAGES;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * KV_STAGES + 1; ++i) mbar_init(full0 + 8 * i, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(saddr(&tmem_slot), 128);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int l = blockIdx.y, c0 = int(blockIdx.x) * 128, nkb = d / TK;
  pdl_wait();
  pdl_trigger();
  if (warp == 0) {
    if (elect_one()) {
      for (int kb = 0; kb < nkb; ++kb) {
        const int st = kb % KV_STAGES;
        if (!mbar_sleep(empty0 + 8 * st, ((kb / KV_STAGES) & 1) ^ 1, abort_flag)) {
          *abort_flag = 1;
          break;
        }
        mbar_expect_tx(full0 + 8 * st, KV_STAGE);
        uint8_t* b = smem + st * KV_STAGE;
        tma_load_2d(saddr(b + A_TILE), &lm.m[l], full0 + 8 * st, kb * TK, c0);
        tma_load_2d(saddr(b), &tmC, full0 + 8 * st, kb * TK, 0);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint64_t da = sw128_desc(saddr(smem)), db = sw128_desc(saddr(smem + A_TILE));
      bool ok = true;
      for (int kb = 0; kb < nkb && ok; ++kb) {
        const int st = kb % KV_STAGES;
        ok = mbar_sleep(full0 + 8 * st, (kb / KV_STAGES) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t so = uint64_t((st * KV_STAGE) >> 4);
#pragma unroll
        for (int kk = 0; kk < TK / 16; ++kk)
          umma_bf16(tmem, da + so + 2 * kk, db + so + 2 * kk, idesc(128, false),
                    (kb > 0 || kk > 0) ? 1u : 0u);
        umma_commit(empty0 + 8 * st);
      }
      if (ok) umma_commit(done);
      else *abort_flag = 1;
    }
  } else {
    const int sp = warp & 3, row = sp * 32 + lane;
    const bool ok = mbar_sleep_warp(done, 0, abort_flag);
    if (ok) {
      tc_fence_after();
      drain_tile(tmem + (uint32_t(sp * 32) << 16), smem, row, lm.bias[l] ? lm.bias[l] + c0 : nullptr);
      fence_proxy_async_smem();
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (warp == 2 && elect_one() && ok) {
      tma_store_3d(&tmT, saddr(smem), c0, 0, layer0 + l);
      tma_store_3d(&tmT, saddr(smem + A_TILE), c0 + 64, 0, layer0 + l);
      bulk_commit();
      bulk_wait_all();
    }
    if (!ok && threadIdx.x == 64) {
      *abort_flag = 1;
      atomicOr(err, DEVERR_TIMEOUT);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

// ------------------------------------------------- folded keys
// G_h = K_h W_xq,h ([M][d], f32 accumulation, stored as bf16) and kb_h =
// K_h b_h of every (layer, head), one CTA each: the head's keys (A, K-major,
// dh padded to a multiple of 16 with zeros) stay in shared memory while
// W_xq,h streams through in 128-column chunks (B, MN-major: its rows are the
// head's dh outputs).  Rows past the text length come out as zero.  Bound by
// the 132 MB of G it writes: 28 layers of 16 heads take 36 us (3.7 TB/s); the
// FMA kernel it replaces took 28 x 64 us.
constexpr int FD_STAGES = 3, FD_THREADS = 192;
template <int DH>
struct FoldCfg {
  static constexpr bool TAIL = DH > 64;
  static constexpr int KD = TAIL ? 80 : 64;  // padded dh
  static constexpr int A32 = TAIL ? TM * 32 : 0;
  static constexpr int ATOM = KD * 128;      // KD rows of 64 columns of W_xq
  static constexpr int CHUNK = 2 * ATOM;
  static constexpr int OUT = 2 * A_TILE;
  static constexpr size_t SMEM =
      size_t(A_TILE) + A32 + FD_STAGES * CHUNK + 2 * OUT + 1024;
};

template <int DH>
__global__ void __launch_bounds__(FD_THREADS, 1)
fold_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmKt,
            const __grid_constant__ LayerMaps lm, const __grid_constant__ CUtensorMap tmG,
            const bf16* __restrict__ text, int layer0, int M, int d, int heads,
            float* __restrict__ kb, unsigned* err) {
  using C = FoldCfg<DH>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* sA = align1024(smem_raw);
  uint8_t* sW = sA + A_TILE + C::A32;
  uint8_t* sO = sW + FD_STAGES * C::CHUNK;
  __shared__ uint64_t bars[2 * FD_STAGES + 5];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;
  const uint32_t full0 = saddr(bars), empty0 = full0 + 8 * FD_STAGES;
  const uint32_t a_full = empty0 + 8 * FD_STAGES, t_full = a_full + 8, t_free = t_full + 16;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * FD_STAGES + 3; ++i) mbar_init(full0 + 8 * i, 1);
    mbar_init(t_free, 128);
    mbar_init(t_free + 8, 128);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(saddr(&tmem_slot), 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int h = blockIdx.x, l = blockIdx.y, layer = layer0 + l, chunks = d / 128;
  pdl_wait();
  pdl_trigger();
  if (warp == 0) {
    if (elect_one()) {
      mbar_expect_tx(a_full, A_TILE + C::A32);
      tma_load_4d(saddr(sA), &tmK, a_full, 0, h, 0, layer);
      if (C::TAIL) tma_load_4d(saddr(sA + A_TILE), &tmKt, a_full, 64, h, 0, layer);
      for (int c = 0; c < chunks; ++c) {
        const int st = c % FD_STAGES;
        if (!mbar_sleep(empty0 + 8 * st, ((c / FD_STAGES) & 1) ^ 1, abort_flag)) {
          *abort_flag = 1;
          break;
        }
        mbar_expect_tx(full0 + 8 * st, C::CHUNK);
        uint8_t* b = sW + st * C::CHUNK;
        tma_load_3d(saddr(b), &lm.m[l], full0 + 8 * st, c * 128, 0, h);
        tma_load_3d(saddr(b + C::ATOM), &lm.m[l], full0 + 8 * st, c * 128 + 64, 0, h);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint64_t da = sw128_desc(saddr(sA)), dt = sw32_kmajor_desc(saddr(sA + A_TILE));
      bool ok = mbar_sleep(a_full, 0, abort_flag);
      for (int c = 0; c < chunks && ok; ++c) {
        const int st = c % FD_STAGES;
        ok = mbar_sleep(full0 + 8 * st, (c / FD_STAGES) & 1, abort_flag) &&
             mbar_sleep(t_free + 8 * (c & 1), ((c >> 1) & 1) ^ 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t db = sw128_mnmajor_desc_lbo(saddr(sW + st * C::CHUNK), C::ATOM);
        const uint32_t acc = tmem + 128u * uint32_t(c & 1);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)  // 16 of the head's dims: 16 rows of 128 bytes of W
          umma_bf16(acc, da + 2 * kk, db + 128 * kk, idesc(128, true), kk > 0 ? 1u : 0u);
        if (C::TAIL) umma_bf16(acc, dt, db + 128 * 4, idesc(128, true), 1u);
        umma_commit(empty0 + 8 * st);
        umma_commit(t_full + 8 * (c & 1));
      }
      if (!ok) *abort_flag = 1;
    }
  } else {
    const int sp = warp & 3, row = sp * 32 + lane;
    const size_t g0 = size_t(layer) * heads + h;
    if (row < M) {  // the key's bias, f32, in ascending order of the head's dims
      const bf16* kr = text + (size_t(layer) * M + row) * 2 * d + h * DH;
      const float* b = lm.bias[l] + h * DH;
      float a = 0.f;
#pragma unroll
      for (int j = 0; j < DH / 8; ++j) {
        const uint4 u = *reinterpret_cast<const uint4*>(kr + 8 * j);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = unpack_bf16x2(w[i]);
          a = fmaf(f.x, __ldg(b + 8 * j + 2 * i), a);
          a = fmaf(f.y, __ldg(b + 8 * j + 2 * i + 1), a);
        }
      }
      kb[g0 * XQ_KEYS + row] = a;
    }
    bool ok = true;
    for (int c = 0; c < chunks; ++c) {
      uint8_t* out = sO + (c & 1) * C::OUT;
      if (ok) ok = mbar_sleep_warp(t_full + 8 * (c & 1), (c >> 1) & 1, abort_flag);
      // the buffer's store of two chunks ago has been read (its issuer waits)
      if (warp == 2) bulk_wait_read<1>();
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (ok) {
        tc_fence_after();
        drain_tile(tmem + 128u * uint32_t(c & 1) + (uint32_t(sp * 32) << 16), out, row, nullptr);
        tc_fence_before();
        mbar_arrive(t_free + 8 * (c & 1));
        fence_proxy_async_smem();
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (threadIdx.x == 64 && ok) {
        tma_store_3d(&tmG, saddr(out), c * 128, 0, int(g0));
        tma_store_3d(&tmG, saddr(out + A_TILE), c * 128 + 64, 0, int(g0));
        bulk_commit();
      }
    }
    if (threadIdx.x == 64) {
      bulk_wait_all();
      if (!ok) {
        *abort_flag = 1;
        atomicOr(err, DEVERR_TIMEOUT);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

// ------------------------------------------------- localisation scores
// scores[i][j] = mean over layers and heads of softmax_j'((x_i G_h^T + kb_h)
// / sqrt(dh))[j] for the listed columns j.  Persistent, one CTA an SM; a unit
// is one layer and two heads of a token tile: S = x G^T with the two heads' key
// rows, each rounded up to 8, as N <= 256 columns.  Two token tiles share a
// unit as a CTA pair (M = 256): a CTA then holds 16 + 16 KB a k-block instead of
// 16 + 32, so 7 k-blocks are in flight instead of 4 over a load latency of
// 1400 cycles and more.  Bound by the tensor pipe under the power cap, so the
// two 256-column accumulators alternate and eight warps take the softmax of
// one unit under the MMAs of the next.  4096 tokens x 28 layers x 16 heads x
// 120 keys: 329 us with single CTAs and all 128 rows a head, 318 without the
// rows past the text, 296 (1.7 PFLOP/s) in pairs.  Units are handed out in
// contiguous ranges, tokens outermost: a thread keeps its token's sums over
// layers and heads in registers and adds them to memory once per range and
// token tile.
constexpr int SC_THREADS = 384;
// CTAs a unit, stages of the ring and bytes of one in a CTA
template <int CL>
struct ScoreCfg {
  static constexpr int STAGES = CL == 2 ? 7 : 4;
  static constexpr int STAGE = A_TILE + 2 / CL * XQ_KEYS * 128;
  static constexpr size_t SMEM = size_t(STAGES) * STAGE + 1024;
};
constexpr int SC_MAX = 8;  // listed columns

template <int CL>
__global__ void __launch_bounds__(SC_THREADS, 1)
scores_kernel(const __grid_constant__ CUtensorMap tmX0, const __grid_constant__ CUtensorMap tmX,
              const __grid_constant__ CUtensorMap tmG, const float* __restrict__ kb, int N, int d,
              int layers, int heads, int xrow0, int xrow_step, int grow0, int Nk,
              float scale_log2, const __grid_constant__ AttnCapture cap, unsigned* err) {
  using C = ScoreCfg<CL>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  __shared__ uint64_t bars[2 * C::STAGES + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;
  const uint32_t full0 = saddr(bars), empty0 = full0 + 8 * C::STAGES;
  const uint32_t t_full = empty0 + 8 * C::STAGES, t_free = t_full + 16;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < C::STAGES; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(t_full + 8 * i, 1);
      mbar_init(t_free + 8 * i, 8 * CL);  // one arrival a softmax warp
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (CL == 2) tmem_alloc_pair(saddr(&tmem_slot), 512);
    else tmem_alloc(saddr(&tmem_slot), 512);
  }
  tc_fence_before();
  if (CL == 2) cluster_sync();  // (the peer's barriers are set up)
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int rank = CL == 2 ? int(cluster_ctarank()) : 0;
  const int pairs = heads / 2, per_tile = layers * pairs, nkb = d / TK;
  const int keys = (Nk + 7) & ~7;  // rows of a head in a stage
  const long long units = (long long)((N + CL * TM - 1) / (CL * TM)) * per_tile;
  const int pos = int(blockIdx.x) / CL, np = int(gridDim.x) / CL;
  const int u0 = int(units * pos / np), u1 = int(units * (pos + 1) / np);
  pdl_wait();
  pdl_trigger();
  if (warp == 0 || warp == 2) {
    // warp 0 loads the token rows, warp 2 the folded keys: one thread issuing
    // both is close to the time of a k-block's MMAs
    if (elect_one()) {
      int st = 0;
      uint32_t ph = 1;
      for (int u = u0; u < u1; ++u) {
        const int qt = u / per_tile, rest = u - qt * per_tile, l = rest / pairs;
        const int grow = grow0 + (l * heads + 2 * (rest - l * pairs)) * XQ_KEYS;
        // layer 0 reads the embedding, layer l the cached output of l - 1
        const CUtensorMap* mx = l ? &tmX : &tmX0;
        const int xrow = (qt * CL + rank) * TM + (l ? xrow0 + (l - 1) * xrow_step : 0);
        for (int k = 0; k < nkb; ++k) {
          if (!mbar_wait(empty0 + 8 * st, ph, abort_flag)) {
            *abort_flag = 1;
            goto out;
          }
          uint8_t* b = smem + st * C::STAGE;
          if (CL == 2) {  // all of a pair's bytes are counted by rank 0's barrier
            const uint32_t fb = mapa_shared(full0 + 8 * st, 0);
            if (warp == 2) {
              tma_load_2d_pair(saddr(b + A_TILE), &tmG, fb, k * TK, grow + rank * XQ_KEYS);
            } else {
              if (rank == 0)
                mbar_expect_tx(full0 + 8 * st, uint32_t(2 * (A_TILE + keys * 128)));
              tma_load_2d_pair(saddr(b), mx, fb, k * TK, xrow);
            }
          } else if (warp == 2) {
            for (int g = 0; g < 2; ++g)
              tma_load_2d(saddr(b + A_TILE + g * keys * 128), &tmG, full0 + 8 * st, k * TK,
                          grow + g * XQ_KEYS);
          } else {
            mbar_expect_tx(full0 + 8 * st, uint32_t(A_TILE + 2 * keys * 128));
            tma_load_2d(saddr(b), mx, full0 + 8 * st, k * TK, xrow);
          }
          if (++st == C::STAGES) { st = 0; ph ^= 1; }
        }
      }
      // every stage has been freed: no arrival is on its way to this CTA when
      // it leaves
      for (int i = 0; CL == 2 && i < C::STAGES; ++i) {
        if (!mbar_wait(empty0 + 8 * st, ph, abort_flag)) goto out;
        if (++st == C::STAGES) { st = 0; ph ^= 1; }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      const uint64_t da = sw128_desc(saddr(smem)), db = sw128_desc(saddr(smem + A_TILE));
      // (M = 256 over a pair: bits 24.. hold M / 16)
      const uint32_t id = (idesc(0, false) + (CL == 2 ? uint32_t(TM >> 4) << 24 : 0u)) |
                          (uint32_t(2 * keys) >> 3 << 17);
      int st = 0;
      uint32_t ph = 0;
      bool ready = false;  // the current stage was seen full already
      for (int u = u0; u < u1; ++u) {
        const int i = u - u0;
        if (!mbar_wait(t_free + 8 * (i & 1), ((i >> 1) & 1) ^ 1, abort_flag)) {
          *abort_flag = 1;
          goto out;
        }
        tc_fence_after();
        const uint32_t acc = tmem + 256u * uint32_t(i & 1);
        for (int k = 0; k < nkb; ++k) {
          if (!ready && !mbar_wait(full0 + 8 * st, ph, abort_flag)) {
            *abort_flag = 1;
            goto out;
          }
          const uint64_t so = uint64_t((st * C::STAGE) >> 4);
          const uint32_t eb = empty0 + 8 * st;
          if (++st == C::STAGES) { st = 0; ph ^= 1; }
          ready = mbar_test(full0 + 8 * st, ph);  // (beside this stage's MMAs)
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < TK / 16; ++kk) {
            const uint32_t add = (k > 0 || kk > 0) ? 1u : 0u;
            if (CL == 2) umma_bf16_pair(acc, da + so + 2 * kk, db + so + 2 * kk, id, add);
            else umma_bf16(acc, da + so + 2 * kk, db + so + 2 * kk, id, add);
          }
          if (CL == 2) umma_commit_pair(eb);
          else umma_commit(eb);
        }
        if (CL == 2) umma_commit_pair(t_full + 8 * (i & 1));
        else umma_commit(t_full + 8 * (i & 1));
      }
    }
  } else if (warp >= 4) {
    const int sp = warp & 3, half = (warp - 4) >> 2;
    float acc[SC_MAX];
#pragma unroll
    for (int q = 0; q < SC_MAX; ++q) acc[q] = 0.f;
    int qt = u0 / per_tile;
    auto flush = [&]() {
      const int tok = (qt * CL + rank) * TM + sp * 32 + lane;
      if (tok < N) {
#pragma unroll
        for (int q = 0; q < SC_MAX; ++q)
          if (q < cap.n) atomicAdd(cap.out + size_t(tok) * cap.ldo + cap.id[q], cap.w * acc[q]);
      }
#pragma unroll
      for (int q = 0; q < SC_MAX; ++q) acc[q] = 0.f;
    };
    for (int u = u0; u < u1; ++u) {
      const int i = u - u0, nqt = u / per_tile, rest = u - nqt * per_tile, l = rest / pairs;
      const int h = 2 * (rest - l * pairs) + half;
      if (nqt != qt) {
        flush();
        qt = nqt;
      }
      if (!mbar_sleep_warp(t_full + 8 * (i & 1), (i >> 1) & 1, abort_flag)) {
        *abort_flag = 1;
        if (threadIdx.x == 128) atomicOr(err, DEVERR_TIMEOUT);
        goto out;
      }
      tc_fence_after();
      const uint32_t ts =
          tmem + 256u * uint32_t(i & 1) + uint32_t(half * keys) + (uint32_t(sp * 32) << 16);
      const float* b = kb + size_t(grow0) + (size_t(l) * heads + h) * XQ_KEYS;
      float r[XQ_KEYS];
#pragma unroll
      for (int c = 0; c < XQ_KEYS / 16; ++c)
        tmem_ld16_nowait(ts + 16u * c, reinterpret_cast<uint32_t*>(r) + 16 * c);
      tmem_wait_ld();
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < XQ_KEYS / 4; ++c) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(b) + c);
        const float a[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          r[4 * c + e] = 4 * c + e < Nk ? r[4 * c + e] + a[e] : -INFINITY;
          mx[e] = fmaxf(mx[e], r[4 * c + e]);
        }
      }
      const float m = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale_log2;
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < XQ_KEYS; ++c) s[c & 3] += ex2_ftz(fmaf(r[c], scale_log2, -m));
      const float sum = (s[0] + s[1]) + (s[2] + s[3]);
      const float inv = sum > 0.f ? 1.f / sum : 0.f;
      // the listed columns again, one by one (the column is the same for
      // the whole warp)
#pragma unroll
      for (int q = 0; q < SC_MAX; ++q)
        if (q < cap.n) {
          const uint32_t v = tmem_ld1_nowait(ts + uint32_t(cap.id[q]));
          tmem_wait_ld();
          acc[q] += ex2_ftz(fmaf(__uint_as_float(v) + __ldg(b + cap.id[q]), scale_log2, -m)) * inv;
        }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CL == 2) mbar_arrive_cluster(mapa_shared(t_free + 8 * (i & 1), 0));
        else mbar_arrive(t_free + 8 * (i & 1));
      }
    }
    if (u1 > u0) flush();
  }
out:
  tc_fence_before();
  __syncthreads();
  if (CL == 2) cluster_sync();  // the peer's loads and arrivals in this CTA are done
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if (CL == 2) tmem_dealloc_pair(tmem, 512);
    else tmem_dealloc(tmem, 512);
  }
}

int turn_sms() {
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (!sms[dev]) {
    int v = 0;
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(text_kv_kernel, attr, int(KV_SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(fold_kernel<72>, attr, int(FoldCfg<72>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(fold_kernel<64>, attr, int(FoldCfg<64>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(scores_kernel<1>, attr, int(ScoreCfg<1>::SMEM)) != cudaSuccess ||
        cudaFuncSetAttribute(scores_kernel<2>, attr, int(ScoreCfg<2>::SMEM)) != cudaSuccess)
      return 0;
    sms[dev] = v;
  }
  return sms[dev];
}

}  // namespace

cudaError_t launch_text_kv(const bf16* ctx, const TextLayer* layers, int L, int M, int d,
                           bf16* text, unsigned* err, cudaStream_t st) {
  if (M < 1 || M > TM || d % 128) return cudaErrorInvalidValue;
  if (!turn_sms()) return cudaErrorInvalidDevice;
  CUtensorMap tc, tt;
  {
    const cuuint64_t dims[2] = {cuuint64_t(d), cuuint64_t(M)}, str[1] = {cuuint64_t(d)};
    const cuuint32_t box[2] = {TK, TM};
    RC_TRY(tma_map(ctx, 2, dims, str, box, &tc));
  }
  {
    // (column, text row, layer): rows past the text length are not written
    const cuuint64_t dims[3] = {cuuint64_t(2 * d), cuuint64_t(M), cuuint64_t(L)};
    const cuuint64_t str[2] = {cuuint64_t(2 * d), cuuint64_t(M) * 2 * d};
    const cuuint32_t box[3] = {64, TM, 1};
    RC_TRY(tma_map(text, 3, dims, str, box, &tt));
  }
  for (int l0 = 0; l0 < L; l0 += LAYERS_PER_LAUNCH) {
    const int n = L - l0 < LAYERS_PER_LAUNCH ? L - l0 : LAYERS_PER_LAUNCH;
    LayerMaps lm{};
    for (int i = 0; i < n; ++i) {
      const cuuint64_t dims[2] = {cuuint64_t(d), cuuint64_t(2 * d)}, str[1] = {cuuint64_t(d)};
      const cuuint32_t box[2] = {TK, 128};
      RC_TRY(tma_map(layers[l0 + i].W_xkv, 2, dims, str, box, &lm.m[i]));
      lm.bias[i] = layers[l0 + i].b_xkv;
    }
    RC_TRY(launch_k(text_kv_kernel, dim3(2 * d / 128, n), dim3(KV_THREADS), KV_SMEM, st, tc, lm,
                    tt, l0, d, err));
    count_launches(1);
  }
  return cudaSuccess;
}

cudaError_t launch_xq_fold(const bf16* text, const TextLayer* layers, int L, int M, int heads,
                           int dh, bf16* G, float* kb, unsigned* err, cudaStream_t st) {
  const int d = heads * dh;
  if (M < 1 || M > XQ_KEYS || (dh != 72 && dh != 64) || d % 128) return cudaErrorInvalidValue;
  if (!turn_sms()) return cudaErrorInvalidDevice;
  CUtensorMap tk, tkt, tg;
  {
    // (head dim, head, text row, layer): reads past dh or the text length are zero
    const cuuint64_t dims[4] = {cuuint64_t(dh), cuuint64_t(heads), cuuint64_t(M), cuuint64_t(L)};
    const cuuint64_t str[3] = {cuuint64_t(dh), cuuint64_t(2 * d), cuuint64_t(M) * 2 * d};
    cuuint32_t box[4] = {64, 1, TM, 1};
    RC_TRY(tma_map(text, 4, dims, str, box, &tk));
    box[0] = 16;
    RC_TRY(tma_map(text, 4, dims, str, box, &tkt));
  }
  {
    const cuuint64_t dims[3] = {cuuint64_t(d), XQ_KEYS, cuuint64_t(L) * heads};
    const cuuint64_t str[2] = {cuuint64_t(d), cuuint64_t(XQ_KEYS) * d};
    const cuuint32_t box[3] = {64, TM, 1};
    RC_TRY(tma_map(G, 3, dims, str, box, &tg));
  }
  for (int l0 = 0; l0 < L; l0 += LAYERS_PER_LAUNCH) {
    const int n = L - l0 < LAYERS_PER_LAUNCH ? L - l0 : LAYERS_PER_LAUNCH;
    LayerMaps lm{};
    for (int i = 0; i < n; ++i) {
      // (input column, the head's output, head): outputs past dh read as zero
      const cuuint64_t dims[3] = {cuuint64_t(d), cuuint64_t(dh), cuuint64_t(heads)};
      const cuuint64_t str[2] = {cuuint64_t(d), cuuint64_t(dh) * d};
      const cuuint32_t box[3] = {64, cuuint32_t(dh == 72 ? FoldCfg<72>::KD : FoldCfg<64>::KD), 1};
      RC_TRY(tma_map(layers[l0 + i].W_xq, 3, dims, str, box, &lm.m[i]));
      lm.bias[i] = layers[l0 + i].b_xq;
    }
    RC_TRY(launch_k(dh == 72 ? fold_kernel<72> : fold_kernel<64>, dim3(heads, n),
                    dim3(FD_THREADS), dh == 72 ? FoldCfg<72>::SMEM : FoldCfg<64>::SMEM, st, tk,
                    tkt, lm, tg, text, l0, M, d, heads, kb, err));
    count_launches(1);
  }
  return cudaSuccess;
}

cudaError_t launch_scores(const bf16* x0, int x0_rows, const bf16* cache, long long cache_rows,
                          int xrow0, int xrow_step, const bf16* G, long long g_rows, int grow0,
                          const float* kb, int N, int layers, int heads, int dh, int Nk,
                          const AttnCapture& cap, unsigned* err, cudaStream_t st) {
  const int d = heads * dh, sms = turn_sms();
  if (!sms) return cudaErrorInvalidDevice;
  // (hidden is a multiple of 128 and dh 64 or 72, so heads come in pairs)
  if (N < 1 || x0_rows < N || d % TK || heads % 2 || Nk < 1 || Nk > XQ_KEYS || cap.n < 1 || cap.n > SC_MAX ||
      !cap.out)
    return cudaErrorInvalidValue;
  for (int q = 0; q < cap.n; ++q)
    if (cap.id[q] < 0 || cap.id[q] >= Nk || cap.id[q] >= cap.ldo) return cudaErrorInvalidValue;
  if (xrow0 < 0 || grow0 < 0 || grow0 + (long long)layers * heads * XQ_KEYS > g_rows ||
      (layers > 1 && xrow0 + (long long)(layers - 2) * xrow_step + N > cache_rows) ||
      cache_rows >= (1ll << 31) || g_rows >= (1ll << 31))
    return cudaErrorInvalidValue;
  const long long units = (long long)((N + TM - 1) / TM) * layers * (heads / 2);
  if (units >= (1ll << 31)) return cudaErrorInvalidValue;
  CUtensorMap t0, tx, tg;
  const cuuint64_t str[1] = {cuuint64_t(d)};
  cuuint64_t dims[2] = {cuuint64_t(d), cuuint64_t(x0_rows)};
  cuuint32_t box[2] = {TK, TM};
  RC_TRY(tma_map(x0, 2, dims, str, box, &t0));
  dims[1] = cuuint64_t(cache_rows);
  RC_TRY(tma_map(cache, 2, dims, str, box, &tx));
  dims[1] = cuuint64_t(g_rows);
  box[1] = cuuint32_t((Nk + 7) & ~7);
  RC_TRY(tma_map(G, 2, dims, str, box, &tg));
  const float scale_log2 = float(1.4426950408889634 / sqrt(double(dh)));
  // pairs wherever there are two token tiles; a single one would leave half of
  // each pair idle (the whole call with single CTAs / pairs, us: 128 tokens 38.8
  // / 39.4, 256 41.6 / 39.7, 384 79.1 / 50.4, 1024 91.6 / 83.2, 4096 344 / 316)
  if (N > TM && sms >= 2) {
    const long long pairs = (long long)((N + 2 * TM - 1) / (2 * TM)) * layers * (heads / 2);
    const int grid = 2 * int(pairs < sms / 2 ? pairs : sms / 2);
    RC_TRY(launch_k_cluster(scores_kernel<2>, dim3(grid), dim3(SC_THREADS),
                            ScoreCfg<2>::SMEM, 2, st, t0, tx, tg, kb, N, d, layers, heads, xrow0, xrow_step, grow0, Nk,
                            scale_log2, cap, err));
  } else {
    const int grid = int(units < sms ? units : sms);
    RC_TRY(launch_k(scores_kernel<1>, dim3(grid), dim3(SC_THREADS), ScoreCfg<1>::SMEM, st,
                    t0, tx, tg, kb, N, d, layers, heads, xrow0, xrow_step, grow0, Nk, scale_log2, cap, err));
  }
  count_launches(1);
  return cudaSuccess;
}

}  // namespace rc
