// Weight-streaming projection GEMM for sm_100a:  P[s][m][n] = sum_{k in split s} X[m][k] * W[n][k]
// (Sec. 4.1 Step 2: the one forward pass over the window; every projection of the decoder).
//
// Shape of the problem: M = batch * window is mostly 8..64 rows, the weight matrices (bf16) are tens to
// hundreds of MB and are read exactly once per step, so the kernel is bound by HBM bandwidth and its
// job is to keep every SM's TMA queue full.  More rows (batches of images, pre-fill passes) run on CTA
// pairs, see gemm_pair_kernel.
//   * W is the 128-row operand of tcgen05.mma (M = 128), the tokens are the N dimension.  The fp32
//     activations arrive split into two bf16 planes, hi = bf16(x) and lo = bf16(x - hi); both planes
//     are columns of the same MMA (N = 2 * Mp), and the epilogue adds the two halves: activations keep
//     ~16 bits of mantissa at no cost in weight bytes.  (Multiplying the hi plane alone, i.e. plain
//     bf16 activations, would halve the tensor work of the many-row case but misses the 2e-2 logits
//     tolerance at d_model 4096 already after two layers: 4.0e-2.  So both planes, always, and the
//     useful tensor throughput of the many-row case cannot pass half the peak.)
//   * One CTA per (128-row weight tile, K split); two CTAs are resident per SM.  A launch covers up to
//     three weight matrices that share the activation operand (Q|K|V, gate|up), so their tiles form
//     one grid.  With more than one K split every CTA writes an fp32 partial plane; the consumer
//     kernel (residual + RMSNorm, RoPE + cache append, SwiGLU, or a plain sum) adds the planes in
//     split order: deterministic, no atomics, no serial reduction tail inside the GEMM.
//   * Warp 0 issues TMA loads of 128B-swizzled 128x64 W tiles (evict-first L2 policy) into a ring of shared-memory stages
//     guarded by mbarriers, warp 6 those of the activation tiles into a shorter ring of their own; warp 1 issues the
//     MMAs into a TMEM accumulator and commits to the k-block's "done" barrier, which frees both stages; warps 2-5 drain the
//     accumulator with tcgen05.ld and store.
//   * Every wait is bounded: after ~2 s a role records an error in the status word and leaves; the
//     CTA still frees its TMEM.
#include <cuda.h>
#include <string.h>

#include <atomic>

#include "tcgen05.cuh"

namespace sjd {
SJD_TIMELINE_TU(gemm)
namespace {

constexpr int TILE_N = 128;   // weight rows per tile (MMA M)
constexpr int TILE_K = 64;    // bf16 elements per k-block = one 128-byte swizzle atom
constexpr int UMMA_K = 16;
constexpr int W_TILE_BYTES = TILE_N * TILE_K * 2;
constexpr int kThreads = 224;   // weight producer, issuer, four epilogue warps, activation producer
constexpr int kMaxStages = 8;
// tunables (defaults chosen by measurement on B200)
#ifndef SJD_GEMM_SMEM_BUDGET
#define SJD_GEMM_SMEM_BUDGET (104 * 1024)   // ring bytes per CTA when two CTAs share an SM, see ring_stages
#endif
#ifndef SJD_GEMM_DEEP_RING
#define SJD_GEMM_DEEP_RING (200 * 1024)     // and when the grid has at most one CTA per SM
#endif
#ifndef SJD_GEMM_L2_PROMO
#define SJD_GEMM_L2_PROMO CU_TENSOR_MAP_L2_PROMOTION_L2_256B
#endif
#ifndef SJD_GEMM_MIN_KB
#define SJD_GEMM_MIN_KB 8                   // fewest k-blocks (of 16 KB of weights) a CTA should stream (8: the O projection runs 32 x 8 CTAs whose whole share fits the prefetched ring; 3.51 against 3.54 ms per step with 16)
#endif
#ifndef SJD_GEMM_CTAS_PER_SM
#define SJD_GEMM_CTAS_PER_SM 2
#endif
// CTA t starts t * kTileSkew k-blocks into its range of K.  In step, all of a launch's CTAs ask L2 for the same few lines of the
// activations at the same time (gate|up, 172 CTAs: 34.2 us, with skew 32.5; logits 91 and 86.4; us of a step of 16 layers, 7B,
// 32 rows: skew 0 / 4 / 8 / 12: 1655 / 1617 / 1616 / 1614, also skewed where K is split 1600 against 1605; two layers and the logits,
// 0 and 8: 7B 48 rows 350 and 344, 64 rows 364 and 356, 8B 64 rows 600 and 592).  Of eight k-blocks (the O projection) all start at the first.
constexpr int kTileSkew = 8;
constexpr int kSmemBudget = SJD_GEMM_SMEM_BUDGET, kDeepRing = SJD_GEMM_DEEP_RING;

struct GemmParams {
  void *out;              // fp32 planes [splits][M][ldc], or bf16 [M][ldc] when store_bf16
  size_t plane_stride;    // elements between planes
  int ldc;
  int M;                  // valid token rows
  int Mp;                 // token rows of one slab, a multiple of 16, on CTA pairs of 8 (MMA N = 2 * Mp: hi and lo plane)
  int n_slabs;            // token slabs (CTA pairs only: more than one)
  int x_lo_row;           // row of the lo plane inside the activation tensor map
  int k_blocks, splits;   // K / 64, K splits (gridDim.y)
  int tile_end[3];        // matrix j owns tiles [tile_end[j-1], tile_end[j])
  int col_off[3];         // first output column of matrix j
  int stages, x_stages;
  int store_bf16;
  int *status;            // device status word (non-zero = a bounded wait ran out)
  const float *ss_part;   // optional [M][n_part] partial sums of squares: rows are scaled by
  int n_part;             //   1 / sqrt(sum_j ss_part[m][j] * inv_d + eps) before they are stored
  float inv_d, eps;
  int tile_rows;          // weight rows a tile really holds (<= 128; the rest of the MMA's 128 rows is idle)
  int n_out[3];           // output features of matrix j (the last tile of a matrix may be partial)
  // gate|up mode (template GU): tile t holds rows [t*tile_rows, (t+1)*tile_rows) of the gate matrix in MMA
  // rows 0.. and the same rows of the up matrix in MMA rows 64..; the epilogue stores
  // silu(gate) * up as bf16 hi/lo planes [M][F]
  __nv_bfloat16 *act_hi;
  size_t act_lo_off;
  int F;
};

// AND of a predicate over the 128 epilogue threads (named barrier 1): keeps their control flow uniform
__device__ __forceinline__ bool epilogue_all(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred)
      : "memory");
  return r != 0;
}

// 16 tokens of one output column: out[i * ld] = v[i] (times scale[i], if any), the first n of them.  Nothing but
// independent adds and stores: an epilogue has a warp or two per scheduler, so every dependent instruction costs its latency
// (with bounds, type and scale tested per element, 128 tokens took 7 us).
template <typename O>
__device__ __forceinline__ void store_column(O *out, size_t ld, float *v, const float *scale, int n) {
  if (scale) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] *= scale[i];
  }
  auto put = [&](int i) {
    if constexpr (sizeof(O) == 2) out[i * ld] = __float2bfloat16_rn(v[i]);
    else out[i * ld] = v[i];
  };
  if (n >= 16) {
#pragma unroll
    for (int i = 0; i < 16; ++i) put(i);
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < n) put(i);
  }
}

constexpr int kTcBarriers = 3 * kMaxStages + 1;
// behind the rings of a CTA
struct TcShared {
  uint64_t full[kMaxStages], x_full[kMaxStages];   // (one array of kTcBarriers to set up)
  uint64_t done[kMaxStages];                       // k-block it has been multiplied: number it % kMaxStages
  uint64_t acc_full;
  uint32_t tmem_base;
  float scale[TILE_N];   // per-row output scales (epilogue)
};

// ---------------------------------------------------------------------------------- kernel
// GU: the gate|up launch that applies SwiGLU in its epilogue
template <bool GU>
__global__ void __launch_bounds__(kThreads, 2)
gemm_tc_kernel(const __grid_constant__ CUtensorMap w_map0, const __grid_constant__ CUtensorMap w_map1,
               const __grid_constant__ CUtensorMap w_map2, const __grid_constant__ CUtensorMap x_map, const GemmParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];   // no static shared memory: it starts on 1024 bytes
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tile = blockIdx.x, split = blockIdx.y;
  constexpr int m_base = 0;   // one slab: more rows run on CTA pairs
  const int NN = 2 * p.Mp;                           // MMA N
  const int x_tile_bytes = NN * TILE_K * 2;
  uint8_t *smem_x = smem + p.stages * W_TILE_BYTES;
  TcShared &sh = *reinterpret_cast<TcShared *>(smem_x + p.x_stages * x_tile_bytes);
  float *s_scale = sh.scale;

  pdl_trigger();   // the next kernel in the stream may be scheduled as soon as every CTA got here
  SJD_TL(TL_GEMM, 0, threadIdx.x == 0);
  const int R = p.tile_rows;
  const uint32_t w_tx = (uint32_t)((GU ? 2 : 1) * R * TILE_K * 2);   // bytes the copies of a weight stage deliver

  // which weight matrix this tile belongs to
  const int mat = GU ? 0 : (tile < p.tile_end[0] ? 0 : (tile < p.tile_end[1] ? 1 : 2));
  const CUtensorMap *w_map = mat == 0 ? &w_map0 : (mat == 1 ? &w_map1 : &w_map2);
  const int tile_in_mat = tile - (mat == 0 ? 0 : p.tile_end[mat - 1]);
  // this CTA's k-blocks
  const int kb_begin = (int)(((long)split * p.k_blocks) / p.splits);
  const int kb_end = (int)(((long)(split + 1) * p.k_blocks) / p.splits);
  const int n_kb = kb_end - kb_begin;

  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < NN) tmem_cols <<= 1;

  if (tid == 0) {
    tma_prefetch_desc(w_map);
    tma_prefetch_desc(&x_map);
  }
  if (tid < kTcBarriers) {
    mbar_init(&sh.full[tid], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = sh.tmem_base;

  if (warp == 0 || warp == 6) {
    // ------------------------------------------------------------------ TMA producers: weights (0), activations (6)
    // The weights do not depend on the preceding kernel: they are streamed from the start, the activations that it produced are
    // waited for.
    const bool is_w = warp == 0;
    const int ring = is_w ? p.stages : p.x_stages;
    uint64_t *full = is_w ? sh.full : sh.x_full;
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    if (!is_w) pdl_wait();
    // (the swizzled tiles have to start on 1024 bytes; not before the wait: sjd_gemm's split kernel clears the word)
    if (!is_w && lane == 0 && (smem_u32(smem) & 1023u) != 0) atomicExch(p.status, 5);
    SJD_TL(TL_GEMM, 1, !is_w && lane == 0);
    const int first = (tile * kTileSkew) % n_kb;
    int s = 0, it = 0;
    bool ok = true;
    for (; it < n_kb; ++it) {
      const int of = it - ring;   // the k-block whose stage this is
      if (of >= 0 && !warp_wait(&sh.done[of % kMaxStages], (uint32_t)(of / kMaxStages) & 1u)) { ok = false; break; }
      if (elect_one()) {
        const int kcol = (kb_begin + (it + first < n_kb ? it + first : it + first - n_kb)) * TILE_K;
        if (is_w) {
          uint8_t *dst = smem + s * W_TILE_BYTES;
          mbar_expect_tx(&full[s], w_tx);
          if (GU) {
            tma_load_2d(dst, &w_map0, kcol, tile * R, &full[s], policy);
            tma_load_2d(dst + W_TILE_BYTES / 2, &w_map1, kcol, tile * R, &full[s], policy);
          } else {
            tma_load_2d(dst, w_map, kcol, tile_in_mat * R, &full[s], policy);
          }
        } else {
          uint8_t *dst = smem_x + s * x_tile_bytes;
          mbar_expect_tx(&full[s], (uint32_t)x_tile_bytes);
          tma_load_2d_nohint(dst, &x_map, kcol, m_base, &full[s]);
          tma_load_2d_nohint(dst + x_tile_bytes / 2, &x_map, kcol, p.x_lo_row + m_base, &full[s]);
        }
      }
      __syncwarp();
      if (++s == ring) s = 0;
    }
    if (!ok) {
      if (lane == 0) atomicExch(p.status, 1);
      // leave no copy in flight: wait (bounded) for the stages armed most recently
      const int armed = it < ring ? it : ring;
      for (int j = it - armed; j < it; ++j) warp_wait(&full[j % ring], (uint32_t)((j / ring) & 1));
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t idesc = umma_idesc_bf16(NN);
    const uint64_t desc0 = umma_desc_sw128(0);
    int s = 0, sx = 0;
    uint32_t ph = 0, phx = 0;
    bool ok = true;
    for (int it = 0; it < n_kb; ++it) {
      if (!warp_wait_both(&sh.full[s], ph, &sh.x_full[sx], phx)) { ok = false; break; }
      tc_fence_after();
      if (elect_one()) {
        const uint64_t a = desc0 | (uint64_t)(smem_u32(smem + s * W_TILE_BYTES) >> 4);
        const uint64_t b = desc0 | (uint64_t)(smem_u32(smem_x + sx * x_tile_bytes) >> 4);
#pragma unroll
        for (int k = 0; k < TILE_K / UMMA_K; ++k) umma_bf16(tmem_base, a + k * 2, b + k * 2, idesc, !(it == 0 && k == 0));
        umma_commit(&sh.done[it % kMaxStages]);   // frees both stages once these MMAs have read them
      }
      __syncwarp();
      if (++s == p.stages) { s = 0; ph ^= 1u; }
      if (++sx == p.x_stages) { sx = 0; phx ^= 1u; }
    }
    if (ok) {
      if (elect_one()) umma_commit(&sh.acc_full);
    } else if (lane == 0) {
      atomicExch(p.status, 2);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ epilogue warps (2..5)
    const int quarter = warp & 3;                 // TMEM lane quarter this warp may read
    const int row = quarter * 32 + lane;          // weight row inside the tile
    const bool ok = epilogue_all(warp_wait(&sh.acc_full, 0));
    if (ok) {
      tc_fence_after();
      pdl_wait();   // the planes may still be read, and the row scales written, by the preceding kernel
      float *plane = reinterpret_cast<float *>(p.out) + (size_t)split * p.plane_stride;
      __nv_bfloat16 *out_bf16 = reinterpret_cast<__nv_bfloat16 *>(p.out);
      if (p.ss_part || GU) {   // RMS scale of each token row, once per CTA (epilogue thread e: row m_base + e)
        const int e = tid - 64, m = m_base + e;
        float sc = 1.0f;
        if (p.ss_part && e < p.Mp && m < p.M) {
          float tot = 0.0f;
          for (int jj = 0; jj < p.n_part; ++jj) tot += __ldg(p.ss_part + (size_t)m * p.n_part + jj);
          sc = rsqrtf(tot * p.inv_d + p.eps);
        }
        s_scale[e] = sc;
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      if (GU) {
        // MMA rows 0..63 hold gate features, rows 64..127 the same features of the up matrix.  The warps
        // that read the up rows (TMEM lane quarters 2, 3) pass their values through shared memory (the
        // ring is idle by now) to the warps that read the gate rows, which finish the activation.
        // Every epilogue warp parks its 32 accumulator rows (scaled) in shared memory, row-major with an odd
        // stride; after one barrier the 128 threads share the activation work: thread t finishes feature
        // t % 64 for every second token, so that a warp's stores cover 32 adjacent features of one token.
        float *ex = reinterpret_cast<float *>(smem);   // [128][Mp + 1]
        const int ldx = p.Mp + 1;
        const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
        for (int m0 = 0; m0 < p.Mp; m0 += 16) {
          uint32_t hi[16], lo[16];
          tmem_ld16_issue(t_addr + m0, hi);
          tmem_ld16_issue(t_addr + p.Mp + m0, lo);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i)
            ex[row * ldx + m0 + i] = (__uint_as_float(hi[i]) + __uint_as_float(lo[i])) * s_scale[m0 + i];
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const int e = tid - 64, fr = e & 63;
        const int f = tile * R + fr;
        if (fr < R && f < p.F) {
#pragma unroll 8
          for (int mm = e >> 6; mm < p.M; mm += 2) {
            const float g = ex[fr * ldx + mm], u = ex[(64 + fr) * ldx + mm];
            const float v = g / (1.0f + expf(-g)) * u;
            const __nv_bfloat16 vh = __float2bfloat16_rn(v);
            p.act_hi[(size_t)mm * p.F + f] = vh;
            p.act_hi[p.act_lo_off + (size_t)mm * p.F + f] = __float2bfloat16_rn(v - __bfloat162float(vh));
          }
        }
      } else {
      const int n_local = tile_in_mat * R + row;
      const int n = p.col_off[mat] + n_local;
      const bool live = row < R && n_local < p.n_out[mat];
      for (int m0 = 0; m0 < p.Mp; m0 += 16) {                    // first token row of the chunk
        const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
        uint32_t hi[16], lo[16];
        tmem_ld16_issue(t_addr + m0, hi);
        tmem_ld16_issue(t_addr + p.Mp + m0, lo);
        tmem_ld_wait();
        if (!live) continue;
        const float *scale = p.ss_part ? s_scale + m0 : nullptr;
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
        if (p.store_bf16) store_column(out_bf16 + (size_t)m0 * p.ldc + n, p.ldc, v, scale, p.M - m0);
        else store_column(plane + (size_t)m0 * p.ldc + n, p.ldc, v, scale, p.M - m0);
      }
      }
    } else if (tid == 64) {
      atomicExch(p.status, 3);
    }
    SJD_TL(TL_GEMM, 2, tid == 64);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ---------------------------------------------------------------------------------- many rows: CTA pairs
// More than 64 token rows.  The tensor pipe is the bound (both activation planes are multiplied), and with one CTA per tile the
// shared memory is: a 128 x 256 MMA moves 192 bytes of operands per clock through a port of 128 (measured: 57 % tensor
// activity, 29-35 % of the bf16 peak useful).  Here two CTAs of a cluster work on 256 weight rows x one slab of up to 128
// tokens with cta_group::2 MMAs: each holds its own 128 weight rows and one activation plane (rank 0 hi, rank 1 lo), i.e. half
// of the bytes.  One CTA per SM, persistent: a pair runs through (weight tile pair, K split, token slab) units, slabs
// innermost so that the pairs at work share weight tiles in L2; two accumulators in tensor memory, so that a unit's epilogue
// runs under the next unit's products.  Kernel alone, before -> now, us: 128 x 12288 x 4096 31.5 -> 25, 256 x 12288 x 4096 59 -> 42,
// 200 x 22016 x 4096 102 -> 61, 1024 x 12288 x 4096 169 -> 135 (1.5 PFLOP/s issued).
constexpr int kPairStages = 8;
constexpr int kPairThreads = 64 + 256;   // producer, issuer, eight epilogue warps
constexpr int kPairSmem = 232448 - 2048; // most dynamic shared memory of a CTA, beside its static part
constexpr int kShareParts = 4;           // most pairs that share a unit
constexpr int kExTokens = 16;            // tokens of one exchange round of the gate|up epilogue

struct PairParams {
  GemmParams g;
  int tiles;             // 128-row weight tiles
  int n_units;
  // Units of the last, partial round (from unit `full` on) that several pairs share: `parts` pairs take a range of K each and
  // leave their sums in scratch [unit][part][rank][token][128].  The one that arrives last adds them, in the order of the parts,
  // and goes on to the epilogue: nobody waits for another pair, so it does not matter which of them are resident.
  int full, parts;
  float *scratch;
  int *flags;            // [unit][rank] arrivals, zero before and after a launch
};

__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void pair_load(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void pair_load_nohint(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void pair_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// arrives on the barrier at this offset in both CTAs once every MMA issued so far is done
__device__ __forceinline__ void pair_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "h"((unsigned short)3)
               : "memory");
}

// AND over the 256 epilogue threads (named barrier 1): keeps their control flow uniform
__device__ __forceinline__ bool pair_epilogue_all(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, 1, 256, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred)
      : "memory");
  return r != 0;
}

template <bool GU>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap w_map0, const __grid_constant__ CUtensorMap w_map1,
                 const __grid_constant__ CUtensorMap w_map2, const __grid_constant__ CUtensorMap x_map, const PairParams q) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t bar_full[kPairStages], bar_empty[kPairStages], acc_full[2], acc_empty[2];
  __shared__ uint32_t s_tmem_base;
  __shared__ float s_scale[TILE_N];
  const GemmParams &p = q.g;
  pdl_trigger();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = blockIdx.x & 1u;
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int R = p.tile_rows, NN = 2 * p.Mp, x_bytes = p.Mp * TILE_K * 2;
  const int stage_bytes = W_TILE_BYTES + x_bytes;
  // bytes that the copies of both CTAs bring into a stage
  const uint32_t stage_tx = 2u * (uint32_t)((GU ? 2 : 1) * R * TILE_K * 2 + x_bytes);
  uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < 2 * NN) tmem_cols <<= 1;

  if (tid == 0) {
    tma_prefetch_desc(&w_map0);
    tma_prefetch_desc(&x_map);
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 16);   // eight epilogue warps of both CTAs
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // both CTAs' barriers are set up
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem_base = s_tmem_base;

  // the n-th unit of this pair: this CTA's weight tile, k-blocks, slab; part of a shared unit
  struct Unit {
    int tile, kb0, kb1, split, slab, part, shared;   // shared: index among the shared units, -1: not one
  };
  const int n_full = q.parts > 1 ? q.full / n_pairs : (q.n_units - pair + n_pairs - 1) / n_pairs;
  const int n_local = n_full + (q.parts > 1 && pair < (q.n_units - q.full) * q.parts ? 1 : 0);
  auto unit_of = [&](int n) {
    Unit t;
    t.part = 0;
    t.shared = -1;
    int u = pair + n * n_pairs;
    if (n >= n_full) {
      t.shared = pair / q.parts;
      t.part = pair - t.shared * q.parts;
      u = q.full + t.shared;
    }
    t.slab = u % p.n_slabs;
    const int v = u / p.n_slabs;
    t.split = v % p.splits;
    t.tile = (v / p.splits) * 2 + (int)rank;
    const int at = t.shared >= 0 ? t.part : t.split, of = t.shared >= 0 ? q.parts : p.splits;
    t.kb0 = (int)(((long)at * p.k_blocks) / of);
    t.kb1 = (int)(((long)(at + 1) * p.k_blocks) / of);
    return t;
  };
  auto mat_of = [&](int tile) { return GU ? 0 : tile < p.tile_end[0] ? 0 : tile < p.tile_end[1] ? 1 : 2; };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (each CTA its half)
    uint64_t policy;   // several slabs read a weight tile again from L2
    if (p.n_slabs > 1) asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
    else asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    const uint32_t full0 = cluster_addr(&bar_full[0], 0), smem0 = smem_u32(smem);
    struct Src {
      const CUtensorMap *map;
      int row;
    };
    auto src_of = [&](const Unit &t) {   // (a tile past the last: rows outside the matrix, filled with zeros)
      const int mat = mat_of(t.tile);
      return Src{mat == 0 ? &w_map0 : mat == 1 ? &w_map1 : &w_map2, (t.tile - (mat ? p.tile_end[mat - 1] : 0)) * R};
    };
    auto load_w = [&](const Src &c, int kb, int s) {
      const uint32_t dst = smem0 + s * stage_bytes, bar = full0 + s * 8;
      if (rank == 0) mbar_expect_tx(&bar_full[s], stage_tx);
      pair_load(dst, c.map, kb * TILE_K, c.row, bar, policy);
      if (GU) pair_load(dst + W_TILE_BYTES / 2, &w_map1, kb * TILE_K, c.row, bar, policy);
    };
    // the weights do not depend on the preceding kernel: those of the first stages are fetched before the wait
    int pre = 0, it = 0;
    if (n_local > 0) {
      const Unit t = unit_of(0);
      const Src c = src_of(t);
      for (; pre < p.stages && t.kb0 + pre < t.kb1; ++pre) {
        if (elect_one()) load_w(c, t.kb0 + pre, pre);
        __syncwarp();
      }
    }
    pdl_wait();
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int n = 0; n < n_local && ok; ++n) {
      const Unit t = unit_of(n);
      const Src c = src_of(t);
      const int x_row = (rank ? p.x_lo_row : 0) + t.slab * p.Mp;
      for (int kb = t.kb0; kb < t.kb1; ++kb, ++it) {
        if (it >= pre && !warp_wait(&bar_empty[s], ph ^ 1u)) { ok = false; break; }
        if (elect_one()) {
          if (it >= pre) load_w(c, kb, s);
          pair_load_nohint(smem0 + s * stage_bytes + W_TILE_BYTES, &x_map, kb * TILE_K, x_row, full0 + s * 8);
        }
        __syncwarp();
        if (++s == p.stages) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok) {   // leave no copy in flight: they are short, give them ample time
      if (lane == 0) atomicExch(p.status, 1);
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 20000000ull) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (rank 0 for the pair)
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      const uint64_t desc0 = umma_desc_sw128(0);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int n = 0; n < n_local && ok; ++n) {
        const Unit t = unit_of(n);
        const int buf = n & 1;
        if (!warp_wait(&acc_empty[buf], ((n >> 1) & 1) ^ 1u)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d = tmem_base + buf * NN;
        for (int kb = t.kb0; kb < t.kb1; ++kb) {
          if (!warp_wait(&bar_full[s], ph)) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
            const uint32_t at = smem_u32(smem + s * stage_bytes);
            const uint64_t a = desc0 | (uint64_t)(at >> 4), b = desc0 | (uint64_t)((at + W_TILE_BYTES) >> 4);
#pragma unroll
            for (int k = 0; k < TILE_K / UMMA_K; ++k) pair_mma(d, a + k * 2, b + k * 2, idesc, !(kb == t.kb0 && k == 0));
            pair_commit(&bar_empty[s]);
          }
          __syncwarp();
          if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
        if (ok && elect_one()) pair_commit(&acc_full[buf]);
        __syncwarp();
      }
      if (!ok && lane == 0) atomicExch(p.status, 2);
    }
  } else {
    // ------------------------------------------------------------------ epilogue warps (2..9): two groups of four, 16 tokens in turn
    const int quarter = warp & 3, row = quarter * 32 + lane, grp = (warp - 2) >> 2, e = (tid - 64) & 127;
    float *ex = reinterpret_cast<float *>(smem + p.stages * stage_bytes) + grp * TILE_N * (kExTokens + 1);   // GU: [128][kExTokens + 1]
    pdl_wait();   // the planes may still be read, and the row scales written, by the preceding kernel
    int have_slab = -1;
    for (int n = 0; n < n_local; ++n) {
      const Unit t = unit_of(n);
      const int buf = n & 1, m_base = t.slab * p.Mp;
      if ((p.ss_part || GU) && have_slab != t.slab) {   // RMS scale of the slab's token rows
        have_slab = t.slab;
        pair_epilogue_all(true);
        if (grp == 0) {
          float sc = 1.0f;
          if (p.ss_part && e < p.Mp && m_base + e < p.M) {
            float tot = 0.0f;
#pragma unroll 8
            for (int jj = 0; jj < p.n_part; ++jj) tot += __ldg(p.ss_part + (size_t)(m_base + e) * p.n_part + jj);
            sc = rsqrtf(tot * p.inv_d + p.eps);
          }
          s_scale[e] = sc;
        }
        pair_epilogue_all(true);
      }
      if (!pair_epilogue_all(warp_wait(&acc_full[buf], (n >> 1) & 1))) {
        if (tid == 64) atomicExch(p.status, 3);
        break;
      }
      tc_fence_after();
      const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * NN;
      const int mat = mat_of(t.tile), m_left = min(p.M - m_base, p.Mp);   // (the last 16 tokens of a slab may be eight)
      const size_t piece = (size_t)2 * p.Mp * TILE_N;
      float *share = q.scratch + (size_t)(t.shared < 0 ? 0 : t.shared) * q.parts * piece + (size_t)rank * p.Mp * TILE_N + row;
      bool finish = true, gather = false;   // this CTA does the unit's epilogue; from the parts' sums
      if (t.shared >= 0) {
        float *dst = share + t.part * piece;
        for (int m0 = grp * 16; m0 < p.Mp; m0 += 32) {
          uint32_t hi[16], lo[16];
          tmem_ld16_issue(t_addr + m0, hi);
          tmem_ld16_issue(t_addr + p.Mp + m0, lo);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (i < 8 || m0 + 8 < p.Mp) dst[(size_t)(m0 + i) * TILE_N] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
        }
        __threadfence();
        pair_epilogue_all(true);
        bool last = true;
        if (tid == 64) {
          int *flag = q.flags + t.shared * 2 + rank;
          last = atomicAdd(flag, 1) == q.parts - 1;
          if (last) *flag = 0;
          __threadfence();
        }
        finish = gather = pair_epilogue_all(last);
      }
      // 16 tokens of this thread's row: hi + lo plane, or the sums of a shared unit's parts
      auto sums = [&](int m0, float *v) {
        if (gather) {   // all loads in flight at once: one round trip per 16 tokens
          float w[kShareParts][16];
#pragma unroll
          for (int k = 0; k < kShareParts; ++k)
#pragma unroll
            for (int i = 0; i < 16; ++i) w[k][i] = k < q.parts && (i < 8 || m0 + 8 < p.Mp) ? __ldcg(share + k * piece + (size_t)(m0 + i) * TILE_N) : 0.0f;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            v[i] = w[0][i];
#pragma unroll
            for (int k = 1; k < kShareParts; ++k) v[i] += w[k][i];
          }
          return;
        }
        uint32_t hi[16], lo[16];
        tmem_ld16_issue(t_addr + m0, hi);
        tmem_ld16_issue(t_addr + p.Mp + m0, lo);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
      };
      if (!finish) {
        // (another pair finishes this unit)
      } else if (GU) {
        // MMA rows 0..63 hold gate features, rows 64..127 the same features of the up matrix: they meet in shared memory, 16
        // tokens at a time; then thread e finishes feature e % 64 for every second token
        const int fr = e & 63, f = t.tile * R + fr, odd = e >> 6;
        const bool live = fr < R && f < p.F;
        for (int m0 = grp * 16; m0 < p.Mp; m0 += 32) {
          float a[16];
          sums(m0, a);
#pragma unroll
          for (int i = 0; i < 16; ++i) ex[row * (kExTokens + 1) + i] = a[i] * s_scale[m0 + i];
          asm volatile("bar.sync %0, 128;" ::"r"(grp + 2) : "memory");
          if (live) {
            __nv_bfloat16 *dst = p.act_hi + (size_t)(m_base + m0 + odd) * p.F + f;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float g = ex[fr * (kExTokens + 1) + 2 * i + odd], up = ex[(64 + fr) * (kExTokens + 1) + 2 * i + odd];
              v[i] = g / (1.0f + expf(-g)) * up;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if (m0 + odd + 2 * i >= m_left) break;
              const __nv_bfloat16 vh = __float2bfloat16_rn(v[i]);
              dst[(size_t)(2 * i) * p.F] = vh;
              dst[p.act_lo_off + (size_t)(2 * i) * p.F] = __float2bfloat16_rn(v[i] - __bfloat162float(vh));
            }
          }
          asm volatile("bar.sync %0, 128;" ::"r"(grp + 2) : "memory");
        }
      } else {
        const int n_local = (t.tile - (mat ? p.tile_end[mat - 1] : 0)) * R + row;
        const int col = p.col_off[mat] + n_local;
        const bool live = t.tile < q.tiles && row < R && n_local < p.n_out[mat];
        float *plane = reinterpret_cast<float *>(p.out) + (size_t)t.split * p.plane_stride + (size_t)m_base * p.ldc + col;
        __nv_bfloat16 *logits = reinterpret_cast<__nv_bfloat16 *>(p.out) + (size_t)m_base * p.ldc + col;
        for (int m0 = grp * 16; m0 < p.Mp; m0 += 32) {
          float v[16];
          sums(m0, v);
          if (!live) continue;
          const float *scale = p.ss_part ? s_scale + m0 : nullptr;
          if (p.store_bf16) store_column(logits + (size_t)m0 * p.ldc, p.ldc, v, scale, m_left - m0);
          else store_column(plane + (size_t)m0 * p.ldc, p.ldc, v, scale, m_left - m0);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0)   // the accumulator is free (rank 0 issues into both CTAs' tensor memory)
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr(&acc_empty[buf], 0)) : "memory");
    }
  }

  tc_fence_before();
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // neither CTA leaves while the other may reach into it
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// plain sum of split planes (sjd_gemm): out[m][n] (+)= sum_s P[s][m][n]; V: entries per thread (4 when out is 16-byte aligned)
template <typename V>
__global__ void sum_planes_kernel(const float *__restrict__ planes, size_t plane_stride, int splits, float *__restrict__ out,
                                  size_t total, int accumulate) {
  pdl_wait();
  constexpr int E = sizeof(V) / 4;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total / E; i += (size_t)gridDim.x * blockDim.x) {
    float acc[E] = {};
    for (int s = 0; s < splits; ++s) {
      const V v = __ldcg(reinterpret_cast<const V *>(planes + (size_t)s * plane_stride) + i);
      const float *f = reinterpret_cast<const float *>(&v);
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] += f[e];
    }
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = accumulate ? out[i * E + e] + acc[e] : acc[e];
    *(reinterpret_cast<V *>(out) + i) = *reinterpret_cast<const V *>(acc);
  }
}

}  // namespace

// bf16 row-major [rows][cols] matrix viewed as boxes of box_rows x 64 columns with 128-byte swizzle
int make_tensor_map_bf16(TensorMap *out, const void *base, long rows, long cols, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return SJD_ERR_UNSUPPORTED;
  if (((uintptr_t)base & 15u) != 0 || (cols * 2) % 16 != 0 || box_rows < 1 || box_rows > 256) return SJD_ERR_UNSUPPORTED;
  static_assert(sizeof(TensorMap) == sizeof(CUtensorMap), "tensor map size");
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)TILE_K, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(reinterpret_cast<CUtensorMap *>(out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base),
                        dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        SJD_GEMM_L2_PROMO, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? SJD_OK : SJD_ERR_CUDA;
}

bool gemm_tc_supported(int M, int N, int K) { return M >= 1 && M <= 1024 && N % TILE_N == 0 && K % TILE_K == 0; }

// How M token rows are laid over the MMA N dimension (at most 256 columns per accumulator, two per token
// row: hi and lo plane): slabs of at most 128 rows, in steps of 16 for one CTA per tile and of 8 for CTA pairs, whose CTAs hold a
// plane each (the tensor pipe is their bound: 200 rows are two slabs of 104 and not of 112).
GemmTcPlan gemm_tc_plan(int M) {
  GemmTcPlan pl;
  pl.n_slabs = (M + 127) / 128;
  const int per = (M + pl.n_slabs - 1) / pl.n_slabs, step = M > 64 ? 8 : 16;
  pl.slab_rows = (per + step - 1) / step * step;
  return pl;
}

// K splits for a launch of `tiles` weight tiles.  Few rows: a single wave of the resident CTAs (two per SM), at least
// SJD_GEMM_MIN_KB k-blocks per CTA so that set-up and drain stay small next to the streaming.  Many rows (CTA pairs): the split
// with the shortest schedule, counted in k-blocks of a full tile (0.27 us): rounds of the grid, about three k-blocks of
// ramp per round, and the traffic of the planes through L2.
int gemm_tc_splits(const GemmTcPlan &pl, int tiles, int k_blocks, int n_sms) {
  const int sms = n_sms < 132 ? 132 : n_sms > 160 ? 160 : n_sms;   // the range scratch is sized for
  if (gemm_tc_pairs(pl)) {
    const int units = (tiles + 1) / 2 * pl.n_slabs, pairs = sms / 2;
    const double per_kb = pl.slab_rows / 128.0, plane = (double)tiles * 128.0 * pl.n_slabs * pl.slab_rows * 8.0 / 2.7e6;
    int best = 1;
    double best_cost = 0.0;
    for (int s = 1; s <= 16 && s * 4 <= k_blocks; ++s) {
      const int rounds = (units * s + pairs - 1) / pairs;
      const double cost = rounds * ((k_blocks + s - 1) / s + 3) * per_kb + s * plane;
      if (s == 1 || cost < best_cost) {
        best = s;
        best_cost = cost;
      }
    }
    return best;
  }
  const int ctas = tiles * pl.n_slabs;
  int s = (SJD_GEMM_CTAS_PER_SM * n_sms) / (ctas > 0 ? ctas : 1);
  const int cap = k_blocks / SJD_GEMM_MIN_KB > 1 ? k_blocks / SJD_GEMM_MIN_KB : 1;
  s = s > cap ? cap : s;
  s = s > 16 ? 16 : s;
  return s < 1 ? 1 : s;
}
size_t gemm_tc_share_floats() { return (size_t)(160 / 2) * 2 * 128 * TILE_N; }   // a shared part per pair: 128 tokens of both CTAs

int gemm_tc_splits_max(const GemmTcPlan &pl, int tiles, int k_blocks) {
  int most = 1;
  for (int sms = 132; sms <= 160; sms += 2) {
    const int s = gemm_tc_splits(pl, tiles, k_blocks, sms);
    most = s > most ? s : most;
  }
  return most;
}

// every kernel here may ask for as much shared memory as its largest launch needs; set once per device
static int allow_gemm_smem() {
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  SJD_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SJD_ERR_UNSUPPORTED;
  if (done.load() >> dev & 1) return SJD_OK;
  constexpr size_t kMost = (kDeepRing > kSmemBudget ? kDeepRing : kSmemBudget) + sizeof(TcShared);
  int rc = allow_smem(gemm_tc_kernel<false>, kMost);
  if (rc == SJD_OK) rc = allow_smem(gemm_tc_kernel<true>, kMost);
  if (rc == SJD_OK) rc = allow_smem(gemm_pair_kernel<false>, kPairSmem);
  if (rc == SJD_OK) rc = allow_smem(gemm_pair_kernel<true>, kPairSmem);
  if (rc == SJD_OK) done.fetch_or(1ull << dev);
  return rc;
}

// Stages of the two rings of a gemm_tc_kernel CTA.  Weights come from HBM and want as many bytes in flight as there is room for;
// activations come from L2, but under the stream of weights that still takes two to three k-blocks.  Two CTAs of an SM have to
// leave a few KB: without them no CTA of the next kernel can wait beside them, and its launch and the weights that it
// prefetches come late.  us of a step of 16 layers, stages of weights + activations: 7B, 32 rows: 6 + 2 (no
// room left) 1755, 5 + 2 1696, 4 + 3 1663, 5 + 3 1646, 4 + 4 1670; 64 rows: 3 + 3 1946, 4 + 2 1905, 4 + 3 (no room left) 1937.
// 48 rows, two layers and the logits: 7B 5 + 2 344, 4 + 3 338; 8B 570 and 559.  Where K is split a CTA has 8 to 24 k-blocks, and the
// room is worth more than the fifth stage (7B, 32 rows, two layers and the logits 311, with 4 + 3 there 307; sjd_gemm
// 32 x 4096 x 4096 12.2 and 11.7, one ring for both operands 11.6).
// At most one CTA per SM (small models, short K): both rings hold all or much of K.
void ring_stages(bool deep, bool split, int x_bytes, int *stages, int *x_stages) {
  if (deep) {
    const int n = kDeepRing / (W_TILE_BYTES + x_bytes);
    *stages = *x_stages = n > kMaxStages ? kMaxStages : n;
    return;
  }
  *x_stages = x_bytes <= W_TILE_BYTES * 3 / 4 ? 3 : 2;
  const int n = (kSmemBudget - *x_stages * x_bytes) / W_TILE_BYTES, most = split ? 4 : kMaxStages;
  *stages = n > most ? most : n;
}

static int launch_gemm_pair(const GemmTcCall &g, const GemmParams &p, int tiles, cudaStream_t stream) {
  PairParams q;
  q.g = p;
  q.tiles = tiles;
  // the second half of a last pair without a tile is the tile past the last matrix: zeros, not rows of a matrix once more
  for (int j = g.n_mats - 1; j < 3; ++j) q.g.tile_end[j] += tiles & 1;
  q.n_units = (tiles + 1) / 2 * p.n_slabs * p.splits;
  const bool gu = g.act_hi != nullptr;
  const int stage_bytes = W_TILE_BYTES + p.Mp * TILE_K * 2;
  const int ex = gu ? 2 * TILE_N * (kExTokens + 1) * 4 : 0;
  const int budget = kPairSmem - 1024 - ex;
  int stages = budget / stage_bytes;
  stages = stages > kPairStages ? kPairStages : stages;
  q.g.stages = stages;
  const size_t smem = (size_t)stages * stage_bytes + 1024 + ex;
  const CUtensorMap &w0 = reinterpret_cast<const CUtensorMap &>(*g.w_map[0]);
  const CUtensorMap &w1 = reinterpret_cast<const CUtensorMap &>(*g.w_map[g.n_mats > 1 ? 1 : 0]);
  const CUtensorMap &w2 = reinterpret_cast<const CUtensorMap &>(*g.w_map[g.n_mats > 2 ? 2 : 0]);
  const CUtensorMap &xm = reinterpret_cast<const CUtensorMap &>(*g.x_map);
  auto kernel = gu ? gemm_pair_kernel<true> : gemm_pair_kernel<false>;
  const int sms = g.n_sms > 1 ? g.n_sms : 148;
  // The units of a partial last round are shared where K may not be split otherwise and the launch has few rounds: one token slab
  // (7B gate|up at 128 rows: 86 units for 74 pairs, 2 rounds without, 1.25 with; 8 layers 1131 -> 1084 us at 80 rows, 1280 ->
  // 1240 at 128; at 192 and 256 rows, 3 rounds against 2.4, nothing to 2 % slower).
  int pairs = sms / 2;
  q.full = q.n_units / pairs * pairs;
  const int tail = q.n_units - q.full;
  q.parts = tail > 0 ? pairs / tail : 1;
  if (q.parts > p.k_blocks / 4) q.parts = p.k_blocks / 4;
  if (q.parts > kShareParts) q.parts = kShareParts;
  q.scratch = g.share;
  q.flags = g.share_flags;
  if (!g.share || p.splits != 1 || p.n_slabs > 1 || q.parts < 2) {
    q.parts = 1;
    pairs = q.n_units < pairs ? q.n_units : pairs;
  }
  SJD_CUDA(launch_kernel(kernel, dim3(2 * pairs), dim3(kPairThreads), smem, stream, w0, w1, w2, xm, q));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

int launch_gemm_tc(const GemmTcCall &g, cudaStream_t stream) {
  if (g.n_mats < 1 || g.n_mats > 3 || g.splits < 1) return SJD_ERR_BAD_ARG;
  GemmParams p;
  memset(&p, 0, sizeof(p));
  const bool gu = g.act_hi != nullptr;
  const int R = g.tile_rows > 0 ? g.tile_rows : TILE_N;
  if (R > TILE_N || (gu && (R > TILE_N / 2 || g.n_mats != 2 || g.n_out[0] != g.n_out[1] || g.splits != 1)))
    return SJD_ERR_BAD_ARG;
  int tiles = 0;
  for (int j = 0; j < 3; ++j) {
    if (j < g.n_mats && !(gu && j == 1)) {
      if (g.M < 1 || g.K % TILE_K != 0 || g.n_out[j] < 1) return SJD_ERR_UNSUPPORTED;
      if (R == TILE_N && g.n_out[j] % TILE_N != 0) return SJD_ERR_UNSUPPORTED;
      tiles += (g.n_out[j] + R - 1) / R;
    }
    p.tile_end[j] = tiles;
    p.col_off[j] = j < g.n_mats ? g.col_off[j] : 0;
    p.n_out[j] = j < g.n_mats ? g.n_out[j] : 0;
  }
  if (g.store_bf16 && g.splits != 1) return SJD_ERR_BAD_ARG;
  p.out = g.out;
  p.plane_stride = g.plane_stride;
  p.ldc = g.ldc;
  const GemmTcPlan pl = gemm_tc_plan(g.M);
  p.M = g.M;
  p.Mp = pl.slab_rows;
  p.n_slabs = pl.n_slabs;
  p.x_lo_row = g.x_lo_row;
  p.k_blocks = g.K / TILE_K;
  p.splits = g.splits;
  p.store_bf16 = g.store_bf16;
  p.status = g.status;
  p.ss_part = g.ss_part;
  p.n_part = g.n_part;
  p.inv_d = g.inv_d;
  p.eps = g.eps;
  p.tile_rows = R;
  p.act_hi = g.act_hi;
  p.act_lo_off = g.act_lo_off;
  p.F = gu ? g.n_out[0] : 0;
  const int rc = allow_gemm_smem();
  if (rc != SJD_OK) return rc;
  if (gemm_tc_pairs(pl)) return launch_gemm_pair(g, p, tiles, stream);
  const int x_bytes = 2 * p.Mp * TILE_K * 2;
  const int ctas = tiles;
  const bool deep = g.n_sms > 0 && ctas * g.splits <= g.n_sms;
  ring_stages(deep, g.splits > 1, x_bytes, &p.stages, &p.x_stages);
  const size_t smem = (size_t)p.stages * W_TILE_BYTES + (size_t)p.x_stages * x_bytes + sizeof(TcShared);
  const CUtensorMap &w0 = reinterpret_cast<const CUtensorMap &>(*g.w_map[0]);
  const CUtensorMap &w1 = reinterpret_cast<const CUtensorMap &>(*g.w_map[g.n_mats > 1 ? 1 : 0]);
  const CUtensorMap &w2 = reinterpret_cast<const CUtensorMap &>(*g.w_map[g.n_mats > 2 ? 2 : 0]);
  const CUtensorMap &xm = reinterpret_cast<const CUtensorMap &>(*g.x_map);
  const dim3 grid(ctas, g.splits);
  if (gu)
    SJD_CUDA(launch_kernel(gemm_tc_kernel<true>, grid, dim3(kThreads), smem, stream, w0, w1, w2, xm, p));
  else
    SJD_CUDA(launch_kernel(gemm_tc_kernel<false>, grid, dim3(kThreads), smem, stream, w0, w1, w2, xm, p));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

int launch_sum_planes(const float *planes, size_t plane_stride, int splits, float *out, size_t total, int accumulate,
                      cudaStream_t stream) {
  const bool vec = ((uintptr_t)out & 15u) == 0 && total % 4 == 0 && plane_stride % 4 == 0;
  const size_t groups = vec ? total / 4 : total;
  const int blocks = (int)((groups + 255) / 256 < 1184 ? (groups + 255) / 256 : 1184);
  auto kernel = vec ? sum_planes_kernel<float4> : sum_planes_kernel<float>;
  SJD_CUDA(launch_kernel(kernel, dim3(blocks), dim3(256), 0, stream, planes, plane_stride, splits, out, total, accumulate));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

}  // namespace sjd
