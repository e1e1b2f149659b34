// One forward pass of a few dozen rows as ONE cooperative launch (Sec. 4.1 Step 2): embedding, every decoder layer and
// the logits projection, one CTA per SM.
//
// What bounds it: a pass of M = batch * window <= 64 rows has to stream every weight once (13.5 GB at the 7B shapes:
// 2.09 ms at the measured copy bandwidth) through a chain of about nine dependent steps per layer.  As separate launches
// (fused_kernels.cu, gemm_tc.cu, attention_mma.cu; still used for more rows) every link of that chain costs 4 to 7 us
// however little it does, and HBM idles meanwhile.  Here the weight stream never waits for the chain: a producer warp runs
// through the weight tiles of the whole pass in order, held back only by the space in its ring of shared memory
// (about 145 KB per SM, 21 MB in all: 3.3 us of HBM time that fills while the chain is between two projections).
//
//   warp 0      weight producer: TMA into the ring, all layers, no dependency on activations (the CTAs walk K in step: their
//               128-byte row pieces then share 256-byte fetches and DRAM pages; each starting at another k-block was 1.2 % slower)
//   warp 1      activation producer: hi/lo planes of the current projection's input once the grid has finished it;
//               K/V tiles during attention
//   warp 2      issues tcgen05.mma (weights = the 128-row operand, hi and lo planes of the tokens = N columns)
//   warp 3      allocates tensor memory
//   warps 4-11  "workers": accumulator epilogues, and between the projections the residual, rotary / append, attention
//               and merge steps, spread over the whole grid; they also carry the grid barriers
//
// Work split.  A weight tile has up to 2 * h rows (two accumulators when more than 128); h is such that the gate|up
// projection gives every CTA one tile of ceil(F / #SMs) gate rows and the same up rows over the whole K (a thread of the epilogue then
// holds both and applies SwiGLU).  The other projections cut tiles * k-blocks evenly over the CTAs; a tile's pieces
// are fp32 planes that the consumer adds in order (deterministic, no atomics).  Short ones (K <= 2048) and the logits
// projection deal whole tiles.
//
// Every wait is bounded (2 s).  A wait that runs out sets the status word and a CTA-wide flag; from then on all waits
// of the CTA return at once and nothing is issued any more, so that control flow (and the named barriers) stay uniform to
// the end, where the copies in flight are waited for and the tensor memory is freed.
#include <cuda.h>
#include <string.h>

#include "common.cuh"

namespace sjd {
SJD_TIMELINE_TU(pass)
// timeline builds: CTA 0's first worker stamps every step of the chain, before and after the grid barriers
#ifdef SJD_TIMELINE
#define PASS_TL(tag_, phase_)                                                               \
  do {                                                                                      \
    if (x.c == 0 && x.w == 0 && x.lane == 0 && g_tl_buf && g_tl_buf->n < (1u << 16)) {       \
      const unsigned int i_ = g_tl_buf->n++;                                                \
      g_tl_buf->rec[i_].t = now_ns();                                                       \
      g_tl_buf->rec[i_].tag = tag_;                                                         \
      g_tl_buf->rec[i_].phase = phase_;                                                     \
    }                                                                                       \
  } while (0)
#else
#define PASS_TL(tag, phase) do { } while (0)
#endif
namespace {

constexpr int kWorkers = 256, kPassThreads = 128 + kWorkers;
constexpr int kMaxW = 16;
constexpr int kKvSlots = 8, kKvKeys = 16;          // attention: slots of 16 keys
constexpr int kXRegion = 64 * 1024;                // activation ring; K/V slots and exchange buffer during attention
constexpr unsigned long long kPassWaitNs = 2000000000ull, kDrainNs = 20000000ull;

// ---------------------------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t s32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint64_t *b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(b)), "r"(n));
}
__device__ __forceinline__ void bar_expect(uint64_t *b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s32(b)) : "memory");
}
__device__ __forceinline__ bool bar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
struct Life {            // the CTA's "a wait ran out" flag and the context's status word
  volatile int *dead;    // shared
  int *status;           // global
};
// The code of a pass runs once per layer from a cold instruction cache: what is not hot inside a loop is kept out of line or
// in a single place (inlined everywhere, the kernel was 357 KB and the steps between the projections took up to twice as long).
__device__ __noinline__ void life_fail(volatile int *dead, int *status, int code) {
  *dead = 1;
  atomicExch(status, code);
}
__device__ __noinline__ bool bar_wait_slow(uint32_t bar, uint32_t parity, volatile int *dead, int *status, int code) {
  const unsigned long long t0 = now_ns();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (bar_test(bar, parity)) return true;
    if (*dead) return false;
    if (now_ns() - t0 > kPassWaitNs) {
      life_fail(dead, status, code);
      return false;
    }
  }
}
__device__ __forceinline__ bool bar_wait(uint64_t *b, uint32_t parity, const Life &life, int code) {
  if (bar_test(s32(b), parity)) return true;
  return bar_wait_slow(s32(b), parity, life.dead, life.status, code);
}
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
__device__ __forceinline__ void fence_proxy() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(s32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_2d_hint(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint64_t *bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(s32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(s32(bar))
      : "memory");
}
// shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(bar)) : "memory");
}
__device__ __forceinline__ void fence_tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t *r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t *r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t *r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_trans(uint32_t addr, uint32_t *r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float *c, const uint32_t *a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// two floats -> packed bf16 hi pair and bf16 lo pair (lo = value - hi, rounded)
__device__ __forceinline__ void split2(float x, float y, uint32_t &hi, uint32_t &lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const float2 f = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}

__device__ __forceinline__ KvLayout pass_kv(const PassParams &p, int l) {
  KvLayout kv;
  kv.n_kv_heads = p.n_kv_heads;
  kv.max_seq = p.max_seq;
  kv.head_dim = p.head_dim;
  kv.layer = l;
  kv.n_layers = p.n_layers;
  kv.page_table = p.page_table;
  kv.pages_per_seq = p.pages_per_seq;
  kv.base = reinterpret_cast<__nv_bfloat16 *>(p.kv_base) + (p.page_table ? 0 : (size_t)l * p.planes_per_layer * p.max_seq * p.head_dim);
  return kv;
}

enum PassKind { PK_QKV = 0, PK_O = 1, PK_GU = 2, PK_DOWN = 3, PK_LOGITS = 4 };
// ---------------------------------------------------------------------------------- work schedule
struct Seg {
  int tile, kb0, kb1, piece;
};
// the pieces of one projection that a CTA computes, in order; every role of the CTA walks the same list
struct SegIter {
  int u, end, kb, step, full, U, G, c;
  __device__ void init(const PassGemm &g, int cta, int n_ctas) {
    kb = g.kb;
    full = g.full;
    G = n_ctas;
    c = cta;
    if (full) {
      u = cta;
      end = g.tiles;
    } else {
      U = g.tiles * g.kb;
      u = U * cta / n_ctas;
      end = U * (cta + 1) / n_ctas;
    }
  }
  __device__ bool next(Seg &s) {
    if (u >= end) return false;
    if (full) {
      s = Seg{u, 0, kb, 0};
      u += G;
    } else {
      s.tile = u / kb;
      s.kb0 = u - s.tile * kb;
      s.kb1 = min(kb, s.kb0 + (end - u));
      s.piece = c - ((s.tile * kb + 1) * G - 1) / U;
      u += s.kb1 - s.kb0;
    }
    return true;
  }
};
// Where column `col` of a projection's output lies in the partial planes: piece 0 of row 0, and the pieces.  From a host-made
// table with an entry per 8 columns (tile heights are multiples of 8): {tile * max_pieces, row in the tile | pieces << 16}.
struct Where {
  const float *p;
  int n;
};
__device__ __forceinline__ Where locate(const PassParams &p, const int2 *loc, int col) {
  const int2 e = __ldg(loc + (col >> 3));
  return Where{p.part + (size_t)e.x * (p.M * p.part_ld) + (e.y & 0xFFFF) + (col & 7), e.y >> 16};
}

// ---------------------------------------------------------------------------------- shared state
struct PassShared {
  uint64_t full[kMaxW], empty[kMaxW], acc_full[2], acc_empty[2];   // full: the weight and the activation part of a block have landed
  uint64_t kvfull[kKvSlots], kvempty[kKvSlots], qfull;
  uint32_t tmem;
  int dead;
  uint32_t ready;   // inputs the workers have released to the activation producer so far
  int pos[64], len[64], seq[64];
  float scale[64];
  float2 ml[128];   // attention: maximum and sum of every (key group, row)
};

struct Ctx {
  const PassParams &p;
  PassShared &sh;
  uint32_t wring, xring;   // shared addresses
  uint8_t *xptr;
  int c, G, w, lane;       // CTA, CTAs, warp of the role's group, lane
  Life life;
};

// Grid barrier, carried by the workers: everything written before it (by any thread of any worker group) is visible
// after it; TMA reads of it follow a proxy fence of the activation producer (wait_ready).  `target` is the arrival count that completes it.
__device__ __noinline__ void grid_sync_at(uint32_t *counter, uint32_t target, bool leader, volatile int *dead, int *status) {
  workers_sync();
  if (leader && !*dead) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
    uint32_t v;
    unsigned long long t0 = 0;
#pragma unroll 1
    for (int i = 0;; ++i) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((i & 255) == 255) {
        if (t0 == 0) t0 = now_ns();
        if (*dead) break;
        if (now_ns() - t0 > kPassWaitNs) {
          life_fail(dead, status, 16);
          break;
        }
      }
    }
  }
  workers_sync();
}
__device__ __forceinline__ void grid_sync(const Ctx &x, uint32_t &target) {
  target += x.G;
  grid_sync_at(x.p.counter, target, x.w == 0 && x.lane == 0, x.life.dead, x.life.status);
}
// lets the activation producer start on the next projection (or attention unit)
__device__ __forceinline__ void signal_ready(const Ctx &x) {
  if (x.w == 0 && x.lane == 0) asm volatile("red.release.cta.shared::cta.add.u32 [%0], 1;" ::"r"(s32(&x.sh.ready)) : "memory");
}
__device__ __forceinline__ void wait_ready(const Ctx &x, uint32_t &seen) {
  ++seen;
  unsigned long long t0 = 0;
  for (int i = 0;; ++i) {
    uint32_t v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(s32(&x.sh.ready)) : "memory");
    if ((int)(v - seen) >= 0 || *x.life.dead) break;
    if ((i & 255) == 255) {
      if (t0 == 0) t0 = now_ns();
      if (now_ns() - t0 > kPassWaitNs) life_fail(x.life.dead, x.life.status, 17);
    }
  }
  fence_proxy();
}

// ---------------------------------------------------------------------------------- residual + gain
// x[m][:] += the pieces of the projection before (or the embedding row), emitted times the norm gain as bf16 hi/lo
// planes, with one partial of sum(x^2) per 128 columns.  One warp per (row, 128 columns): a single round of loads.
__device__ __forceinline__ void resid_gain(const Ctx &x, const int2 *loc, const __nv_bfloat16 *gain) {
  const PassParams &p = x.p;
  const int nch = p.d / 128, n = p.M * nch;
  for (int u = x.c + x.G * x.w; u < n; u += x.G * 8) {
    const int m = u / nch, ch = u - m * nch, col = ch * 128 + x.lane * 4;
    const size_t idx = (size_t)m * p.d + col;
    const uint2 gb = __ldg(reinterpret_cast<const uint2 *>(gain + col));
    float4 v;
    if (loc) {
      const Where w = locate(p, loc, col);
      const float *src = w.p + (size_t)m * p.part_ld;
      const size_t stride = (size_t)p.M * p.part_ld;
      float4 t[kPassMaxPieces];
      v = __ldcg(reinterpret_cast<const float4 *>(p.x + idx));
#pragma unroll
      for (int i = 0; i < kPassMaxPieces; ++i)
        t[i] = i < w.n ? __ldcg(reinterpret_cast<const float4 *>(src + i * stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < kPassMaxPieces; ++i) {
        v.x += t[i].x; v.y += t[i].y; v.z += t[i].z; v.w += t[i].w;
      }
    } else {
      const int tok = min(max(p.in_tok[m], 0), p.vocab - 1);
      const uint2 e = __ldg(reinterpret_cast<const uint2 *>(p.tok_emb + (size_t)tok * p.d + col));
      const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&e.x));
      const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&e.y));
      v = make_float4(a.x, a.y, b.x, b.y);
    }
    *reinterpret_cast<float4 *>(p.x + idx) = v;
    const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gb.x));
    const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&gb.y));
    uint2 hi, lo;
    split2(v.x * g0.x, v.y * g0.y, hi.x, lo.x);
    split2(v.z * g1.x, v.w * g1.y, hi.y, lo.y);
    *reinterpret_cast<uint2 *>(p.h.base + idx) = hi;
    *reinterpret_cast<uint2 *>(p.h.base + p.h.lo_offset + idx) = lo;
    const float ss = warp_sum(v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w);
    if (x.lane == 0) p.ss_part[(size_t)m * nch + ch] = ss;
  }
}
// RMS scale of every row into shared memory (after the barrier that follows resid_gain)
__device__ __forceinline__ void row_scales(const Ctx &x) {
  const PassParams &p = x.p;
  const int nch = p.d / 128;
#pragma unroll 4
  for (int m = x.w; m < p.M; m += 8) {
    float t = 0.0f;
    for (int j = x.lane; j < nch; j += 32) t += __ldcg(p.ss_part + (size_t)m * nch + j);
    t = warp_sum(t);
    if (x.lane == 0) x.sh.scale[m] = rsqrtf(t / (float)p.d + p.eps);
  }
  workers_sync();
}

// ---------------------------------------------------------------------------------- rotary step + cache append
// q, k, v = scale * sum of the pieces; q and k rotated by the row's position; q times log2(e) / sqrt(hd) -> bf16 hi/lo
// planes, k and v -> cache.  One warp per (row, head).  The step is one round trip to L2 under a full load of weight
// copies (about 1.5 us), so the loads of three heads are in flight before the first is used.
template <int HD>
__device__ __forceinline__ void qkv_finish(const Ctx &x, const PassLayer &L, KvLayout kv) {
  const PassParams &p = x.p;
  constexpr int PER = HD / 64;   // adjacent entries of a half head per lane
  constexpr int NU = 3, NP = 4;
  const int H = p.n_heads, KV = p.n_kv_heads, slots = H + 2 * KV, n = p.M * slots;
  __nv_bfloat16 *cache = reinterpret_cast<__nv_bfloat16 *>(kv.base);
  const size_t stride = (size_t)p.M * p.part_ld;
  const int j0 = x.lane * PER;
  for (int u0 = x.c + x.G * x.w; u0 < n; u0 += x.G * 8 * NU) {
    float v[NU][2][PER];
    const float *src[NU][2];
    int np[NU][2], row[NU], slot[NU];
#pragma unroll
    for (int k = 0; k < NU; ++k) {
      const int u = u0 + k * x.G * 8;
      const bool on = u < n;
      row[k] = on ? u / slots : 0;
      slot[k] = on ? u - row[k] * slots : 0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const Where w = locate(p, p.loc_qkv, slot[k] * HD + h * (HD / 2) + j0);
        src[k][h] = w.p + (size_t)row[k] * p.part_ld;
        np[k][h] = on ? w.n : 0;
#pragma unroll
        for (int i = 0; i < PER; ++i) v[k][h][i] = 0.0f;
      }
    }
    for (int q0 = 0; q0 < p.gemm[PK_QKV].max_pieces; q0 += NP) {
      float t[NU][2][NP][PER];
#pragma unroll
      for (int k = 0; k < NU; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            const float *a = src[k][h] + (q0 + q) * stride;
            const bool on = q0 + q < np[k][h];
            if (PER == 2) {
              const float2 f = on ? __ldcg(reinterpret_cast<const float2 *>(a)) : make_float2(0.f, 0.f);
              t[k][h][q][0] = f.x;
              t[k][h][q][PER - 1] = f.y;
            } else {
              t[k][h][q][0] = on ? __ldcg(a) : 0.0f;
            }
          }
#pragma unroll
      for (int k = 0; k < NU; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int i = 0; i < PER; ++i) v[k][h][i] += t[k][h][q][i];
    }
#pragma unroll
    for (int k = 0; k < NU; ++k) {
      const int m = row[k], pos = x.sh.pos[m];
      if (u0 + k * x.G * 8 >= n || pos < 0) continue;
      float *a = v[k][0], *b = v[k][1];
      const float sc = x.sh.scale[m];
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        a[i] *= sc;
        b[i] *= sc;
      }
      const int seq = x.sh.seq[m / p.rows];
      const bool is_q = slot[k] < H, is_v = slot[k] >= H + KV;
      if (!is_v) {
        if (L.q_norm) {
          float ss = 0.0f;
#pragma unroll
          for (int i = 0; i < PER; ++i) ss += a[i] * a[i] + b[i] * b[i];
          const float r = rsqrtf(warp_sum(ss) / (float)HD + p.eps);
          const __nv_bfloat16 *gain = is_q ? L.q_norm : L.k_norm;
#pragma unroll
          for (int i = 0; i < PER; ++i) {
            a[i] *= r * __bfloat162float(gain[j0 + i]);
            b[i] *= r * __bfloat162float(gain[j0 + HD / 2 + i]);
          }
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
          const float2 cs = __ldg(p.rope + (size_t)pos * (HD / 2) + j0 + i);
          const float r1 = a[i] * cs.x - b[i] * cs.y, r2 = b[i] * cs.x + a[i] * cs.y;
          a[i] = r1;
          b[i] = r2;
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float *e = v[k][h];
        const int j = j0 + h * (HD / 2);
        if (is_q) {
          const float f = 1.4426950408889634f * rsqrtf((float)HD);
          uint32_t hi, lo;
          split2(e[0] * f, e[PER - 1] * f, hi, lo);
          __nv_bfloat16 *dst = p.qs.base + (size_t)m * H * HD + slot[k] * HD + j;
          if (PER == 2) {
            *reinterpret_cast<uint32_t *>(dst) = hi;
            *reinterpret_cast<uint32_t *>(dst + p.qs.lo_offset) = lo;
          } else {
            *reinterpret_cast<uint16_t *>(dst) = (uint16_t)hi;
            *reinterpret_cast<uint16_t *>(dst + p.qs.lo_offset) = (uint16_t)lo;
          }
        } else {
          __nv_bfloat16 *dst = cache + kv_row_offset(kv, seq, is_v ? 1 : 0, slot[k] - (is_v ? H + KV : H), pos) + j;
          if (PER == 2) *reinterpret_cast<__nv_bfloat162 *>(dst) = __floats2bfloat162_rn(e[0], e[PER - 1]);
          else dst[0] = __float2bfloat16_rn(e[0]);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------------- attention
// Key ranges of a segment: one while a CTA gets through its keys in about the time a merge would take (four rounds of
// 16 keys per key group), else as many as the grid has room for.
__device__ __forceinline__ int key_chunk(const PassParams &p, int len) {
  const int single = kKvKeys * 4 * p.key_groups;
  if (len <= single || p.splits == 1) return (len + kKvKeys - 1) / kKvKeys * kKvKeys;
  const int c = (len + p.splits - 1) / p.splits;
  return (c + kKvKeys - 1) / kKvKeys * kKvKeys;
}
struct AttUnit {
  int seg, h, split, k0, k1, n_act;
};
__device__ __forceinline__ bool att_unit(const Ctx &x, int u, AttUnit &a) {
  const PassParams &p = x.p;
  a.h = u % p.n_heads;
  const int t = u / p.n_heads;
  a.seg = t % p.n_segs;
  a.split = t / p.n_segs;
  const int len = x.sh.len[a.seg];
  if (len == 0) {                     // a segment without an active row: its rows are zeros, written by split 0
    a.k0 = a.k1 = 0;
    a.n_act = 1;
    return a.split == 0;
  }
  const int chunk = key_chunk(p, len);
  a.n_act = (len + chunk - 1) / chunk;
  a.k0 = a.split * chunk;
  a.k1 = min(len, a.k0 + chunk);
  return a.split < a.n_act;
}

// Shared memory during attention (the activation region): the rows' queries [plane][64-entry half][row][128 B], then the tile
// ring; after the last tile the whole region holds the key groups' outputs.
template <int HD>
struct AttSmem {
  static constexpr int SLOT = kKvKeys * HD * 4, HALF = kKvKeys * 128;   // K then V, each in 64-entry halves
  int q_half, q_bytes, slots;
  __device__ AttSmem(const PassParams &p) {
    q_half = (p.rows + 7) / 8 * 1024;
    q_bytes = 2 * (HD / 64) * q_half;
    const int n = (kXRegion - q_bytes) / SLOT;
    slots = n < kKvSlots ? n : kKvSlots;
  }
};

// activation producer's part of attention: queries and 16-key tiles of this CTA's units
template <int HD>
__device__ __forceinline__ void attention_loads(const Ctx &x, int plane0, KvLayout kv, uint32_t &ready_n, int &kv_slot, uint32_t &kv_phase,
                                                bool &alive) {
  const PassParams &p = x.p;
  using S = AttSmem<HD>;
  const S sm(p);
  const int n_units = p.n_heads * p.n_segs * p.splits;
  for (int u = x.c; u < n_units; u += x.G) {
    AttUnit a;
    if (!att_unit(x, u, a)) continue;
    wait_ready(x, ready_n);
    const int seq = x.sh.seq[a.seg], kvh = a.h / (p.n_heads / p.n_kv_heads);
    const int n_tiles = (a.k1 - a.k0 + kKvKeys - 1) / kKvKeys;
    if (alive && elect_one()) {
      bar_expect(&x.sh.qfull, 2 * (HD / 64) * p.rows * 128);
#pragma unroll
      for (int i = 0; i < 2 * (HD / 64); ++i)
        tma_2d(x.xring + i * sm.q_half, reinterpret_cast<const CUtensorMap *>(&p.q_map), a.h * HD + (i % (HD / 64)) * 64,
               a.seg * p.rows + (i / (HD / 64)) * p.x_lo_row, &x.sh.qfull);
    }
    for (int t = 0; t < n_tiles; ++t) {
      alive = alive && __all_sync(0xffffffffu, bar_wait(&x.sh.kvempty[kv_slot], ((kv_phase >> kv_slot) & 1u) ^ 1u, x.life, 18));
      kv_phase ^= 1u << kv_slot;
      const uint32_t dst = x.xring + sm.q_bytes + kv_slot * S::SLOT;
      uint64_t *bar = &x.sh.kvfull[kv_slot];
      if (++kv_slot == sm.slots) kv_slot = 0;
      int key = a.k0 + t * kKvKeys;
      int pk = plane0 + (seq * 2) * p.n_kv_heads + kvh;
      if (kv.page_table) {
        const int page = __ldg(kv.page_table + seq * kv.pages_per_seq + key / KV_PAGE);
        pk = ((page * kv.n_layers + kv.layer) * 2) * p.n_kv_heads + kvh;
        key %= KV_PAGE;
      }
      if (alive && elect_one()) {
        bar_expect(bar, S::SLOT);
#pragma unroll
        for (int hf = 0; hf < HD / 64; ++hf) {
          tma_3d(dst + hf * S::HALF, reinterpret_cast<const CUtensorMap *>(&p.kv_map), hf * 64, key, pk, bar);
          tma_3d(dst + S::SLOT / 2 + hf * S::HALF, reinterpret_cast<const CUtensorMap *>(&p.kv_map), hf * 64, key, pk + p.n_kv_heads, bar);
        }
      }
      __syncwarp();
    }
  }
}

// workers' part: the tiles go round the key groups (8 / KG warps, 16 query rows each; no more groups than slots); online
// softmax in base 2, the queries and the probabilities split hi / lo (neither operand loses more than about 2^-17 relative).
// The query fragments are read from shared memory for every tile: 64 registers less than keeping them.
template <int HD, int KG>
__device__ __forceinline__ void attention(const Ctx &x, int &kv_slot, uint32_t &kv_phase, uint32_t &q_phase) {
  const PassParams &p = x.p;
  using S = AttSmem<HD>;
  const S sm(p);
  constexpr int NRW = 8 / KG;
  const int rw = x.w % NRW, kg = x.w / NRW, g = x.lane >> 2, tq = x.lane & 3;
  const int W = p.rows, H = p.n_heads;
  const int n_units = H * p.n_segs * p.splits;
  bool first = true;
  for (int u = x.c; u < n_units; u += x.G) {
    AttUnit a;
    if (!att_unit(x, u, a)) continue;
    if (!first) workers_sync();   // the exchange buffer of the unit before becomes the query and tile region again
    signal_ready(x);
    first = false;
    const int m0 = a.seg * W;
    const int r0 = rw * 16 + g, r1 = r0 + 8;
    const int lim0 = min(r0 < W ? x.sh.pos[m0 + r0] : -1, a.k1 - 1), lim1 = min(r1 < W ? x.sh.pos[m0 + r1] : -1, a.k1 - 1);
    float o[HD / 8][4];
#pragma unroll
    for (int i = 0; i < HD / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.0f;
    float mr[2] = {-INFINITY, -INFINITY}, lr[2] = {0.0f, 0.0f};
    const int n_tiles = (a.k1 - a.k0 + kKvKeys - 1) / kKvKeys;
    bar_wait(&x.sh.qfull, q_phase, x.life, 27);
    q_phase ^= 1u;
    // A fragments by ldmatrix: rows rw * 16 + (0..15), 16-byte chunks 2 * ks and 2 * ks + 1
    const int qrow = rw * 16 + (x.lane & 15);
    const uint32_t qaddr = x.xring + (qrow < W ? qrow : 0) * 128, qswz = (qrow < W ? qrow : 0) & 7;
    const int groups = min(KG, sm.slots);
    int turn = groups - 1;
    for (int t = 0; t < n_tiles; ++t) {
      const int slot = kv_slot;
      const uint32_t ph = (kv_phase >> slot) & 1u;
      kv_phase ^= 1u << slot;
      if (++kv_slot == sm.slots) kv_slot = 0;
      if (++turn == groups) turn = 0;
      if (turn != kg) continue;
      // The slot's tile before this one belongs to another group, which may be behind: with only its parity to go by, `full` of
      // that tile would look like ours.  Its consumption (`empty`) cannot be mistaken: the producer is past the tile before
      // that, because this group's last tile was issued after it (groups <= slots).
      bar_wait(&x.sh.kvempty[slot], ph ^ 1u, x.life, 29);
      bar_wait(&x.sh.kvfull[slot], ph, x.life, 19);
      const uint32_t kb = x.xring + sm.q_bytes + slot * S::SLOT, vb = kb + S::SLOT / 2;
      const int key0 = a.k0 + t * kKvKeys;
      float sa[2][4], sb[2][4];   // hi and lo plane apart: four independent accumulation chains
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) sa[i][e] = sb[i][e] = 0.0f;
#pragma unroll
      for (int ks = 0; ks < HD / 16; ++ks) {
        const int row = (x.lane & 7) + ((x.lane >> 4) & 1) * 8, ch = (ks & 3) * 2 + ((x.lane >> 3) & 1);
        const uint32_t qch = (((ks & 3) * 2 + (x.lane >> 4)) ^ qswz) << 4;
        uint32_t kf[4], qh[4], ql[4];
        ldsm4(kb + (ks >> 2) * S::HALF + row * 128 + ((ch ^ (row & 7)) << 4), kf);
        ldsm4(qaddr + (ks >> 2) * sm.q_half + qch, qh);
        ldsm4(qaddr + (HD / 64 + (ks >> 2)) * sm.q_half + qch, ql);
        mma_16816(sa[0], qh, kf[0], kf[1]);
        mma_16816(sa[1], qh, kf[2], kf[3]);
        mma_16816(sb[0], ql, kf[0], kf[1]);
        mma_16816(sb[1], ql, kf[2], kf[3]);
      }
      float s[2][4];
      float t0 = -INFINITY, t1 = -INFINITY;
#pragma unroll
      for (int nb = 0; nb < 2; ++nb) {
        const int j = key0 + nb * 8 + tq * 2;
#pragma unroll
        for (int e = 0; e < 4; ++e) s[nb][e] = j + (e & 1) <= (e < 2 ? lim0 : lim1) ? sa[nb][e] + sb[nb][e] : -INFINITY;
        t0 = fmaxf(t0, fmaxf(s[nb][0], s[nb][1]));
        t1 = fmaxf(t1, fmaxf(s[nb][2], s[nb][3]));
      }
      t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 1));
      t0 = fmaxf(t0, __shfl_xor_sync(0xffffffffu, t0, 2));
      t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 1));
      t1 = fmaxf(t1, __shfl_xor_sync(0xffffffffu, t1, 2));
      const float n0 = fmaxf(mr[0], t0), n1 = fmaxf(mr[1], t1);
      if (__any_sync(0xffffffffu, n0 > mr[0] || n1 > mr[1])) {   // some row has a new maximum: rescale
        const float a0 = n0 > -INFINITY ? exp2f(mr[0] - n0) : 1.0f, a1 = n1 > -INFINITY ? exp2f(mr[1] - n1) : 1.0f;
        lr[0] *= a0;
        lr[1] *= a1;
#pragma unroll
        for (int i = 0; i < HD / 8; ++i) {
          o[i][0] *= a0; o[i][1] *= a0;
          o[i][2] *= a1; o[i][3] *= a1;
        }
        mr[0] = n0;
        mr[1] = n1;
      }
      const float u0 = mr[0] > -INFINITY ? mr[0] : 0.0f, u1 = mr[1] > -INFINITY ? mr[1] : 0.0f;
      uint32_t ph_[4], pl_[4];
#pragma unroll
      for (int nb = 0; nb < 2; ++nb) {
        const float p0 = exp2f(s[nb][0] - u0), p1 = exp2f(s[nb][1] - u0), p2 = exp2f(s[nb][2] - u1), p3 = exp2f(s[nb][3] - u1);
        lr[0] += p0 + p1;
        lr[1] += p2 + p3;
        split2(p0, p1, ph_[nb * 2], pl_[nb * 2]);
        split2(p2, p3, ph_[nb * 2 + 1], pl_[nb * 2 + 1]);
      }
#pragma unroll
      for (int c8 = 0; c8 < HD / 8; c8 += 2) {
        const int row = (x.lane & 7) + ((x.lane >> 3) & 1) * 8, ch = c8 + ((x.lane >> 4) & 1);
        uint32_t vf[4];
        ldsm4_trans(vb + (ch >> 3) * S::HALF + row * 128 + (((ch & 7) ^ (row & 7)) << 4), vf);
        mma_16816(o[c8], ph_, vf[0], vf[1]);
        mma_16816(o[c8 + 1], ph_, vf[2], vf[3]);
        mma_16816(o[c8], pl_, vf[0], vf[1]);
        mma_16816(o[c8 + 1], pl_, vf[2], vf[3]);
      }
      __syncwarp();
      if (x.lane == 0) {   // the slot is free when the group's warps have read it: the barrier counts 8 / KG
        bar_arrive(&x.sh.kvempty[slot]);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      lr[i] += __shfl_xor_sync(0xffffffffu, lr[i], 1);
      lr[i] += __shfl_xor_sync(0xffffffffu, lr[i], 2);
    }
    // Every group leaves its (max, sum, output) per row in the idle region; then each warp finishes whole rows.  Entries
    // of eight floats are rotated by the row so that the fragment stores do not meet in a bank.
    workers_sync();
    float *xch = reinterpret_cast<float *>(x.xptr);
    const int band = (kg * NRW + rw) * 16;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int r = band + g + rr * 8;
      if (tq == 0) x.sh.ml[r] = make_float2(mr[rr], lr[rr]);
#pragma unroll
      for (int i = 0; i < HD / 8; ++i)
        *reinterpret_cast<float2 *>(xch + r * HD + (((i ^ (r & 7)) << 3) | (tq * 2))) = make_float2(o[i][rr * 2], o[i][rr * 2 + 1]);
    }
    workers_sync();
    constexpr int PER = HD / 32;
    for (int r = x.w; r < W; r += 8) {
      float2 ml[KG];
      float mx = -INFINITY, den = 0.0f, acc[PER];
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        ml[k] = x.sh.ml[k * NRW * 16 + r];
        mx = fmaxf(mx, ml[k].x);
      }
#pragma unroll
      for (int i = 0; i < PER; ++i) acc[i] = 0.0f;
#pragma unroll
      for (int k = 0; k < KG; ++k) {
        const float w = ml[k].x > -INFINITY ? exp2f(ml[k].x - mx) : 0.0f;
        den += ml[k].y * w;
        const int rk = k * NRW * 16 + r, j = x.lane * PER;
        const float *src = xch + rk * HD + ((((j >> 3) ^ (rk & 7)) << 3) | (j & 7));
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] += src[i] * w;
      }
      const size_t rec = (size_t)(m0 + r) * H + a.h;
      if (a.n_act == 1) {
        const float inv = den > 0.0f ? 1.0f / den : 0.0f;   // inactive rows: zeros
#pragma unroll
        for (int i = 0; i < PER; i += 2) {
          uint32_t hi, lo;
          split2(acc[i] * inv, acc[i + 1] * inv, hi, lo);
          const size_t idx = rec * HD + x.lane * PER + i;
          *reinterpret_cast<uint32_t *>(p.attn.base + idx) = hi;
          *reinterpret_cast<uint32_t *>(p.attn.base + p.attn.lo_offset + idx) = lo;
        }
      } else {   // record of this key range: output, and max and sum
        float *dst = p.partial + (rec * p.splits + a.split) * HD + x.lane * PER;
#pragma unroll
        for (int i = 0; i < PER; i += 2) *reinterpret_cast<float2 *>(dst + i) = make_float2(acc[i], acc[i + 1]);
        if (x.lane == 0) reinterpret_cast<float2 *>(p.partial_ml)[rec * p.splits + a.split] = make_float2(mx, den);
      }
    }
  }
}
// merge of the key ranges: one warp per (row, head)
template <int HD>
__device__ __forceinline__ void attention_merge(const Ctx &x) {
  const PassParams &p = x.p;
  constexpr int PER = HD / 32;
  const int n = p.M * p.n_heads;
  for (int u = x.c + x.G * x.w; u < n; u += x.G * 8) {
    const int m = u / p.n_heads, len = x.sh.len[m / p.rows];
    if (len == 0) continue;
    const int chunk = key_chunk(p, len), n_act = (len + chunk - 1) / chunk;
    if (n_act == 1) continue;   // written by its only key range
    const float *src = p.partial + (size_t)u * p.splits * HD + x.lane * PER;
    float mx = -INFINITY, den = 0.0f, acc[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = 0.0f;
#pragma unroll 1
    for (int s0 = 0; s0 < n_act; s0 += 4) {   // four records in flight
      float2 ml[4];
      float v[4][PER];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const bool on = s0 + s < n_act;
        ml[s] = on ? __ldcg(reinterpret_cast<const float2 *>(p.partial_ml) + (size_t)u * p.splits + s0 + s) : make_float2(-INFINITY, 0.0f);
#pragma unroll
        for (int i = 0; i < PER; i += 2) {
          const float2 t = on ? __ldcg(reinterpret_cast<const float2 *>(src + (size_t)(s0 + s) * HD + i)) : make_float2(0.f, 0.f);
          v[s][i] = t.x;
          v[s][i + 1] = t.y;
        }
      }
      float mn = mx;
#pragma unroll
      for (int s = 0; s < 4; ++s) mn = fmaxf(mn, ml[s].x);
      if (!(mn > -INFINITY)) continue;
      const float keep = exp2f(mx - mn);
      den *= keep;
#pragma unroll
      for (int i = 0; i < PER; ++i) acc[i] *= keep;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const float w = exp2f(ml[s].x - mn);
        den += ml[s].y * w;
#pragma unroll
        for (int i = 0; i < PER; ++i) acc[i] += v[s][i] * w;
      }
      mx = mn;
    }
    const float inv = x.sh.pos[m] >= 0 && den > 0.0f ? 1.0f / den : 0.0f;
    const size_t idx = (size_t)u * HD + x.lane * PER;
#pragma unroll
    for (int i = 0; i < PER; i += 2) {
      uint32_t hi, lo;
      split2(acc[i] * inv, acc[i + 1] * inv, hi, lo);
      *reinterpret_cast<uint32_t *>(p.attn.base + idx + i) = hi;
      *reinterpret_cast<uint32_t *>(p.attn.base + p.attn.lo_offset + idx + i) = lo;
    }
  }
}

// ---------------------------------------------------------------------------------- projections
// The projections of a pass in order: 4 per layer (Q|K|V, O, gate|up, down), then the logits.  A pre-fill pass (no logits)
// ends with the last layer's Q|K|V.
__device__ __forceinline__ int pass_gemms(const PassParams &p) { return p.logits ? 4 * p.n_layers + 1 : 4 * p.n_layers - 3; }
__device__ __forceinline__ int pass_kind(const PassParams &p, int i) { return i == 4 * p.n_layers ? PK_LOGITS : i & 3; }
// matrix of a tile (only Q|K|V has several), its rows, and how the tile lies in the accumulators: up to 128 rows in one; else
// (and gate | up) two, the second starting `second` rows (a multiple of 8) into the tile's shared memory
struct TileShape {
  int j, R, row0, second;
  bool two;
};
__device__ __forceinline__ TileShape tile_shape(const PassGemm &g, int kind, int tile) {
  TileShape t;
  t.j = kind != PK_QKV || tile < g.tile_end[0] ? 0 : tile < g.tile_end[1] ? 1 : 2;
  t.R = g.rows[t.j];
  t.row0 = (tile - (t.j ? g.tile_end[t.j - 1] : 0)) * t.R;
  t.two = kind == PK_GU || t.R > 128;
  t.second = kind == PK_GU ? (t.R + 7) / 8 * 8 : (t.R / 2 + 7) / 8 * 8;
  return t;
}

// The workers' side of one projection: TMEM lane = weight row, columns = tokens (hi plane, then lo plane).
__device__ __forceinline__ void epilogue(const Ctx &x, const PassGemm &g, int kind, uint32_t tmem, uint32_t &acc_n) {
  const PassParams &p = x.p;
  const int quarter = x.w & 3, grp = x.w >> 2, row = quarter * 32 + x.lane;
  const int NN = 2 * p.Mp;
  SegIter it;
  it.init(g, x.c, x.G);
  Seg s;
#pragma unroll 1
  while (it.next(s)) {
    const int buf = acc_n & 1u;
    const TileShape t = tile_shape(g, kind, s.tile);
    const int n_left = g.n_out[t.j] - t.row0;   // rows of the tile that exist
    bar_wait(&x.sh.acc_full[buf], (acc_n >> 1) & 1u, x.life, 20);
    ++acc_n;
    fence_tc_after();
    const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + buf * 2 * NN;
    // (stores of 8 or 16 tokens without a test between them: two warps per scheduler cannot hide dependent instructions)
    if (kind == PK_GU) {
      const bool live = row < t.R && row < n_left;
      __nv_bfloat16 *dst = p.act.base + t.row0 + row;
#pragma unroll 1
      for (int m0 = grp * 8; m0 < p.M; m0 += 16) {
        uint32_t gh[8], gl[8], uh[8], ul[8];
        tmem_ld8(base + m0, gh);
        tmem_ld8(base + p.Mp + m0, gl);
        tmem_ld8(base + NN + m0, uh);
        tmem_ld8(base + NN + p.Mp + m0, ul);
        tmem_wait_ld();
        __nv_bfloat16 hi[8], lo[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float sc = x.sh.scale[m0 + i];
          const float gv = (__uint_as_float(gh[i]) + __uint_as_float(gl[i])) * sc;
          const float uv = (__uint_as_float(uh[i]) + __uint_as_float(ul[i])) * sc;
          const float v = gv / (1.0f + expf(-gv)) * uv;
          hi[i] = __float2bfloat16_rn(v);
          lo[i] = __float2bfloat16_rn(v - __bfloat162float(hi[i]));
        }
        if (!live) continue;
        __nv_bfloat16 *o = dst + (size_t)m0 * p.F;
        const int n = p.M - m0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (i < n) {
            o[(size_t)i * p.F] = hi[i];
            o[p.act.lo_offset + (size_t)i * p.F] = lo[i];
          }
        }
      }
    } else {
      // two accumulators: warps 0-3 take the first, 4-7 the second; one: they share its token columns
      const int half = t.two ? grp : 0, r = half * t.second + row;
      const bool live = row < (half ? t.R - t.second : t.two ? t.second : t.R) && r < n_left;
      float *dst = p.part + (size_t)(s.tile * g.max_pieces + s.piece) * p.M * p.part_ld + r;
      __nv_bfloat16 *lg = p.logits + (size_t)t.row0 + r;
#pragma unroll 1
      for (int m0 = t.two ? 0 : grp * 16; m0 < p.M; m0 += t.two ? 16 : 32) {
        uint32_t hi[16], lo[16];
        tmem_ld16(base + half * NN + m0, hi);
        tmem_ld16(base + half * NN + p.Mp + m0, lo);
        tmem_wait_ld();
        if (!live) continue;
        const int n = p.M - m0;
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
        if (kind == PK_LOGITS) {
          __nv_bfloat16 *o = lg + (size_t)m0 * p.vocab;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (i < n) o[(size_t)i * p.vocab] = __float2bfloat16_rn(v[i] * x.sh.scale[m0 + i]);
        } else {
          float *o = dst + (size_t)m0 * p.part_ld;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (i < n) o[(size_t)i * p.part_ld] = v[i];
        }
      }
    }
    fence_tc_before();
    __syncwarp();
    if (x.lane == 0) bar_arrive(&x.sh.acc_empty[buf]);
  }
}

template <int HD, int KG>
__global__ void __launch_bounds__(kPassThreads, 1) pass_kernel(const __grid_constant__ PassParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ PassShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (*reinterpret_cast<volatile int *>(p.status) != 0) return;   // an earlier launch gave up: the counters are void
  uint8_t *smem = smem_raw;   // 1024-byte aligned by its declaration (the swizzle pattern depends on it: checked below)
  const uint32_t wring = s32(smem), xring = wring + p.n_w * p.slot_bytes;
  const int NN = 2 * p.Mp, x_bytes = NN * 128, n_x = min(kXRegion / x_bytes, p.n_w);
  uint32_t cols = 32;
  while ((int)cols < 4 * NN) cols <<= 1;
  if ((wring & 1023u) != 0) {
    if (tid == 0) atomicExch(p.status, 28);
    return;
  }
  const uint32_t epoch = *reinterpret_cast<volatile uint32_t *>(p.counter + 1);
  if (tid == 0) {
    for (int i = 0; i < p.n_w; ++i) { bar_init(&sh.full[i], 2); bar_init(&sh.empty[i], 1); }
    for (int i = 0; i < 2; ++i) { bar_init(&sh.acc_full[i], 1); bar_init(&sh.acc_empty[i], 8); }
    for (int i = 0; i < kKvSlots; ++i) { bar_init(&sh.kvfull[i], 1); bar_init(&sh.kvempty[i], 8 / p.key_groups); }
    bar_init(&sh.qfull, 1);
    sh.ready = 0;
    sh.dead = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy();
  }
  if (tid < 64) sh.pos[tid] = tid < p.M ? p.in_pos[tid] : -1;
  if (tid >= 64 && tid < 64 + p.n_segs) {
    const int s = tid - 64;
    int len = 0;
    for (int i = 0; i < p.rows; ++i) len = max(len, p.in_pos[s * p.rows + i] + 1);
    sh.len[s] = len;
    sh.seq[s] = p.seg_seq ? p.seg_seq[s] : s;
  }
  // The layers' tensor maps were copied into global memory by the host: a fence per map before any use by this CTA.
  for (int i = tid; i < (p.n_layers + 1) * 7; i += kPassThreads)
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(p.layers[i / 7].w + i % 7) : "memory");
  if (warp == 3) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&sh.tmem)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_tc_before();
  __syncthreads();
  fence_tc_after();
  const uint32_t tmem = sh.tmem;
  const Life life{&sh.dead, p.status};
  const Ctx x{p, sh, wring, xring, smem + (size_t)p.n_w * p.slot_bytes, (int)blockIdx.x, (int)gridDim.x,
              warp >= 4 ? warp - 4 : warp, lane, life};

  // Blocks (64 columns of K of one tile) are numbered through the pass.  Block i sits in weight slot i % n_w and activation
  // slot i % n_x (n_x <= n_w); full[i % n_w] flips when both have landed, empty[i % n_w] when the MMAs have read them.
  // A role whose wait has run out issues nothing any more (alive).
  // The three warps below run converged and elect a lane to issue: the operands stay in uniform registers.
  bool alive = true;
  if (warp == 0) {
    // ------------------------------------------------------------------ weight producer
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    int slot = 0;
    uint32_t ph = 0;
#pragma unroll 1
    for (int i = 0, n = pass_gemms(p); i < n; ++i) {
      const int kind = pass_kind(p, i);
      const PassGemm &g = p.gemm[kind];
      const TensorMap *maps = p.layers[i >> 2].w;   // the logits matrix stands first in the entry after the last layer
      SegIter it;
      it.init(g, x.c, x.G);
      Seg s;
#pragma unroll 1
      while (it.next(s)) {
        const TileShape t = tile_shape(g, kind, s.tile);
        const CUtensorMap *map = reinterpret_cast<const CUtensorMap *>(
            maps + (kind == PK_LOGITS ? 0 : kind == PK_QKV ? t.j : kind == PK_O ? 3 : kind == PK_GU ? 4 : 6));
        const uint32_t bytes = (kind == PK_GU ? 2 : 1) * t.R * 128;
#pragma unroll 1
        for (int kb = s.kb0; kb < s.kb1; ++kb) {
          alive = alive && __all_sync(0xffffffffu, bar_wait(&sh.empty[slot], ph ^ 1u, life, 21));
          if (alive && elect_one()) {
            const uint32_t dst = wring + slot * p.slot_bytes;
            const int kcol = kb * 64;
            bar_expect(&sh.full[slot], bytes);
            tma_2d_hint(dst, map, kcol, t.row0, &sh.full[slot], policy);
            if (kind == PK_GU) tma_2d_hint(dst + t.second * 128, map + 1, kcol, t.row0, &sh.full[slot], policy);
          }
          __syncwarp();
          if (++slot == p.n_w) { slot = 0; ph ^= 1u; }
        }
      }
    }
    if (*life.dead) {   // leave no copy in flight: give the last ones ample time to land
      const unsigned long long t0 = now_ns();
      while (now_ns() - t0 < kDrainNs) {}
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ activation producer
    int slot = 0, xs = 0, eslot = 0, kv_slot = 0;
    uint32_t eph = 0, ready_n = 0, kv_phase = 0;
    int fill = 0;   // blocks before the first reuse of an activation slot
#pragma unroll 1
    for (int i = 0, n = pass_gemms(p); i < n; ++i) {
      const int kind = pass_kind(p, i);
      const PassGemm &g = p.gemm[kind];
      if (kind == PK_O) attention_loads<HD>(x, (i >> 2) * p.planes_per_layer, pass_kv(p, i >> 2), ready_n, kv_slot, kv_phase, alive);
      const CUtensorMap *map = reinterpret_cast<const CUtensorMap *>(kind == PK_O ? &p.attn_map : kind == PK_DOWN ? &p.act_map : &p.h_map);
      wait_ready(x, ready_n);
      SegIter it;
      it.init(g, x.c, x.G);
      Seg s;
#pragma unroll 1
      while (it.next(s)) {
#pragma unroll 1
        for (int kb = s.kb0; kb < s.kb1; ++kb) {
          if (fill == n_x) {   // the block n_x back has been read
            alive = alive && __all_sync(0xffffffffu, bar_wait(&sh.empty[eslot], eph, life, 23));
            if (++eslot == p.n_w) { eslot = 0; eph ^= 1u; }
          } else {
            ++fill;
          }
          if (alive && elect_one()) {
            const uint32_t dst = xring + xs * x_bytes;
            bar_expect(&sh.full[slot], x_bytes);
            const int kcol = kb * 64;
            tma_2d(dst, map, kcol, 0, &sh.full[slot]);
            tma_2d(dst + x_bytes / 2, map, kcol, p.x_lo_row, &sh.full[slot]);
          }
          __syncwarp();
          if (++slot == p.n_w) slot = 0;
          if (++xs == n_x) xs = 0;
        }
      }
    }
    if (*life.dead) {
      const unsigned long long t0 = now_ns();
      while (now_ns() - t0 < kDrainNs) {}
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NN >> 3) << 17) | (8u << 24);
    const uint64_t desc0 = desc_sw128(0);
    int ws = 0, xs = 0;
    uint32_t wph = 0, acc_n = 0;
#pragma unroll 1
    for (int i = 0, n = pass_gemms(p); i < n; ++i) {
      const int kind = pass_kind(p, i);
      const PassGemm &g = p.gemm[kind];
      SegIter it;
      it.init(g, x.c, x.G);
      Seg s;
#pragma unroll 1
      while (it.next(s)) {
        const TileShape t = tile_shape(g, kind, s.tile);
        const uint32_t second = t.second * 8;   // in 16-byte units
        const int buf = acc_n & 1u;
        alive = alive && __all_sync(0xffffffffu, bar_wait(&sh.acc_empty[buf], ((acc_n >> 1) & 1u) ^ 1u, life, 24));
        ++acc_n;
        fence_tc_after();
        const uint32_t d = tmem + buf * 2 * NN;
#pragma unroll 1
        for (int kb = s.kb0; kb < s.kb1; ++kb) {
          alive = alive && __all_sync(0xffffffffu, bar_wait(&sh.full[ws], wph, life, 25));
          fence_tc_after();
          if (alive && elect_one()) {
            const uint64_t a = desc0 | (uint64_t)((wring + ws * p.slot_bytes) >> 4), b = desc0 | (uint64_t)((xring + xs * x_bytes) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              mma_f16(d, a + k * 2, b + k * 2, idesc, kb > s.kb0 || k > 0);
              if (t.two) mma_f16(d + NN, a + second + k * 2, b + k * 2, idesc, kb > s.kb0 || k > 0);
            }
            mma_commit(&sh.empty[ws]);
          }
          __syncwarp();
          if (++ws == p.n_w) { ws = 0; wph ^= 1u; }
          if (++xs == n_x) xs = 0;
        }
        if (alive && elect_one()) mma_commit(&sh.acc_full[buf]);
        __syncwarp();
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ workers
    uint32_t target = epoch, acc_n = 0;
    uint32_t kv_phase = 0, q_phase = 0;   // kv_phase: bit per slot, phase of its next tile
    int kv_slot = 0;
    bool merge = false;   // some segment's keys are spread over several CTAs
    for (int s = 0; s < p.n_segs; ++s) merge = merge || (sh.len[s] > 0 && key_chunk(p, sh.len[s]) < sh.len[s]);
    const int n_gemms = pass_gemms(p);
#pragma unroll 1
    for (int i = 0; i < n_gemms + (p.logits ? 0 : 1); ++i) {   // pre-fill: one round more for the last layer's keys and values
      const int kind = pass_kind(p, i), l = i >> 2;
      const PassLayer &L = p.layers[l];   // (of the logits: the entry after the last layer)
      if (kind == PK_O) {
        PASS_TL(TL_QKV, 0);
        qkv_finish<HD>(x, L, pass_kv(p, l));
        PASS_TL(TL_QKV, 1);
        if (i == n_gemms) break;
        grid_sync(x, target);
        PASS_TL(TL_ATTN, 0);
        attention<HD, KG>(x, kv_slot, kv_phase, q_phase);
        PASS_TL(TL_ATTN, 1);
        grid_sync(x, target);
        if (merge) {
          PASS_TL(TL_COMBINE, 0);
          attention_merge<HD>(x);
          PASS_TL(TL_COMBINE, 1);
          grid_sync(x, target);
        }
      } else if (kind != PK_DOWN) {
        PASS_TL(TL_RESID, kind);
        resid_gain(x, kind == PK_GU ? p.loc_o : i ? p.loc_down : nullptr, kind == PK_GU ? L.ffn_norm : L.attn_norm);
        PASS_TL(TL_RESID, kind + 1);
        grid_sync(x, target);
      }
      PASS_TL(TL_GEMM, kind * 2);
      signal_ready(x);
      if (kind != PK_O && kind != PK_DOWN) row_scales(x);
      epilogue(x, p.gemm[kind], kind, tmem, acc_n);
      PASS_TL(TL_GEMM, kind * 2 + 1);
      if (kind != PK_LOGITS) grid_sync(x, target);
    }
    // nobody reads the epoch any more in this launch: every CTA is past its first barrier
    if (x.c == 0 && x.w == 0 && lane == 0 && !sh.dead) *reinterpret_cast<volatile uint32_t *>(p.counter + 1) = target;
  }
  fence_tc_before();
  __syncthreads();
  if (warp == 3) {
    fence_tc_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
  }
}

inline int up8(int v) { return (v + 7) / 8 * 8; }

// tiles of a projection over matrices of n[j] rows: whole tiles for short K, else units cut evenly
void plan_gemm(PassGemm &g, const int *n, int n_mats, int kb, int slot_rows, int n_sms) {
  memset(&g, 0, sizeof(g));
  g.kb = kb;
  g.full = kb <= 32;
  int total = 0;
  for (int j = 0; j < n_mats; ++j) total += n[j];
  int want = g.full ? up8((total + n_sms - 1) / n_sms) : slot_rows;
  want = want > slot_rows ? slot_rows : want;
  for (int j = 0; j < 3; ++j) {
    if (j < n_mats) {
      const int t = (n[j] + want - 1) / want;
      g.rows[j] = up8((n[j] + t - 1) / t);
      g.n_out[j] = n[j];
      g.tiles += (n[j] + g.rows[j] - 1) / g.rows[j];
    }
    g.tile_end[j] = g.tiles;
  }
  g.max_pieces = 1;
  if (!g.full)
    for (int t = 0; t < g.tiles; ++t) {
      const int U = g.tiles * kb;
      const int np = ((t + 1) * kb * n_sms - 1) / U - ((t * kb + 1) * n_sms - 1) / U + 1;
      g.max_pieces = np > g.max_pieces ? np : g.max_pieces;
    }
}

}  // namespace

bool pass_plan(const sjd_model_cfg &c, int n_sms, PassPlan *pl) {
  const int nq = c.n_heads * c.head_dim, nk = c.n_kv_heads * c.head_dim;
  if (n_sms < 1 || (c.head_dim != 64 && c.head_dim != 128)) return false;
  const int f = (c.ffn_hidden + n_sms - 1) / n_sms;   // gate rows (and up rows) per CTA
  if (f > 128) return false;
  const int slot_rows = 2 * (up8(f) > 64 ? up8(f) : 64);
  pl->slot_bytes = slot_rows * 128;
  const int qkv[3] = {nq, nk, nk}, d[1] = {c.d_model}, F[1] = {c.ffn_hidden}, V[1] = {c.vocab};
  plan_gemm(pl->gemm[PK_QKV], qkv, 3, c.d_model / 64, slot_rows, n_sms);
  plan_gemm(pl->gemm[PK_O], d, 1, nq / 64, slot_rows, n_sms);
  plan_gemm(pl->gemm[PK_DOWN], d, 1, c.ffn_hidden / 64, slot_rows, n_sms);
  plan_gemm(pl->gemm[PK_GU], F, 1, c.d_model / 64, slot_rows, n_sms);
  pl->gemm[PK_GU].full = 1;      // one tile of f gate rows and the same up rows per CTA
  pl->gemm[PK_GU].rows[0] = f;
  pl->gemm[PK_GU].tiles = (c.ffn_hidden + f - 1) / f;
  pl->gemm[PK_GU].max_pieces = 1;
  plan_gemm(pl->gemm[PK_LOGITS], V, 1, c.d_model / 64, slot_rows, n_sms);
  pl->gemm[PK_LOGITS].full = 1;    // whole tiles, as many rounds of the grid as the slot size asks for
  const int rounds = (c.vocab + n_sms * slot_rows - 1) / (n_sms * slot_rows);
  pl->gemm[PK_LOGITS].rows[0] = up8((c.vocab + n_sms * rounds - 1) / (n_sms * rounds));
  pl->gemm[PK_LOGITS].tiles = (c.vocab + pl->gemm[PK_LOGITS].rows[0] - 1) / pl->gemm[PK_LOGITS].rows[0];
  pl->gemm[PK_LOGITS].max_pieces = 1;
  for (PassGemm *g : {&pl->gemm[PK_GU], &pl->gemm[PK_LOGITS]}) g->tile_end[0] = g->tile_end[1] = g->tile_end[2] = g->tiles;
  pl->part_ld = 0;
  size_t part = 0;
  for (const PassGemm *g : {&pl->gemm[PK_QKV], &pl->gemm[PK_O], &pl->gemm[PK_DOWN]}) {
    if (g->max_pieces > kPassMaxPieces || (!g->full && g->tiles * g->kb < n_sms)) return false;
    for (int j = 0; j < 3; ++j) pl->part_ld = g->rows[j] > pl->part_ld ? g->rows[j] : pl->part_ld;
    part = (size_t)g->tiles * g->max_pieces > part ? (size_t)g->tiles * g->max_pieces : part;
  }
  pl->part_bytes = part * kPassMaxRows * pl->part_ld * sizeof(float);
  const int ring = 232448 - 3072 - kXRegion;   // shared memory of a CTA less the static part and the activation region
  pl->n_w = ring / pl->slot_bytes < kMaxW ? ring / pl->slot_bytes : kMaxW;
  static_assert(sizeof(PassShared) <= 3072, "static shared memory");
  return pl->n_w >= 3;
}

// the location tables of the Q|K|V, O and down projections, one after the other
void pass_locations(const PassPlan &pl, int n_sms, int2 *out) {
  for (int kind : {PK_QKV, PK_O, PK_DOWN}) {
    const PassGemm *g = &pl.gemm[kind];
    const int U = g->tiles * g->kb;
    for (int j = 0; j < 3; ++j)
      for (int col = 0; col < g->n_out[j]; col += 8) {
        const int t = (j ? g->tile_end[j - 1] : 0) + col / g->rows[j];
        const int np = g->full ? 1 : ((t + 1) * g->kb * n_sms - 1) / U - ((t * g->kb + 1) * n_sms - 1) / U + 1;
        *out++ = make_int2(t * g->max_pieces, col % g->rows[j] | np << 16);
      }
  }
}

int launch_pass(const PassParams &p, int n_sms, cudaStream_t stream) {
  auto kernel = p.head_dim == 128 ? (p.key_groups == 8 ? pass_kernel<128, 8> : p.key_groups == 4 ? pass_kernel<128, 4> : pass_kernel<128, 2>)
                                  : (p.key_groups == 8 ? pass_kernel<64, 8> : p.key_groups == 4 ? pass_kernel<64, 4> : pass_kernel<64, 2>);
  const size_t smem = (size_t)p.n_w * p.slot_bytes + kXRegion;
  SJD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(n_sms);
  cfg.blockDim = dim3(kPassThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SJD_CUDA(cudaLaunchKernelEx(&cfg, kernel, p));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

}  // namespace sjd
