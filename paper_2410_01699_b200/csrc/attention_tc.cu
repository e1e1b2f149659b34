// Window-causal split-KV attention on the tensor cores for bf16 caches (Sec. 3.2 / Sec. 4.1 Step 2: the W window queries
// attend the cached prefix plus the in-window causal block).
//
// A stream is one (query head, segment of W rows, key range); a CTA works on two of them.  Keys are the rows of both products and
// the queries their columns, because a window has far fewer queries than an MMA has rows:
//   S^T [128 keys x 2 Wp]  =  K [128 keys x HD] . [Q hi | Q lo]^T
//   O^T [HD x 2 Wp]       +=  V^T [HD x 128 keys] . [P hi | P lo]
// Q (pre-scaled) and the probabilities are split into bf16 hi + lo planes, which are columns of the same MMA; the halves are
// added when they are read from tensor memory, so neither operand loses more than about 2^-17 relative.  K and V tiles of 128
// keys come by TMA (128-byte swizzle, boxes of 64 keys x 64 dims: a box lies in one page of a paged cache) into one ring that
// both streams take their tiles from in a fixed order; V needs no transposition, it is an MN-major operand as it is stored.
// Eight warps, a thread per key and stream, turn S^T into probabilities: the reference of a query's exponents is the maximum of
// its first tile, and is renewed (and O^T rescaled) only if a later score passes it by 2^40, so that a tile needs no maximum over
// lanes; the sums of the probabilities stay in registers until the end.
//
// Bound: the bytes of K and V (a tile of 64 KB takes the tensor pipe 500 to 1000 cycles, an SM's share of HBM about 2800).
// One CTA per SM, with all of its shared memory (head_dim 64 and up to 32 columns: 147 KB, the six tiles of the longest ring): 96 to
// 160 KB of tiles in flight.
// (us a call, 32 heads of 128, mma.sync with a CTA per stream and tiles of 64 keys -> now: 8 x 32 rows x 4009 keys 123 -> 101 (K and V
// at 5.2 TB/s, launch included; 82 in a graph, 6.4 TB/s), 8 x 64 rows 202 -> 119 (95 in a graph), 5 x 32 x 3032 94 -> 62, 1 x 32 x 2232
// with the merge 31 -> 23 (13 in a graph).  Windows of up to 32 rows take 64 columns, longer ones 128: with 128 the ring holds three tiles and not five, and a thread
// has twice the columns.  Over few keys that thread is the bound: 10 x 48 rows x 64 keys, two rounds of the grid, 20 -> 22.)
// Partials (reference, sum, unnormalised output) go to the merge kernel of attention.cu.  Every barrier wait is bounded.
#include <type_traits>

#include "tcgen05.cuh"

namespace sjd {
SJD_TIMELINE_TU(attn)
namespace {

constexpr int KT = 128;                // keys per tile
constexpr int kBoxKeys = 64;           // keys per TMA box
constexpr int kAttnThreads = 320;      // 2 x 4 softmax warps, producer, issuer
constexpr int kAttnSlots = 6;          // most tiles in the ring
constexpr int kAttnSmem = 232448;      // most dynamic shared memory of a CTA
constexpr float kRenewAt = 40.0f;      // log2 by which a score may pass its query's reference

struct AttnParams {
  const float *q;        // [M][H*HD]
  const int32_t *in_pos; // [M]
  float *partial;        // [M][H][splits][HD], then (reference, sum) [M][H][splits][2]
  float *out;            // [M][H*HD], OUT only: written here when splits == 1 (no merge launch needed)
  HiLoOut hilo;          // optional bf16 hi/lo planes of out (same case)
  int *status;
  int clear_status;      // the word is this call's own: it starts at zero
  int q_aligned;         // q starts on 16 bytes (else on 8)
  int M, rows_per_seq, n_segs, n_heads, n_kv_heads, splits;
  int slots;             // tiles in the ring
  int plane0;            // first cache plane of this layer: planes are [b][k|v][kv_head]
  // paged cache: planes are [page][layer][k|v][kv_head], one page (kBoxKeys positions) per box
  const int32_t *page_table;   // [B][pages_per_seq]; null: contiguous
  int pages_per_seq, layer, n_layers;
  const int32_t *seg_seq;      // PACKED: sequence of every segment
};

// behind Q, P and the ring
struct AttnShared {
  float red[2][4][64];   // per stream: a value per softmax warp and query; rows 0 and 1 also hold a renewed rescale factor and reference
  int pos[2][64];        // position of every query, -1: none
  int len[2], first[2];  // keys that the last query sees; smallest position of an active query
  uint64_t full[kAttnSlots], empty[kAttnSlots];
  uint64_t q_ready[2], s_full[2], s_free[2], p_full[2], pv_done[2];
  uint32_t tmem_base;
};
constexpr int kAttnBarriers = 2 * kAttnSlots + 10;

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t *r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};"
      ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ float4 load_stream4(const float *p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// value i of 32, combined over the lanes of the warp, in lane i (31 exchanges)
template <typename F>
__device__ __forceinline__ float lanes_combine(float *v, const F &f) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (j >= o) break;
      const float send = lane & o ? v[j] : v[j + o], keep = lane & o ? v[j + o] : v[j];
      v[j] = f(keep, __shfl_xor_sync(0xffffffffu, send, o));
    }
  }
  return v[0];
}
// OR / AND of a predicate over the 128 softmax threads of a stream (named barrier 1 + stream)
__device__ __forceinline__ bool stream_any(int st, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, %2, 128, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(1 + st)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void stream_sync(int st) { asm volatile("bar.sync %0, 128;" ::"r"(1 + st) : "memory"); }

struct Stream {
  int h, seg, split, b, m0, k_begin, k_end, n_tiles;
};

// HD: head_dim; WP: columns of a plane (W padded to 32 or 64).  PACKED: a pre-fill pass, whose rows are segments of prompts, several
// of one sequence among them.  OUT: the fp32 output is wanted (else only its planes).
template <int HD, int WP, bool PACKED, bool OUT>
__global__ void __launch_bounds__(kAttnThreads, 1) attention_tc_kernel(const __grid_constant__ CUtensorMap kv_map, const AttnParams p) {
  constexpr int HALVES = HD / 64;                    // 64-dim (128-byte) columns of boxes
  constexpr int HALF_BYTES = KT * 128;               // 128 keys x 64 dims
  constexpr int TILE_BYTES = HALVES * HALF_BYTES;    // one of K or V
  constexpr int Q_BYTES = 2 * WP * HD * 2;           // both planes of a stream's queries
  constexpr int P_BYTES = KT * (WP == 32 ? 128 : 256);
  constexpr int NC = WP / 16;                        // chunks of 16 queries
  // Tensor memory of a stream: S^T, then O^T (both planes: 2 WP columns each); where there is room, odd tiles have an O^T of their
  // own, which halves the chains of truncating additions (8 x 32 rows x 4009 keys against fp64: 5.7e-6 with one).
  constexpr int NO = WP == 32 ? 2 : 1;
  constexpr int T_COLS = (1 + NO) * 2 * WP, T_ALL = 512;
  extern __shared__ __align__(1024) uint8_t attn_smem[];   // no static shared memory: it starts on 1024 bytes
  uint8_t *ring = attn_smem + 2 * (Q_BYTES + P_BYTES);
  AttnShared &sh = *reinterpret_cast<AttnShared *>(ring + p.slots * TILE_BYTES);

  SJD_TL(TL_ATTN, 0, threadIdx.x == 0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int W = p.rows_per_seq;
  const int n_streams = p.n_heads * p.n_segs * p.splits;
  // The swizzled tiles have to start on 1024 bytes (the same for every CTA of a launch); any other error is 2 s away.
  const bool skewed = (smem_u32(attn_smem) & 1023u) != 0;
  if (tid == 0 && (skewed || (p.clear_status && blockIdx.x == 0))) *p.status = skewed ? 5 : 0;
  if (PACKED) pdl_wait();   // (a window's positions, and its keys before it, are older than the step: see embed_kernel)

  auto stream_of = [&](int st) {
    Stream s;
    const int u = blockIdx.x * 2 + st;
    s.h = u % p.n_heads;
    const int v = u / p.n_heads;
    s.seg = v % p.n_segs;
    s.split = v / p.n_segs;
    if (PACKED) s.seg = p.n_segs - 1 - s.seg;   // later segments of a prompt see more keys, they start first
    s.b = PACKED && s.split < p.splits ? __ldg(p.seg_seq + s.seg) : s.seg;
    s.m0 = s.seg * W;
    return s;
  };
  if (warp == 0 || warp == 4) {
    const int st = warp >> 2;
    const bool have = (int)blockIdx.x * 2 + st < n_streams;
    const int m0 = have ? stream_of(st).m0 : 0;
    int len = 0, first = 0x7FFFFFFF;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int i = lane + 32 * j, pos = have && i < W ? p.in_pos[m0 + i] : -1;
      sh.pos[st][i] = pos;
      len = max(len, pos + 1);
      if (pos >= 0) first = min(first, pos);
    }
    len = __reduce_max_sync(0xffffffffu, len);
    first = __reduce_min_sync(0xffffffffu, first);
    if (lane == 0) {
      sh.len[st] = len;
      sh.first[st] = first;
    }
  }
  if (warp == 8 && lane < kAttnBarriers) {
    mbar_init(&sh.full[lane], lane < 2 * kAttnSlots ? 1 : lane < 2 * kAttnSlots + 2 ? 4 : lane < 2 * kAttnSlots + 4 ? 1 : lane < 2 * kAttnSlots + 8 ? 4 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // key range of a stream
  auto range_of = [&](Stream &s, int st) {
    const int len = sh.len[st];
    int chunk = (len + p.splits - 1) / p.splits;
    chunk = (chunk + KT - 1) / KT * KT;
    s.k_begin = s.split * chunk;
    s.k_end = min(len, s.k_begin + chunk);
    s.n_tiles = s.k_end > s.k_begin ? (s.k_end - s.k_begin + KT - 1) / KT : 0;
  };
  Stream s0 = stream_of(0), s1 = stream_of(1);
  range_of(s0, 0);
  range_of(s1, 1);
  const int n0 = s0.n_tiles, n1 = s1.n_tiles, n_max = max(n0, n1);
  const int my = warp < 8 ? warp >> 2 : 0;      // softmax warps: their stream
  const Stream me = my ? s1 : s0;
  const bool have = (int)blockIdx.x * 2 + my < n_streams;
  float *ml = p.partial + (size_t)p.M * p.n_heads * p.splits * HD;
  if (n_max == 0 && p.splits > 1) {   // key ranges beyond the last key: empty records
    pdl_wait();   // (the merge of an earlier layer may still read its records)
    const int i = tid & 127;
    if (warp < 8 && have && i < W)
      *reinterpret_cast<float2 *>(ml + (((size_t)(me.m0 + i) * p.n_heads + me.h) * p.splits + me.split) * 2) = make_float2(-INFINITY, 0.0f);
    return;
  }

  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_base)), "r"(T_ALL) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();   // (not before the allocation: a CTA of a later kernel that holds tensor memory waits for this one)
  const uint32_t tmem = sh.tmem_base;

  if (warp == 8) {
    // ------------------------------------------------------------------ TMA producer
    // Tiles in the order in which the issuer takes them: K of tile t of both streams, then V of tile t - 1 of both.
    const int group = p.n_heads / p.n_kv_heads;
    const int kvh0 = s0.h / group, kvh1 = s1.h / group;
    int it = 0, s = 0;
    uint32_t ph = 1;   // (a ring that has not been filled yet is not waited for)
    bool ok = true, waited = PACKED;
    auto load = [&](const Stream &c, int kvh, int first, int t, int is_v) {
      const int key0 = c.k_begin + t * KT;
      // keys before the window were written by earlier steps; the kernel before this one wrote the others
      if (!waited && key0 + KT > first) {
        pdl_wait();
        waited = true;
      }
      if (it >= p.slots && !warp_wait(&sh.empty[s], ph)) { ok = false; return; }
      if (elect_one()) {
        const bool two = c.k_end - key0 > kBoxKeys;
        const uint32_t dst = smem_u32(ring) + s * TILE_BYTES;
        uint64_t *bar = &sh.full[s];
        mbar_expect_tx(bar, (two ? 2u : 1u) * (kBoxKeys * HD * 2));
        auto box = [&](int j) {
          int key = key0 + j * kBoxKeys, plane = p.plane0 + (c.b * 2 + is_v) * p.n_kv_heads + kvh;
          if (p.page_table != nullptr) {   // ranges start on multiples of a tile: a box is exactly one page
            const int page = __ldg(p.page_table + c.b * p.pages_per_seq + key / kBoxKeys);
            plane = ((page * p.n_layers + p.layer) * 2 + is_v) * p.n_kv_heads + kvh;
            key = 0;
          }
#pragma unroll
          for (int hf = 0; hf < HALVES; ++hf)
            tma_load_3d(dst + hf * HALF_BYTES + j * (kBoxKeys * 128), &kv_map, hf * 64, key, plane, bar);
        };
        box(0);
        if (two) box(1);
      }
      __syncwarp();
      ++it;
      if (++s == p.slots) { s = 0; ph ^= 1u; }
    };
    const int f0 = sh.first[0], f1 = sh.first[1];
    for (int t = 0; t <= n_max && ok; ++t) {
      if (t < n0) load(s0, kvh0, f0, t, 0);
      if (t < n1 && ok) load(s1, kvh1, f1, t, 0);
      if (t >= 1 && t - 1 < n0 && ok) load(s0, kvh0, f0, t - 1, 1);
      if (t >= 1 && t - 1 < n1 && ok) load(s1, kvh1, f1, t - 1, 1);
    }
    if (!waited) pdl_wait();
    if (!ok && lane == 0) atomicExch(p.status, 4);
    // leave no copy in flight, whatever the other roles do
    for (int j = it > p.slots ? it - p.slots : 0; j < it; ++j) warp_wait(&sh.full[j % p.slots], (uint32_t)((j / p.slots) & 1));
  } else if (warp == 9) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t idesc = umma_idesc_bf16(2 * WP);
    const uint32_t idesc_v = idesc | (1u << 15) | (1u << 16);   // both operands MN-major
    const uint64_t desc_k = umma_desc_sw128(0);
    // MN-major, 128-byte swizzle: 8-key groups 1024 bytes apart, 64-element columns LBO apart.  (V at head_dim 64: both halves of
    // the MMA's rows read the same 64 dims, the second is ignored.)
    const uint64_t desc_mn = desc_k & ~((uint64_t)0x3FFF << 16);
    const uint64_t desc_v = desc_mn | (uint64_t)(HALVES == 2 ? HALF_BYTES >> 4 : 0) << 16;
    const uint64_t desc_p = desc_mn | (uint64_t)(WP == 64 ? (KT * 128) >> 4 : 1) << 16;
    const uint32_t ring0 = smem_u32(ring), q_at = smem_u32(attn_smem), p_at = q_at + 2 * Q_BYTES;
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    auto next = [&]() {
      __syncwarp();
      if (++s == p.slots) { s = 0; ph ^= 1u; }
    };
    auto scores = [&](int st, int t) {
      if (!(t == 0 ? warp_wait_both(&sh.full[s], ph, &sh.q_ready[st], 0) : warp_wait_both(&sh.full[s], ph, &sh.s_free[st], (uint32_t)((t - 1) & 1)))) {
        ok = false;
        return;
      }
      tc_fence_after();
      if (elect_one()) {
        const uint64_t a = desc_k | (uint64_t)((ring0 + s * TILE_BYTES) >> 4);
        const uint64_t b = desc_k | (uint64_t)((q_at + st * Q_BYTES) >> 4);
#pragma unroll
        for (int k = 0; k < HD / 16; ++k)
          umma_bf16(tmem + st * T_COLS, a + (k >> 2) * (HALF_BYTES >> 4) + (k & 3) * 2, b + (k >> 2) * ((2 * WP * 128) >> 4) + (k & 3) * 2,
                    idesc, k > 0);
        umma_commit(&sh.empty[s]);
        umma_commit(&sh.s_full[st]);
      }
      next();
    };
    auto values = [&](const Stream &c, int st, int t) {
      if (!warp_wait_both(&sh.full[s], ph, &sh.p_full[st], (uint32_t)(t & 1))) { ok = false; return; }
      tc_fence_after();
      if (elect_one()) {
        const uint64_t a = desc_v | (uint64_t)((ring0 + s * TILE_BYTES) >> 4);
        const uint64_t b = desc_p | (uint64_t)((p_at + st * P_BYTES) >> 4);
        const int keys = c.k_end - c.k_begin - t * KT;   // no further than the last one: rows past it may be anything
        const uint32_t d = tmem + st * T_COLS + (1 + t % NO) * 2 * WP;
#pragma unroll
        for (int k = 0; k < KT / 16; ++k)
          if (k * 16 < keys) umma_bf16(d, a + k * (16 * 128 >> 4), b + k * (16 * 128 >> 4), idesc_v, t >= NO || k > 0);
        umma_commit(&sh.empty[s]);
        umma_commit(&sh.pv_done[st]);
      }
      next();
    };
    for (int t = 0; t <= n_max && ok; ++t) {
      if (t < n0) scores(0, t);
      if (t < n1 && ok) scores(1, t);
      if (t >= 1 && t - 1 < n0 && ok) values(s0, 0, t - 1);
      if (t >= 1 && t - 1 < n1 && ok) values(s1, 1, t - 1);
    }
    if (!ok && lane == 0) atomicExch(p.status, 4);
  } else if (have) {
    // ------------------------------------------------------------------ softmax warps: thread = key of the tile
    const int st = my, ts = tid & 127, w = warp & 3;
    const int n = me.n_tiles;
    uint8_t *Ps = attn_smem + 2 * Q_BYTES + st * P_BYTES;
    const uint32_t row_bytes = ts * 128, sw = (uint32_t)(ts & 7) << 4;
    pdl_wait();   // the queries
    SJD_TL(TL_ATTN, 1, threadIdx.x == 0);
    {
      // Q, pre-scaled by log2(e) / sqrt(HD), as K-major planes: rows 0.. hi, rows WP.. lo
      uint8_t *Qs = attn_smem + st * Q_BYTES;
      const float sc = 1.4426950408889634f * rsqrtf((float)HD);
      // A warp takes whole rows, four entries a thread.  All loads are in flight at once: none stands behind a test (rows that are not
      // wanted are loaded all the same, those past the window from its last row), and they are volatile, so that the compiler does not
      // move them to their uses one by one.  (Behind a test of its row each load was a round trip of its own, eight in a row at 64 rows of
      // 128: the attention of a 7B layer at 64 rows, 80 keys, 12.7 us of the step's chain, now 10.3; 8 x 64 rows x 214 keys 21.0 -> 16.7 us a call.)
      constexpr int NQ = WP * (HD / 4) / 128;
      auto at = [&](int j) {
        const int i = ts + j * 128;
        return p.q + ((size_t)(me.m0 + min(i / (HD / 4), W - 1)) * p.n_heads + me.h) * HD + i % (HD / 4) * 4;
      };
      auto put = [&](int j, float4 v) {
        const int i = ts + j * 128, r = i / (HD / 4), c = i % (HD / 4);
        uint2 hi = make_uint2(0u, 0u), lo = hi;
        if (sh.pos[st][r] >= 0) {
          split_pair(v.x * sc, v.y * sc, hi.x, lo.x);
          split_pair(v.z * sc, v.w * sc, hi.y, lo.y);
        }
        uint8_t *dst = Qs + (c >> 4) * (2 * WP * 128) + r * 128 + ((c * 8 & 127) ^ ((r & 7) << 4));
        *reinterpret_cast<uint2 *>(dst) = hi;
        *reinterpret_cast<uint2 *>(dst + WP * 128) = lo;
      };
      if (__builtin_expect(p.q_aligned, 1)) {
        float4 v[NQ];
#pragma unroll
        for (int j = 0; j < NQ; ++j) v[j] = load_stream4(at(j));
#pragma unroll
        for (int j = 0; j < NQ; ++j) put(j, v[j]);
      } else {   // (a caller's q may start on 8 bytes)
#pragma unroll 1
        for (int j = 0; j < NQ; ++j) {
          const float2 a = *reinterpret_cast<const float2 *>(at(j)), b = *reinterpret_cast<const float2 *>(at(j) + 2);
          put(j, make_float4(a.x, a.y, b.x, b.y));
        }
      }
      if (W <= WP - 16)   // columns of queries that do not exist
        for (int i = ts; i < P_BYTES / 16; i += 128) reinterpret_cast<uint4 *>(Ps)[i] = make_uint4(0u, 0u, 0u, 0u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      stream_sync(st);   // (a row of P is cleared by one thread and written by another)
      if (lane == 0) mbar_arrive(&sh.q_ready[st]);
    }
    const uint32_t t_s = tmem + ((uint32_t)(w * 32) << 16) + st * T_COLS, t_o = t_s + 2 * WP;
    float l_acc[WP];
#pragma unroll
    for (int i = 0; i < WP; ++i) l_acc[i] = 0.0f;
    float my_ref = 0.0f;   // thread i < W: the reference of query i
    bool ok = true;
    const int first = sh.first[st];
    for (int t = 0; t < n; ++t) {
      const int key0 = me.k_begin + t * KT, key = key0 + ts;
      ok = warp_wait(&sh.s_full[st], (uint32_t)(t & 1));   // (a wait that ran out is noticed at the vote below)
      tc_fence_after();
      float sv[WP];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c * 16 < W) {
          uint32_t hi[16], lo[16];
          tmem_ld16_issue(t_s + c * 16, hi);
          tmem_ld16_issue(t_s + WP + c * 16, lo);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) sv[c * 16 + i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) sv[c * 16 + i] = -INFINITY;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.s_free[st]);
      if (key0 + KT - 1 > first || key0 + KT > me.k_end) {   // some query does not see some key of this tile
        const int lim = key < me.k_end ? key : 0x7FFFFFFF;
#pragma unroll
        for (int i = 0; i < WP; i += 4) {
          const int4 at = *reinterpret_cast<const int4 *>(&sh.pos[st][i]);
          if (lim > at.x) sv[i] = -INFINITY;
          if (lim > at.y) sv[i + 1] = -INFINITY;
          if (lim > at.z) sv[i + 2] = -INFINITY;
          if (lim > at.w) sv[i + 3] = -INFINITY;
        }
      }
      // the tile before is multiplied: P may be written, O^T is at rest
      if (t > 0) ok = warp_wait(&sh.pv_done[st], (uint32_t)((t - 1) & 1)) && ok;
      float over = 0.0f;
      if (t > 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (c * 16 < W) {
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
              const float4 r = *reinterpret_cast<const float4 *>(&sh.red[st][1][c * 16 + i]);
              sv[c * 16 + i] -= r.x;
              sv[c * 16 + i + 1] -= r.y;
              sv[c * 16 + i + 2] -= r.z;
              sv[c * 16 + i + 3] -= r.w;
              over = fmaxf(over, fmaxf(sv[c * 16 + i], sv[c * 16 + i + 1]));
              over = fmaxf(over, fmaxf(sv[c * 16 + i + 2], sv[c * 16 + i + 3]));
            }
          }
        }
      }
      if (stream_any(st, !ok || t == 0 || !(over <= kRenewAt))) {
        if (stream_any(st, !ok)) { ok = false; break; }
        // ---- renew the references: the maximum over the tile (scores are relative to the old reference after the first tile)
#pragma unroll
        for (int g = 0; g < WP / 32; ++g) {
          float mx[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) mx[i] = sv[g * 32 + i];
          sh.red[st][w][g * 32 + lane] = lanes_combine(mx, [](float a, float b) { return fmaxf(a, b); });
        }
        stream_sync(st);
        if (ts < WP) {   // by how much the reference of query ts grows
          const float mx = fmaxf(fmaxf(sh.red[st][0][ts], sh.red[st][1][ts]), fmaxf(sh.red[st][2][ts], sh.red[st][3][ts]));
          const float up = t > 0 ? fmaxf(mx, 0.0f) : mx > -INFINITY ? mx : 0.0f;   // (a query that does not see the first key of the range sees none)
          my_ref += up;
          // row 2: what to subtract from this tile's scores; row 1: the reference from now on; row 0: the factor of the sums so far
          sh.red[st][2][ts] = up;
          sh.red[st][1][ts] = my_ref;
          sh.red[st][0][ts] = ex2(-up);
        }
        stream_sync(st);
#pragma unroll
        for (int i = 0; i < WP; i += 4) {
          const float4 r = *reinterpret_cast<const float4 *>(&sh.red[st][2][i]);
          sv[i] -= r.x;
          sv[i + 1] -= r.y;
          sv[i + 2] -= r.z;
          sv[i + 3] -= r.w;
        }
        if (t > 0) {
#pragma unroll
          for (int i = 0; i < WP; i += 4) {
            const float4 r = *reinterpret_cast<const float4 *>(&sh.red[st][0][i]);
            l_acc[i] *= r.x;
            l_acc[i + 1] *= r.y;
            l_acc[i + 2] *= r.z;
            l_acc[i + 3] *= r.w;
          }
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < 2 * NC * min(t, NO); ++c) {
            uint32_t o[16];
            tmem_ld16_issue(t_o + c * 16, o);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * sh.red[st][0][(c * 16 + i) & (WP - 1)]);
            tmem_st16(t_o + c * 16, o);
          }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
      }
      // ---- probabilities, split hi / lo, as MN-major planes: row = key, 128 bytes of queries
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (c * 16 >= W) continue;
        uint32_t ph[8], pl[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float a = ex2(sv[c * 16 + 2 * i]), b = ex2(sv[c * 16 + 2 * i + 1]);
          l_acc[c * 16 + 2 * i] += a;
          l_acc[c * 16 + 2 * i + 1] += b;
          split_pair(a, b, ph[i], pl[i]);
        }
        uint8_t *hi_at = Ps + row_bytes, *lo_at = WP == 32 ? hi_at : hi_at + KT * 128;
        constexpr uint32_t lo_col = WP == 32 ? 64 : 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t col = c * 32 + j * 16;
          *reinterpret_cast<uint4 *>(hi_at + (col ^ sw)) = make_uint4(ph[4 * j], ph[4 * j + 1], ph[4 * j + 2], ph[4 * j + 3]);
          *reinterpret_cast<uint4 *>(lo_at + ((lo_col + col) ^ sw)) = make_uint4(pl[4 * j], pl[4 * j + 1], pl[4 * j + 2], pl[4 * j + 3]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.p_full[st]);
    }
    SJD_TL(TL_ATTN, 2, threadIdx.x == 0);
    // ---- the sums over the keys, while the last tile is multiplied; then the output rows
    stream_sync(st);
#pragma unroll
    for (int g = 0; g < WP / 32; ++g) {
      float v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = l_acc[g * 32 + i];
      sh.red[st][w][g * 32 + lane] = lanes_combine(v, [](float a, float b) { return a + b; });
    }
    if (ok && n > 0) ok = warp_wait(&sh.pv_done[st], (uint32_t)((n - 1) & 1));
    if (!stream_any(st, !ok)) {
      tc_fence_after();
      const bool direct = p.splits == 1;
      const size_t rec_step = (size_t)p.n_heads * p.splits;   // from a query's record to the next one's
      const size_t rec0 = (size_t)me.m0 * rec_step + (size_t)me.h * p.splits + me.split;
      float l = 0.0f;
      if (ts < W) {
        l = sh.pos[st][ts] >= 0 ? (sh.red[st][0][ts] + sh.red[st][1][ts]) + (sh.red[st][2][ts] + sh.red[st][3][ts]) : 0.0f;
        if (!direct)   // (reference in natural log units)
          *reinterpret_cast<float2 *>(ml + (rec0 + ts * rec_step) * 2) = make_float2(l > 0.0f ? my_ref * 0.6931471805599453f : -INFINITY, l);
      }
      if (direct) {
        // inactive rows: zeros; the NaN of a score that is not finite stays  (each thread has read its column only)
        if (ts < WP) sh.red[st][0][ts] = l == 0.0f ? 0.0f : 1.0f / l;
        stream_sync(st);
      }
      const int dim = w * 32 + lane;
      if ((n > 0 || direct) && w * 32 < HD) {
        const size_t step = direct ? (size_t)p.n_heads * HD : rec_step * HD;
        const size_t at0 = direct ? ((size_t)me.m0 * p.n_heads + me.h) * HD + dim : rec0 * HD + dim;
#pragma unroll 1
        for (int c = 0; c < NC; ++c) {
          if (c * 16 >= W) break;
          uint32_t hi[16], lo[16];
          float v[16];
          if (n > 0) {
            tmem_ld16_issue(t_o + c * 16, hi);
            tmem_ld16_issue(t_o + WP + c * 16, lo);
            tmem_ld_wait();
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
          if (NO == 2 && n > 1) {
            tmem_ld16_issue(t_o + 2 * WP + c * 16, hi);
            tmem_ld16_issue(t_o + 3 * WP + c * 16, lo);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
          }
          const size_t at = at0 + (size_t)(c * 16) * step;
          const int left = W - c * 16;
          auto each = [&](auto store) {   // (no tests per row but in a ragged chunk)
            if (left >= 16) {
#pragma unroll
              for (int i = 0; i < 16; ++i) store(i);
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i)
                if (i < left) store(i);
            }
          };
          if (!direct) {
            float *dst = p.partial + at;
            each([&](int i) { dst[i * step] = v[i]; });
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float inv = sh.red[st][0][c * 16 + i];
              v[i] = inv == 0.0f ? 0.0f : v[i] * inv;
            }
            if constexpr (OUT) {
              float *dst = p.out + at;
              each([&](int i) { dst[i * step] = v[i]; });
            }
            if (p.hilo.base) {
              __nv_bfloat16 *dst = p.hilo.base + at, *dst_lo = dst + p.hilo.lo_offset;
              each([&](int i) {
                const __nv_bfloat16 vh = __float2bfloat16_rn(v[i]);
                dst[i * step] = vh;
                dst_lo[i * step] = __float2bfloat16_rn(v[i] - __bfloat162float(vh));
              });
            }
          }
        }
      }
    } else if (ts == 0) {
      atomicExch(p.status, 4);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T_ALL) : "memory");
  }
}

}  // namespace

// bf16 cache [planes][max_seq][head_dim] as boxes of 64 keys x 64 dims, 128-byte swizzle
int make_kv_tensor_map(TensorMap *out, const void *base, long planes, long max_seq, int head_dim) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return SJD_ERR_UNSUPPORTED;
  if (((uintptr_t)base & 15u) != 0 || (head_dim != 64 && head_dim != 128)) return SJD_ERR_UNSUPPORTED;
  cuuint64_t dims[3] = {(cuuint64_t)head_dim, (cuuint64_t)max_seq, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)head_dim * 2, (cuuint64_t)max_seq * head_dim * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)kBoxKeys, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = fn(reinterpret_cast<CUtensorMap *>(out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base),
                        dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? SJD_OK : SJD_ERR_CUDA;
}

bool attention_tc_supported(int head_dim, int rows_per_seq) { return (head_dim == 64 || head_dim == 128) && rows_per_seq <= 64; }

// With splits > 1 the kernel leaves partial records and the caller merges them with the combine kernel of
// attention.cu; with a single key range it writes `out` (and `hilo`) itself and no merge is needed.
int launch_attention_tc(const TensorMap &kv_map, int plane0, KvLayout kv, const float *q, const int32_t *in_pos, float *partial,
                        float *out, HiLoOut hilo, int *status, int M, RowSegs segs, int n_heads, int n_kv_heads, int head_dim,
                        int splits, bool clear_status, cudaStream_t stream) {
  const int rows_per_seq = segs.rows;
  if (!attention_tc_supported(head_dim, rows_per_seq) || M % rows_per_seq != 0) return SJD_ERR_UNSUPPORTED;
  AttnParams p;
  p.q = q;
  p.in_pos = in_pos;
  p.partial = partial;
  p.out = out;
  p.hilo = hilo;
  p.status = status;
  p.clear_status = clear_status ? 1 : 0;
  p.q_aligned = ((uintptr_t)q & 15u) == 0;
  p.M = M;
  p.rows_per_seq = rows_per_seq;
  p.n_segs = M / rows_per_seq;
  p.seg_seq = segs.seq;
  p.n_heads = n_heads;
  p.n_kv_heads = n_kv_heads;
  p.splits = splits;
  p.plane0 = plane0;
  static_assert(kBoxKeys == KV_PAGE, "one box per cache page");
  p.page_table = kv.page_table;
  p.pages_per_seq = kv.pages_per_seq;
  p.layer = kv.layer;
  p.n_layers = kv.n_layers;
  const int wp = rows_per_seq <= 32 ? 32 : 64;
  const long streams = (long)n_heads * p.n_segs * splits;
  const CUtensorMap &km = reinterpret_cast<const CUtensorMap &>(kv_map);
  const int tile = KT * head_dim * 2, fixed = 2 * (2 * wp * head_dim * 2 + KT * (wp == 32 ? 128 : 256));
  p.slots = (kAttnSmem - (int)sizeof(AttnShared) - fixed) / tile;
  p.slots = p.slots > kAttnSlots ? kAttnSlots : p.slots;
  const size_t smem = (size_t)fixed + (size_t)p.slots * tile + sizeof(AttnShared);
  auto launch = [&](auto kernel) -> int {
    const int rc = allow_smem(kernel, smem);   // (the size follows from the kernel's head_dim and columns)
    if (rc != SJD_OK) return rc;
    SJD_CUDA(launch_kernel(kernel, dim3((unsigned)((streams + 1) / 2)), dim3(kAttnThreads), smem, stream, km, p));
    SJD_CHECK_LAUNCH();
    return SJD_OK;
  };
  auto pick = [&](auto packed, auto wants_out) -> int {
    constexpr bool P = decltype(packed)::value, O = decltype(wants_out)::value;
    if (head_dim == 128) return wp == 32 ? launch(attention_tc_kernel<128, 32, P, O>) : launch(attention_tc_kernel<128, 64, P, O>);
    return wp == 32 ? launch(attention_tc_kernel<64, 32, P, O>) : launch(attention_tc_kernel<64, 64, P, O>);
  };
  if (segs.seq) return out ? SJD_ERR_UNSUPPORTED : pick(std::true_type(), std::false_type());
  return out ? pick(std::false_type(), std::true_type()) : pick(std::false_type(), std::false_type());
}

}  // namespace sjd
