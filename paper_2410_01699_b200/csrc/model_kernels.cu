// Generic kernels of the decoder forward pass (Sec. 3.1: the auto-regressive transformer; Sec. 4.1
// Step 2: one pass over the window).  These cover every shape and both dtypes with plain FMA
// arithmetic and fp32 accumulation.  Activations between kernels are fp32 (they are a few hundred KB);
// only weights, the KV cache and the stored logits are in the model dtype.
#include <type_traits>

#include "common.cuh"

namespace sjd {
namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// E = 4 adjacent entries (aligned) or one, as they are stored: they are converted where they are used, so that nothing waits for a
// load that was issued ahead.
template <typename T, int E>
struct Group {
  uint32_t w[E * sizeof(T) / 4 ? E * sizeof(T) / 4 : 1];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (uint32_t &x : w) x = 0u;
  }
  __device__ __forceinline__ void load(const T *p) {
    if constexpr (E == 1 && sizeof(T) == 4) {
      w[0] = __float_as_uint(p[0]);
    } else if constexpr (E == 1) {
      w[0] = *reinterpret_cast<const unsigned short *>(p);
    } else if constexpr (sizeof(T) == 4) {
      const uint4 t = *reinterpret_cast<const uint4 *>(p);
      w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
    } else {
      const uint2 t = *reinterpret_cast<const uint2 *>(p);
      w[0] = t.x; w[1] = t.y;
    }
  }
  __device__ __forceinline__ float get(int e) const {
    if constexpr (sizeof(T) == 4) return __uint_as_float(w[e]);
    else return __uint_as_float(e & 1 ? w[e / 2] & 0xFFFF0000u : w[e / 2] << 16);
  }
};

__device__ __forceinline__ void store_hilo(const HiLoOut &o, size_t idx, float v) {
  if (!o.base) return;
  const __nv_bfloat16 hi = __float2bfloat16_rn(v);
  o.base[idx] = hi;
  o.base[o.lo_offset + idx] = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// ------------------------------------------------------------------------------------ projections (FMA)
// Small or odd-shaped matrices and fp32 models.  With few rows a step is a chain of launches that each cost their own latency (two
// layers of d 256 and 16 rows: 29 launches, 418 us of projections in a 476 us step with 32 x 64 tiles that walked K in slices of
// 32, one dependent load after the other; 16 launches and the verification in 107 us now).  Hence: the eight warps of a CTA
// split every chunk of KC columns between them, so that a whole chunk is one round trip to memory, and the next chunk is
// on its way while this one is multiplied.  The RMS normalisation before a projection (its row scale commutes with the
// product), the residual add, SwiGLU and the rotary step with its cache append are part of the launch.  Any M, N, K; the sums have one fixed order.
// A tile: 4 * MI rows x 8 * NJ weight rows; BLOCKS: CTAs that an SM has registers for.  (LD: + 4, rows eight apart meet in
// different banks.)
template <int MI_, int NJ_, int KC_, int BLOCKS_>
struct RowsTile {
  static constexpr int MI = MI_, NJ = NJ_, KC = KC_, BLOCKS = BLOCKS_, BM = 4 * MI, BN = 8 * NJ, LD = KC + 4;
  static constexpr size_t kOperands = (size_t)(BM + BN) * LD, kSums = (size_t)8 * BM * (BN + 1);
  static constexpr size_t kSmem = (kOperands > kSums ? kOperands : kSums) * sizeof(float);
};
// Few rows: 16 x 16 (small matrices: half the work per CTA) or 16 x 32, with all the registers they want (two CTAs on an SM: a
// step of the fp32 model of d 256 with 192 rows 160 us, one: 142).  More rows: 32 x 32, which loads a third less per product, with
// two CTAs on an SM.  (With 16 x 32 alone, one CTA on an SM and the CTAs of one weight tile far apart in the grid, passes of
// many rows were slower than the 32 x 64 tiles had been.  us, 32 x 64 / 16 x 32 / now: fp32 512 x 12288 x 4096 2655 / 2915 /
// 1681, 256 x 8192 x 1024 234 / 265 / 158; bf16 1280 x 22016 x 4096 11460 / 17392 / 6769, 512 x 2560 x 961 168 / 345 / 148.)
using RowsNarrow = RowsTile<4, 2, 256, 1>;
using RowsFew = RowsTile<4, 4, 256, 1>;
using RowsMany = RowsTile<8, 4, 128, 2>;

// VEC: rows of x and of every matrix can be read in groups of four entries
template <typename T, typename Tile, bool VEC>
__global__ void __launch_bounds__(256, Tile::BLOCKS) gemm_rows_kernel(const RowsGemm g) {
  constexpr int MI = Tile::MI, NJ = Tile::NJ, RG_M = Tile::BM, BN = Tile::BN, RG_K = Tile::KC, RG_LD = Tile::LD;
  extern __shared__ float smem[];
  float *xs = smem, *ws = smem + RG_M * RG_LD;
  __shared__ float s_ss[RG_M][8];
  pdl_trigger();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * RG_M, t0 = blockIdx.y + blockIdx.z * gridDim.y;   // (blocks that share weight rows run side by side)
  const bool qkv = g.epilogue == RG_QKV, glu = g.epilogue == RG_SWIGLU || qkv;   // an output column is made of two weight rows
  const int half = g.kv.head_dim >> 1;
  const T *gain = reinterpret_cast<const T *>(g.gain);
  // weight row r of this tile: under SwiGLU the first half of the rows are gate features, the second the same up features; of
  // rotated pairs the first half of the rows holds the first entries, the second the others
  auto wrow = [&](int r) -> const T * {
    int n, j = 0;
    if (glu) {
      j = r >= BN / 2;
      n = t0 * (BN / 2) + r - j * (BN / 2);
      if (qkv) {
        if (n >= g.N) return nullptr;
        n = n / half * (2 * half) + n % half + j * half;
        j = 0;
        while (j < 2 && n >= g.n[j]) n -= g.n[j++];
      }
    } else {
      n = t0 * BN + r;
      while (j < 2 && n >= g.n[j]) n -= g.n[j++];
    }
    return n < g.n[j] ? reinterpret_cast<const T *>(g.w[j]) + (size_t)n * g.K : nullptr;
  };
  constexpr int E = VEC ? 4 : 1, PER = 256 / (RG_K / E);        // entries per load, rows per round of the block
  constexpr int NXL = RG_M / PER, NWL = BN / PER;
  const int col = tid % (RG_K / E) * E, r0 = tid / (RG_K / E);
  Group<float, E> xr[NXL];
  Group<T, E> wr[NWL], gr;
  float ss[NXL];
  const T *wp[NWL];   // this thread's weight rows (each is looked up on the way to its first load)
#pragma unroll
  for (int i = 0; i < NXL; ++i) ss[i] = 0.0f;
  auto load_w = [&](int k0, auto first) {
    const int k = k0 + col;
#pragma unroll
    for (int i = 0; i < NWL; ++i) {
      if constexpr (decltype(first)::value) wp[i] = wrow(r0 + i * PER);
      wr[i].clear();
      if (wp[i] && k < g.K) wr[i].load(wp[i] + k);
    }
    gr.clear();
    if (gain && k < g.K) gr.load(gain + k);
  };
  auto load_x = [&](int k0) {
    const int k = k0 + col;
#pragma unroll
    for (int i = 0; i < NXL; ++i) {
      const int m = m0 + r0 + i * PER;
      xr[i].clear();
      if (m < g.M && k < g.K) xr[i].load(g.x + (size_t)m * g.ldx + k);
    }
  };
  load_w(0, std::true_type());     // the weights do not depend on the kernel before
  pdl_wait();
  load_x(0);
  const int lm = lane >> 3, ln = lane & 7;
  float acc[MI][NJ];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = 0.0f;
  for (int k0 = 0; k0 < g.K; k0 += RG_K) {
    if (k0) __syncthreads();
#pragma unroll
    for (int i = 0; i < NXL; ++i)
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float v = xr[i].get(e);
        ss[i] = fmaf(v, v, ss[i]);
        xs[(r0 + i * PER) * RG_LD + col + e] = gain ? v * gr.get(e) : v;
      }
#pragma unroll
    for (int i = 0; i < NWL; ++i)
#pragma unroll
      for (int e = 0; e < E; ++e) ws[(r0 + i * PER) * RG_LD + col + e] = wr[i].get(e);
    __syncthreads();
    if (k0 + RG_K < g.K) {
      load_w(k0 + RG_K, std::false_type());
      load_x(k0 + RG_K);
    }
    const int kw = warp * (RG_K / 8);
#pragma unroll
    for (int k = 0; k < RG_K / 8; k += 4) {
      float4 xv[MI], wv[NJ];
#pragma unroll
      for (int i = 0; i < MI; ++i) xv[i] = *reinterpret_cast<const float4 *>(xs + (lm + 4 * i) * RG_LD + kw + k);
#pragma unroll
      for (int j = 0; j < NJ; ++j) wv[j] = *reinterpret_cast<const float4 *>(ws + (ln + 8 * j) * RG_LD + kw + k);
#pragma unroll
      for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
          acc[i][j] = fmaf(xv[i].w, wv[j].w, fmaf(xv[i].z, wv[j].z, fmaf(xv[i].y, wv[j].y, fmaf(xv[i].x, wv[j].x, acc[i][j]))));
    }
  }
  // sums of squares of the rows (their columns lie over 256 / PER threads, whole warps of one row each)
  if (gain) {
#pragma unroll
    for (int i = 0; i < NXL; ++i) {
      const float t = warp_sum(ss[i]);
      if (lane == 0) s_ss[r0 + i * PER][warp % (8 / PER)] = t;
    }
  }
  __syncthreads();
  float *red = smem;   // [warp][row][BN + 1]
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) red[(warp * RG_M + lm + 4 * i) * (BN + 1) + ln + 8 * j] = acc[i][j];
  __syncthreads();
  auto total = [&](int r, int c) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[(w * RG_M + r) * (BN + 1) + c];
    return t;
  };
  const int cols = glu ? BN / 2 : BN;
  for (int i = tid; i < RG_M * cols; i += 256) {
    const int r = i / cols, c = i - r * cols, m = m0 + r, n = t0 * cols + c;
    if (m >= g.M || n >= g.N) continue;
    float scale = 1.0f;
    if (gain) {
      float t = 0.0f;
#pragma unroll
      for (int w = 0; w < 8 / PER; ++w) t += s_ss[r][w];
      scale = rsqrtf(t / (float)g.K + g.eps);
    }
    float v = total(r, c) * scale;
    if (qkv) {
      const float u = total(r, c + BN / 2) * scale;
      const int pos = g.in_pos[m];
      if (pos < 0) continue;
      const int head = n / half, j = n % half, kh = head - g.n_heads, nkv = g.kv.n_kv_heads;
      const bool is_v = kh >= nkv;
      float x1 = v, x2 = u;
      if (!is_v) {
        const float2 cs = g.rope[(size_t)pos * half + j];
        x1 = v * cs.x - u * cs.y;
        x2 = u * cs.x + v * cs.y;
      }
      if (kh < 0) {
        float *dst = reinterpret_cast<float *>(g.out) + (size_t)m * g.ldc + head * 2 * half + j;
        dst[0] = x1;
        dst[half] = x2;
      } else {
        T *dst = reinterpret_cast<T *>(g.kv.base) +
                 kv_row_offset(g.kv, seg_sequence(g.segs, m / g.segs.rows), is_v ? 1 : 0, kh - (is_v ? nkv : 0), pos) + j;
        dst[0] = from_f<T>(x1);
        dst[half] = from_f<T>(x2);
      }
      continue;
    }
    if (glu) {
      const float u = total(r, c + BN / 2) * scale;
      v = v / (1.0f + expf(-v)) * u;
    }
    const size_t idx = (size_t)m * g.ldc + n;
    if (g.epilogue == RG_ADD) reinterpret_cast<float *>(g.out)[idx] += v;
    else if (g.epilogue == RG_LOGITS) reinterpret_cast<T *>(g.out)[idx] = from_f<T>(v);
    else reinterpret_cast<float *>(g.out)[idx] = v;
  }
}

template <typename T, typename Tile>
int gemm_rows_tile(const RowsGemm &g, bool vec, cudaStream_t stream) {
  const int cols = g.epilogue == RG_SWIGLU || g.epilogue == RG_QKV ? Tile::BN / 2 : Tile::BN;
  const int n_tiles = (g.N + cols - 1) / cols, layers = (n_tiles + 65534) / 65535;
  const dim3 grid((g.M + Tile::BM - 1) / Tile::BM, (n_tiles + layers - 1) / layers, layers);
  auto launch = [&](auto kernel) -> int {
    const int rc = Tile::kSmem > 40 * 1024 ? allow_smem(kernel, Tile::kSmem) : SJD_OK;
    if (rc != SJD_OK) return rc;
    SJD_CUDA(launch_kernel(kernel, grid, dim3(256), Tile::kSmem, stream, g));
    SJD_CHECK_LAUNCH();
    return SJD_OK;
  };
  return vec ? launch(gemm_rows_kernel<T, Tile, true>) : launch(gemm_rows_kernel<T, Tile, false>);
}

template <typename T>
int gemm_rows_t(const RowsGemm &g, cudaStream_t stream) {
  auto tiles = [&](int rows, int cols) { return (long)((g.M + rows - 1) / rows) * ((g.N + cols - 1) / cols); };
  const int glu = g.epilogue == RG_SWIGLU || g.epilogue == RG_QKV ? 2 : 1;   // weight rows of an output column
  bool vec = g.K % 4 == 0 && g.ldx % 4 == 0 && ((uintptr_t)g.x & 15u) == 0 && ((uintptr_t)g.gain & (4 * sizeof(T) - 1)) == 0;
  for (int j = 0; j < 3; ++j) vec = vec && ((uintptr_t)g.w[j] & (4 * sizeof(T) - 1)) == 0;
  // us, smallest / middle / largest tile.  The smallest while its grid is one wave (fp32 64 x 256 x 683: 8.3 / 14.5 / 18.5), the
  // middle one up to two (64 x 1024 x 2816: 25 / 23 / 35; 64 x 4096 x 4096, more than that: 123 / 103 / 85; a step of four layers
  // of d 1024 and 128 rows 957 us, 1007 if the line is at one wave).  The largest is not for rows that would fill half of it (16 x
  // 12288 x 4096: 108 / 82 / 125).
  constexpr int kSms = 148;
  if (tiles(RowsNarrow::BM, RowsNarrow::BN / glu) <= kSms) return gemm_rows_tile<T, RowsNarrow>(g, vec, stream);
  if (g.M <= RowsFew::BM || tiles(RowsFew::BM, RowsFew::BN / glu) <= 2 * kSms) return gemm_rows_tile<T, RowsFew>(g, vec, stream);
  return gemm_rows_tile<T, RowsMany>(g, vec, stream);
}

// ------------------------------------------------------------------------------------ embedding
template <typename T>
__global__ void embed_kernel(const T *__restrict__ emb, const int32_t *__restrict__ tok, float *__restrict__ x, int d,
                             int vocab) {
  pdl_wait();
  // First kernel of a pass, and in a step the only one that lets the next one start after its own wait (the attention of a pre-fill pass
  // does so too): whatever was written before the pass (positions, the cache of earlier steps) is there for every later kernel of the
  // pass, also before that kernel's wait.
  pdl_trigger();
  const int m = blockIdx.x;
  int t = tok[m];
  t = min(max(t, 0), vocab - 1);
  const T *row = emb + (size_t)t * d;
  for (int i = threadIdx.x; i < d; i += blockDim.x) x[(size_t)m * d + i] = to_f<T>(row[i]);
}

// ------------------------------------------------------------------------------------ RoPE + KV append
// of models with QK-norm; without it both are part of the query-key-value launch (RG_QKV).
template <typename T>
__global__ void rope_append_kernel(const float *__restrict__ qkv, const int32_t *__restrict__ in_pos,
                                   const float2 *__restrict__ rope, float *__restrict__ q, KvLayout kv, RowSegs segs,
                                   int n_heads, QkNorm qkn) {
  pdl_trigger();
  pdl_wait();
  const int m = blockIdx.x;
  const int pos = in_pos[m];
  if (pos < 0) return;
  const int b = seg_sequence(segs, m / segs.rows);
  const int hd = kv.head_dim, half = hd >> 1, nkv = kv.n_kv_heads;
  const int nq = n_heads * hd, nk = nkv * hd;
  const float *row = qkv + (size_t)m * (nq + 2 * nk);
  const float2 *cs = rope + (size_t)pos * half;
  T *cache = reinterpret_cast<T *>(kv.base);
  // rotated pairs of q and k
  for (int i = threadIdx.x; i < (n_heads + nkv) * half; i += blockDim.x) {
    const int head = i / half, j = i % half;
    const float2 c = cs[j];
    // this head's RMS over its hd entries (every thread of the head sums them itself)
    const float *hv = row + (head < n_heads ? head * hd : nq + (head - n_heads) * hd);
    float ss = 0.0f;
    for (int t = 0; t < hd; ++t) ss += hv[t] * hv[t];
    const float rinv = rsqrtf(ss / (float)hd + qkn.eps);
    const T *gain = reinterpret_cast<const T *>(head < n_heads ? qkn.q_gain : qkn.k_gain);
    const float g1 = rinv * to_f<T>(gain[j]), g2 = rinv * to_f<T>(gain[j + half]);
    if (head < n_heads) {
      const float x1 = g1 * row[head * hd + j], x2 = g2 * row[head * hd + j + half];
      q[(size_t)m * nq + head * hd + j] = x1 * c.x - x2 * c.y;
      q[(size_t)m * nq + head * hd + j + half] = x2 * c.x + x1 * c.y;
    } else {
      const int kh = head - n_heads;
      const float x1 = g1 * row[nq + kh * hd + j], x2 = g2 * row[nq + kh * hd + j + half];
      T *dst = cache + kv_row_offset(kv, b, 0, kh, pos);
      dst[j] = from_f<T>(x1 * c.x - x2 * c.y);
      dst[j + half] = from_f<T>(x2 * c.x + x1 * c.y);
    }
  }
  for (int i = threadIdx.x; i < nk; i += blockDim.x) {
    const int kh = i / hd, j = i % hd;
    cache[kv_row_offset(kv, b, 1, kh, pos) + j] = from_f<T>(row[nq + nk + i]);
  }
}

}  // namespace

#define SJD_DISPATCH(dtype, CALL)                         \
  do {                                                    \
    if ((dtype) == SJD_F32) { using T = float; CALL; }    \
    else if ((dtype) == SJD_BF16) { using T = __nv_bfloat16; CALL; } \
    else return SJD_ERR_UNSUPPORTED;                      \
  } while (0)

int launch_gemm_rows(int dtype, const RowsGemm &g, cudaStream_t stream) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0) return SJD_ERR_BAD_ARG;
  SJD_DISPATCH(dtype, return gemm_rows_t<T>(g, stream));
}

int launch_embed(int dtype, const void *tok_emb, const int32_t *tok, float *x, int M, int d, int vocab,
                 cudaStream_t stream) {
  SJD_DISPATCH(dtype, SJD_CUDA(launch_kernel(embed_kernel<T>, dim3(M), dim3(256), 0, stream, reinterpret_cast<const T *>(tok_emb),
                                             tok, x, d, vocab)));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

int launch_rope_append(int dtype, const float *qkv, const int32_t *in_pos, const float2 *rope_table, float *q,
                       KvLayout kv, int M, RowSegs segs, int n_heads, QkNorm qkn, cudaStream_t stream) {
  if (!qkn.q_gain || !qkn.k_gain) return SJD_ERR_BAD_ARG;
  SJD_DISPATCH(dtype, SJD_CUDA(launch_kernel(rope_append_kernel<T>, dim3(M), dim3(256), 0, stream, qkv, in_pos, rope_table, q, kv,
                                             segs, n_heads, qkn)));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

}  // namespace sjd

namespace sjd {
namespace {
// VEC: four entries per thread and round (both sides 16-byte aligned).  Also clears the call's status word.
template <int VEC>
__global__ void split_hilo_kernel(const float *__restrict__ x, HiLoOut o, size_t groups, int *status) {
  pdl_trigger();
  if (status && blockIdx.x == 0 && threadIdx.x == 0) *status = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < groups; i += (size_t)gridDim.x * blockDim.x) {
    if constexpr (VEC == 4) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(x) + i);
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
      const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
      const __nv_bfloat162 l0 = __floats2bfloat162_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2bfloat162_rn(v.z - f1.x, v.w - f1.y);
      *reinterpret_cast<uint2 *>(o.base + i * 4) =
          make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
      *reinterpret_cast<uint2 *>(o.base + o.lo_offset + i * 4) =
          make_uint2(*reinterpret_cast<const uint32_t *>(&l0), *reinterpret_cast<const uint32_t *>(&l1));
    } else {
      store_hilo(o, i, x[i]);
    }
  }
}
}  // namespace

// hi/lo bf16 planes of an fp32 matrix (same row stride; total a multiple of 4), for the tensor-core GEMM
int launch_split_hilo(const float *x, HiLoOut o, size_t total, int *status, cudaStream_t stream) {
  const bool vec = ((uintptr_t)x & 15u) == 0 && total % 4 == 0 && o.lo_offset % 4 == 0;
  const size_t groups = vec ? total / 4 : total;
  const int blocks = (int)((groups + 255) / 256 < 1184 ? (groups + 255) / 256 : 1184);
  if (vec) SJD_CUDA(launch_kernel(split_hilo_kernel<4>, dim3(blocks), dim3(256), 0, stream, x, o, groups, status));
  else SJD_CUDA(launch_kernel(split_hilo_kernel<1>, dim3(blocks), dim3(256), 0, stream, x, o, groups, status));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}
}  // namespace sjd
