// Generic kernels of the decoder forward pass (Sec. 3.1: the auto-regressive transformer; Sec. 4.1
// Step 2: one pass over the window).  These cover every shape and both dtypes with plain FMA
// arithmetic and fp32 accumulation.  Activations between kernels are fp32 (they are a few hundred KB);
// only weights, the KV cache and the stored logits are in the model dtype.
#include "common.cuh"

namespace sjd {
namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// E = 4 adjacent entries (aligned) or one
template <typename T, int E>
__device__ __forceinline__ void load_group(const T *p, float *v) {
  if constexpr (E == 1) {
    v[0] = to_f<T>(p[0]);
  } else if constexpr (sizeof(T) == 4) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
    const uint2 t = *reinterpret_cast<const uint2 *>(p);
    v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xFFFF0000u);
    v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xFFFF0000u);
  }
}

__device__ __forceinline__ void store_hilo(const HiLoOut &o, size_t idx, float v) {
  if (!o.base) return;
  const __nv_bfloat16 hi = __float2bfloat16_rn(v);
  o.base[idx] = hi;
  o.base[o.lo_offset + idx] = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// ------------------------------------------------------------------------------------ projections (FMA)
// A projection of a few rows through small or odd-shaped matrices, where a step is a chain of launches that each cost their
// own latency (two layers of d 256 and 16 rows: 29 launches, 418 us of projections in a 476 us step with 32 x 64 tiles that
// walked K in slices of 32, one dependent load after the other; 14 launches and 101 us a step now).  Hence: one CTA per 16 rows x 8 * NJ weight rows, the
// eight warps split every 256-column chunk of K between them, so that a whole chunk is one round trip to memory, and the
// next chunk is on its way while this one is multiplied.  The RMS normalisation before a projection (its row scale
// commutes with the product), the residual add and SwiGLU are part of the launch.  Any M, N, K; the sums have one fixed order.
constexpr int RG_M = 16, RG_K = 256, RG_LD = RG_K + 4;   // + 4: rows eight apart meet in different banks

// VEC: rows of x and of every matrix can be read in groups of four entries
template <typename T, int NJ, bool VEC>
__global__ void __launch_bounds__(256) gemm_rows_kernel(const RowsGemm g) {
  constexpr int BN = 8 * NJ;
  extern __shared__ float smem[];
  float *xs = smem, *ws = smem + RG_M * RG_LD;
  __shared__ float s_ss[RG_M][8];
  pdl_trigger();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * RG_M, t0 = blockIdx.x;
  const bool glu = g.epilogue == RG_SWIGLU;
  const T *gain = reinterpret_cast<const T *>(g.gain);
  // weight row r of this tile: under SwiGLU the first half of the rows are gate features, the second the same up features
  auto wrow = [&](int r) -> const T * {
    int n, j = 0;
    if (glu) {
      j = r >= BN / 2;
      n = t0 * (BN / 2) + r - j * (BN / 2);
    } else {
      n = t0 * BN + r;
      while (j < 2 && n >= g.n[j]) n -= g.n[j++];
    }
    return n < g.n[j] ? reinterpret_cast<const T *>(g.w[j]) + (size_t)n * g.K : nullptr;
  };
  constexpr int E = VEC ? 4 : 1, PER = 256 / (RG_K / E);        // entries per load, rows per round of the block
  constexpr int NXL = RG_M / PER, NWL = BN / PER;
  const int col = tid % (RG_K / E) * E, r0 = tid / (RG_K / E);
  float xr[NXL][E], wr[NWL][E], gr[E], ss[NXL];
#pragma unroll
  for (int i = 0; i < NXL; ++i) ss[i] = 0.0f;
  auto load_w = [&](int k0) {
    const int k = k0 + col;
#pragma unroll
    for (int i = 0; i < NWL; ++i) {
      const T *row = wrow(r0 + i * PER);
#pragma unroll
      for (int e = 0; e < E; ++e) wr[i][e] = 0.0f;
      if (row && k < g.K) load_group<T, E>(row + k, wr[i]);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) gr[e] = 1.0f;
    if (gain && k < g.K) load_group<T, E>(gain + k, gr);
  };
  auto load_x = [&](int k0) {
    const int k = k0 + col;
#pragma unroll
    for (int i = 0; i < NXL; ++i) {
      const int m = m0 + r0 + i * PER;
#pragma unroll
      for (int e = 0; e < E; ++e) xr[i][e] = 0.0f;
      if (m < g.M && k < g.K) load_group<float, E>(g.x + (size_t)m * g.ldx + k, xr[i]);
    }
  };
  load_w(0);     // the weights do not depend on the kernel before
  pdl_wait();
  load_x(0);
  const int lm = lane >> 3, ln = lane & 7;
  float acc[4][NJ];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = 0.0f;
  for (int k0 = 0; k0 < g.K; k0 += RG_K) {
    if (k0) __syncthreads();
#pragma unroll
    for (int i = 0; i < NXL; ++i)
#pragma unroll
      for (int e = 0; e < E; ++e) {
        ss[i] = fmaf(xr[i][e], xr[i][e], ss[i]);
        xs[(r0 + i * PER) * RG_LD + col + e] = xr[i][e] * gr[e];
      }
#pragma unroll
    for (int i = 0; i < NWL; ++i)
#pragma unroll
      for (int e = 0; e < E; ++e) ws[(r0 + i * PER) * RG_LD + col + e] = wr[i][e];
    __syncthreads();
    if (k0 + RG_K < g.K) {
      load_w(k0 + RG_K);
      load_x(k0 + RG_K);
    }
    const int kw = warp * (RG_K / 8);
#pragma unroll
    for (int k = 0; k < RG_K / 8; k += 4) {
      float4 xv[4], wv[NJ];
#pragma unroll
      for (int i = 0; i < 4; ++i) xv[i] = *reinterpret_cast<const float4 *>(xs + (lm + 4 * i) * RG_LD + kw + k);
#pragma unroll
      for (int j = 0; j < NJ; ++j) wv[j] = *reinterpret_cast<const float4 *>(ws + (ln + 8 * j) * RG_LD + kw + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
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
  for (int i = 0; i < 4; ++i)
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

template <typename T>
int gemm_rows_t(const RowsGemm &g, cudaStream_t stream) {
  const int mt = (g.M + RG_M - 1) / RG_M;
  const int wide = g.epilogue == RG_SWIGLU ? 16 : 32;   // output columns of a CTA with four weight rows per lane
  // two weight rows per lane while that still leaves the grid within one wave (half the work per CTA)
  const bool narrow = mt * ((g.N + wide / 2 - 1) / (wide / 2)) <= 148;
  bool vec = g.K % 4 == 0 && g.ldx % 4 == 0 && ((uintptr_t)g.x & 15u) == 0 && ((uintptr_t)g.gain & (4 * sizeof(T) - 1)) == 0;
  for (int j = 0; j < 3; ++j) vec = vec && ((uintptr_t)g.w[j] & (4 * sizeof(T) - 1)) == 0;
  const int cols = narrow ? wide / 2 : wide, bn = narrow ? 16 : 32;
  const size_t smem = (size_t)(RG_M + bn) * RG_LD * sizeof(float);
  const dim3 grid((g.N + cols - 1) / cols, mt);
  auto launch = [&](auto kernel) -> int {
    const int rc = smem > 40 * 1024 ? allow_smem(kernel, smem) : SJD_OK;   // (the size follows from the kernel's tile)
    if (rc != SJD_OK) return rc;
    SJD_CUDA(launch_kernel(kernel, grid, dim3(256), smem, stream, g));
    SJD_CHECK_LAUNCH();
    return SJD_OK;
  };
  if (narrow) return vec ? launch(gemm_rows_kernel<T, 2, true>) : launch(gemm_rows_kernel<T, 2, false>);
  return vec ? launch(gemm_rows_kernel<T, 4, true>) : launch(gemm_rows_kernel<T, 4, false>);
}

// ------------------------------------------------------------------------------------ embedding
template <typename T>
__global__ void embed_kernel(const T *__restrict__ emb, const int32_t *__restrict__ tok, float *__restrict__ x, int d,
                             int vocab) {
  pdl_trigger();
  pdl_wait();
  const int m = blockIdx.x;
  int t = tok[m];
  t = min(max(t, 0), vocab - 1);
  const T *row = emb + (size_t)t * d;
  for (int i = threadIdx.x; i < d; i += blockDim.x) x[(size_t)m * d + i] = to_f<T>(row[i]);
}

// ------------------------------------------------------------------------------------ RoPE + KV append
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
    float g1 = 1.0f, g2 = 1.0f;
    if (qkn.q_gain) {   // QK-norm: this head's RMS over its hd entries (every thread of the head sums them itself)
      const float *hv = row + (head < n_heads ? head * hd : nq + (head - n_heads) * hd);
      float ss = 0.0f;
      for (int t = 0; t < hd; ++t) ss += hv[t] * hv[t];
      const float rinv = rsqrtf(ss / (float)hd + qkn.eps);
      const T *gain = reinterpret_cast<const T *>(head < n_heads ? qkn.q_gain : qkn.k_gain);
      g1 = rinv * to_f<T>(gain[j]);
      g2 = rinv * to_f<T>(gain[j + half]);
    }
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
