// Window-causal attention of the W window queries over the cached prefix plus the in-window causal
// block (Sec. 3.2 / Sec. 4.1 Step 2: one forward pass over the window under a causal mask), as split-KV
// flash decoding: every block owns one (sequence, head, key range), keeps an online softmax per query
// and writes an unnormalised partial; a second kernel merges the partials.  Generic FMA version that
// serves fp32 and bf16 storage with fp32 arithmetic.
#include <float.h>

#include "common.cuh"

namespace sjd {
SJD_TIMELINE_TU(combine)
namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

constexpr int TK = 32;        // keys per tile (one per lane)
constexpr int NWARPS = 8;
constexpr int MAXQ = 8;       // queries per warp: window <= 64
constexpr int MAXD = 4;       // head dims per lane: head_dim <= 128

template <typename T>
__global__ void __launch_bounds__(NWARPS * 32) attention_partial_kernel(
    const float *__restrict__ q, KvLayout kv, const int32_t *__restrict__ in_pos, float *__restrict__ partial,
    RowSegs segs, int n_heads, int splits) {
  extern __shared__ float smem[];
  const int hd = kv.head_dim;
  const int W = segs.rows;
  float *Qs = smem;                       // [W][hd]
  float *Ks = Qs + W * hd;                // [TK][hd + 1]
  float *Vs = Ks + TK * (hd + 1);         // [TK][hd]
  float *Ss = Vs + TK * hd;               // [W][TK]
  __shared__ int s_pos[64];
  __shared__ int s_len;

  pdl_trigger();
  pdl_wait();
  const int h = blockIdx.x, seg = blockIdx.y, s = blockIdx.z;
  const int b = seg_sequence(segs, seg);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int kvh = h / (n_heads / kv.n_kv_heads);
  const int m0 = seg * W;

  if (tid < 64) s_pos[tid] = tid < W ? in_pos[m0 + tid] : -1;
  __syncthreads();
  if (tid == 0) {
    int len = 0;
    for (int i = 0; i < W; ++i) len = max(len, s_pos[i] + 1);
    s_len = len;
  }
  for (int i = tid; i < W * hd; i += blockDim.x) {
    const int qi = i / hd, d = i % hd;
    Qs[i] = q[((size_t)(m0 + qi) * n_heads + h) * hd + d];
  }
  __syncthreads();
  const int len = s_len;
  int chunk = (len + splits - 1) / splits;
  chunk = (chunk + TK - 1) / TK * TK;
  const int k_begin = s * chunk;
  const int k_end = min(len, k_begin + chunk);

  static_assert(KV_PAGE % TK == 0, "a key tile must lie inside one cache page");
  const T *cache = reinterpret_cast<const T *>(kv.base);
  const float scale = rsqrtf((float)hd);

  float m_run[MAXQ], l_run[MAXQ], o[MAXQ][MAXD];
#pragma unroll
  for (int i = 0; i < MAXQ; ++i) {
    m_run[i] = -INFINITY;
    l_run[i] = 0.0f;
#pragma unroll
    for (int j = 0; j < MAXD; ++j) o[i][j] = 0.0f;
  }

  for (int t0 = k_begin; t0 < k_end; t0 += TK) {
    const int nk = min(TK, k_end - t0);
    const T *kbase = cache + kv_row_offset(kv, b, 0, kvh, t0);   // the tile's rows are contiguous
    const T *vbase = cache + kv_row_offset(kv, b, 1, kvh, t0);
    for (int i = tid; i < TK * hd; i += blockDim.x) {
      const int r = i / hd, d = i % hd;
      float kx = 0.0f, vx = 0.0f;
      if (r < nk) {
        kx = to_f<T>(kbase[(size_t)r * hd + d]);
        vx = to_f<T>(vbase[(size_t)r * hd + d]);
      }
      Ks[r * (hd + 1) + d] = kx;
      Vs[r * hd + d] = vx;
    }
    __syncthreads();
    // scores: lane = key, this warp's queries
    float sc[MAXQ];
#pragma unroll
    for (int i = 0; i < MAXQ; ++i) sc[i] = 0.0f;
    for (int d = 0; d < hd; ++d) {
      const float kx = Ks[lane * (hd + 1) + d];
#pragma unroll
      for (int i = 0; i < MAXQ; ++i) {
        const int qi = warp + i * NWARPS;
        if (qi < W) sc[i] = fmaf(Qs[qi * hd + d], kx, sc[i]);
      }
    }
    const int key = t0 + lane;
#pragma unroll
    for (int i = 0; i < MAXQ; ++i) {
      const int qi = warp + i * NWARPS;
      if (qi >= W) continue;
      const bool visible = lane < nk && key <= s_pos[qi];
      const float sv = visible ? sc[i] * scale : -INFINITY;
      const float tmax = warp_max(sv);
      const float m_new = fmaxf(m_run[i], tmax);
      // (no finite score so far: zeros, or the NaN that a maximum does not show)
      const float pexp = visible ? expf(sv - (m_new > -INFINITY ? m_new : 0.0f)) : 0.0f;
      const float alpha = m_run[i] > -INFINITY ? expf(m_run[i] - m_new) : 1.0f;
      const float psum = warp_sum(pexp);
      l_run[i] = l_run[i] * alpha + psum;
      m_run[i] = m_new;
      Ss[qi * TK + lane] = pexp;
#pragma unroll
      for (int j = 0; j < MAXD; ++j) o[i][j] *= alpha;
    }
    __syncwarp();
    // P V: lane = head dims lane, lane+32, ...
#pragma unroll
    for (int i = 0; i < MAXQ; ++i) {
      const int qi = warp + i * NWARPS;
      if (qi >= W) continue;
      for (int kk = 0; kk < nk; ++kk) {
        const float pv = Ss[qi * TK + kk];
#pragma unroll
        for (int j = 0; j < MAXD; ++j) {
          const int d = lane + 32 * j;
          if (d < hd) o[i][j] = fmaf(pv, Vs[kk * hd + d], o[i][j]);
        }
      }
    }
    __syncthreads();
  }

  // partial records: o [row][head][split][hd], then (m, l) [row][head][split]
  float *ml = partial + (size_t)gridDim.y * W * n_heads * splits * hd;
#pragma unroll
  for (int i = 0; i < MAXQ; ++i) {
    const int qi = warp + i * NWARPS;
    if (qi >= W) continue;
    const size_t rec = ((size_t)(m0 + qi) * n_heads + h) * splits + s;
    if (lane == 0) *reinterpret_cast<float2 *>(ml + rec * 2) = make_float2(m_run[i], l_run[i]);
#pragma unroll
    for (int j = 0; j < MAXD; ++j) {
      const int d = lane + 32 * j;
      if (d < hd) partial[rec * hd + d] = o[i][j];
    }
  }
}

// Merge of the key ranges: a warp per (row, head), whose loads are all in flight at once (those of the records do not wait for the
// references): the launch is a link of the chain of a step and costs a round trip or two, not its work.  (A block per (row, head) whose
// threads each read every reference took three round trips with more than eight ranges: 5.8 us of a layer of the 7B step.)
constexpr int kCombineWarps = 4;
constexpr int kCombineSplits = 16;

__global__ void __launch_bounds__(kCombineWarps * 32) attention_combine_kernel(const float *__restrict__ partial,
                                                                               const int32_t *__restrict__ in_pos,
                                                                               float *__restrict__ out, int M, int n_heads, int hd,
                                                                               int splits, HiLoOut hilo) {
  pdl_trigger();
  SJD_TL(TL_COMBINE, 0, threadIdx.x == 0);
  pdl_wait();
  SJD_TL(TL_COMBINE, 1, threadIdx.x == 0);
  const int lane = threadIdx.x & 31, mh = blockIdx.x * kCombineWarps + (threadIdx.x >> 5);
  if (mh >= M * n_heads) return;
  const float *src = partial + (size_t)mh * splits * hd + 2 * lane;
  const float *ml = partial + (size_t)M * n_heads * splits * hd + (size_t)mh * splits * 2;
  const int pos = in_pos[mh / n_heads];
  const float2 r = lane < splits ? *reinterpret_cast<const float2 *>(ml + 2 * lane) : make_float2(-INFINITY, 0.0f);
  const bool on0 = 2 * lane < hd, on1 = 2 * lane + 64 < hd;   // (hd is even)
  float2 v0[kCombineSplits], v1[kCombineSplits];
#pragma unroll
  for (int s = 0; s < kCombineSplits; ++s) {
    v0[s] = v1[s] = make_float2(0.0f, 0.0f);
    if (s < splits && on0) v0[s] = *reinterpret_cast<const float2 *>(src + (size_t)s * hd);
    if (s < splits && on1) v1[s] = *reinterpret_cast<const float2 *>(src + (size_t)s * hd + 64);
  }
  const float g = warp_max(r.x);
  const float wgt = r.x > -INFINITY ? expf(r.x - g) : 0.0f;
  const float denom = warp_sum(r.y * wgt);
  float2 a0 = make_float2(0.0f, 0.0f), a1 = a0;
#pragma unroll
  for (int s = 0; s < kCombineSplits; ++s) {
    if (s >= splits) break;
    const float w = __shfl_sync(0xffffffffu, wgt, s);
    if (w > 0.0f) {   // (the record of an empty range is not written)
      a0.x += v0[s].x * w;
      a0.y += v0[s].y * w;
      a1.x += v1[s].x * w;
      a1.y += v1[s].y * w;
    }
  }
  const bool live = pos >= 0 && denom != 0.0f;   // (a range with a NaN among its scores has a NaN for its sum: the row becomes NaN)
  auto put = [&](int d, float2 a) {
    const float x = live ? a.x / denom : 0.0f, y = live ? a.y / denom : 0.0f;
    const size_t idx = (size_t)mh * hd + d;
    if (out && ((uintptr_t)out & 7u) == 0) {
      *reinterpret_cast<float2 *>(out + idx) = make_float2(x, y);
    } else if (out) {   // (a caller's buffer may start on any float)
      out[idx] = x;
      out[idx + 1] = y;
    }
    if (hilo.base) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
      const float2 f = __bfloat1622float2(h);
      *reinterpret_cast<__nv_bfloat162 *>(hilo.base + idx) = h;
      *reinterpret_cast<__nv_bfloat162 *>(hilo.base + hilo.lo_offset + idx) = __floats2bfloat162_rn(x - f.x, y - f.y);
    }
  };
  if (on0) put(2 * lane, a0);
  if (on1) put(2 * lane + 64, a1);
}

template <typename T>
int attention_t(const float *q, KvLayout kv, const int32_t *in_pos, float *out, float *partial, int M, RowSegs segs,
                int n_heads, int splits, cudaStream_t stream, HiLoOut hilo) {
  const int hd = kv.head_dim, W = segs.rows;
  if (W > NWARPS * MAXQ || hd > 32 * MAXD || M % W != 0) return SJD_ERR_UNSUPPORTED;
  const size_t smem = sizeof(float) * ((size_t)W * hd + TK * (hd + 1) + TK * hd + (size_t)W * TK);
  constexpr int WM = NWARPS * MAXQ, HM = 32 * MAXD;   // the most rows and head entries
  const int rc = allow_smem(attention_partial_kernel<T>, sizeof(float) * (WM * HM + TK * (HM + 1) + TK * HM + WM * TK));
  if (rc != SJD_OK) return rc;
  dim3 grid(n_heads, M / W, splits);
  SJD_CUDA(launch_kernel(attention_partial_kernel<T>, grid, dim3(NWARPS * 32), smem, stream, q, kv, in_pos, partial, segs,
                         n_heads, splits));
  SJD_CHECK_LAUNCH();
  return launch_attention_combine(partial, in_pos, out, M, n_heads, hd, splits, stream, hilo);
}

}  // namespace

int launch_attention_combine(const float *partial, const int32_t *in_pos, float *out, int M, int n_heads, int head_dim,
                             int splits, cudaStream_t stream, HiLoOut hilo) {
  if (splits > kCombineSplits || head_dim > 128) return SJD_ERR_UNSUPPORTED;
  SJD_CUDA(launch_kernel(attention_combine_kernel, dim3((M * n_heads + kCombineWarps - 1) / kCombineWarps), dim3(kCombineWarps * 32), 0,
                         stream, partial, in_pos, out, M, n_heads, head_dim, splits, hilo));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

int launch_attention(int dtype, const float *q, KvLayout kv, const int32_t *in_pos, float *out, float *partial, int M,
                     RowSegs segs, int n_heads, int splits, cudaStream_t stream, HiLoOut hilo) {
  if (dtype == SJD_F32)
    return attention_t<float>(q, kv, in_pos, out, partial, M, segs, n_heads, splits, stream, hilo);
  if (dtype == SJD_BF16)
    return attention_t<__nv_bfloat16>(q, kv, in_pos, out, partial, M, segs, n_heads, splits, stream, hilo);
  return SJD_ERR_UNSUPPORTED;
}

}  // namespace sjd
