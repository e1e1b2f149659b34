// Consumer kernels of the tensor-core path.  The weight-streaming GEMM leaves one fp32 partial plane
// per K split; each kernel here adds the planes in split order (fixed order: deterministic) while doing
// the element-wise work that follows the projection in the decoder layer (Sec. 3.1 / Sec. 4.1 Step 2),
// and emits the next GEMM's activation operand directly as bf16 hi + lo planes.
#include "common.cuh"

namespace sjd {
SJD_TIMELINE_TU(fused)
namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// N adjacent entries (4 or 2, aligned) as fp32
template <int N>
__device__ __forceinline__ void load_gain(const __nv_bfloat16 *p, float *v) {
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const float2 f = __bfloat1622float2(__ldg(reinterpret_cast<const __nv_bfloat162 *>(p + i)));
    v[i] = f.x;
    v[i + 1] = f.y;
  }
}

// Per-row RMS scale from the partial sums of squares a resid_gain launch left:
// scale(m) = 1 / sqrt(mean(x[m]^2) + eps).  The scale is a per-row scalar, so it commutes with the
// projection that follows the normalisation and is applied by that projection's consumer.
// The row index is uniform over the (full) warp: lanes share the loads.  The partials are added in a fixed
// tree order, so every caller gets the same bits.
__device__ __forceinline__ float row_scale_warp(const RowScale &rs, int m) {
  if (!rs.ss_part) return 1.0f;
  const int lane = threadIdx.x & 31;
  float tot = 0.0f;
  for (int j = lane; j < rs.n_part; j += 32) tot += __ldg(rs.ss_part + (size_t)m * rs.n_part + j);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  return rsqrtf(tot * rs.inv_d + rs.eps);
}

// x[m][:] += sum_s P[s][m][:]  (residual connection); emits x * gain as bf16 hi/lo planes (the RMS
// scale is applied downstream) and one partial of sum(x^2) per 128 columns (= per warp, = per weight
// tile of the projections, which write the same partials when they fold this step into their
// epilogue).  Grid (rows, column chunks of 1024).
constexpr int RG_THREADS = 256;
constexpr int RG_COLS = RG_THREADS * 4;

template <typename T>
__global__ void __launch_bounds__(RG_THREADS) resid_gain_kernel(float *__restrict__ x, PlaneSet ps, const T *__restrict__ gain,
                                                               HiLoOut h, float *__restrict__ ss_part, int d) {
  pdl_trigger();
  SJD_TL(TL_RESID, 0, threadIdx.x == 0);
  pdl_wait();
  SJD_TL(TL_RESID, 1, threadIdx.x == 0);
  const int m = blockIdx.x, chunk = blockIdx.y, tid = threadIdx.x;
  const int c0 = chunk * RG_COLS + tid * 4;
  float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (c0 < d) {   // d is a multiple of 4; the gain row may start on any element of its dtype
    float gv[4];
    if (((uintptr_t)gain & 3u) == 0) {
      load_gain<4>(gain + c0, gv);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) gv[i] = to_f<T>(gain[c0 + i]);
    }
    const float4 t = *reinterpret_cast<const float4 *>(x + (size_t)m * d + c0);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    for (int s = 0; s < ps.splits; ++s) {
      const float4 pv = __ldg(reinterpret_cast<const float4 *>(ps.base + (size_t)s * ps.plane_stride + (size_t)m * ps.ld + c0));
      v[0] += pv.x; v[1] += pv.y; v[2] += pv.z; v[3] += pv.w;
    }
    if (ps.splits > 0) *reinterpret_cast<float4 *>(x + (size_t)m * d + c0) = make_float4(v[0], v[1], v[2], v[3]);
    uint2 hi, lo;
    split_pair(v[0] * gv[0], v[1] * gv[1], hi.x, lo.x);
    split_pair(v[2] * gv[2], v[3] * gv[3], hi.y, lo.y);
    *reinterpret_cast<uint2 *>(h.base + (size_t)m * d + c0) = hi;
    *reinterpret_cast<uint2 *>(h.base + h.lo_offset + (size_t)m * d + c0) = lo;
  }
  float ss = v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  ss = warp_sum(ss);
  const int part = chunk * (RG_THREADS / 32) + (tid >> 5), n_part = (d + 127) / 128;
  if ((tid & 31) == 0 && part < n_part) ss_part[(size_t)m * n_part + part] = ss;
  SJD_TL(TL_RESID, 2, threadIdx.x == 0);
}

// q,k,v = scale * sum of the QKV planes; rotate q and k (pairs i, i + hd/2) by the row's absolute
// position; q -> fp32 [M][H*hd]; k, v -> cache row in_pos[m].  A warp per (row, head slot), eight slots per block;
// a lane holds up to two entries of each half of the head: adjacent ones at head_dim 128 (VEC), so that planes, q and cache are
// accessed in 8-byte (cache: 4-byte) groups, else those 32 apart (any even head_dim up to 128).
template <typename T, bool VEC>
__global__ void __launch_bounds__(256) qkv_finish_kernel(PlaneSet ps, RowScale rs, const int32_t *__restrict__ in_pos,
                                                         const float2 *__restrict__ rope, float *__restrict__ q, KvLayout kv,
                                                         RowSegs segs, int n_heads, QkNorm qkn) {
  pdl_trigger();
  SJD_TL(TL_QKV, 0, threadIdx.x == 0);
  pdl_wait();
  SJD_TL(TL_QKV, 1, threadIdx.x == 0);
  constexpr int PER = 2;
  const int HD = VEC ? 128 : kv.head_dim, HALF = HD >> 1;
  const int m = blockIdx.x, lane = threadIdx.x & 31;
  auto at = [&](int i) { return VEC ? lane * 2 + i : lane + 32 * i; };   // entry i of this lane in a half
  auto on = [&](int i) { return VEC || at(i) < HALF; };
  const int nkv = kv.n_kv_heads, nq = n_heads * HD;
  const float *row = ps.base + (size_t)m * ps.ld;
  T *cache = reinterpret_cast<T *>(kv.base);
  // The loads of the projection planes depend on nothing, the row's position and RMS scale are loads of their
  // own and the rotary entry depends on the position: the plane loads of a slot are issued first, so that the
  // kernel waits for two memory round trips in a row and not three.
  int pos = 0, b = 0;
  float sc = 0.0f;
  bool first = true;
  for (int slot = blockIdx.y * 8 + (threadIdx.x >> 5); slot < n_heads + 2 * nkv; slot += gridDim.y * 8) {
    float v[2][PER];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int i = 0; i < PER; ++i) v[h][i] = 0.0f;
      const float *src = row + slot * HD + h * HALF;
#pragma unroll 4
      for (int s = 0; s < ps.splits; ++s) {
        const float *a = src + (size_t)s * ps.plane_stride;
        if constexpr (VEC) {
          const float2 f = __ldg(reinterpret_cast<const float2 *>(a) + lane);
          v[h][0] += f.x;
          v[h][1] += f.y;
        } else {
#pragma unroll
          for (int i = 0; i < PER; ++i)
            if (on(i)) v[h][i] += __ldg(a + at(i));
        }
      }
    }
    if (first) {
      pos = in_pos[m];
      b = seg_sequence(segs, m / segs.rows);
      sc = row_scale_warp(rs, m);
      first = false;
      if (pos < 0) return;
    }
    const bool is_q = slot < n_heads, is_v = slot >= n_heads + nkv;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < PER; ++i) v[h][i] *= sc;
    if (!is_v) {
      if (qkn.q_gain) {   // QK-norm: RMS over the head's entries
        float ss = 0.0f;
#pragma unroll
        for (int i = 0; i < PER; ++i) ss += v[0][i] * v[0][i] + v[1][i] * v[1][i];
        const float rinv = rsqrtf(warp_sum(ss) / (float)HD + qkn.eps);
        const T *gain = reinterpret_cast<const T *>(is_q ? qkn.q_gain : qkn.k_gain);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
          if (!on(i)) continue;
          v[0][i] *= rinv * to_f<T>(gain[at(i)]);
          v[1][i] *= rinv * to_f<T>(gain[at(i) + HALF]);
        }
      }
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (!on(i)) continue;
        const float2 c = rope[(size_t)pos * HALF + at(i)];
        const float r1 = v[0][i] * c.x - v[1][i] * c.y, r2 = v[1][i] * c.x + v[0][i] * c.y;
        v[0][i] = r1;
        v[1][i] = r2;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T *kvd = nullptr;
      if (!is_q) kvd = cache + kv_row_offset(kv, b, is_v ? 1 : 0, slot - n_heads - (is_v ? nkv : 0), pos) + h * HALF;
      float *qd = q + (size_t)m * nq + slot * HD + h * HALF;
      if constexpr (VEC && sizeof(T) == 2) {
        if (is_q) reinterpret_cast<float2 *>(qd)[lane] = make_float2(v[h][0], v[h][1]);
        else reinterpret_cast<__nv_bfloat162 *>(kvd)[lane] = __floats2bfloat162_rn(v[h][0], v[h][1]);
      } else {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
          if (!on(i)) continue;
          if (is_q) qd[at(i)] = v[h][i];
          else kvd[at(i)] = from_f<T>(v[h][i]);
        }
      }
    }
  }
}

}  // namespace

int resid_gain_parts(int d) { return (d + 127) / 128; }

int launch_resid_gain(float *x, PlaneSet ps, const void *gain, HiLoOut h, float *ss_part, int M, int d,
                      cudaStream_t stream) {
  if (d % 4 != 0) return SJD_ERR_UNSUPPORTED;
  const dim3 grid(M, (d + RG_COLS - 1) / RG_COLS);
  SJD_CUDA(launch_kernel(resid_gain_kernel<__nv_bfloat16>, grid, dim3(RG_THREADS), 0, stream, x, ps,
                         reinterpret_cast<const __nv_bfloat16 *>(gain), h, ss_part, d));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

int launch_qkv_finish(PlaneSet ps, RowScale rs, const int32_t *in_pos, const float2 *rope_table, float *q,
                      KvLayout kv, int M, RowSegs segs, int n_heads, QkNorm qkn, cudaStream_t stream) {
  if (kv.head_dim > 128) return SJD_ERR_UNSUPPORTED;
  // a block per eight head slots for a few dozen rows; fewer blocks per row (each walking more slots) as
  // the rows grow, about eight blocks per SM in all
  int per_row = (n_heads + 2 * kv.n_kv_heads + 7) / 8;
  const int cap = 1184 / M > 0 ? 1184 / M : 1;
  per_row = per_row < cap ? per_row : cap;
  auto kernel = kv.head_dim == 128 ? qkv_finish_kernel<__nv_bfloat16, true> : qkv_finish_kernel<__nv_bfloat16, false>;
  SJD_CUDA(launch_kernel(kernel, dim3(M, per_row), dim3(256), 0, stream, ps, rs, in_pos, rope_table, q, kv, segs, n_heads, qkn));
  SJD_CHECK_LAUNCH();
  return SJD_OK;
}

}  // namespace sjd
