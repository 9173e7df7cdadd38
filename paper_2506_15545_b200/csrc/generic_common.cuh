// Building blocks of the portable fp32-FMA kernels: padded shared-memory tiles, the
// softmax feature map of Section 3.1 on a tile, and register-tiled products
// (16x16 thread grid, strided micro-tiles so float4 shared-memory reads are conflict-free).
#pragma once
#include "rattn_internal.h"

namespace rattn {
namespace generic {

constexpr int NT = 256;       // threads per CTA
constexpr int PAD = 4;        // fp32 padding per smem row (keeps float4 reads conflict-free)

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  uint2 u = *reinterpret_cast<const uint2*>(p);
  __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&u.x);
  __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162*>(&u.y);
  float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
  return make_float4(fa.x, fa.y, fb.x, fb.y);
}
template <typename T> __device__ __forceinline__ void store4(T* p, float4 v);
template <> __device__ __forceinline__ void store4<float>(float* p, float4 v) {
  *reinterpret_cast<float4*>(p) = v;
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
  __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&a);
  u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}

// Where head (b, h) of a caller's tensor with H heads and T rows per head starts, and the distance
// between its rows, in elements: [B, H, T, D] (layout 0) or [B, T, H, D] (layout 1).
template <int D>
__device__ __forceinline__ size_t head_base(int b, int h, int H, int T, int layout) {
  return layout ? ((size_t)b * T * H + h) * D : ((size_t)b * H + h) * (size_t)T * D;
}
template <int D>
__device__ __forceinline__ size_t row_pitch(int H, int layout) { return layout ? (size_t)H * D : (size_t)D; }

// Copy a [ROWS, D] tile (rows row0.., zero beyond n_rows; `pitch` elements between rows) into padded fp32
// shared memory.
template <typename TIO, int D, int ROWS>
__device__ __forceinline__ void load_tile(float* dst, const TIO* src, int row0, int n_rows, int tid, size_t pitch = D) {
  constexpr int LD = D + PAD;
  constexpr int V4 = D / 4;
  for (int i = tid; i < ROWS * V4; i += NT) {
    int r = i / V4, c = (i % V4) * 4;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row0 + r < n_rows) x = load4<TIO>(src + (size_t)(row0 + r) * pitch + c);
    *reinterpret_cast<float4*>(dst + r * LD + c) = x;
  }
}

// phi of each of the ROWS (<= 64) rows of src, written to dst (Section 3.1): softmax over the
// D features, or one of the element-wise maps of the paper's ablation.  Four threads per row.
template <int D, int ROWS>
__device__ __forceinline__ void feature_map_tile(float* dst, const float* src, int tid, int phi) {
  constexpr int LD = D + PAD;
  int r = tid >> 2, part = tid & 3;
  if (r >= ROWS) return;            // whole warps drop out (ROWS is a multiple of 8)
  const float* s = src + r * LD;
  if (phi != RATTN_PHI_SOFTMAX) {
    float* o = dst + r * LD;
    for (int a = part; a < D; a += 4) o[a] = phi == RATTN_PHI_RELU ? fmaxf(s[a], 0.f) : s[a];
    return;
  }
  float m = -INFINITY;
  for (int a = part; a < D; a += 4) m = fmaxf(m, s[a]);
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
  float sum = 0.f;
  float* o = dst + r * LD;
  for (int a = part; a < D; a += 4) {
    float e = __expf(s[a] - m);
    o[a] = e;
    sum += e;
  }
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  float inv = 1.f / sum;
  for (int a = part; a < D; a += 4) o[a] *= inv;
}

// Gradient through the feature map for one element: f = phi(x), df = dL/df, dot = <df, f> over
// the row (used by the softmax map only).
__device__ __forceinline__ float feature_map_grad(int phi, float f, float df, float dot) {
  if (phi == RATTN_PHI_SOFTMAX) return f * (df - dot);
  if (phi == RATTN_PHI_RELU) return f > 0.f ? df : 0.f;       // relu(x) > 0 exactly where x > 0
  return df;
}

__device__ __forceinline__ float group16_max(float x) {
  x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
  x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
  x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 4));
  x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 8));
  return x;
}
__device__ __forceinline__ float group16_sum(float x) {
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 4);
  x += __shfl_xor_sync(0xffffffffu, x, 8);
  return x;
}

// scores[i][j] = sum_a A[ty+16i][a] * Bt[tx+16j][a]   (A has 16*NA rows, Bt has 16*NB rows)
template <int D, int NA, int NB>
__device__ __forceinline__ void tile_scores(float (&s)[NA][NB], const float* A, const float* Bt,
                                            int ty, int tx) {
  constexpr int LD = D + PAD;
#pragma unroll
  for (int i = 0; i < NA; ++i)
#pragma unroll
    for (int j = 0; j < NB; ++j) s[i][j] = 0.f;
#pragma unroll 4
  for (int a = 0; a < D; a += 4) {
    float4 av[NA], bv[NB];
#pragma unroll
    for (int i = 0; i < NA; ++i) av[i] = *reinterpret_cast<const float4*>(A + (ty + 16 * i) * LD + a);
#pragma unroll
    for (int j = 0; j < NB; ++j) bv[j] = *reinterpret_cast<const float4*>(Bt + (tx + 16 * j) * LD + a);
#pragma unroll
    for (int i = 0; i < NA; ++i)
#pragma unroll
      for (int j = 0; j < NB; ++j)
        s[i][j] += av[i].x * bv[j].x + av[i].y * bv[j].y + av[i].z * bv[j].z + av[i].w * bv[j].w;
  }
}

// acc[i][c] += sum_{j<NJ} P[ty+16i][j] * V[j][tx*4 + 64c .. +3]   (P has 16*NA rows of NJ+PAD)
template <int D, int NA, int NJ>
__device__ __forceinline__ void tile_pv(float4 (&acc)[NA][D / 64], const float* P, const float* V,
                                        int ty, int tx) {
  constexpr int LD = D + PAD;
  constexpr int LP = NJ + PAD;
#pragma unroll 2
  for (int j = 0; j < NJ; j += 4) {
    float4 p[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) p[i] = *reinterpret_cast<const float4*>(P + (ty + 16 * i) * LP + j);
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
#pragma unroll
      for (int c = 0; c < D / 64; ++c) {
        float4 v = *reinterpret_cast<const float4*>(V + (j + jj) * LD + tx * 4 + 64 * c);
#pragma unroll
        for (int i = 0; i < NA; ++i) {
          float pv = jj == 0 ? p[i].x : jj == 1 ? p[i].y : jj == 2 ? p[i].z : p[i].w;
          acc[i][c].x += pv * v.x;
          acc[i][c].y += pv * v.y;
          acc[i][c].z += pv * v.z;
          acc[i][c].w += pv * v.w;
        }
      }
    }
  }
}

// ---- chunk states ------------------------------------------------------------------------------
// Over whole chunks of 64 tokens the residual sums are read from running sums of d x d matrices (Eq. 2): S_c = sum over
// the chunks before c of phi(K)^T V for the forward and dq, R_c = sum over the chunks from c on of phi(Q)^T g_r, over the
// group's heads, for dk and dv.  Their terms are formed by a CTA each; a second kernel turns them into the running sums
// in place.  In quadratic form the residual part is O(T^2): at T = 1024, w = 128 the last query tile of a head walked 16
// key tiles, one after another, where it now walks five and a matrix.
constexpr int GC = 64;        // tokens of a chunk

// term[bh, c] = sum over the output's `group` heads of phi(X_c)^T Y_c for the chunks c = first .. first + gridDim.x - 1 of n;
// X (type TX) is mapped through phi, Y (type TY) taken as it is; both have H_out * group heads per batch entry.
template <typename TX, typename TY, int D>
__global__ void __launch_bounds__(NT) chunk_term_kernel(const TX* __restrict__ x, const TY* __restrict__ y, float* __restrict__ out,
                                                        int T, int H_out, int group, int x_layout, int y_layout, int phi,
                                                        int first, int n) {
  constexpr int LD = D + PAD, M = D / 16;
  extern __shared__ __align__(16) float smem[];
  float* Xs = smem;
  float* Fs = Xs + GC * LD;
  float* Ys = Fs + GC * LD;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int c = first + blockIdx.x, bh = blockIdx.y, b = bh / H_out, ho = bh - b * H_out, H = H_out * group;
  float acc[M][M];
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M; ++j) acc[i][j] = 0.f;
  for (int g = 0; g < group; ++g) {
    const int h = ho * group + g;
    __syncthreads();
    load_tile<TX, D, GC>(Xs, x + head_base<D>(b, h, H, T, x_layout), c * GC, T, tid, row_pitch<D>(H, x_layout));
    load_tile<TY, D, GC>(Ys, y + head_base<D>(b, h, H, T, y_layout), c * GC, T, tid, row_pitch<D>(H, y_layout));
    __syncthreads();
    feature_map_tile<D, GC>(Fs, Xs, tid, phi);          // a row beyond T maps to something, but its Y row is zero
    __syncthreads();
#pragma unroll 2
    for (int t = 0; t < GC; ++t) {
      float f[M], v[M];
#pragma unroll
      for (int i = 0; i < M; i += 4) {
        *reinterpret_cast<float4*>(f + i) = *reinterpret_cast<const float4*>(Fs + t * LD + ty * 4 + 16 * i);
        *reinterpret_cast<float4*>(v + i) = *reinterpret_cast<const float4*>(Ys + t * LD + tx * 4 + 16 * i);
      }
#pragma unroll
      for (int i = 0; i < M; ++i)
#pragma unroll
        for (int j = 0; j < M; ++j) acc[i][j] += f[i] * v[j];
    }
  }
  float* o = out + ((size_t)bh * n + c) * D * D;
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M; j += 4)
      *reinterpret_cast<float4*>(o + (size_t)(ty * 4 + 16 * (i & ~3) + (i & 3)) * D + tx * 4 + 16 * j) =
          make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
}

// In place along the first (suffix = 0) or last (1) n_chunks of each head's n slots: suffix = 0: slot c := sum of the slots
// before it (the last slot has no term of its own); 1: sum of the slots from it on.  A thread walks one float4 of the
// matrix, eight loads in flight.
static __global__ void __launch_bounds__(256) chunk_sum_kernel(float4* __restrict__ s, int n_chunks, int n, int vecs, int suffix) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= vecs) return;
  float4* p = s + (size_t)blockIdx.y * n * vecs + i + (suffix ? (size_t)(n - 1) * vecs : 0);
  const int n_terms = suffix ? n_chunks : n_chunks - 1;
  const ptrdiff_t step = suffix ? -(ptrdiff_t)vecs : (ptrdiff_t)vecs;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c0 = 0; c0 < n_chunks; c0 += 8) {
    float4 d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = c0 + k < n_terms ? p[(c0 + k) * step] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (c0 + k >= n_chunks) break;
      if (!suffix) p[(c0 + k) * step] = acc;
      acc.x += d[k].x; acc.y += d[k].y; acc.z += d[k].z; acc.w += d[k].w;
      if (suffix) p[(c0 + k) * step] = acc;
    }
  }
}

// Forms the states that some tile reads, where the sizes leave any: a tile of 32 (or 64) query rows from q0 on reads S_c for
// c = (q0 - w) / 64, one of 32 (or 64) key rows from j0 on R_c for c = (j0 + 32 + w) / 64 rounded up, or a later one.  With a
// window about as long as the sequence that is next to nothing (64/16 heads of 64, T = 100, w = 512: the states of all
// chunks took 16 of a training step's 178 us for nobody).
template <typename TX, typename TY, int D>
cudaError_t launch_chunk_states(const TX* x, const TY* y, float* out, int B, int T, int w, int H_out, int group, int x_layout,
                                int y_layout, int phi, int suffix, cudaStream_t s) {
  const int n = (T + GC - 1) / GC, q_last = (T - 1) / 32 * 32;
  const int n_sums = suffix ? n - (int)(((long long)w + 32 + GC - 1) / GC) : q_last > w ? (q_last - w) / GC + 1 : 0;
  const int n_terms = suffix ? n_sums : n_sums - 1, first = suffix ? n - n_terms : 0;      // (S_c takes the chunks before c)
  if (n_terms <= 0) return cudaSuccess;
  constexpr int smem = 3 * GC * (D + PAD) * (int)sizeof(float);
  const cudaError_t e = allow_smem<chunk_term_kernel<TX, TY, D>>(smem);
  if (e != cudaSuccess) return e;
  { KernelTimer kt("generic_terms", s);
    chunk_term_kernel<TX, TY, D><<<dim3(n_terms, B * H_out), NT, smem, s>>>(x, y, out, T, H_out, group, x_layout, y_layout, phi,
                                                                            first, n); }
  { KernelTimer kt("generic_sums", s);
    chunk_sum_kernel<<<dim3((D * D / 4 + 255) / 256, B * H_out), 256, 0, s>>>(reinterpret_cast<float4*>(out), n_sums, n, D * D / 4,
                                                                              suffix); }
  count_launches(2);
  return cudaGetLastError();
}

// acc[i][c] += sum_f P[ty+16i][f] * M[f][tx*4 + 64c ..] over all D columns of the fp32 tile P (16*NA rows) and the D x D
// matrix m in global memory (transposed: M[f][v] = m[v][f]), 64 rows of M at a time through `stage` ([64][D+PAD]) and the
// column slice of P through `slice` ([16*NA][64+PAD]).
template <int D, int NA>
__device__ __forceinline__ void tile_matrix(float4 (&acc)[NA][D / 64], const float* P, const float* m, bool transposed,
                                            float* stage, float* slice, int tid, int ty, int tx) {
  constexpr int LD = D + PAD, LP = 64 + PAD;
  for (int f0 = 0; f0 < D; f0 += 64) {
    __syncthreads();
    if (!transposed) {
      for (int i = tid; i < 64 * (D / 4); i += NT) {
        const int r = i / (D / 4), c = (i % (D / 4)) * 4;
        *reinterpret_cast<float4*>(stage + r * LD + c) = *reinterpret_cast<const float4*>(m + (size_t)(f0 + r) * D + c);
      }
    } else {
      for (int i = tid; i < D * 16; i += NT) {
        const int r = i >> 4, c = (i & 15) * 4;          // row r of m, columns f0 + c ..: column r of the stage
        const float4 v = *reinterpret_cast<const float4*>(m + (size_t)r * D + f0 + c);
        stage[(c + 0) * LD + r] = v.x;
        stage[(c + 1) * LD + r] = v.y;
        stage[(c + 2) * LD + r] = v.z;
        stage[(c + 3) * LD + r] = v.w;
      }
    }
    for (int i = tid; i < 16 * NA * 64; i += NT) {
      const int r = i >> 6, c = i & 63;
      slice[r * LP + c] = P[r * LD + f0 + c];
    }
    __syncthreads();
    tile_pv<D, NA, 64>(acc, slice, stage, ty, tx);
  }
}

}  // namespace generic
}  // namespace rattn
