// Pieces shared by the tensor-core kernels (forward and backward): the shared-memory tile
// layout a 128-byte-swizzled TMA load produces, the tcgen05 operand descriptors for it, the
// 128 x 128 x 128 MMA chains, the in-place feature map and the host-side tensor maps.
#pragma once

#include <cuda_fp16.h>

#include "rattn_internal.h"
#include "tc_ptx.cuh"

namespace rattn {
namespace tc {

using namespace ptx;

constexpr int TILE = 128;
constexpr int HALF_BYTES = TILE * 64 * 2;   // one [128 x 64] bf16 sub-tile, 128-byte rows
constexpr int TILE_BYTES = 2 * HALF_BYTES;

// Operand descriptors.  The descriptor of a tile is built once from its base address; the
// eight (or four) reduction steps of a product then only add a constant to its start-address
// field (bytes / 16; shared-memory addresses stay below 2^18, so the field never carries).
//   K-major operand: [128 rows x 128 reduction] as two 64-wide halves; 16 reduction elements
//   per MMA = 32 bytes along the 128-byte row.
//   MN-major operand: rows are the reduction index (128-byte rows of 64 columns, two column
//   halves 16 KB apart); 16 reduction rows per MMA = 2048 bytes.
__device__ __forceinline__ uint64_t kmajor_base(uint32_t base) { return smem_desc(base, 16, 1024); }
__device__ __forceinline__ uint64_t mnmajor_base(uint32_t base) { return smem_desc(base, HALF_BYTES, 1024); }
__host__ __device__ constexpr uint32_t kstep_k(int k, int half_bytes) { return (uint32_t)(((k >> 2) * half_bytes + (k & 3) * 32) >> 4); }
__host__ __device__ constexpr uint32_t kstep_mn(int k) { return (uint32_t)((k * 2048) >> 4); }
__device__ __forceinline__ uint64_t mnmajor_desc(uint32_t base, int kstep) { return mnmajor_base(base) + kstep_mn(kstep); }

// D[128x128] (+)= A B^T-style products over a reduction of 128, 8 MMAs of K = 16.  (Unrolled on
// purpose: with rolled issue loops the MMA warps, which sit on the critical path, measured 6-25 % slower.)
__device__ __forceinline__ void mma_kk(uint32_t d, uint32_t a_base, uint32_t b_base, bool acc) {
  constexpr uint32_t idesc = instr_desc(128, 128, 0, 0);
  const uint64_t a0 = kmajor_base(a_base), b0 = kmajor_base(b_base);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    mma_bf16(d, a0 + kstep_k(k, HALF_BYTES), b0 + kstep_k(k, HALF_BYTES), idesc, (acc || k > 0) ? 1u : 0u);
}
template <int AB_BF16>
__device__ __forceinline__ void mma_kmn(uint32_t d, uint32_t a_base, uint32_t b_base, bool acc) {
  constexpr uint32_t idesc = instr_desc(128, 128, 0, 1, AB_BF16);
  const uint64_t a0 = kmajor_base(a_base), b0 = mnmajor_base(b_base);
#pragma unroll
  for (int k = 0; k < 8; ++k) mma_bf16(d, a0 + kstep_k(k, HALF_BYTES), b0 + kstep_mn(k), idesc, (acc || k > 0) ? 1u : 0u);
}
__device__ __forceinline__ void mma_mnmn(uint32_t d, uint32_t a_base, uint32_t b_base, bool acc) {
  constexpr uint32_t idesc = instr_desc(128, 128, 1, 1);
  const uint64_t a0 = mnmajor_base(a_base), b0 = mnmajor_base(b_base);
#pragma unroll
  for (int k = 0; k < 8; ++k) mma_bf16(d, a0 + kstep_mn(k), b0 + kstep_mn(k), idesc, (acc || k > 0) ? 1u : 0u);
}

// ---- half tiles: [64 rows x 128 columns] bf16 as two [64 x 64] boxes of 8 KB ------------
constexpr int HT_HALF = 64 * 64 * 2;
constexpr int HT_BYTES = 2 * HT_HALF;
// B operand, K-major: the half tile's 64 rows are N, its 128 columns the reduction (8 steps)
__device__ __forceinline__ uint64_t kmajor_base_h(uint32_t base) { return smem_desc(base, 16, 1024); }
// B operand, MN-major: the half tile's 128 columns are N, its 64 rows the reduction (4 steps)
__device__ __forceinline__ uint64_t mnmajor_base_h(uint32_t base) { return smem_desc(base, HT_HALF, 1024); }
// D[128 x 64] = A[128 x 128] (K-major full tile) . B[64 x 128]^T (K-major half tile)
__device__ __forceinline__ void mma_k_kh(uint32_t d, uint32_t a_base, uint32_t b_base) {
  constexpr uint32_t idesc = instr_desc(128, 64, 0, 0);
  const uint64_t a0 = kmajor_base(a_base), b0 = kmajor_base_h(b_base);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    mma_bf16(d, a0 + kstep_k(k, HALF_BYTES), b0 + kstep_k(k, HT_HALF), idesc, k > 0 ? 1u : 0u);
}
// D[128 x 128] (+)= A[128 x 64] (bf16 in TMEM, 32 columns) . B[64 x 128] (MN-major half tile)
__device__ __forceinline__ void mma_ts_h(uint32_t d, uint32_t a_tmem, uint32_t b_base, bool acc) {
  constexpr uint32_t idesc = instr_desc(128, 128, 0, 1);
  const uint64_t b0 = mnmajor_base_h(b_base);
#pragma unroll
  for (int k = 0; k < 4; ++k) mma_bf16_ts(d, a_tmem + 8 * k, b0 + kstep_mn(k), idesc, (acc || k > 0) ? 1u : 0u);
}
// A caller's tensor (q, k, v, out and the gradients): its heads may be dense ([B, H, T, d]) or interleaved
// ([B, T, H, d]), so its map has four dimensions (d, T, H, B) and a matrix index z = b * H + h is split.
struct alignas(64) UMap {
  CUtensorMap m;
  int H;
};
__device__ __forceinline__ void prefetch_map(const UMap* tm) { prefetch_tensormap(&tm->m); }
__device__ __forceinline__ void load_tile(unsigned char* dst, const UMap* tm, uint64_t* bar, int row, int z) {
  const int b = z / tm->H, h = z - b * tm->H;
  tma_load_4d(dst, &tm->m, bar, 0, row, h, b);
  tma_load_4d(dst + HALF_BYTES, &tm->m, bar, 64, row, h, b);
}
// `tm` must have a [64 columns x 64 rows] box
__device__ __forceinline__ void load_half_tile(unsigned char* dst, const UMap* tm, uint64_t* bar, int row, int z) {
  const int b = z / tm->H, h = z - b * tm->H;
  tma_load_4d(dst, &tm->m, bar, 0, row, h, b);
  tma_load_4d(dst + HT_HALF, &tm->m, bar, 64, row, h, b);
}
__device__ __forceinline__ void load_tile(unsigned char* dst, const CUtensorMap* tm, uint64_t* bar, int row, int z) {
  tma_load_3d(dst, tm, bar, 0, row, z);
  tma_load_3d(dst + HALF_BYTES, tm, bar, 64, row, z);
}
// `tm` must have a [64 columns x 64 rows] box
__device__ __forceinline__ void load_half_tile(unsigned char* dst, const CUtensorMap* tm, uint64_t* bar, int row, int z) {
  tma_load_3d(dst, tm, bar, 0, row, z);
  tma_load_3d(dst + HT_HALF, tm, bar, 64, row, z);
}

// The element-wise maps of the paper's ablation (Table 6) on packed bf16 pairs: ReLU; the
// identity needs no arithmetic at all.
__device__ __forceinline__ uint4 relu_bf16x8(uint4 u) {
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
  const __nv_bfloat162 z = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
  for (int e = 0; e < 4; ++e) h[e] = __hmax2(h[e], z);
  return u;
}
// phi over the 128 features of one row by a pair of adjacent lanes, of which this one (`ch`, its parity) owns the 64
// columns of one column half; `src` and `dst` point at that half of the row (128 bytes, chunks swizzled by row & 7) and may
// be the same.  normalise = false: the softmax map leaves exp(x - max).  Returns 1 / sum (1 for the element-wise maps) for
// callers that scale whatever is linear in the row afterwards.  The two lanes walk the chunks four apart: the halves lie
// a multiple of 8 KB from each other, and in the same order both lanes would meet in the same banks.
__device__ __forceinline__ float feature_map_half_row(const unsigned char* src, unsigned char* dst, int row, int ch, int phi,
                                                      bool normalise) {
  const int sw = (row & 7) ^ (ch << 2);
  if (phi != RATTN_PHI_SOFTMAX) {
    if (phi == RATTN_PHI_IDENTITY && src == dst) return 1.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint4 u = *reinterpret_cast<const uint4*>(src + ((c ^ sw) << 4));
      *reinterpret_cast<uint4*>(dst + ((c ^ sw) << 4)) = phi == RATTN_PHI_RELU ? relu_bf16x8(u) : u;
    }
    return 1.f;
  }
  float x[64], m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint4 u = *reinterpret_cast<const uint4*>(src + ((c ^ sw) << 4));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      x[c * 8 + 2 * e] = __uint_as_float(w[e] << 16);
      x[c * 8 + 2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
      m0 = fmaxf(m0, x[c * 8 + 2 * e]);
      m1 = fmaxf(m1, x[c * 8 + 2 * e + 1]);
    }
  }
  float m = fmaxf(m0, m1);
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
  const float ml = m * 1.4426950408889634f;
  const float2 l2e = make_float2(1.4426950408889634f, 1.4426950408889634f), nml = make_float2(-ml, -ml);
  float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 64; i += 2) {
    const float2 y = __ffma2_rn(make_float2(x[i], x[i + 1]), l2e, nml);
    const float2 p = make_float2(ex2(y.x), ex2(y.y));
    x[i] = p.x;
    x[i + 1] = p.y;
    if (i & 2) s1 = __fadd2_rn(s1, p);
    else s0 = __fadd2_rn(s0, p);
  }
  float sum = (s0.x + s0.y) + (s1.x + s1.y);
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  const float inv = 1.f / sum, sc = normalise ? inv : 1.f;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    *reinterpret_cast<uint4*>(dst + ((c ^ sw) << 4)) =
        make_uint4(pack_bf16(x[c * 8 + 0] * sc, x[c * 8 + 1] * sc), pack_bf16(x[c * 8 + 2] * sc, x[c * 8 + 3] * sc),
                   pack_bf16(x[c * 8 + 4] * sc, x[c * 8 + 5] * sc), pack_bf16(x[c * 8 + 6] * sc, x[c * 8 + 7] * sc));
  return inv;
}
// ... normalised, by four lanes per row, of which this one (q) owns 32 columns; `src` and `dst` point at the row in the
// first column half's box, the second half's lies `half_stride` behind.
// PAIR_SUMS = false: q = lane & 3.  A quarter-warp (two rows) touches every bank once: the lanes of the second half walk
// their chunks two apart from the first's.
// PAIR_SUMS = true: the softmax map's sums are formed in feature_map_half_row's order, so that both leave the same bits:
// of a half's two lanes (q, q ^ 1: neighbours; the other half's lie 8 lanes away) the second carries on from the first's
// partial sums.  A quarter-warp touches every bank once with one half of four rows.
template <bool PAIR_SUMS = false>
__device__ __forceinline__ void feature_map_quad(const unsigned char* src, unsigned char* dst, int half_stride, int row, int q,
                                                 int phi) {
  const int sw = (row & 7) ^ ((q & 1) << 2) ^ (PAIR_SUMS ? 0 : q & 2);
  src += (q >> 1) * half_stride;
  dst += (q >> 1) * half_stride;
  if (phi != RATTN_PHI_SOFTMAX) {
    if (phi == RATTN_PHI_IDENTITY && src == dst) return;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const uint4 u = *reinterpret_cast<const uint4*>(src + ((c ^ sw) << 4));
      *reinterpret_cast<uint4*>(dst + ((c ^ sw) << 4)) = phi == RATTN_PHI_RELU ? relu_bf16x8(u) : u;
    }
    return;
  }
  float x[32];
  __nv_bfloat162 mx[4];                                   // packed: two values per instruction
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint4 u = *reinterpret_cast<const uint4*>(src + ((c ^ sw) << 4));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(w);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      x[c * 8 + 2 * e] = __uint_as_float(w[e] << 16);
      x[c * 8 + 2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
      mx[e] = c == 0 ? h[e] : __hmax2(mx[e], h[e]);
    }
  }
  const float2 m2 = __bfloat1622float2(__hmax2(__hmax2(mx[0], mx[1]), __hmax2(mx[2], mx[3])));
  float m = fmaxf(m2.x, m2.y);
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, PAIR_SUMS ? 8 : 2));
  const float ml = m * 1.4426950408889634f;
  const float2 l2e = make_float2(1.4426950408889634f, 1.4426950408889634f), nml = make_float2(-ml, -ml);
  float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    const float2 y = __ffma2_rn(make_float2(x[i], x[i + 1]), l2e, nml);
    const float2 p = make_float2(ex2(y.x), ex2(y.y));
    x[i] = p.x;
    x[i + 1] = p.y;
    if (i & 2) s1 = __fadd2_rn(s1, p);
    else s0 = __fadd2_rn(s0, p);
  }
  float sum;
  if (PAIR_SUMS) {
    // a pair's lane walks the first half's chunks 0 .. 7, the second half's 4 .. 7, 0 .. 3: first are q = 0 and q = 3
    s0.x = __shfl_xor_sync(0xffffffffu, s0.x, 1); s0.y = __shfl_xor_sync(0xffffffffu, s0.y, 1);
    s1.x = __shfl_xor_sync(0xffffffffu, s1.x, 1); s1.y = __shfl_xor_sync(0xffffffffu, s1.y, 1);
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
      s0 = __fadd2_rn(s0, make_float2(x[i], x[i + 1]));
      s1 = __fadd2_rn(s1, make_float2(x[i + 2], x[i + 3]));
    }
    sum = (s0.x + s0.y) + (s1.x + s1.y);                  // of a half, in q = 1 and q = 2
    const int lane0 = (int)(threadIdx.x & 31) & ~9;       // q = 0 of this row
    sum = __shfl_sync(0xffffffffu, sum, lane0 + 1) + __shfl_sync(0xffffffffu, sum, lane0 + 8);
  } else {
    sum = (s0.x + s0.y) + (s1.x + s1.y);
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  }
  const float sc = 1.f / sum;
  const float2 sc2 = make_float2(sc, sc);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 y = __fmul2_rn(make_float2(x[c * 8 + 2 * e], x[c * 8 + 2 * e + 1]), sc2);
      w[e] = pack_bf16(y.x, y.y);
    }
    *reinterpret_cast<uint4*>(dst + ((c ^ sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// byte offset of 16-byte chunk c (0..15) of row r inside a swizzled [128 x 128] bf16 tile
__device__ __forceinline__ uint32_t swz(int r, int c) {
  return (uint32_t)((c >> 3) * HALF_BYTES + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}

// x[i] *= g[i] for 16 consecutive columns; every lane reads the same 64 bytes, as four 16-byte loads (gains are 16-byte
// aligned and 16 columns are 64 bytes).
__device__ __forceinline__ void apply_gain16(float (&x)[16], const float* __restrict__ g) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(g) + i);
    x[4 * i] *= v.x; x[4 * i + 1] *= v.y; x[4 * i + 2] *= v.z; x[4 * i + 3] *= v.w;
  }
}

// 64 threads bring a head's two gain vectors into L1 (16 bytes each): consecutive units of a CTA are units of other heads, and
// by the epilogue's own loads, in sixteen batches, each an L2 latency, the gains took a tenth of a long prefill's time.
__device__ __forceinline__ void prefetch_gains(const float* g_swa, const float* g_rla, int head, int i) {
  const float* g = i < 32 ? g_swa : g_rla;
  if (!g) return;
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(g + (size_t)head * 128 + 4 * (i & 31)));
}

// One [128 x 128] bf16 tile staged in shared memory (swizzled like a loaded tile) goes to
// rows row0.. of matrix z of a tensor map: two 64-column boxes; rows past the end are clipped.
__device__ __forceinline__ void store_tile(const UMap* tm, const unsigned char* tile, int row0, int z) {
  const int b = z / tm->H, h = z - b * tm->H;
  tma_store_4d(&tm->m, tile, 0, row0, h, b);
  tma_store_4d(&tm->m, tile + HALF_BYTES, 64, row0, h, b);
}
// one 64-column half of a staged tile
__device__ __forceinline__ void store_half(const UMap* tm, const unsigned char* half, int x, int row0, int z) {
  const int b = z / tm->H, h = z - b * tm->H;
  tma_store_4d(&tm->m, half, x, row0, h, b);
}
__device__ __forceinline__ void store_half(const CUtensorMap* tm, const unsigned char* half, int x, int row0, int z) {
  tma_store_3d(tm, half, x, row0, z);
}
__device__ __forceinline__ void store_tile(const CUtensorMap* tm, const unsigned char* tile, int row0, int z) {
  tma_store_3d(tm, tile, 0, row0, z);
  tma_store_3d(tm, tile + HALF_BYTES, 64, row0, z);
}

// Bit e of the result says whether column 32*c + e of a [128 x 128] score tile is kept for row
// r: on the diagonal tile the keys j <= r, on the oldest tile of the band the keys j >= r.
__device__ __forceinline__ uint32_t keep_bits(int r, int c, bool diag, bool bound) {
  const int rd = r - 32 * c;                      // column of the row's own position in this chunk
  uint32_t m = 0xffffffffu;
  if (diag) m &= rd >= 31 ? 0xffffffffu : (rd < 0 ? 0u : ((2u << rd) - 1u));
  if (bound) m &= rd <= 0 ? 0xffffffffu : (rd > 31 ? 0u : ~((1u << rd) - 1u));
  return m;
}

// bits e >= rd, e > rd, e <= rd of a 32-bit chunk mask (any integer rd)
__device__ __forceinline__ uint32_t bits_ge(int rd) { return rd <= 0 ? 0xffffffffu : (rd > 31 ? 0u : ~((1u << rd) - 1u)); }
__device__ __forceinline__ uint32_t bits_gt(int rd) { return bits_ge(rd + 1); }
__device__ __forceinline__ uint32_t bits_le(int rd) { return ~bits_gt(rd); }
__device__ __forceinline__ uint32_t bits_lt(int rd) { return ~bits_ge(rd); }

// Maximum of 32 registers as four independent chains (the row threads run two or three warps per
// scheduler, so a 32-long dependent chain would sit exposed at full latency).
__device__ __forceinline__ float max32(const float (&x)[32]) {
  float m0 = x[0], m1 = x[1], m2 = x[2], m3 = x[3];
#pragma unroll
  for (int e = 4; e < 32; e += 4) {
    m0 = fmaxf(m0, x[e]);
    m1 = fmaxf(m1, x[e + 1]);
    m2 = fmaxf(m2, x[e + 2]);
    m3 = fmaxf(m3, x[e + 3]);
  }
  return fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
}
// columns whose keep bit is clear become -inf: no part in the maximum, weight exactly zero
__device__ __forceinline__ void mask32(float (&x)[32], uint32_t keep) {
#pragma unroll
  for (int e = 0; e < 32; ++e) x[e] = (keep >> e) & 1u ? x[e] : -INFINITY;
}
// The helpers below walk a row in sixteen 16-byte steps with a rolled loop: compact code
// matters more than loop overhead here (large unrolled kernels are instruction-fetch bound).
// Row maximum of row r of a swizzled bf16 tile.
__device__ __forceinline__ float row_max_bf16(const unsigned char* tile, int r) {
  // packed bf16 maxima (two values per instruction), four independent chains
  __nv_bfloat162 m[4];
  {
    const uint4 u = *reinterpret_cast<const uint4*>(tile + swz(r, 0));
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = h[e];
  }
#pragma unroll 3
  for (int c = 1; c < 16; ++c) {
    const uint4 u = *reinterpret_cast<const uint4*>(tile + swz(r, c));
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int e = 0; e < 4; ++e) m[e] = __hmax2(m[e], h[e]);
  }
  const float2 f = __bfloat1622float2(__hmax2(__hmax2(m[0], m[1]), __hmax2(m[2], m[3])));
  return fmaxf(f.x, f.y);
}
// x -> exp(x - max) over row r, in place, as fp16 (FP16 = true) or bf16; returns the row sum.
template <bool FP16>
__device__ __forceinline__ float row_exp_inplace(unsigned char* tile, int r, float ml) {
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 2
  for (int c = 0; c < 16; ++c) {
    uint4 u = *reinterpret_cast<const uint4*>(tile + swz(r, c));
    uint32_t* w = reinterpret_cast<uint32_t*>(&u);
    float ex[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
      ex[2 * e] = ex2(f.x * 1.4426950408889634f - ml);
      ex[2 * e + 1] = ex2(f.y * 1.4426950408889634f - ml);
      w[e] = FP16 ? pack_f16(ex[2 * e], ex[2 * e + 1]) : pack_bf16(ex[2 * e], ex[2 * e + 1]);
    }
    s0 += ex[0] + ex[4];
    s1 += ex[1] + ex[5];
    s2 += ex[2] + ex[6];
    s3 += ex[3] + ex[7];
    *reinterpret_cast<uint4*>(tile + swz(r, c)) = u;
  }
  return (s0 + s1) + (s2 + s3);
}
// Un-normalised feature map of row r, in place: x -> exp(x - max) (bf16); returns 1 / sum so
// that the caller can scale whatever is linear in this row afterwards.
__device__ __forceinline__ float feature_map_row_unnorm_inplace(unsigned char* tile, int r) {
  const float ml = row_max_bf16(tile, r) * 1.4426950408889634f;
  return 1.f / row_exp_inplace<false>(tile, r, ml);
}
// phi of row r, in place, with few live registers: the exponentials are parked in the tile
// itself as fp16 between the summation and the normalisation (one bf16 rounding in the end).
__device__ __forceinline__ void feature_map_row_inplace_lr(unsigned char* tile, int r) {
  const float ml = row_max_bf16(tile, r) * 1.4426950408889634f;
  const float inv = 1.f / row_exp_inplace<true>(tile, r, ml);
#pragma unroll 1
  for (int c = 0; c < 16; ++c) {
    uint4 u = *reinterpret_cast<const uint4*>(tile + swz(r, c));
    uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
      w[e] = pack_bf16(f.x * inv, f.y * inv);
    }
    *reinterpret_cast<uint4*>(tile + swz(r, c)) = u;
  }
}

// phi (softmax over the 128 features) of row r of a swizzled bf16 tile, in place.
// NORMALISE = false leaves exp(x - max) (bf16) and returns 1 / sum, for callers that scale
// whatever is linear in this row afterwards.  The row lives in 128 registers in between: one
// read and one write of shared memory.
template <bool NORMALISE = true>
__device__ __forceinline__ float feature_map_row_inplace(unsigned char* tile, int r) {
  float x[128];
  float m = -INFINITY;
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    uint4 u = *reinterpret_cast<const uint4*>(tile + swz(r, c));
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float2 f = __bfloat1622float2(h[e]);
      x[c * 8 + 2 * e] = f.x;
      x[c * 8 + 2 * e + 1] = f.y;
      m = fmaxf(m, fmaxf(f.x, f.y));
    }
  }
  float sum = 0.f;
  const float ml = m * 1.4426950408889634f;
#pragma unroll
  for (int i = 0; i < 128; ++i) {
    x[i] = ex2(x[i] * 1.4426950408889634f - ml);
    sum += x[i];
  }
  const float inv = 1.f / sum, sc = NORMALISE ? inv : 1.f;
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    uint4 u;
    u.x = pack_bf16(x[c * 8 + 0] * sc, x[c * 8 + 1] * sc);
    u.y = pack_bf16(x[c * 8 + 2] * sc, x[c * 8 + 3] * sc);
    u.z = pack_bf16(x[c * 8 + 4] * sc, x[c * 8 + 5] * sc);
    u.w = pack_bf16(x[c * 8 + 6] * sc, x[c * 8 + 7] * sc);
    *reinterpret_cast<uint4*>(tile + swz(r, c)) = u;
  }
  return inv;
}

// phi of row r of a swizzled bf16 tile, in place, for any map.  NORMALISE = false: the softmax
// map leaves exp(x - max) and returns 1 / sum (see feature_map_row_inplace); the element-wise
// maps have no normalisation and return 1.
// The softmax map comes in two forms: fully unrolled with the row in 128 registers (one read and one
// write of shared memory, but 16 KB of code per call site) and compact (rolled loops, two or three
// passes over the row in shared memory, twice the cycles).  The kernels that call this are larger
// than the instruction cache; a caller whose launch executes much other code (the training-mode
// forward) is faster with the compact form, the others with the unrolled one.
template <bool NORMALISE>
__device__ __forceinline__ float feature_map_row_any(unsigned char* tile, int r, int phi, bool compact = false) {
  if (phi == RATTN_PHI_SOFTMAX) {
    if (!compact) return feature_map_row_inplace<NORMALISE>(tile, r);
    if (NORMALISE) {
      feature_map_row_inplace_lr(tile, r);
      return 1.f;
    }
    return feature_map_row_unnorm_inplace(tile, r);
  }
  if (phi == RATTN_PHI_RELU) {
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
      uint4* p = reinterpret_cast<uint4*>(tile + swz(r, c));
      *p = relu_bf16x8(*p);
    }
  }
  return 1.f;
}

// ------------------------------------------------------------------------ timeline
// For tuning (compiled in only with -DRATTN_TIMELINE): one CTA of the kernel in this file records (event id, clock) pairs
// per role.
#ifdef RATTN_TIMELINE
static __device__ unsigned long long g_timeline[4][2048];
static __device__ int g_timeline_n[4];
#define TL_DECL(on_expr) const bool tl_on = (on_expr); int tl_i = 0; (void)tl_on; (void)tl_i
#define TL(role, id) do { if (tl_on && tl_i < 1000) { unsigned long long c_; asm volatile("mov.u64 %0, %%clock64;" : "=l"(c_) :: "memory"); \
    g_timeline[role][2 * tl_i] = (unsigned long long)(id); g_timeline[role][2 * tl_i + 1] = c_; ++tl_i; g_timeline_n[role] = tl_i; } } while (0)
// the records so far, which are cleared; whether there were any
static bool read_timeline(unsigned long long* out, int* n) {
  const int none[4] = {0, 0, 0, 0};
  cudaMemcpyFromSymbol(out, g_timeline, sizeof(g_timeline));
  cudaMemcpyFromSymbol(n, g_timeline_n, sizeof(g_timeline_n));
  cudaMemcpyToSymbol(g_timeline_n, none, sizeof(none));
  return n[0] + n[1] + n[2] + n[3] > 0;
}
#else
#define TL_DECL(on_expr) do { } while (0)
#define TL(role, id) do { } while (0)
#endif

// ------------------------------------------------------------------------ work items
// Of persistent kernels: a CTA's next item comes from a device-wide counter, so that CTAs that start late
// (the SM was still running another kernel) or meet heavy items simply take fewer.  The loader warp draws it and
// publishes it in a small ring that the other roles read in order; a slot is rewritten once every reader has read it.
// A loader that gives up (a wait that ran out, here or in another role) notes how many items it has published.  The row
// threads, which meet at named barriers, leave on the end of that list and on nothing else (see mbar_wait), and so all at
// the same place.
constexpr int SCHED_SLOTS = 4;
struct SchedRing {
  uint64_t full[SCHED_SLOTS], free_[SCHED_SLOTS];
  int item[SCHED_SLOTS];
  int published, closed;   // items so far; items in all, once the loader has given up
};
__device__ __forceinline__ void sched_init(SchedRing* r, int readers) {
  r->published = 0;
  r->closed = INT_MAX;
  for (int i = 0; i < SCHED_SLOTS; ++i) {
    mbar_init(&r->full[i], 1);
    mbar_init(&r->free_[i], readers);
  }
}
// the loader warp's side: item n of this CTA is i (-1: there is none left)
__device__ __forceinline__ bool sched_publish(SchedRing* r, int n, int i, volatile int* abort) {
  const int slot = n % SCHED_SLOTS, use = n / SCHED_SLOTS;
  if (use >= 1) { if (!mbar_wait_warp(&r->free_[slot], (use - 1) & 1, abort)) return false; }
  if ((threadIdx.x & 31) == 0) {
    r->item[slot] = i;
    r->published = n + 1;
    mbar_arrive(&r->full[slot]);
  }
  __syncwarp();
  return true;
}
// ... the end of the list, by one thread of a loader that gives up
__device__ __forceinline__ void sched_close(SchedRing* r) { *(volatile int*)&r->closed = r->published; }
// ... drawn from the counter
__device__ __forceinline__ bool sched_draw(SchedRing* r, int* counter, int n_items, int n, volatile int* abort, int* out) {
  int i = 0;
  if ((threadIdx.x & 31) == 0) i = atomicAdd(counter, 1);
  i = __shfl_sync(0xffffffffu, i, 0);
  *out = i < n_items ? i : -1;
  return sched_publish(r, n, *out, abort);
}
// a reading thread's side
__device__ __forceinline__ bool sched_read(SchedRing* r, int n, volatile int* abort, int* out) {
  const int slot = n % SCHED_SLOTS, use = n / SCHED_SLOTS;
  if (!mbar_wait(&r->full[slot], use & 1, abort)) return false;
  *out = r->item[slot];
  mbar_arrive(&r->free_[slot]);
  return true;
}
// ... of the threads that share named barriers: item n, or -1 where the list has ended.  Whether item n has been published
// does not depend on when a thread asks.  (The loader's own waits are bounded; the limit here is four of them.)
__device__ __forceinline__ int sched_read_all(SchedRing* r, int n) {
  const int slot = n % SCHED_SLOTS, use = n / SCHED_SLOTS;
#pragma unroll 1
  for (int it = 0; !mbar_try_wait(&r->full[slot], use & 1); ++it)
    if (it == 4 * kWaitPolls || ((it & 63) == 63 && *(volatile int*)&r->closed <= n)) return -1;
  const int i = r->item[slot];
  mbar_arrive(&r->free_[slot]);
  return i;
}
// ... and a whole warp's (one of its lanes is counted)
__device__ __forceinline__ bool sched_read_warp(SchedRing* r, int n, volatile int* abort, int* out) {
  const int slot = n % SCHED_SLOTS, use = n / SCHED_SLOTS;
  if (!mbar_wait_warp(&r->full[slot], use & 1, abort)) return false;
  *out = r->item[slot];
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(&r->free_[slot]);
  return true;
}

// Bounded wait (whole warp) until a progress word of another kernel reaches `need`; the TMA loads
// that follow are ordered behind the acquiring read.
__device__ __forceinline__ bool wait_published(const int* word, int need, volatile int* abort) {
#pragma unroll 1
  for (int it = 0; it < (1 << 20); ++it) {
    if (ld_acquire_gpu(word) >= need) {
      fence_proxy_async_all();
      return true;
    }
    if ((it & 15) == 15 && *abort) return false;
    __nanosleep(200);
  }
  *abort = 1;
  return false;
}

// ------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) return (EncodeTiledFn) nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// [n_mats, rows, 128] bf16, box = 64 columns x 128 rows x 1, 128-byte swizzle, zero fill.
inline bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t n_mats, uint32_t box_rows = 128) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {128, rows, n_mats};
  const cuuint64_t strides[2] = {128 * 2, rows * 128 * 2};
  const cuuint32_t box[3] = {64, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// A caller's tensor with T rows per head, H heads, B batch entries: [B, H, T, 128] (layout 0) or
// [B, T, H, 128] (layout 1), bf16; box = 64 columns x box_rows rows of one head.
inline bool make_user_map(UMap* u, const void* base, uint64_t T, uint64_t H, uint64_t B, int layout,
                          uint32_t box_rows = 128) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  u->H = (int)H;
  const cuuint64_t dims[4] = {128, T, H, B};
  const cuuint64_t row = 128 * 2;
  const cuuint64_t strides[3] = {layout ? H * row : row, layout ? row : T * row, T * H * row};
  const cuuint32_t box[4] = {64, box_rows, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(&u->m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// The same tensor read as whole rows: box = 128 columns x box_rows rows of one head, no swizzle.
inline bool make_row_map(CUtensorMap* m, const void* base, uint64_t T, uint64_t H, uint64_t B, int layout,
                         uint32_t box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {128, T, H, B};
  const cuuint64_t row = 128 * 2;
  const cuuint64_t strides[3] = {layout ? H * row : row, layout ? row : T * row, T * H * row};
  const cuuint32_t box[4] = {128, box_rows, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// [n_mats, 128, 128] bf16 chunk states.  Modes without a linear branch keep none: the kernels
// then never use the map, which is encoded over one matrix of `any` (some valid bf16 buffer of
// at least 128 x 128 elements) so that it is well formed.
inline bool make_state_map(CUtensorMap* m, const void* states, const void* any, uint64_t n_mats, uint32_t box_rows = 128) {
  return states ? make_map(m, states, 128, n_mats, box_rows) : make_map(m, any, 128, 1, box_rows);
}

}  // namespace tc
}  // namespace rattn
