// Single-token decode step for bf16, d = 128, windows that are a multiple of 64 and groups of up
// to 8 query heads: the ring and the state stream through shared memory by TMA.
//
// The step reads the K ring, the V ring and the fp32 state of a K/V head once and writes the
// state back (Section 2.1: a cache of at most w+1 tokens; Eq. 4: the state), so it is bound by
// HBM traffic, or, for few sequences, by the latency of one CTA's share of it.  A (batch entry, K/V head) is therefore
// shared by a cluster of 1, 2, 4 or 8 CTAs: each takes a run of ring pieces and of state rows, forms the partial
// softmax sums and read-outs of them, and the cluster combines these through distributed shared memory.  Everything a
// CTA will read is requested up front as 16 KB pieces (64 ring slots, or up to 32 state rows) that pass through a
// ring of stages (eight, or as many as let two CTAs share an SM), refilled by whichever warp reads a stage last, so the memory
// system always has the next pieces in flight, whatever the warps are doing.
//
// The ring is one pass over K and V pieces together: four warps take the even pieces and four the odd ones, 16 slots
// each, with an online softmax of their own (maximum, sum and output per warp), so no barrier falls between the first
// K piece and the last V piece; the warps' outputs meet once at the end.  The two groups of warps have half of the
// stages each, and nothing of the other's passes through them: a stage's barrier tells only whether the last or the
// last but one of its uses has landed, so everyone who waits on it must have waited for all uses before.  Both products are warp-level mma with the
// group's query heads as rows (q K^T, then P V; the pieces arrive 128-byte swizzled, so the fragment loads are
// conflict-free): with at most 8 rows they are far too small for tcgen05's 64-row minimum.  The weights stay in
// registers, where the fragment of q K^T is the fragment P V wants; they enter as a bf16 pair, the leading part in rows
// 0-7 and the remainder in rows 8-15, so one product keeps 16 bits of them.  The state is read out and updated
// in fp32 on the CUDA cores.
#include "rattn_internal.h"
#include "tc_common.cuh"
#include "tc_ptx.cuh"

namespace rattn {
namespace {

using namespace ptx;

constexpr int DT_THREADS = 256;
constexpr int DT_WARPS = DT_THREADS / 32;
constexpr int DT_MAX_STAGES = 8;
constexpr int DT_PIECE = 16384;            // 64 ring slots x 128 bf16, or 32 state rows x 128 fp32
constexpr int D = 128;
constexpr int QB_STRIDE = D + 8;           // bf16 elements; 272 bytes: rows fall 16 bytes apart modulo 128

__device__ int g_decode_status;            // RATTN_ERR_TIMEOUT once a bounded wait has expired

struct DecodeTcArgs {
  const __nv_bfloat16* q; const __nv_bfloat16* k; const __nv_bfloat16* v;
  __nv_bfloat16* k_ring; __nv_bfloat16* v_ring; float* state; __nv_bfloat16* out;
  const float* gamma_swa; const float* gamma_rla;
  const int* pos_dev;
  int B, H_q, H_kv, w, pos, group, phi, cluster;
  int debug_wait;             // debug build only, 2: a wait of the last CTA of each cluster counts as run out
  float scale, eps;
};

struct DecodeTcMaps {
  CUtensorMap k, v;                        // [B*H_kv, w, 128] bf16, box 64 columns x 64 slots
};

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// phi over the 128 features by one warp (softmax, or one of the element-wise maps)
__device__ __forceinline__ void warp_feature_map(float* dst, const float* src, int lane, int phi) {
  float x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = src[lane + 32 * i];
  if (phi == RATTN_PHI_SOFTMAX) {
    const float m = warp_max(fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])));
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = __expf(x[i] - m);
      s += x[i];
    }
    const float inv = 1.f / warp_sum(s);
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] *= inv;
  } else if (phi == RATTN_PHI_RELU) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = fmaxf(x[i], 0.f);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) dst[lane + 32 * i] = x[i];
}

__device__ __forceinline__ void ldmatrix_x2(uint32_t addr, uint32_t (&r)[2]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// c[16 x 8] += a[16 x 16] b[16 x 8], bf16 in, fp32 accumulate
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
               "{%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A fragment register holds the values of slots s (low half) and s + 1 (high half): zero those
// at or beyond `live`.
__device__ __forceinline__ uint32_t keep_valid(uint32_t pair, int s, int live) {
  return pair & (s < live ? 0x0000ffffu : 0u) | pair & (s + 1 < live ? 0xffff0000u : 0u);
}

// Shared-memory plan (bytes, after the 1024-byte aligned stages).
struct Plan {
  int stages, q_b, zero, q_f, fq, vec, o_warp, o_swa, o_rla, w_stat, stat, bars, total;
};
__host__ __device__ inline Plan plan_with(int g, int stages) {
  Plan p;
  p.stages = stages;
  int off = stages * DT_PIECE;
  auto take = [&](int bytes) { const int at = off; off += (bytes + 15) & ~15; return at; };
  p.q_b = take(8 * QB_STRIDE * 2);         // bf16 [8][136]: the group's queries, rows >= g zero
  p.q_f = p.o_swa = take(g * D * 4);       // fp32 raw q; the ring's output once that has been used
  p.fq = take(g * D * 4);                  // phi(q)
  p.vec = take(5 * D * 4);                 // k_new, v_new, k_old, v_old, phi(k_old)
  p.o_warp = take(DT_WARPS * g * D * 4);   // per warp: un-normalised output over its slots
  // read-out of the state, per group of warps.  For 7 and 8 heads it takes the place of o_warp, behind a barrier of its
  // own: otherwise one CTA per SM is all that fits (148 heads of 8: 30.8 us a step against 22.0).
  p.o_rla = g > 6 ? p.o_warp : take(2 * g * D * 4);
  p.w_stat = take(2 * DT_WARPS * 8 * 4);   // per warp and head: maximum, sum
  p.stat = take(3 * 8 * 4);                // per head: this CTA's maximum and sum, logit of the incoming token
  p.bars = take(8 * DT_MAX_STAGES + 4 * DT_MAX_STAGES + 4 * DT_MAX_STAGES + 16);
  p.total = off + 1024;                    // room to align the stages
  return p;
}
constexpr int DT_SMEM = 227 * 1024, DT_SMEM_SHARED = (DT_SMEM - 2048) / 2;      // of a CTA alone on its SM; of each of two
// As many stages as let two CTAs share an SM, at least four.
inline int lean_stages(int g) { return plan_with(g, 6).total <= DT_SMEM_SHARED ? 6 : 4; }

// ---- cluster: barrier halves, and a read from another CTA's shared memory
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ float ld_cluster(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
// pieces of the ring that one CTA of a cluster of cs takes, of np
__host__ __device__ inline int pieces_per_rank(int np, int cs) { return (np + cs - 1) / cs; }

// G: query heads of a group, at most; NS: stages (known when compiled: a piece's stage and the phase of its barrier are
// divisions by it)
template <int G, int NS>
__global__ void __launch_bounds__(DT_THREADS, NS == DT_MAX_STAGES ? 1 : 2)
decode_tc_kernel(const __grid_constant__ DecodeTcArgs a, const __grid_constant__ DecodeTcMaps maps) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int g = a.group, w = a.w;
  const int CS = a.cluster, rank = CS > 1 ? (int)(blockIdx.x % CS) : 0;
  const Plan P = plan_with(g, NS);
  constexpr int NG = NS / 2;                                    // stages of each group of warps
  __nv_bfloat16* q_b = reinterpret_cast<__nv_bfloat16*>(sm + P.q_b);
  float* q_f = reinterpret_cast<float*>(sm + P.q_f);
  float* fq_s = reinterpret_cast<float*>(sm + P.fq);
  float* k_new = reinterpret_cast<float*>(sm + P.vec);
  float* v_new = k_new + D;
  float* k_old = v_new + D;
  float* v_old = k_old + D;
  float* fk_old = v_old + D;
  float* o_swa = reinterpret_cast<float*>(sm + P.o_swa);
  float* o_rla = reinterpret_cast<float*>(sm + P.o_rla);
  float* o_warp = reinterpret_cast<float*>(sm + P.o_warp);     // [8 warps][g][128]
  float* st_max = reinterpret_cast<float*>(sm + P.stat);       // [8] maximum over this CTA's logits
  float* st_sum = st_max + 8;                                  // [8] sum of its weights
  float* l_new = st_sum + 8;                                   // [8] scaled logit of the incoming token
  float* w_max = reinterpret_cast<float*>(sm + P.w_stat);      // [8 warps][8 heads]
  float* w_sum = w_max + DT_WARPS * 8;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + P.bars);
  int* readers = reinterpret_cast<int*>(full + DT_MAX_STAGES); // per stage: warps that have read its piece
  int* issued = readers + DT_MAX_STAGES;                       // per stage: pieces requested so far
  volatile int* abort = issued + DT_MAX_STAGES;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int z = blockIdx.x / CS, b = z / a.H_kv, hk = z % a.H_kv;
  // The next kernel on the stream may be set up; what this one reads may still be on its way from the one before.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) {
    prefetch_tensormap(&maps.k);
    prefetch_tensormap(&maps.v);
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], 1);
      readers[i] = issued[i] = 0;
    }
    *abort = 0;
    fence_mbar_init();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int pos = a.pos_dev ? a.pos_dev[b] : a.pos;
  const bool evict = pos - w >= 0;
  const int slot = pos % w;
  const int n_valid = pos < w ? pos : w;
  const int np_all = (n_valid + 63) >> 6;                      // K (and V) pieces that hold valid slots
  const int ppr = pieces_per_rank(np_all, CS), piece0 = min(rank * ppr, np_all);
  const int np = min(ppr, np_all - piece0);                    // ... this CTA's
  const int live_all = max(0, min(n_valid - 64 * piece0, 64 * np));   // its slots that hold a token
  const int st_rows = D / CS, st_piece = st_rows < 64 ? st_rows / 2 : 32, row0 = rank * st_rows;   // its state rows
  // this group's pieces: K and V of the ring pieces grp, grp + 2, ..., then the state pieces grp, grp + 2, ...
  const int grp = warp >> 2, n_kv = 2 * ((np - grp + 1) >> 1), n_pieces = n_kv + (st_rows / st_piece) / 2;

  const __nv_bfloat16* qg = a.q + ((size_t)b * a.H_q + (size_t)hk * g) * D;
  const __nv_bfloat16* kg = a.k + (size_t)z * D;
  const __nv_bfloat16* vg = a.v + (size_t)z * D;
  __nv_bfloat16* kr = a.k_ring + (size_t)z * w * D;
  __nv_bfloat16* vr = a.v_ring + (size_t)z * w * D;
  float* S = a.state + (size_t)z * D * D;
  __nv_bfloat16* og = a.out + ((size_t)b * a.H_q + (size_t)hk * g) * D;

  // The step's small operands are requested before any bulk traffic: behind 20 MB of ring pieces
  // they would wait microseconds.  They go to registers here and to shared memory once the pieces
  // have been asked for.
  uint4 q_reg = make_uint4(0u, 0u, 0u, 0u);                      // thread (row, 16-byte chunk) of the group's queries
  if (tid < g * 16) q_reg = reinterpret_cast<const uint4*>(qg)[tid];
  __nv_bfloat16 kn = __float2bfloat16_rn(0.f), vn = kn, ko = kn, vo_ = kn;
  if (tid < D) {
    kn = kg[tid];
    vn = vg[tid];
    if (evict) {
      ko = kr[(size_t)slot * D + tid];
      vo_ = vr[(size_t)slot * D + tid];
    }
  }
  __syncthreads();

  // piece p of the group's stream into its stage p % NG (one whole warp)
  auto stage_of = [&](int p) { return grp * NG + p % NG; };
  auto issue = [&](int p) {
    const int st = stage_of(p);
    unsigned char* dst = sm + st * DT_PIECE;
    uint64_t* bar = &full[st];
    if (lane == 0) ++issued[st];
    if (p < n_kv) {
      const CUtensorMap* m = (p & 1) ? &maps.v : &maps.k;
      const int row = (piece0 + grp + 2 * (p >> 1)) * 64;
      mbar_arrive_expect_tx(bar, DT_PIECE);
      tma_load_3d(dst, m, bar, 0, row, z);
      tma_load_3d(dst + DT_PIECE / 2, m, bar, 64, row, z);
    } else {
      const uint32_t bytes = (uint32_t)st_piece * D * 4;
      mbar_arrive_expect_tx(bar, bytes);
      bulk_load_1d(dst, S + (size_t)(row0 + (grp + 2 * (p - n_kv)) * st_piece) * D, bytes, bar);
    }
  };
  auto wait_piece = [&](int p) { return mbar_wait_warp(&full[stage_of(p)], (uint32_t)(p / NG) & 1u, abort); };
  // this warp has read piece p; the last of the group's four to do so requests the piece that takes its stage
  auto release = [&](int p) {
    __syncwarp();
    int last = 0;
    if (lane == 0) {
      last = atomicAdd(&readers[stage_of(p)], 1) == 3;
      if (last) readers[stage_of(p)] = 0;
    }
    if (__shfl_sync(0xffffffffu, last, 0) && p + NG < n_pieces) issue(p + NG);
  };
  if ((warp & 3) == 0)
    for (int p = 0; p < NG && p < n_pieces; ++p) issue(p);

  // queries: bf16 rows for the fragments (rows beyond the group zero), fp32 for phi and the new logit
  if (tid < 128) {
    const int r = tid >> 4, c = tid & 15;
    *reinterpret_cast<uint4*>(q_b + r * QB_STRIDE + c * 8) = q_reg;
    if (r < g) {
      const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&q_reg);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 x = __bfloat1622float2(h2[i]);
        q_f[r * D + c * 8 + 2 * i] = x.x;
        q_f[r * D + c * 8 + 2 * i + 1] = x.y;
      }
    }
  }
  if (tid < D) {
    k_new[tid] = __bfloat162float(kn);
    v_new[tid] = __bfloat162float(vn);
    k_old[tid] = __bfloat162float(ko);
    v_old[tid] = __bfloat162float(vo_);
  }
  __syncthreads();

  // query fragments: rows 0..7 from q_b (rows 8..15 of the 16-row product are zero)
  uint32_t qa[8][2];
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
    ldmatrix_x2(smem_u32(q_b + (lane & 7) * QB_STRIDE + (kk * 2 + ((lane >> 3) & 1)) * 8), qa[kk]);

  // phi(q), phi(k_old) and the incoming token's logit (Section 2.1), while the first pieces are on their way
  for (int r = warp; r <= g; r += DT_WARPS) {
    if (r < g) warp_feature_map(fq_s + r * D, q_f + r * D, lane, a.phi);
    else warp_feature_map(fk_old, k_old, lane, a.phi);
  }
  if (warp == DT_WARPS - 1) {
    for (int hh = 0; hh < g; ++hh) {
      float x = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) x += q_f[hh * D + lane + 32 * i] * k_new[lane + 32 * i];
      x = warp_sum(x);
      if (lane == 0) l_new[hh] = x * a.scale;
    }
  }

  // ---- one pass over the ring: this warp's pieces, 16 slots of each -----------------------------------
  bool ok = true;
  float m_run = -INFINITY, l_run = 0.f;                          // head lane / 4: maximum (quad-wide), sum (this thread's columns)
  float o[16][4];                                                // feature tile, fragment: rows 0-7 leading parts, 8-15 remainders
#pragma unroll
  for (int i = 0; i < 64; ++i) o[i >> 2][i & 3] = 0.f;
  const int slot0 = 16 * (warp & 3);                             // of the piece's 64
  for (int pk = 0; pk < n_kv; pk += 2) {
    const int pv = pk + 1, j = grp + pk;                         // ring piece j of this CTA's
    ok = wait_piece(pk);
    if (!ok) break;
    float c[2][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i >> 2][i & 3] = 0.f;
    {
      const uint32_t base = smem_u32(sm + stage_of(pk) * DT_PIECE);
      const int row = slot0 + (lane & 7) + ((lane >> 4) << 3);   // slots 0-7, 8-15 for the two column tiles
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const int chunk = kk * 2 + ((lane >> 3) & 1);
        uint32_t kb[4];
        ldmatrix_x4(base + (chunk >> 3) * (DT_PIECE / 2) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4), kb);
        const uint32_t qf[4] = {qa[kk][0], 0u, qa[kk][1], 0u};
        mma_16816(c[0], qf, kb[0], kb[1]);
        mma_16816(c[1], qf, kb[2], kb[3]);
      }
    }
    release(pk);
    const int live = live_all - 64 * j - slot0;                  // of this warp's 16 slots, those below hold a token
    const int s0 = 2 * (lane & 3);
    float p[4];                                                  // slots s0, s0 + 1, s0 + 8, s0 + 9
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = s0 + (i & 1) + 8 * (i >> 1) < live ? c[i >> 1][i & 1] * a.scale : -INFINITY;
    float mx = fmaxf(fmaxf(p[0], p[1]), fmaxf(p[2], p[3]));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float m_new = fmaxf(m_run, mx), m_safe = m_new == -INFINITY ? 0.f : m_new;
    if (__any_sync(0xffffffffu, m_new > m_run)) {
      const float f = __expf(m_run - m_safe);
      l_run *= f;
#pragma unroll
      for (int i = 0; i < 64; ++i) o[i >> 2][i & 3] *= f;
      m_run = m_new;
    }
    uint32_t pa[4];
    {
      float lo[4];
      uint32_t hi[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        p[i] = __expf(p[i] - m_safe);
        l_run += p[i];
      }
      hi[0] = pack_bf16(p[0], p[1]);
      hi[1] = pack_bf16(p[2], p[3]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        lo[i] = p[i] - __uint_as_float((i & 1) ? hi[i >> 1] & 0xffff0000u : hi[i >> 1] << 16);
      pa[0] = hi[0]; pa[1] = pack_bf16(lo[0], lo[1]); pa[2] = hi[1]; pa[3] = pack_bf16(lo[2], lo[3]);
    }
    ok = wait_piece(pv);
    if (!ok) break;
    if (live > 0) {
      const uint32_t base = smem_u32(sm + stage_of(pv) * DT_PIECE);
      const int row = slot0 + (lane & 15);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int chunk = 2 * t + (lane >> 4);
        uint32_t vb[4];
        ldmatrix_x4_trans(base + (chunk >> 3) * (DT_PIECE / 2) + row * 128 + (((chunk & 7) ^ (row & 7)) << 4), vb);
        if (live < 16) {
          // a slot without a token may hold anything; its weight is zero, but 0 * NaN is not
          vb[0] = keep_valid(vb[0], s0, live);
          vb[2] = keep_valid(vb[2], s0, live);
          vb[1] = keep_valid(vb[1], s0 + 8, live);
          vb[3] = keep_valid(vb[3], s0 + 8, live);
        }
        mma_16816(o[2 * t], pa, vb[0], vb[1]);
        mma_16816(o[2 * t + 1], pa, vb[2], vb[3]);
      }
    }
    release(pv);
  }
  l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
  l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
  {
    const int hh = lane >> 2;
    if ((lane & 3) == 0) {
      w_max[warp * 8 + hh] = m_run;
      w_sum[warp * 8 + hh] = l_run;
    }
    if (hh < g) {
#pragma unroll
      for (int t = 0; t < 16; ++t)
        *reinterpret_cast<float2*>(o_warp + (warp * g + hh) * D + 8 * t + 2 * (lane & 3)) =
            make_float2(o[t][0] + o[t][2], o[t][1] + o[t][3]);
    }
  }
  ok = __syncthreads_and(ok) != 0;
  // the warps' shares meet; the incoming token is rank 0's
  for (int i = tid; i < g * D; i += DT_THREADS) {
    const int hh = i >> 7, c = i & (D - 1);
    float m = rank == 0 ? l_new[hh] : -INFINITY;
#pragma unroll
    for (int wv = 0; wv < DT_WARPS; ++wv) m = fmaxf(m, w_max[wv * 8 + hh]);
    const float ms = m == -INFINITY ? 0.f : m, en = rank == 0 ? __expf(l_new[hh] - ms) : 0.f;
    float x = en * v_new[c], l = en;
#pragma unroll
    for (int wv = 0; wv < DT_WARPS; ++wv) {
      const float f = __expf(w_max[wv * 8 + hh] - ms);           // 0 for a warp without a valid slot
      x += f * o_warp[(wv * g + hh) * D + c];
      l += f * w_sum[wv * 8 + hh];
    }
    o_swa[i] = x;
    if (c == 0) {
      st_max[hh] = m;
      st_sum[hh] = l;
    }
  }

  // ---- the state: read-out phi(q) S and the update S += phi(k_old)^T v_old (Eq. 4), fp32 -----------
  // thread = two float4 column groups (c4, c4 + 16) and one of 8 row lanes (rl) that sit in the same warp; a piece
  // belongs to one group of four warps
  {
    const int rl = (lane >> 2) & 7, c4 = (lane & 3) | ((warp & 3) << 2);
    float4 ar[G][2], vo[2];
#pragma unroll
    for (int hh = 0; hh < G; ++hh) ar[hh][0] = ar[hh][1] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 2; ++u) vo[u] = *reinterpret_cast<const float4*>(v_old + (c4 + 16 * u) * 4);
    for (int p = n_kv; p < n_pieces && ok; ++p) {
      ok = wait_piece(p);
#ifdef RATTN_DEBUG_KNOBS
      if (a.debug_wait == 2 && rank == CS - 1 && warp == 0) {     // as if this wait had run out
        ok = false;
        *abort = 1;
      }
#endif
      if (!ok) break;
      const float* piece = reinterpret_cast<const float*>(sm + stage_of(p) * DT_PIECE);
      const int r0 = row0 + (grp + 2 * (p - n_kv)) * st_piece;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int rp = rl + 8 * m, r = r0 + rp;
        if (rp >= st_piece) break;
        const float fk = fk_old[r];
        float4 s4[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) s4[u] = *reinterpret_cast<const float4*>(piece + rp * D + (c4 + 16 * u) * 4);
#pragma unroll
        for (int hh = 0; hh < G; ++hh) {
          const float f = hh < g ? fq_s[hh * D + r] : 0.f;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            ar[hh][u].x += f * s4[u].x; ar[hh][u].y += f * s4[u].y; ar[hh][u].z += f * s4[u].z; ar[hh][u].w += f * s4[u].w;
          }
        }
        if (evict) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            s4[u].x += fk * vo[u].x; s4[u].y += fk * vo[u].y; s4[u].z += fk * vo[u].z; s4[u].w += fk * vo[u].w;
            *reinterpret_cast<float4*>(S + (size_t)r * D + (c4 + 16 * u) * 4) = s4[u];
          }
        }
      }
      release(p);
    }
    if (P.o_rla == P.o_warp) __syncthreads();                    // everybody has read the warps' shares of the ring
#pragma unroll
    for (int hh = 0; hh < G; ++hh) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
          ar[hh][u].x += __shfl_xor_sync(0xffffffffu, ar[hh][u].x, off);
          ar[hh][u].y += __shfl_xor_sync(0xffffffffu, ar[hh][u].y, off);
          ar[hh][u].z += __shfl_xor_sync(0xffffffffu, ar[hh][u].z, off);
          ar[hh][u].w += __shfl_xor_sync(0xffffffffu, ar[hh][u].w, off);
        }
        if (rl == 0 && hh < g) *reinterpret_cast<float4*>(o_rla + (grp * g + hh) * D + (c4 + 16 * u) * 4) = ar[hh][u];
      }
    }
  }
  ok = __syncthreads_and(ok) != 0;
  if (CS > 1) {
    cluster_arrive();                                              // partial sums of every CTA are in place
    cluster_wait();
    // a wait that ran out in one of the CTAs ends the step for all of them
    ok = !__any_sync(0xffffffffu, lane < CS && __float_as_uint(ld_cluster(cluster_addr((const void*)abort, lane))) != 0u);
  }
  // The incoming token takes the evicted token's slot: every CTA has read the evicted token, and the one whose piece that
  // is has consumed it (a slot beyond the valid pieces is read by nobody).
  if (ok && tid < D && rank == min((slot >> 6) / max(ppr, 1), CS - 1)) {
    kr[(size_t)slot * D + tid] = __float2bfloat16_rn(k_new[tid]);
    vr[(size_t)slot * D + tid] = __float2bfloat16_rn(v_new[tid]);
  }

  // ---- combine, Section 3.2: two RMS norms and the sum: one warp per head, heads spread over the cluster -----
  const int hh = CS > 1 ? rank + CS * warp : warp;
  if (ok && hh < g) {
    const int h = hk * g + hh, c0 = 4 * lane;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
    if (CS == 1) {
      const float inv = 1.f / st_sum[hh];
      const float4 p = *reinterpret_cast<const float4*>(o_swa + hh * D + c0);
      x = make_float4(p.x * inv, p.y * inv, p.z * inv, p.w * inv);
      const float4 ya = *reinterpret_cast<const float4*>(o_rla + hh * D + c0);
      const float4 yb = *reinterpret_cast<const float4*>(o_rla + (g + hh) * D + c0);
      y = make_float4(ya.x + yb.x, ya.y + yb.y, ya.z + yb.z, ya.w + yb.w);
    } else {
      // lane r has rank r's maximum and sum
      float m_r = -INFINITY, l_r = 0.f;
      if (lane < CS) {
        m_r = ld_cluster(cluster_addr(st_max + hh, lane));
        l_r = ld_cluster(cluster_addr(st_sum + hh, lane));
      }
      float4 p[8], r4[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if (r < CS) {
          p[r] = ld_cluster4(cluster_addr(o_swa + hh * D + c0, r));
          const float4 ya = ld_cluster4(cluster_addr(o_rla + hh * D + c0, r));
          const float4 yb = ld_cluster4(cluster_addr(o_rla + (g + hh) * D + c0, r));
          r4[r] = make_float4(ya.x + yb.x, ya.y + yb.y, ya.z + yb.z, ya.w + yb.w);
        }
      }
      const float m = warp_max(m_r), f = __expf(m_r - m);          // a CTA without a valid slot: exp(-inf) = 0
      const float inv = 1.f / warp_sum(f * l_r);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if (r < CS) {
          const float fr = __shfl_sync(0xffffffffu, f, r) * inv;
          x.x += fr * p[r].x; x.y += fr * p[r].y; x.z += fr * p[r].z; x.w += fr * p[r].w;
          y.x += r4[r].x; y.y += r4[r].y; y.z += r4[r].z; y.w += r4[r].w;
        }
      }
    }
    const float ss = warp_sum(x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w);
    const float sr = warp_sum(y.x * y.x + y.y * y.y + y.z * y.z + y.w * y.w);
    const float is = rsqrtf(ss / D + a.eps), ir = rsqrtf(sr / D + a.eps);
    const float4 one = make_float4(1.f, 1.f, 1.f, 1.f);
    const float4 gs = a.gamma_swa ? *reinterpret_cast<const float4*>(a.gamma_swa + (size_t)h * D + c0) : one;
    const float4 gr = a.gamma_rla ? *reinterpret_cast<const float4*>(a.gamma_rla + (size_t)h * D + c0) : one;
    *reinterpret_cast<uint2*>(og + (size_t)hh * D + c0) =
        make_uint2(pack_bf16(gs.x * x.x * is + gr.x * y.x * ir, gs.y * x.y * is + gr.y * y.y * ir),
                   pack_bf16(gs.z * x.z * is + gr.z * y.z * ir, gs.w * x.w * is + gr.w * y.w * ir));
  }
  if (!ok && tid == 0) {
    // a wait ran out: give what is still in flight a bounded time to land, report (neither output nor rings are written)
    for (int i = 0; i < NS; ++i)
      for (int it = 0; it < kWaitPolls && issued[i] > 0 && !mbar_try_wait(&full[i], (uint32_t)(issued[i] - 1) & 1u); ++it) {}
    g_decode_status = RATTN_ERR_TIMEOUT;
  }
  if (CS > 1) {                                                    // nobody leaves while its sums are being read
    __syncwarp();
    cluster_arrive();
    cluster_wait();
  }
}

struct Launch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  Launch(int n_heads, int cluster, int smem, cudaStream_t s) {
    cfg.gridDim = dim3((unsigned)(n_heads * cluster));
    cfg.blockDim = dim3(DT_THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    // the kernel waits for its predecessor itself (griddepcontrol.wait), after its set-up
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
  }
  Launch(const Launch&) = delete;
  Launch& operator=(const Launch&) = delete;
};

// Clusters of `cluster` CTAs that the current device runs at once, asked of the driver when a device meets another size of
// shared memory than before (0: it would not say).
template <int G, int NS>
int clusters_at_once(int cluster, int smem) {
  static std::atomic<uint64_t> known[kMaxDevices][4][4];             // smem << 32 | clusters
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  std::atomic<uint64_t>& k = known[dev][cluster == 1 ? 0 : cluster == 2 ? 1 : cluster == 4 ? 2 : 3][(smem >> 12) & 3];
  const uint64_t seen = k.load(std::memory_order_relaxed);
  if ((int)(seen >> 32) == smem) return (int)(seen & 0xffffffffu);
  int n = 0, n_sm = 0;
  cudaError_t e = allow_smem<decode_tc_kernel<G, NS>>(smem);
  if (e == cudaSuccess && cluster == 1) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, decode_tc_kernel<G, NS>, DT_THREADS, (size_t)smem);
    if (e == cudaSuccess) e = sm_count(&n_sm);
    n *= n_sm;
  } else if (e == cudaSuccess) {
    Launch l(1, cluster, smem, nullptr);
    e = cudaOccupancyMaxActiveClusters(&n, decode_tc_kernel<G, NS>, &l.cfg);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  k.store((uint64_t)smem << 32 | (uint32_t)n, std::memory_order_relaxed);
  return n;
}

// CTAs per (batch entry, K/V head), for a ring of `pieces` pieces: as many as still find room on the GPU at once -- a second
// wave costs more than the shorter shares save, and room for the CTAs is not yet room for their clusters, which do not span
// GPCs (4 heads a group, w = 512: 64 heads by 4 take 11.1 us a step, 72 heads by 4 20.5 and by 2 13.4) -- and no more than
// there are pieces to share out: a share of the state alone costs as much as it saves (w = 128, 64 heads: 8.9 us undivided,
// 9.1 by 2).  0: not even one CTA each finds room.
template <int G, int NS>
int cluster_size(int n_heads, int pieces, int g) {
  const int smem = plan_with(g, NS).total;
  if (clusters_at_once<G, NS>(1, smem) < n_heads) return 0;
  int cs = 1;
  while (cs < 8 && pieces > 2 && 2 * cs <= pieces && clusters_at_once<G, NS>(2 * cs, smem) >= n_heads) cs *= 2;
  return cs;
}

template <int G, int NS>
cudaError_t launch_with(DecodeTcArgs a, const DecodeTcMaps& m, int cluster, cudaStream_t s) {
  const int smem = plan_with(a.group, NS).total;
  cudaError_t e = allow_smem<decode_tc_kernel<G, NS>>(smem);
  if (e != cudaSuccess) return e;
  a.cluster = cluster > 0 ? cluster : 1;
  {
    KernelTimer kt("decode_step", s);
    const Launch l(a.B * a.H_kv, a.cluster, smem, s);
    e = cudaLaunchKernelEx(&l.cfg, decode_tc_kernel<G, NS>, a, m);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  return cudaGetLastError();
}

template <int G>
cudaError_t launch_g(const DecodeTcArgs& a, const DecodeTcMaps& m, int pieces, cudaStream_t s) {
  const int n_heads = a.B * a.H_kv, knob = tuning(RATTN_TUNE_DECODE_STAGES) & ~1;
  const int stages = knob >= 4 ? knob : lean_stages(a.group);
  const int shared = stages == 4 ? cluster_size<G, 4>(n_heads, pieces, a.group)
                   : stages == 6 ? cluster_size<G, 6>(n_heads, pieces, a.group) : 0;
  // Where the CTAs find room one to an SM, each takes eight stages: nearly everything it reads is then under way from the
  // start, and the scheduler cannot put two of them on one SM while others idle (16 sequences of 32/8 heads, w = 64: 11.1 ->
  // 9.0 us; 8 of w = 256 10.4 -> 9.3; 9 of w = 512 13.4 -> 11.2).  Not where that halves the cluster and leaves eight
  // pieces or more to a CTA (12 sequences of w = 1024: 22.3 us, shared by two 19.6).
  const int alone = knob == 8 || knob < 4 ? cluster_size<G, 8>(n_heads, pieces, a.group) : 0;
  if (knob == 8 || (alone > 0 && (alone >= shared || pieces < 8 * alone))) return launch_with<G, 8>(a, m, alone, s);
  return stages == 4 ? launch_with<G, 4>(a, m, shared, s) : launch_with<G, 6>(a, m, shared, s);
}

}  // namespace

bool decode_tc_applies(const Args& p, int w) {
  return p.dtype == RATTN_BF16 && p.d == 128 && w % 64 == 0 && p.group <= 8;
}

cudaError_t launch_decode_tc(const Args& p, void* k_ring, void* v_ring, float* state, int pos, const int* pos_dev,
                             cudaStream_t s) {
  DecodeTcArgs a;
  a.q = static_cast<const __nv_bfloat16*>(p.q);
  a.k = static_cast<const __nv_bfloat16*>(p.k);
  a.v = static_cast<const __nv_bfloat16*>(p.v);
  a.k_ring = static_cast<__nv_bfloat16*>(k_ring);
  a.v_ring = static_cast<__nv_bfloat16*>(v_ring);
  a.state = state;
  a.out = static_cast<__nv_bfloat16*>(p.out);
  a.gamma_swa = p.gamma_swa; a.gamma_rla = p.gamma_rla;
  a.pos_dev = pos_dev;
  a.B = p.B; a.H_q = p.H_q; a.H_kv = p.H_kv; a.w = p.w; a.pos = pos; a.group = p.group; a.phi = p.phi;
  a.scale = p.scale; a.eps = p.eps;
  DecodeTcMaps m;
  if (!tc::make_map(&m.k, k_ring, (uint64_t)p.w, (uint64_t)p.B * p.H_kv, 64) ||
      !tc::make_map(&m.v, v_ring, (uint64_t)p.w, (uint64_t)p.B * p.H_kv, 64))
    return cudaErrorInvalidValue;
  a.debug_wait = debug_wait();
  a.cluster = 0;                            // launch_g
  const int pieces = ((pos_dev || pos >= p.w ? p.w : pos) + 63) / 64;
  if (p.group == 1) return launch_g<1>(a, m, pieces, s);
  if (p.group == 2) return launch_g<2>(a, m, pieces, s);
  if (p.group <= 4) return launch_g<4>(a, m, pieces, s);
  return launch_g<8>(a, m, pieces, s);
}

int decode_tc_status(cudaStream_t s, cudaError_t* err) {
  int word = 0;
  cudaError_t e = cudaMemcpyFromSymbolAsync(&word, g_decode_status, sizeof(int), 0, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && word != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbolAsync(g_decode_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  *err = e;
  return word;
}

}  // namespace rattn
