// Tensor-core backward for bf16, d = 128, window a multiple of 128 (sm_100a: TMA + tcgen05 + TMEM).
//
// The paper prints no backward formulas; these follow from its definitions by the chain rule
// (Section 2.1 for the window branch, Eq. 4 in the chunkwise form of Eq. 2-3 for the residual
// branch, Section 3.1 for the feature map, Section 3.2 for the two norms).  With 128-token
// tiles, chunk c = key tile c, lag wt = w / 128, and for query tile i the "boundary" chunk
// cb = i - wt (the chunk the residual branch reads in intra form, masked to j < t - w):
//
//   prep      per row: gradients g_s, g_r of the two un-normalised branch outputs (through the
//             RMS norms and gains), D_t = g_s . o_swa, all from the forward's residuals.
//   window    P = exp(scale q.k - lse),  dP = g_s V^T,  dS = P * (dP - D) * scale,
//             dQ += dS K,   dK += dS^T Q,   dV += P^T g_s.
//   residual  forward states S_c = sum_{c' < c} phi(K_c')^T V_c' (saved by the forward) and
//             reverse states R_c = sum_{i > c + wt} phi(Q_i)^T g_r,i (summed over the query
//             heads of the group; computed here by an outer-product kernel and a suffix scan):
//               dphi_q = g_r S_cb^T + ((g_r V_cb^T) masked) phi(K_cb)
//               dphi_k = V_c R_c^T  + ((V_c g_r^T) masked) phi(Q_{c+wt})
//               dV    += phi(K_c) R_c + ((phi(K_c) phi(Q_{c+wt})^T) masked) g_r
//   feature   dq += phi(q) * (dphi_q - <dphi_q, phi(q)>), the same for k.
//
// Two main kernels, so that every output tile has one owner and nothing is accumulated with
// atomics (results are deterministic):
//   tc_bwd_dq_kernel   a (query head, query tile) item loops over the key tiles of its band;
//   tc_bwd_dkv_kernel  a (K/V head, key tile) item loops over the group's query heads and, for
//                      each, over the query half tiles whose band contains the key tile.
// Both are persistent (one CTA per SM walks its items, the next item's loads in flight while
// the current one's epilogue drains) and warp-specialised: row threads share the accumulator
// rows (row = TMEM lane), a loader warp issues the TMA copies, MMA warps the tcgen05 products; all accumulation is fp32 in TMEM, and the weight matrices of each tile
// pair (P, dS) are rounded to bf16 and handed to the tensor core through TMEM.
#include "tc_common.cuh"

namespace rattn {
namespace {

using namespace ptx;
using namespace tc;

constexpr float LOG2E = 1.4426950408889634f;

struct BwdArgs {
  __nv_bfloat16* dq;
  __nv_bfloat16* dk;
  __nv_bfloat16* dv;
  const float* lse;     // [B,H_q,T]  natural-log log-sum-exp of the window logits
  const float* delta;   // [B,H_q,T]  D_t
  const float* lse2p;   // [B*H_q, t_pad]  lse * log2(e), +inf beyond T   (t_pad = T rounded up to 128)
  const float* dscp;    // [B*H_q, t_pad]  D_t * scale, 0 beyond T
  int t_pad;
  int* status;
  int* counter;         // next item of the launch (device memory, zero at launch)
  int wait_first;       // 1: wait for the kernel ahead right after the set-up
  int wait_before;      // 1: the kernel ahead (the reverse states' chain) may still be running; not to end before it
  int T, w, H_q, group, mode, n_chunks, n_bh;   // n_bh: query heads (dq), K/V heads times parts (dk/dv) over the batch
  int split;            // dk/dv: parts that the group's heads are split into
  float4* part;         // ... and where their dK, dV go in fp32 (null: one part, straight to the outputs)
  int phi;              // rattn_feature_map
  float scale, scale_log2;
  int debug_wait;       // debug build only, 2: the first wait of some of the row threads counts as run out
};

#define WAIT_OR_RETURN(bar, parity) \
  do { if (!mbar_wait(&(bar), (parity), &bars->abort)) return false; } while (0)
// for roles run by a whole converged warp
#define WAIT_OR_RETURN_W(bar, parity) \
  do { if (!mbar_wait_warp(&(bar), (parity), &bars->abort)) return false; } while (0)

// of threads that share named barriers: see mbar_wait
#define WAIT_ON(bar, parity) mbar_wait(&(bar), (parity), &bars->abort)

// ------------------------------------------------------------------------------ prep
// A pure stream: dO and the two un-normalised branch outputs in, g_s and g_r out (bf16), plus the
// per-row statistics; bound by HBM.  The unit is a chunk of 32 rows of one head (8 KB per tensor,
// contiguous), which travels global -> shared -> global as bulk asynchronous copies through a ring
// of stages, so the bytes in flight do not depend on where the warps are; the rows are transformed
// in place in shared memory (g_s over o_swa, g_r over o_rla).  The warps meet only at the ring's barriers and take
// turns with the copies: chunk n is stored, and its stage refilled, by warp n mod 8 (with all of that on one warp
// behind a __syncthreads per chunk, that warp's path, 5500 cycles a chunk, was everybody's).  GAINS: without gains
// neither they nor the sums of their gradients take registers.  Eight neighbouring lanes hold a row:
// lane l has features [8l, 8l+8) and [64+8l, 64+8l+8).  Every CTA takes an equal contiguous share of
// the chunks (head-major), so it meets few heads and keeps its gain-gradient sums in registers.
// With n = o / r (r the rms incl. eps), gh = dy * gain, A = gh . o:
//   g = (gh - n * (A / (128 r))) / r,   D = g . o = (A - A ss / (128 r^2)) / r,
// so each branch needs two row sums (ss = o . o and A).
constexpr int PREP_THREADS = 256;
constexpr int PREP_ROWS = 32;                       // rows of a chunk
constexpr int PREP_CHUNK = PREP_ROWS * 256;         // bytes of a chunk of one tensor
constexpr int PREP_STAGES = 4;
constexpr int PREP_SMEM = PREP_STAGES * 3 * PREP_CHUNK + 128;

struct PrepArgs {
  const __nv_bfloat16* o_s; const __nv_bfloat16* o_r;
  const float* gamma_s; const float* gamma_r;
  __nv_bfloat16* g_s; __nv_bfloat16* g_r;
  float* delta; float* dgamma_s; float* dgamma_r;
  const float* lse; float* lse2p; float* dscp;              // lse2p, dscp: -lse * log2(e) and -D * scale, padded
  int* status;
  int* counters;        // work counters of the two main kernels: cleared here
  int n_heads, T, t_pad, H_q, rla_on;
  float eps, scale;
};

__device__ __forceinline__ void unpack8(const unsigned char* p, float (&x)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(w[i] << 16);
    x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}

template <bool GAINS>
__global__ void __launch_bounds__(PREP_THREADS, 2)
tc_bwd_prep_kernel(const __grid_constant__ PrepArgs a, const __grid_constant__ CUtensorMap dy_map) {
  extern __shared__ __align__(128) unsigned char psm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(psm + PREP_STAGES * 3 * PREP_CHUNK);
  uint64_t* done = full + PREP_STAGES;                              // the chunk in the stage has been transformed
  volatile int* abort = reinterpret_cast<volatile int*>(done + PREP_STAGES);
  const int tid = threadIdx.x, l = tid & 7, row = tid >> 3;
  const int cph = a.t_pad / PREP_ROWS;                              // chunks per head
  const long long n_all = (long long)a.n_heads * cph;
  const int lo = (int)(n_all * blockIdx.x / gridDim.x), hi = (int)(n_all * (blockIdx.x + 1) / gridDim.x);
  const int n_in = a.rla_on ? 3 : 2;                                // tensors read per chunk

  if (tid == 0) {
    prefetch_tensormap(&dy_map);
    for (int i = 0; i < PREP_STAGES; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&done[i], PREP_THREADS / 32);
    }
    *abort = 0;
    fence_mbar_init();
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");        // the forward's residuals
  if (blockIdx.x == 0 && tid == 0) a.counters[0] = a.counters[1] = 0;
  __syncthreads();

  // chunk i: head i / cph, rows t0 .. t0 + 31 of it; rows at or beyond T are padding (nothing is copied)
  auto rows_of = [&](int i) { const int t0 = (i % cph) * PREP_ROWS; return a.T - t0 < 0 ? 0 : a.T - t0 < PREP_ROWS ? a.T - t0 : PREP_ROWS; };
  // `ahead` is the next chunk with data to ask for, the n_ahead-th of this CTA's; every thread follows it
  int ahead = lo, n_ahead = 0;
  auto skip_padding = [&] { while (ahead < hi && rows_of(ahead) == 0) ++ahead; };
  auto issue_ahead = [&]() {                                        // one thread
    const int rows = rows_of(ahead), slot = n_ahead % PREP_STAGES;
    const int bq = ahead / cph, t0 = (ahead - bq * cph) * PREP_ROWS, b = bq / a.H_q, h = bq - b * a.H_q;
    const size_t at = ((size_t)bq * a.T + t0) * 128;
    unsigned char* dst = psm + (size_t)slot * 3 * PREP_CHUNK;
    uint64_t* bar = &full[slot];
    const uint32_t bytes = (uint32_t)rows * 256;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 ::"r"(smem_u32(bar)), "r"((uint32_t)PREP_CHUNK + bytes * (n_in - 1)) : "memory");
    // dO is the caller's tensor (either head layout): a tiled copy of 32 whole rows, rows beyond T read as zero
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(smem_u32(dst)), "l"(&dy_map), "r"(smem_u32(bar)), "r"(0), "r"(t0), "r"(h), "r"(b)
                 : "memory");
    const __nv_bfloat16* src[3] = {nullptr, a.o_s, a.o_r};
    for (int k = 1; k < n_in; ++k)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(smem_u32(dst + k * PREP_CHUNK)), "l"(src[k] + at), "r"(bytes), "r"(smem_u32(bar)) : "memory");
  };
  for (int k = 0; k < PREP_STAGES; ++k) {
    skip_padding();
    if (ahead >= hi) break;
    if (tid == 0) issue_ahead();
    ++ahead;
    ++n_ahead;
  }

  float gs_lo[8], gs_hi[8], gr_lo[8], gr_hi[8], acc_s[16], acc_r[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) acc_s[e] = acc_r[e] = 0.f;
#pragma unroll
  for (int e = 0; e < 8; ++e) gs_lo[e] = gs_hi[e] = gr_lo[e] = gr_hi[e] = 1.f;
  int cur_h = -1;
  // This CTA's sums for head cur_h.  The four rows of a warp are added first and share the additions to memory: with every
  // row adding for itself these were 4.8 million at 40 heads, T = 8192 (145 -> 113 us with gains).
  auto flush = [&]() {
    if (cur_h < 0) return;
    const int part = (tid >> 3) & 3;                                // 0, 1: the window branch's halves, 2, 3: the other's
    float* dst = part < 2 ? a.dgamma_s : a.rla_on ? a.dgamma_r : nullptr;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float v[4] = {acc_s[e], acc_s[8 + e], acc_r[e], acc_r[8 + e]};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 8);
        v[k] += __shfl_xor_sync(0xffffffffu, v[k], 16);
      }
      if (dst) atomicAdd(dst + (size_t)cur_h * 128 + 64 * (part & 1) + 8 * l + e, part & 2 ? (part & 1 ? v[3] : v[2]) : (part & 1 ? v[1] : v[0]));
      acc_s[e] = acc_s[8 + e] = acc_r[e] = acc_r[8 + e] = 0.f;
    }
  };

  int i = lo, n_cons = 0;                                           // n_cons: chunks with data consumed so far
  bool ok = true;
  for (; i < hi; ++i) {
    const int bq = i / cph, t0 = (i % cph) * PREP_ROWS, rows = rows_of(i);
    const int t = t0 + row;
    const size_t prow = (size_t)bq * a.t_pad + t;
    if (rows == 0) {                                                // padding only: statistics that make every weight zero
      if (l == 0) { a.lse2p[prow] = -INFINITY; a.dscp[prow] = 0.f; }
      continue;
    }
    const int h = bq % a.H_q;
    if (GAINS && h != cur_h) {
      if (a.dgamma_s || a.dgamma_r) flush();
      cur_h = h;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        gs_lo[e] = a.gamma_s ? __ldg(a.gamma_s + (size_t)h * 128 + 8 * l + e) : 1.f;
        gs_hi[e] = a.gamma_s ? __ldg(a.gamma_s + (size_t)h * 128 + 64 + 8 * l + e) : 1.f;
        gr_lo[e] = a.gamma_r ? __ldg(a.gamma_r + (size_t)h * 128 + 8 * l + e) : 1.f;
        gr_hi[e] = a.gamma_r ? __ldg(a.gamma_r + (size_t)h * 128 + 64 + 8 * l + e) : 1.f;
      }
    }
    const int slot = n_cons % PREP_STAGES;
    unsigned char* buf = psm + (size_t)slot * 3 * PREP_CHUNK + row * 256 + 16 * l;
    const bool live = row < rows;
    // the row's log-sum-exp is asked for before the wait, so that its latency passes under it
    const float lse_row = (live && l == 0) ? __ldg(a.lse + (size_t)bq * a.T + t) : 0.f;
    const bool got = mbar_wait_warp(&full[slot], (uint32_t)(n_cons / PREP_STAGES) & 1u, abort);
    ok = got;
    if (!ok) break;
    {
      float g_lo[8], g_hi[8];
      if (live) {
        unpack8(buf, g_lo); unpack8(buf + 128, g_hi);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) g_lo[e] = g_hi[e] = 0.f;
      }
      // one branch after the other (both at once, with gains and sums, do not fit the registers); returns D = g . o
      auto branch = [&](unsigned char* p, const float (&ga_lo)[8], const float (&ga_hi)[8], float (&acc)[16], bool window) -> float {
        float o_lo[8], o_hi[8];
        if (live) {
          unpack8(p, o_lo); unpack8(p + 128, o_hi);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) o_lo[e] = o_hi[e] = 0.f;
        }
        float ss = 0.f, A = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          ss += o_lo[e] * o_lo[e] + o_hi[e] * o_hi[e];
          A += g_lo[e] * ga_lo[e] * o_lo[e] + g_hi[e] * ga_hi[e] * o_hi[e];
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
          ss += __shfl_xor_sync(0xffffffffu, ss, o);
          A += __shfl_xor_sync(0xffffffffu, A, o);
        }
        const float ir = rsqrtf(ss * (1.f / 128.f) + a.eps), c = A * ir * ir * (1.f / 128.f);   // c = mean(gh n) / r
        // gh - n A / (128 r): which of the two products is rounded on its own is said here and not left to the compiler, whose
        // choice, and with it the last bit of some g, changed with the code around
        auto diff = [&](float g, float ga, float o) {
          return GAINS && window ? fmaf(g, ga, -__fmul_rn(o, c)) : fmaf(-o, c, __fmul_rn(g, ga));
        };
        if (live) {
          uint32_t w_lo[4], w_hi[4];
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            w_lo[e >> 1] = pack_bf16(diff(g_lo[e], ga_lo[e], o_lo[e]) * ir, diff(g_lo[e + 1], ga_lo[e + 1], o_lo[e + 1]) * ir);
            w_hi[e >> 1] = pack_bf16(diff(g_hi[e], ga_hi[e], o_hi[e]) * ir, diff(g_hi[e + 1], ga_hi[e + 1], o_hi[e + 1]) * ir);
          }
          *reinterpret_cast<uint4*>(p) = make_uint4(w_lo[0], w_lo[1], w_lo[2], w_lo[3]);
          *reinterpret_cast<uint4*>(p + 128) = make_uint4(w_hi[0], w_hi[1], w_hi[2], w_hi[3]);
#pragma unroll
          for (int e = 0; GAINS && e < 8; ++e) {
            acc[e] += g_lo[e] * o_lo[e] * ir;
            acc[8 + e] += g_hi[e] * o_hi[e] * ir;
          }
        }
        return (A - c * ss) * ir;
      };
      const float dl = branch(buf + PREP_CHUNK, gs_lo, gs_hi, acc_s, true);            // D_t = g_s . o_swa
      if (a.rla_on) branch(buf + 2 * PREP_CHUNK, gr_lo, gr_hi, acc_r, false);
      if (l == 0) {
        if (live) {
          const size_t grow = (size_t)bq * a.T + t;
          a.delta[grow] = dl;
          a.lse2p[prow] = -lse_row * LOG2E;
          a.dscp[prow] = -dl * a.scale;
        } else {
          a.lse2p[prow] = -INFINITY;
          a.dscp[prow] = 0.f;
        }
      }
      fence_proxy_async_smem();
    }
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&done[slot]);
    skip_padding();
    if ((tid >> 5) == n_cons % (PREP_THREADS / 32)) {               // this warp's turn with the copies
      ok = mbar_wait_warp(&done[slot], (uint32_t)(n_cons / PREP_STAGES) & 1u, abort);
      if (!ok) break;
      if ((tid & 31) == 0) {
        const size_t at = ((size_t)bq * a.T + t0) * 128;
        unsigned char* src = psm + (size_t)slot * 3 * PREP_CHUNK;
        const uint32_t bytes = (uint32_t)rows * 256;
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(a.g_s + at), "r"(smem_u32(src + PREP_CHUNK)), "r"(bytes) : "memory");
        if (a.rla_on)
          asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(a.g_r + at), "r"(smem_u32(src + 2 * PREP_CHUNK)), "r"(bytes) : "memory");
        tma_store_commit();
        if (ahead < hi) {
          tma_store_wait_read();                                    // the stage has been read out
          issue_ahead();
        }
      }
      __syncwarp();
    }
    if (ahead < hi) { ++ahead; ++n_ahead; }
    ++n_cons;
  }
  if ((tid & 31) == 0) tma_store_wait();
  if (!ok) {
    // give the copies still in flight a bounded time to land before the CTA's memory goes away
    if (tid == 0) {
      for (int n = n_cons; n < n_cons + PREP_STAGES; ++n)
        for (int it = 0; it < (1 << 14) && !mbar_try_wait(&full[n % PREP_STAGES], (uint32_t)(n / PREP_STAGES) & 1u); ++it) {}
    }
    if ((tid & 31) == 0) atomicExch(a.status, RATTN_ERR_TIMEOUT);
  }
  if (GAINS && ok && (a.dgamma_s || a.dgamma_r)) flush();
}

// ================================================================================ dq
// Persistent: one CTA per SM walks a list of (query head, query tile) items, so that an item's
// first loads are in flight while the previous item's epilogue drains (at w = 512 the fixed
// cost per tile -- first TMA touch, output staging -- is larger than the band itself).
//   loader warp   Q, g_s, K tiles through a ring of three slots, V tiles through two; for the residual part g_r follows in
//                 g_s's buffer and the stored state in the K ring.  dQ leaves through the slot of the item's last K tile.
//   MMA warp      per key tile S = Q K^T, dP = g_s V^T; after the row threads have overwritten S
//                 with dS (bf16, in TMEM): dQ += dS K.  Then the residual part.
//   row threads   512: query row = TMEM lane, and a quarter of the 128 columns
// TMEM holds S twice (the second buffer is dphi_q's, which only the residual part needs), so that S of the next key tile
// is formed beside the row threads' work; dP of the next tile goes out the moment they are done, ahead of this tile's dQ.
// K is read by S in the step before its own and by dQ at the end of it, V by dP early in its step: three slots of K and two
// of V keep the loads (1750 cycles each) off the path; two of each, released together, put one into every step (4150 cycles
// a step), and so did a single V (3800).  Q is read to the end of the window loop, phi(q) being kept in registers.
// With one buffer, two threads per row and the epilogue on 128 of them, an item of 5 key tiles took 31k cycles.
// All barriers run on with phase counters that every role advances in the same way.
constexpr int DQ_NK = 3, DQ_NV = 2;
constexpr int DQ_OFF_Q = 0;
constexpr int DQ_OFF_G = 1 * TILE_BYTES;
constexpr int DQ_OFF_K = 2 * TILE_BYTES;   // DQ_NK slots
constexpr int DQ_OFF_V = 5 * TILE_BYTES;   // DQ_NV slots
constexpr int DQ_OFF_BAR = 7 * TILE_BYTES;
constexpr int DQ_OFF_EX = DQ_OFF_BAR + 384;   // one word per row thread
constexpr int DQ_ROW_WARPS = 16;
constexpr int DQ_SMEM = DQ_OFF_EX + 32 * DQ_ROW_WARPS * 4;
constexpr int DQ_THREADS = 32 * (DQ_ROW_WARPS + 4);   // row threads, MMA warp, loader warp (and two idle)

struct DqBars {
  uint64_t q_full, q_free, g_full, g_free, v_full[DQ_NV], v_free[DQ_NV], k_full[DQ_NK], k_free[DQ_NK], s_full, ds_full,
      phik_ready, o_done, acc_free, out_staged, drain;
  SchedRing sched;
  uint32_t tmem_base;
  int abort;
};

static_assert(sizeof(DqBars) <= DQ_OFF_EX - DQ_OFF_BAR, "barriers");

struct DqItem {
  int q0, bh_q, bh_kv, n_kt, st_index;
  bool has_boundary, has_rla, has_state;
};

__device__ __forceinline__ DqItem dq_item(const BwdArgs& a, int idx, int n_qt) {
  DqItem it;
  const int rank = idx / a.n_bh;                           // long bands first
  it.bh_q = idx - rank * a.n_bh;
  const int qt = n_qt - 1 - rank;
  it.q0 = qt * TILE;
  const int b = it.bh_q / a.H_q, h = it.bh_q % a.H_q;
  it.bh_kv = b * (a.H_q / a.group) + h / a.group;
  const int wt = a.w / TILE;
  it.has_boundary = (a.mode != RATTN_MODE_FULL_CAUSAL) && (qt - wt >= 0);
  it.n_kt = (it.has_boundary ? wt : qt) + 1;
  it.has_rla = it.has_boundary && (a.mode == RATTN_MODE_RATTN);
  const int cb = qt - wt;
  it.has_state = it.has_rla && cb > 0;
  it.st_index = it.bh_kv * a.n_chunks + (cb > 0 ? cb : 0);
  return it;
}

struct DqMaps {
  UMap q, k, v, dq;             // the caller's tensors (either head layout)
  CUtensorMap gs, gr, st;
};

__device__ bool dq_loader(const DqMaps& tm, const BwdArgs& a, unsigned char* smem, DqBars* bars, int n_items, int n_qt) {
  int kc = 0, vc = 0, gc = 0, n = 0;                       // uses of the K and V rings and of the g buffer; items so far
  // dQ of an item is staged in the slot of its last K tile, from where this warp stores it before it refills that slot
  int out_use = -1, out_row = 0, out_z = 0, out_n = 0;     // the K use and the item whose dQ is still to go
  auto store_out = [&]() -> bool {
    WAIT_OR_RETURN_W(bars->out_staged, out_n & 1);
    if ((threadIdx.x & 31) == 0) {
      store_tile(&tm.dq, smem + DQ_OFF_K + out_use % DQ_NK * TILE_BYTES, out_row, out_z);
      tma_store_commit();
      tma_store_wait_read();
    }
    __syncwarp();
    out_use = -1;
    return true;
  };
  for (;; ++n) {
    int idx;
    if (!sched_draw(&bars->sched, a.counter, n_items, n, &bars->abort, &idx)) return false;
    if (idx < 0) break;
    const DqItem it = dq_item(a, idx, n_qt);
    auto k_slot = [&](int& st) -> bool {                   // the next K slot, once its previous use is consumed
      st = kc % DQ_NK;
      const int use = kc / DQ_NK;
      if (use >= 1) WAIT_OR_RETURN_W(bars->k_free[st], (use - 1) & 1);
      if (out_use >= 0 && kc == out_use + DQ_NK && !store_out()) return false;
      ++kc;
      return true;
    };
    auto load_k = [&](int i) -> bool {
      int st;
      if (!k_slot(st)) return false;
      mbar_arrive_expect_tx(&bars->k_full[st], TILE_BYTES);
      load_tile(smem + DQ_OFF_K + st * TILE_BYTES, &tm.k, &bars->k_full[st], it.q0 - i * TILE, it.bh_kv);
      return true;
    };
    auto load_g = [&](const CUtensorMap* map) -> bool {
      if (gc >= 1) WAIT_OR_RETURN_W(bars->g_free, (gc - 1) & 1);
      mbar_arrive_expect_tx(&bars->g_full, TILE_BYTES);
      load_tile(smem + DQ_OFF_G, map, &bars->g_full, it.q0, it.bh_q);
      ++gc;
      return true;
    };
    if (n >= 1) WAIT_OR_RETURN_W(bars->q_free, (n - 1) & 1);
    mbar_arrive_expect_tx(&bars->q_full, TILE_BYTES);
    load_tile(smem + DQ_OFF_Q, &tm.q, &bars->q_full, it.q0, it.bh_q);
    if (!load_k(0) || !load_g(&tm.gs)) return false;
    int last_use = kc - 1;
    for (int i = 0; i < it.n_kt; ++i, ++vc) {
      const int st = vc % DQ_NV, use = vc / DQ_NV;
      if (use >= 1) WAIT_OR_RETURN_W(bars->v_free[st], (use - 1) & 1);
      mbar_arrive_expect_tx(&bars->v_full[st], TILE_BYTES);
      load_tile(smem + DQ_OFF_V + st * TILE_BYTES, &tm.v, &bars->v_full[st], it.q0 - i * TILE, it.bh_kv);
      if (i + 1 < it.n_kt) {
        if (!load_k(i + 1)) return false;
        last_use = kc - 1;
      }
    }
    if (it.has_rla) {
      if (it.has_state) {
        int st;
        if (!k_slot(st)) return false;
        mbar_arrive_expect_tx(&bars->k_full[st], TILE_BYTES);
        load_tile(smem + DQ_OFF_K + st * TILE_BYTES, &tm.st, &bars->k_full[st], 0, it.st_index);
      }
      if (!load_g(&tm.gr)) return false;
    }
    if (out_use >= 0 && !store_out()) return false;        // a short item has not come to that slot
    out_use = last_use;
    out_row = it.q0;
    out_z = it.bh_q;
    out_n = n;
  }
  if (out_use >= 0 && !store_out()) return false;
  if ((threadIdx.x & 31) == 0) tma_store_wait();           // the last store has completed
  return true;
}

__device__ bool dq_mma(const BwdArgs& a, unsigned char* smem, DqBars* bars, uint32_t tmem, int n_qt) {
  const uint32_t sQ = smem_u32(smem + DQ_OFF_Q), sG = smem_u32(smem + DQ_OFF_G);
  const uint32_t sK = smem_u32(smem + DQ_OFF_K), sV = smem_u32(smem + DQ_OFF_V);
  const uint32_t tS = tmem, tP = tmem + 128, tQ = tmem + 256, tF = tmem + 384;
  constexpr uint32_t idesc_ts = instr_desc(128, 128, 0, 1);
  int kc = 0, vc = 0, gc = 0, n = 0, cs = 0, cr = 0;       // K, V and g uses, items, score hand-overs, residual items
  for (;; ++n) {
    int idx;
    if (!sched_read_warp(&bars->sched, n, &bars->abort, &idx)) return false;
    if (idx < 0) break;
    const DqItem it = dq_item(a, idx, n_qt);
    auto k_landed = [&](int use) -> bool {
      WAIT_OR_RETURN_W(bars->k_full[use % DQ_NK], (use / DQ_NK) & 1);
      return true;
    };
    auto v_landed = [&]() -> bool {
      WAIT_OR_RETURN_W(bars->v_full[vc % DQ_NV], (vc / DQ_NV) & 1);
      return true;
    };
    // dP = g_s V^T of key tile i, with the releases behind it (the last tile's V is read once more by the residual part)
    auto dp_products = [&](int i) {
      mma_kk(tP, sG, sV + vc % DQ_NV * TILE_BYTES, false);
      mma_commit(&bars->s_full);
      if (!(it.has_rla && i + 1 == it.n_kt)) mma_commit(&bars->v_free[vc % DQ_NV]);
      if (i + 1 == it.n_kt) mma_commit(&bars->g_free);
      ++vc;
    };
    WAIT_OR_RETURN_W(bars->q_full, n & 1);
    if (!k_landed(kc)) return false;
    tc_fence_after();
    mma_kk(tS, sQ, sK + kc % DQ_NK * TILE_BYTES, false);   // S = Q K^T
    WAIT_OR_RETURN_W(bars->g_full, gc & 1);
    ++gc;
    if (!v_landed()) return false;
    tc_fence_after();
    dp_products(0);
    for (int i = 0; i < it.n_kt; ++i, ++kc, ++cs) {
      const int st = kc % DQ_NK;
      const uint32_t tSi = (i & 1) ? tF : tS, tSn = (i & 1) ? tS : tF;
      const bool more = i + 1 < it.n_kt;
      if (more && !k_landed(kc + 1)) return false;
      if (i == 0 && n >= 1) WAIT_OR_RETURN_W(bars->acc_free, (n - 1) & 1);   // the previous item's epilogue has read dQ and dphi_q
      if (more) {
        tc_fence_after();
        mma_kk(tSn, sQ, sK + (kc + 1) % DQ_NK * TILE_BYTES, false);   // the next tile's S, while the row threads work on this one's
        if (!v_landed()) return false;
      }
      WAIT_OR_RETURN_W(bars->ds_full, cs & 1);
      tc_fence_after();
      if (more) dp_products(i + 1);                        // ahead of dQ: the row threads wait for it
#pragma unroll
      for (int k = 0; k < 8; ++k)                          // dQ += dS K, dS read from TMEM
        mma_bf16_ts(tQ, tSi + 32 * (k >> 1) + 8 * (k & 1), mnmajor_desc(sK + st * TILE_BYTES, k), idesc_ts, (i > 0 || k > 0) ? 1u : 0u);
      // the last tile's K turns into phi(K) for the residual part: its slot is released there
      if (!(it.has_rla && !more)) mma_commit(&bars->k_free[st]);
      // the products that overwrite what these read follow them in the tensor pipe, which runs in issue order
    }
    if (it.has_rla) {
      const int last_st = (kc - 1) % DQ_NK, xs = kc % DQ_NK, vs = (vc - 1) % DQ_NV;   // K_cb; the stored state; V_cb
      mma_commit(&bars->o_done);                           // (interim) every window product done: K_cb may be rewritten
      WAIT_OR_RETURN_W(bars->g_full, gc & 1);              // g_r
      ++gc;
      tc_fence_after();
      mma_kk(tS, sG, sV + vs * TILE_BYTES, false);         // dA = g_r V_cb^T
      mma_commit(&bars->s_full);
      mma_commit(&bars->v_free[vs]);
      if (it.has_state) {
        if (!k_landed(kc)) return false;
        tc_fence_after();
        mma_kk(tF, sG, sK + xs * TILE_BYTES, false);       // g_r S_cb^T
        mma_commit(&bars->k_free[xs]);
        ++kc;
      }
      mma_commit(&bars->g_free);
      WAIT_OR_RETURN_W(bars->phik_ready, cr & 1);
      WAIT_OR_RETURN_W(bars->ds_full, cs & 1);
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < 8; ++k)                          // (dA masked) phi(K_cb)
        mma_bf16_ts(tF, tS + 32 * (k >> 1) + 8 * (k & 1), mnmajor_desc(sK + last_st * TILE_BYTES, k), idesc_ts, (it.has_state || k > 0) ? 1u : 0u);
      mma_commit(&bars->k_free[last_st]);
      ++cs; ++cr;
    }
    mma_commit(&bars->o_done);
  }
  return true;
}

// Row thread (r, part): query row r = TMEM lane, columns 32 part .. 32 part + 31.
__device__ bool dq_rows(const BwdArgs& a, unsigned char* smem, DqBars* bars, uint32_t tmem, int part, int r,
                        int n_qt) {
  const uint32_t lane_off = ((uint32_t)((r & ~31) << 16)) + 32 * part;
  const uint32_t tS = tmem + lane_off, tP = tmem + 128 + lane_off, tQ = tmem + 256 + lane_off,
                 tF = tmem + 384 + lane_off;
  int kc = 0, n = 0, cs = 0, co = 0;                       // ring uses, items, score hand-overs, o_done completions
  const unsigned char* sQ = smem + DQ_OFF_Q;
  const bool soft = (a.phi == RATTN_PHI_SOFTMAX);
  const float2 sl2 = make_float2(a.scale_log2, a.scale_log2), sc2 = make_float2(a.scale, a.scale);
  // one value per thread, shared by the four threads of a row (the four warps of the same 32 rows meet; sync again before
  // the words are used once more)
  float* ex = reinterpret_cast<float*>(smem + DQ_OFF_EX);
  auto row_sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(4 + (r >> 5)) : "memory"); };
  auto exchange = [&](float mine, float (&all)[4]) {
    ex[part * TILE + r] = mine;
    row_sync();
#pragma unroll
    for (int k = 0; k < 4; ++k) all[k] = ex[k * TILE + r];
  };
  for (;; ++n) {
    const int idx = sched_read_all(&bars->sched, n);
    if (idx < 0) break;
    const DqItem it = dq_item(a, idx, n_qt);
    const int n_kt = it.n_kt;
    const int t = it.q0 + r;
    const bool live = t < a.T;
    const size_t row = (size_t)it.bh_q * a.T + t;
    const float nl2 = live ? -a.lse[row] * LOG2E : -INFINITY;
    const float nD = live ? -a.delta[row] * a.scale : 0.f;

    for (int i = 0; i < n_kt; ++i, ++cs) {
      WAIT_ON(bars->s_full, cs & 1);
#ifdef RATTN_DEBUG_KNOBS
      if (a.debug_wait == 2 && part == 1 && n == 0 && i == 0) bars->abort = 1;
#endif
      tc_fence_after();
      const bool diag = (i == 0), bound = it.has_boundary && (i == n_kt - 1);
      const uint32_t tSi = (i & 1) ? tF : tS;
      float s[32], dp[32];
      tmem_ld32(tSi, s);
      tmem_ld32(tP, dp);
      tmem_wait_ld();
      if (diag || bound) mask32(s, keep_bits(r, part, diag, bound));   // the two edge tiles; exp2(-inf) = 0
      uint32_t pk[16];
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        const float2 y = __ffma2_rn(make_float2(s[e], s[e + 1]), sl2, make_float2(nl2, nl2));
        const float2 d = __fmul2_rn(make_float2(ex2(y.x), ex2(y.y)),
                                    __ffma2_rn(make_float2(dp[e], dp[e + 1]), sc2, make_float2(nD, nD)));
        pk[e >> 1] = pack_bf16(d.x, d.y);
      }
      tmem_st16(tSi, pk);                                    // dS (bf16, two per column) over this thread's own S columns
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&bars->ds_full);
    }
    const int last = (kc + n_kt - 1) % DQ_NK;                // the slot of K_cb
    kc += n_kt + (it.has_state ? 1 : 0);

    float ph[32];                                            // phi(q), this thread's columns
    if (it.has_rla) {
      // phi(q), while the last window products run (for the element-wise maps q itself)
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const uint4 u = *reinterpret_cast<const uint4*>(sQ + swz(r, 4 * part + cc));
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          ph[8 * cc + 2 * e] = __uint_as_float(w[e] << 16);
          ph[8 * cc + 2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
        }
      }
    }
    mbar_arrive(&bars->q_free);                              // every S has been formed
    if (it.has_rla) {
      if (soft) {
        float all[4];
        exchange(max32(ph), all);
        const float nml = -fmaxf(fmaxf(all[0], all[1]), fmaxf(all[2], all[3])) * LOG2E;
        float2 s0 = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const float2 y = __ffma2_rn(make_float2(ph[e], ph[e + 1]), make_float2(LOG2E, LOG2E), make_float2(nml, nml));
          ph[e] = ex2(y.x);
          ph[e + 1] = ex2(y.y);
          s0 = __fadd2_rn(s0, make_float2(ph[e], ph[e + 1]));
        }
        row_sync();
        exchange(s0.x + s0.y, all);
        const float inv = 1.f / ((all[0] + all[1]) + (all[2] + all[3]));
#pragma unroll
        for (int e = 0; e < 32; ++e) ph[e] *= inv;
        row_sync();
      }
      WAIT_ON(bars->o_done, co & 1);                    // every window product done: K_cb is no longer read raw
      ++co;
      {
        const int t4 = part * TILE + r, krow = t4 >> 2;        // four threads per key row
        unsigned char* kp = smem + DQ_OFF_K + last * TILE_BYTES + krow * 128;
        feature_map_quad(kp, kp, HALF_BYTES, krow, t4 & 3, a.phi);
      }
      fence_proxy_async_smem();
      mbar_arrive(&bars->phik_ready);
      WAIT_ON(bars->s_full, cs & 1);
      tc_fence_after();
      {
        float x[32];
        tmem_ld32(tS, x);
        tmem_wait_ld();
        const uint32_t keep = bits_lt(r - 32 * part);            // residual keys of row r in this chunk: j < r
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 32; e += 2)
          pk[e >> 1] = pack_bf16((keep >> e) & 1u ? x[e] : 0.f, (keep >> (e + 1)) & 1u ? x[e + 1] : 0.f);
        tmem_st16(tS, pk);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&bars->ds_full);
      ++cs;
    }

    // ---- dq = dQ + phi(q) * (dphi_q - <dphi_q, phi(q)>) -----------------------------------
    WAIT_ON(bars->o_done, co & 1);
    ++co;
    tc_fence_after();
    float dot = 0.f;
    if (it.has_rla && soft) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float df[16];
        tmem_ld16(tF + 16 * c, df);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) dot += ph[16 * c + e] * df[e];
      }
      float all[4];
      exchange(dot, all);
      dot = (all[0] + all[1]) + (all[2] + all[3]);
    }
    // every product has completed: the slot of the last K tile stages the output, which the loader warp stores
    unsigned char* sOut = smem + DQ_OFF_K + last * TILE_BYTES;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float x[16];
      tmem_ld16(tQ + 16 * c, x);
      if (it.has_rla) {
        float df[16];
        tmem_ld16(tF + 16 * c, df);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          // element-wise maps: ReLU passes the gradient where q > 0, the identity everywhere
          if (soft) x[e] += ph[16 * c + e] * (df[e] - dot);
          else x[e] += (a.phi == RATTN_PHI_RELU && !(ph[16 * c + e] > 0.f)) ? 0.f : df[e];
        }
      } else {
        tmem_wait_ld();
      }
#pragma unroll
      for (int e = 0; e < 2; ++e)
        *reinterpret_cast<uint4*>(sOut + swz(r, 4 * part + 2 * c + e)) =
            make_uint4(pack_bf16(x[8 * e + 0], x[8 * e + 1]), pack_bf16(x[8 * e + 2], x[8 * e + 3]),
                       pack_bf16(x[8 * e + 4], x[8 * e + 5]), pack_bf16(x[8 * e + 6], x[8 * e + 7]));
    }
    tc_fence_before();
    mbar_arrive(&bars->acc_free);          // the dQ / dphi_q columns have been read
    fence_proxy_async_smem();
    mbar_arrive(&bars->out_staged);
    if (it.has_rla && soft) row_sync();                      // the last exchanged value has been read
  }
  return *(volatile int*)&bars->abort == 0;
}

__global__ void __launch_bounds__(DQ_THREADS, 1)
tc_bwd_dq_kernel(const __grid_constant__ DqMaps tm, BwdArgs a, int n_items, int n_qt) {
  extern __shared__ __align__(1024) unsigned char smem[];
  DqBars* bars = reinterpret_cast<DqBars*>(smem + DQ_OFF_BAR);
  const int tid = threadIdx.x, warp = tid >> 5;
  if ((smem_u32(smem) & 1023u) != 0) {
    if (tid == 0 && a.status) atomicExch(a.status, 2);
    return;
  }
  if (tid == 0) {
    sched_init(&bars->sched, 32 * DQ_ROW_WARPS + 1);
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->q_free, 32 * DQ_ROW_WARPS);
    mbar_init(&bars->g_full, 1);
    mbar_init(&bars->g_free, 1);
    for (int i = 0; i < DQ_NV; ++i) {
      mbar_init(&bars->v_full[i], 1);
      mbar_init(&bars->v_free[i], 1);
    }
    for (int i = 0; i < DQ_NK; ++i) {
      mbar_init(&bars->k_full[i], 1);
      mbar_init(&bars->k_free[i], 1);
    }
    mbar_init(&bars->s_full, 1);
    mbar_init(&bars->ds_full, 32 * DQ_ROW_WARPS);
    mbar_init(&bars->phik_ready, 32 * DQ_ROW_WARPS);
    mbar_init(&bars->o_done, 1);
    mbar_init(&bars->acc_free, 32 * DQ_ROW_WARPS);
    mbar_init(&bars->out_staged, 32 * DQ_ROW_WARPS);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == DQ_ROW_WARPS) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  if (a.wait_first) asm volatile("griddepcontrol.wait;" ::: "memory");
  // A kernel that does not read dq may take the SMs that run out of items.  (Behind the wait: the terms of the reverse
  // states start on this signal alone, and what they read is complete only then.)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (warp == DQ_ROW_WARPS + 1 && (tid & 31) == 0) {
    prefetch_map(&tm.q);
    prefetch_map(&tm.k);
    prefetch_map(&tm.v);
    prefetch_tensormap(&tm.gs);
    prefetch_tensormap(&tm.gr);
    prefetch_tensormap(&tm.st);
    prefetch_map(&tm.dq);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  // registers follow the work: 512 x 104 + 128 x 64 = 640 x 96, the CTA's allocation
  bool ok = true;
  if (warp < DQ_ROW_WARPS) setmaxnreg_inc<104>();
  else setmaxnreg_dec<64>();
  if (warp < DQ_ROW_WARPS) {
    ok = dq_rows(a, smem, bars, tmem, warp >> 2, tid & 127, n_qt);
  } else if (warp == DQ_ROW_WARPS) {
    ok = dq_mma(a, smem, bars, tmem, n_qt);
    if (!ok) {
      mma_commit(&bars->drain);
      for (int it = 0; it < (1 << 16) && !mbar_try_wait(&bars->drain, 0); ++it) {}
    }
  } else if (warp == DQ_ROW_WARPS + 1) {
    ok = dq_loader(tm, a, smem, bars, n_items, n_qt);
    if (!ok && (tid & 31) == 0) sched_close(&bars->sched);
  }
  if (!ok && a.status) atomicExch(a.status, 1);
  if (a.wait_before) asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  if (warp == DQ_ROW_WARPS) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// =============================================================================== dkv
// One CTA per (key tile j, K/V head).  K_j, V_j (and phi(K_j)) stay in shared memory, the dV
// and dK accumulators in TMEM.  The work is a list of items, one per (query head of the
// group, query half tile of 64 rows): first the residual-branch items (query tile j + wt),
// then the window items (query tiles j .. j + wt).  Two row groups of 256 threads (two per key
// row = TMEM lane) take the items alternately, so that one group's exponentials overlap the
// other group's products.  One TMEM buffer holds the scores of an item: they are read into registers at once, and the
// next item's replace them; each group has columns of its own for its weights.  (With scores and weights in a slot per
// group, the scores of an item waited for the products of the one two before: 488 -> 476 us at 8 x 16/16 heads, T = 4096,
// w = 512.)
//   loader warp     TMA: K, V, [R_j], then per item Q_h, g_h and the query-side row statistics; stores dV, dK
//   score warp      per item: S^T = K Q_h^T and dP^T = V g_h^T (128 x 64 each)
//   accumulate warp from the row group's bf16 P^T and dS^T:
//                   dV += P^T g_h, dK += dS^T Q_h with the A operand read from TMEM
//   row group       P^T = exp2(S^T * scale_log2 - lse2[q]), dS^T = P^T (dP^T scale - D[q] scale)
// The residual items run first and leave dphi_k in the dK accumulator; the row groups then fold
// the feature-map Jacobian into it (dK := phi(k) (dphi_k - <dphi_k, phi(k)>)) and the window
// items accumulate on top.
constexpr int KV_NS = 4;                                   // item stages (the last two of a key tile stage its dV and dK)
constexpr int KV_OFF_K = 0;
constexpr int KV_OFF_V = 1 * TILE_BYTES;
constexpr int KV_OFF_KPHI = 2 * TILE_BYTES;                // phi(K_j)
constexpr int KV_OFF_STAGE = 3 * TILE_BYTES;               // KV_NS x [Q_h 16 KB | g_h 16 KB]
constexpr int KV_OFF_STAT = KV_OFF_STAGE + KV_NS * TILE_BYTES;   // KV_NS x (lse2[64], D*scale[64]) fp32
constexpr int KV_OFF_BAR = KV_OFF_STAT + KV_NS * 512;
constexpr int KV_SMEM = KV_OFF_BAR + 384;                  // 231,808 bytes of the 232,448 a CTA may have
constexpr int KV_ROW_WARPS = 16;
constexpr int KV_THREADS = 32 * (KV_ROW_WARPS + 4);        // 2 row groups; score, loader and accumulate warp (and one idle)

struct KvBars {
  uint64_t kv_full, kphi_ready, full[KV_NS], acc_done[KV_NS], s_full[2], s_read, p_ready[2], p_free[2], phiq_ready[2],
      r_acc_done, fold_done, all_done, acc_free, kv_free, out_staged, drain, drain2;
  SchedRing sched;
  uint32_t tmem_base;
  int abort;
};

static_assert(sizeof(KvBars) <= KV_SMEM - KV_OFF_BAR, "barriers");

struct KvMaps {
  UMap k, v, qh, dk, dv;        // the caller's tensors (either head layout)
  CUtensorMap rs, gsh, grh;
};

// One key tile (j, K/V head) of the persistent CTA's work list, and how its half-tile items
// are numbered.  Counters that run on across key tiles (ring slots, items, barrier
// phases) are kept by every role in the same way.
struct KvPlan {
  int j, bh_kv, head0, part_index, rs_index, n_qt, wt, group, n_R, n_s_tiles, N;
  bool windowed, has_inter;
  __device__ bool is_r(int n) const { return n < n_R; }
  __device__ int head(int n) const { return n < n_R ? (n >> 1) : (n - n_R) / (2 * n_s_tiles); }
  __device__ int qtile(int n) const { return n < n_R ? j + wt : j + (((n - n_R) % (2 * n_s_tiles)) >> 1); }
  __device__ int half(int n) const { return n < n_R ? (n & 1) : ((n - n_R) & 1); }
};

__device__ __forceinline__ KvPlan kv_plan(const BwdArgs& a, int idx) {
  KvPlan pl;
  pl.n_qt = (a.T + TILE - 1) / TILE;
  pl.j = idx / a.n_bh;                                     // most query tiles first
  const int rem = idx - pl.j * a.n_bh;
  pl.bh_kv = rem / a.split;
  const int part = rem - pl.bh_kv * a.split;
  pl.part_index = (pl.bh_kv * pl.n_qt + pl.j) * a.split + part;
  pl.rs_index = pl.bh_kv * a.n_chunks + pl.j;
  pl.wt = a.w / TILE;
  pl.group = a.group / a.split;
  pl.head0 = pl.bh_kv * a.group + part * pl.group;
  pl.windowed = (a.mode != RATTN_MODE_FULL_CAUSAL);
  const int i_hi = (pl.windowed && pl.j + pl.wt < pl.n_qt - 1) ? pl.j + pl.wt : pl.n_qt - 1;
  pl.n_s_tiles = i_hi - pl.j + 1;
  const bool r_tile = pl.windowed && (a.mode == RATTN_MODE_RATTN) && (pl.j + pl.wt <= pl.n_qt - 1);
  pl.n_R = r_tile ? 2 * pl.group : 0;
  pl.has_inter = part == 0 && r_tile && (pl.j + pl.wt + 1 <= pl.n_qt - 1);
  pl.N = pl.n_R + 2 * pl.group * pl.n_s_tiles;
  return pl;
}

// running counters shared by the three roles: key tiles done, ring slots used, half-tile items
// done, key tiles with residual items done
struct KvCount {
  int it, seq, gi, cr;
};

__device__ bool kv_loader(const KvMaps& tm, const BwdArgs& a, unsigned char* smem, KvBars* bars, int n_items) {
  KvCount c = {0, 0, 0, 0};
  // dV and dK of a key tile are staged in the ring slots of its last two items, which the next key tile uses third and
  // fourth.  This warp stores them, so that nobody else has to wait for the stores to have read the slots out: as soon as
  // they are staged and before the first of the slots is refilled.
  int out_row = 0, out_z = 0, out_seq = -1;                 // the key tile whose gradients are still to go
  auto store_out = [&]() -> bool {
    WAIT_OR_RETURN_W(bars->out_staged, (c.it - 1) & 1);
    if ((threadIdx.x & 31) == 0) {
      store_tile(&tm.dv, smem + KV_OFF_STAGE + out_seq % KV_NS * TILE_BYTES, out_row, out_z);
      tma_store_commit();
      store_tile(&tm.dk, smem + KV_OFF_STAGE + (out_seq + 1) % KV_NS * TILE_BYTES, out_row, out_z);
      tma_store_commit();
      asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // dV has left its slot; dK's is refilled next
    }
    __syncwarp();
    out_seq = -1;
    return true;
  };
  for (;; ++c.it) {
    int idx;
    if (!sched_draw(&bars->sched, a.counter, n_items, c.it, &bars->abort, &idx)) return false;
    if (idx < 0) break;
    const KvPlan pl = kv_plan(a, idx);
    const int j0 = pl.j * TILE;
    // K_j, V_j replace the previous key tile's once its last scores have been formed (the residual products that read V_j
    // come before those): they arrive while its last items and its epilogue are still under way
    if (c.it >= 1) WAIT_OR_RETURN_W(bars->kv_free, (c.it - 1) & 1);
    mbar_arrive_expect_tx(&bars->kv_full, 2 * TILE_BYTES);
    load_tile(smem + KV_OFF_K, &tm.k, &bars->kv_full, j0, pl.bh_kv);
    load_tile(smem + KV_OFF_V, &tm.v, &bars->kv_full, j0, pl.bh_kv);
    auto ring = [&](int& st) -> bool {                     // next ring slot, once its previous user is consumed
      st = c.seq % KV_NS;
      const int use = c.seq / KV_NS;
      if (use >= 1) WAIT_OR_RETURN_W(bars->acc_done[st], (use - 1) & 1);
      if (c.seq == out_seq + KV_NS && out_seq >= 0) {
        if (!store_out()) return false;
      } else {
        if ((threadIdx.x & 31) == 0) tma_store_wait_read();   // dK of the previous key tile has left its slot
        __syncwarp();
      }
      ++c.seq;
      return true;
    };
    if (pl.has_inter) {
      int st;
      if (!ring(st)) return false;
      mbar_arrive_expect_tx(&bars->full[st], TILE_BYTES);
      load_tile(smem + KV_OFF_STAGE + st * TILE_BYTES, &tm.rs, &bars->full[st], 0, pl.rs_index);
    }
    for (int n = 0; n < pl.N; ++n) {
      int st;
      if (!ring(st)) return false;
      unsigned char* dst = smem + KV_OFF_STAGE + st * TILE_BYTES;
      const int z = pl.head0 + pl.head(n);
      const int row = pl.qtile(n) * TILE + 64 * pl.half(n);
      if (pl.is_r(n)) {
        mbar_arrive_expect_tx(&bars->full[st], 2 * HT_BYTES);
        load_half_tile(dst, &tm.qh, &bars->full[st], row, z);
        load_half_tile(dst + HT_BYTES, &tm.grh, &bars->full[st], row, z);
      } else {
        mbar_arrive_expect_tx(&bars->full[st], 2 * HT_BYTES + 512);
        load_half_tile(dst, &tm.qh, &bars->full[st], row, z);
        load_half_tile(dst + HT_BYTES, &tm.gsh, &bars->full[st], row, z);
        float* stat = reinterpret_cast<float*>(smem + KV_OFF_STAT + st * 512);
        bulk_load_1d(stat, a.lse2p + (size_t)z * a.t_pad + row, 256, &bars->full[st]);
        bulk_load_1d(stat + 64, a.dscp + (size_t)z * a.t_pad + row, 256, &bars->full[st]);
      }
    }
    if (out_seq >= 0 && !store_out()) return false;        // a key tile of two ring uses has not come to those slots
    if (!a.part) {
      out_row = j0;
      out_z = pl.bh_kv;
      out_seq = c.seq - 2;
    }
  }
  if (out_seq >= 0 && !store_out()) return false;
  if ((threadIdx.x & 31) == 0) tma_store_wait();           // the last store has completed
  return true;
}

// The products are issued by two warps: the score warp issues S^T and dP^T of every item, the accumulate
// warp everything that writes the dV / dK accumulators, so that the waits of one (a wait that is already
// satisfied still costs an issuing warp some 300 cycles) pass under the products of the other.  A third
// issuer (S^T and dP^T apart) measured no faster.  Order between the two warps:
//   scores(n) -> row group -> p_ready -> accumulate(n)        (existing barriers)
//   scores(n - 1) in registers -> scores(n)                   (s_read)
//   accumulate(n - 2) complete -> the group's next weights     (p_free)
__device__ bool kv_mma_scores(const BwdArgs& a, unsigned char* smem, KvBars* bars, uint32_t tmem) {
  const uint32_t sK = smem_u32(smem + KV_OFF_K), sV = smem_u32(smem + KV_OFF_V), sKphi = smem_u32(smem + KV_OFF_KPHI);
  const uint32_t sStage = smem_u32(smem + KV_OFF_STAGE);
  const uint32_t tS = tmem + 256, tP = tmem + 320;
  KvCount c = {0, 0, 0, 0};
  int cq0 = 0, cq1 = 0;                                    // phi(Q_h) hand-overs per row group

  for (;; ++c.it) {
    int idx;
    if (!sched_read_warp(&bars->sched, c.it, &bars->abort, &idx)) return false;
    if (idx < 0) break;
    const KvPlan pl = kv_plan(a, idx);
    WAIT_OR_RETURN_W(bars->kv_full, c.it & 1);
    if (pl.n_R > 0) WAIT_OR_RETURN_W(bars->kphi_ready, c.cr & 1);
    if (pl.has_inter) ++c.seq;                             // the reverse state's ring slot (accumulate warp)
    const int seq0 = c.seq, gi0 = c.gi;
    for (int n = 0; n < pl.N; ++n) {
      const int st = (seq0 + n) % KV_NS, use = (seq0 + n) / KV_NS, slot = (gi0 + n) & 1;
      const uint32_t sQh = sStage + st * TILE_BYTES, sGh = sQh + HT_BYTES;
      // the reverse state's use of this slot is over (this warp has not followed it, and may not skip a phase)
      if (n == KV_NS - 1 && pl.has_inter) WAIT_OR_RETURN_W(bars->acc_done[st], (use - 1) & 1);
      WAIT_OR_RETURN_W(bars->full[st], use & 1);
      if (gi0 + n >= 1) WAIT_OR_RETURN_W(bars->s_read, (gi0 + n - 1) & 1);   // the item before is in registers
      if (pl.is_r(n)) {
        WAIT_OR_RETURN_W(bars->phiq_ready[slot], (slot ? cq1 : cq0) & 1);
        if (slot) ++cq1; else ++cq0;
      }
      tc_fence_after();
      mma_k_kh(tS, pl.is_r(n) ? sKphi : sK, sQh);          // S^T  = K Q_h^T   (phi(K) phi(Q_h)^T)
      mma_k_kh(tP, sV, sGh);                               // dP^T = V g_h^T
      mma_commit(&bars->s_full[slot]);
      if (n == pl.N - 1) mma_commit(&bars->kv_free);
    }
    c.seq += pl.N;
    c.gi += pl.N;
    if (pl.n_R > 0) ++c.cr;
  }
  return true;
}

__device__ bool kv_mma_accum(const BwdArgs& a, unsigned char* smem, KvBars* bars, uint32_t tmem) {
  const uint32_t sV = smem_u32(smem + KV_OFF_V), sKphi = smem_u32(smem + KV_OFF_KPHI);
  const uint32_t sStage = smem_u32(smem + KV_OFF_STAGE);
  const uint32_t tV = tmem, tK = tmem + 128;
  const uint32_t tW = tmem + 384;                          // the weights of row group g at columns 64 g: P^T, then dS^T
  KvCount c = {0, 0, 0, 0};

  for (;; ++c.it) {
    int idx;
    if (!sched_read_warp(&bars->sched, c.it, &bars->abort, &idx)) return false;
    if (idx < 0) break;
    const KvPlan pl = kv_plan(a, idx);
    bool accV = false, accK = false;
    // the previous key tile's epilogue has read the two accumulators
    bool acc_ok = (c.it == 0);
    if (pl.has_inter) {
      const int st = c.seq % KV_NS, use = c.seq / KV_NS;
      ++c.seq;
      WAIT_OR_RETURN_W(bars->kv_full, c.it & 1);
      WAIT_OR_RETURN_W(bars->kphi_ready, c.cr & 1);
      WAIT_OR_RETURN_W(bars->full[st], use & 1);
      if (!acc_ok) { WAIT_OR_RETURN_W(bars->acc_free, (c.it - 1) & 1); acc_ok = true; }
      tc_fence_after();
      mma_kk(tK, sV, sStage + st * TILE_BYTES, false);     // dphi_k = V_j R_j^T
      mma_kmn<1>(tV, sKphi, sStage + st * TILE_BYTES, false);   // dV     = phi(K_j) R_j
      mma_commit(&bars->acc_done[st]);
      accV = accK = true;
    }
    const int seq0 = c.seq, gi0 = c.gi;
    for (int m = 0; m < pl.N; ++m) {
      const int st = (seq0 + m) % KV_NS, slot = (gi0 + m) & 1;
      const uint32_t sQh = sStage + st * TILE_BYTES, sGh = sQh + HT_BYTES;
      WAIT_OR_RETURN_W(bars->p_ready[slot], ((gi0 + m) >> 1) & 1);
      if (m == pl.n_R && pl.n_R > 0) WAIT_OR_RETURN_W(bars->fold_done, c.cr & 1);
      if (!acc_ok) { WAIT_OR_RETURN_W(bars->acc_free, (c.it - 1) & 1); acc_ok = true; }
      tc_fence_after();
      mma_ts_h(tV, tW + 64 * slot, sGh, accV);             // dV += P^T g_h
      mma_ts_h(tK, tW + 64 * slot + 32, sQh, accK);        // dK += dS^T Q_h   (dphi_k += dA^T phi(Q_h))
      accV = accK = true;
      mma_commit(&bars->p_free[slot]);
      mma_commit(&bars->acc_done[st]);
      if (m == pl.n_R - 1) mma_commit(&bars->r_acc_done);
    }
    c.seq += pl.N;
    c.gi += pl.N;
    if (pl.n_R > 0) ++c.cr;
    mma_commit(&bars->all_done);
  }
  return true;
}

__device__ bool kv_rows(const BwdArgs& a, unsigned char* smem, KvBars* bars, uint32_t tmem, int g, int h, int r) {
  // Two groups of 256 threads.  A thread is key row r = TMEM lane and half h of its item's 64 query
  // columns: with all 64 on one thread a warp had a scheduler almost to itself and an item's arithmetic took 1530 cycles.
  const uint32_t lane_off = (uint32_t)((r & ~31) << 16);
  const uint32_t tV = tmem + lane_off, tK = tmem + 128 + lane_off;
  const uint32_t tS = tmem + 256 + 32 * h + lane_off, tP = tS + 64, tW = tmem + 384 + 64 * g + 16 * h + lane_off;
  const int gt = h * 128 + r;                                  // thread of the group
  KvCount cnt = {0, 0, 0, 0};

  for (;;) {
  const int idx = sched_read_all(&bars->sched, cnt.it);
  if (idx < 0) break;
  const KvPlan pl = kv_plan(a, idx);
  if (pl.n_R > 0) {
    // phi(K_j) into its own tile, four threads per row.  (Only here do these threads follow kv_full: without residual
    // items the next key tile's K and V may land before they look.)
    WAIT_ON(bars->kv_full, cnt.it & 1);
    const int row = (g * 256 + gt) >> 2;
    feature_map_quad(smem + KV_OFF_K + row * 128, smem + KV_OFF_KPHI + row * 128, HALF_BYTES, row, gt & 3, a.phi);
    fence_proxy_async_smem();
    mbar_arrive(&bars->kphi_ready);
  }
  const int seq0 = cnt.seq + (pl.has_inter ? 1 : 0), gi0 = cnt.gi;

  for (int n = 0; n < pl.N; ++n) {
    if (((gi0 + n) & 1) != g) continue;                       // the other group's item
    const int st = (seq0 + n) % KV_NS, use = (seq0 + n) / KV_NS;
    const bool is_r = pl.is_r(n);
    const int i = pl.qtile(n), hf = pl.half(n);
    unsigned char* sQh = smem + KV_OFF_STAGE + st * TILE_BYTES;
    // A group sees every second item, so it follows a slot's uses with gaps, and a wait by parity cannot skip a phase:
    // the previous use of the slot must be known to be over.
    if (use >= 1) WAIT_ON(bars->acc_done[st], (use - 1) & 1);
    WAIT_ON(bars->full[st], use & 1);
    if (is_r) {
      // phi(Q_h) in place: 64 rows, four threads per row
      const int row = gt >> 2;
      feature_map_quad(sQh + row * 128, sQh + row * 128, HT_HALF, row, gt & 3, a.phi);
      fence_proxy_async_smem();
      mbar_arrive(&bars->phiq_ready[g]);
    }
    WAIT_ON(bars->s_full[g], ((gi0 + n) >> 1) & 1);
#ifdef RATTN_DEBUG_KNOBS
    if (a.debug_wait == 2 && g == 1 && h == 1 && cnt.it == 0 && n < 2) bars->abort = 1;
#endif
    tc_fence_after();
    const bool diag = !is_r && (i == pl.j), bound = !is_r && pl.windowed && (i == pl.j + pl.wt);
    float s[32], dp[32];
    tmem_ld32(tS, s);
    tmem_ld32(tP, dp);
    tmem_wait_ld();
    tc_fence_before();
    mbar_arrive(&bars->s_read);                                // the next item's scores may come
    const int rd = r - (64 * hf + 32 * h);                     // key row relative to this thread's first query
    uint32_t pk1[16], pk2[16];
    if (is_r) {
      const uint32_t keep = bits_gt(rd);                       // keep key r < query q
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        const bool k0 = (keep >> e) & 1u, k1 = (keep >> (e + 1)) & 1u;
        pk1[e >> 1] = pack_bf16(k0 ? s[e] : 0.f, k1 ? s[e + 1] : 0.f);
        pk2[e >> 1] = pack_bf16(k0 ? dp[e] : 0.f, k1 ? dp[e + 1] : 0.f);
      }
    } else {
      // the item's statistics, -lse2 and -D scale of its queries
      const float* nl = reinterpret_cast<const float*>(smem + KV_OFF_STAT + st * 512) + 32 * h;
      // diagonal tile: queries q >= r; oldest tile of the band: queries q <= r; no mask in between
      const uint32_t keep = (diag ? bits_ge(rd) : 0xffffffffu) & (bound ? bits_le(rd) : 0xffffffffu);
      const float2 sl2 = make_float2(a.scale_log2, a.scale_log2), sc2 = make_float2(a.scale, a.scale);
      if (diag || bound) mask32(s, keep);                      // exp2(-inf) = 0: weight and score gradient vanish
#pragma unroll
      for (int e4 = 0; e4 < 32; e4 += 4) {
        const float4 lv = *reinterpret_cast<const float4*>(nl + e4);
        const float4 dv = *reinterpret_cast<const float4*>(nl + 64 + e4);
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
          const int e = e4 + u;
          const float2 y = __ffma2_rn(make_float2(s[e], s[e + 1]), sl2, u ? make_float2(lv.z, lv.w) : make_float2(lv.x, lv.y));
          const float2 p = make_float2(ex2(y.x), ex2(y.y));
          const float2 d = __fmul2_rn(p, __ffma2_rn(make_float2(dp[e], dp[e + 1]), sc2, u ? make_float2(dv.z, dv.w) : make_float2(dv.x, dv.y)));
          pk1[e >> 1] = pack_bf16(p.x, p.y);
          pk2[e >> 1] = pack_bf16(d.x, d.y);
        }
      }
    }
    // bf16 results, two per column, once the group's previous ones have been consumed
    const int gn = (gi0 + n) >> 1;
    if (gn >= 1) WAIT_ON(bars->p_free[g], (gn - 1) & 1);
    tc_fence_after();
    tmem_st16(tW, pk1);
    tmem_st16(tW + 32, pk2);
    tmem_wait_st();
    tc_fence_before();
    mbar_arrive(&bars->p_ready[g]);

    if (is_r && n + 2 >= pl.n_R) {                              // this group's last residual item of this key tile
      // end of the residual items: dK := dphi_k through the feature map's gradient (softmax map:
      // phi(k) (dphi_k - <dphi_k, phi(k)>)), a quarter of the columns per thread: every window item waits for it
      WAIT_ON(bars->r_acc_done, cnt.cr & 1);
      tc_fence_after();
      // the identity map leaves dphi_k as it is
      if (a.phi != RATTN_PHI_IDENTITY) {
        const bool soft = (a.phi == RATTN_PHI_SOFTMAX);
        const int part = 2 * g + h;
        unsigned char* sKphi = smem + KV_OFF_KPHI;
        float df[32];
        tmem_ld32(tK + 32 * part, df);
        tmem_wait_ld();
        uint4 u[4];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) u[cc] = *reinterpret_cast<const uint4*>(sKphi + swz(r, 4 * part + cc));
        float dot = 0.f;
        if (soft) {
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&u[cc]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 f = __bfloat1622float2(h2[e]);
              dot += f.x * df[8 * cc + 2 * e] + f.y * df[8 * cc + 2 * e + 1];
            }
          }
          // the four parts of a row meet in its phi(k), which nothing reads any more
          *reinterpret_cast<float*>(sKphi + swz(r, 4 * part)) = dot;
          asm volatile("bar.sync %0, 128;" ::"r"(4 + (r >> 5)) : "memory");   // the four warps of these 32 rows
          float d4[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) d4[k] = *reinterpret_cast<const float*>(sKphi + swz(r, 4 * k));
          dot = (d4[0] + d4[1]) + (d4[2] + d4[3]);
        }
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&u[cc]);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(h2[e]);
            float &d0 = df[8 * cc + 2 * e], &d1 = df[8 * cc + 2 * e + 1];
            d0 = soft ? f.x * (d0 - dot) : f.x > 0.f ? d0 : 0.f;             // ReLU: relu(k) > 0 exactly where k > 0
            d1 = soft ? f.y * (d1 - dot) : f.y > 0.f ? d1 : 0.f;
          }
        }
        tmem_st32(tK + 32 * part, df);
        tmem_wait_st();
      }
      tc_fence_before();
      mbar_arrive(&bars->fold_done);
    }
  }

  // every product has completed: group 1 stages dV and group 0 dK in the ring slots of this tile's last two items, from
  // where the loader warp stores them
  {
    WAIT_ON(bars->all_done, cnt.it & 1);
    tc_fence_after();
    const uint32_t tOut = (g == 0 ? tK : tV) + 64 * h;
    float x[2][32];
    tmem_ld32(tOut, x[0]);
    tmem_ld32(tOut + 32, x[1]);
    tmem_wait_ld();
    tc_fence_before();
    mbar_arrive(&bars->acc_free);                              // the accumulators have been read
    if (a.part) {
      // one of several parts: fp32, float4 columns outermost ([32][128 rows]), so that a warp's stores are whole runs
      float4* dst = a.part + ((size_t)pl.part_index * 2 + g) * 4096 + 16 * h * 128 + r;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const float* y = &x[e >> 3][4 * (e & 7)];
        dst[e * 128] = make_float4(y[0], y[1], y[2], y[3]);
      }
    } else {
      unsigned char* sOut = smem + KV_OFF_STAGE + (seq0 + pl.N - 1 - g) % KV_NS * TILE_BYTES;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float* y = &x[e >> 2][8 * (e & 3)];
        *reinterpret_cast<uint4*>(sOut + swz(r, 8 * h + e)) =
            make_uint4(pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]), pack_bf16(y[4], y[5]), pack_bf16(y[6], y[7]));
      }
      fence_proxy_async_smem();
      mbar_arrive(&bars->out_staged);
    }
  }
  cnt.seq = seq0 + pl.N;
  cnt.gi += pl.N;
  if (pl.n_R > 0) ++cnt.cr;
  ++cnt.it;
  }
  return *(volatile int*)&bars->abort == 0;
}

__global__ void __launch_bounds__(KV_THREADS, 1)
tc_bwd_dkv_kernel(const __grid_constant__ KvMaps tm, BwdArgs a, int n_items) {
  extern __shared__ __align__(1024) unsigned char smem[];
  KvBars* bars = reinterpret_cast<KvBars*>(smem + KV_OFF_BAR);
  const int tid = threadIdx.x, warp = tid >> 5;
  if ((smem_u32(smem) & 1023u) != 0) {
    if (tid == 0 && a.status) atomicExch(a.status, 2);
    return;
  }
  if (tid == 0) {
    sched_init(&bars->sched, 32 * KV_ROW_WARPS + 2);
    mbar_init(&bars->kv_full, 1);
    mbar_init(&bars->kphi_ready, 32 * KV_ROW_WARPS);
    for (int i = 0; i < KV_NS; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->acc_done[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->p_ready[i], 16 * KV_ROW_WARPS);
      mbar_init(&bars->p_free[i], 1);
      mbar_init(&bars->phiq_ready[i], 16 * KV_ROW_WARPS);
    }
    mbar_init(&bars->s_read, 16 * KV_ROW_WARPS);
    mbar_init(&bars->r_acc_done, 1);
    mbar_init(&bars->fold_done, 32 * KV_ROW_WARPS);
    mbar_init(&bars->all_done, 1);
    mbar_init(&bars->acc_free, 32 * KV_ROW_WARPS);
    mbar_init(&bars->kv_free, 1);
    mbar_init(&bars->out_staged, 32 * KV_ROW_WARPS);
    mbar_init(&bars->drain, 1);
    mbar_init(&bars->drain2, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == KV_ROW_WARPS) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp == KV_ROW_WARPS + 1 && (tid & 31) == 0) {
    prefetch_map(&tm.k);
    prefetch_map(&tm.v);
    prefetch_tensormap(&tm.rs);
    prefetch_map(&tm.qh);
    prefetch_tensormap(&tm.gsh);
    prefetch_tensormap(&tm.grh);
    prefetch_map(&tm.dk);
    prefetch_map(&tm.dv);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  // registers follow the work: 512 x 104 + 128 x 64 = 640 x 96, the CTA's allocation
  bool ok = true;
  if (warp < KV_ROW_WARPS) setmaxnreg_inc<104>();
  else setmaxnreg_dec<64>();
  if (warp < KV_ROW_WARPS) {
    ok = kv_rows(a, smem, bars, tmem, warp >> 3, (warp >> 2) & 1, tid & 127);
  } else if (warp == KV_ROW_WARPS || warp == KV_ROW_WARPS + 2) {
    ok = warp == KV_ROW_WARPS ? kv_mma_scores(a, smem, bars, tmem) : kv_mma_accum(a, smem, bars, tmem);
    if (!ok) {                                             // let this warp's products in flight finish
      uint64_t* drain = warp == KV_ROW_WARPS ? &bars->drain : &bars->drain2;
      mma_commit(drain);
      for (int it = 0; it < (1 << 16) && !mbar_try_wait(drain, 0); ++it) {}
    }
  } else if (warp == KV_ROW_WARPS + 1) {
    ok = kv_loader(tm, a, smem, bars, n_items);
    if (!ok && (tid & 31) == 0) sched_close(&bars->sched);
  }
  if (!ok && a.status) atomicExch(a.status, 1);
  tc_fence_before();
  __syncthreads();
  if (warp == KV_ROW_WARPS) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// dK, dV of an item = the sum of its parts, rounded once.  Mapping as in the sum of the chunk-state terms: a warp reads
// 128-byte runs of the parts and writes whole 32-byte sectors of eight rows.
struct KvSumArgs {
  const float4* part;
  __nv_bfloat16* out[2];
  int split, n_qt, T, H_kv, layout;
};
__global__ void __launch_bounds__(256) tc_bwd_kv_sum_kernel(const KvSumArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int item = blockIdx.x >> 4, piece = blockIdx.x & 15, which = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = 32 * (piece & 3) + 8 * (warp & 3) + (lane & 7), c4 = 8 * (piece >> 2) + 4 * (warp >> 2) + (lane >> 3);
  const int bh = item / a.n_qt, t = (item - bh * a.n_qt) * TILE + row;
  if (t >= a.T) return;
  const float4* src = a.part + ((size_t)item * a.split * 2 + which) * 4096 + c4 * 128 + row;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int p0 = 0; p0 < a.split; p0 += 4) {
    float4 d[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = p0 + k < a.split ? __ldcg(src + (size_t)(p0 + k) * 2 * 4096) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 4; ++k) { acc.x += d[k].x; acc.y += d[k].y; acc.z += d[k].z; acc.w += d[k].w; }
  }
  const int b = bh / a.H_kv, h = bh - b * a.H_kv;
  const size_t at = (a.layout == RATTN_LAYOUT_BTHD ? ((size_t)b * a.T + t) * a.H_kv + h : (size_t)bh * a.T + t) * 128 + 4 * c4;
  *reinterpret_cast<uint2*>(a.out[which] + at) = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
}

}  // namespace

cudaError_t launch_tc_backward(const Args& a, cudaStream_t s) {
  __nv_bfloat16* g_s = reinterpret_cast<__nv_bfloat16*>(a.do_swa);
  __nv_bfloat16* g_r = reinterpret_cast<__nv_bfloat16*>(a.do_rla);
  const bool rla_on = (a.mode == RATTN_MODE_RATTN);
  const int n_qt = (a.T + TILE - 1) / TILE;
  const int wt = a.w / TILE;
  int n_sm = 0;
  cudaError_t e = sm_count(&n_sm);
  if (e != cudaSuccess) return e;
  if (a.dgamma_swa) {
    e = cudaMemsetAsync(a.dgamma_swa, 0, sizeof(float) * a.H_q * 128, s);
    if (e != cudaSuccess) return e;
  }
  if (a.dgamma_rla) {
    e = cudaMemsetAsync(a.dgamma_rla, 0, sizeof(float) * a.H_q * 128, s);
    if (e != cudaSuccess) return e;
  }
  const int t_pad = a.n_chunks * TILE;
  {
    PrepArgs pa;
    pa.o_s = reinterpret_cast<const __nv_bfloat16*>(a.o_swa);
    pa.o_r = reinterpret_cast<const __nv_bfloat16*>(a.o_rla);
    pa.gamma_s = a.gamma_swa; pa.gamma_r = a.gamma_rla;
    pa.g_s = g_s; pa.g_r = g_r;
    pa.delta = a.delta; pa.dgamma_s = a.dgamma_swa; pa.dgamma_r = a.dgamma_rla;
    pa.lse = a.lse; pa.lse2p = a.lse2p; pa.dscp = a.dscp;
    pa.status = a.status; pa.counters = a.work_counter + 1;
    pa.n_heads = a.B * a.H_q; pa.T = a.T; pa.t_pad = t_pad; pa.H_q = a.H_q; pa.rla_on = rla_on ? 1 : 0;
    pa.eps = a.eps; pa.scale = a.scale;
    const bool gains = a.gamma_swa || a.gamma_rla || a.dgamma_swa || a.dgamma_rla;
    e = gains ? allow_smem<tc_bwd_prep_kernel<true>>(PREP_SMEM) : allow_smem<tc_bwd_prep_kernel<false>>(PREP_SMEM);
    if (e != cudaSuccess) return e;
    const long long n_chunks_all = (long long)pa.n_heads * (t_pad / PREP_ROWS);
    const int grid = (int)(n_chunks_all < 2ll * n_sm ? n_chunks_all : 2ll * n_sm);
    CUtensorMap dy_map;
    if (!make_row_map(&dy_map, a.dout, a.T, a.H_q, a.B, a.layout, PREP_ROWS)) return cudaErrorInvalidValue;
    KernelTimer kt("tc_bwd_prep", s);
    e = launch_pdl(gains ? tc_bwd_prep_kernel<true> : tc_bwd_prep_kernel<false>, dim3(grid), dim3(PREP_THREADS), PREP_SMEM, s, !a.dgamma_swa && !a.dgamma_rla, pa, dy_map);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);

  UMap tm_q, tm_k, tm_v, tm_dq, tm_dk, tm_dv;
  CUtensorMap tm_gs, tm_gr, tm_st, tm_rs;
  const uint64_t nq = (uint64_t)a.B * a.H_q, nkv = (uint64_t)a.B * a.H_kv;
  if (!make_user_map(&tm_q, a.q, a.T, a.H_q, a.B, a.layout) || !make_user_map(&tm_k, a.k, a.T, a.H_kv, a.B, a.layout) ||
      !make_user_map(&tm_v, a.v, a.T, a.H_kv, a.B, a.layout) ||
      !make_map(&tm_gs, g_s, a.T, nq) || !make_map(&tm_gr, g_r, a.T, nq) ||
      !make_user_map(&tm_dq, a.dq, a.T, a.H_q, a.B, a.layout) || !make_user_map(&tm_dk, a.dk, a.T, a.H_kv, a.B, a.layout) ||
      !make_user_map(&tm_dv, a.dv, a.T, a.H_kv, a.B, a.layout) ||
      !make_state_map(&tm_st, a.chunk_state, a.k, nkv * a.n_chunks) || !make_state_map(&tm_rs, a.rstate, a.k, nkv * a.n_chunks))
    return cudaErrorInvalidValue;

  BwdArgs t;
  t.dq = reinterpret_cast<__nv_bfloat16*>(a.dq);
  t.dk = reinterpret_cast<__nv_bfloat16*>(a.dk);
  t.dv = reinterpret_cast<__nv_bfloat16*>(a.dv);
  t.lse = a.lse; t.delta = a.delta; t.status = a.status;
  t.lse2p = a.lse2p; t.dscp = a.dscp; t.t_pad = t_pad;
  t.T = a.T; t.w = a.w; t.H_q = a.H_q; t.group = a.group; t.mode = a.mode; t.n_chunks = a.n_chunks;
  t.scale = a.scale; t.scale_log2 = a.scale * LOG2E;
  t.phi = a.phi;
  t.debug_wait = debug_wait();
  e = allow_smem<tc_bwd_dq_kernel>(DQ_SMEM);
  if (e != cudaSuccess) return e;
  e = allow_smem<tc_bwd_dkv_kernel>(KV_SMEM);
  if (e != cudaSuccess) return e;

  // Reverse states of the residual branch: R_c for c = 0 .. n_r-1 (chunks with a query tile beyond c + wt), a running
  // sum that walks the query tiles from the last one down to wt+1.  The dq kernel does not read them, so the two share
  // the GPU.  A serial chain (one CTA per K/V head) goes first, and the dq kernel runs beside it on the other SMs; that
  // costs least as long as the chain is over by then (1.4 us per tile and query head -- alone 1.7 with one head to a K/V
  // head, 1.34 with two, 1.20 with eight -- against about 1.45 us per key tile + 5 us for a dq item; up to 15 % longer is still cheaper than the other way).  Where it would
  // outlast the dq kernel, its terms are formed in parallel behind that kernel, on the SMs it runs out of items on: at
  // 1 x 16/4 heads, T = 1111, w = 128 the chain took 46 us on four SMs beside a dq kernel of 16 us, the terms and their
  // sum end 11 us behind it.  With a chain on more than half of the SMs there is nothing to share.
  const int n_r = rla_on && a.mode != RATTN_MODE_FULL_CAUSAL ? n_qt - wt - 1 : 0;
  const long long chain_ns = 1400ll * n_r * a.group, dq_ns = 10ll * n_qt * (long long)nq * (145 * (wt + 1) + 500) / n_sm;
  const bool few_heads = 2 * (int)nkv <= n_sm;
  const bool parallel_terms = n_r > 0 && a.rdelta != nullptr && few_heads && 100 * chain_ns > 115 * dq_ns;
  const bool chain_beside = n_r > 0 && !parallel_terms && few_heads;
  const int parts = a.kvpart ? head_split((long long)n_qt * (long long)nkv, a.group) : 1;
  StateLaunch L;
  L.ready = nullptr;
  L.x = a.q; L.y = g_r; L.out = a.rstate;
  L.x_heads = a.H_q; L.x_layout = a.layout; L.y_heads = 0; L.y_layout = 0;
  L.T = a.T; L.n_kv = (int)nkv; L.group = a.group; L.n_chunks = a.n_chunks;
  L.n_steps = n_r; L.first = n_qt - 1; L.dir = -1; L.out_first = n_qt - wt - 2;
  L.store_every = 1; L.store_phase = 0; L.handoff = 0; L.w = a.w; L.final_out = nullptr;
  L.state_in = nullptr; L.seq_lens = nullptr; L.kv_per_batch = 1;
  L.phi = a.phi;
  L.status = a.status; L.name = "tc_state_bwd";
  L.delta = parallel_terms ? a.rdelta : nullptr;
  L.h_split = parts;
  L.after_independent = parallel_terms;
  L.wait_first = false;                                    // (under prep: no difference)
  if (!parallel_terms) {
    e = launch_tc_states(L, s);
    if (e != cudaSuccess) return e;
  }
  {
    DqMaps dm;
    dm.q = tm_q; dm.k = tm_k; dm.v = tm_v; dm.gs = tm_gs; dm.gr = tm_gr; dm.st = tm_st; dm.dq = tm_dq;
    const int n_items = n_qt * (int)nq;
    t.n_bh = (int)nq;
    t.counter = a.work_counter + 1;
    t.wait_before = chain_beside ? 1 : 0;
    t.wait_first = chain_beside ? 0 : 1;
    t.split = 1; t.part = nullptr;
    KernelTimer kt("tc_bwd_dq", s);
    e = launch_pdl(tc_bwd_dq_kernel, dim3((unsigned)(n_items < n_sm ? n_items : n_sm)), dim3(DQ_THREADS), DQ_SMEM, s, true, dm, t,
                   n_items, n_qt);
    if (e != cudaSuccess) return e;
  }
  if (parallel_terms) {
    e = launch_tc_states(L, s);
    if (e != cudaSuccess) return e;
  }
  KvMaps km;
  km.k = tm_k; km.v = tm_v; km.rs = tm_rs; km.dk = tm_dk; km.dv = tm_dv;
  if (!make_user_map(&km.qh, a.q, a.T, a.H_q, a.B, a.layout, 64) || !make_map(&km.gsh, g_s, a.T, nq, 64) ||
      !make_map(&km.grh, g_r, a.T, nq, 64))
    return cudaErrorInvalidValue;
  {
    const int n_items = n_qt * (int)nkv * parts;
    t.n_bh = (int)nkv * parts;
    t.split = parts;
    t.part = parts > 1 ? reinterpret_cast<float4*>(a.kvpart) : nullptr;
    t.counter = a.work_counter + 2;
    t.wait_before = 0;
    KernelTimer kt("tc_bwd_dkv", s);
    e = launch_pdl(tc_bwd_dkv_kernel, dim3((unsigned)(n_items < n_sm ? n_items : n_sm)), dim3(KV_THREADS), KV_SMEM, s, true, km, t,
                   n_items);
    if (e != cudaSuccess) return e;
  }
  if (parts > 1) {
    KvSumArgs sa;
    sa.part = reinterpret_cast<const float4*>(a.kvpart);
    sa.out[0] = t.dk; sa.out[1] = t.dv;
    sa.split = parts; sa.n_qt = n_qt; sa.T = a.T; sa.H_kv = a.H_kv; sa.layout = a.layout;
    KernelTimer kt("tc_bwd_kv_sum", s);
    e = launch_pdl(tc_bwd_kv_sum_kernel, dim3((unsigned)(n_qt * (int)nkv * 16), 2), dim3(256), 0, s, true, sa);
    if (e != cudaSuccess) return e;
    count_launches(1);
  }
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace rattn
