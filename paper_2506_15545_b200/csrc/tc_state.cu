// Chunk states of the linear branch, one pass (sm_100a: TMA + tcgen05 + TMEM).
//
// Forward (Eq. 2 of the paper, chunk C = 128):  S_[c+1] = S_[c] + phi(K_c)^T V_c,  S_[0] = 0.
// Backward, the mirror image over query tiles:   R_c = sum_{i > c + w/128} sum_heads phi(Q_i)^T g_r,i.
// Both are running sums of 128 x 128 outer-product blocks along the sequence, so one kernel
// serves both: a CTA owns one K/V head, walks the chunks in order and keeps the running sum in
// TMEM (fp32).  The sum leaves as bf16 (the operand type of the products that read it) after
// every `store_every`-th chunk -- the paper's "states stored every m chunks" -- and, when the
// caller wants the decode state, once more in fp32 at the end.  phi (softmax over the head
// features, Section 3.1) is applied to the loaded tile in shared memory.
//
// The chain is a pipeline of five roles, so that a step costs little more than its slowest
// stage (the feature map, bound by the exponential unit):
//   loader warp    TMA: X and Y tiles of the next chunks into a ring of three stages
//   16 phi warps   feature map of the X tile in place, four lanes per row
//   MMA warp       acc += phi(X)^T Y as soon as the tile is mapped
//   8 flush warps  after a stored step: accumulator -> registers (the MMA warp goes on as soon as
//                  the TMEM loads have landed) -> bf16 -> staging tile; two threads per row
//   store warp     staging tile -> TMA store, and the number of stored states where they are published
// A step takes 1.64 us where every sum is stored, 1.30 where every second one is and 2.3 where they are published (4 to 16
// heads on a GPU to itself; with eight phi and four flush warps, which looked for the staging tile only once they held the
// sum, 2.6 and 1.65).
#include <climits>

#include "tc_common.cuh"

namespace rattn {
namespace {

using namespace ptx;
using namespace tc;

constexpr int ST_NS = 3;                                   // ring stages
constexpr int ST_STAGE = 2 * TILE_BYTES;                   // X tile + Y tile
constexpr int ST_OFF_OUT = ST_NS * ST_STAGE;               // staging for one [128 x 128] bf16 matrix
constexpr int ST_OFF_BAR = ST_OFF_OUT + TILE_BYTES;
constexpr int ST_SMEM = ST_OFF_BAR + 128;
constexpr int ST_PHI_WARPS = 16, ST_FLUSH_WARP = 20;      // 16: MMA warp, 17: loader warp, 18: store warp (19 is idle)
constexpr int ST_THREADS = 32 * (ST_FLUSH_WARP + 8);

struct StateArgs {
  int n_steps;      // chunks to walk
  int first, dir;   // chunk index of step s: first + dir * s
  int group;        // heads summed per chunk (X/Y matrix index = kv * group + head)
  int out_first;    // output matrix of step s: kv * n_chunks + out_first + dir * s
  int n_chunks;
  int store_every;  // the sum after step s is stored iff (out_first + dir * s) % store_every == store_phase
  int store_phase;
  int handoff;      // forward chain that also yields the decode state (see StateLaunch)
  int T, w;         // rows per head in memory, window
  float* final_out; // optional fp32 [n_kv, 128, 128]: the sum after the last step
  const float* state_in;   // optional fp32 [n_kv, 128, 128]: the sum starts from it; matrix out_first - dir holds it
  const int* seq_lens;     // optional: valid rows per batch entry
  int kv_per_batch;
  int phi;          // rattn_feature_map
  int* status;
  int* ready;       // optional [n_kv]: number of leading output matrices stored so far (forward chain)
  float* delta;     // optional: the CTA forms the term of one step alone and leaves it here in fp32, matrix
                    // (kv * n_split + step), its float4 columns outermost ([32][128 rows][4])
  int n_ctas;       // CTAs with work: the grid may have one more
  int n_split;      // steps that the grid is split into (delta)
  int h_split;      // ... and the group's heads: term matrix ((kv * n_split + step) * h_split + part)
  int wait_before;  // 1: the kernel ahead may still be running; not to end before it
  int wait_first;   // 1: set up under the kernel ahead, whose results this one reads
  int debug_wait;   // debug build only, 2 (4): the first (last) wait for a sum of some of the flush threads counts as run out
};

struct StBars {
  uint64_t full[ST_NS], phi_ready[ST_NS], free_[ST_NS], done, acc_free, staged, stage_free;
  uint32_t tmem_base;
  int abort;
};

// steps of a head's chain: the caller's count, or -- variable-length batches -- what the entry's own length asks for; with
// the hand-off the tokens from len - w on are still inside the window
__device__ __forceinline__ int head_len(const StateArgs& a, int kv) {
  return a.seq_lens ? min(a.T, a.seq_lens[kv / a.kv_per_batch]) : a.T;
}
__device__ __forceinline__ int head_steps(const StateArgs& a, int kv) {
  if (!a.seq_lens) return a.n_steps;
  const int len = head_len(a, kv), nd = max(0, (len + TILE - 1) / TILE - 1 - a.w / TILE);
  return (a.handoff && len > a.w) ? nd + 1 : nd;
}
__device__ __forceinline__ bool stored_step(const StateArgs& a, int s) {
  const int o = a.out_first + a.dir * s;
  return o >= 0 && (o % a.store_every) == a.store_phase;
}
__device__ __forceinline__ bool flushed_step(const StateArgs& a, int s, int n_steps) {
  return a.delta != nullptr || stored_step(a, s) || (a.final_out != nullptr && s == n_steps - 1);
}

__global__ void __launch_bounds__(ST_THREADS, 1)
tc_state_scan_kernel(const __grid_constant__ UMap tm_x, const __grid_constant__ UMap tm_y,
                     const __grid_constant__ CUtensorMap tm_out, StateArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  StBars* bars = reinterpret_cast<StBars*>(smem + ST_OFF_BAR);
  if ((int)blockIdx.x >= a.n_ctas) return;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int unit = a.delta ? (int)blockIdx.x / a.h_split : (int)blockIdx.x;      // (K/V head, step)
  const int kv = a.delta ? unit / a.n_split : unit;
  const int first = a.delta ? a.first + a.dir * (unit - kv * a.n_split) : a.first;
  const int group = a.delta ? a.group / a.h_split : a.group, head0 = a.delta ? group * ((int)blockIdx.x - unit * a.h_split) : 0;
  // The kernel that follows may start its own prologue, and whatever does not read the states; where this kernel itself is set
  // up under the one ahead, behind its wait, because the next one relies on what is ahead of this one.
  if (!a.wait_first) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if ((smem_u32(smem) & 1023u) != 0) {
    if (tid == 0 && a.status) atomicExch(a.status, 2);
    return;
  }
  if (tid == 0) {
    for (int i = 0; i < ST_NS; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->phi_ready[i], 32 * ST_PHI_WARPS);
      mbar_init(&bars->free_[i], 1);
    }
    mbar_init(&bars->done, 1);
    mbar_init(&bars->acc_free, 256);
    mbar_init(&bars->staged, 256);
    mbar_init(&bars->stage_free, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == ST_PHI_WARPS) {
    tmem_alloc(&bars->tmem_base, 128);
    tmem_relinquish();
  }
  if (tid == 32 * (ST_PHI_WARPS + 1)) {
    prefetch_map(&tm_x);
    prefetch_map(&tm_y);
    prefetch_tensormap(&tm_out);
  }
  if (a.wait_first) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  int n_steps = head_steps(a, kv);
  const int row_limit = a.handoff ? head_len(a, kv) - a.w : INT_MAX;
  if (a.delta) n_steps = unit - kv * a.n_split < n_steps ? 1 : 0;     // one term, or none beyond this head's length
  const bool has_init = (a.state_in != nullptr) && !a.delta;        // of terms the incoming state is none
  const int n_items = n_steps * group;
  bool ok = true;

  // registers follow the work: 512 x 64 + 128 x 48 + 256 x 96, within the CTA's 896 x 72
  if (warp < ST_PHI_WARPS) {
    setmaxnreg_dec<64>();
    // ---- feature map of the X tile, in place: four lanes per row ---------------------------
    const int row = 8 * warp + 4 * ((tid >> 4) & 1) + ((tid >> 1) & 3), q = 2 * ((tid >> 3) & 1) + (tid & 1);
    for (int it = 0; it < n_items && ok; ++it) {
      const int st = it % ST_NS, use = it / ST_NS;
      ok = mbar_wait_warp(&bars->full[st], use & 1, &bars->abort);
      if (!ok) break;
      unsigned char* x = smem + st * ST_STAGE + row * 128;
      const int token = (first + a.dir * (it / group)) * TILE + row;
      // every lane maps its row (the softmax map exchanges partial results between the lanes
      // of a row with full-warp shuffles, so no lane may skip it); rows past the limit are then cleared
      feature_map_quad<true>(x, x, HALF_BYTES, row, q, a.phi);
      __syncwarp();
      if (token >= row_limit) {
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(x + (q >> 1) * HALF_BYTES + ((4 * (q & 1) + c) << 4)) = make_uint4(0, 0, 0, 0);
      }
      fence_proxy_async_smem();
      mbar_arrive(&bars->phi_ready[st]);
    }
  } else if (warp >= ST_FLUSH_WARP) {
    setmaxnreg_inc<96>();
    // ---- flush: thread = accumulator row (its warp's TMEM lane quarter) and one half of the columns
    const int r = (warp & 3) * 32 + (tid & 31), half = (warp - ST_FLUSH_WARP) >> 2;
    const uint32_t t_row = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 64 * half;
    unsigned char* s_out = smem + ST_OFF_OUT;
    int n_flush = 0, n_stored = 0;
    // The staging tile has left; all of these warps or none of them go on.
    auto stage_free = [&]() -> bool {
      if (n_stored >= 1) mbar_wait(&bars->stage_free, (n_stored - 1) & 1, &bars->abort);
      return !named_any(4, 256, *(volatile int*)&bars->abort);
    };
    // bf16 copy of this thread's half row of the sum -> staging; the store warp sends it off, unless a thread has given up
    // waiting for the sum and does not say that its share is there
    auto store_row = [&](const float (&x)[2][32], bool arrived) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          uint4 u;
          u.x = pack_bf16(x[c][8 * e + 0], x[c][8 * e + 1]);
          u.y = pack_bf16(x[c][8 * e + 2], x[c][8 * e + 3]);
          u.z = pack_bf16(x[c][8 * e + 4], x[c][8 * e + 5]);
          u.w = pack_bf16(x[c][8 * e + 6], x[c][8 * e + 7]);
          *reinterpret_cast<uint4*>(s_out + swz(r, 8 * half + 4 * c + e)) = u;
        }
      }
      fence_proxy_async_smem();
      if (arrived) mbar_arrive(&bars->staged);
      ++n_stored;
    };
    auto write_final = [&](const float (&x)[2][32]) {
      float* dst = a.final_out + ((size_t)kv * 128 + r) * 128 + 64 * half;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          *reinterpret_cast<float4*>(dst + 32 * c + 4 * e) =
              make_float4(x[c][4 * e], x[c][4 * e + 1], x[c][4 * e + 2], x[c][4 * e + 3]);
      }
    };
    if (has_init || (a.final_out != nullptr && n_steps == 0 && !a.delta)) {
      // the chain starts from the incoming state (zero without one): into the accumulator, into the
      // matrix in front of the first step's, and -- when no token leaves the window -- straight out
      float x[2][32];
      const float* src = has_init ? a.state_in + ((size_t)kv * 128 + r) * 128 + 64 * half : nullptr;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float4 f = src ? *reinterpret_cast<const float4*>(src + 32 * c + 4 * e) : make_float4(0.f, 0.f, 0.f, 0.f);
          x[c][4 * e] = f.x; x[c][4 * e + 1] = f.y; x[c][4 * e + 2] = f.z; x[c][4 * e + 3] = f.w;
        }
      }
      if (has_init) {
#pragma unroll
        for (int c = 0; c < 2; ++c) tmem_st32(t_row + 32 * c, x[c]);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bars->acc_free);
        if (stored_step(a, -1)) store_row(x, true);
      }
      if (a.final_out != nullptr && n_steps == 0) write_final(x);
    }
    for (int s = 0; s < n_steps && ok; ++s) {
      if (!flushed_step(a, s, n_steps)) continue;
      // (ahead of the wait, so that the last store passes under it)
      if (!a.delta && stored_step(a, s) && !stage_free()) { ok = false; break; }
      bool arrived = mbar_wait(&bars->done, n_flush & 1, &bars->abort);
#ifdef RATTN_DEBUG_KNOBS
      if (warp == ST_FLUSH_WARP && (a.debug_wait == 2 ? n_flush == 0 : a.debug_wait == 4 && s == n_steps - 1)) {
        bars->abort = 1;
        arrived = false;
      }
#endif
      ++n_flush;
      tc_fence_after();
      float x[2][32];
#pragma unroll
      for (int c = 0; c < 2; ++c) tmem_ld32(t_row + 32 * c, x[c]);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&bars->acc_free);                            // the next step may accumulate
      if (a.delta) {                                           // rows are neighbours in memory: whole 512-byte runs per store
        float4* dst = reinterpret_cast<float4*>(a.delta) + (size_t)blockIdx.x * 4096 + 16 * half * 128 + r;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            dst[(8 * c + e) * 128] = make_float4(x[c][4 * e], x[c][4 * e + 1], x[c][4 * e + 2], x[c][4 * e + 3]);
        continue;
      }
      if (stored_step(a, s)) store_row(x, arrived);
      if (a.final_out != nullptr && s == n_steps - 1) write_final(x);
    }
  } else {
    setmaxnreg_dec<48>();
    if (warp == ST_PHI_WARPS) {
      // ---- acc[128 features x 128] += phi(X)^T Y   (both operands MN-major: rows are the tokens)
      int n_wait = 0;                                          // hand-backs of the accumulator so far
      for (int it = 0; it < n_items && ok; ++it) {
        const int st = it % ST_NS, use = it / ST_NS;
        const int s = it / group, hh = it - s * group;
        ok = mbar_wait_warp(&bars->phi_ready[st], use & 1, &bars->abort);
        // the flush warps hold the previous sum, or are still writing the incoming state into the accumulator
        if (ok && hh == 0 && ((s > 0 && flushed_step(a, s - 1, n_steps)) || (s == 0 && has_init))) {
          ok = mbar_wait_warp(&bars->acc_free, n_wait & 1, &bars->abort);
          ++n_wait;
        }
        if (!ok) break;
        tc_fence_after();
        mma_mnmn(tmem, smem_u32(smem + st * ST_STAGE), smem_u32(smem + st * ST_STAGE + TILE_BYTES), it > 0 || has_init);
        mma_commit(&bars->free_[st]);
        if (hh == group - 1 && flushed_step(a, s, n_steps)) mma_commit(&bars->done);
      }
    } else if (warp == ST_PHI_WARPS + 2) {
      // ---- store: staged sums to memory, in order -----------------------------------------------
      int n = 0;
      for (int s = (has_init ? -1 : 0); s < n_steps && ok && !a.delta; ++s) {
        if (!stored_step(a, s)) continue;
        const int mat = a.out_first + a.dir * s;
        ok = mbar_wait_warp(&bars->staged, n & 1, &bars->abort);
        if (!ok) break;
        ++n;
        if ((tid & 31) == 0) {
          store_tile(&tm_out, smem + ST_OFF_OUT, 0, kv * a.n_chunks + mat);
          tma_store_commit();
          tma_store_wait_read();
          mbar_arrive(&bars->stage_free);
          if (a.ready) {
            // The kernel that reads the states runs beside this one and takes them as they appear: the matrix must be in
            // memory, not merely read out of the staging tile, before its index is shown.  (Shown one store later, without
            // this wait, the reader lost more than the chain gained: 129.5 -> 131 us for a chunk of 2 x 32/8 heads, T = 2048.)
            tma_store_wait();
            fence_proxy_async_all();
            __threadfence();
            st_release_gpu(a.ready + kv, mat + 1);
          }
        }
        __syncwarp();
      }
      if ((tid & 31) == 0) tma_store_wait();
    } else if (warp == ST_PHI_WARPS + 1) {
      // ---- loader ---------------------------------------------------------------------------
      for (int it = 0; it < n_items && ok; ++it) {
        const int st = it % ST_NS, use = it / ST_NS;
        const int s = it / group, hh = it - s * group;
        if (use >= 1) ok = mbar_wait_warp(&bars->free_[st], (use - 1) & 1, &bars->abort);
        if (!ok) break;
        const int row = (first + a.dir * s) * TILE, z = kv * a.group + head0 + hh;
        unsigned char* dst = smem + st * ST_STAGE;
        mbar_arrive_expect_tx(&bars->full[st], ST_STAGE);
        load_tile(dst, &tm_x, &bars->full[st], row, z);
        load_tile(dst + TILE_BYTES, &tm_y, &bars->full[st], row, z);
      }
    }
  }
  if (a.wait_before) asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  // every wait that has run out has raised the flag, the last one of a role too
  if (tid == 0 && bars->abort && a.status) atomicExch(a.status, 1);
  if (warp == ST_PHI_WARPS) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

// Running sums of the terms left by the kernel above: state(s) = incoming state + the terms 0 .. s (each h_split matrices),
// as bf16, row-major, and the last one in fp32 where the decode state is asked for.  A pure stream (64 KB in per term
// matrix, 32 KB out per state): a thread owns one float4 of the matrix and walks the terms with eight loads in flight.  A
// warp covers 8 rows x 4 float4 columns, so that it reads 128-byte runs of the column-major terms and writes whole 32-byte
// sectors of the row-major states.
__global__ void __launch_bounds__(256) tc_state_sum_kernel(const StateArgs a, uint2* __restrict__ out) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int kv = blockIdx.x >> 4, part = blockIdx.x & 15;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = 32 * (part & 3) + 8 * (warp & 3) + (lane & 7), c4 = 8 * (part >> 2) + 4 * (warp >> 2) + (lane >> 3);
  const int n = head_steps(a, kv) * a.h_split;
  const float4* src = reinterpret_cast<const float4*>(a.delta) + (size_t)kv * a.n_split * a.h_split * 4096 + c4 * 128 + row;
  uint2* dst = out + (size_t)kv * a.n_chunks * 4096 + row * 32 + c4;
  const size_t at = (size_t)kv * 4096 + row * 32 + c4;              // of a row-major fp32 matrix, in float4
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  auto store = [&](int s) {
    if (stored_step(a, s))
      dst[(ptrdiff_t)(a.out_first + a.dir * s) * 4096] = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
  };
  if (a.state_in) {
    acc = reinterpret_cast<const float4*>(a.state_in)[at];
    store(-1);
  }
  int left = a.h_split, s = 0;
  for (int i0 = 0; i0 < n; i0 += 8) {
    float4 d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) d[k] = i0 + k < n ? __ldcg(src + (size_t)(i0 + k) * 4096) : acc;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (i0 + k >= n) break;
      acc.x += d[k].x; acc.y += d[k].y; acc.z += d[k].z; acc.w += d[k].w;
      if (--left == 0) {
        store(s++);
        left = a.h_split;
      }
    }
  }
  if (a.final_out) reinterpret_cast<float4*>(a.final_out)[at] = acc;
}

}  // namespace

// x, y: [n_kv * group, T, 128] bf16; out: [n_kv * n_chunks, 128, 128] bf16.
cudaError_t launch_tc_states(const StateLaunch& L, cudaStream_t s) {
  if (L.n_steps <= 0 && !L.state_in && !(L.seq_lens && L.final_out)) return cudaSuccess;
  UMap tm_x, tm_y;
  CUtensorMap tm_out;
  const uint64_t n_mats = (uint64_t)L.n_kv * L.group;
  auto user = [&](UMap* m, const void* base, int heads, int layout) {
    return heads > 0 ? make_user_map(m, base, L.T, heads, n_mats / heads, layout) : make_user_map(m, base, L.T, n_mats, 1, 0);
  };
  if (!user(&tm_x, L.x, L.x_heads, L.x_layout) || !user(&tm_y, L.y, L.y_heads, L.y_layout) ||
      !make_map(&tm_out, L.out, 128, (uint64_t)L.n_kv * L.n_chunks))
    return cudaErrorInvalidValue;
  StateArgs a;
  a.n_steps = L.n_steps; a.first = L.first; a.dir = L.dir; a.group = L.group; a.out_first = L.out_first;
  a.n_chunks = L.n_chunks; a.status = L.status;
  a.store_every = L.store_every > 0 ? L.store_every : 1;
  a.store_phase = L.store_phase;
  a.handoff = L.handoff; a.T = L.T; a.w = L.w;
  a.final_out = L.final_out;
  a.state_in = L.state_in;
  a.seq_lens = L.seq_lens; a.kv_per_batch = L.kv_per_batch > 0 ? L.kv_per_batch : 1;
  a.phi = L.phi;
  a.ready = (L.dir > 0 && L.group == 1) ? L.ready : nullptr;
  a.delta = L.delta;
  a.n_split = L.delta ? L.n_steps : 1;
  a.h_split = L.delta ? L.h_split : 1;
  a.n_ctas = L.n_kv * a.n_split * a.h_split;
  a.wait_before = L.after_independent ? 1 : 0;
  a.wait_first = L.wait_first ? 1 : 0;
  a.debug_wait = debug_wait();
  cudaError_t e = allow_smem<tc_state_scan_kernel>(ST_SMEM);
  if (e != cudaSuccess) return e;
  {
    KernelTimer kt(L.name, s);
    // CTAs that are set up under a kernel whose CTAs are just leaving find their SMs here and there, and one that shares a TPC
    // with a CTA of the main kernel is slower, the slowest by a fifth: 4 x 8/8 heads, T = 6144, w = 1408, hand-off 233 us in full
    // order, 252 so.  As pairs, which take a TPC's two SMs like the CTAs of a launch onto an empty GPU, 232; in the mean over
    // 352 sizes of 8 to 36 heads 3 % faster than in full order (and 0.8 without the pairs, a quarter of them slower).
    const int cluster = L.wait_first && a.n_ctas > 1 ? 2 : 1;
    e = launch_pdl_cluster(tc_state_scan_kernel, dim3((unsigned)((a.n_ctas + cluster - 1) / cluster * cluster)), dim3(ST_THREADS),
                           ST_SMEM, s, L.after_independent || L.wait_first, cluster, tm_x, tm_y, tm_out, a);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  if (L.delta) {
    KernelTimer kt("tc_state_sum", s);
    e = launch_pdl(tc_state_sum_kernel, dim3((unsigned)L.n_kv * 16), dim3(256), 0, s, true, a, reinterpret_cast<uint2*>(L.out));
    if (e != cudaSuccess) return e;
    count_launches(1);
  }
  return cudaGetLastError();
}

}  // namespace rattn
