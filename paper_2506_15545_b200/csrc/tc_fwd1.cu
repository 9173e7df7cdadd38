// Tensor-core forward for windows with a linear branch, one query tile per CTA and two CTAs per SM (bf16, d = 128,
// window a multiple of 128; sm_100a: TMA + tcgen05 + TMEM).
//
// Persistent kernel.  A work unit is one query tile (128 rows) of one query head; its key tiles, t down to t - w/128, are
// walked in half tiles of 64 keys ("steps"):
//
//   8 row warps   (thread = query row = TMEM lane, and one half of the columns) SWA (Section 2.1): online softmax
//                 straight out of TMEM; the weights of a step (fp16) are written back over its score columns and read
//                 from there by the P V product, so they never touch shared memory
//   MMA warp      S = Q K^T, O += P V (A operand from TMEM), the residual-branch products
//   loader warp   TMA: Q, and the stream of K and V half tiles and state halves through a ring of five 16 KB slots
//   2 helper warps re-encode each V half tile bf16 -> fp16 in place (tcgen05 needs A and B of one type)
//
//   RLA (Eq. 4 in the chunkwise form of Eq. 2-3 with the window lag): when the window loop ends, its normalised output is
//   parked in registers (fp16) and the same accumulator is reused.  With c = t - w/128 the chunk the tile reads in "intra"
//   form and S_[c] the stored state (sum over the chunks before c of phi(K)^T V):
//       O_rla = phi(Q) S_[c] + ((phi(Q) phi(K_c)^T) masked to j < t - w) V_c
//   phi (softmax over the head features, Section 3.1) is applied to the Q and K tiles in shared memory, in place: it never
//   goes to HBM.
//   Section 3.2: y = g_s * o_swa / rms(o_swa) + g_r * o_rla / rms(o_rla), staged in the tile's Q buffer and written by TMA.
//
// Why two small CTAs. A unit is a chain of dependent phases (scores -> row threads -> products, then the feature maps, the
// residual products, the epilogue), none of which fills the SM alone, and the window loop is less than half of it. The pair
// kernel (tc_fwd2.cu: one CTA per SM, two adjacent tiles sharing each K/V tile) has both tiles in the same phase most of
// the time: 41k cycles per pair at w = 512 for the late units (up to 60k for earlier ones), of which the tensor pipe works
// 14k and the exponential unit 13k. Two independent CTAs drift apart, so that one's feature maps and epilogue pass under
// the other's window loop: 34 - 42k cycles per tile and CTA, i.e. 17 - 21k per tile against 20.5k and more (2 x 16/16
// heads, T = 4096; clock stamps of single units). Half of TMEM (256 columns) holds the accumulator and two 64-column score
// buffers, so the scores of the next step are ready when the row threads come for them. The price: every K/V tile is
// fetched once per query tile (L2 delivers that: measured 70 bytes per clock and SM to two CTAs with copies in flight, half
// of it used), the N = 64 score products read Q from shared memory twice as often (shared memory carries 2.0k cycles per
// tile and key tile against the pair's 1.3k, about what the row threads take), and every tile reads a state of its own, so
// all of them are stored. Without the residual part (control modes) the pair kernel is the faster one.
#include <type_traits>

#include "tc_common.cuh"

namespace rattn {
namespace {

using namespace ptx;
using namespace tc;

constexpr int F_NS = 5;                          // ring slots: a half tile of K or V, or half of a state
constexpr int F_OFF_Q = 0;
constexpr int F_OFF_RING = TILE_BYTES;
constexpr int F_OFF_BAR = F_OFF_RING + F_NS * HT_BYTES;
constexpr int F_OFF_EX = F_OFF_BAR + 384;        // one word per row, between its two threads
constexpr int F_SMEM = F_OFF_EX + TILE * 4;      // 115,584 bytes: two CTAs share the SM's 228 KB
constexpr int F_THREADS = 384;                   // 8 row warps, MMA, loader, 2 converters
constexpr float LOG2E = 1.4426950408889634f;

struct FBars {
  // Ring slots: K or a state landed, V landed, consumed, V re-encoded.  V has a barrier of its own because the converters
  // follow the V uses alone: a wait by parity cannot skip a phase (two loads in flight may land in either order).
  uint64_t full[F_NS], v_full[F_NS], free_[F_NS], v_ready[F_NS];
  uint64_t q_full, q_free, s_full[2], p_ready[2], pv_done, o_ready, stash_done, phi_ready, o_free, drain;
  SchedRing sched;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(FBars) <= F_OFF_EX - F_OFF_BAR, "barriers");

struct FArgs {
  float* lse;
  __nv_bfloat16* o_swa;   // training mode: un-normalised branch outputs [B*H_q, T, 128] as bf16
  __nv_bfloat16* o_rla;   // (the tensor-core backward reads them in that form)
  const float* gamma_swa;
  const float* gamma_rla;
  int* status;
  int* clear_status;      // status word that nothing ahead of this kernel has cleared
  int* work_counter;      // next unit to hand out (device memory, zero at launch); null: static round-robin
  int T, w, H_q, group, n_chunks, n_qt, n_units, n_bh;
  int phi;                // rattn_feature_map
  int off;                // key tile of query tile 0 (a resumed sequence carries w/128 history tiles in front)
  int first_state;        // smallest chunk index whose state is stored: 1 (S_[0] = 0), or 0 with an incoming state
  const int* seq_lens;    // optional [B]: valid query rows per batch entry
  int n_stateless;        // tiles that read no stored state; their units come first
  int wait_first;         // the kernel ahead produces what this one reads: wait for it after the set-up
  int wait_for_states;    // a chunk-state kernel runs ahead of this one: wait for it before the first state load
  const int* state_ready; // ... or, per K/V head, for the number of states it has published so far (null: the former)
  int ascending;          // units in sequence order, the order in which their states appear
  int debug_wait;         // debug build only, 1: the row threads withhold their first hand-over (a wait then runs out); 2: the
                          // first wait of one half of them counts as run out
  float scale_log2, eps;
};

struct FMaps {
  UMap q, k, v, out;          // the caller's tensors (either head layout); k, v in half tiles
  CUtensorMap st;             // chunk states, in halves of 64 features
  CUtensorMap o_swa, o_rla;   // training mode: the un-normalised branch outputs, [B*H_q, T, 128] bf16
};

// What one unit consists of; every role derives the same plan from the unit index.
struct Unit {
  int bh_q, bh_kv, h;
  int t;                    // key-space index of the query tile; -1: beyond this batch entry's length
  int n;                    // key tiles t, t-1, ..., t-n+1; two steps each, the lower 64 keys first
  int c;                    // the chunk of the residual part (rla)
  bool rla, has_state;
};

__device__ __forceinline__ Unit make_unit(const FArgs& a, int u) {
  Unit un;
  // Order: first the tiles that read no stored state (they can run while the chunk-state kernel
  // is still at work), then the others, heaviest first.
  const int pr = u / a.n_bh;
  un.bh_q = u - pr * a.n_bh;
  const int p = (a.ascending || pr < a.n_stateless) ? pr : a.n_qt - 1 - (pr - a.n_stateless);
  const int b = un.bh_q / a.H_q;
  un.h = un.bh_q - b * a.H_q;
  un.bh_kv = b * (a.H_q / a.group) + un.h / a.group;
  const int wt = a.w / TILE;
  // tile indices are key-space positions: query tile i of the call sits at key tile i + off
  const int n_qt = a.seq_lens ? (min(a.T, a.seq_lens[b]) + TILE - 1) / TILE : a.n_qt;
  un.t = p < n_qt ? a.off + p : -1;
  un.c = un.t - wt;
  un.rla = un.t >= 0 && un.c >= 0;
  un.n = (un.rla ? wt : un.t) + 1;
  un.has_state = un.rla && un.c >= a.first_state;
  return un;
}

// The ring order of a unit with L steps.  Loads and releases run in the same order,
//   K0 K1 V0 K2 V1 K3 ... K(L-1) V(L-2) V(L-1),
// except that a unit with a residual part, which reads the last tile's K and V once more, brings V(L-3) in front of
// K(L-2): the four half tiles that are kept are then the last four, and the two state halves that follow take the slots
// of V(L-3) and K(L-2).
__device__ __forceinline__ int pos_k(int s, int L, bool rla) { return s < 2 ? s : (rla && s == L - 2) ? 2 * s : 2 * s - 1; }
__device__ __forceinline__ int pos_v(int s, int L, bool rla) {
  return s == L - 1 ? 2 * L - 1 : (rla && s == L - 3) ? 2 * s + 1 : 2 * s + 2;
}
__device__ __forceinline__ int unit_uses(const Unit& un) { return 4 * un.n + (un.has_state ? 2 : 0); }
// ring position -> slot and phase of its use
struct Ring {
  int base = 0;                                  // uses of the units before
  __device__ __forceinline__ int slot(int pos) const { return (base + pos) % F_NS; }
  __device__ __forceinline__ uint32_t phase(int pos) const { return (uint32_t)((base + pos) / F_NS) & 1u; }   // of free_
};
// full, v_full and v_ready complete once per use of their own kind: parity of the next such use of each slot
struct UsePhase {
  uint32_t bits = 0;
  __device__ __forceinline__ uint32_t take(int st) {
    const uint32_t p = (bits >> st) & 1u;
    bits ^= 1u << st;
    return p;
  }
};

#define WAIT_OR_RETURN(bar, parity) \
  do { if (!mbar_wait(&(bar), (parity), &bars->abort)) return false; } while (0)
#define WAIT_OR_RETURN_W(bar, parity) \
  do { if (!mbar_wait_warp(&(bar), (parity), &bars->abort)) return false; } while (0)

// of threads that share named barriers: see mbar_wait
#define WAIT_ON(bar, parity) mbar_wait(&(bar), (parity), &bars->abort)

// D[128x128] (+)= P[128 x 64 keys] (fp16 in TMEM, 32 columns) . V[64 keys x 128] (fp16, MN-major half tile)
__device__ __forceinline__ void mma_pv(uint32_t d, uint32_t p_tmem, uint32_t v_base, bool acc) {
  constexpr uint32_t idesc = instr_desc(128, 128, 0, 1, 0);
  const uint64_t b0 = mnmajor_base_h(v_base);
#pragma unroll
  for (int k = 0; k < 4; ++k) mma_bf16_ts(d, p_tmem + 8 * k, b0 + kstep_mn(k), idesc, (acc || k > 0) ? 1u : 0u);
}
// D[128x128] (+)= phi(Q)[128 x 64 features] (column half `half` of the Q tile) . S[64 features x 128] (MN-major)
__device__ __forceinline__ void mma_q_state(uint32_t d, uint32_t q_base, int half, uint32_t s_base, bool acc) {
  constexpr uint32_t idesc = instr_desc(128, 128, 0, 1);
  const uint64_t a0 = kmajor_base(q_base + half * HALF_BYTES), b0 = mnmajor_base_h(s_base);
#pragma unroll
  for (int k = 0; k < 4; ++k) mma_bf16(d, a0 + kstep_k(k, HALF_BYTES), b0 + kstep_mn(k), idesc, (acc || k > 0) ? 1u : 0u);
}

// ----------------------------------------------------------------------------- loader
__device__ bool fwd_loader(const FMaps& tm, const FArgs& a, unsigned char* smem, FBars* bars) {
  Ring ring;
  int cu = 0;                                    // units so far
  bool states_ready = (a.wait_for_states == 0);
  for (int n = 0;; ++n) {
    int u;
    if (a.work_counter) {
      if (!sched_draw(&bars->sched, a.work_counter, a.n_units, n, &bars->abort, &u)) return false;
    } else {
      u = blockIdx.x + n * gridDim.x;            // dealt round-robin
      if (u >= a.n_units) u = -1;
      if (!sched_publish(&bars->sched, n, u, &bars->abort)) return false;
    }
    if (u < 0) break;
    const Unit un = make_unit(a, u);
    if (un.t < 0) continue;                      // beyond this batch entry's length
    const int L = 2 * un.n;
    auto slot_wait = [&](int pos) -> bool {      // the slot's previous use has been consumed
      const int use = (ring.base + pos) / F_NS;
      if (use >= 1) WAIT_OR_RETURN_W(bars->free_[ring.slot(pos)], (use - 1) & 1);
      return true;
    };
    auto half_tile = [&](int pos, const UMap* map, uint64_t* landed, int s) -> bool {
      if (!slot_wait(pos)) return false;
      const int st = ring.slot(pos);
      mbar_arrive_expect_tx(&landed[st], HT_BYTES);
      load_half_tile(smem + F_OFF_RING + st * HT_BYTES, map, &landed[st], (un.t - (s >> 1)) * TILE + 64 * (s & 1), un.bh_kv);
      return true;
    };
    // K0 may come while the previous unit's output still occupies the Q buffer
    if (!half_tile(0, &tm.k, bars->full, 0)) return false;
    if (cu >= 1) WAIT_OR_RETURN_W(bars->q_free, (cu - 1) & 1);
    mbar_arrive_expect_tx(&bars->q_full, TILE_BYTES);
    load_tile(smem + F_OFF_Q, &tm.q, &bars->q_full, (un.t - a.off) * TILE, un.bh_q);
    ++cu;
    if (!half_tile(1, &tm.k, bars->full, 1)) return false;
    for (int s = 0; s < L; ++s) {                // V(s) and K(s+2), in ring order
      if (!(un.rla && s == L - 3) && !half_tile(pos_v(s, L, un.rla), &tm.v, bars->v_full, s)) return false;
      if (un.rla && s == L - 4 && !half_tile(pos_v(s + 1, L, un.rla), &tm.v, bars->v_full, s + 1)) return false;
      if (s + 2 < L && !half_tile(pos_k(s + 2, L, un.rla), &tm.k, bars->full, s + 2)) return false;
    }
    if (un.has_state) {
      if (a.state_ready) {
        // the chunk-state kernel, still running beside this one, has stored and published S_[c]
        if (!wait_published(a.state_ready + un.bh_kv, un.c + 1, &bars->abort)) return false;
      } else if (!states_ready) {
        // the chunk-state kernel launched ahead of this one has completed and its stores are visible
        asm volatile("griddepcontrol.wait;" ::: "memory");
        states_ready = true;
      }
      for (int k = 0; k < 2; ++k) {
        if (!slot_wait(2 * L + k)) return false;
        const int st = ring.slot(2 * L + k);
        mbar_arrive_expect_tx(&bars->full[st], HT_BYTES);
        load_half_tile(smem + F_OFF_RING + st * HT_BYTES, &tm.st, &bars->full[st], 64 * k, un.bh_kv * a.n_chunks + un.c);
      }
    }
    ring.base += unit_uses(un);
  }
  return true;
}

// -------------------------------------------------------------------------- V re-encoding
__device__ bool fwd_convert(const FArgs& a, unsigned char* smem, FBars* bars, int cid) {
  Ring ring;
  UsePhase vf;
  for (int n = 0;; ++n) {
    int u;
    if (!sched_read(&bars->sched, n, &bars->abort, &u)) return false;
    if (u < 0) break;
    const Unit un = make_unit(a, u);
    if (un.t < 0) continue;
    prefetch_gains(a.gamma_swa, a.gamma_rla, un.h, cid);
    const int L = 2 * un.n;
    for (int s = 0; s < L; ++s) {
      const int st = ring.slot(pos_v(s, L, un.rla));
      WAIT_OR_RETURN(bars->v_full[st], vf.take(st));
      unsigned char* tile = smem + F_OFF_RING + st * HT_BYTES;
#pragma unroll 4
      for (int c = cid; c < HT_BYTES / 16; c += 64) {
        uint4 x = *reinterpret_cast<uint4*>(tile + c * 16);
        x.x = bf16x2_to_f16x2(x.x);
        x.y = bf16x2_to_f16x2(x.y);
        x.z = bf16x2_to_f16x2(x.z);
        x.w = bf16x2_to_f16x2(x.w);
        *reinterpret_cast<uint4*>(tile + c * 16) = x;
      }
      fence_proxy_async_smem();
      mbar_arrive(&bars->v_ready[st]);
    }
    ring.base += unit_uses(un);
  }
  return true;
}

// ----------------------------------------------------------------------------- MMA warp
__device__ bool fwd_mma(const FArgs& a, unsigned char* smem, FBars* bars, uint32_t tmem) {
  const uint32_t sQ = smem_u32(smem + F_OFF_Q), sR = smem_u32(smem + F_OFF_RING);
  const uint32_t tS = tmem, tO = tmem + 128;
  Ring ring;
  UsePhase kp, vp;                               // K and state uses, V uses
  int cu = 0, cs = 0, cr = 0;                    // units, score hand-overs per buffer, residual units so far

  for (int n = 0;; ++n) {
    int u;
    if (!sched_read_warp(&bars->sched, n, &bars->abort, &u)) return false;
    if (u < 0) break;
    const Unit un = make_unit(a, u);
    if (un.t < 0) continue;
    const int L = 2 * un.n;
    auto scores = [&](int s, bool keep) {                  // S of step s into its buffer; K is released unless kept
      const int st = ring.slot(pos_k(s, L, un.rla));
      mma_k_kh(tS + 64 * (s & 1), sQ, sR + st * HT_BYTES);
      mma_commit(&bars->s_full[s & 1]);
      if (!keep) mma_commit(&bars->free_[st]);
    };
    WAIT_OR_RETURN_W(bars->q_full, cu & 1);
#pragma unroll
    for (int s = 0; s < 2; ++s) {                // a unit with a residual part has at least four steps
      const int kst = ring.slot(pos_k(s, L, un.rla));
      WAIT_OR_RETURN_W(bars->full[kst], kp.take(kst));
      tc_fence_after();
      scores(s, false);
    }
    for (int s = 0; s < L; ++s) {
      // The operands of this step are awaited ahead of the weights, so that the product and the next
      // scores go out the moment the row threads hand their weights over (a wait costs this warp a few
      // hundred cycles even when it is already satisfied).
      const int vst = ring.slot(pos_v(s, L, un.rla));
      WAIT_OR_RETURN_W(bars->v_ready[vst], vp.take(vst));
      if (s + 2 < L) {
        const int kst = ring.slot(pos_k(s + 2, L, un.rla));
        WAIT_OR_RETURN_W(bars->full[kst], kp.take(kst));
      }
      if (s == 0 && cu >= 1) WAIT_OR_RETURN_W(bars->o_free, (cu - 1) & 1);   // the previous unit has read O
      WAIT_OR_RETURN_W(bars->p_ready[s & 1], (cs + (s >> 1)) & 1);
      tc_fence_after();
      mma_pv(tO, tS + 64 * (s & 1), sR + vst * HT_BYTES, s > 0);             // O += P V
      if (!(un.rla && s >= L - 2)) mma_commit(&bars->free_[vst]);
      else if (s == L - 2) mma_commit(&bars->pv_done);
      if (s == L - 1) mma_commit(&bars->o_ready);
      if (s + 2 < L) scores(s + 2, un.rla && s + 2 >= L - 2);
    }
    cs += un.n;
    // ---- residual branch ---------------------------------------------------------------
    if (un.rla) {
      const int ka = ring.slot(2 * L - 4), kb = ring.slot(2 * L - 3), va = ring.slot(2 * L - 2), vb = ring.slot(2 * L - 1);
      const int sa = ring.slot(2 * L), sb = ring.slot(2 * L + 1);
      WAIT_OR_RETURN_W(bars->phi_ready, cr & 1);
      tc_fence_after();
      mma_k_kh(tS, sQ, sR + ka * HT_BYTES);                                  // phi(Q) phi(K_c)^T, lower 64 keys
      mma_commit(&bars->s_full[0]);
      mma_commit(&bars->free_[ka]);
      mma_k_kh(tS + 64, sQ, sR + kb * HT_BYTES);                             // upper 64 keys
      mma_commit(&bars->s_full[1]);
      mma_commit(&bars->free_[kb]);
      if (un.has_state) WAIT_OR_RETURN_W(bars->full[sa], kp.take(sa));
      WAIT_OR_RETURN_W(bars->stash_done, cr & 1);
      tc_fence_after();
      if (un.has_state) {
        mma_q_state(tO, sQ, 0, sR + sa * HT_BYTES, false);     // phi(Q) S_[c], features 0 .. 63
        mma_commit(&bars->free_[sa]);
      }
      WAIT_OR_RETURN_W(bars->p_ready[0], cs & 1);
      tc_fence_after();
      mma_pv(tO, tS, sR + va * HT_BYTES, un.has_state);
      mma_commit(&bars->free_[va]);
      WAIT_OR_RETURN_W(bars->p_ready[1], cs & 1);
      tc_fence_after();
      mma_pv(tO, tS + 64, sR + vb * HT_BYTES, true);
      mma_commit(&bars->free_[vb]);
      if (un.has_state) {
        WAIT_OR_RETURN_W(bars->full[sb], kp.take(sb));
        tc_fence_after();
        mma_q_state(tO, sQ, 1, sR + sb * HT_BYTES, true);  // features 64 .. 127
        mma_commit(&bars->free_[sb]);
      }
      mma_commit(&bars->o_ready);
      ++cs;
      ++cr;
    }
    ring.base += unit_uses(un);
    ++cu;
  }
  return true;
}

// ------------------------------------------------------------------------------ row threads
__device__ __forceinline__ uint32_t lane_base(int r) { return (uint32_t)((r & ~31) << 16); }
// barrier of the two warps that hold the two column halves of the same 32 rows (ids 4 .. 7), and the same with a vote
__device__ __forceinline__ void pair_sync(int wq) { asm volatile("bar.sync %0, 64;" ::"r"(4 + wq) : "memory"); }
__device__ __forceinline__ bool pair_any(int wq, bool p) { return named_any(4 + wq, 64, p); }
// One value per row, combined over the two column halves: half 1 hands its own over, half 0 combines and hands the
// result back (one word per row).
template <typename F>
__device__ __forceinline__ float pair_combine(float* ex, int wq, int h, float mine, F&& op) {
  if (h) *ex = mine;
  pair_sync(wq);
  if (!h) *ex = mine = op(mine, *ex);
  pair_sync(wq);
  return h ? *ex : mine;
}

// Row threads: thread = query row r and column half h (32 of a step's 64 keys, 64 of the 128 features).  With one
// thread per row the kernel executed 0.37 instructions per clock and scheduler with two row warps on each: every phase
// was a chain of dependent instructions, and nothing else was there to issue (8 x 32/8 heads, T = 32768, w = 512: 6.14 ms
// against 5.92).  The halves agree on the reference maximum once per step by a two-warp barrier that also carries the vote
// for a rescale; sums stay per half until the end.
__device__ bool fwd_rows(const FMaps& tm, const FArgs& a, unsigned char* smem, FBars* bars, uint32_t tmem, int h, int r) {
  const uint32_t tS = tmem + lane_base(r), tO = tmem + 128 + 64 * h + lane_base(r);
  unsigned char* sQ = smem + F_OFF_Q;
  float* ex0 = reinterpret_cast<float*>(smem + F_OFF_EX);
  float* ex = ex0 + r;
  Ring ring;
  int cs = 0, co = 0, cr = 0;                      // score hand-overs per buffer, o_ready completions, residual units
  const int wq = r >> 5;                           // this warp's quarter of the tile's rows
  auto max2 = [](float p, float q) { return fmaxf(p, q); };
  auto add2 = [](float p, float q) { return p + q; };

  TL_DECL(blockIdx.x == 7 && r == 0);
  for (int n = 0;; ++n) {
    const int u = sched_read_all(&bars->sched, n);
    if (u < 0) break;
    const Unit un = make_unit(a, u);
    if (un.t < 0) continue;
    TL(h, 1000 + u);
    const int L = 2 * un.n;
    const int q0 = (un.t - a.off) * TILE;          // first query row of the tile (un.t is its key-space index)

    // ---- window branch: online softmax over the steps of the band ------------------------
    // On the two edge tiles of the band a warp's 32 rows keep whole 32-column chunks, drop whole chunks
    // (no exponentials: zero weights) and mask exactly one chunk, the one their own positions fall into:
    // diagonal tile -> chunks 0 .. wq, oldest tile -> chunks wq .. 3 (of the tile's four; a step has two,
    // one per half).
    float m_ref = -INFINITY, l = 0.f;
#pragma unroll 1
    for (int s = 0; s < L; ++s) {
      const int b = s & 1, chunk = 2 * b + h;
      WAIT_ON(bars->s_full[b], (cs + (s >> 1)) & 1);
#ifdef RATTN_DEBUG_KNOBS
      if (a.debug_wait == 2 && h == 1 && n == 0 && s == 0) bars->abort = 1;      // as if this half's wait had run out
#endif
      TL(h, 200 + s);
      tc_fence_after();
      const bool diag = s < 2, bound = un.c >= 0 && s >= L - 2;
      const bool kept = !(diag && chunk > wq) && !(bound && chunk < wq);
      float x[32];
      tmem_ld32(tS + 64 * b + 32 * h, x);
      tmem_wait_ld();
      tc_fence_before();                           // the other half writes its weights over score columns read here
      if ((diag || bound) && chunk == wq) mask32(x, keep_bits(r, wq, diag, bound));
      const float mx = kept ? max32(x) * a.scale_log2 : -INFINITY;     // scale > 0
      // lazy rescale: the reference maximum only moves when the row maximum grew by more than 2^8
      if (s == 0) {
        m_ref = pair_combine(ex, wq, h, mx, max2);
      } else if (pair_any(wq, mx > m_ref + 8.f)) {
        const float m_new = fmaxf(m_ref, pair_combine(ex, wq, h, mx, max2));
        // the product of the previous step must have completed: its V slot is released then (the one of the
        // last step but one of a residual unit is kept, and reported apart)
        if (un.rla && s == L - 1) WAIT_ON(bars->pv_done, cr & 1);
        else WAIT_ON(bars->free_[ring.slot(pos_v(s - 1, L, un.rla))], ring.phase(pos_v(s - 1, L, un.rla)));
        tc_fence_after();
        const float f = ex2(m_ref - m_new);
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float o[16];
          tmem_ld16(tO + 16 * c, o);
          tmem_wait_ld();
          uint32_t ow[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) ow[e] = __float_as_uint(o[e] * f);
          tmem_st16(tO + 16 * c, ow);
        }
        l *= f;
        m_ref = m_new;
      }
      tc_fence_after();
      TL(h, 300 + s);
      // weights, written back (fp16, two per column) over the score columns
      uint32_t pk[16];
      if (kept) {
        const float2 sc2 = make_float2(a.scale_log2, a.scale_log2), nm2 = make_float2(-m_ref, -m_ref);
        float2 ps0 = make_float2(0.f, 0.f), ps1 = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float2 y = __ffma2_rn(make_float2(x[2 * e], x[2 * e + 1]), sc2, nm2);
          const float2 pp = make_float2(ex2(y.x), ex2(y.y));
          if (e & 1) ps1 = __fadd2_rn(ps1, pp);
          else ps0 = __fadd2_rn(ps0, pp);
          pk[e] = pack_f16(pp.x, pp.y);
        }
        l += (ps0.x + ps0.y) + (ps1.x + ps1.y);
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e) pk[e] = 0u;
      }
      tmem_st16(tS + 64 * b + 16 * h, pk);
      tmem_wait_st();
      tc_fence_before();
#ifdef RATTN_DEBUG_KNOBS
      // failure injection for the time-out test: an arrival that nothing else depends on is left
      // out, so the MMA warp's bounded wait expires and every role takes the abort path
      if (!(a.debug_wait == 1 && n == 0 && s == 0))
#endif
      mbar_arrive(&bars->p_ready[b]);
      TL(h, 400 + s);
    }
    cs += un.n;

    // ---- residual branch, first part: feature maps ------------------------------------------
    // Done right here, while the last P V of the window loop is still running.  Every Q K^T has completed
    // (the commit behind the last scores covers them).  Two neighbouring lanes share a row.  phi(Q) stays
    // without its normalisation: everything that follows is linear in the row, so 1/sum is applied to the
    // accumulator row at the end.
    float inv_q = 1.f;
    if (un.rla) {
      const int row = 32 * wq + 16 * h + ((r & 31) >> 1), ch = r & 1;        // rows of this warp pair
      pair_sync(wq);                               // a rescale in the last step has been read
      unsigned char* sK = smem + F_OFF_RING + ring.slot(2 * L - 4 + (row >> 6)) * HT_BYTES;   // rows 0..63, 64..127 of chunk c
#pragma unroll 1
      for (int k = 0; k < 2; ++k) {
        unsigned char* p = k ? sK + ch * HT_HALF + (row & 63) * 128 : sQ + ch * HALF_BYTES + row * 128;
        const float inv = feature_map_half_row(p, p, row, ch, a.phi, k != 0);
        if (k == 0 && ch == 0) ex0[row] = inv;
      }
      fence_proxy_async_smem();
      mbar_arrive(&bars->phi_ready);
      TL(h, 503);
      pair_sync(wq);
      inv_q = *ex;
      pair_sync(wq);
    }
    l = pair_combine(ex, wq, h, l, add2);

    // ---- park the normalised window output (Section 3.2, first norm) in registers ---------
    WAIT_ON(bars->o_ready, co & 1);
    ++co;
    TL(h, 501);
    tc_fence_after();
    const float inv_l = 1.f / l;
    uint32_t stash[32];
    float ss = 0.f;
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      float o[32];
      tmem_ld32(tO + 32 * c, o);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 32; ++e) ss += o[e] * o[e];
    }
    ss = pair_combine(ex, wq, h, ss, add2);
    const float ms = ss * inv_l * inv_l * (1.f / 128.f) + a.eps;     // mean square of o_swa, plus eps
    const float rs = rsqrtf(ms);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float o[32];
      tmem_ld32(tO + 32 * c, o);
      tmem_wait_ld();
#pragma unroll
      for (int e = 0; e < 16; ++e) stash[16 * c + e] = pack_f16(o[2 * e] * inv_l * rs, o[2 * e + 1] * inv_l * rs);
    }

    // ---- residual branch, second part -------------------------------------------------------
    TL(h, 502);
    float rr = 0.f;
    if (un.rla) {
      tc_fence_before();
      mbar_arrive(&bars->stash_done);
#pragma unroll 1
      for (int b = 0; b < 2; ++b) {
        WAIT_ON(bars->s_full[b], cs & 1);
        tc_fence_after();
        float x[32];
        tmem_ld32(tS + 64 * b + 32 * h, x);
        tmem_wait_ld();
        tc_fence_before();
        pair_sync(wq);                             // both halves have read the columns that the weights overwrite
        tc_fence_after();
        const uint32_t keep = bits_lt(r - 64 * b - 32 * h);            // residual keys of row r in its chunk: j < r
        uint32_t pk[16];
#pragma unroll
        for (int e = 0; e < 16; ++e)
          pk[e] = pack_f16((keep >> (2 * e)) & 1u ? x[2 * e] : 0.f, (keep >> (2 * e + 1)) & 1u ? x[2 * e + 1] : 0.f);
        tmem_st16(tS + 64 * b + 16 * h, pk);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bars->p_ready[b]);
      }
      ++cs;
      ++cr;
      WAIT_ON(bars->o_ready, co & 1);
      ++co;
      tc_fence_after();
      float sr = 0.f;
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        float o[32];
        tmem_ld32(tO + 32 * c, o);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 32; ++e) sr += o[e] * o[e];
      }
      sr = pair_combine(ex, wq, h, sr, add2);
      rr = inv_q * rsqrtf(sr * inv_q * inv_q * (1.f / 128.f) + a.eps);     // o_rla = inv_q * accumulator
    }
    ring.base += unit_uses(un);
    TL(h, 530);

    // ---- Section 3.2: gains, sum; outputs leave through the tile's Q buffer ---------------
    // (every product that reads Q has completed) by TMA: plain 16-byte global stores from row owners keep
    // the load/store unit busy under everything else.  Each column half has its own 64-column box of the
    // buffer, its own barrier and its own storing thread.
    unsigned char* stage = sQ + h * HALF_BYTES;
    auto send = [&](const auto* map, bool last) {
      fence_proxy_async_smem();
      group_sync(h);
      if (r == 0) {
        store_half(map, stage, 64 * h, q0, un.bh_q);
        tma_store_commit();
        tma_store_wait_read();
        if (last) mbar_arrive(&bars->q_free);      // the next unit's Q may come
      }
      if (!last) group_sync(h);
    };
    if (a.o_swa) {
      // training mode: the un-normalised branch outputs (bf16) for the backward
      const float rms_s = ms * rs;                                     // sqrt(mean square + eps)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        uint32_t wv[4];
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&stash[4 * e + k2]));
          wv[k2] = pack_bf16(f.x * rms_s, f.y * rms_s);
        }
        *reinterpret_cast<uint4*>(stage + swz(r, e)) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
      }
      send(&tm.o_swa, false);
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        float x[16];
        if (un.rla) {
          tmem_ld16(tO + 16 * c, x);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) x[e] *= inv_q;
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) x[e] = 0.f;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
          *reinterpret_cast<uint4*>(stage + swz(r, 2 * c + e)) =
              make_uint4(pack_bf16(x[8 * e], x[8 * e + 1]), pack_bf16(x[8 * e + 2], x[8 * e + 3]),
                         pack_bf16(x[8 * e + 4], x[8 * e + 5]), pack_bf16(x[8 * e + 6], x[8 * e + 7]));
      }
      send(&tm.o_rla, false);
    }
    TL(h, 535);
    const float* gs = a.gamma_swa ? a.gamma_swa + (size_t)un.h * 128 + 64 * h : nullptr;
    const float* gr = a.gamma_rla ? a.gamma_rla + (size_t)un.h * 128 + 64 * h : nullptr;
    // The branches on "gains given" and "tile has a residual branch" are taken once, outside the loops.
    auto emit_y = [&](auto has_gains_t, auto has_rla_t) {
      constexpr bool has_gains = decltype(has_gains_t)::value, has_rla = decltype(has_rla_t)::value;
#pragma unroll
      for (int c = 0; c < 4; ++c) {                                    // 16 columns at a time
        float orl[16];
        if constexpr (has_rla) {
          tmem_ld16(tO + 16 * c, orl);
          tmem_wait_ld();
        }
        uint32_t yk[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {                                  // four of them: sixteen outputs and gains at once spill
          const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&stash[8 * c + 2 * e]));
          const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&stash[8 * c + 2 * e + 1]));
          float4 y = make_float4(f0.x, f0.y, f1.x, f1.y);
          if constexpr (has_gains) {
            if (gs) {
              const float4 g = __ldg(reinterpret_cast<const float4*>(gs + 16 * c) + e);
              y.x *= g.x; y.y *= g.y; y.z *= g.z; y.w *= g.w;
            }
          }
          if constexpr (has_rla) {
            float4 x = make_float4(orl[4 * e] * rr, orl[4 * e + 1] * rr, orl[4 * e + 2] * rr, orl[4 * e + 3] * rr);
            if constexpr (has_gains) {
              if (gr) {
                const float4 g = __ldg(reinterpret_cast<const float4*>(gr + 16 * c) + e);
                x.x *= g.x; x.y *= g.y; x.z *= g.z; x.w *= g.w;
              }
            }
            y.x += x.x; y.y += x.y; y.z += x.z; y.w += x.w;
          }
          yk[2 * e] = pack_bf16(y.x, y.y);
          yk[2 * e + 1] = pack_bf16(y.z, y.w);
        }
        *reinterpret_cast<uint4*>(stage + swz(r, 2 * c)) = make_uint4(yk[0], yk[1], yk[2], yk[3]);
        *reinterpret_cast<uint4*>(stage + swz(r, 2 * c + 1)) = make_uint4(yk[4], yk[5], yk[6], yk[7]);
      }
      tc_fence_before();
      mbar_arrive(&bars->o_free);        // last read of the accumulator
    };
    const bool gains = gs != nullptr || gr != nullptr;
    if (gains) {
      if (un.rla) emit_y(std::true_type{}, std::true_type{});
      else emit_y(std::true_type{}, std::false_type{});
    } else {
      if (un.rla) emit_y(std::false_type{}, std::true_type{});
      else emit_y(std::false_type{}, std::false_type{});
    }
    send(&tm.out, true);
    const int t = q0 + r;
    TL(h, 540);
    if (h == 0 && t < a.T && a.lse) a.lse[(size_t)un.bh_q * a.T + t] = (m_ref + log2f(l)) * 0.6931471805599453f;
  }
  if (r == 0) tma_store_wait();          // this thread's stores have completed before the CTA may go
  return *(volatile int*)&bars->abort == 0;
}

__global__ void __launch_bounds__(F_THREADS, 2)
tc_fwd1_kernel(const __grid_constant__ FMaps tm, FArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  FBars* bars = reinterpret_cast<FBars*>(smem + F_OFF_BAR);
  const int tid = threadIdx.x, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");    // the next kernel may be set up in the tail
  if ((smem_u32(smem) & 1023u) != 0) {
    if (tid == 0 && a.status) atomicExch(a.status, 2);
    return;
  }
  if (tid == 0) {
    for (int i = 0; i < F_NS; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->v_full[i], 1);
      mbar_init(&bars->free_[i], 1);
      mbar_init(&bars->v_ready[i], 64);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->p_ready[i], 256);
    }
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->q_free, 2);
    mbar_init(&bars->pv_done, 1);
    mbar_init(&bars->o_ready, 1);
    mbar_init(&bars->stash_done, 256);
    mbar_init(&bars->phi_ready, 256);
    mbar_init(&bars->o_free, 256);
    mbar_init(&bars->drain, 1);
    sched_init(&bars->sched, 256 + 1 + 64);      // row threads, the MMA warp's lane 0, the converter threads
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 8) {
    tmem_alloc(&bars->tmem_base, 256);
    tmem_relinquish();
  }
  if (tid == 288) {
    prefetch_map(&tm.q);
    prefetch_map(&tm.k);
    prefetch_map(&tm.v);
    prefetch_tensormap(&tm.st);
    prefetch_map(&tm.out);
    prefetch_tensormap(&tm.o_swa);
    prefetch_tensormap(&tm.o_rla);
  }
  if (a.wait_first) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (a.clear_status && blockIdx.x == 0 && tid == 0) *a.clear_status = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;

  // Registers follow the work: 256 x 88 + 128 x 64 = 384 x 80, the CTA's allocation.
  bool ok = true;
  if (warp < 8) setmaxnreg_inc<88>();
  else setmaxnreg_dec<64>();
  if (warp < 8) {
    ok = fwd_rows(tm, a, smem, bars, tmem, warp >> 2, tid & 127);
  } else if (warp == 8) {
    ok = fwd_mma(a, smem, bars, tmem);
    if (!ok) {
      mma_commit(&bars->drain);
      for (int it = 0; it < (1 << 16) && !mbar_try_wait(&bars->drain, 0); ++it) {}
    }
  } else if (warp == 9) {
    ok = fwd_loader(tm, a, smem, bars);
    if (!ok && (tid & 31) == 0) sched_close(&bars->sched);
  } else {
    ok = fwd_convert(a, smem, bars, tid - 320);
  }
  if (!ok && a.status) atomicExch(a.status, 1);
  // Not to end before the chunk-state kernel, whether or not this CTA has read a state: what follows on the stream may
  // wait for this kernel alone and read the decode state that the other one leaves.
  if (a.wait_for_states) asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

}  // namespace

#ifdef RATTN_TIMELINE
bool read_timeline_single(unsigned long long* out, int* n) { return tc::read_timeline(out, n); }
#endif

cudaError_t launch_tc_forward_single(const Args& a, cudaStream_t s, bool after_states) {
  FMaps tm;
  if (!make_user_map(&tm.q, a.q, a.T, a.H_q, a.B, a.layout) || !make_user_map(&tm.k, a.k, a.Tk, a.H_kv, a.B, a.kv_layout, 64) ||
      !make_user_map(&tm.v, a.v, a.Tk, a.H_kv, a.B, a.kv_layout, 64) || !make_user_map(&tm.out, a.out, a.T, a.H_q, a.B, a.layout) ||
      !make_state_map(&tm.st, a.chunk_state, a.k, (uint64_t)a.B * a.H_kv * a.n_chunks, 64) ||
      !make_map(&tm.o_swa, a.o_swa ? (const void*)a.o_swa : a.out, a.T, (uint64_t)a.B * a.H_q) ||
      !make_map(&tm.o_rla, a.o_rla ? (const void*)a.o_rla : a.out, a.T, (uint64_t)a.B * a.H_q))
    return cudaErrorInvalidValue;
  int n_sm = 0;
  cudaError_t e = sm_count(&n_sm);
  if (e != cudaSuccess) return e;
  FArgs t;
  t.lse = a.lse;
  t.o_swa = reinterpret_cast<__nv_bfloat16*>(a.o_swa);   // the fp32-sized regions of the workspace hold bf16 here
  t.o_rla = reinterpret_cast<__nv_bfloat16*>(a.o_rla);
  t.gamma_swa = a.gamma_swa; t.gamma_rla = a.gamma_rla; t.status = a.status;
  t.T = a.T; t.w = a.w; t.H_q = a.H_q; t.group = a.group; t.n_chunks = a.n_chunks;
  t.n_qt = (a.T + TILE - 1) / TILE;
  t.n_bh = a.B * a.H_q;
  t.n_units = t.n_qt * t.n_bh;
  t.scale_log2 = a.scale * LOG2E; t.eps = a.eps;
  t.phi = a.phi;
  t.off = a.q_off / TILE;
  t.first_state = a.state_in ? 0 : 1;
  t.seq_lens = a.seq_lens;
  // tiles t with t - w/128 <= 0 read no stored state (a resumed sequence has none: every tile reads one); they come first
  // when the chunk-state kernel leaves many SMs free for them (it runs one CTA per K/V head)
  t.n_stateless = 0;
  const int order = tuning(RATTN_TUNE_UNIT_ORDER);
  const bool stateless_first = order == 1 || (order == 0 && 2 * a.B * a.H_kv <= n_sm);
  if (after_states && !a.state_in && stateless_first) t.n_stateless = a.w / TILE + 1 < t.n_qt ? a.w / TILE + 1 : t.n_qt;
  t.wait_for_states = after_states ? 1 : 0;
  t.wait_first = after_states ? 0 : 1;
  t.state_ready = after_states ? a.state_ready : nullptr;
  t.ascending = (t.state_ready && t.n_stateless > 0) ? 1 : 0;
  t.debug_wait = debug_wait();
  int grid = 2 * n_sm;
  if (tuning(RATTN_TUNE_GRID) > 0 && tuning(RATTN_TUNE_GRID) < grid) grid = tuning(RATTN_TUNE_GRID);
  if (t.n_units < grid) grid = t.n_units;
  // One unit per CTA needs no counter; behind a chunk-state kernel, whose CTAs keep whole SMs for a while, it does: the CTAs
  // that find no room until then would start their units last.
  t.work_counter = (order != 3 && (after_states || t.n_units > 2 * n_sm)) ? a.work_counter : nullptr;
  t.clear_status = after_states ? nullptr : a.clear_status;
  e = allow_smem<tc_fwd1_kernel>(F_SMEM);
  if (e != cudaSuccess) return e;
  {
    KernelTimer kt("tc_fwd", s);
    // Behind a chunk-state kernel this one may begin while that one still runs (its loader waits before the first state
    // load); behind any other it waits right after its set-up.
    e = launch_pdl(tc_fwd1_kernel, dim3((unsigned)grid), dim3(F_THREADS), F_SMEM, s,
                   !after_states || tuning(RATTN_TUNE_OVERLAP), tm, t);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace rattn
