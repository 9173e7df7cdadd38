// Tensor-core forward for bf16, d = 128, window a multiple of 128: the chunk states of the linear
// branch first (tc_state.cu), then the main kernel (tc_fwd1.cu: single query tiles, two CTAs per SM;
// tc_fwd2.cu: pairs of tiles).
//
// Chunk states S_[c] = sum_{c' < c} phi(K_c')^T V_c' (Eq. 2): one CTA per K/V head walks the chunks
// with the sum in TMEM.  The pair kernel reads S_[c] only for c = 2p - w/128 (one stored state serves
// a pair of query tiles), so before it an inference forward stores every second state -- the paper's
// "states stored every m chunks" with m = 2; a training forward stores all of them, because the backward
// reads one per query tile, and so does the single-tile kernel.  When the caller asks for the decode state,
// the chain runs one chunk further (tokens up to T - w, the rest of that chunk masked) and leaves its fp32
// sum there.  The main kernel is launched so that it may start while the chain still runs (programmatic
// dependent launch): its window loops need no state, and it waits for the chain only before its
// first state load.
#include "tc_common.cuh"

namespace rattn {

// How a forward is run.
struct Plan {
  bool chain;        // a chunk-state kernel runs ahead of the main kernel
  bool terms;        // ... as terms formed in parallel and their sums
  bool progress;     // the main kernel takes the states as the chain publishes them
  bool single;       // tc_fwd1.cu instead of tc_fwd2.cu
  bool single_tiles; // tc_fwd2.cu with units of one tile
  int n_steps;       // chunks of the chain
};
static Plan make_plan(const Args& a, int n_sm) {
  Plan p;
  const int n_kt = (a.Tk + tc::TILE - 1) / tc::TILE, n_qt = (a.T + tc::TILE - 1) / tc::TILE, wt = a.w / tc::TILE;
  const bool rla = a.mode == RATTN_MODE_RATTN, want_state = rla && a.state_out != nullptr;
  const int n_kv = a.B * a.H_kv, n_q = a.B * a.H_q;
  // S_[c] for c = 1 .. n_delta: the states some query tile reads (S_[0] is the incoming state, zero
  // for a fresh sequence, where it is never read)
  const int n_delta = rla ? n_kt - 1 - wt : 0;
  p.n_steps = (want_state && (a.Tk > a.w || a.seq_lens)) ? n_delta + 1 : n_delta;
  if (p.n_steps < 0) p.n_steps = 0;
  p.chain = n_delta > 0 || (want_state && (a.Tk > a.w || a.seq_lens)) || (a.state_in && rla);
  const int knob = tuning(RATTN_TUNE_STATE_PROGRESS);
  // Estimates, for which the lines below are drawn: the chain 2.6 us per step, the main kernel 30 ns per query tile and 12 ns
  // per tile and key tile, and no less than 40 us as far as this matters.  (A step with the GPU to itself takes 1.64 us where
  // every state is stored, 1.30 where every second one is, 2.3 where they are published.)  (Fitted on a B200
  // with all of its 148 SMs at work and every window full: short sequences, whose first tiles read less, and ragged batches
  // have less work than this says.)  Where the chain of a long sequence on few heads would outlast the main kernel, its terms
  // are formed in parallel (1 x 8/1 heads, T = 16384, w = 512: 202 -> 113 us).
  const long long chain_ns = 2600ll * p.n_steps;
  const long long work_ns = (long long)n_qt * n_q * (30 + 12 * (wt + 1)), main_ns = work_ns < 40000 ? 40000 : work_ns;
  p.terms = p.chain && a.rdelta && knob == 0 && n_kt >= kMinTermChunks && (long long)n_kv * a.n_chunks <= kMaxForwardTerms &&
            chain_ns > main_ns;
  // The single-tile kernel wins where the window loop is not everything: 1.05 - 1.28 times where measured up to w = 768 (8 x
  // 32/8 heads, T = 4397, w = 128, training: 748 -> 610 us; 4 x 16/16, T = 4096, w = 512: 215 -> 201), in training, where all
  // states are stored and three outputs leave per tile, up to w = 1536; at w = 1408 and 2048 the pair kernel is 8 - 10 % faster
  // in inference.  The lines are drawn at 7 key tiles (w = 896) and, in training, at 12.  It needs every state, in bf16, where
  // of a pair the second tile takes the chunk in between exactly: a chain that outlasts the main kernel by far decides against
  // it (16 heads, T = 16384, w = 128), in inference, where the pair kernel's chain stores half of the states, from 1.2 - 1.4
  // times on (1 x 16/4 heads, T = 6298, w = 768: 203 us against 167; 1 x 16/16, T = 2200, w = 128: 88 against 73; but 1 x 40/8,
  // T = 3541, w = 128, at 1.1: 92 against 116), and the element-wise maps' signed sums feel the rounding (of the output's bound
  // of 2e-2 the last rounding alone takes 1.6e-2 above 4).
  const bool chain_fits = a.training ? 2 * chain_ns <= 3 * main_ns
                                     : 5 * chain_ns <= (wt <= 4 ? 7 : 6) * (work_ns < 16000 ? 16000 : work_ns);
  // Where the pairs all run at once, everything else is over within a unit's time, about 20 us: a chain much
  // longer than that decides, and the pair kernel's is the shorter one (inference) or leaves it less to do at
  // the end (1 x 16/4 heads, T = 2200, w = 512: 47 us as single tiles, 37 as pairs; w = 768, two steps fewer: 42 and 41;
  // training, w = 128: 55 and 50).
  const bool chain_decides = (long long)((n_qt + 1) / 2) * n_q <= n_sm && chain_ns > (a.training ? 36000 : 30000);
  // A head of one tile has no pairs, whatever its window: two tiles per SM instead of one (T = 116, w = 1024, 100 / 160 / 290 / 600
  // tiles: 10.6 / 19.0 / 21.9 / 38.9 us as units of the pair kernel, 9.8 / 10.6 / 10.7 / 24.7 as single tiles; of two tiles a head
  // the two are alike, from four on the pairs are faster).
  p.single = rla && (a.phi == RATTN_PHI_SOFTMAX || !p.chain) && (wt <= (a.training ? 12 : 7) || (!a.training && n_kt == 1)) &&
             (p.terms || (chain_fits && !chain_decides)) &&
             !(p.chain && !a.training && tuning(RATTN_TUNE_STATE_STRIDE) == 2);
  // The pair kernel where there are no more tiles than SMs: a tile of its own per CTA ends sooner.  (With more, the second
  // wave costs more than that: 32 heads, T = 1000, w = 256, window only: 26.7 us as 256 tiles, 18.6 as 128 pairs.)
  p.single_tiles = !p.single && !rla && (long long)n_qt * n_q <= n_sm;
  // The main kernel can take the chunk states as the chain publishes them instead of waiting for the whole
  // chain.  That pays where the chain is long and leaves most SMs to the main kernel, which otherwise runs out
  // of work that needs no state (2 x 32/8 heads, T = 8192, w = 512: 422 -> 357 us; 1 x 32/8, T = 2048: 64 -> 58); elsewhere
  // publishing only slows the chain.  With wide windows the units without a state are many and heavy already, and taking
  // the units in sequence order (light ones first) costs more at the tail than the earlier start gains.
  const bool few = 4 * n_kv <= n_sm && n_kt >= 48 && wt <= (p.single ? 8 : 4);
  const bool fewer = p.single && 8 * n_kv <= n_sm && n_kt >= 16;
  p.progress = p.chain && !p.terms && a.state_ready && (knob == 1 || (knob == 0 && (few || fewer)));
  return p;
}
bool tc_forward_clears_status(const Args& a) {
  int n_sm = 0;
  if (sm_count(&n_sm) != cudaSuccess) return false;
  const Plan p = make_plan(a, n_sm);
  const int n_qt = (a.T + tc::TILE - 1) / tc::TILE, per = p.single || p.single_tiles ? 1 : 2;
  return !p.chain && (long long)((n_qt + per - 1) / per) * a.B * a.H_q <= (p.single ? 2 : 1) * n_sm;
}

cudaError_t launch_tc_forward(const Args& a, cudaStream_t s) {
  int n_sm = 0;
  cudaError_t e = sm_count(&n_sm);
  if (e != cudaSuccess) return e;
  const Plan p = make_plan(a, n_sm);
  const int wt = a.w / tc::TILE, off = a.q_off / tc::TILE;       // a resumed sequence carries its w-token history in front
  const int n_kv = a.B * a.H_kv;
  const bool want_state = a.mode == RATTN_MODE_RATTN && a.state_out != nullptr;
  if (want_state && a.Tk <= a.w && !a.seq_lens && !a.zero_state) {
    // nothing has left the window yet
    e = cudaMemsetAsync(a.state_out, 0, sizeof(float) * (size_t)n_kv * 128 * 128, s);
    if (e != cudaSuccess) return e;
  }
  if (p.chain) {
    StateLaunch L;
    L.x = a.k; L.y = a.v; L.out = a.chunk_state;
    L.x_heads = L.y_heads = a.H_kv; L.x_layout = L.y_layout = a.kv_layout;
    L.T = a.Tk; L.n_kv = n_kv; L.group = 1; L.n_chunks = a.n_chunks;
    L.n_steps = p.n_steps; L.first = 0; L.dir = +1; L.out_first = 1;
    // the pair kernel reads S_[c] for c = off + 2p - wt only
    const bool every = a.training || p.single || tuning(RATTN_TUNE_STATE_STRIDE) == 1;
    L.store_every = every ? 1 : 2;
    L.store_phase = every ? 0 : ((off + wt) & 1);
    L.handoff = want_state ? 1 : 0;
    L.w = a.w;
    L.final_out = want_state ? a.state_out : nullptr;
    L.state_in = a.state_in;
    L.seq_lens = a.seq_lens; L.kv_per_batch = a.H_kv;
    L.phi = a.phi;
    L.status = a.status; L.name = "tc_state_fwd";
    L.ready = p.progress ? a.state_ready : nullptr;
    L.delta = p.terms ? a.rdelta : nullptr;
    L.h_split = 1;
    L.after_independent = false;
    // Behind the call's own copies (gather, ring hand-off) the chain is set up under them where it has few heads.  Resumed
    // chunks in full order and so: 1 x 40/8 heads, T = 300, w = 256 26.6 and 24.6 us; w = 512: 2 x 32/8, T = 2048 126.8 and 121.9,
    // 4 x 32/8, T = 1024 120.5 and 115.3.  Heads are counted and not CTAs, of which parallel terms have one per head and step:
    // 1 x 8/1, T = 8192 63.2 and 60.2, 1 x 16/4 127.4 and 122.5.  (The line lies where the chain's CTAs lost when they did not yet
    // come in pairs, 5 x 32/8, T = 1024 139.8 and 144.9; as pairs they gain beyond it too, 139.1 and 136.1, 8 x 32/8 217.3 and
    // 214.1.)
    L.wait_first = a.kernel_ahead && 4 * n_kv <= n_sm;
    e = launch_tc_states(L, s);
    if (e != cudaSuccess) return e;
  }
  Args m = a;
  m.single_tiles = p.single_tiles;
  if (!p.progress) m.state_ready = nullptr;          // the main kernel waits for the whole chain instead
  return p.single ? launch_tc_forward_single(m, s, p.chain) : launch_tc_forward_main(m, s, p.chain);
}

#ifdef RATTN_TIMELINE
bool read_timeline_single(unsigned long long* out, int* n);
bool read_timeline_pair(unsigned long long* out, int* n);
#endif

}  // namespace rattn

#ifdef RATTN_TIMELINE
// Records of the forward kernel that has run since the last call; how many query tiles its units have (0: no record).
extern "C" int rattn_timeline_read(unsigned long long* out, int* n) {
  return rattn::read_timeline_single(out, n) ? 1 : rattn::read_timeline_pair(out, n) ? 2 : 0;
}
#endif
