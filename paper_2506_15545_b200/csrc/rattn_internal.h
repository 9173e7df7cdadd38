// Internal declarations shared by the translation units of librattn.so.
// Nothing here is part of the public ABI (include/rattn.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <utility>

#include "rattn.h"

namespace rattn {

// Byte offsets inside the caller's workspace.  Every region is 256-byte aligned; a region the
// call's mode and flags do not need has offset kAbsent and takes no room.
struct WorkspaceLayout {
  size_t status;        // 256 bytes; word 0 = device status, word 1 = detail code; behind it, on the tensor-core
                        // path with a linear branch, one progress word per K/V head (status_bytes in all)
  size_t status_bytes;  // what a forward clears before its kernels
  size_t lse;           // fp32 [B,H_q,T]      log-sum-exp of the SWA logits (natural log)
  size_t o_swa;         // fp32 [B,H_q,T,d]    un-normalised SWA branch output (bf16 on the tensor-core path)
  size_t o_rla;         // fp32 [B,H_q,T,d]    un-normalised RLA branch output (likewise)
  size_t do_swa;        // fp32 [B,H_q,T,d]    backward scratch (the tensor-core path keeps bf16 there)
  size_t do_rla;        // fp32 [B,H_q,T,d]    backward scratch (likewise)
  size_t delta;         // fp32 [B,H_q,T]      backward scratch
  size_t chunk_state;   // bf16 [B,H_kv,n_chunks,d,d]  exclusive prefix over chunks
  size_t rstate;        // bf16 [B,H_kv,n_chunks,d,d]  backward: suffix sums of phi(Q)^T g_r
  size_t gstate;        // fp32 [B,H_kv,ceil(T/64),d,d]  portable training path: sums of phi(K)^T V over the chunks before
  size_t grstate;       // fp32 [B,H_kv,ceil(T/64),d,d]  ... and of phi(Q)^T g_r over the chunks from this one on
  size_t rdelta;        // fp32 [B,H_kv,n_chunks,head_split,d,d]  backward: their terms, where these are formed in parallel
  size_t kvpart;        // fp32 [B,H_kv,n_chunks,head_split,2,d,d]  backward: partial dK, dV of a share of a group's heads
  size_t lse2p;         // fp32 [B*H_q, n_chunks*128]  backward: lse * log2(e), +inf in the padding
  size_t dscp;          // fp32 [B*H_q, n_chunks*128]  backward: D_t * scale, 0 in the padding
  size_t k_ext;         // I/O type [B,H_kv,w+T,d]  chunked prefill: history + chunk keys, in time order
  size_t v_ext;         //                          ... values
  size_t total;
  int n_chunks;         // ceil(T / 128)
};

// The reverse states of the backward are a running sum over the query tiles of each K/V head.  Walked by one CTA per
// head (tc_state.cu) the chain takes a microsecond per tile and query head of the group on as few SMs as there are
// heads.  Up to this many terms (64 KB each; twice as many of long chains) they are formed by a CTA each and summed by a
// second kernel instead; with more of them the chain runs beside the dq kernel, which hides it.
constexpr long long kMaxParallelTerms = 512;

// The forward's chain, one CTA per K/V head, takes 2.6 us per chunk when every state is stored.  For long sequences of few
// heads that is longer than everything else; the workspace then has room for the terms, so that they too can be formed in
// parallel.  (From 64 chunks on: shorter chains hide under the main kernel.  Up to 384 terms: with more of them, 80 ns each,
// the chain whose states the main kernel takes as they appear is over sooner: 1 x 16/16 heads, T = 8192, w = 512, 960 terms:
// 170 us against 119; 1 x 32/8, w = 128, 496: 165 against 155; 1 x 16/4, 240: 92 against 115.)
constexpr int kMinTermChunks = 64;
constexpr long long kMaxForwardTerms = 384;

// Grouped heads: where the (key tile, K/V head) items of the dk/dv kernel leave most of the GPU idle, an item is split
// over the group's query heads, whose contributions (fp32) a second kernel adds.  The largest divisor of the group for
// which the parts still run at once, one per SM of a B200: 148 is written in because the workspace's layout depends on
// this and is computed without a device.
inline int head_split(long long items, int group) {
  for (int n = group; n > 1; --n)
    if (group % n == 0 && items * n <= 148) return n;
  return 1;
}

// Offset of a region the call does not use.
constexpr size_t kAbsent = ~(size_t)0;

// T: query rows of the call; history: 1 when the call resumes a sequence (chunked prefill)
WorkspaceLayout workspace_layout(int B, int H_q, int H_kv, int T, int d, int w, int dtype, int mode,
                                 unsigned flags, int history = 0);

// Resolved arguments handed to the kernel launchers (all device pointers).
struct Args {
  const void* q;
  const void* k;
  const void* v;
  void* out;
  int B, H_q, H_kv, T, d, w;   // w already replaced by T for FULL_CAUSAL
  // Chunked prefill: k, v then point at the history (the w tokens before the chunk, in time
  // order) followed by the chunk, Tk = w + T rows per head, and query row t sits at key
  // position t + q_off (q_off = w); state_in holds the sum over the tokens before the history.
  // A fresh sequence has Tk = T, q_off = 0, state_in = null.
  int Tk, q_off;
  const float* state_in;
  const int* seq_lens;         // optional device [B]: valid tokens of each batch entry (fresh sequences only)
  int pos_shift;               // sequence position of key row 0 (pos0 - w for a resumed sequence, else 0)
  int group;                   // H_q / H_kv
  int dtype, mode;
  unsigned flags;              // rattn_params.flags
  int layout;                  // rattn_layout of q, out, dout, dq (and of k, v, dk, dv unless kv_layout says otherwise)
  int kv_layout;               // layout of the k, v the kernels read: dense when they are the gathered history + chunk
  int phi;                     // rattn_feature_map
  float scale, eps;
  const float* gamma_swa;
  const float* gamma_rla;
  // residuals (may be null in inference mode)
  float* lse;
  float* o_swa;
  float* o_rla;
  // tensor-path scratch
  __nv_bfloat16* chunk_state;
  __nv_bfloat16* rstate;
  float* gstate;               // portable path, training: see WorkspaceLayout (null: residual sums in quadratic form)
  float* grstate;
  float* rdelta;
  float* kvpart;
  float* lse2p;
  float* dscp;
  int n_chunks;
  int* status;                 // device status word (may be null when no workspace)
  int* clear_status;           // the status word, where no kernel ahead of the forward's first one has cleared it
  bool kernel_ahead;           // the last thing put on the stream is a kernel of this call that signals its successor
  bool single_tiles;           // the pair kernel's work units are single query tiles
  int* work_counter;           // the forward's work counter, zero at launch (null: units are dealt round-robin);
                               // the backward's two kernels use the two words behind it
  int* state_ready;            // [B*H_kv], zero at launch: chunk states the chunk-state kernel has stored so far
                               // (null: the main kernel waits for that whole kernel instead)
  bool training;               // the backward will read every chunk state
  // hand-off
  float* state_out;
  void* k_ring_out;
  void* v_ring_out;
  bool zero_state;             // the ring hand-off also clears state_out (no token has left the window)
  // backward
  const void* dout;
  void* dq;
  void* dk;
  void* dv;
  float* dgamma_swa;
  float* dgamma_rla;
  float* do_swa;               // fp32 [B,H_q,T,d]  gradient w.r.t. the SWA branch output
  float* do_rla;               // fp32 [B,H_q,T,d]  gradient w.r.t. the RLA branch output
  float* delta;                // fp32 [B,H_q,T]    do_swa . o_swa per row
};

// Launchers; each returns the cudaError_t of its launches (cudaGetLastError).
cudaError_t launch_generic_forward(const Args& a, cudaStream_t s);
cudaError_t launch_generic_backward(const Args& a, cudaStream_t s);
cudaError_t launch_decode(const Args& a, void* k_ring, void* v_ring, float* state, int pos, const int* pos_dev,
                          cudaStream_t s);
// The TMA-staged decode step (bf16, d = 128, w a multiple of 64, groups of up to 8 heads) and
// its status word (RATTN_ERR_TIMEOUT once a bounded wait has expired; reading clears it).
bool decode_tc_applies(const Args& a, int w);
cudaError_t launch_decode_tc(const Args& a, void* k_ring, void* v_ring, float* state, int pos, const int* pos_dev,
                             cudaStream_t s);
int decode_tc_status(cudaStream_t s, cudaError_t* err);
// prefill -> decode hand-off: the rings, and (state_too) the state by the portable kernel.  `clear` (clear_ints of them):
// words to set to zero beside it
cudaError_t launch_handoff(const Args& a, cudaStream_t s, bool state_too, int* clear = nullptr, int clear_ints = 0);
cudaError_t launch_tc_forward(const Args& a, cudaStream_t s);        // chunk states, then the main kernel
bool tc_forward_clears_status(const Args& a);   // one kernel, one unit per CTA: only Args::clear_status has to be set
// after_states: a chunk-state kernel was launched just before on the same stream
cudaError_t launch_tc_forward_main(const Args& a, cudaStream_t s, bool after_states);     // pairs of query tiles (tc_fwd2.cu)
cudaError_t launch_tc_forward_single(const Args& a, cudaStream_t s, bool after_states);   // single tiles (tc_fwd1.cu)
// Running sums of phi(X_c)^T Y_c over the chunks first, first+dir, ... (n_steps of them) for every
// K/V head (tc_state.cu).  The sum after step s goes, as bf16, to matrix out_first + dir*s of the
// head when that index is congruent to store_phase modulo store_every.  With `handoff` the chain
// is the forward's and also yields the decode state: per head it walks ceil((len - w) / 128) chunks
// (len = T, or the batch entry's own length), tokens at positions >= len - w contribute nothing,
// and the final sum goes to final_out in fp32.
struct StateLaunch {
  const void* x;            // [n_kv * group, T, 128] bf16, mapped through phi
  const void* y;            // [n_kv * group, T, 128] bf16
  // x and y as the caller's tensors: heads per batch entry and head layout (rattn_layout); 0 heads = a dense
  // internal tensor of n_kv * group matrices
  int x_heads, x_layout, y_heads, y_layout;
  void* out;                // [n_kv * n_chunks, 128, 128] bf16
  int T, n_kv, group, n_chunks;
  int n_steps, first, dir, out_first;
  int store_every, store_phase;
  int handoff;              // 1: the chain ends with the decode state (tokens before len - w, len = T or the
  int w;                    //    entry's own length), left in final_out; the step count follows the length
  float* final_out;
  const float* state_in;    // optional fp32 [n_kv,128,128]: the sum starts from it and matrix 0 holds it
  const int* seq_lens;      // optional [n_kv / kv_per_batch]: valid rows of each batch entry
  int kv_per_batch;
  int phi;                  // rattn_feature_map applied to x
  int* status;
  int* ready;               // optional [n_kv] (forward chain): matrices stored so far, published after each store
  float* delta;             // optional fp32 scratch, n_kv * n_steps * h_split matrices: the terms are formed in parallel
                            // and summed by a second kernel
  int h_split;              // ... each by this many CTAs, a share of the group's heads each
  bool wait_first;          // the kernel before on the stream signals its successor: this one is set up under it, and waits
  bool after_independent;   // the kernel before on the stream neither feeds this one nor is fed by it: they may overlap
  const char* name;         // label of the timing record
};
cudaError_t launch_tc_states(const StateLaunch& L, cudaStream_t s);
cudaError_t launch_tc_backward(const Args& a, cudaStream_t s);
// chunked prefill: k_ext/v_ext[b,hk] = the ring's tokens pos0-w .. pos0-1 in time order, then the chunk
cudaError_t launch_gather_history(const Args& a, const void* k_chunk, const void* v_chunk, const void* k_ring,
                                  const void* v_ring, void* k_ext, void* v_ext, void* k_ring_out, void* v_ring_out, int pos0,
                                  int* clear, int clear_ints, cudaStream_t s);

int debug_wait();                    // always 0 outside the debug build
int tuning(int knob);                       // current value of a rattn_knob
void count_launches(int n);
void set_last_cuda_error(int cuda_error);   // what rattn_last_cuda_error() reports for this thread

// Multiprocessors of the current device, asked of the driver once per device.
cudaError_t sm_count(int* n_sm);
constexpr int kMaxDevices = 64;
// Lets the kernel use `bytes` of dynamic shared memory on the current device.  The driver is called only when a
// device meets a larger size than before: as a call per launch it cost small launches a microsecond of host time.
template <auto Kernel>
cudaError_t allow_smem(int bytes) {
  static std::atomic<int> granted[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (granted[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
  static std::mutex mu;                    // of two threads the one with the larger size must come last
  std::lock_guard<std::mutex> lk(mu);
  if (granted[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) granted[dev].store(bytes, std::memory_order_relaxed);
  return e;
}

// Launch with or without programmatic stream serialisation: with it the kernel may be set up while the one ahead of it on
// the stream still runs, and has to wait for that one itself (griddepcontrol.wait) before it reads or overwrites anything
// the other uses -- and in any case before it ends, so that whatever follows may rely on both.
// cluster > 1: in clusters of that many CTAs, of which the grid is a multiple.
template <typename... P, typename... A>
cudaError_t launch_pdl_cluster(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool overlap, int cluster,
                               A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool overlap, A&&... args) {
  return launch_pdl_cluster(kernel, grid, block, smem, s, overlap, 1, std::forward<A>(args)...);
}

// Records a CUDA event pair around one kernel launch on its stream while per-kernel
// timing is enabled (rattn_timing_enable); free otherwise.
class KernelTimer {
 public:
  KernelTimer(const char* name, cudaStream_t s);
  ~KernelTimer();
 private:
  cudaStream_t stream_;
  int slot_;
};

}  // namespace rattn
