// Middle of the decode step in ONE launch (paper Section 2.3, steps 8-10): finish the joint
// softmax reductions of every sequence from the per-CTA partials of the logits kernel, select the
// token (argmax or Gumbel-max sample, or the caller's forced code; a sequence may sit out), apply the online LZW update,
// and build the work list of new codebook entries for the hyper-encoder pass that follows.
// One block per sequence: its four warps merge the partials, the first one does the rest, and the block
// that finishes last compacts the work list from the records that all of them left.
//
// Latency is all that counts here (a chain of dependent loads between two streams of weights): as one
// block of 32 warps the kernel pulled the partials of the whole batch (148 per row, 32 bytes each)
// through one SM and took 7.8 us at 8 sequences, 13 at 32 and 23 at 90; its 42 KB of shared memory also
// kept it from being resident before the logits kernel had ended.
#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_lzw_dev.cuh"
#include "z2z_sm100.cuh"

namespace z2z {

namespace {

constexpr int kUpdateThreads = 128;         // also the most sequences a fused step takes

// What a block leaves for the last one: entry number + 1 (0: none), base tokens of the entry, hypertokens
// of the sequence after the step, then the entry's tokens.
struct StepRecord { int created, len, n, pad, tok[kMaxM]; };
static_assert(sizeof(StepRecord) <= 64, "64 bytes per sequence are set aside");

__device__ __forceinline__ RowRed shfl_xor_red(const RowRed& r, int off) {
  RowRed o;
  o.m = __shfl_xor_sync(0xffffffffu, r.m, off);
  o.s = __shfl_xor_sync(0xffffffffu, r.s, off);
  o.idx = __shfl_xor_sync(0xffffffffu, r.idx, off);
  o.gm = __shfl_xor_sync(0xffffffffu, r.gm, off);
  o.gidx = __shfl_xor_sync(0xffffffffu, r.gidx, off);
  return o;
}

}  // namespace

__global__ void __launch_bounds__(kUpdateThreads) k_decode_update(CbView cb, DecodeUpdateArgs a, EntryList el) {
  __shared__ RowRed s_red[kUpdateThreads / 32];
  __shared__ int s_warp[kUpdateThreads / 32], s_last;
  sm100::pdl_trigger();
  sm100::pdl_wait();               // the logits partials and the codebook state come from earlier kernels
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = blockIdx.x;
  LzwPrev state{};
  if (warp == 0) state = warp_lzw_load(cb, b);               // independent of the selection: loaded ahead of it
  // ---- merge the partial reductions of hidden row b
  const LogitPartial* lp = a.lpart + (size_t)b * a.part_stride;
  RowRed red; red.init();
  for (int g = tid; g < a.part_count; g += kUpdateThreads) red.merge(load_partial(lp + g));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) red.merge(shfl_xor_red(red, off));
  if (lane == 0) s_red[warp] = red;
  __syncthreads();
  StepRecord* rec = reinterpret_cast<StepRecord*>(reinterpret_cast<char*>(a.records) + (size_t)b * 64);
  if (warp == 0) {
    red = s_red[0];
#pragma unroll
    for (int w = 1; w < kUpdateThreads / 32; ++w) red.merge(s_red[w]);
    const int amax = red.idx == 0x7fffffff ? -1 : red.idx;
    const int smp = red.gidx == 0x7fffffff ? -1 : red.gidx;
    const int sel = a.select == Z2Z_SELECT_GUMBEL ? smp : amax;
    int code = a.forced ? a.forced[b] : sel;
    if (code == Z2Z_CODE_SELECTED) code = sel;
    const bool sits_out = a.forced && code == Z2Z_CODE_NONE;   // a finished sequence of the batch
    if (lane == 0) {
      if (a.lse) a.lse[b] = red.m + logf(red.s);
      if (a.selected) a.selected[b] = sel;
      a.next_codes[b] = code;
    }
    // ---- online LZW update with the applied code
    int new_tok = -1;
    const int created = sits_out ? -1 : warp_lzw_step(cb, b, code, state, &new_tok);
    if (lane < cb.M) rec->tok[lane] = new_tok;
    if (lane == 0) {
      if (a.new_entry) a.new_entry[b] = created;
      rec->created = created + 1;
      rec->len = created >= 0 ? state.plen + 1 : 0;
      rec->n = state.n + (created >= 0 ? 1 : 0);
    }
    __threadfence();                                         // the record is out before the block counts as done
    __syncwarp();
    if (lane == 0) s_last = atomicInc(a.done, gridDim.x - 1) == gridDim.x - 1;     // (returns to 0 by itself)
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // ---- the last block: compact the new entries into the encoder's work list (exclusive scan over
  // sequences): an entry's slot in the list, and the first of the PACKED rows that its base tokens
  // take (the tensor-core pass keeps no padding rows).  Both sums travel in one word: entries in the
  // low half, rows in the high half (at most 128 entries of at most 8 rows).
  const StepRecord* mine_rec = reinterpret_cast<const StepRecord*>(reinterpret_cast<const char*>(a.records) + (size_t)tid * 64);
  int4 head = make_int4(0, 0, 0, 0);
  int emb[2] = {0, 0};
  int tok[kMaxM];
#pragma unroll
  for (int i = 0; i < kMaxM; ++i) tok[i] = -1;
  if (tid < cb.B) {
    emb[0] = cb.n_emb[tid]; emb[1] = cb.n_emb[cb.B + tid];
    head = __ldcg(reinterpret_cast<const int4*>(mine_rec));
    const int4 t0 = __ldcg(reinterpret_cast<const int4*>(mine_rec) + 1), t1 = __ldcg(reinterpret_cast<const int4*>(mine_rec) + 2);
    tok[0] = t0.x; tok[1] = t0.y; tok[2] = t0.z; tok[3] = t0.w;
    tok[4] = t1.x; tok[5] = t1.y; tok[6] = t1.z; tok[7] = t1.w;
  }
  const int mine = head.x, flag = mine > 0 ? 1 : 0, my_len = flag ? head.y : 0;
  const int val = flag | (my_len << 16);
  int incl = val;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kUpdateThreads / 32; ++w) {
    if (w < warp) before += s_warp[w];
    all += s_warp[w];
  }
  const int excl_both = incl - val + before;
  const int excl = excl_both & 0xffff, row0 = excl_both >> 16;
  const int total = all & 0xffff, total_rows = all >> 16;
  if (tid < cb.B) el.off[tid] = excl;
  if (tid == 0) {
    el.off[cb.B] = total; el.off[cb.B + 1] = total < el.chunk ? total : el.chunk;
    el.row_off[cb.B] = total_rows;                 // the pass that follows is sized for B entries
  }
  if (flag && excl < el.chunk) {
    el.seq[excl] = tid; el.idx[excl] = mine - 1;
    el.len[excl] = my_len;
    el.row_off[excl] = row0;
#pragma unroll
    for (int i = 0; i < kMaxM; ++i) {
      if (i >= cb.M) break;
      el.tok[(size_t)excl * cb.M + i] = tok[i];
      if (i < my_len) { el.row_src[row0 + i] = excl * cb.M + i; el.row_tok[row0 + i] = tok[i]; }
    }
  }
  for (int e = total + tid; e < el.chunk && e < cb.B; e += kUpdateThreads) {
    el.seq[e] = -1; el.idx[e] = 0; el.len[e] = 0; el.row_off[e] = total_rows;
    for (int i = 0; i < cb.M; ++i) el.tok[(size_t)e * cb.M + i] = -1;
  }
  // both caches will hold every entry once the encoder pass that follows has run, unless a bounded call left some out
  int full = 1;
  if (tid < cb.B) {
    const int n = head.z;
    if (emb[0] >= 0) cb.n_emb[tid] = n;
    if (emb[1] >= 0) cb.n_emb[cb.B + tid] = n;
    full = n >= cb.cap && mine == 0;             // full already when this step began: it created nothing
  }
  // Once every codebook is full no step creates an entry any more.  The host learns it through a
  // word in its own memory and stops launching the hyper-encoder pass (the session number guards
  // against a late store from before a reset).  The word is only written by a step that found every
  // codebook full on entry: the step that creates the last entry still needs its encoder pass, and
  // the host may read the word at any time after this kernel was enqueued.
  if (a.frozen_flag) {
    const int all_full = __syncthreads_and(full);
    if (all_full && tid == 0) *reinterpret_cast<volatile int*>(a.frozen_flag) = a.epoch;
  }
}

cudaError_t launch_decode_update(const CbView& cb, const DecodeUpdateArgs& a, const EntryList& el,
                                 cudaStream_t s) {
  if (cb.B > kUpdateThreads) return cudaErrorInvalidValue;
  return launch_pdl(k_decode_update, dim3(cb.B), dim3(kUpdateThreads), 0, s, cb, a, el);
}

}  // namespace z2z
