// Weight-streaming skinny GEMM on tcgen05 tensor cores, for the HBM-bound decode regime.
//
//   D[r, j] = sum_k A[r, k] * W[j, k]      A: activation rows (bf16, K-major), few
//                                          W: weight rows streamed once from HBM (bf16, K-major)
//
// One persistent CTA per SM.  Warp 0 issues TMA loads into a ring of shared-memory stages, warp 1
// issues tcgen05.mma (fp32 accumulators in tensor memory, double buffered), warps 2-5 (logits: 2-13)
// drain accumulators.  Two kernels share the ring and its barriers:
//   * hyper-encoder linear layers (k_stream_gemm): a tile of 128 weight rows is the MMA's M
//     operand, the packed activation rows (hi and lo part of a row in adjacent operand rows) its
//     N operand, as wide as the rows that exist; work is cut stream-K style, every CTA gets the
//     same number of (tile, k-step) units and adds its accumulators into one fp32 result matrix
//     with reductions in global memory (sums of a few partial tiles in arrival order; where the bits
//     must not depend on it, two matrices of at most two partials each);
//   * joint logits for 33 .. 128 hidden rows of a batch (k_stream_logits; paper Section 2.3 steps 7-9):
//     the hidden rows are the 128-row M operand, tiles run over W_U and then over the visible
//     rows of each sequence's U_h; the epilogue keeps max / sum-exp / argmax / best perturbed
//     score per hidden row in registers, so the logits are never written.  Only the hidden rows
//     that exist are loaded: the MMA also reads the shared memory behind them, which only feeds
//     accumulator rows nobody reads (rows of D depend on the same rows of A only).
#include <mutex>
#include <unordered_map>

#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_sm100.cuh"
#include "z2z_stream.h"

namespace z2z {
using namespace sm100;

namespace {

constexpr int kThreads = 192;
// The logits kernel drains with twelve warps, three per tensor-memory lane quarter that take every third 32 columns: a
// sampled column costs its row some 30 instructions, and four warps, of which a batch of 43 rows keeps two busy, take
// longer than the weights (V = 128256, d = 4096, 128 rows: sampled with 4 / 8 / 12 warps 276 / 214 / 199 us, argmax 180).
constexpr int kLogitEpiWarps = 12;
constexpr int kLogitEpiGroups = kLogitEpiWarps / 4;
constexpr int kLogitThreads = 64 + 32 * kLogitEpiWarps;

struct Ctrl {                            // at most 512 bytes of shared memory
  unsigned long long full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2], pref_ready;
  uint32_t tmem_base;
  int abort;
};

__host__ __device__ constexpr int tmem_cols(int nt) {
  return 2 * nt <= 32 ? 32 : (2 * nt <= 64 ? 64 : (2 * nt <= 128 ? 128 : (2 * nt <= 256 ? 256 : 512)));
}

// A job of the logits kernel: weight rows [wrow, wrow + nrows) of tensor wmap (0: W_U, 1: U_h).
struct Job {
  int wmap, wrow;
  int col0, nvalid, owner, k0;           // first column id, valid rows, owning sequence, first entry
  int nrows;                             // the MMA's N, a multiple of kLogitGran
  int kb;                                // k-blocks of 64 columns per stage
  int group;                             // >= 0: only this group of 8 hidden rows is loaded
};

// ---- logits schedule ----------------------------------------------------------------------------
// Columns are dealt in granules of kLogitGran rows: every CTA takes an even share of the granules of W_U, and then one
// of those of the visible rows of each sequence's U_h.  (One share of both in a row gives some CTAs nothing but
// hypertokens, whose jobs are short and cost more per granule: V = 128256, d = 4096, 90 sequences of 29 hypertokens
// 385 us, even shares 190.)  With fewer than kLogitEvenGrans granules of W_U per CTA it is their jobs that would get
// short, with all hidden rows each: there it is one share of both in a row (d = 3072, 149 hypertokens each, even shares
// and one: V = 6020, 54 rows 38 and 33 us, V = 12000 43 and 37; V = 17000, 128 rows 54 and 61).  A job is a run of up to
// kLogitNT / kLogitGran granules inside one segment (W_U, or one sequence).
constexpr int kLogitEvenGrans = 3;
constexpr int kNoGroup = 254, kManyGroups = 255;       // a sequence without a row; one with rows in several groups of 8
struct LogitSched {
  const StreamLogitsParams& p;
  const int* pref;       // shared: prefix of per-sequence granule counts, [B + 1]
  const uint8_t* groups; // shared, with row_seq: the group of 8 hidden rows that holds all rows of a sequence, [B]
  int u, u1;
  bool hyper;
  // (pref has to be there unless the shares are even)
  __device__ LogitSched(const StreamLogitsParams& pp, const int* s_pref) : p(pp), pref(s_pref), groups(nullptr), hyper(false) {
    if (p.la.row_seq) groups = reinterpret_cast<const uint8_t*>(pref + p.cb.B + 1);
    const int ns = n_static(p);
    if (even(p)) { share(ns); return; }
    share(ns + pref[p.cb.B]);
    u = u < ns ? u : ns;
    u1 = u1 < ns ? u1 : ns;
  }
  static __device__ int n_static(const StreamLogitsParams& p) { return (p.cb.V + kLogitGran - 1) / kLogitGran; }
  static __device__ bool even(const StreamLogitsParams& p) { return n_static(p) >= kLogitEvenGrans * (int)gridDim.x; }
  __device__ void share(int total) {
    const int G = gridDim.x, c = blockIdx.x;
    u = (int)((long long)c * total / G);
    u1 = (int)((long long)(c + 1) * total / G);
  }
  __device__ void begin_hyper() {                    // (pref is there by now)
    hyper = true;
    if (even(p)) { share(pref[p.cb.B]); return; }
    const int ns = n_static(p);
    share(ns + pref[p.cb.B]);
    u = u < ns ? 0 : u - ns;
    u1 = u1 < ns ? 0 : u1 - ns;
  }
  __device__ bool next(Job& j) {
    if (u >= u1) return false;
    int remaining, total_rows, g0;
    if (!hyper) {
      g0 = u; remaining = u1 - u; total_rows = p.cb.V;
      j.wmap = 0; j.wrow = g0 * kLogitGran; j.col0 = g0 * kLogitGran; j.owner = -1; j.k0 = 0;
    } else {
      int lo = 0, hi = p.cb.B - 1;                 // last b with pref[b] <= u
      while (lo < hi) { int mid = (lo + hi + 1) >> 1; if (pref[mid] <= u) lo = mid; else hi = mid - 1; }
      g0 = u - pref[lo]; remaining = pref[lo + 1] - pref[lo] - g0; total_rows = p.cb.n[lo];
      j.owner = lo; j.k0 = g0 * kLogitGran;
      j.wmap = 1; j.wrow = lo * p.cb.cap + j.k0; j.col0 = p.cb.V + j.k0;
    }
    int ng = kLogitNT / kLogitGran;
    if (remaining < ng) ng = remaining;
    if (u1 - u < ng) ng = u1 - u;
    j.nrows = ng * kLogitGran;
    j.nvalid = total_rows - g0 * kLogitGran < j.nrows ? total_rows - g0 * kLogitGran : j.nrows;
    u += ng;
    // A sequence's hypertokens meet the hidden rows of that sequence only.  Where those lie in one group of 8 rows, just
    // that group is loaded, to where all rows would put it (the other rows of the operand are what
    // is left there, and nobody reads their accumulators), and a job of few rows takes several k-blocks per stage: with
    // one, a job of 64 rows had 8 KB a stage in flight, and took as long as one of 256 (V = 128256, d = 4096, 90
    // sequences of 59 hypertokens 301 us, of 256 hypertokens 218).
    j.kb = 1; j.group = -1;
    const int group = j.owner < 0 ? kManyGroups : groups ? groups[j.owner] : j.owner < p.la.N ? j.owner >> 3 : kNoGroup;
    if (group != kManyGroups) {
      j.group = group == kNoGroup ? 0 : group;
      if (ng <= 4) {                               // up to 128 rows: one box, of 1, 2 or 4 granules
        if (ng == 3) j.nrows = 4 * kLogitGran;
        j.kb = logit_short_kb(ng > 2 ? 2 : ng - 1);
      }
    } else if (j.owner >= 0 && ng <= 2) {
      j.kb = 2;         // all hidden rows, two k-blocks of them (V = 32064, d = 3072, 33 rows of 11 sequences, 250 hypertokens: 79 -> 57 us)
    }
    return true;
  }
  __device__ bool next_of_both(Job& j) {
    if (next(j)) return true;
    if (hyper) return false;
    begin_hyper();
    return next(j);
  }
};

// Weight rows of a stage: behind the hidden rows, and behind the further k-blocks of the last group of 8.  (The MMA reads
// 128 hidden rows from a k-block's start; those that are not there lie in the weight rows.)
__host__ __device__ constexpr uint32_t logit_w_offset(int a_box_rows) { return (uint32_t)a_box_rows * 128u + 3u * 1024u; }
// Where a job's hidden rows and weight rows of k-block i lie in a stage.  (Two k-blocks of all hidden rows push the weight rows
// back; 64 of them at most then end where 256 would.)
struct LogitStage {
  uint32_t w_off, a_step;
  __device__ LogitStage(const StreamLogitsParams& p, const Job& j) : w_off(logit_w_offset(p.a_box_rows)), a_step(1024u) {
    if (j.group < 0) a_step = (uint32_t)p.a_box_rows * 128u;
    if (j.group < 0 && j.kb > 1) w_off = (uint32_t)j.kb * a_step;
  }
};
static_assert(2 * 128 * 128 + 2 * 64 * 128 <= 128 * 128 + 3 * 1024 + kLogitNT * 128, "two k-blocks of 128 hidden and 64 weight rows fit a stage");

// ---- producer and MMA role of the logits kernel -----------------------------------------------------
// Everything that is loaded, W_U among it, may come from the kernel ahead: nothing is issued before the dependency wait.
template <int STAGES>
__device__ __forceinline__ void logits_producer(const StreamLogitsParams& p, const int* s_pref, Ctrl* ctrl, uint32_t stage_base,
                                                const LogitMaps& tm) {
  const uint32_t a_bytes = (uint32_t)p.a_box_rows * 128;
  const uint32_t stage_bytes = logit_w_offset(p.a_box_rows) + kLogitNT * 128;      // smem stride of a stage
  const uint64_t pol_w = policy_evict_first(), pol_a = policy_evict_last();
  int stage = 0; uint32_t phase = 0;
  pdl_wait();
  if (!LogitSched::even(p) && !mbar_wait(smem_u32(&ctrl->pref_ready), 0, &ctrl->abort)) return;
  LogitSched sched(p, s_pref);
  Job j;
  auto w_boxes = [&](uint32_t dst, int ks, uint32_t full) {
    // the rows of the job go out as few boxes as possible: largest power-of-two box first
    for (int r0 = 0; r0 < j.nrows;) {
      int cls = kLogitBoxClasses - 1;
      while (cls > 0 && (kLogitGran << cls) > j.nrows - r0) --cls;
      tma_load_3d(dst + r0 * 128, &tm.w[j.wmap * kLogitBoxClasses + cls], 0, j.wrow + r0, ks, full, pol_w);
      r0 += kLogitGran << cls;
    }
  };
  // W_U in a loop of its own: one loop for both kinds of jobs cost it 4 us of 168 (V = 128256, d = 4096, 33 rows)
  while (sched.next(j)) {
    const uint32_t w_off = logit_w_offset(p.a_box_rows), bytes = a_bytes + (uint32_t)j.nrows * 128u;
    for (int ks = 0; ks < p.ksteps; ++ks) {
      if (!mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, &ctrl->abort)) return;
      const uint32_t full = smem_u32(&ctrl->full[stage]);
      const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
      mbar_expect_tx(full, bytes);
      tma_load_3d(sb, &tm.h, 0, 0, ks, full, pol_a);
      w_boxes(sb + w_off, ks, full);
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
    }
  }
  if (!mbar_wait(smem_u32(&ctrl->pref_ready), 0, &ctrl->abort)) return;
  sched.begin_hyper();
  while (sched.next(j)) {                              // the sequences' hypertokens
    const uint32_t w_off = LogitStage(p, j).w_off;
    // (k-blocks beyond the last one, and rows outside the tensors, are zero-filled and counted)
    const uint32_t bytes = (uint32_t)j.kb * ((uint32_t)j.nrows * 128u + (j.group < 0 ? a_bytes : 1024u));
    for (int ks = 0; ks < p.ksteps; ks += j.kb) {
      if (!mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, &ctrl->abort)) return;
      const uint32_t full = smem_u32(&ctrl->full[stage]);
      const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
      mbar_expect_tx(full, bytes);
      if (j.group < 0) tma_load_3d(sb, j.kb > 1 ? &tm.h2 : &tm.h, 0, 0, ks, full, pol_a);
      else tma_load_3d(sb + (uint32_t)j.group * 1024u, &tm.h8[j.kb >> 1], 0, 8 * j.group, ks, full, pol_a);
      if (j.kb == 1) w_boxes(sb + w_off, ks, full);
      else if (j.group < 0) tma_load_3d(sb + w_off, &tm.u2[j.nrows == kLogitGran ? 0 : 1], 0, j.wrow, ks, full, pol_w);
      else tma_load_3d(sb + w_off, &tm.u[j.nrows == kLogitGran ? 0 : j.nrows == 2 * kLogitGran ? 1 : 2], 0, j.wrow, ks, full, pol_w);
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
    }
  }
}

template <int STAGES>
__device__ __forceinline__ void logits_mma(const StreamLogitsParams& p, const int* s_pref, Ctrl* ctrl, uint32_t stage_base,
                                           uint32_t tmem_base) {
  const uint32_t stage_bytes = logit_w_offset(p.a_box_rows) + kLogitNT * 128;
  int stage = 0; uint32_t phase = 0;
  uint32_t job_i = 0;
  LogitSched sched(p, s_pref);
  Job j;
  while (sched.next_of_both(j)) {
    const uint32_t idesc = idesc_bf16_f32(128, j.nrows);
    const uint32_t buf = job_i & 1u, aph = (job_i >> 1) & 1u;
    if (!mbar_wait_warp(smem_u32(&ctrl->acc_empty[buf]), aph ^ 1u, &ctrl->abort)) return;
    tc_fence_after();
    const uint32_t d = tmem_base + buf * kLogitNT;
    const LogitStage at(p, j);
    uint32_t acc = 0;
    for (int ks = 0; ks < p.ksteps; ks += j.kb) {
      if (!mbar_wait_warp(smem_u32(&ctrl->full[stage]), phase, &ctrl->abort)) return;
      tc_fence_after();
      const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
      if (elect_one()) {
        for (int i = 0; i < j.kb; ++i) {
          const uint32_t ab = sb + (uint32_t)i * at.a_step, wb = sb + at.w_off + (uint32_t)(i * j.nrows) * 128u;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_bf16(d, smem_desc_sw128(ab + k * 32), smem_desc_sw128(wb + k * 32), idesc, i || k ? 1u : acc);
        }
        umma_commit(smem_u32(&ctrl->empty[stage]));        // frees the stage when the MMAs are done
      }
      __syncwarp();
      acc = 1;
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
    }
    if (elect_one()) umma_commit(smem_u32(&ctrl->acc_full[buf]));
    __syncwarp();
    ++job_i;
  }
}

template <int STAGES, int EPI_WARPS = 4>
__device__ __forceinline__ void setup_barriers(Ctrl* ctrl) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&ctrl->full[s]), 1);
      mbar_init(smem_u32(&ctrl->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctrl->acc_full[b]), 1);
      mbar_init(smem_u32(&ctrl->acc_empty[b]), EPI_WARPS);
    }
    mbar_init(smem_u32(&ctrl->pref_ready), 2);         // logits: the sequences' granules are counted, their rows found
    ctrl->abort = 0;
    mbar_init_fence();
  }
}

// =================================================================================================
// GEMM kernel: weights as the M operand, activation rows (hi | lo) as the N operand
// =================================================================================================
struct GemmJob { int g, wrow, kb0, kb1; };
struct GemmWalk {
  const StreamGemmParams& p;
  int mid;                               // > 0: a job ends there
  long long u, u1;
  __device__ GemmWalk(const StreamGemmParams& pp) : p(pp), mid(pp.half_stride ? pp.ksteps / 2 : 0) {
    const long long U = (long long)p.groups * p.tiles_per_group * p.ksteps, G = gridDim.x, c = blockIdx.x;
    u = c * U / G;
    u1 = (c + 1) * U / G;
  }
  __device__ bool next(GemmJob& j) {
    if (u >= u1) return false;
    const long long tile = u / p.ksteps;
    j.kb0 = (int)(u - tile * p.ksteps);
    const long long left = u1 - u;
    const int end = j.kb0 < mid ? mid : p.ksteps;
    j.kb1 = (int)((end - j.kb0) < left ? end : j.kb0 + left);
    j.g = (int)tile / p.tiles_per_group;
    j.wrow = ((int)tile - j.g * p.tiles_per_group) * kGemmNT;
    u += j.kb1 - j.kb0;
    return true;
  }
};

__host__ __device__ constexpr uint32_t gemm_tmem_cols(int n_act) {
  return 2 * n_act <= 32 ? 32u : (2 * n_act <= 64 ? 64u : (2 * n_act <= 128 ? 128u : (2 * n_act <= 256 ? 256u : 512u)));
}

// Operand rows (hi and lo) of `live` > 0 packed rows, up to a multiple of `step`.
__device__ __forceinline__ int gemm_op_rows(const StreamGemmParams& p, int live, int step) {
  const int n = (2 * live + step - 1) / step * step;
  return n < p.a_box_rows ? n : p.a_box_rows;
}

template <int KSB, int STAGES>
__global__ void __launch_bounds__(kThreads, 1)
k_stream_gemm(const StreamGemmParams p, const __grid_constant__ StreamGemmMaps tm) {
  constexpr int NT = kGemmNT;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(sm);
  const uint32_t stage_base = smem_u32(sm + 1024);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t a_bytes = (uint32_t)KSB * p.a_box_rows * 128;
  const uint32_t stage_bytes = a_bytes + (uint32_t)KSB * NT * 128;
  pdl_trigger();                                   // the next kernel may get resident behind this one
  // (the word may still be that of the pass before: it only decides whether weights are loaded ahead)
  const int hint = threadIdx.x == 0 && p.peek ? __ldcg(p.rows_dev) : 1;
  setup_barriers<STAGES>(ctrl);
  if (warp == 0 && lane == 0) { prefetch_tmap(&tm.w[0]); if (p.groups > 1) prefetch_tmap(&tm.w[1]); }
  __syncthreads();
  if (warp == 2) { tmem_alloc(smem_u32(&ctrl->tmem_base), gemm_tmem_cols(p.a_box_rows)); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = ctrl->tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      // ---- TMA producer.  The weight tiles depend on no earlier kernel, the activation rows and their
      // count do: during the first pass over the ring only the weight boxes are issued and the
      // activation boxes are noted; once the ring is full (or the work ends) the producer waits for the
      // preceding kernel, picks the box that covers the live rows and issues them.  (A box of the pass's
      // capacity would bring 1.5 bytes of activations per byte of weights at 96 rows of which 55 are live,
      // and what an SM takes in from L2 bounds a batch of this size, not HBM: 546 instead of 511 us per step of
      // 32 sequences at d = 4096.)  With an ordinary launch the wait returns at once.  A pass without a live row (a
      // step that created no entry, an empty range) streams nothing: the producer takes in what it loaded ahead,
      // and the other roles have no work (one sequence, d = 3072: 77 us such a step, 227 with the weights).
      const uint64_t pol_w = policy_evict_first(), pol_a = policy_evict_last();
      struct Deferred { int g, kb; };
      Deferred def[kMaxStages];                       // load i of the first pass uses stage i
      int n_def = 0, issued = 0, box = 0;
      uint32_t box_bytes = 0;
      bool deps = false, ok = true;
      auto need_deps = [&]() {
        if (deps) return;
        pdl_wait();
        deps = true;
        const int live = *p.rows_dev;
        if (live < 1) {
          ok = false;
          for (int i = 0; i < n_def; ++i) mbar_arrive(smem_u32(&ctrl->full[i]));
          for (int i = 0; i < n_def; ++i) mbar_wait(smem_u32(&ctrl->full[i]), 0, &ctrl->abort);
          return;
        }
        const int rows = gemm_op_rows(p, live, p.box_step);
        box = rows / p.box_step - 1;
        box_bytes = (uint32_t)KSB * rows * 128;
        for (int i = 0; i < n_def; ++i) {
          const uint32_t full = smem_u32(&ctrl->full[i]);
          mbar_expect_tx(full, box_bytes);
          tma_load_3d(stage_base + (uint32_t)i * stage_bytes, &tm.a[def[i].g][box], 0, 0, def[i].kb, full, pol_a);
        }
      };
      if (hint < 1) need_deps();
      int stage = 0; uint32_t phase = 0;
      GemmWalk walk(p);
      GemmJob j;
      while (ok && walk.next(j)) {
        for (int ks = j.kb0; ks < j.kb1; ++ks) {
          if (issued == STAGES) need_deps();
          if (!ok) break;
          if (!mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, &ctrl->abort)) { ok = false; break; }
          const uint32_t full = smem_u32(&ctrl->full[stage]);
          const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
          if (deps) mbar_expect_tx(full, KSB * NT * 128 + box_bytes);   // rows outside the tensor are zero-filled and counted
          else mbar_expect_only(full, KSB * NT * 128);
          tma_load_3d(sb + a_bytes, &tm.w[j.g], 0, j.wrow, ks * KSB, full, pol_w);
          if (deps) tma_load_3d(sb, &tm.a[j.g][box], 0, 0, ks * KSB, full, pol_a);
          else { def[n_def].g = j.g; def[n_def].kb = ks * KSB; ++n_def; }
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      need_deps();
    }
  } else if (warp == 1) {
    {  // the whole warp: elect_one()
      // ---- MMA issue: D[128 weight rows][n] += W tile (M operand) x live activation rows (N operand)
      pdl_wait();                                      // the live-row count comes from an earlier kernel
      const int live = *p.rows_dev;
      const uint32_t box_kb = (uint32_t)gemm_op_rows(p, live, p.box_step) * 128;    // one k-block of the activation box
      const uint32_t idesc = idesc_bf16_f32(128, gemm_op_rows(p, live, 16));
      int stage = 0; uint32_t phase = 0, job_i = 0;
      bool ok = live > 0;
      GemmWalk walk(p);
      GemmJob j;
      while (ok && walk.next(j)) {
        const uint32_t buf = job_i & 1u, aph = (job_i >> 1) & 1u;
        if (!mbar_wait_warp(smem_u32(&ctrl->acc_empty[buf]), aph ^ 1u, &ctrl->abort)) break;
        tc_fence_after();
        const uint32_t d = tmem_base + buf * (uint32_t)p.a_box_rows;
        uint32_t acc = 0;
        for (int ks = j.kb0; ks < j.kb1; ++ks) {
          if (!mbar_wait_warp(smem_u32(&ctrl->full[stage]), phase, &ctrl->abort)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
          if (elect_one()) {
#pragma unroll
            for (int i = 0; i < KSB; ++i) {
              const uint32_t ab = sb + (uint32_t)i * box_kb;
              const uint32_t wb = sb + a_bytes + (uint32_t)i * NT * 128;
#pragma unroll
              for (int k = 0; k < 4; ++k)
                umma_bf16(d, smem_desc_sw128(wb + k * 32), smem_desc_sw128(ab + k * 32), idesc, i || k ? 1u : acc);
            }
            umma_commit(smem_u32(&ctrl->empty[stage]));        // frees the stage when the MMAs are done
          }
          __syncwarp();
          acc = 1;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (elect_one()) umma_commit(smem_u32(&ctrl->acc_full[buf]));
        __syncwarp();
        ++job_i;
      }
    }
  } else {
    // ---- epilogue: a thread owns one output feature of the tile (its TMEM lane) and walks the
    // live activation rows (pairs of TMEM columns): hi + lo in registers, one reduction per
    // (row, feature)
    pdl_wait();                                      // the result matrix may still be read by the kernel before
    int rows = *p.rows_dev;
    rows = rows < p.a_box_rows / 2 ? rows : p.a_box_rows / 2;
    const int q = warp & 3;                          // TMEM lane quarter this warp may read
    const int feature = q * 32 + lane;
    uint32_t job_i = 0;
    GemmWalk walk(p);
    GemmJob j;
    while (rows > 0 && walk.next(j)) {
      const uint32_t buf = job_i & 1u, aph = (job_i >> 1) & 1u;
      if (!mbar_wait(smem_u32(&ctrl->acc_full[buf]), aph, &ctrl->abort)) break;
      tc_fence_after();
      float* dst = p.out + (j.kb0 >= walk.mid ? p.half_stride : 0) + (size_t)j.g * p.Rt * p.J + j.wrow + feature;
      const uint32_t t0 = tmem_base + ((uint32_t)(q * 32) << 16) + buf * (uint32_t)p.a_box_rows;
#pragma unroll 1
      for (int r0 = 0; r0 < rows; r0 += 8) {
        uint32_t v[16];
        tmem_ld16(t0 + 2 * r0, v);
        tmem_ld_wait();
#pragma unroll
        for (int x = 0; x < 8; ++x)
          if (r0 + x < rows) red_add_f32(dst + (size_t)(r0 + x) * p.J, __uint_as_float(v[2 * x]) + __uint_as_float(v[2 * x + 1]));
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctrl->acc_empty[buf]));
      ++job_i;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.err, 1);
  if (warp == 2) tmem_dealloc(tmem_base, gemm_tmem_cols(p.a_box_rows));
}

// =================================================================================================
// Logits kernel: fused reductions
// =================================================================================================
static_assert(sizeof(Ctrl) <= 512, "the sequences' tables lie behind it");
template <int STAGES>
__global__ void __launch_bounds__(kLogitThreads, 1)
k_stream_logits(const StreamLogitsParams p, const __grid_constant__ LogitMaps tm) {
  constexpr int NT = kLogitNT;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(sm);
  int* s_pref = reinterpret_cast<int*>(sm + 512);               // [B + 1], then the groups of the sequences: <= 5124 bytes
  const uint32_t stage_base = smem_u32(sm + 1024 + 5120);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  setup_barriers<STAGES, kLogitEpiWarps>(ctrl);
  if (warp == 3) {
    if (lane < 1 + 2 * kLogitBoxClasses) prefetch_tmap(lane == 0 ? &tm.h : &tm.w[lane - 1]);
    if (lane < 3) { prefetch_tmap(&tm.h8[lane]); prefetch_tmap(&tm.u[lane]); prefetch_tmap(lane < 2 ? &tm.u2[lane] : &tm.h2); }
  }
  __syncthreads();                                 // barriers exist, which is all that the producer needs

  if (warp == 0) {
    if (lane == 0) logits_producer<STAGES>(p, s_pref, ctrl, stage_base, tm);
  } else {
    if (warp == 2) { tmem_alloc(smem_u32(&ctrl->tmem_base), tmem_cols(NT)); tmem_relinquish(); }
    pdl_wait();                                    // codebook counters, row tables and partial slots are dependent
    pdl_trigger();                                 // (behind the wait: a step's encoder pass loads weights ahead of its own)
    if (warp == 1) {                               // prefix of the sequences' granule counts
      int carry = 0;
      for (int b0 = 0; b0 < p.cb.B; b0 += 32) {
        const int b = b0 + lane;
        int v = b < p.cb.B ? (p.cb.n[b] + kLogitGran - 1) / kLogitGran : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int x = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += x; }
        if (b < p.cb.B) s_pref[b + 1] = carry + v;
        carry += __shfl_sync(0xffffffffu, v, 31);
      }
      if (lane == 0) s_pref[0] = 0;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctrl->pref_ready));
    }
    if (warp == 3) {                               // the group of each sequence's rows, where they are given
      if (p.la.row_seq) {
        uint8_t* s_group = reinterpret_cast<uint8_t*>(s_pref + p.cb.B + 1);
        for (int b = lane; b < p.cb.B; b += 32) s_group[b] = kNoGroup;
        int seq[4];
        bool other[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          seq[i] = 32 * i + lane < p.la.N ? p.la.row_seq[32 * i + lane] : -1;
          if (seq[i] >= p.cb.B) seq[i] = -1;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i)                // one of a sequence's rows has the say,
          if (seq[i] >= 0) s_group[seq[i]] = (uint8_t)(4 * i + (lane >> 3));
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i)                // and any in another group objects
          other[i] = seq[i] >= 0 && s_group[seq[i]] != 4 * i + (lane >> 3);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (other[i]) s_group[seq[i]] = kManyGroups;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctrl->pref_ready));
    }
    tc_fence_before();
    asm volatile("bar.sync 2, %0;" ::"n"(kLogitThreads - 32) : "memory");      // all but the producer warp
    tc_fence_after();
  }
  if (warp == 1) {
    logits_mma<STAGES>(p, s_pref, ctrl, stage_base, ctrl->tmem_base);
  } else if (warp >= 2) {
    const uint32_t tmem_base = ctrl->tmem_base;
    LogitSched sched(p, s_pref);
    const int q = warp & 3;                        // tensor-memory lane quarter this warp may read
    const int group = (warp - 2) >> 2;             // which 32-column groups of a job it takes
    const LogitsArgs& a = p.la;
    const uint32_t k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    const uint32_t c2 = (uint32_t)a.step, c3 = (uint32_t)(a.step >> 32);
    const size_t ldbg = (size_t)p.cb.V + p.cb.cap;
    RowRed red; red.init();
    const int r = q * 32 + lane;
    int my_seq = -1, my_nvis = 0, my_tgt = -1;
    if (r < a.N) {
      my_seq = a.row_seq ? a.row_seq[r] : r;
      if (my_seq < 0 || my_seq >= p.cb.B) my_seq = -1;
      if (my_seq >= 0) {
        my_nvis = p.cb.n[my_seq];
        if (a.row_nvis) { const int x = a.row_nvis[r]; my_nvis = x < my_nvis ? (x < 0 ? 0 : x) : my_nvis; }
      }
      if (a.targets) my_tgt = a.targets[r];
    }
    uint32_t job_i = 0;
    Job j;
    while (sched.next_of_both(j)) {
      const uint32_t buf = job_i & 1u, aph = (job_i >> 1) & 1u;
      if (!mbar_wait(smem_u32(&ctrl->acc_full[buf]), aph, &ctrl->abort)) break;
      tc_fence_after();
      int limit = 0;
      if (my_seq >= 0) limit = j.owner < 0 ? j.nvalid : (my_seq == j.owner ? min(j.nvalid, my_nvis - j.k0) : 0);
      if (__any_sync(0xffffffffu, limit > 0)) {
#pragma unroll 1
        for (int c0 = 32 * group; c0 < j.nrows; c0 += 32 * kLogitEpiGroups) {
          if (!__any_sync(0xffffffffu, limit > c0)) break;
          uint32_t v[32];
          tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + buf * NT + c0, v);
          tmem_ld_wait();
          const int col0 = j.col0 + c0;
          if (a.select == Z2Z_SELECT_GUMBEL) sample_row32(v, limit - c0, col0, a.inv_temperature, (uint32_t)(a.row_base + r), c2, c3, k0, k1, red);
          if (a.logits_debug) {
#pragma unroll
            for (int x = 0; x < 32; ++x)
              if (c0 + x < limit) a.logits_debug[(size_t)r * ldbg + col0 + x] = __uint_as_float(v[x]);
          }
          const int at = my_tgt - col0;                 // the row's target column, if it lies here and exists
          if (at >= 0 && at < 32 && at < limit - c0 && a.target_logit) a.target_logit[r] = pick32(v, at);
          fold_row32(v, limit - c0, col0, red);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&ctrl->acc_empty[buf]));
      ++job_i;
    }
    // every load has been consumed: the ring's first stage takes the other warps' reductions
    RowRed* others = reinterpret_cast<RowRed*>(sm + 1024 + 5120) + q * 32 + lane;
    if (group > 0) others[(group - 1) * 128] = red;
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kLogitEpiWarps) : "memory");
    if (group == 0)
      for (int g = 1; g < kLogitEpiGroups; ++g) red.merge(others[(g - 1) * 128]);
    if (group == 0 && r < a.N) {
      LogitPartial* lp = reinterpret_cast<LogitPartial*>(a.lpart) + (size_t)r * p.part_stride + blockIdx.x;
      lp->m = red.m; lp->s = red.s; lp->idx = red.idx; lp->gm = red.gm; lp->gidx = red.gidx;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.err, 1);
  if (warp == 2) tmem_dealloc(ctrl->tmem_base, tmem_cols(NT));
}

// One warp per row: merge the partial reductions of the G CTAs.
__global__ void __launch_bounds__(128) k_stream_logits_merge(StreamLogitsParams p, int G) {
  pdl_wait();
  pdl_trigger();
  const LogitsArgs& a = p.la;
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= a.N) return;
  const LogitPartial* lp = reinterpret_cast<const LogitPartial*>(a.lpart) + (size_t)r * p.part_stride;
  RowRed red; red.init();
  for (int g = lane; g < G; g += 32) red.merge(load_partial(lp + g));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    RowRed o;
    o.m = __shfl_xor_sync(0xffffffffu, red.m, off);
    o.s = __shfl_xor_sync(0xffffffffu, red.s, off);
    o.idx = __shfl_xor_sync(0xffffffffu, red.idx, off);
    o.gm = __shfl_xor_sync(0xffffffffu, red.gm, off);
    o.gidx = __shfl_xor_sync(0xffffffffu, red.gidx, off);
    red.merge(o);
  }
  if (lane == 0) {
    if (a.lse) a.lse[r] = red.m + logf(red.s);
    if (a.argmax) a.argmax[r] = red.idx == 0x7fffffff ? -1 : red.idx;
    if (a.max_logit) a.max_logit[r] = red.m;
    if (a.sample) a.sample[r] = red.gidx == 0x7fffffff ? -1 : red.gidx;
  }
}

__global__ void k_fill_nan_f32(float* p, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = __int_as_float(0x7fc00000);
}

// ---- host helpers ---------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(f);
  }
  return fn;
}

}  // namespace

// Tensor map over a row-major bf16 matrix [rows, cols]; box = 64 columns x box_rows rows,
// 128-byte swizzle, out-of-range elements read as zero.
bool make_tmap_bf16(CUtensorMap* m, const void* base, long long rows, long long cols, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (cols % 8) || box_rows < 1 || box_rows > 256 || rows < 1) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tensor map over the same matrix seen as [cols / 64 k-blocks][rows][64]: one box brings
// `box_kb` k-blocks of `box_rows` rows, laid out k-block after k-block (each k-block is then a
// K-major 128-byte-swizzled operand tile).
//
// A map is a pure function of (base, rows, cols, box): the encoded maps are kept, so that a decode
// step, whose operands sit at the same addresses step after step, encodes none in steady state.
namespace {
struct TmapKey {
  const void* base; long long rows, cols; int box_rows, box_kb;
  bool operator==(const TmapKey& o) const {
    return base == o.base && rows == o.rows && cols == o.cols && box_rows == o.box_rows && box_kb == o.box_kb;
  }
};
struct TmapKeyHash {
  size_t operator()(const TmapKey& k) const {
    size_t h = reinterpret_cast<uintptr_t>(k.base) * 0x9E3779B97F4A7C15ull;
    h ^= (size_t)k.rows * 0xC2B2AE3D27D4EB4Full + (size_t)k.cols * 0x165667B19E3779F9ull;
    h ^= ((size_t)k.box_rows << 20) ^ (size_t)k.box_kb;
    return h;
  }
};
constexpr size_t kTmapCacheMax = 4096;           // entries kept; the cache starts over beyond that
std::unordered_map<TmapKey, CUtensorMap, TmapKeyHash> g_tmap_cache;
std::mutex g_tmap_mu;
}  // namespace

bool make_tmap_bf16_kblocks(CUtensorMap* m, const void* base, long long rows, long long cols, int box_rows,
                            int box_kb) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (cols % 64) || box_rows < 1 || box_rows > 256 || box_kb < 1 ||
      box_kb > 256 || rows < 1)
    return false;
  const TmapKey key{base, rows, cols, box_rows, box_kb};
  {
    std::lock_guard<std::mutex> lock(g_tmap_mu);
    auto it = g_tmap_cache.find(key);
    if (it != g_tmap_cache.end()) { *m = it->second; return true; }
  }
  cuuint64_t dims[3] = {64, (cuuint64_t)rows, (cuuint64_t)(cols / 64)};
  cuuint64_t strides[2] = {(cuuint64_t)cols * 2, 128};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)box_kb};
  cuuint32_t es[3] = {1, 1, 1};
  if (fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  std::lock_guard<std::mutex> lock(g_tmap_mu);
  if (g_tmap_cache.size() >= kTmapCacheMax) g_tmap_cache.clear();
  g_tmap_cache.emplace(key, *m);
  return true;
}
// Capacity of the activation box (hi and lo rows of R packed rows) and the step of its heights: eight
// heights cover it.
static int gemm_box_step(int R) { return 2 * R <= 128 ? 16 : 32; }
static int gemm_box_rows(int R) { return (2 * R + gemm_box_step(R) - 1) / gemm_box_step(R) * gemm_box_step(R); }

// Stages of the GEMM ring that fit beside the control block (every operand row an MMA reads is
// loaded or zero-filled, so no readable padding is needed behind the ring).
static int gemm_stages(int ksb, int a_box_rows) {
  const int stage = ksb * a_box_rows * 128 + ksb * kGemmNT * 128;
  const int s = (227 * 1024 - 2048) / stage;
  return s > kMaxStages ? kMaxStages : s;
}
// Two k-blocks per stage (fewer TMA operations per byte) while at least four stages still fit.
int stream_gemm_ksb(int R) { return gemm_stages(2, gemm_box_rows(R)) >= 4 ? 2 : 1; }

// Tensor maps of one activation operand ([2 Rt, K], hi and lo rows interleaved): one per box height.
bool stream_gemm_act_maps(CUtensorMap* maps, const void* act, int Rt, int K, int R) {
  const int step = gemm_box_step(R), n = gemm_box_rows(R) / step, ksb = stream_gemm_ksb(R);
  for (int i = 0; i < 8; ++i) {
    if (i >= n) { maps[i] = maps[n - 1]; continue; }
    if (!make_tmap_bf16_kblocks(&maps[i], act, 2ll * Rt, K, step * (i + 1), ksb)) return false;
  }
  return true;
}

template <int KSB, int STAGES>
static cudaError_t launch_gemm_t(const StreamGemmParams& p, const StreamGemmMaps& maps, int grid, cudaStream_t s) {
  const size_t stage = (size_t)KSB * p.a_box_rows * 128 + (size_t)KSB * kGemmNT * 128;
  const size_t smem = 1024 + 1024 + STAGES * stage;
  auto kern = k_stream_gemm<KSB, STAGES>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(grid), dim3(kThreads), smem, s, p, maps);
}

template <int KSB>
static cudaError_t launch_stream_gemm_k(const StreamGemmParams& p, const StreamGemmMaps& maps, int grid, cudaStream_t s) {
  const int st = gemm_stages(KSB, p.a_box_rows);
  if (st >= 8) return launch_gemm_t<KSB, 8>(p, maps, grid, s);
  if (st >= 6) return launch_gemm_t<KSB, 6>(p, maps, grid, s);
  if (st >= 5) return launch_gemm_t<KSB, 5>(p, maps, grid, s);
  return launch_gemm_t<KSB, 4>(p, maps, grid, s);
}
cudaError_t launch_stream_gemm(StreamGemmParams p, const StreamGemmMaps& maps, int n_sm, cudaStream_t s) {
  if (!p.out || !p.err || !p.rows_dev || p.R < 1 || p.R > 128) return cudaErrorInvalidValue;
  p.box_step = gemm_box_step(p.R);
  p.a_box_rows = gemm_box_rows(p.R);
  p.tiles_per_group = p.J / kGemmNT;
  const long long tiles = (long long)p.groups * p.tiles_per_group, units = tiles * p.ksteps;
  const int most = p.half_stride ? fixed_order_workers(tiles, n_sm, 2) : n_sm;
  const int grid = units < most ? (int)units : most;           // every CTA owns >= 1 unit
  return stream_gemm_ksb(p.R) == 2 ? launch_stream_gemm_k<2>(p, maps, grid, s) : launch_stream_gemm_k<1>(p, maps, grid, s);
}

constexpr int kLogitSmemFixed = 1024 + 1024 + 5120;
static int logit_stage_bytes(int a_box_rows) { return (int)logit_w_offset(a_box_rows) + kLogitNT * 128; }
template <int STAGES>
static cudaError_t launch_logits_t(const StreamLogitsParams& p, const LogitMaps& maps, int grid, cudaStream_t s) {
  const size_t smem = kLogitSmemFixed + STAGES * (size_t)logit_stage_bytes(p.a_box_rows);
  auto kern = k_stream_logits<STAGES>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(grid), dim3(kLogitThreads), smem, s, p, maps);
}

cudaError_t run_logits_stream(const CbView& cb, const LogitsArgs& a, int* err_word, LogitsPartInfo* info, Prof* prof,
                              cudaStream_t s) {
  if (a.N > 128) return cudaErrorInvalidValue;
  static int n_sm = 0;
  if (!n_sm) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (n_sm <= 0) n_sm = 148;
  }
  StreamLogitsParams p{};
  p.cb = cb; p.la = a;
  p.ksteps = a.d / 64;
  p.a_box_rows = (a.N + 7) / 8 * 8;
  p.err = err_word;
  LogitMaps maps;
  if (!make_tmap_bf16_kblocks(&maps.h, a.hidden, a.N, a.d, p.a_box_rows, 1)) return cudaErrorInvalidValue;
  const bool hyper = cb.cap > 0;                       // (otherwise no job uses the maps)
  if (!make_tmap_bf16_kblocks(&maps.h2, a.hidden, a.N, a.d, p.a_box_rows, 2)) return cudaErrorInvalidValue;
  for (int c = 0; c < 2; ++c)
    if (!make_tmap_bf16_kblocks(&maps.u2[c], hyper ? a.Uh : a.WU, hyper ? (long long)cb.B * cb.cap : cb.V, a.d, kLogitGran << c, 2))
      return cudaErrorInvalidValue;
  for (int c = 0; c < 3; ++c) {
    if (!make_tmap_bf16_kblocks(&maps.h8[c], a.hidden, a.N, a.d, 8, 1 << c)) return cudaErrorInvalidValue;
    if (!make_tmap_bf16_kblocks(&maps.u[c], hyper ? a.Uh : a.WU, hyper ? (long long)cb.B * cb.cap : cb.V, a.d, kLogitGran << c,
                                logit_short_kb(c)))
      return cudaErrorInvalidValue;
  }
  for (int c = 0; c < kLogitBoxClasses; ++c) {
    if (!make_tmap_bf16_kblocks(&maps.w[c], a.WU, cb.V, a.d, kLogitGran << c, 1)) return cudaErrorInvalidValue;
    if (cb.cap > 0) {
      if (!make_tmap_bf16_kblocks(&maps.w[kLogitBoxClasses + c], a.Uh, (long long)cb.B * cb.cap, a.d, kLogitGran << c, 1))
        return cudaErrorInvalidValue;
    } else {
      maps.w[kLogitBoxClasses + c] = maps.w[c];
    }
  }
  // every CTA must own at least one unit: the granules of W_U alone are a lower bound on the units
  const int units_lb = (cb.V + kLogitGran - 1) / kLogitGran;
  const int grid = units_lb < n_sm ? units_lb : n_sm;
  p.part_stride = grid + 2;
  if ((size_t)a.N * p.part_stride * sizeof(LogitPartial) > a.lpart_bytes) return cudaErrorMemoryAllocation;
  if (info) { info->stride = p.part_stride; info->count = grid; }
  if (a.target_logit) {
    ProfScope ps(prof, kProfLogitsMerge, 1, s);
    k_fill_nan_f32<<<(a.N + 255) / 256, 256, 0, s>>>(a.target_logit, a.N);
  }
  cudaError_t e;
  {
    ProfScope ps(prof, kProfLogits, 1, s);
    const int st = (227 * 1024 - kLogitSmemFixed) / logit_stage_bytes(p.a_box_rows);        // stages that fit, 4 or more
    e = st >= 5 ? launch_logits_t<5>(p, maps, grid, s) : launch_logits_t<4>(p, maps, grid, s);
  }
  if (e != cudaSuccess || info) return e;
  ProfScope ps(prof, kProfLogitsMerge, 1, s);
  return launch_pdl(k_stream_logits_merge, dim3((a.N + 3) / 4), dim3(128), 0, s, p, grid);
}

}  // namespace z2z
