// Weight-streaming skinny GEMM on CTA pairs, for hyper-encoder passes of a large decode batch or of a call
// bounded to some hundred activation rows (more than 128, fewer than a prompt-sized pass has):
//
//   out[group][r][j] += sum_k A[group][r][k] * W[group][j][k]
//
// A weight byte crosses HBM once, but the activation rows have to be brought from L2 into every SM
// for every weight tile it streams, and that ingest is what bounds a batch of this size.  One CTA per
// weight tile and row tile of 128 rows brought the weights again for every row tile, also for tiles
// without a live row.  Here
//   * two CTAs share a tile of 256 weight rows (tcgen05.mma.cta_group::2, M = 256): each loads its own
//     128 weight rows and HALF of the activation rows;
//   * the activation box follows the LIVE rows, a count that only the device knows: one tensor map
//     per box height (16, 32, .. 128 rows), picked once the preceding kernel is done.  The weight
//     boxes of the first pass over the ring are issued before that;
//   * up to 256 packed rows ride on one stream of the weights: hi and lo part of a row are two columns
//     of tensor memory, two accumulators of 128 rows.  More live rows run as several such blocks, the same
//     weight tile one after the other, so that it comes from L2 the second time;
//   * an accumulator takes in one product per weight, hi and lo in columns of their own, and at most 8192
//     weights before it is drained: tensor-core sums lose low bits with every product added.  (Both parts
//     in one column would let 512 rows ride on one stream - 384 rows of both encoders, d = 3072: 687
//     instead of 787 us a step, 640 rows 1392 against 1173 - but the error against fp64, in units of the
//     rows' rms, is then 2.5e-5 instead of 1.35e-5 at d = 4096 and 2.1e-5 instead of 1.1e-5 at d = 3072.)
// A decode step of 90 sequences (d = 3072, one encoder, 270 rows of capacity, about 150 live) takes 1.7 times as
// long with one CTA per weight tile and 128 rows.
//
// Work is cut stream-K style: cluster c of C owns units [floor(c U / C), floor((c + 1) U / C)) of the
// (group, weight tile, row block, k-step) space and adds its accumulators into the fp32 result with
// reductions in global memory, like k_stream_gemm.
//
// Operand layout: packed row r of the activations is rows 2 r (bf16 hi) and 2 r + 1 (lo) of
// [2 Rt, K], seen as [k-block][operand row][64].  An epilogue thread owns one output feature.
//
// Roles per CTA: warp 0 lane 0 TMA producer, warp 1 MMA issuer (an elected lane; leader CTA only), warps 2-9
// epilogue.  Every mbarrier wait is bounded.
#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_sm100.cuh"
#include "z2z_stream.h"

namespace z2z {
using namespace sm100;

namespace {

constexpr int kEpiWarps = 8;             // two per tensor-memory lane quarter, one for each half of a row block
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kSpMaxStages = 8;
constexpr int kSpBlockRows = 256;        // packed rows that share one stream of the weights
constexpr int kSpHalfRows = kSpBlockRows / 2;                     // ... of one accumulator
constexpr int kSpChain = 128;            // k-blocks of 64 columns an accumulator takes in
constexpr int kSpSmem = 227 * 1024;

struct SpCtrl {
  unsigned long long full[kSpMaxStages], empty[kSpMaxStages], acc_full, acc_empty;
  uint32_t tmem_base;
  int abort;
};

struct SpJob { int g, wrow, block, kb0, kb1; };
struct SpWalk {
  const StreamPairParams& p;
  int blocks, chain;                     // a job takes at most `chain` k-steps
  long long u, u1;
  __device__ SpWalk(const StreamPairParams& pp, int live_blocks, int chain_) : p(pp), blocks(live_blocks), chain(chain_) {
    const long long U = (long long)p.groups * p.tiles_per_group * blocks * p.ksteps, C = gridDim.x >> 1, c = blockIdx.x >> 1;
    u = c * U / C;
    u1 = (c + 1) * U / C;
  }
  __device__ bool next(SpJob& j) {
    if (u >= u1) return false;
    const long long job = u / p.ksteps;
    j.kb0 = (int)(u - job * p.ksteps);
    const long long left = u1 - u;
    int end = (j.kb0 / chain + 1) * chain;
    end = end < p.ksteps ? end : p.ksteps;
    j.kb1 = (int)((end - j.kb0) < left ? end : j.kb0 + left);
    const long long tile = job / blocks;
    j.block = (int)(job - tile * blocks);
    j.g = (int)(tile / p.tiles_per_group);
    j.wrow = ((int)tile - j.g * p.tiles_per_group) * 256;
    u += j.kb1 - j.kb0;
    return true;
  }
};

// Columns of tensor memory (the MMA's N, a multiple of 32) that half `h` of a row block takes, 0 if it has
// no live row.
__device__ __forceinline__ int sp_cols(int live, int block, int h) {
  int rows = live - block * kSpBlockRows - h * kSpHalfRows;
  if (rows < 1) return 0;
  if (rows > kSpHalfRows) rows = kSpHalfRows;
  return (2 * rows + 31) & ~31;
}
// Bytes per CTA of the activation box for n columns: half of the operand rows.
__device__ __forceinline__ uint32_t sp_box_bytes(int n) { return (uint32_t)n * 64u; }
// Row blocks with a live row (at least one).  A pass whose capacity is one block does not need the count.
__device__ __forceinline__ int sp_live_blocks(const StreamPairParams& p, int live) {
  return p.blocks > 1 && live > kSpBlockRows ? (live + kSpBlockRows - 1) / kSpBlockRows : 1;
}

// 4 x 4 transpose among four neighbouring lanes: f[x] of lane t becomes f[t] of lane x.
__device__ __forceinline__ void transpose4(float (&f)[4], int lane) {
  float s0 = (lane & 1) ? f[0] : f[1], s1 = (lane & 1) ? f[2] : f[3];
  s0 = __shfl_xor_sync(0xffffffffu, s0, 1);
  s1 = __shfl_xor_sync(0xffffffffu, s1, 1);
  if (lane & 1) { f[0] = s0; f[2] = s1; } else { f[1] = s0; f[3] = s1; }
  s0 = (lane & 2) ? f[0] : f[2]; s1 = (lane & 2) ? f[1] : f[3];
  s0 = __shfl_xor_sync(0xffffffffu, s0, 2);
  s1 = __shfl_xor_sync(0xffffffffu, s1, 2);
  if (lane & 2) { f[0] = s0; f[1] = s1; } else { f[2] = s0; f[3] = s1; }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_stream_pair(const StreamPairParams p, const __grid_constant__ StreamPairMaps tm) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  SpCtrl* ctrl = reinterpret_cast<SpCtrl*>(sm);
  const uint32_t stage_base = smem_u32(sm + 1024);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();          // 0: leader (issues the MMAs), 1: peer
  const uint32_t stage_bytes = (uint32_t)p.act_bytes + 16384u;
  const int STAGES = p.stages;
  pdl_trigger();                                    // the next kernel may get resident behind this one
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&ctrl->full[s]), 1);        // leader: its producer's arrive + bytes of both CTAs
      mbar_init(smem_u32(&ctrl->empty[s]), 1);       // one multicast commit
    }
    mbar_init(smem_u32(&ctrl->acc_full), 1);         // one multicast commit
    mbar_init(smem_u32(&ctrl->acc_empty), 2 * kEpiWarps);        // leader: epilogue warps of both CTAs
    ctrl->abort = 0;
    mbar_init_fence();
    prefetch_tmap(&tm.w[0]);
    if (p.groups > 1) prefetch_tmap(&tm.w[1]);
  }
  __syncthreads();
  if (warp == 2) { tmem_alloc_pair(smem_u32(&ctrl->tmem_base), 512); tmem_relinquish_pair(); }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // both CTAs' barriers exist before any remote signal
  tc_fence_after();
  const uint32_t tmem_base = ctrl->tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer (both CTAs) ---------------------------------------------------
      const uint64_t pol_a = policy_evict_last();
      const uint64_t pol_w = p.blocks > 1 ? policy_evict_last() : policy_evict_first();
      uint32_t full_leader[kSpMaxStages];
      for (int s = 0; s < STAGES; ++s) full_leader[s] = map_to_cta(smem_u32(&ctrl->full[s]), 0);
      // Weight tiles depend on no earlier kernel, activations and their row count do: during the first
      // pass over the ring only the weight boxes are issued and the activation boxes are noted.
      SpJob def[kSpMaxStages];                        // load i of the first pass uses stage i; kb0 = its k-step
      int n_def = 0, issued = 0, live = 0;
      bool deps = false, ok = true;
      auto act_bytes = [&](int block) { return sp_box_bytes(sp_cols(live, block, 0) + sp_cols(live, block, 1)); };
      auto load_act = [&](int st, const SpJob& j, int ks) {
        const uint32_t sb = stage_base + (uint32_t)st * stage_bytes;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int n = sp_cols(live, j.block, h);
          if (n == 0) continue;
          tma_load_3d_pair(sb + h * 16384u, &tm.a[j.g][(n >> 5) - 1], 0,
                           2 * (j.block * kSpBlockRows + h * kSpHalfRows) + (int)rank * (n >> 1), ks, full_leader[st], pol_a);
        }
      };
      auto need_deps = [&]() {
        if (deps) return;
        pdl_wait();
        live = *p.rows_dev;
        live = live < p.R ? live : p.R;
        deps = true;
        if (live < 1) {
          // a pass without a row: the leader takes in what both CTAs loaded ahead, and the peer stays until then
          // (the cluster leaves together).  Such a step of 90 sequences, d = 3072, one encoder: 122 us, 264 with the weights.
          ok = false;
          if (rank == 0) {
            for (int i = 0; i < n_def; ++i) mbar_arrive(smem_u32(&ctrl->full[i]));
            for (int i = 0; i < n_def; ++i) mbar_wait(smem_u32(&ctrl->full[i]), 0, &ctrl->abort);
          }
          return;
        }
        for (int i = 0; i < n_def; ++i) {
          if (rank == 0) mbar_expect_tx(smem_u32(&ctrl->full[i]), 2 * act_bytes(def[i].block));
          load_act(i, def[i], def[i].kb0);
        }
      };
      if (p.blocks > 1) need_deps();                   // the walk itself depends on the row count
      int stage = 0; uint32_t phase = 0;
      SpWalk walk(p, sp_live_blocks(p, live), p.ksteps);      // (where an accumulator ends does not matter to the loads)
      SpJob j;
      while (ok && walk.next(j)) {
        for (int ks = j.kb0; ks < j.kb1; ++ks) {
          if (issued == STAGES) need_deps();
          if (!ok) break;
          if (!mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, &ctrl->abort)) { ok = false; break; }
          if (rank == 0) {
            const uint32_t full = smem_u32(&ctrl->full[stage]);
            if (deps) mbar_expect_tx(full, 2 * (16384u + act_bytes(j.block)));
            else mbar_expect_only(full, 2 * 16384u);
          }
          const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
          tma_load_3d_pair(sb + p.act_bytes, &tm.w[j.g], 0, j.wrow + (int)rank * 128, ks, full_leader[stage], pol_w);
          if (deps) load_act(stage, j, ks);
          else { def[n_def] = j; def[n_def].kb0 = ks; ++n_def; }
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      need_deps();
    }
  } else {
    pdl_wait();                                       // the row count and the result matrix belong to earlier kernels
    int live = *p.rows_dev;
    live = live < p.R ? live : p.R;
    const int n_blocks = sp_live_blocks(p, live);
    const int chain = p.parts > 1 ? p.ksteps / p.parts : kSpChain;
    if (warp == 1) {
      if (rank == 0) {                                 // (the whole warp: elect_one())
        // ---------------- MMA issuer (leader only): D[256 weight rows][n] += W tile x activation rows -----
        int stage = 0; uint32_t phase = 0, job_i = 0;
        bool ok = live > 0;
        SpWalk walk(p, n_blocks, chain);
        SpJob j;
        while (ok && walk.next(j)) {
          const uint32_t aph = job_i & 1u;
          if (!mbar_wait_warp(smem_u32(&ctrl->acc_empty), aph ^ 1u, &ctrl->abort)) break;
          tc_fence_after();
          const int n0 = sp_cols(live, j.block, 0), n1 = sp_cols(live, j.block, 1);
          const uint32_t id0 = idesc_bf16_f32(256, n0), id1 = idesc_bf16_f32(256, n1 ? n1 : 32);
          const uint32_t d = tmem_base;
          uint32_t acc = 0;
          for (int ks = j.kb0; ks < j.kb1; ++ks) {
            if (!mbar_wait_warp(smem_u32(&ctrl->full[stage]), phase, &ctrl->abort)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
            const uint32_t wb = sb + p.act_bytes;
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                umma_bf16_pair(d, smem_desc_sw128(wb + k * 32), smem_desc_sw128(sb + k * 32), id0, k ? 1u : acc);
                if (n1) umma_bf16_pair(d + 256, smem_desc_sw128(wb + k * 32), smem_desc_sw128(sb + 16384u + k * 32), id1, k ? 1u : acc);
              }
              umma_commit_pair(smem_u32(&ctrl->empty[stage]));    // frees the stage in both CTAs
            }
            __syncwarp();
            acc = 1;
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          if (elect_one()) umma_commit_pair(smem_u32(&ctrl->acc_full));       // wakes the epilogues of both CTAs
          __syncwarp();
          ++job_i;
        }
      }
    } else {
      // ---------------- epilogue (both CTAs): thread = output feature -----------------------------------
      // Nothing overlaps the epilogue, as both accumulators are in use, and one reduction instruction per
      // row and feature is what it costs: four lanes transpose four rows x four features among
      // themselves and add 16 bytes each.  (Two passes of 217 rows, one per encoder, d = 3072, with the parse
      // and the logits around them: 859 us with single words on four warps, 805 with 16 bytes, 714 with
      // whole clusters per tile, 654 on eight warps.)
      const int q = warp & 3;                          // TMEM lane quarter this warp may read
      const int group = (warp - 2) >> 2;               // takes every other 32 columns
      const uint32_t acc_empty_leader = map_to_cta(smem_u32(&ctrl->acc_empty), 0);
      uint32_t job_i = 0;
      SpWalk walk(p, n_blocks, chain);
      SpJob j;
      while (live > 0 && walk.next(j)) {
        const uint32_t aph = job_i & 1u;
        if (!mbar_wait(smem_u32(&ctrl->acc_full), aph, &ctrl->abort)) break;
        tc_fence_after();
        const int feature0 = j.wrow + (int)rank * 128;
        if (feature0 < p.J) {                          // the last tile may be half outside (J is a multiple of 128)
          const size_t part = p.parts > 1 ? (j.kb0 / chain) * p.part_stride : 0;
          const int row0 = j.block * kSpBlockRows;
          const int rows = live - row0 < kSpBlockRows ? live - row0 : kSpBlockRows;
          // this lane's row of every four, and the first of the four features it adds
          float* dst = p.out + part + ((size_t)j.g * p.Rt + row0 + (lane & 3)) * p.J + feature0 + q * 32 + (lane & ~3);
          const uint32_t t0 = tmem_base + ((uint32_t)(q * 32) << 16);
          auto add4 = [&](float (&f)[4], int r) {      // rows r .. r + 3
            transpose4(f, lane);
            if (r + (lane & 3) < rows) red_add_f32x4(dst + (size_t)r * p.J, f[0], f[1], f[2], f[3]);
          };
#pragma unroll 1
          for (int c0 = 32 * group; c0 < 2 * rows; c0 += 64) {
            uint32_t v[32];
            tmem_ld32(t0 + c0, v);
            tmem_ld_wait();
#pragma unroll
            for (int y = 0; y < 4; ++y) {
              float f[4];
#pragma unroll
              for (int x = 0; x < 4; ++x) f[x] = __uint_as_float(v[8 * y + 2 * x]) + __uint_as_float(v[8 * y + 2 * x + 1]);
              add4(f, c0 / 2 + 4 * y);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty_leader);
        ++job_i;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.err, 1);
  cluster_sync_all();                               // nobody leaves while the pair's MMAs may read its memory
  if (warp == 2) tmem_dealloc_pair(tmem_base, 512);
}

int round32(int n) { return (n + 31) / 32 * 32; }

// Shared memory of one stage's activation boxes per CTA, for a pass of at most R > 128 rows.
int pair_act_bytes(int R) {
  return 16384 + (R < kSpBlockRows ? round32(2 * (R - kSpHalfRows)) * 64 : 16384);
}

}  // namespace

// Tensor maps of one activation operand ([2 Rt, K], hi and lo rows interleaved): one per box height.
bool stream_pair_act_maps(CUtensorMap* maps, const void* act, int Rt, int K) {
  for (int i = 0; i < 8; ++i)
    if (!make_tmap_bf16_kblocks(&maps[i], act, 2ll * Rt, K, 16 * (i + 1), 1)) return false;
  return true;
}

cudaError_t launch_stream_pair(StreamPairParams p, const StreamPairMaps& maps, int n_sm, cudaStream_t s) {
  if (!p.out || !p.err || !p.rows_dev || p.R <= 128 || p.parts < 1 || p.ksteps % p.parts) return cudaErrorInvalidValue;
  p.tiles_per_group = (p.J + 255) / 256;
  p.blocks = (p.R + kSpBlockRows - 1) / kSpBlockRows;
  p.act_bytes = pair_act_bytes(p.R);
  const int stage = p.act_bytes + 16384;
  p.stages = (kSpSmem - 2048) / stage;
  if (p.stages > kSpMaxStages) p.stages = kSpMaxStages;
  const size_t smem = 2048 + (size_t)p.stages * stage;
  const long long units = (long long)p.groups * p.tiles_per_group * p.ksteps;      // every cluster owns >= 1 unit
  int clusters = units < n_sm / 2 ? (int)units : n_sm / 2;
  // A whole number of clusters per tile leaves every cluster with one piece of one tile, and so with one
  // epilogue instead of two; worth up to a seventh of the clusters (decode steps with all rows live, 74 -> whole:
  // d = 3072 180 rows of both encoders 426 -> 405 us, 384 811 -> 789, d = 1024 640 rows 343 -> 311; d = 2048 640 rows
  // lose, 664 -> 678).
  const int tiles = p.groups * p.tiles_per_group, whole = clusters / tiles * tiles;
  if (p.parts > 1) clusters = fixed_order_workers(tiles, clusters, p.parts);
  else if (7 * whole >= 6 * clusters) clusters = whole;
  cudaError_t e = cudaFuncSetAttribute(k_stream_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_stream_pair, dim3(2 * clusters), dim3(kThreads), smem, s, p, maps);
}

}  // namespace z2z
