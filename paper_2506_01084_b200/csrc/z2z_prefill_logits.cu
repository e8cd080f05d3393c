// Joint logits with fused reductions for many hidden rows (chunks of positions, prompt scoring; paper
// Section 2.3 steps 7-9).  This is a contraction
//     [N rows] x [V + n_b columns] x d
// and runs on the tcgen05 tensor cores with CTA pairs:
//
//   * a cluster of two CTAs owns a tile of 256 hidden rows x up to 256 vocabulary columns;
//     `tcgen05.mma.cta_group::2` (M = 256, N = 64 .. 256, K = 16) reads 128 rows of the hidden tile
//     and half of the weight rows from EACH CTA's shared memory, so every CTA loads only its
//     own halves (plain TMA loads, no multicast) and the operand traffic per flop is halved.  With at
//     most 192 rows in all a CTA takes (and loads) half of them, up to a multiple of 32;
//   * fp32 accumulators live in tensor memory, 128 lanes x 256 columns per CTA, double
//     buffered: while the pair's tensor cores work on column tile j + 1, the four epilogue
//     warps of each CTA fold tile j into a running (max, sum-exp, argmax) per hidden row, one
//     thread per row, so no logit is ever written;
//   * work unit = (row tile, column strip): a strip is a share of W_U's columns (in granules of 64) and
//     of the visible hypertokens of the sequences present in the row tile, and the pair sweeps it in
//     tiles of up to 256 columns with the running reduction in registers.  Units are dealt round-robin
//     to the clusters, so that neighbouring clusters read the same weight tiles at about the same
//     time (L2 reuse).
//
// Up to 256 rows the kernel is bound by the weight stream, beyond by the tensor cores.  From 129 rows on it
// replaced a kernel of single CTAs that streams all weights once per 128 rows (V = 128256, d = 4096:
// 343 -> 231 us at 129 rows, 988 -> 570 at 700, 2714 -> 1395 at 2000).
//
// Roles per CTA: warp 0 lane 0 TMA producer, warp 1 MMA issuer (an elected lane; leader CTA only),
// warps 2-5 epilogue.  Every mbarrier wait is bounded; on a timeout the CTA raises an abort flag,
// all roles leave their loops, tensor memory is released and an error word is set.
#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_sm100.cuh"
#include "z2z_stream.h"

namespace z2z {
using namespace sm100;

namespace {

// Epilogue warps: one per tensor-memory lane quarter, or two that take every other 32 columns when every
// column costs random numbers (128 sequences at V = 12000, sampled: 433 -> 395 us a step).
__host__ __device__ constexpr int epi_warps(bool generic) { return generic ? 8 : 4; }
__host__ __device__ constexpr int prefill_threads(bool generic) { return 64 + 32 * epi_warps(generic); }
constexpr int kTileRows = 256;           // hidden rows per cluster tile (128 per CTA)
constexpr int kTileCols = 256;           // most vocabulary columns per tile (half of the weight rows per CTA)
constexpr int kGran = 64;                // columns are dealt in granules of this many
constexpr int kPrefillStages = 11;           // a stage holds the CTA's hidden rows and up to 128 weight rows, 64 columns
constexpr int kRingBytes = 221 * 1024;   // each: 6 stages of 32 KB with 128 hidden rows, 11 of 20 KB with 32

struct PCtrl {
  unsigned long long full[kPrefillStages], empty[kPrefillStages], acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(PCtrl) <= 1024 && 128 * sizeof(RowRed) <= 3072, "control block and hand-over area");

// Tensor maps: hidden rows, then W_U and U_h in boxes of 32, 64, 96 and 128 rows (half a tile).
struct PrefillMaps { CUtensorMap h, w[2][4]; };

// ---- schedule --------------------------------------------------------------------------------------
// Columns of a row tile: the 64-column granules of W_U, then for each sequence b in [lo, hi] (the
// sequences that own rows of the tile) the tiles of up to 256 visible rows of U_h[b].  Strips are cut by
// COST: a column tile of ng granules loads ng * 32 weight rows and all hidden rows of the CTA per k-step,
// so that a short hypertoken tile costs nearly as much as a full one (equal shares of the columns
// gave the last cluster one job per sequence: 50 instead of 27 us at V = 16000, d = 2048, five
// sequences of 30 entries).  With h = 32-row units of hidden rows per CTA (1 .. 4) a granule of W_U
// costs 4 + h (h is shared by the four of a full tile) and a hypertoken tile 4 (h + ng).
struct TileRef { int wmap; int wrow; int col0; int owner; int k0; int nvalid; int ng; };

__device__ __forceinline__ int tile_cost(const PrefillLogitsParams& p, int ng) { return 4 * (p.cta_rows / 32 + ng); }
// Cost of all hypertoken tiles of a sequence of n entries.
__device__ __forceinline__ int seq_cost(const PrefillLogitsParams& p, int n) {
  const int rest = n % kTileCols;
  return n / kTileCols * tile_cost(p, kTileCols / kGran) + (rest ? tile_cost(p, (rest + kGran - 1) / kGran) : 0);
}

struct UnitWalk {
  const PrefillLogitsParams& p;
  int rt, hi;                   // row tile, last sequence present
  int v, v1;                    // granules of W_U left in the strip
  int b, tb;                    // hypertokens: sequence, tile inside it
  long long at, h1;             // cost at the start of sequence b, end of the strip (0 = behind W_U)
  __device__ UnitWalk(const PrefillLogitsParams& pp) : p(pp) {}
  __device__ void begin(long long unit) {
    rt = (int)(unit / p.strips);
    const int strip = (int)(unit - (long long)rt * p.strips);
    b = p.tile_lo[rt]; hi = p.tile_hi[rt];
    const int cs = 4 + p.cta_rows / 32;
    const long long stat = (long long)p.n_static * cs, total = stat + p.tile_nh[rt];
    const long long u0 = strip * total / p.strips, u1 = (strip + 1) * total / p.strips;
    v = (int)(u0 < stat ? (u0 + cs - 1) / cs : p.n_static);
    v1 = (int)(u1 < stat ? (u1 + cs - 1) / cs : p.n_static);
    const long long h0 = u0 > stat ? u0 - stat : 0;
    h1 = u1 - stat;                             // not positive: no hypertoken tile starts in this strip
    tb = 0; at = 0;
    if (h1 > 0 && h0 > 0) {                     // a tile belongs to the strip in which its cost starts
      const int full = tile_cost(p, kTileCols / kGran);
      while (b <= hi) {
        const int n = p.cb.n[b], nt = (n + kTileCols - 1) / kTileCols;
        tb = h0 > at ? (int)((h0 - at + full - 1) / full) : 0;
        if (tb < nt) break;
        at += seq_cost(p, n);
        ++b; tb = 0;
      }
    }
  }
  __device__ bool next(TileRef& t) {
    if (v < v1) {
      t.wmap = 0; t.wrow = v * kGran; t.col0 = t.wrow; t.owner = -1; t.k0 = 0;
      t.ng = v1 - v < kTileCols / kGran ? v1 - v : kTileCols / kGran;
      t.nvalid = p.cb.V - t.wrow < t.ng * kGran ? p.cb.V - t.wrow : t.ng * kGran;
      v += t.ng;
      return true;
    }
    while (h1 > at && b <= hi) {
      const int n = p.cb.n[b], k0 = tb * kTileCols;
      if (k0 < n) {
        if (at + (long long)tb * tile_cost(p, kTileCols / kGran) >= h1) return false;
        t.wmap = 1; t.owner = b; t.k0 = k0;
        t.wrow = b * p.cb.cap + k0; t.col0 = p.cb.V + k0;
        t.nvalid = n - k0 < kTileCols ? n - k0 : kTileCols;
        t.ng = (t.nvalid + kGran - 1) / kGran;
        ++tb;
        return true;
      }
      at += seq_cost(p, n);
      ++b; tb = 0;
    }
    return false;
  }
};

// ---- plan: sequence range and cost of the hypertoken tiles of every row tile; target logits start as NaN -----------------------------------
__global__ void __launch_bounds__(256) k_prefill_plan(PrefillLogitsParams p) {
  __shared__ int s_lo, s_hi, s_nh;
  pdl_trigger();
  pdl_wait();
  const int rt = blockIdx.x;
  if (threadIdx.x == 0) { s_lo = 0x7fffffff; s_hi = -1; s_nh = 0; }
  __syncthreads();
  const int r = rt * kTileRows + threadIdx.x;
  if (r < p.la.N) {
    if (p.la.target_logit) p.la.target_logit[r] = __int_as_float(0x7fc00000);
    int sq = p.la.row_seq ? p.la.row_seq[r] : r;
    if (sq >= 0 && sq < p.cb.B) { atomicMin(&s_lo, sq); atomicMax(&s_hi, sq); }
  }
  __syncthreads();
  int nh = 0;
  const int n_seq = s_hi < s_lo ? 0 : s_hi - s_lo + 1;          // (none when no row of the tile has an owner)
  for (int i = threadIdx.x; i < n_seq; i += blockDim.x) nh += seq_cost(p, p.cb.n[s_lo + i]);
  if (nh) atomicAdd(&s_nh, nh);
  __syncthreads();
  if (threadIdx.x == 0) { p.tile_lo[rt] = s_lo; p.tile_hi[rt] = s_hi; p.tile_nh[rt] = s_nh; }
}

// =================================================================================================
// Barrier of the epilogue warps; true if `ok` was true in all their threads.
template <int THREADS>
__device__ __forceinline__ bool epilogue_all(bool ok) {
  uint32_t all;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(all)
      : "r"(ok ? 1u : 0u), "n"(THREADS)
      : "memory");
  return all != 0;
}

template <bool GENERIC>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(prefill_threads(GENERIC), 1)
k_prefill_logits(const PrefillLogitsParams p, const __grid_constant__ PrefillMaps tm) {
  constexpr int EW = epi_warps(GENERIC);
  constexpr int GROUPS = EW / 4;                    // epilogue warps per lane quarter
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  PCtrl* ctrl = reinterpret_cast<PCtrl*>(sm);
  RowRed* s_red = reinterpret_cast<RowRed*>(sm + 1024);
  const uint32_t stage_base = smem_u32(sm + 4096);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();          // 0: leader (issues the MMAs), 1: peer
  const long long n_clusters = gridDim.x >> 1, cluster_id = blockIdx.x >> 1;
  const long long n_units = (long long)p.row_tiles * p.strips;
  const int STAGES = p.stages;
  // An MMA reads 128 hidden rows from a stage's start; with fewer loaded it reads on into the stage's
  // weight rows, which only feeds accumulator lanes that nobody looks at.
  const uint32_t w_off = (uint32_t)p.cta_rows * 128, stage_bytes = w_off + 16384u;
  pdl_trigger();                                    // the next kernel may get resident behind this one

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&ctrl->full[s]), 1);        // leader: its producer's arrive + bytes of both CTAs
      mbar_init(smem_u32(&ctrl->empty[s]), 1);       // one multicast commit
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&ctrl->acc_full[b]), 1);    // one multicast commit
      mbar_init(smem_u32(&ctrl->acc_empty[b]), 2 * EW);   // leader: epilogue warps of both CTAs
    }
    ctrl->abort = 0;
    mbar_init_fence();
    prefetch_tmap(&tm.h); prefetch_tmap(&tm.w[0][3]);
  }
  __syncthreads();
  if (warp == 2) { tmem_alloc_pair(smem_u32(&ctrl->tmem_base), 512); tmem_relinquish_pair(); }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                               // both CTAs' barriers exist before any remote signal
  tc_fence_after();
  const uint32_t tmem_base = ctrl->tmem_base;
  pdl_wait();                                       // the plan, the codebook state and the hidden rows

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer (both CTAs): own hidden rows, own half of the weight rows ------
      const uint64_t pol_a = policy_evict_last();
      const uint64_t pol_w = p.row_tiles == 1 ? policy_evict_first() : policy_evict_last();   // read once, or by every row tile
      uint32_t full_leader[kPrefillStages];
      for (int s = 0; s < STAGES; ++s) full_leader[s] = map_to_cta(smem_u32(&ctrl->full[s]), 0);
      UnitWalk w(p);
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (long long u = cluster_id; u < n_units && ok; u += n_clusters) {
        w.begin(u);
        const int arow = w.rt * kTileRows + (int)rank * p.cta_rows;
        TileRef t;
        while (ok && w.next(t)) {
          const CUtensorMap* wm = &tm.w[t.wmap][t.ng - 1];
          const int half = t.ng * (kGran / 2);
          const int wrow = t.wrow + (int)rank * half;
          const uint32_t bytes = 2u * 128u * (uint32_t)(p.cta_rows + half);        // of both CTAs
          for (int ks = 0; ks < p.ksteps; ++ks) {
            if (!mbar_wait(smem_u32(&ctrl->empty[stage]), phase ^ 1u, &ctrl->abort)) { ok = false; break; }
            if (rank == 0) mbar_expect_tx(smem_u32(&ctrl->full[stage]), bytes);
            const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
            tma_load_2d_pair(sb, &tm.h, ks * 64, arow, full_leader[stage], pol_a);
            tma_load_2d_pair(sb + w_off, wm, ks * 64, wrow, full_leader[stage], pol_w);
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------- MMA issuer (leader only, the whole warp: elect_one()) ------------------------------------------------------
      UnitWalk w(p);
      int stage = 0; uint32_t phase = 0, job_i = 0;
      bool ok = true;
      for (long long u = cluster_id; u < n_units && ok; u += n_clusters) {
        w.begin(u);
        TileRef t;
        while (ok && w.next(t)) {
          const uint32_t buf = job_i & 1u, aph = (job_i >> 1) & 1u;
          if (!mbar_wait_warp(smem_u32(&ctrl->acc_empty[buf]), aph ^ 1u, &ctrl->abort)) { ok = false; break; }
          tc_fence_after();
          const uint32_t idesc = idesc_bf16_f32(kTileRows, t.ng * kGran);
          const uint32_t d = tmem_base + buf * kTileCols;
          uint32_t acc = 0;
          for (int ks = 0; ks < p.ksteps; ++ks) {
            if (!mbar_wait_warp(smem_u32(&ctrl->full[stage]), phase, &ctrl->abort)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sb = stage_base + (uint32_t)stage * stage_bytes;
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < 4; ++k)
                umma_bf16_pair(d, smem_desc_sw128(sb + k * 32), smem_desc_sw128(sb + w_off + k * 32), idesc, k ? 1u : acc);
              umma_commit_pair(smem_u32(&ctrl->empty[stage]));    // frees the stage in both CTAs
            }
            __syncwarp();
            acc = 1;
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          if (elect_one()) umma_commit_pair(smem_u32(&ctrl->acc_full[buf]));       // wakes the epilogues of both CTAs
          __syncwarp();
          ++job_i;
        }
      }
    }
  } else {
    // ---------------- epilogue (both CTAs): thread = hidden row (x half of the columns) ---------------------
    const int q = warp & 3;                           // tensor-memory lane quarter this warp may read
    const int half = (warp - 2) >> 2;                 // which 32-column groups of a tile it takes
    const LogitsArgs& a = p.la;
    const uint32_t k0s = (uint32_t)a.seed, k1s = (uint32_t)(a.seed >> 32);
    const uint32_t c2 = (uint32_t)a.step, c3 = (uint32_t)(a.step >> 32);
    const size_t ldbg = (size_t)p.cb.V + p.cb.cap;
    uint32_t acc_empty_leader[2];
    acc_empty_leader[0] = map_to_cta(smem_u32(&ctrl->acc_empty[0]), 0);
    acc_empty_leader[1] = map_to_cta(smem_u32(&ctrl->acc_empty[1]), 0);
    UnitWalk w(p);
    uint32_t job_i = 0;
    bool ok = true;
    for (long long u = cluster_id; u < n_units && ok; u += n_clusters) {
      w.begin(u);
      const int strip = (int)(u - (long long)w.rt * p.strips);
      const int in_cta = q * 32 + lane;                // accumulator lanes beyond the CTA's rows hold nothing
      const int r = in_cta < p.cta_rows ? w.rt * kTileRows + (int)rank * p.cta_rows + in_cta : a.N;
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
      RowRed red; red.init();
      TileRef t;
      while (w.next(t)) {
        const uint32_t buf = job_i & 1u, aph = (job_i >> 1) & 1u;
        if (!mbar_wait(smem_u32(&ctrl->acc_full[buf]), aph, &ctrl->abort)) { ok = false; break; }
        tc_fence_after();
        int limit = 0;
        if (my_seq >= 0) limit = t.owner < 0 ? t.nvalid : (my_seq == t.owner ? min(t.nvalid, my_nvis - t.k0) : 0);
        const uint32_t tbase = tmem_base + ((uint32_t)(q * 32) << 16) + buf * kTileCols;
#pragma unroll 1
        for (int c0 = 32 * half; c0 < t.ng * kGran; c0 += 32 * GROUPS) {
          if (!__any_sync(0xffffffffu, limit > c0)) break;
          uint32_t v[32];
          tmem_ld32(tbase + c0, v);
          tmem_ld_wait();
          const int col0 = t.col0 + c0;
          if (GENERIC) {                                // sampling, or every logit stored
            if (a.select == Z2Z_SELECT_GUMBEL) sample_row32(v, limit - c0, col0, a.inv_temperature, (uint32_t)(a.row_base + r), c2, c3, k0s, k1s, red);
            if (a.logits_debug) {
#pragma unroll
              for (int x = 0; x < 32; ++x)
                if (c0 + x < limit) a.logits_debug[(size_t)r * ldbg + col0 + x] = __uint_as_float(v[x]);
            }
          }
          const int at = my_tgt - col0;                 // the row's target column, if it lies here and exists
          if (at >= 0 && at < 32 && at < limit - c0 && a.target_logit) a.target_logit[r] = pick32(v, at);
          fold_row32(v, limit - c0, col0, red);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty_leader[buf]);
        ++job_i;
      }
      // The two warps of a lane quarter merge their halves of the columns.  A wait that ran out in one
      // warp ends the loop for all of them, so that none is left alone at a barrier.
      if (GROUPS == 2) {
        ok = epilogue_all<32 * EW>(ok);
        if (ok && half == 1) s_red[in_cta] = red;
        ok = epilogue_all<32 * EW>(ok);
        if (ok && half == 0) red.merge(s_red[in_cta]);
      }
      if (ok && half == 0 && r < a.N) {
        LogitPartial* lp = reinterpret_cast<LogitPartial*>(a.lpart) + (size_t)r * p.strips + strip;
        lp->m = red.m; lp->s = red.s; lp->idx = red.idx; lp->gm = red.gm; lp->gidx = red.gidx;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctrl->abort) atomicOr(p.err, 1);
  cluster_sync_all();                               // nobody leaves while the pair's MMAs may read its memory
  if (warp == 2) tmem_dealloc_pair(tmem_base, 512);
}

// Eight lanes per row: merge the partial reductions of the strips, write the outputs.
__global__ void __launch_bounds__(256) k_prefill_merge(PrefillLogitsParams p) {
  pdl_wait();
  pdl_trigger();
  const LogitsArgs& a = p.la;
  const int r = blockIdx.x * (blockDim.x / 8) + (threadIdx.x >> 3), lane = threadIdx.x & 7;
  RowRed red; red.init();
  if (r < a.N) {
    const LogitPartial* lp = reinterpret_cast<const LogitPartial*>(a.lpart) + (size_t)r * p.strips;
    for (int g = lane; g < p.strips; g += 8) red.merge(load_partial(lp + g));
  }
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) {
    RowRed o;
    o.m = __shfl_xor_sync(0xffffffffu, red.m, off);
    o.s = __shfl_xor_sync(0xffffffffu, red.s, off);
    o.idx = __shfl_xor_sync(0xffffffffu, red.idx, off);
    o.gm = __shfl_xor_sync(0xffffffffu, red.gm, off);
    o.gidx = __shfl_xor_sync(0xffffffffu, red.gidx, off);
    red.merge(o);
  }
  if (lane != 0 || r >= a.N) return;
  if (a.lse) a.lse[r] = red.m + logf(red.s);
  if (a.argmax) a.argmax[r] = red.idx == 0x7fffffff ? -1 : red.idx;
  if (a.max_logit) a.max_logit[r] = red.m;
  if (a.sample) a.sample[r] = red.gidx == 0x7fffffff ? -1 : red.gidx;
}

}  // namespace

bool logits_tc_supported(int d, int dtype) { return dtype == Z2Z_DTYPE_BF16 && d % 64 == 0; }

long long prefill_logits_max_rows(size_t lpart_bytes, size_t plan_bytes, int strips) {
  long long by_part = (long long)(lpart_bytes / sizeof(LogitPartial)) / (strips < 1 ? 1 : strips);
  long long by_plan = (long long)(plan_bytes / (3 * sizeof(int32_t))) * kTileRows;
  long long m = by_part < by_plan ? by_part : by_plan;
  return m / kTileRows * kTileRows;
}

static int sm_count_prefill() {
  static int n_sm = 0;
  if (!n_sm) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (n_sm <= 0) n_sm = 148;
  }
  return n_sm;
}

static size_t l2_bytes_prefill() {
  static size_t l2 = 0;
  if (!l2) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev);
    l2 = v > 0 ? (size_t)v : ((size_t)64 << 20);
  }
  return l2;
}

// Number of column strips per row tile.  Two conditions:
//   * the hidden-row tiles that are in work at the same time must stay in the L2 cache, because a
//     pair re-reads its 256 x d tile for every column tile of its strip: n_clusters / strips tiles
//     of 512 d bytes within a third of the cache (with one strip at d = 4096 the 74 pairs keep
//     148 MB of tiles in work, more than the cache holds, and every column tile fetches its
//     hidden rows from HBM again: 0.92 instead of 1.15 PFLOP/s at 1.8e5 rows);
//   * the cost that the busiest cluster sweeps (rounds x cost of a strip, in the schedule's units) should
//     be low.  With fewer row tiles than kPrefillMaxStrips strips can spread over the clusters the
//     split goes on: 700 rows are three row tiles, of 24 strips each.
// The cheapest split; among equals the finest as long as every cluster has one unit (what the host cannot
// see, the hypertokens, then finds room), else the coarsest.
static int pick_strips(int row_tiles, int n_clusters, int d, int n_static, int cta_rows) {
  const size_t tile_bytes = (size_t)kTileRows * d * 2;
  const size_t budget = l2_bytes_prefill() / 3;
  int s_min = (int)(((size_t)n_clusters * tile_bytes + budget - 1) / budget);
  if (row_tiles < n_clusters) s_min = (int)(((size_t)row_tiles * tile_bytes + budget - 1) / budget);
  s_min = s_min < 1 ? 1 : (s_min > kPrefillMaxStrips ? kPrefillMaxStrips : s_min);
  const int spread = n_clusters / row_tiles;
  const int s_max = spread > kPrefillMaxStrips ? spread : kPrefillMaxStrips;
  int best = s_min;
  long long best_cost = -1;
  for (int s = s_min; s <= s_max; ++s) {
    const long long rounds = ((long long)row_tiles * s + n_clusters - 1) / n_clusters;
    const int g = (n_static + s - 1) / s;
    const long long cost = rounds * (4 * g + cta_rows / 8 * ((g + 3) / 4));
    if (best_cost < 0 || cost < best_cost || (cost == best_cost && s <= spread)) { best_cost = cost; best = s; }
  }
  return best;
}

static int cta_rows_of(int N) { return N > 192 ? 128 : ((N + 1) / 2 + 31) / 32 * 32; }

int prefill_logits_strips(int N, int d, int V) {
  return pick_strips((N + kTileRows - 1) / kTileRows, sm_count_prefill() / 2, d, (V + kGran - 1) / kGran,
                     cta_rows_of(N));
}

cudaError_t run_logits_prefill(const CbView& cb, const LogitsArgs& a, int32_t* plan, int* err_word, int strips_override,
                               Prof* prof, cudaStream_t s) {
  const int n_sm = sm_count_prefill();
  PrefillLogitsParams p{};
  p.cb = cb; p.la = a;
  p.ksteps = a.d / 64;
  p.row_tiles = (a.N + kTileRows - 1) / kTileRows;
  p.cta_rows = cta_rows_of(a.N);
  p.n_static = (cb.V + kGran - 1) / kGran;
  const int max_clusters = n_sm / 2;
  p.strips = strips_override > 0 ? strips_override : pick_strips(p.row_tiles, max_clusters, a.d, p.n_static, p.cta_rows);
  if (p.strips > p.n_static) p.strips = p.n_static;          // every strip gets at least one granule
  p.tile_lo = plan; p.tile_hi = plan + p.row_tiles; p.tile_nh = plan + 2 * p.row_tiles;
  p.err = err_word;
  if ((size_t)a.N * p.strips * sizeof(LogitPartial) > a.lpart_bytes) return cudaErrorMemoryAllocation;
  PrefillMaps maps;
  if (!make_tmap_bf16(&maps.h, a.hidden, a.N, a.d, p.cta_rows)) return cudaErrorInvalidValue;
  for (int i = 0; i < 4; ++i) {
    if (!make_tmap_bf16(&maps.w[0][i], a.WU, cb.V, a.d, 32 * (i + 1))) return cudaErrorInvalidValue;
    if (cb.cap == 0) maps.w[1][i] = maps.w[0][i];
    else if (!make_tmap_bf16(&maps.w[1][i], a.Uh, (long long)cb.B * cb.cap, a.d, 32 * (i + 1))) return cudaErrorInvalidValue;
  }
  const long long units = (long long)p.row_tiles * p.strips;
  const int clusters = units < max_clusters ? (int)units : max_clusters;
  const bool generic = a.select == Z2Z_SELECT_GUMBEL || a.logits_debug;
  cudaError_t e;
  {
    ProfScope ps(prof, kProfLogitsMerge, 1, s);
    if ((e = launch_pdl(k_prefill_plan, dim3(p.row_tiles), dim3(kTileRows), 0, s, p)) != cudaSuccess) return e;
  }
  {
    ProfScope ps(prof, kProfLogits, 1, s);
    const int stage = p.cta_rows * 128 + 16384;
    p.stages = kRingBytes / stage < kPrefillStages ? kRingBytes / stage : kPrefillStages;
    const size_t smem = 1024 + 4096 + (size_t)p.stages * stage;      // alignment; barriers and hand-over; ring
    auto kern = generic ? k_prefill_logits<true> : k_prefill_logits<false>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    if ((e = launch_pdl(kern, dim3(2 * clusters), dim3(prefill_threads(generic)), smem, s, p, maps)) != cudaSuccess) return e;
  }
  ProfScope ps(prof, kProfLogitsMerge, 1, s);
  return launch_pdl(k_prefill_merge, dim3((a.N + 31) / 32), dim3(256), 0, s, p);
}

}  // namespace z2z
