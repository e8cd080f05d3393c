// LZW decompression on the device (Section 2.1, property 2: the compressed stream decodes
// without a shipped codebook; Section 2.3 steps 11-12: the generated hypertoken stream is turned
// back into base tokens).
//
// Two kernels:
//   k_lzw_replay  rebuilds (or continues) each sequence's codebook from the code stream alone by
//                 replaying the online update once per code, a window of codes at a time.
//   k_lzw_expand  turns codes into base tokens with the codebook that is resident: an exclusive
//                 scan of phrase lengths gives every code its output offset, each thread then
//                 copies one phrase.  Blocks are (sequence, chunk of codes); a block finds its
//                 start offset by summing the lengths of the codes before its chunk.
#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_lzw_dev.cuh"

namespace z2z {

namespace {

constexpr int kExpandThreads = 256;
constexpr int kExpandChunk = 2048;          // codes per block

__device__ __forceinline__ int entry_first(const CbView& cb, int b, int code) {
  return code < cb.V ? code : cb.cons[((size_t)b * cb.cap + (code - cb.V)) * cb.M];
}
__device__ __forceinline__ int entry_len(const CbView& cb, int b, int code) {
  return code < cb.V ? 1 : (int)cb.len[(size_t)b * cb.cap + (code - cb.V)];
}

}  // namespace

// Replays the online update (Figure 1; Section 2.3 step 10) for codes[b][0 .. code_lens[b]).
// n_valid[b] = number of codes accepted; replay of a sequence stops at the first code that names
// no hypertoken (BAD_TOKEN; the state is the one after the last accepted code).
//
// One block per sequence; a window of LANES codes at a time (z2z_lzw_dev.cuh).  Code i asks
// for the entry (code i - 1, first token of code i), which depends on no other code of the window
// as long as both name entries from before it: the window ends before the first code that does not
// (the entry it names is known once the codes before it are in), and before the first lane whose bid
// for a slot lost.  The code that names the very entry it creates can only be the window's first.
//
// Bound by the latency of one window (the codes' first tokens and lengths from L2, one lookup, four
// barriers); one thread that replayed code by code took 170 ns per code with the table in shared
// memory and 260 with it in global memory.
template <int LANES, bool SMEM>
__global__ void __launch_bounds__(parse_threads(LANES)) k_lzw_replay(CbView cb, const int32_t* __restrict__ codes,
                                                              const int32_t* __restrict__ code_lens, int Tc_max,
                                                              int32_t* __restrict__ n_valid) {
  constexpr int WARPS = LANES / 32;
  extern __shared__ __align__(16) unsigned char s_parse[];
  __shared__ int s_code[LANES + 1], s_first[LANES + 1];   // [0]: the code before the window
  __shared__ uint8_t s_len[LANES + 4];
  __shared__ uint32_t s_known[WARPS], s_ins[WARPS];
  __shared__ int s_n1, s_bad0, s_prev0[3], s_lost[2];      // first loser of this window, of the next one
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int V = cb.V, M = cb.M, cap = cb.cap;
  int32_t* const cons = cb.cons + (size_t)b * cap * M;
  uint8_t* const elen = cb.len + (size_t)b * cap;
  const int n0 = cb.n[b];
  int Tc = code_lens ? code_lens[b] : Tc_max;
  Tc = Tc < 0 ? 0 : (Tc > Tc_max ? Tc_max : Tc);
  const int32_t* zs = codes + (size_t)b * Tc_max;
  ParseTable<SMEM> table;
  table.open(cb, b, n0, s_parse);
  if (tid == 0) {
    const int prev = cb.prev[b];
    s_prev0[0] = prev;
    s_prev0[1] = prev >= 0 ? entry_first(cb, b, prev) : -1;
    s_prev0[2] = prev >= 0 ? entry_len(cb, b, prev) : 0;
    s_n1 = n0;
    s_bad0 = 0;
    s_lost[0] = s_lost[1] = LANES;
  }
  __syncthreads();
  if (tid < LANES) {
    int n = n0, st = 0, base = 0;
    int z = tid < Tc ? zs[tid] : -1;
    int prev0 = s_prev0[0], first0 = s_prev0[1], plen0 = s_prev0[2];       // the code before the window
    for (int par = 0; base < Tc; par ^= 1) {
      const int z_ahead = base + LANES + tid < Tc ? zs[base + LANES + tid] : -1;
      const int i = base + tid;
      // ---- first token and length of every code, as far as known
      bool known = i < Tc && z >= 0 && z < V + n;
      int f = -1, l = 0;
      if (known) { f = entry_first(cb, b, z); l = entry_len(cb, b, z); }
      const bool self_ref = tid == 0 && z == V + n && prev0 >= 0 && plen0 < M && n < cap;   // the entry this code creates
      if (self_ref) { known = true; f = first0; l = plen0 + 1; }
      s_code[tid + 1] = z; s_first[tid + 1] = f; s_len[tid + 1] = (uint8_t)l;
      if (tid == 0) { s_code[0] = prev0; s_first[0] = first0; s_len[0] = (uint8_t)plen0; }
      const uint32_t v_known = __ballot_sync(0xffffffffu, known);
      if (lane == 0) s_known[warp] = v_known;
      parse_sync<LANES>();
      int limit = LANES;                       // first lane that is not known
#pragma unroll
      for (int k = WARPS - 1; k >= 0; --k)
        if (~s_known[k]) limit = k * 32 + __ffs((int)~s_known[k]) - 1;
      // the table in global memory keeps no keys to rebuild a row from later: a row is written at once,
      // which needs the previous code's row to be there
      if (!SMEM && limit > 1 && s_code[1] == V + n) limit = 1;
      const int pz = s_code[tid], pf = s_first[tid], pl = s_len[tid];
      bool want = tid < limit && pz >= 0 && pl < M && n < cap;
      int slot = -1;
      if (want) {
        const bool found = table.probe((uint32_t)pz, (uint32_t)f, slot) >= 0;
        if (found && self_ref) s_bad0 = 1;           // that phrase already has another id
        if (!found && slot < 0) st |= Z2Z_ST_TABLE_FULL;
        want = !found && slot >= 0;
      }
      parse_sync<LANES>();
      if (tid == 0) s_lost[par ^ 1] = LANES;           // (read ahead of this window's first barrier)
      if (want) {
        const int loser = table.bid(slot, tid, LANES);
        if (loser < LANES) atomicMin(&s_lost[par], loser);
      }
      const uint32_t v_ins = __ballot_sync(0xffffffffu, want);
      if (lane == 0) s_ins[warp] = v_ins;
      parse_sync<LANES>();
      uint32_t ins[WARPS];
#pragma unroll
      for (int k = 0; k < WARPS; ++k) ins[k] = s_ins[k];
      int stop = s_lost[par];
      if (stop > limit) stop = limit;
      if (s_bad0) stop = 0;
      const int room = cap - n;
      int made;
      const int new_before = parse_rank(ins, warp, lane, made);
      if (stop < LANES) made = parse_count_below(ins, stop);
      if (want) {
        if (tid < stop && new_before < room) {
          const int entry = n + new_before;
          table.settle(slot, (uint32_t)pz, (uint32_t)f, entry);
          int32_t* row = cons + (size_t)entry * M;
          row[0] = pf;                               // what later windows ask for; SMEM: the rest follows below
          if (!SMEM) {
            const int32_t* from = pz < V ? nullptr : cons + (size_t)(pz - V) * M;
            for (int j = 1; j < M; ++j) row[j] = j < pl ? from[j] : (j == pl ? f : -1);
          }
          elen[entry] = (uint8_t)(pl + 1);
        } else {
          table.withdraw(slot, tid);
        }
      }
      if (made > 0) {
        n += made < room ? made : room;
        if (n >= cap) st |= Z2Z_ST_CAP_FROZEN;
      }
      if (stop == 0) { st |= Z2Z_ST_BAD_TOKEN; break; }        // the window's first code names no hypertoken
      prev0 = s_code[stop]; first0 = s_first[stop]; plen0 = s_len[stop];
      base += stop;
      z = stop == LANES ? z_ahead : (base + tid < Tc ? zs[base + tid] : -1);
      parse_sync<LANES>();                             // rows, lengths and slots are there for the next window
    }
    if (tid == 0) {
      s_n1 = n;
      cb.n[b] = n;
      if (base > 0) cb.prev[b] = prev0;
      n_valid[b] = base;
    }
    if (st) atomicOr(&cb.status[b], st);
  }
  __syncthreads();
  const int n1 = s_n1;
  table.close(n0, n1);
  if (!SMEM) return;
  // constituent rows of the entries created here: walk back through the prefixes (each at most
  // M - 1 steps); only rows from before this call are read
  for (int e = n0 + tid; e < n1; e += blockDim.x) {
    int tok[kMaxM];
#pragma unroll
    for (int j = 0; j < kMaxM; ++j) tok[j] = -1;
    int pos = (int)elen[e] - 1, cur = e;
    for (int hop = 0; hop < kMaxM && pos > 0; ++hop) {
      const int p = (int)table.prefix_of(cur);
#pragma unroll
      for (int j = 0; j < kMaxM; ++j) if (j == pos) tok[j] = (int)table.token_of(cur);
      --pos;
      if (p < V) {
        if (pos == 0) tok[0] = p;
        break;
      }
      if (p - V < n0) {
#pragma unroll
        for (int j = 0; j < kMaxM; ++j) if (j <= pos) tok[j] = cons[(size_t)(p - V) * M + j];
        break;
      }
      cur = p - V;
    }
#pragma unroll
    for (int j = 0; j < kMaxM; ++j) if (j < M) cons[(size_t)e * M + j] = tok[j];
  }
}

// Block-wide exclusive scan of one int per thread (kExpandThreads threads); returns the
// thread's exclusive prefix, *total = sum over the block.
__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();                               // warp_sums free to overwrite
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kExpandThreads / 32; ++w) {
    int s = warp_sums[w];
    if (w < warp) before += s;
    all += s;
  }
  *total = all;
  return before + inc - v;
}

// Codes -> base tokens with the resident codebook.  grid = (chunks, B).  limit[b] (or code_lens,
// or Tc_max) bounds the codes of sequence b; expansion stops at the first code that is not below
// V + n_b (BAD_TOKEN) and at T_out_max tokens (OUTPUT_TRUNCATED; token_lens[b] is then T_out_max).
// Eight blocks per SM, so that 1024 sequences are there at once (40 registers leave six: 9.6 us instead of 7.0 for 64
// tokens each); six codes ahead fit the 32 registers.
__global__ void __launch_bounds__(kExpandThreads, 8) k_lzw_expand(
    CbView cb, const int32_t* __restrict__ codes, const int32_t* __restrict__ code_lens,
    const int32_t* __restrict__ limit, int Tc_max, int32_t* __restrict__ tokens,
    int32_t* __restrict__ token_lens, int T_out_max) {
  __shared__ int warp_sums[kExpandThreads / 32];
  __shared__ int s_first_bad;
  const int b = blockIdx.y;
  const int tid = threadIdx.x;
  int Tc = code_lens ? code_lens[b] : Tc_max;
  Tc = Tc < 0 ? 0 : (Tc > Tc_max ? Tc_max : Tc);
  const int lim = limit ? (limit[b] < Tc ? limit[b] : Tc) : Tc;
  const int n = cb.n[b];
  const int32_t* zs = codes + (size_t)b * Tc_max;
  const int lo = blockIdx.x * kExpandChunk;
  if (lo > lim) return;                          // the block that holds position `lim` reports the length
  const int hi = lo + kExpandChunk < lim ? lo + kExpandChunk : lim;
  if (tid == 0) s_first_bad = 0x7fffffff;
  __syncthreads();
  // codes before this chunk: total length and validity
  int before = 0;
  constexpr int kAhead = 6;                      // codes a thread looks at together: their lengths are a second round of loads
  for (int i0 = tid; i0 < lo; i0 += kAhead * kExpandThreads) {
    int z[kAhead], l[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) z[u] = i0 + u * kExpandThreads < lo ? zs[i0 + u * kExpandThreads] : 0;
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      l[u] = i0 + u * kExpandThreads < lo && z[u] >= 0 && z[u] < cb.V + n ? entry_len(cb, b, z[u]) : 0;
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      before += l[u];
      if (z[u] < 0 || z[u] >= cb.V + n) atomicMin(&s_first_bad, i0 + u * kExpandThreads);
    }
  }
  int total = 0;
  block_exclusive_scan(before, warp_sums, &total);
  __syncthreads();
  if (s_first_bad != 0x7fffffff) return;         // an earlier block holds the end of the valid prefix
  int offset = total;
  int32_t* out = tokens + (size_t)b * T_out_max;
  bool truncated = false;
  int end_pos = hi;                              // first position this block does not expand
  for (int c0 = lo; c0 < hi; c0 += kExpandThreads) {
    const int i = c0 + tid;
    int z = -1, l = 0;
    if (i < hi) {
      z = zs[i];
      if (z < 0 || z >= cb.V + n) { atomicMin(&s_first_bad, i); z = -1; }
      else l = entry_len(cb, b, z);
    }
    __syncthreads();
    const int first_bad = s_first_bad;
    if (i >= first_bad) l = 0;                   // nothing at or after the first bad code is written
    int sum = 0;
    const int ex = block_exclusive_scan(l, warp_sums, &sum);
    if (l > 0) {
      const int at = offset + ex;
      if (z < cb.V) {
        if (at < T_out_max) out[at] = z; else truncated = true;
      } else {
        const int32_t* src = cb.cons + ((size_t)b * cb.cap + (z - cb.V)) * cb.M;
        for (int j = 0; j < l; ++j) {
          if (at + j < T_out_max) out[at + j] = src[j]; else truncated = true;
        }
      }
    }
    offset += sum;
    if (first_bad != 0x7fffffff) { end_pos = first_bad; break; }
  }
  const int any_trunc = __syncthreads_or(truncated ? 1 : 0);
  const bool bad = end_pos < hi || (s_first_bad != 0x7fffffff);
  // exactly one block owns the end of the expanded prefix: the one where expansion stopped at a
  // bad code, or the one whose chunk holds position `lim`
  const bool owns_end = bad || (lim < lo + kExpandChunk);
  if (tid == 0) {
    int st = 0;
    if (any_trunc) st |= Z2Z_ST_OUTPUT_TRUNCATED;
    if (bad) st |= Z2Z_ST_BAD_TOKEN;           // (a replay that stopped early has set it already)
    if (st) atomicOr(&cb.status[b], st);
    if (owns_end) token_lens[b] = offset < T_out_max ? offset : T_out_max;
  }
}

cudaError_t launch_lzw_decode(const CbView& cb, const int32_t* codes, const int32_t* code_lens,
                              int Tc_max, int replay, int32_t* n_valid, int32_t* tokens,
                              int32_t* token_lens, int T_out_max, cudaStream_t s) {
  if (replay) {
    const ParseLaunch pl = parse_launch(cb, Tc_max);             // as for prompt compression
    auto kern = pl.lanes == kParseLanes ? (pl.smem_bytes ? k_lzw_replay<kParseLanes, true> : k_lzw_replay<kParseLanes, false>)
                                        : (pl.smem_bytes ? k_lzw_replay<kParseLanesMany, true> : k_lzw_replay<kParseLanesMany, false>);
    if (pl.smem_bytes) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem_bytes);
      if (e != cudaSuccess) return e;
    }
    kern<<<cb.B, parse_threads(pl.lanes), pl.smem_bytes, s>>>(cb, codes, code_lens, Tc_max, n_valid);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  dim3 grid(Tc_max / kExpandChunk + 1, cb.B);
  k_lzw_expand<<<grid, kExpandThreads, 0, s>>>(cb, codes, code_lens, replay ? n_valid : nullptr,
                                               Tc_max, tokens, token_lens, T_out_max);
  return cudaGetLastError();
}

}  // namespace z2z
