// LZW codebook kernels: session reset, prompt compression, online update.
//
// The codebook of a sequence is an open-addressing hash table in global memory keyed by (prefix
// code, next base token), probed linearly from an even slot; the online update probes it with one
// warp (one coalesced 256-byte load of 32 consecutive slots followed by a ballot).  Entries are
// never deleted and an insert always takes the first empty slot in probe order, so an empty slot
// proves absence.
// Prompt compression gives every sequence a block (paper Section 2.4: compression is per document)
// that parses a window of positions at a time.
#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_lzw_dev.cuh"
#include "z2z_sm100.cuh"

namespace z2z {

// Session reset.  An empty slot and an absent constituent are all ones, and the workspace plan puts the two
// tables behind one another and the lengths behind them, each from a 256-byte boundary: 16-byte stores.
// zero / n_zero: words of the hyper-encoder's result matrix that have to be zero before its first pass.
__global__ void k_codebook_clear(CbView cb, uint4* zero, size_t n_zero) {
  uint4* const ones = reinterpret_cast<uint4*>(cb.hash);
  uint4* const lens = reinterpret_cast<uint4*>(cb.len);
  const size_t n_ones = (size_t)(lens - ones), n_lens = (size_t)(reinterpret_cast<uint4*>(cb.n) - lens);
  const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = tid; i < n_ones; i += stride) ones[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  for (size_t i = tid; i < n_zero; i += stride) zero[i] = make_uint4(0u, 0u, 0u, 0u);
  for (size_t i = tid; i < n_lens; i += stride) lens[i] = make_uint4(0u, 0u, 0u, 0u);
  for (size_t i = tid; i < (size_t)cb.B; i += stride) {
    cb.n[i] = 0; cb.prev[i] = -1; cb.status[i] = 0; cb.n_emb[i] = 0; cb.n_emb[cb.B + i] = 0;
  }
}
static_assert(kEmptySlot == ~0ull, "an empty slot is all ones");

// All threads of the block: constituent rows of entries [n0, n1), whose first word is the position of their first token:
// tokens [start, start + len), -1 padded.  (AT_ONCE entries of a thread at a time: their loads do not wait for one another)
template <int AT_ONCE>
__device__ __forceinline__ void write_rows(const CbView& cb, int b, const int32_t* __restrict__ x, int n0, int n1) {
  const int V = cb.V, M = cb.M, cap = cb.cap;
  for (int e0 = n0 + (int)threadIdx.x; e0 < n1; e0 += AT_ONCE * (int)blockDim.x) {
    int start[AT_ONCE], L[AT_ONCE], tok[AT_ONCE][kMaxM];
#pragma unroll
    for (int u = 0; u < AT_ONCE; ++u) {
      const int e = e0 + u * (int)blockDim.x;
      start[u] = L[u] = 0;
      if (e < n1) { start[u] = cb.cons[((size_t)b * cap + e) * M]; L[u] = cb.len[(size_t)b * cap + e]; }
    }
#pragma unroll
    for (int u = 0; u < AT_ONCE; ++u)
#pragma unroll
      for (int j = 0; j < kMaxM; ++j) tok[u][j] = j < L[u] ? x[start[u] + j] : -1;
#pragma unroll
    for (int u = 0; u < AT_ONCE; ++u) {
      const int e = e0 + u * (int)blockDim.x;
      if (e >= n1) break;
      int32_t* row = cb.cons + ((size_t)b * cap + e) * M;
#pragma unroll
      for (int j = 0; j < kMaxM; ++j)
        if (j < M) row[j] = j < L[u] && (unsigned)tok[u][j] >= (unsigned)V ? 0 : tok[u][j];
    }
  }
}

// Prompt compression (Section 2.1; Section 2.3 step 2).  One block per sequence; a window of
// LANES input positions at a time (z2z_lzw_dev.cuh).
//
// Each lane follows the longest match from its own position (at most M - 1 dependent lookups).
// Which positions start a phrase is a walk position -> position + match length: inside a warp by
// pointer doubling (five rounds carry the set of visited lanes and the exit), across the
// warps by looking up the exit of one as the entry of the next (a match is at most kMaxM long, so
// only the first kMaxM lanes of a warp can be entered: a warp's exits fit one word, four bits each).
//
// Bound by the latency of one window (a few dependent shared-memory lookups, ten shuffles, three
// barriers).  One thread that walks the chain token by token takes 180 ns per token with the table in
// shared memory, 220 with it in global memory: four texts of 32768 tokens (cap 16384), to codes and back
// with both session resets, 9.6 ms; in windows, here and in the replay, 0.55.
// At most 64 registers: narrow windows are for calls of many sequences, seven per SM at 1024.
template <int LANES, bool SMEM>
__global__ void __launch_bounds__(parse_threads(LANES), 1024 / parse_threads(LANES)) k_lzw_encode(CbView cb, const int32_t* __restrict__ tokens,
                                                              const int32_t* __restrict__ lens, int T_max,
                                                              int32_t* __restrict__ codes,
                                                              int32_t* __restrict__ code_lens,
                                                              int32_t* __restrict__ entries_after) {
  constexpr int WARPS = LANES / 32, kTokRing = 2 * LANES;      // (a window's tokens and a match behind it fit the ring)
  extern __shared__ __align__(16) unsigned char s_parse[];
  __shared__ int s_tok[kTokRing];                    // token of position p at p mod kTokRing
  __shared__ uint32_t s_exit[WARPS];           // per warp, four bits per entry lane: the next warp's entry lane
  __shared__ ParseVotes<WARPS> s_votes;
  __shared__ int s_prev, s_n1, s_st, s_lost[2];      // first loser of this window, of the next one
  static_assert(kMaxM * 4 <= 32, "a warp's exits fit one word");
  constexpr uint32_t kInputEnd = 15;           // instead of an entry lane
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int V = cb.V, M = cb.M, cap = cb.cap;
  const int n0 = cb.n[b];
  int T = lens ? lens[b] : T_max;
  T = T < 0 ? 0 : (T > T_max ? T_max : T);
  const int32_t* x = tokens + (size_t)b * T_max;
  ParseTable<SMEM> table;
  table.open(cb, b, n0, s_parse);
  if (tid == 0) { s_prev = -1; s_st = 0; s_n1 = n0; s_lost[0] = s_lost[1] = LANES; }
  __syncthreads();
  if (tid < LANES) {
    int32_t* out = codes + (size_t)b * T_max;
    int32_t* aft = entries_after ? entries_after + (size_t)b * T_max : nullptr;
    int n = n0, n_out = 0, st = 0;
    int loaded = 0;                                  // tokens already in s_tok
    int ahead = tid < T ? x[tid] : 0;                // token loaded + tid
    for (int p0 = 0, par = 0; p0 < T; par ^= 1) {    // p0: a phrase starts here
      // Positions below p0 + LANES + kMaxM are looked at; the ring is filled as far as it goes, so
      // that a token has been on its way for a window before it is stored.  (A window moves p0 by 257 on
      // average where no phrase repeats in it: with nothing in reserve every other window would wait for
      // the last few tokens.  s_tok is only read ahead of a window's second barrier, so that the tokens
      // of the last window may be overwritten here.)
      const int need = p0 + LANES + kMaxM < T ? p0 + LANES + kMaxM : T;
      const int room_end = p0 + kTokRing < T ? p0 + kTokRing : T;
      do {
        const int cnt = room_end - loaded < LANES ? room_end - loaded : LANES;
        if (tid < cnt) {
          int c = ahead;
          if ((unsigned)c >= (unsigned)V) { st |= Z2Z_ST_BAD_TOKEN; c = 0; }     // not a base token
          s_tok[(loaded + tid) & (kTokRing - 1)] = c;
        }
        loaded += cnt;
        ahead = loaded + tid < T ? x[loaded + tid] : 0;
      } while (loaded < need);
      parse_sync<LANES>();
      // ---- longest match from every position of the window
      const int q = p0 + tid;
      const bool live = q < T;
      int w = -1, len = 1, slot = -1, c = 0;
      bool miss = false;
      if (live) {
        w = s_tok[q & (kTokRing - 1)];
        int next = s_tok[(q + 1) & (kTokRing - 1)];            // (the ring's slot is there whether or not its token is)
        while (len < M && q + len < T) {
          c = next;
          next = s_tok[(q + len + 1) & (kTokRing - 1)];
          const int e = table.probe((uint32_t)w, (uint32_t)c, slot);
          if (e < 0) { miss = true; break; }
          w = V + e; ++len;
        }
      }
      // ---- positions on the chain
      uint32_t visited = live ? 1u << lane : 0u;
      int to = live ? lane + len : lane;
#pragma unroll
      for (int r = 0; r < 5; ++r) {
        const uint32_t v2 = __shfl_sync(0xffffffffu, visited, to & 31);
        const int t2 = __shfl_sync(0xffffffffu, to, to & 31);
        if (to < 32) { visited |= v2; to = t2; }
      }
      const uint32_t exits = __reduce_or_sync(0xffffffffu, lane < kMaxM ? (to >= 32 ? (uint32_t)(to - 32) : kInputEnd) << (4 * lane) : 0u);
      if (lane == 0) s_exit[warp] = exits;
      parse_sync<LANES>();
      if (tid == 0) s_lost[par ^ 1] = LANES;         // (read ahead of this window's first barrier)
      uint32_t at = 0, entered = kInputEnd;          // entry lane of warp k, and of this thread's
#pragma unroll
      for (int k = 0; k < WARPS; ++k) {
        if (k == warp) entered = at;
        if (at != kInputEnd) at = (s_exit[k] >> (4 * at)) & 15u;
      }
      const uint32_t chain = __shfl_sync(0xffffffffu, visited, (int)entered);
      const bool on = entered != kInputEnd && ((chain >> lane) & 1u);
      // ---- new phrases of the chain bid for their slots
      const bool ins = on && miss && n < cap && slot >= 0;
      if (on && miss && n < cap && slot < 0) st |= Z2Z_ST_TABLE_FULL;
      if (ins) {
        const int loser = table.bid(slot, tid, LANES);
        if (loser < LANES) atomicMin(&s_lost[par], loser);
      }
      const uint32_t v_on = __ballot_sync(0xffffffffu, on), v_ins = __ballot_sync(0xffffffffu, ins);
      if (lane == 0) { s_votes.on[warp] = v_on; s_votes.ins[warp] = v_ins; }
      parse_sync<LANES>();
      const ParseVotes<WARPS> votes = s_votes;
      const int stop = s_lost[par];                  // lanes below it are final
      const int room = cap - n;
      int made, emitted;
      const int new_before = parse_rank(votes.ins, warp, lane, made), on_before = parse_rank(votes.on, warp, lane, emitted);
      if (stop < LANES) { made = parse_count_below(votes.ins, stop); emitted = parse_count_below(votes.on, stop); }
      if (ins) {
        if (tid < stop && new_before < room) {       // the phrase and its next token: input from q on (expanded below)
          const int entry = n + new_before;
          table.settle(slot, (uint32_t)w, (uint32_t)c, entry);
          cb.cons[((size_t)b * cap + entry) * M] = q;
          cb.len[(size_t)b * cap + entry] = (uint8_t)(len + 1);
        } else {
          table.withdraw(slot, tid);
        }
      }
      if (on && tid < stop) {
        const int pos = n_out + on_before;
        out[pos] = w;
        const int mine_too = new_before + (ins ? 1 : 0);
        if (aft) aft[pos] = n + (mine_too < room ? mine_too : room);
        if (on_before == emitted - 1) s_prev = w;
      }
      if (made > 0) {
        n += made < room ? made : room;
        if (n >= cap) st |= Z2Z_ST_CAP_FROZEN;
      }
      n_out += emitted;
      p0 = stop < LANES ? p0 + stop : at == kInputEnd ? T : p0 + LANES + (int)at;
      // (the barrier at the head of the next window orders these writes before its lookups; s_votes
      // and s_exit are rewritten behind further barriers)
    }
    if (st) atomicOr(&s_st, st);
    if (tid == 0) { code_lens[b] = n_out; s_n1 = n; }
  }
  __syncthreads();
  if (tid == 0) {
    cb.n[b] = s_n1;
    if (s_prev >= 0) cb.prev[b] = s_prev;
    if (s_st) atomicOr(&cb.status[b], s_st);
  }
  table.close(n0, s_n1);
  if (write_back_four(n0, s_n1)) write_rows<4>(cb, b, x, n0, s_n1);
  else write_rows<1>(cb, b, x, n0, s_n1);
}

// Online update with one new code per sequence (Figure 1; Section 2.3 step 10).
// none_sits_out: a code equal to Z2Z_CODE_NONE marks a sequence that takes no part in this step.
__global__ void __launch_bounds__(128) k_lzw_step(CbView cb, const int32_t* new_codes, const uint8_t* active,
                                                  int none_sits_out, int32_t* new_entry) {
  sm100::pdl_wait();
  sm100::pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (b >= cb.B) return;
  if ((active && !active[b]) || (none_sits_out && new_codes[b] == Z2Z_CODE_NONE)) {
    if (lane == 0 && new_entry) new_entry[b] = -1;
    return;
  }
  const int created = warp_lzw_step(cb, b, new_codes[b]);
  if (lane == 0 && new_entry) new_entry[b] = created;
}

cudaError_t launch_codebook_clear(const CbView& cb, void* zero, size_t zero_bytes, cudaStream_t s) {
  size_t work = (size_t)(reinterpret_cast<char*>(cb.len) - reinterpret_cast<char*>(cb.hash)) / 16;
  if (work < zero_bytes / 16) work = zero_bytes / 16;
  int blocks = (int)((work + 255) / 256);
  if (blocks > 148 * 8) blocks = 148 * 8;
  if (blocks < 1) blocks = 1;
  k_codebook_clear<<<blocks, 256, 0, s>>>(cb, reinterpret_cast<uint4*>(zero), zero_bytes / 16);
  return cudaGetLastError();
}

// The wide window while at most two sequences share an SM: with 1024 sequences its blocks ran in two waves (cap
// 1024, 200 tokens: 106 us, narrow 29; 49 with a warp or a thread per sequence).  The table goes to shared
// memory when it fits for all sequences of an SM at once - in waves, 1024 sequences of cap 16384 took 173 us and
// 263 for a second call, which brings the codebooks in, from global memory 43 and 13 - and when the call is long
// enough to repay bringing it in: 16 tokens of one sequence, cap 16384, second call 19 against 10 us.
ParseLaunch parse_launch(const CbView& cb, int T) {
  static int n_sm = 0;
  if (!n_sm) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (n_sm <= 0) n_sm = 148;
  }
  const int per_sm = (cb.B + n_sm - 1) / n_sm;
  ParseLaunch p{per_sm > 2 ? kParseLanesMany : kParseLanes, 0};
  const size_t bytes = parse_smem_bytes(cb.n_slots, cb.cap), fixed = 4096;      // fixed: the kernels' own arrays and the block's reserve
  const bool fits = cb.cap <= kParseSmemMaxCap && (per_sm == 1 || per_sm * (bytes + fixed) <= (size_t)227 * 1024);
  if (fits && (long long)T * 512 >= cb.n_slots) p.smem_bytes = bytes;
  return p;
}

cudaError_t launch_lzw_encode(const CbView& cb, const int32_t* tokens, const int32_t* lens,
                              int T_max, int32_t* codes, int32_t* code_lens,
                              int32_t* entries_after, cudaStream_t s) {
  const ParseLaunch pl = parse_launch(cb, T_max);
  auto kern = pl.lanes == kParseLanes ? (pl.smem_bytes ? k_lzw_encode<kParseLanes, true> : k_lzw_encode<kParseLanes, false>)
                                      : (pl.smem_bytes ? k_lzw_encode<kParseLanesMany, true> : k_lzw_encode<kParseLanesMany, false>);
  if (pl.smem_bytes) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem_bytes);
    if (e != cudaSuccess) return e;
  }
  kern<<<cb.B, parse_threads(pl.lanes), pl.smem_bytes, s>>>(cb, tokens, lens, T_max, codes, code_lens, entries_after);
  return cudaGetLastError();
}

cudaError_t launch_lzw_step(const CbView& cb, const int32_t* new_codes, const uint8_t* active,
                            int none_sits_out, int32_t* new_entry, cudaStream_t s) {
  int wpb = 4;
  return launch_pdl(k_lzw_step, dim3((cb.B + wpb - 1) / wpb), dim3(wpb * 32), 0, s, cb, new_codes, active, none_sits_out, new_entry);
}

}  // namespace z2z
