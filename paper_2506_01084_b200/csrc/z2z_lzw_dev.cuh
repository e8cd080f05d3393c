// Warp-level device functions of the LZW codebook, shared by the LZW kernels and by the fused
// decode-step update kernel.  All 32 lanes of a warp call these together for one sequence.
#pragma once
#include "z2z_common.cuh"

namespace z2z {

// Result of a warp probe.
struct Probe {
  int found;        // entry number, or -1
  int slot;         // if absent: first empty slot in probe order (-1: table full)
};

// First slot of the probe sequence of (prefix, token): linear probing from an even slot, so that
// a single thread can walk the sequence two slots (16 bytes) at a time and a warp can look at a
// window of kWindow consecutive slots at once.  Entries are never deleted and an insert takes the
// first empty slot of the sequence, so an empty slot proves that the key is absent.
__device__ __forceinline__ int probe_start(int n_slots, uint32_t prefix, uint32_t token) {
  return (int)(hash_pair(prefix, token) & (uint32_t)(n_slots - 1)) & ~1;
}

// All 32 lanes must call this together: lane l looks at slot (start + l) of the sequence.
__device__ __forceinline__ Probe warp_probe(const unsigned long long* __restrict__ table,
                                            int n_slots, uint32_t prefix, uint32_t token) {
  const int lane = threadIdx.x & 31;
  const unsigned long long key = pack_slot(prefix, token, 0) >> 16;
  int at = probe_start(n_slots, prefix, token);
  Probe r{-1, -1};
  for (int it = 0; it < n_slots / kWindow; ++it) {          // bounded: at most the whole table
    unsigned long long s = table[(at + lane) & (n_slots - 1)];
    unsigned hit = __ballot_sync(0xffffffffu, (s >> 16) == key && s != kEmptySlot);
    if (hit) {
      int src = __ffs(hit) - 1;
      unsigned long long v = __shfl_sync(0xffffffffu, s, src);
      r.found = (int)(v & 0xffffu);
      return r;
    }
    unsigned empty = __ballot_sync(0xffffffffu, s == kEmptySlot);
    if (empty) { r.slot = (at + __ffs(empty) - 1) & (n_slots - 1); return r; }
    at = (at + kWindow) & (n_slots - 1);
  }
  return r;
}

// The part of a sequence's state that the update needs and that does not depend on the new code;
// a caller that still has to compute the code can load it ahead.  ptok: base token `lane` of the
// previous phrase (-1 beyond its length), so that writing a new entry needs no further load.
struct LzwPrev { int n, prev, plen, ptok; };
__device__ __forceinline__ LzwPrev warp_lzw_load(const CbView& cb, int b) {
  const int lane = threadIdx.x & 31;
  LzwPrev s;
  s.n = cb.n[b];
  s.prev = cb.prev[b];
  s.plen = 0;
  s.ptok = -1;
  if (s.prev >= 0) {
    if (s.prev < cb.V) {
      s.plen = 1;
      if (lane == 0) s.ptok = s.prev;
    } else {
      const size_t e = (size_t)b * cb.cap + (s.prev - cb.V);
      if (lane < cb.M) s.ptok = cb.cons[e * cb.M + lane];      // -1 padded behind the phrase
      s.plen = (int)cb.len[e];
    }
  }
  return s;
}
// Write entry k = phrase(prev) ++ c from the previous phrase's tokens held by the lanes; returns the
// token this lane wrote (-1: padding, or a lane beyond M).
__device__ __forceinline__ int warp_write_entry_from(const CbView& cb, int b, int k, const LzwPrev& s, int c) {
  const int lane = threadIdx.x & 31;
  int v = -1;
  if (lane < cb.M) {
    if (lane < s.plen) v = s.ptok;
    else if (lane == s.plen) v = c;
    cb.cons[((size_t)b * cb.cap + k) * cb.M + lane] = v;
  }
  if (lane == 0) cb.len[(size_t)b * cb.cap + k] = (uint8_t)(s.plen + 1);
  return v;
}
// Online update of sequence b with the newly selected code z (Figure 1; Section 2.3 step 10).
// Candidate entry = phrase(prev) ++ first(phrase(z)); returns the entry created, or -1.
// A code that names no existing (or about-to-exist) hypertoken raises BAD_TOKEN and leaves the
// sequence untouched.
// new_tok (optional): base token `lane` of the entry created (-1 if none / padding).
__device__ __forceinline__ int warp_lzw_step(const CbView& cb, int b, int z, const LzwPrev& s,
                                             int* new_tok = nullptr) {
  const int lane = threadIdx.x & 31;
  if (new_tok) *new_tok = -1;
  unsigned long long* table = cb.hash + (size_t)b * cb.n_slots;
  const int n = s.n;
  const int prev = s.prev;
  int created = -1;
  int st = 0;
  bool ok = !(z < 0 || z > cb.V + n);
  const int plen = s.plen;
  const bool self_ref = ok && (z == cb.V + n);       // the code this very step would create
  if (self_ref && !(prev >= 0 && plen < cb.M && n < cb.cap)) ok = false;
  if (ok) {
    int first;
    if (self_ref) first = prev < cb.V ? prev : cb.cons[((size_t)b * cb.cap + (prev - cb.V)) * cb.M];
    else first = z < cb.V ? z : cb.cons[((size_t)b * cb.cap + (z - cb.V)) * cb.M];
    if (prev >= 0 && plen < cb.M && n < cb.cap) {
      Probe p = warp_probe(table, cb.n_slots, (uint32_t)prev, (uint32_t)first);
      if (p.found < 0) {
        if (p.slot >= 0) {
          if (lane == 0) table[p.slot] = pack_slot((uint32_t)prev, (uint32_t)first, (uint32_t)n);
          const int wrote = warp_write_entry_from(cb, b, n, s, first);
          if (new_tok) *new_tok = wrote;
          created = n;
          if (n + 1 >= cb.cap) st |= Z2Z_ST_CAP_FROZEN;
        } else {
          st |= Z2Z_ST_TABLE_FULL;
        }
      } else if (self_ref) {
        ok = false;                                    // that phrase already has another id
      }
    }
  }
  if (lane == 0) {
    if (!ok) {
      st |= Z2Z_ST_BAD_TOKEN;                          // state stays as it was
    } else {
      cb.prev[b] = z;
      if (created >= 0) cb.n[b] = n + 1;
    }
    if (st) atomicOr(&cb.status[b], st);
  }
  return ok ? created : -1;
}

__device__ __forceinline__ int warp_lzw_step(const CbView& cb, int b, int z) {
  return warp_lzw_step(cb, b, z, warp_lzw_load(cb, b));
}

// ---------------------------------------------------------------------------------------------
// Windowed parsing, shared by prompt compression and by replay of a code stream.
//
// Both are defined as a chain of one dictionary lookup per token or code, but the dictionary
// changes little while a window of them is looked at: LANES threads look up LANES starting
// points at once in the dictionary as it was before the window, the results that lie on the chain
// are picked out, and only the new phrases of the chain are inserted.  A lookup is invalid only if
// an earlier phrase of the same window inserted exactly the key that it missed; such a lane shares
// its first empty slot with the earlier lane, so one atomicMin of the lane number per new phrase on
// that slot finds it (a loser may also be a different key whose probe sequence ends in the same
// slot; it is treated the same).  The window then ends before the first loser, which is looked up
// again; the lowest lane never loses, so every window makes progress.  Whoever of two bidders comes
// second learns of the other from the atomic and reports the higher lane of both: the lowest lane
// reported is the second lowest bidder of some slot, that is the first loser, known one barrier after the bids.
//
// ParseTable holds the dictionary during the parse.
//   SMEM  (codebooks of at most kParseSmemMaxCap entries): the slot array lies in shared memory as
//         4-byte words (15-bit tag << 16 | entry, four slots per 16-byte load) with the full keys
//         beside it (6 bytes per entry): 224 KB at 16384 entries, where the 8-byte slots of the
//         codebook itself would take 256.  New entries go to the codebook's own hash table at the end.
//   else  the codebook's hash table in global memory is used in place (two slots per 16-byte load).
// ---------------------------------------------------------------------------------------------
// A window of 256 costs little more than one of 128 (two warps per scheduler hide each other's latencies)
// and moves 216 tokens on in long repetitive text where 128 moved 122; 512 would gain there and lose
// where phrases repeat sooner (vocabulary 32064: 93 tokens either way).  Where more than two sequences share an
// SM, its warps have other sequences to turn to and narrow windows leave room for all blocks at once.
constexpr int kParseLanes = 256;          // starting points looked up at once
constexpr int kParseLanesMany = 64;       // ... with many sequences
constexpr int kParseSmemMaxCap = 16384;
constexpr int parse_threads(int lanes) { return 2 * lanes; }      // the other warps only help to fill and to write back

inline size_t parse_smem_bytes(int n_slots, int cap) { return (size_t)n_slots * 4 + (size_t)(cap + (cap & 1)) * 6; }

// Barrier among the parsing threads only.
template <int LANES>
__device__ __forceinline__ void parse_sync() { asm volatile("bar.sync 1, %0;" ::"n"(LANES) : "memory"); }

// Entries [n0, n1) are written back four of a thread at a time where a thread has more than one.  (The code that does it takes
// longer to fetch than one entry takes: 1024 sequences of 200 tokens, M = 2, 16.4 us with it and 14.4 without;
// 400 of 2000 tokens, M = 5, 106 and 120.)
__device__ __forceinline__ bool write_back_four(int n0, int n1) { return n1 - n0 > (int)blockDim.x; }

template <bool SMEM>
struct ParseTable {
  unsigned long long* hash;   // this sequence's table of the codebook
  int n_slots;
  uint32_t* tab;              // SMEM: [n_slots], all-ones = empty
  uint32_t* key0;             // SMEM: [cap] prefix | (token & 0xff) << 24
  uint16_t* key1;             // SMEM: [cap] token >> 8

  static __device__ __forceinline__ uint32_t mix(uint32_t prefix, uint32_t token) {
    return prefix * 0x9E3779B1u ^ hash_token_part(token);
  }
  // The slot index takes bits 13 and up of the mix, the tag the 13 bits below and the top two.
  static __device__ __forceinline__ uint32_t tag_of(uint32_t h) { return (h & 0x1fffu) | ((h >> 30) << 13); }       // below 2^15

  // Entry of (prefix, token), or -1 and the first empty slot of its probe sequence (-1: table full).
  __device__ __forceinline__ int probe(uint32_t prefix, uint32_t token, int& slot) const {
    slot = -1;
    if (SMEM) {
      const uint32_t h = mix(prefix, token), tag = tag_of(h);
      const uint32_t k0 = prefix | (token << 24), k1 = token >> 8;
      uint32_t at = (h >> 13) & (uint32_t)(n_slots - 4);
      for (int it = 0; it < n_slots; it += 4) {                    // bounded: at most the whole table
        // all four slots at once, as bit masks: lanes of a warp differ in where their key or their gap lies
        const uint4 g = *reinterpret_cast<const uint4*>(tab + at);
        const uint32_t gap = (g.x == ~0u ? 1u : 0u) | (g.y == ~0u ? 2u : 0u) | (g.z == ~0u ? 4u : 0u) | (g.w == ~0u ? 8u : 0u);
        uint32_t hit = (g.x >> 16 == tag ? 1u : 0u) | (g.y >> 16 == tag ? 2u : 0u) | (g.z >> 16 == tag ? 4u : 0u) |
                       (g.w >> 16 == tag ? 8u : 0u);               // (an empty slot's tag is never one of a key's)
        while (hit) {
          const uint32_t v = (hit & 1u) ? g.x : (hit & 2u) ? g.y : (hit & 4u) ? g.z : g.w;
          const int e = (int)(v & 0xffffu);
          if ((key0[e] == k0) & (key1[e] == (uint16_t)k1)) return e;      // (both loads under way)
          hit &= hit - 1;
        }
        if (gap) { slot = (int)at + __ffs((int)gap) - 1; return -1; }
        at = (at + 4) & (uint32_t)(n_slots - 1);
      }
    } else {
      const unsigned long long key = pack_slot(prefix, token, 0) >> 16;
      int at = probe_start(n_slots, prefix, token);
      for (int it = 0; it < n_slots; it += 2) {
        const ulonglong2 g = __ldcg(reinterpret_cast<const ulonglong2*>(hash + at));
        if (g.x == kEmptySlot) { slot = at; return -1; }
        if ((g.x >> 16) == key) return (int)(g.x & 0xffffu);
        if (g.y == kEmptySlot) { slot = at + 1; return -1; }
        if ((g.y >> 16) == key) return (int)(g.y & 0xffffu);
        at = (at + 2) & (n_slots - 1);
      }
    }
    return -1;
  }
  // A bid is above every entry's word (tags have 15 bits; no code is 2^24 - 1) and below the empty slot.
  static constexpr uint32_t kBid = 0xffff0000u;
  // A lane bids for its empty slot.  Returns the higher lane when another one has bid before, `none` otherwise.
  __device__ __forceinline__ int bid(int slot, int lane, int none) {
    uint32_t old;
    if (SMEM) old = atomicMin(tab + slot, kBid | (uint32_t)lane);
    else old = (uint32_t)atomicMin(hash + slot, (unsigned long long)0xffffffffu << 32 | (kBid | (uint32_t)lane));
    const int other = (int)(old & 0xffffu);
    return old == ~0u ? none : (other > lane ? other : lane);
  }
  // After a barrier: the owner of a slot (a bidder ahead of all losers) turns its bid into the entry.
  __device__ __forceinline__ void settle(int slot, uint32_t prefix, uint32_t token, int entry) {
    if (SMEM) {
      tab[slot] = (tag_of(mix(prefix, token)) << 16) | (uint32_t)entry;
      key0[entry] = prefix | (token << 24);
      key1[entry] = (uint16_t)(token >> 8);
    } else {
      hash[slot] = pack_slot(prefix, token, (uint32_t)entry);
    }
  }
  // A bidder that gets no entry empties the slot if its bid is the one that stands there.
  __device__ __forceinline__ void withdraw(int slot, int lane) {
    if (SMEM) atomicCAS(tab + slot, kBid | (uint32_t)lane, ~0u);
    else atomicCAS(hash + slot, (unsigned long long)0xffffffffu << 32 | (kBid | (uint32_t)lane), (unsigned long long)kEmptySlot);
  }
  __device__ __forceinline__ uint32_t prefix_of(int e) const { return key0[e] & 0xffffffu; }
  __device__ __forceinline__ uint32_t token_of(int e) const { return (key0[e] >> 24) | ((uint32_t)key1[e] << 8); }

  // All threads of the block: carve the shared memory and take over the codebook's n entries.
  __device__ void open(const CbView& cb, int b, int n, unsigned char* smem) {
    hash = cb.hash + (size_t)b * cb.n_slots;
    n_slots = cb.n_slots;
    if (!SMEM) return;
    tab = reinterpret_cast<uint32_t*>(smem);
    key0 = tab + n_slots;
    key1 = reinterpret_cast<uint16_t*>(key0 + (cb.cap + (cb.cap & 1)));
    for (int i = threadIdx.x; i < n_slots / 4; i += blockDim.x)
      reinterpret_cast<uint4*>(tab)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
    if (n <= 0) return;                                   // (the caller synchronises the block)
    __syncthreads();
    for (int i = threadIdx.x; i < n_slots; i += blockDim.x) {
      const unsigned long long s = hash[i];
      if (s == kEmptySlot) continue;
      const uint32_t prefix = (uint32_t)(s >> 40), token = (uint32_t)(s >> 16) & 0xffffffu, e = (uint32_t)s & 0xffffu;
      key0[e] = prefix | (token << 24);
      key1[e] = (uint16_t)(token >> 8);
      const uint32_t h = mix(prefix, token), word = (tag_of(h) << 16) | e;
      uint32_t at = (h >> 13) & (uint32_t)(n_slots - 4);
      for (int it = 0; it < n_slots; ++it) {
        if (atomicCAS(tab + at, 0xffffffffu, word) == 0xffffffffu) break;
        at = (at + 1) & (uint32_t)(n_slots - 1);
      }
    }
  }
  // All threads of the block: entries [n0, n1) go to the codebook's hash table.
  __device__ void close(int n0, int n1) {
    if (!SMEM) return;
    if (write_back_four(n0, n1)) close_by<4>(n0, n1);
    else close_by<1>(n0, n1);
  }
  // (AT_ONCE entries of a thread at a time: their insertions do not wait for one another)
  template <int AT_ONCE>
  __device__ __forceinline__ void close_by(int n0, int n1) {
    for (int e0 = n0 + (int)threadIdx.x; e0 < n1; e0 += AT_ONCE * (int)blockDim.x) {
      unsigned long long word[AT_ONCE];
      int at[AT_ONCE];
      bool open[AT_ONCE];
#pragma unroll
      for (int u = 0; u < AT_ONCE; ++u) {
        const int e = e0 + u * (int)blockDim.x;
        open[u] = e < n1;
        const uint32_t prefix = open[u] ? prefix_of(e) : 0u, token = open[u] ? token_of(e) : 0u;
        at[u] = probe_start(n_slots, prefix, token);
        word[u] = pack_slot(prefix, token, (uint32_t)e);
      }
      for (int it = 0; it < n_slots; ++it) {
        unsigned long long old[AT_ONCE];
#pragma unroll
        for (int u = 0; u < AT_ONCE; ++u)
          old[u] = open[u] ? atomicCAS(hash + at[u], (unsigned long long)kEmptySlot, word[u]) : kEmptySlot;
        bool more = false;
#pragma unroll
        for (int u = 0; u < AT_ONCE; ++u) {
          open[u] = open[u] && old[u] != kEmptySlot;
          if (open[u]) { at[u] = (at[u] + 1) & (n_slots - 1); more = true; }
        }
        if (!more) break;
      }
    }
  }
};

// How a call of B sequences of at most T tokens or codes is launched (z2z_lzw.cu); smem_bytes 0: SMEM false.
struct ParseLaunch { int lanes; size_t smem_bytes; };
ParseLaunch parse_launch(const CbView& cb, int T);

// What the parsing warps tell each other inside a window: per warp a mask of lanes on the chain, and of
// those that want a new entry.
template <int WARPS>
struct ParseVotes { uint32_t on[WARPS], ins[WARPS]; };

// Bits of m below lane `at` of the window.
template <int WARPS>
__device__ __forceinline__ int parse_count_below(const uint32_t (&m)[WARPS], int at) {
  int c = 0;
#pragma unroll
  for (int k = 0; k < WARPS; ++k) {
    const int left = at - k * 32;
    const uint32_t keep = left >= 32 ? 0xffffffffu : (left <= 0 ? 0u : (1u << left) - 1u);
    c += __popc(m[k] & keep);
  }
  return c;
}
// The same for this thread's own lane, and the number of all bits.
template <int WARPS>
__device__ __forceinline__ int parse_rank(const uint32_t (&m)[WARPS], int warp, int lane, int& total) {
  int below = 0;
  total = 0;
#pragma unroll
  for (int k = 0; k < WARPS; ++k) {
    if (k == warp) below = total + __popc(m[k] & ((1u << lane) - 1u));
    total += __popc(m[k]);
  }
  return below;
}

}  // namespace z2z
