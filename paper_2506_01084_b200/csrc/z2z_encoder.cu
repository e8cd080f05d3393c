// Hyper-encoder (paper Section 2.2; Section 3.1: transformer encoder layers): work-list
// construction and the CUDA-core kernels of one encoder pass.  Activations stay in fp32 here;
// weights are read in their storage type.
//
// Row layout of a pass: entry e of the work list owns rows e*M .. e*M+M-1 ("we pad the input
// sequence to length M"); rows at or beyond the entry's length are padding: they are never
// attended to and never pooled, and are kept at zero so that no NaN can appear in them.
#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_simt_tile.cuh"
#include "z2z_sm100.cuh"

namespace z2z {

// ---------------------------------------------------------------------------------------------
// Work list
// ---------------------------------------------------------------------------------------------
// First entry of sequence b that is due on a side.
__device__ __forceinline__ int due_from(const CbView& cb, int which, int b) {
  const int e = cb.n_emb[which * cb.B + b];
  return e < 0 ? ~e : e;
}

// mode 0: ranges from first/count (NULL: the entries due on side `which`);  mode 1: from new_entry (0/1 each)
__global__ void __launch_bounds__(1024) k_entry_offsets(CbView cb, int which, int mode,
                                                        const int32_t* first, const int32_t* count,
                                                        const int32_t* new_entry, int32_t* off) {
  __shared__ int sm[32];
  sm100::pdl_wait();
  sm100::pdl_trigger();
  const int b = threadIdx.x;
  int c = 0;
  if (b < cb.B) {
    const int n = cb.n[b];
    if (mode == 1) {
      c = (new_entry[b] >= 0 && new_entry[b] < n) ? 1 : 0;
    } else {
      int f = first ? first[b] : due_from(cb, which, b);
      f = f < 0 ? 0 : (f > n ? n : f);
      c = count ? count[b] : n - f;
      c = c < 0 ? 0 : (c > n - f ? n - f : c);
    }
  }
  int total;
  const int excl = block_scan_1024(c, sm, total);
  if (b < cb.B) off[b] = excl;
  if (b == 0) { off[cb.B] = total; off[cb.B + 1] = 0; }
}

// Entry g of the call: its sequence and number within it.
__device__ __forceinline__ void entry_of(const CbView& cb, int which, int mode, const int32_t* first,
                                         const int32_t* new_entry, const EntryList& el, long long g, int& b, int& k) {
  int lo = 0, hi = cb.B - 1;                     // last b with off[b] <= g
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (el.off[mid] <= g) lo = mid; else hi = mid - 1;
  }
  b = lo;
  int f;
  if (mode == 1) f = new_entry[b];
  else {
    f = first ? first[b] : due_from(cb, which, b);
    const int n = cb.n[b];
    f = f < 0 ? 0 : (f > n ? n : f);
  }
  k = f + (int)(g - el.off[b]);
}

// Work list of a pass: entries [g0, g0 + slots) of the call, or those of one pass of pass_first.
__global__ void k_entry_fill(CbView cb, int which, int mode, const int32_t* first, const int32_t* new_entry, EntryList el,
                             long long g0, int slots, const int32_t* pass_first) {
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  long long end = el.off[cb.B];
  if (pass_first) { g0 = pass_first[0]; end = pass_first[1]; }
  if (e == 0) {
    const long long left = end - g0;
    el.off[cb.B + 1] = (int)(left < 0 ? 0 : (left > slots ? slots : left));
  }
  if (e >= slots) return;
  const long long g = g0 + e;
  if (g >= end) {
    el.seq[e] = -1; el.idx[e] = 0; el.len[e] = 0;
    for (int i = 0; i < cb.M; ++i) el.tok[(size_t)e * cb.M + i] = -1;
    return;
  }
  int b, k;
  entry_of(cb, which, mode, first, new_entry, el, g, b, k);
  el.seq[e] = b;
  el.idx[e] = k;
  const bool in_book = k >= 0 && k < cb.cap;
  el.len[e] = in_book ? (int)cb.len[(size_t)b * cb.cap + k] : 0;
  for (int i = 0; i < cb.M; ++i)                       // constituents are -1 padded behind the entry's length
    el.tok[(size_t)e * cb.M + i] = in_book ? cb.cons[((size_t)b * cb.cap + k) * cb.M + i] : -1;
}

// A call of one pass of at most kListSlots entries: offsets of the sequences (unless `have_off`: they are there), the
// work list and the map of the packed rows, in one block - a launch and the latency of its loads for each of the three
// were 4 to 5 us apart, with nothing else on the GPU (two such calls, the logits and the sampling of 16 sequences at
// d = 4096: 628 -> 618 us).  Thread = sequence, then slot of the list.
__global__ void __launch_bounds__(1024) k_entry_list(CbView cb, int which, const int32_t* first, const int32_t* count, EntryList el,
                                                     int slots, int have_off) {
  __shared__ int warp_sums[32], s_off[1024], s_from[1024];
  sm100::pdl_wait();
  sm100::pdl_trigger();
  const int e = threadIdx.x;
  int f = 0, c = 0, off = 0, total;
  if (e < cb.B) {
    const int n = cb.n[e];
    f = first ? first[e] : due_from(cb, which, e);
    f = f < 0 ? 0 : (f > n ? n : f);
    c = count ? count[e] : n - f;
    c = c < 0 ? 0 : (c > n - f ? n - f : c);
    if (have_off) off = el.off[e];
  }
  if (have_off) {
    total = el.off[cb.B];
  } else {
    off = block_scan_1024(c, warp_sums, total);
    if (e < cb.B) el.off[e] = off;
    if (e == 0) el.off[cb.B] = total;
  }
  s_off[e] = off; s_from[e] = f;
  __syncthreads();
  if (e == 0) el.off[cb.B + 1] = total < slots ? total : slots;
  int len = 0, tok[kMaxM];
#pragma unroll
  for (int i = 0; i < kMaxM; ++i) tok[i] = -1;
  if (e < slots) {
    int b = -1, k = 0;
    if (e < total) {
      int lo = 0, hi = cb.B - 1;                   // last b with off[b] <= e
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_off[mid] <= e) lo = mid; else hi = mid - 1;
      }
      b = lo;
      k = s_from[b] + (e - s_off[b]);
      if (k >= 0 && k < cb.cap) {
        len = (int)cb.len[(size_t)b * cb.cap + k];
#pragma unroll
        for (int i = 0; i < kMaxM; ++i)            // constituents are -1 padded behind the entry's length
          if (i < cb.M) tok[i] = cb.cons[((size_t)b * cb.cap + k) * cb.M + i];
      }
    }
    el.seq[e] = b; el.idx[e] = k; el.len[e] = len;
#pragma unroll
    for (int i = 0; i < kMaxM; ++i)
      if (i < cb.M) el.tok[(size_t)e * cb.M + i] = tok[i];
  }
  int rows;
  const int row = block_scan_1024(len, warp_sums, rows);
  if (e < slots) {
    el.row_off[e] = row;
#pragma unroll
    for (int i = 0; i < kMaxM; ++i)
      if (i < len) { el.row_src[row + i] = e * cb.M + i; el.row_tok[row + i] = tok[i]; }
  }
  if (e == 0) el.row_off[slots] = rows;
}

// Packed rows (base tokens) of all entries of the call, added up in el.off[B + 1] (zero before).
__global__ void __launch_bounds__(256) k_entry_rows(CbView cb, int which, const int32_t* first, EntryList el) {
  sm100::pdl_wait();
  sm100::pdl_trigger();
  const int b = blockIdx.x;
  const int count = el.off[b + 1] - el.off[b];
  int f = first ? first[b] : due_from(cb, which, b);
  const int n = cb.n[b];
  f = f < 0 ? 0 : (f > n ? n : f);
  int sum = 0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) sum += (int)cb.len[(size_t)b * cb.cap + f + i];
  sum = __reduce_add_sync(0xffffffffu, sum);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&el.off[cb.B + 1], sum);
}

// First entry of every pass: the entry whose first row is row r of the call belongs to pass r / rows_per, so
// that a pass holds at most rows_per + M - 1 rows.  One block walks the entries 1024 at a time.
__global__ void __launch_bounds__(1024) k_entry_passes(CbView cb, int which, const int32_t* first, EntryList el, int rows_per,
                                                       int n_passes, int32_t* pass_first) {
  __shared__ int sm[32];
  sm100::pdl_wait();
  sm100::pdl_trigger();
  const int total = el.off[cb.B];
  long long before = 0;                          // rows ahead of this batch of entries
  for (int g0 = 0; g0 < total; g0 += 1024) {
    const int g = g0 + (int)threadIdx.x;
    int len = 0;
    if (g < total) {
      int b, k;
      entry_of(cb, which, 0, first, nullptr, el, g, b, k);
      if (k < cb.cap) len = (int)cb.len[(size_t)b * cb.cap + k];
    }
    int rows;
    const int excl = block_scan_1024(len, sm, rows);
    if (g < total) {
      const long long r0 = before + excl;
      const int pass = (int)(r0 / rows_per);
      const int next = (int)((r0 + len) / rows_per);       // pass of the entry that follows
      if (g == 0) pass_first[0] = 0;
      if (next != pass && next <= n_passes && g + 1 < total) pass_first[next] = g + 1;
      if (g + 1 == total) for (int q = pass + 1; q <= n_passes; ++q) pass_first[q] = total;
    }
    before += rows;
  }
}

// After a call (off: offsets of the sequences' entries in it): the entries among its first `bound` are embedded;
// what the bound left out is due for the next call and stays so through decode steps.  After a decode step
// (off == NULL): every entry is embedded, unless a call left some out.
__global__ void k_mark_embedded(CbView cb, int which, const int32_t* off, long long bound) {
  sm100::pdl_wait();
  sm100::pdl_trigger();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= cb.B) return;
  int32_t* emb = cb.n_emb + which * cb.B + b;
  if (!off) {
    if (*emb >= 0) *emb = cb.n[b];
    return;
  }
  const long long beyond = (long long)off[b + 1] - bound;
  const int count = off[b + 1] - off[b];
  const int left_out = beyond <= 0 ? 0 : (beyond < count ? (int)beyond : count);
  *emb = left_out ? ~(cb.n[b] - left_out) : cb.n[b];
}

__device__ __forceinline__ int entry_len(const CbView& cb, const EntryList& el, int e) {
  const int s = el.seq[e];
  return s < 0 ? 0 : (int)cb.len[(size_t)s * cb.cap + el.idx[e]];
}

// ---------------------------------------------------------------------------------------------
// Pass kernels
// ---------------------------------------------------------------------------------------------
// X[r] = table[y_i] + pos[i] for valid rows, 0 for padding.  grid = rows, block = 128.
template <typename T>
__global__ void __launch_bounds__(128) k_enc_gather(CbView cb, EntryList el,
                                                    const T* __restrict__ table,
                                                    const T* __restrict__ pos, float* __restrict__ X,
                                                    int d) {
  const int r = blockIdx.x, e = r / cb.M, i = r - e * cb.M;
  if (e >= el.off[cb.B + 1]) return;             // beyond the entries of this pass
  const int L = entry_len(cb, el, e);
  float* x = X + (size_t)r * d;
  if (i >= L) {
    for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4)
      *reinterpret_cast<float4*>(x + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const int y = cb.cons[((size_t)el.seq[e] * cb.cap + el.idx[e]) * cb.M + i];
  const T* row = table + (size_t)y * d;
  const T* p = pos + (size_t)i * d;
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {
    float a[4], b[4];
    load4<T>(row + c, a);
    load4<T>(p + c, b);
    *reinterpret_cast<float4*>(x + c) = make_float4(a[0] + b[0], a[1] + b[1], a[2] + b[2], a[3] + b[3]);
  }
}

__device__ __forceinline__ float block_sum_256(float v, float* sm) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sm[w] = v;
  __syncthreads();
  float t = (l < (blockDim.x >> 5)) ? sm[l] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// A[r] = LayerNorm(X[r]) * g + b  (eps 1e-5, biased variance) for valid rows, 0 for padding.
template <typename T>
__global__ void __launch_bounds__(256) k_enc_layernorm(CbView cb, EntryList el,
                                                       const float* __restrict__ X,
                                                       const T* __restrict__ g,
                                                       const T* __restrict__ bta,
                                                       float* __restrict__ A, int d) {
  __shared__ float sm[32];
  const int r = blockIdx.x, e = r / cb.M, i = r - e * cb.M;
  if (e >= el.off[cb.B + 1]) return;
  const int L = entry_len(cb, el, e);
  const float* x = X + (size_t)r * d;
  float* a = A + (size_t)r * d;
  if (i >= L) {
    for (int c = threadIdx.x; c < d; c += blockDim.x) a[c] = 0.f;
    return;
  }
  float s = 0.f;
  for (int c = threadIdx.x; c < d; c += blockDim.x) s += x[c];
  const float mean = block_sum_256(s, sm) / (float)d;
  float q = 0.f;
  for (int c = threadIdx.x; c < d; c += blockDim.x) { float t = x[c] - mean; q += t * t; }
  const float var = block_sum_256(q, sm) / (float)d;
  const float rstd = 1.0f / sqrtf(var + kLnEps);
  for (int c = threadIdx.x; c < d; c += blockDim.x)
    a[c] = (x[c] - mean) * rstd * to_f32<T>(g[c]) + to_f32<T>(bta[c]);
}

__device__ __forceinline__ float gelu_erf(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752440f));
}

// Y = epilogue(A W^T + bias).  MODE 0: plain; 1: GELU; 2: Y += (in-place residual).
template <typename TW, int MODE>
__global__ void __launch_bounds__(256) k_enc_linear(const float* __restrict__ A, int K,
                                                    const TW* __restrict__ W, int J,
                                                    const TW* __restrict__ bias,
                                                    float* __restrict__ Y, int R,
                                                    const int32_t* __restrict__ n_entries, int M) {
  __shared__ SimtSmem sm;
  const int j0 = blockIdx.x * kTJ, r0 = blockIdx.y * kTR;
  if (r0 >= n_entries[0] * M) return;             // no live entry in this row tile
  float acc[4][4];
  const int nW = J - j0 < kTJ ? J - j0 : kTJ;
  simt_tile_mainloop<float, TW>(sm, A, K, r0, R, W + (size_t)j0 * K, nW, K, acc);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty * 4 + i;
    if (r >= R) continue;
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int j = j0 + tx * 4 + jj;
      if (j >= J) continue;
      float v = acc[i][jj] + to_f32<TW>(bias[j]);
      if (MODE == 1) v = gelu_erf(v);
      float* y = Y + (size_t)r * J + j;
      if (MODE == 2) v += *y;
      *y = v;
    }
  }
}

// Bidirectional attention inside one entry (keys = its valid rows only).
// grid (entries, heads), block (32, M): warp y is query row y.
__global__ void k_enc_attention(CbView cb, EntryList el, const float* __restrict__ QKV,
                                float* __restrict__ O, int d, int heads) {
  const int e = blockIdx.x, h = blockIdx.y, i = threadIdx.y, lane = threadIdx.x;
  if (e >= el.off[cb.B + 1]) return;
  const int L = entry_len(cb, el, e);
  const int dh = d / heads;
  float* o = O + ((size_t)e * cb.M + i) * d + (size_t)h * dh;
  if (i >= L) {
    for (int c = lane; c < dh; c += 32) o[c] = 0.f;
    return;
  }
  const float* q = QKV + ((size_t)e * cb.M + i) * 3 * d + (size_t)h * dh;
  const float scale = 1.0f / sqrtf((float)dh);
  float s[kMaxM];
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < kMaxM; ++j) {
    s[j] = -INFINITY;
    if (j < L) {
      const float* kp = QKV + ((size_t)e * cb.M + j) * 3 * d + d + (size_t)h * dh;
      float p = 0.f;
      for (int c = lane; c < dh; c += 32) p = fmaf(q[c], kp[c], p);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) p += __shfl_xor_sync(0xffffffffu, p, off);
      s[j] = p * scale;
      mx = fmaxf(mx, s[j]);
    }
  }
  float den = 0.f;
#pragma unroll
  for (int j = 0; j < kMaxM; ++j) { s[j] = j < L ? expf(s[j] - mx) : 0.f; den += s[j]; }
  const float inv = 1.0f / den;
  for (int c = lane; c < dh; c += 32) {
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < L) v = fmaf(s[j] * inv, QKV[((size_t)e * cb.M + j) * 3 * d + 2 * d + (size_t)h * dh + c], v);
    o[c] = v;
  }
}

// cache[seq][idx] = mean over the entry's valid rows.  grid = entries, block = 256.
template <typename T>
__global__ void __launch_bounds__(256) k_enc_pool(CbView cb, EntryList el,
                                                  const float* __restrict__ X, T* __restrict__ cache,
                                                  float* __restrict__ cache_f32, int d) {
  const int e = blockIdx.x;
  if (e >= el.off[cb.B + 1]) return;
  const int L = entry_len(cb, el, e);
  if (L <= 0) return;
  const size_t dst = ((size_t)el.seq[e] * cb.cap + el.idx[e]) * d;
  const float inv = 1.0f / (float)L;
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    float v = 0.f;
    for (int i = 0; i < L; ++i) v += X[((size_t)e * cb.M + i) * d + c];
    v *= inv;
    cache[dst + c] = from_f32<T>(v);
    if (cache_f32) cache_f32[dst + c] = v;
  }
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
cudaError_t launch_entry_offsets(const CbView& cb, int which, const int32_t* first,
                                 const int32_t* count, const EntryList& el, cudaStream_t s) {
  return launch_pdl(k_entry_offsets, dim3(1), dim3(1024), 0, s, cb, which, 0, first, count, nullptr, el.off);
}
cudaError_t launch_entry_offsets_from_new(const CbView& cb, const int32_t* new_entry,
                                          const EntryList& el, cudaStream_t s) {
  return launch_pdl(k_entry_offsets, dim3(1), dim3(1024), 0, s, cb, 0, 1, nullptr, nullptr, new_entry, el.off);
}
cudaError_t launch_entry_fill(const CbView& cb, int which, const int32_t* first,
                              const int32_t* new_entry, const EntryList& el, int chunk_index, int slots,
                              cudaStream_t s) {
  return launch_pdl(k_entry_fill, dim3((slots + 255) / 256), dim3(256), 0, s, cb, which, new_entry ? 1 : 0, first, new_entry,
                    el, (long long)chunk_index * el.chunk, slots, nullptr);
}
cudaError_t launch_entry_list(const CbView& cb, int which, const int32_t* first, const int32_t* count, const EntryList& el,
                              int slots, bool have_off, cudaStream_t s) {
  if (slots > kListSlots) return cudaErrorInvalidValue;
  return launch_pdl(k_entry_list, dim3(1), dim3(1024), 0, s, cb, which, first, count, el, slots, have_off ? 1 : 0);
}
cudaError_t launch_entry_rows(const CbView& cb, int which, const int32_t* first, const EntryList& el, cudaStream_t s) {
  return launch_pdl(k_entry_rows, dim3(cb.B), dim3(256), 0, s, cb, which, first, el);
}
cudaError_t launch_entry_passes(const CbView& cb, int which, const int32_t* first, const EntryList& el, int rows,
                                int n_passes, int32_t* pass_first, cudaStream_t s) {
  return launch_pdl(k_entry_passes, dim3(1), dim3(1024), 0, s, cb, which, first, el, rows - (cb.M - 1), n_passes, pass_first);
}
cudaError_t launch_entry_fill_pass(const CbView& cb, int which, const int32_t* first, const EntryList& el, int pass,
                                   const int32_t* pass_first, int slots, cudaStream_t s) {
  return launch_pdl(k_entry_fill, dim3((slots + 255) / 256), dim3(256), 0, s, cb, which, 0, first, nullptr, el, 0ll, slots,
                    pass_first ? pass_first + pass : nullptr);
}
cudaError_t launch_mark_embedded(const CbView& cb, int which, const int32_t* off, long long bound, cudaStream_t s) {
  return launch_pdl(k_mark_embedded, dim3((cb.B + 255) / 256), dim3(256), 0, s, cb, which, off, bound);
}

template <typename T>
static cudaError_t encoder_pass_simt(const CbView& cb, const EncoderArgs& a, const EntryList& el,
                                     Prof* prof, cudaStream_t s) {
  const int d = a.d, dff = a.dff, M = cb.M;
  const int E = a.entries, R = E * M;
  const int32_t* n_live = el.off + cb.B + 1;
  auto W = [&](int i) { return reinterpret_cast<const T*>(a.w[i]); };
  { ProfScope ps(prof, kProfEncOther, 1, s);
    k_enc_gather<T><<<R, 128, 0, s>>>(cb, el, reinterpret_cast<const T*>(a.table), W(0), a.X, d); }
  const dim3 blk(256);
  const int rt = (R + kTR - 1) / kTR;
  for (int l = 0; l < a.layers; ++l) {
    const int o = 1 + 12 * l;
{ ProfScope ps(prof, kProfEncOther, 1, s);
        k_enc_layernorm<T><<<R, 256, 0, s>>>(cb, el, a.X, W(o + 0), W(o + 1), a.A, d);
      }
{ ProfScope ps(prof, kProfEncGemm, 1, s);
        k_enc_linear<T, 0><<<dim3((3 * d + kTJ - 1) / kTJ, rt), blk, 0, s>>>(a.A, d, W(o + 2), 3 * d,
                                                                          W(o + 3), a.QKV, R, n_live, M);
      }
{ ProfScope ps(prof, kProfEncOther, 1, s);
        k_enc_attention<<<dim3(E, a.heads), dim3(32, M), 0, s>>>(cb, el, a.QKV, a.A, d, a.heads);
      }
{ ProfScope ps(prof, kProfEncGemm, 1, s);
        k_enc_linear<T, 2><<<dim3((d + kTJ - 1) / kTJ, rt), blk, 0, s>>>(a.A, d, W(o + 4), d, W(o + 5),
                                                                      a.X, R, n_live, M);
      }
      if (dff == 0) continue;                          // attention-only layer
{ ProfScope ps(prof, kProfEncOther, 1, s);
        k_enc_layernorm<T><<<R, 256, 0, s>>>(cb, el, a.X, W(o + 6), W(o + 7), a.A, d);
      }
{ ProfScope ps(prof, kProfEncGemm, 1, s);
        k_enc_linear<T, 1><<<dim3((dff + kTJ - 1) / kTJ, rt), blk, 0, s>>>(a.A, d, W(o + 8), dff,
                                                                        W(o + 9), a.H, R, n_live, M);
      }
{ ProfScope ps(prof, kProfEncGemm, 1, s);
        k_enc_linear<T, 2><<<dim3((d + kTJ - 1) / kTJ, rt), blk, 0, s>>>(a.H, dff, W(o + 10), d,
                                                                      W(o + 11), a.X, R, n_live, M);
      }
  }
{ ProfScope ps(prof, kProfEncOther, 1, s);
      k_enc_pool<T><<<E, 256, 0, s>>>(cb, el, a.X, reinterpret_cast<T*>(a.cache), a.cache_f32, d);
      }
  return cudaGetLastError();
}

cudaError_t run_encoder_pass(const CbView& cb, const EncoderArgs& a, const EntryList& el,
                             bool use_tensor_cores, Prof* prof, cudaStream_t s) {
  (void)use_tensor_cores;
  if (a.dtype == Z2Z_DTYPE_FP32) return encoder_pass_simt<float>(cb, a, el, prof, s);
  return encoder_pass_simt<__nv_bfloat16>(cb, a, el, prof, s);
}

}  // namespace z2z
