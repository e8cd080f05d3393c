// Hyper-encoder pass on the tensor cores (bf16 weights): the linear layers run in the stream-K
// tcgen05 kernels of z2z_stream.cu and z2z_stream_pair.cu (prompt-sized passes: z2z_pair_gemm.cu); this file holds the element-wise kernels between them and the
// host-side sequencing.  Both encoders (embedding side and unembedding side, paper Section 2.2)
// go through the same launches as two "groups".
//
// Activations are kept to ~16 mantissa bits on the tensor cores by splitting every fp32
// activation x into bf16 hi = rn(x) and lo = rn(x - hi): with bf16 weights w the products hi*w
// and lo*w are exact in fp32, so A.W^T = hi.W^T + lo.W^T with fp32 accumulation.  Rounding the
// activations to a single bf16 would leave the hyper-embeddings outside the 2e-2 tolerance.
//
// Prompt-sized passes may instead round every activation ONCE to fp16 and multiply by fp16 copies
// of the weights (exact for bf16 values within fp16's range), when the caller has lent memory
// for the copies: one MMA per k-step instead of two.  The rounding error (2^-11 relative per
// operand element) stays inside the tolerance with a margin of about 3 at d = 4096; the two-part
// form keeps a margin of about 200 and remains the default.
//
// Rows are PACKED in both kinds of pass: entry e owns the rows row_off[e] .. row_off[e] + len[e],
// there are no padding rows, and only the device knows how many rows a pass has (the word behind
// the last entry slot of row_off).
// Layout of a hi/lo operand: decode-sized passes (stream-K GEMM) keep the two parts of packed
// row r in operand rows 2r and 2r + 1 of a bf16 [2 * Rt, K] matrix, so that the live rows are one
// contiguous range whatever their number; prompt-sized passes (CTA-pair GEMM) keep hi rows
// [0, Rt) first and lo rows [Rt, 2 Rt) after them.
//
// GEMM output.  Every CTA of the stream-K GEMM adds its partial tiles (hi and lo parts summed
// in registers) into ONE fp32 matrix Y[group][Rt][J] with reductions in global memory; Y is all zero
// whenever no GEMM result is pending.  The element-wise kernel after a GEMM reads each element of
// that GEMM's result exactly once and stores zero back ("consume and clear"), for every live row
// of the pass (the GEMM adds nothing to rows beyond them), which restores the invariant for the
// next GEMM.  The first pass of a session that needs it clears Y.  Sums of three or more partials depend on
// the order in which they arrive: calls whose bits must not (z2z_hyper_embed in a session of prompt size)
// use a matrix for each half or quarter of K (StreamPairParams::parts), and the kernel after the GEMM adds them.
//
// Launches per layer: GEMM(qkv) -> [+ bias, attention] -> GEMM(o) -> [+ bias + residual,
// LayerNorm 2] -> GEMM(1) -> [+ bias, GELU] -> GEMM(2) -> [+ bias + residual, LayerNorm 1 of the
// next layer | mean-pool into the cache].  All are launched with programmatic serialization.
// Between two GEMMs the weight stream stands still, so the small kernels are written for latency:
// what a kernel needs about an entry (its length, the base token of a row) is one load from the
// work list, and every data load is issued before the first value is used - whether a row is valid
// only decides what is stored.
#include <cuda_fp16.h>

#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_sm100.cuh"
#include "z2z_stream.h"

namespace z2z {

namespace {

using bf16 = __nv_bfloat16;
constexpr int kNT = kGemmNT;
constexpr int kRowThreads = 256;
constexpr int kMaxVec4 = 8;            // float4 per thread in the row kernels: d <= 8192
constexpr int kNarrowVec4 = 4;         // ... and for d <= 4096, where half the registers do
// Which linear-layer kernel a pass takes, by its row capacity.  Up to 128 rows one CTA per weight tile streams
// best (24 rows, d = 3072, both encoders: 249 us a step against 272 with pairs; 96 rows, d = 4096: equal);
// beyond, CTA pairs carry up to 256 rows on one stream (270 rows, one encoder: 486 -> 291 us a step).  Passes
// of 1024 rows take whole output tiles.  Those put both operand parts of all of K into one accumulator, which
// costs accuracy (error against fp64 in units of the rows' rms, d = 4096: 4.3e-5, streamed 1.35e-5), so that
// smaller decode steps stay with the stream also where whole tiles would be quicker (one encoder, all rows
// live: d = 4096, 768 rows 1266 against 1188 us a step, 900 rows 1536 against 1446; d = 3072, 930 rows 991 against
// 1012).  Bounded calls in a session of prompt size stream too, with a matrix for each half of K, up to the
// capacity below; beyond they take whole tiles, as every call of such a session did before (us for 510, 639 and
// 768 rows, streamed / whole tiles: d = 1024 205 286 298 / 198 224 231, d = 2048 348 466 486 / 358 397 408, d = 3072
// 501 706 748 / 540 609 618, d = 4096 708 1013 - / 755 1088 1026; the error 4.6e-6 / 1.1e-5, 6.4e-6 / 2.2e-5,
// 8.5e-6 / 3.2e-5, 1.1e-5 / 4.3e-5: between 512 rows and the line accuracy is what speaks for the stream).
constexpr int kStreamSingleRows = 128;
constexpr int kPromptPassRows = 1024;         // rows of a pass, or that a pass of the session can hold, from which it is prompt-sized
static int prompt_call_min_rows(int d) { return d > 3584 ? 720 : 900; }

struct Ptr2 { const void* p[2]; };
struct MPtr2 { void* p[2]; };

__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
__device__ __forceinline__ float4 load_bf16x4(const bf16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(bf_lo(u.x), bf_hi(u.x), bf_lo(u.y), bf_hi(u.y));
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
         ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}
// hi = rn(x), lo = rn(x - hi) for 4 values; 8-byte stores.
__device__ __forceinline__ void split_store4(bf16* hi, bf16* lo, float4 x) {
  const bf16 h0 = __float2bfloat16_rn(x.x), h1 = __float2bfloat16_rn(x.y);
  const bf16 h2 = __float2bfloat16_rn(x.z), h3 = __float2bfloat16_rn(x.w);
  uint2 H, L;
  H.x = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
  H.y = (uint32_t)__bfloat16_as_ushort(h2) | ((uint32_t)__bfloat16_as_ushort(h3) << 16);
  L.x = pack_bf16(x.x - __bfloat162float(h0), x.y - __bfloat162float(h1));
  L.y = pack_bf16(x.z - __bfloat162float(h2), x.w - __bfloat162float(h3));
  *reinterpret_cast<uint2*>(hi) = H;
  *reinterpret_cast<uint2*>(lo) = L;
}
// 4 values rounded once to fp16; one 8-byte store.  `dst` points into an fp16 matrix that shares
// the bf16 operand buffer (same element size).
__device__ __forceinline__ void half_store4(bf16* dst, float4 x) {
  uint2 H;
  H.x = (uint32_t)__half_as_ushort(__float2half_rn(x.x)) | ((uint32_t)__half_as_ushort(__float2half_rn(x.y)) << 16);
  H.y = (uint32_t)__half_as_ushort(__float2half_rn(x.z)) | ((uint32_t)__half_as_ushort(__float2half_rn(x.w)) << 16);
  *reinterpret_cast<uint2*>(dst) = H;
}
// Base tokens of work-list entry e (0 for an unused slot): one load, so that the kernels below can
// issue it together with their data loads instead of ahead of them.
__device__ __forceinline__ int entry_len_tc(const CbView& cb, const EntryList& el, int e) {
  (void)cb;
  return el.len[e];
}
__device__ __forceinline__ float4 unpack_bf16x4(uint2 u) {
  return make_float4(bf_lo(u.x), bf_hi(u.x), bf_lo(u.y), bf_hi(u.y));
}

// A result that lies in several matrices (StreamPairParams::parts): always added in the order of the parts.
__device__ __forceinline__ void add_part(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }

__device__ __forceinline__ float block_sum(float v, float* sm) {
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

// LayerNorm of a row held in registers (x[v] = 4 columns starting at (tid + v * 256) * 4),
// written as hi/lo bf16.  eps 1e-5, biased variance, two-pass.
// gw / gb: gamma and beta of the thread's columns, packed 4 bf16 per uint2 and loaded by the caller
// together with the row, so that no load waits behind the reductions.
template <int NV, bool HALF = false>
__device__ __forceinline__ void layernorm_split_regs(const float4 (&x)[NV], int nvec, const uint2 (&gw)[NV],
                                                     const uint2 (&gb)[NV], bf16* hi, bf16* lo, int d, float* sm) {
  float s = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v)
    if ((int)threadIdx.x + v * kRowThreads < nvec) s += (x[v].x + x[v].y) + (x[v].z + x[v].w);
  const float mean = block_sum(s, sm) / (float)d;
  float q = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v)
    if ((int)threadIdx.x + v * kRowThreads < nvec) {
      const float a = x[v].x - mean, bb = x[v].y - mean, c = x[v].z - mean, e = x[v].w - mean;
      q += (a * a + bb * bb) + (c * c + e * e);
    }
  const float rstd = 1.0f / sqrtf(block_sum(q, sm) / (float)d + kLnEps);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (int)threadIdx.x + v * kRowThreads;
    if (idx < nvec) {
      const float4 gg = unpack_bf16x4(gw[v]), bb = unpack_bf16x4(gb[v]);
      float4 y;
      y.x = (x[v].x - mean) * rstd * gg.x + bb.x;
      y.y = (x[v].y - mean) * rstd * gg.y + bb.y;
      y.z = (x[v].z - mean) * rstd * gg.z + bb.z;
      y.w = (x[v].w - mean) * rstd * gg.w + bb.w;
      if (HALF) half_store4(hi + idx * 4, y);
      else split_store4(hi + idx * 4, lo + idx * 4, y);
    }
  }
}

// X = table[y] + pos for every live packed row; then LN1 of layer 0 -> hi/lo.  grid (rows, groups).
template <int NV>
__global__ void __launch_bounds__(kRowThreads) k_tc_gather_ln(CbView cb, EntryList el, const int* total, Ptr2 table,
                                                              Ptr2 pos, Ptr2 ln_w, Ptr2 ln_b, MPtr2 X, MPtr2 Ahl,
                                                              int d, int has_ln) {
  __shared__ float sm[32];
  sm100::pdl_trigger();            // the next kernel may start its prologue and weight prefetch
  sm100::pdl_wait();               // everything read or written below depends on earlier kernels
  const int r = blockIdx.x, g = blockIdx.y;
  const int y = el.row_tok[r];                    // the row's base token, its place in the entry and the
  const int src = el.row_src[r];                  // row count: three independent loads
  if (r >= *total) return;
  const int i = src % cb.M;
  float* x = reinterpret_cast<float*>(X.p[g]) + (size_t)r * d;
  bf16* hi = reinterpret_cast<bf16*>(Ahl.p[g]) + (size_t)2 * r * d;
  bf16* lo = hi + d;
  const int nvec = d / 4;
  const bf16* row = reinterpret_cast<const bf16*>(table.p[g]) + (size_t)y * d;
  const bf16* pp = reinterpret_cast<const bf16*>(pos.p[g]) + (size_t)i * d;
  const uint2* lw = reinterpret_cast<const uint2*>(ln_w.p[g]);
  const uint2* lb = reinterpret_cast<const uint2*>(ln_b.p[g]);
  float4 xv[NV];
  uint2 gw[NV], gb[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (int)threadIdx.x + v * kRowThreads;
    if (idx < nvec) {
      const float4 a = load_bf16x4(row + idx * 4), b = load_bf16x4(pp + idx * 4);
      gw[v] = lw[idx]; gb[v] = lb[idx];
      xv[v] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
      *reinterpret_cast<float4*>(x + idx * 4) = xv[v];
    }
  }
  if (has_ln) layernorm_split_regs<NV>(xv, nvec, gw, gb, hi, lo, d, sm);
}

// x = X[r] + Y[r] + bias for a live packed row (Y consumed and cleared); then LayerNorm -> hi/lo
// for the next GEMM.  grid (rows, groups).  All loads (row count, Y, X, bias, gamma, beta) are
// issued together; whether the row is live only decides what is stored.
template <int NV, int PARTS>
__global__ void __launch_bounds__(kRowThreads) k_tc_reduce_resid_ln(const int* total, float* Y, size_t part_stride, Ptr2 bias,
                                                                    MPtr2 X, Ptr2 ln_w, Ptr2 ln_b, MPtr2 Ahl,
                                                                    int d, int Rt) {
  __shared__ float sm[32];
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int r = blockIdx.x, g = blockIdx.y;
  const int live = *total;
  float* y = Y + ((size_t)g * Rt + r) * d;
  float* x = reinterpret_cast<float*>(X.p[g]) + (size_t)r * d;
  const uint2* bs = reinterpret_cast<const uint2*>(bias.p[g]);
  const uint2* lw = reinterpret_cast<const uint2*>(ln_w.p[g]);
  const uint2* lb = reinterpret_cast<const uint2*>(ln_b.p[g]);
  const int nvec = d / 4;
  float4 xv[NV], yv[NV], zv[PARTS][NV];            // (zv[0] is not used)
  uint2 bv[NV], gw[NV], gb[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (int)threadIdx.x + v * kRowThreads;
    if (idx < nvec) {
      yv[v] = *reinterpret_cast<const float4*>(y + idx * 4);
#pragma unroll
      for (int k = 1; k < PARTS; ++k) zv[k][v] = *reinterpret_cast<const float4*>(y + k * part_stride + idx * 4);
      xv[v] = *reinterpret_cast<const float4*>(x + idx * 4);
      bv[v] = bs[idx]; gw[v] = lw[idx]; gb[v] = lb[idx];
    }
  }
  if (r >= live) return;                          // nothing was added to this row of Y: it is still zero
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (int)threadIdx.x + v * kRowThreads;
    if (idx < nvec) {
      *reinterpret_cast<float4*>(y + idx * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 1; k < PARTS; ++k) {
        *reinterpret_cast<float4*>(y + k * part_stride + idx * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
        add_part(yv[v], zv[k][v]);
      }
      const float4 b = unpack_bf16x4(bv[v]);
      xv[v] = make_float4(xv[v].x + yv[v].x + b.x, xv[v].y + yv[v].y + b.y, xv[v].z + yv[v].z + b.z,
                          xv[v].w + yv[v].w + b.w);
      *reinterpret_cast<float4*>(x + idx * 4) = xv[v];
    }
  }
  bf16* hi = reinterpret_cast<bf16*>(Ahl.p[g]) + (size_t)2 * r * d;
  layernorm_split_regs<NV>(xv, nvec, gw, gb, hi, hi + d, d, sm);
}

// Last layer: x_i = X[r_i] + Y[r_i] + bias for the entry's rows, cache row = mean_i x_i.
// grid (entries, groups, ceil(d / (4 * kRowThreads))): a thread owns 4 columns of the entry and
// issues the loads of all its rows before it adds.
template <int PARTS>
__global__ void __launch_bounds__(kRowThreads) k_tc_reduce_resid_pool(CbView cb, EntryList el, float* Y, size_t part_stride,
                                                                      Ptr2 bias, MPtr2 X, MPtr2 cache, MPtr2 cache_f32,
                                                                      int d, int Rt) {
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int e = blockIdx.x, g = blockIdx.y;
  const int col = ((int)blockIdx.z * kRowThreads + (int)threadIdx.x) * 4;
  if (col >= d) return;
  const int L = entry_len_tc(cb, el, e);
  const int r0 = el.row_off[e];
  const int seq = el.seq[e], idx = el.idx[e];
  const float4 b = load_bf16x4(reinterpret_cast<const bf16*>(bias.p[g]) + col);
  if (L <= 0) return;
  float4 yv[kMaxM], xv[kMaxM], zv[PARTS][kMaxM];
#pragma unroll
  for (int i = 0; i < kMaxM; ++i)
    if (i < L) {
      const size_t r = (size_t)r0 + i;
      yv[i] = *reinterpret_cast<const float4*>(Y + ((size_t)g * Rt + r) * d + col);
#pragma unroll
      for (int k = 1; k < PARTS; ++k) zv[k][i] = *reinterpret_cast<const float4*>(Y + k * part_stride + ((size_t)g * Rt + r) * d + col);
      xv[i] = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(X.p[g]) + r * d + col);
    }
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < kMaxM; ++i)
    if (i < L) {
      const size_t r = (size_t)r0 + i;
      *reinterpret_cast<float4*>(Y + ((size_t)g * Rt + r) * d + col) = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 1; k < PARTS; ++k) {
        *reinterpret_cast<float4*>(Y + k * part_stride + ((size_t)g * Rt + r) * d + col) = make_float4(0.f, 0.f, 0.f, 0.f);
        add_part(yv[i], zv[k][i]);
      }
      acc.x += xv[i].x + yv[i].x + b.x; acc.y += xv[i].y + yv[i].y + b.y;
      acc.z += xv[i].z + yv[i].z + b.z; acc.w += xv[i].w + yv[i].w + b.w;
    }
  const size_t dst = ((size_t)seq * cb.cap + idx) * d + col;
  const float inv = 1.0f / (float)L;
  const float4 m = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
  uint2 o; o.x = pack_bf16(m.x, m.y); o.y = pack_bf16(m.z, m.w);
  *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(cache.p[g]) + dst) = o;
  float* out32 = reinterpret_cast<float*>(cache_f32.p[g]);
  if (out32) *reinterpret_cast<float4*>(out32 + dst) = m;
}

// Zero-layer encoder (the parameter-free averaging variant): cache row = mean of the entry's X rows.
__global__ void __launch_bounds__(kRowThreads) k_tc_pool(CbView cb, EntryList el, MPtr2 X, MPtr2 cache,
                                                         MPtr2 cache_f32, int d) {
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int e = blockIdx.x, g = blockIdx.y;
  const int L = entry_len_tc(cb, el, e);
  if (L <= 0) return;
  const float* x = reinterpret_cast<const float*>(X.p[g]) + (size_t)el.row_off[e] * d;
  const size_t dst = ((size_t)el.seq[e] * cb.cap + el.idx[e]) * d;
  const float inv = 1.0f / (float)L;
  bf16* out = reinterpret_cast<bf16*>(cache.p[g]);
  float* out32 = reinterpret_cast<float*>(cache_f32.p[g]);
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    float v = 0.f;
    for (int i = 0; i < L; ++i) v += x[(size_t)i * d + c];
    v *= inv;
    out[dst + c] = __float2bfloat16_rn(v);
    if (out32) out32[dst + c] = v;
  }
}

// H = GELU(Y + bias) -> hi/lo (Y consumed and cleared) for the live packed rows.  The
// [groups * R, J] results are one flat range of float4; every thread takes kGeluPerThread of them,
// kGeluThreads apart, and issues all of its loads before it computes.
// grid = ceil(groups * R * J / 4 / (kGeluThreads * kGeluPerThread)), R = row capacity of the pass.
constexpr int kGeluThreads = 256, kGeluPerThread = 4;
template <bool HALVES>
__global__ void __launch_bounds__(kGeluThreads) k_tc_reduce_gelu(const int* total_rows, float* Y, size_t part_stride, Ptr2 bias,
                                                                 MPtr2 Hhl, int J, int R, int Rt, int ng) {
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int J4 = J / 4;
  const long long total = (long long)ng * R * J4;
  const long long base = (long long)blockIdx.x * (kGeluThreads * kGeluPerThread) + threadIdx.x;
  const int live = *total_rows;
  float4 q[kGeluPerThread], bs[kGeluPerThread], q2[HALVES ? kGeluPerThread : 1];
  int row[kGeluPerThread], jj[kGeluPerThread];
#pragma unroll
  for (int k = 0; k < kGeluPerThread; ++k) {
    const long long f = base + (long long)k * kGeluThreads;
    row[k] = -1;
    if (f < total) {
      row[k] = (int)(f / J4);
      jj[k] = (int)(f - (long long)row[k] * J4) * 4;
      const int g = row[k] / R, r = row[k] - g * R;
      q[k] = *reinterpret_cast<const float4*>(Y + ((size_t)g * Rt + r) * J + jj[k]);
      if (HALVES) q2[HALVES ? k : 0] = *reinterpret_cast<const float4*>(Y + part_stride + ((size_t)g * Rt + r) * J + jj[k]);
      bs[k] = load_bf16x4(reinterpret_cast<const bf16*>(bias.p[g]) + jj[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < kGeluPerThread; ++k) {
    if (row[k] < 0) continue;
    const int g = row[k] / R, r = row[k] - g * R;
    if (r >= live) continue;                       // no row there: Y is still zero, nothing reads the operand row
    *reinterpret_cast<float4*>(Y + ((size_t)g * Rt + r) * J + jj[k]) = make_float4(0.f, 0.f, 0.f, 0.f);
    if (HALVES) {
      *reinterpret_cast<float4*>(Y + part_stride + ((size_t)g * Rt + r) * J + jj[k]) = make_float4(0.f, 0.f, 0.f, 0.f);
      add_part(q[k], q2[HALVES ? k : 0]);
    }
    float4 v = make_float4(q[k].x + bs[k].x, q[k].y + bs[k].y, q[k].z + bs[k].z, q[k].w + bs[k].w);
    v.x = 0.5f * v.x * (1.0f + erff(v.x * 0.70710678118654752440f));
    v.y = 0.5f * v.y * (1.0f + erff(v.y * 0.70710678118654752440f));
    v.z = 0.5f * v.z * (1.0f + erff(v.z * 0.70710678118654752440f));
    v.w = 0.5f * v.w * (1.0f + erff(v.w * 0.70710678118654752440f));
    bf16* hi = reinterpret_cast<bf16*>(Hhl.p[g]) + (size_t)2 * r * J + jj[k];
    split_store4(hi, hi + J, v);
  }
}

// q, k, v = Y + bias for one head of one entry (consumed, cleared, staged in shared memory), then
// bidirectional attention over the entry's rows; output as hi/lo.
// grid (entries, heads, groups), block (32, M), dynamic smem M * 3 * dh floats; dh % 4 == 0.
template <bool HALVES>
__global__ void k_tc_qkv_attention(CbView cb, EntryList el, float* Y, size_t part_stride, Ptr2 bias, MPtr2 Ohl, int d,
                                   int heads, int Rt) {
  extern __shared__ float s_qkv[];
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int e = blockIdx.x, h = blockIdx.y, g = blockIdx.z, i = threadIdx.y, lane = threadIdx.x;
  const int L = entry_len_tc(cb, el, e);
  const int r = el.row_off[e] + i;               // packed row of position i (only used while i < L)
  const int dh = d / heads;
  if (i < L) {
    const bf16* bs = reinterpret_cast<const bf16*>(bias.p[g]);
    float* y = Y + ((size_t)g * Rt + r) * 3 * d;
    for (int c = lane * 4; c < dh; c += 128) {
      float4 p[3], b[3], p2[HALVES ? 3 : 1];
#pragma unroll
      for (int w = 0; w < 3; ++w) {                // the loads are independent of one another
        const int col = w * d + h * dh + c;
        p[w] = *reinterpret_cast<const float4*>(y + col);
        if (HALVES) p2[HALVES ? w : 0] = *reinterpret_cast<const float4*>(y + part_stride + col);
        b[w] = load_bf16x4(bs + col);
      }
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        *reinterpret_cast<float4*>(y + w * d + h * dh + c) = make_float4(0.f, 0.f, 0.f, 0.f);
        if (HALVES) {
          *reinterpret_cast<float4*>(y + part_stride + w * d + h * dh + c) = make_float4(0.f, 0.f, 0.f, 0.f);
          add_part(p[w], p2[HALVES ? w : 0]);
        }
        *reinterpret_cast<float4*>(&s_qkv[(i * 3 + w) * dh + c]) =
            make_float4(p[w].x + b[w].x, p[w].y + b[w].y, p[w].z + b[w].z, p[w].w + b[w].w);
      }
    }
  }
  __syncthreads();
  if (i >= L) return;
  const float* q = s_qkv + (i * 3) * dh;
  const float scale = 1.0f / sqrtf((float)dh);
  float s[kMaxM];
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < kMaxM; ++j) {
    s[j] = -INFINITY;
    if (j < L) {
      const float* kp = s_qkv + (j * 3 + 1) * dh;
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
  bf16* hi = reinterpret_cast<bf16*>(Ohl.p[g]) + (size_t)2 * r * d + (size_t)h * dh;
  bf16* lo = hi + d;
  for (int c = lane; c < dh; c += 32) {
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < L) v = fmaf(s[j] * inv, s_qkv[(j * 3 + 2) * dh + c], v);
    const bf16 hh = __float2bfloat16_rn(v);
    hi[c] = hh;
    lo[c] = __float2bfloat16_rn(v - __bfloat162float(hh));
  }
}

// Packed rows: entry e owns rows row_off[e] .. row_off[e] + len[e], there are no padding rows
// inside entries, and rows at or beyond the total carry nothing.  (With M = 3 or 4 a quarter to a
// third of padded rows would be zeros that the GEMMs load and multiply anyway.)
//
// One block: first packed row of every entry (exclusive scan of the lengths), the total behind the
// last entry slot, the way back from a packed row to (entry, position) and the row's base token.
// E <= 1024 * kMapPerThread entries, neighbouring ones per thread.  (The decode step's update kernel
// writes the same map itself.)
//
// UNIQ: also finds the rows that are alike.  Up to the first attention a row depends on its base token and its place in
// the entry only, and the rows of a pass repeat them (of 3072 rows of prompts with vocabulary 32064 a third are
// distinct, of 2304 with 128256 a quarter): LayerNorm and the q, k, v products run on the distinct ones, numbered by
// first appearance.  Dynamic shared memory: uniq_slots words of a hash table of first rows, then the rows' keys.
constexpr int kMapPerThread = kMaxM / 2;
template <bool UNIQ>
__global__ void __launch_bounds__(1024) k_tc_row_map(CbView cb, EntryList el, int E, int uniq_slots, int R) {
  __shared__ int warp_sums[32];
  extern __shared__ uint32_t s_first[];
  uint32_t* s_key = s_first + uniq_slots;
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int tid = threadIdx.x;
  const int per = (E + 1023) / 1024, e0 = tid * per;
  int len[kMapPerThread], mine = 0;
#pragma unroll
  for (int q = 0; q < kMapPerThread; ++q) {
    len[q] = q < per && e0 + q < E ? entry_len_tc(cb, el, e0 + q) : 0;
    mine += len[q];
  }
  int rows;
  int row = block_scan_1024(mine, warp_sums, rows);
#pragma unroll
  for (int q = 0; q < kMapPerThread; ++q) {
    if (q >= per || e0 + q >= E) break;
    el.row_off[e0 + q] = row;
    for (int i = 0; i < len[q]; ++i) {
      const int tok = el.tok[(size_t)(e0 + q) * cb.M + i];
      el.row_src[row + i] = (e0 + q) * cb.M + i;
      el.row_tok[row + i] = tok;
      if (UNIQ && row + i < R) s_key[row + i] = (uint32_t)tok * kMaxM + i;
    }
    row += len[q];
  }
  if (tid == 0) el.row_off[E] = rows;
  if (!UNIQ) return;
  rows = rows < R ? rows : R;
  for (int i = tid; i < uniq_slots; i += 1024) s_first[i] = ~0u;
  __syncthreads();
  // every row bids for the slot of its key: the lowest row of a kind keeps it
  const int rper = (rows + 1023) / 1024, r0 = tid * rper;      // at most kMaxM rows per thread, neighbouring ones
  int slot[kMaxM], fresh = 0;
#pragma unroll
  for (int q = 0; q < kMaxM; ++q) {
    slot[q] = -1;
    if (q >= rper || r0 + q >= rows) continue;
    const uint32_t key = s_key[r0 + q];
    uint32_t at = (key * 0x9E3779B1u >> 8) & (uint32_t)(uniq_slots - 1);
    for (int it = 0; it < uniq_slots; ++it) {                  // bounded; half of the slots stay empty
      const uint32_t old = atomicCAS(s_first + at, ~0u, (uint32_t)(r0 + q));
      if (old == ~0u) break;
      if (s_key[old] == key) { atomicMin(s_first + at, (uint32_t)(r0 + q)); break; }
      at = (at + 1) & (uint32_t)(uniq_slots - 1);
    }
    slot[q] = (int)at;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kMaxM; ++q)
    if (slot[q] >= 0 && s_first[slot[q]] == (uint32_t)(r0 + q)) ++fresh;
  int kinds;
  int u = block_scan_1024(fresh, warp_sums, kinds);
#pragma unroll
  for (int q = 0; q < kMaxM; ++q)
    if (slot[q] >= 0 && s_first[slot[q]] == (uint32_t)(r0 + q)) { s_key[r0 + q] = u; el.row_uniq[r0 + q] = u | kFirstOfKind; ++u; }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kMaxM; ++q)
    if (slot[q] >= 0 && s_first[slot[q]] != (uint32_t)(r0 + q)) el.row_uniq[r0 + q] = (int)s_key[s_first[slot[q]]];
  if (tid == 0) el.row_uniq[el.chunk * cb.M] = kinds;
}

// X = table[y] + pos for every packed row, then LN1 of layer 0 -> hi/lo (uniq: of the distinct rows).  grid (row capacity).
template <int NV, bool HALF>
__global__ void __launch_bounds__(kRowThreads) k_tc_gather_ln_packed(CbView cb, EntryList el, const int* total, const int* uniq,
                                                                     const bf16* table, const bf16* pos, const bf16* ln_w,
                                                                     const bf16* ln_b, float* X, bf16* Ahl, int d, int Rt,
                                                                     int has_ln) {
  __shared__ float sm[32];
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int r = blockIdx.x;
  if (r >= *total) return;
  const int src = el.row_src[r];
  const int u = uniq ? uniq[r] : r | kFirstOfKind;
  const int y = el.tok[src], i = src % cb.M;
  float* x = X + (size_t)r * d;
  bf16* hi = Ahl + (size_t)(u & ~kFirstOfKind) * d;
  const bf16* row = table + (size_t)y * d;
  const bf16* pp = pos + (size_t)i * d;
  const int nvec = d / 4;
  float4 xv[NV];
  uint2 gw[NV], gb[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (int)threadIdx.x + v * kRowThreads;
    if (idx < nvec) {
      const float4 a = load_bf16x4(row + idx * 4), b = load_bf16x4(pp + idx * 4);
      gw[v] = reinterpret_cast<const uint2*>(ln_w)[idx];
      gb[v] = reinterpret_cast<const uint2*>(ln_b)[idx];
      xv[v] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
      *reinterpret_cast<float4*>(x + idx * 4) = xv[v];
    }
  }
  if (has_ln && u < 0) layernorm_split_regs<NV, HALF>(xv, nvec, gw, gb, hi, hi + (size_t)Rt * d, d, sm);
}

// Mean-pool on packed rows: cache row = mean of the entry's rows of X.  grid (entries,
// ceil(d / (4 * kRowThreads))): a thread owns 4 columns and loads all rows before it adds.
__global__ void __launch_bounds__(kRowThreads) k_tc_pool_packed(CbView cb, EntryList el, const float* X, void* cache,
                                                                float* cache_f32, int d) {
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int e = blockIdx.x;
  const int col = ((int)blockIdx.y * kRowThreads + (int)threadIdx.x) * 4;
  if (col >= d) return;
  const int L = entry_len_tc(cb, el, e);
  if (L <= 0) return;
  const float* x = X + (size_t)el.row_off[e] * d + col;
  float4 v[kMaxM];
#pragma unroll
  for (int i = 0; i < kMaxM; ++i)
    if (i < L) v[i] = *reinterpret_cast<const float4*>(x + (size_t)i * d);
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < kMaxM; ++i)
    if (i < L) { acc.x += v[i].x; acc.y += v[i].y; acc.z += v[i].z; acc.w += v[i].w; }
  const size_t dst = ((size_t)el.seq[e] * cb.cap + el.idx[e]) * d + col;
  const float inv = 1.0f / (float)L;
  const float4 m = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
  uint2 o; o.x = pack_bf16(m.x, m.y); o.y = pack_bf16(m.z, m.w);
  *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(cache) + dst) = o;
  if (cache_f32) *reinterpret_cast<float4*>(cache_f32 + dst) = m;
}

// LayerNorm of the packed rows of X -> hi/lo (the GEMM epilogue has already added bias and
// residual into X).  grid (row capacity), one encoder.
template <int NV, bool HALF>
__global__ void __launch_bounds__(kRowThreads) k_tc_ln_rows(const int* total, const float* X, const bf16* ln_w,
                                                            const bf16* ln_b, bf16* Ahl, int d, int Rt) {
  __shared__ float sm[32];
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int r = blockIdx.x;
  if (r >= *total) return;
  const float* x = X + (size_t)r * d;
  const int nvec = d / 4;
  float4 xv[NV];
  uint2 gw[NV], gb[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int idx = (int)threadIdx.x + v * kRowThreads;
    if (idx < nvec) {
      xv[v] = *reinterpret_cast<const float4*>(x + idx * 4);
      gw[v] = reinterpret_cast<const uint2*>(ln_w)[idx];
      gb[v] = reinterpret_cast<const uint2*>(ln_b)[idx];
    }
  }
  bf16* hi = Ahl + (size_t)r * d;
  layernorm_split_regs<NV, HALF>(xv, nvec, gw, gb, hi, hi + (size_t)Rt * d, d, sm);
}

// Bidirectional attention inside one entry from fp32 q, k, v of its packed rows [rows, 3d] (bias
// already added); output as hi/lo.  One WARP per (entry, head): all of the item's q, k, v values
// are loaded into registers at once (a lane holds four columns of every row), the L x L scores are
// warp reductions, no shared memory and no block barrier.  MM = compile-time bound on the merge
// size; dh <= 128 (larger heads take the kernel below).  grid = ceil(entries * heads / 8), block 256.
template <int MM, bool HALF>
__global__ void __launch_bounds__(256) k_tc_attention_rows_warp(CbView cb, EntryList el, const float* QKV,
                                                                const int* uniq, bf16* Ohl, int E, int d, int heads, int Rt) {
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int lane = threadIdx.x & 31;
  const int item = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (item >= E * heads) return;
  const int e = item / heads, h = item - e * heads;
  const int L = entry_len_tc(cb, el, e);
  if (L <= 0) return;
  const int dh = d / heads, c = lane * 4;
  const bool on = c < dh;                      // lanes beyond the head's width hold zeros
  const size_t r0 = el.row_off[e];
  const float* y = QKV + (size_t)h * dh + c;
  size_t at[MM];
#pragma unroll
  for (int i = 0; i < MM; ++i) at[i] = i < L && uniq ? uniq[r0 + i] & ~kFirstOfKind : r0 + i;
  float4 q[MM], k[MM], v[MM];
#pragma unroll
  for (int i = 0; i < MM; ++i) {
    q[i] = k[i] = v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < L && on) {
      const float* yi = y + at[i] * 3 * d;
      q[i] = *reinterpret_cast<const float4*>(yi);
      k[i] = *reinterpret_cast<const float4*>(yi + d);
      v[i] = *reinterpret_cast<const float4*>(yi + 2 * d);
    }
  }
  const float scale = 1.0f / sqrtf((float)dh);
  bf16* hi = Ohl + r0 * d + (size_t)h * dh + c;
  bf16* lo = hi + (size_t)Rt * d;
#pragma unroll
  for (int i = 0; i < MM; ++i) {
    if (i >= L) break;
    float s[MM];
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      float p = q[i].x * k[j].x + q[i].y * k[j].y + q[i].z * k[j].z + q[i].w * k[j].w;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) p += __shfl_xor_sync(0xffffffffu, p, off);
      s[j] = j < L ? p * scale : -INFINITY;
      mx = fmaxf(mx, s[j]);
    }
    float den = 0.f;
#pragma unroll
    for (int j = 0; j < MM; ++j) { s[j] = j < L ? expf(s[j] - mx) : 0.f; den += s[j]; }
    const float inv = 1.0f / den;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < MM; ++j) {
      const float wj = s[j] * inv;
      o.x = fmaf(wj, v[j].x, o.x); o.y = fmaf(wj, v[j].y, o.y); o.z = fmaf(wj, v[j].z, o.z); o.w = fmaf(wj, v[j].w, o.w);
    }
    if (on) {
      if (HALF) half_store4(hi + (size_t)i * d, o);
      else split_store4(hi + (size_t)i * d, lo + (size_t)i * d, o);
    }
  }
}

// The same for heads wider than 128 columns or merge sizes above 4: staged in shared memory.
// grid (entries, heads), block (32, M), dynamic smem M * 3 * dh floats.
__global__ void k_tc_attention_rows(CbView cb, EntryList el, const float* QKV, const int* uniq, bf16* Ohl, int d, int heads,
                                    int Rt, int half) {
  extern __shared__ float s_qkv[];
  sm100::pdl_trigger();
  sm100::pdl_wait();
  const int e = blockIdx.x, h = blockIdx.y, i = threadIdx.y, lane = threadIdx.x;
  const int L = entry_len_tc(cb, el, e);
  if (L <= 0) return;
  const int dh = d / heads;
  const int r = el.row_off[e] + i;
  if (i < L) {
    const float* y = QKV + (size_t)(uniq ? uniq[r] & ~kFirstOfKind : r) * 3 * d;
    for (int w = 0; w < 3; ++w)
      for (int c = lane * 4; c < dh; c += 128)
        *reinterpret_cast<float4*>(&s_qkv[(i * 3 + w) * dh + c]) = *reinterpret_cast<const float4*>(y + w * d + h * dh + c);
  }
  __syncthreads();
  if (i >= L) return;
  const float* q = s_qkv + (i * 3) * dh;
  const float scale = 1.0f / sqrtf((float)dh);
  float s[kMaxM];
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < kMaxM; ++j) {
    s[j] = -INFINITY;
    if (j < L) {
      const float* kp = s_qkv + (j * 3 + 1) * dh;
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
  bf16* hi = Ohl + (size_t)r * d + (size_t)h * dh;
  bf16* lo = hi + (size_t)Rt * d;
  for (int c = lane; c < dh; c += 32) {
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < kMaxM; ++j)
      if (j < L) v = fmaf(s[j] * inv, s_qkv[(j * 3 + 2) * dh + c], v);
    if (half) {
      reinterpret_cast<__half*>(hi)[c] = __float2half_rn(v);
    } else {
      const bf16 hh = __float2bfloat16_rn(v);
      hi[c] = hh;
      lo[c] = __float2bfloat16_rn(v - __bfloat162float(hh));
    }
  }
}

// fp16 copy of a bf16 weight tensor (n a multiple of 8).  A bf16 value inside fp16's range converts
// exactly; a value beyond it cannot be represented and raises bit 1 of the error word.
__global__ void __launch_bounds__(256) k_tc_weights_to_half(const bf16* __restrict__ src, __half* __restrict__ dst,
                                                            size_t n8, int* err) {
  bool over = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += (size_t)gridDim.x * blockDim.x) {
    const uint4 u = reinterpret_cast<const uint4*>(src)[i];
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    uint32_t o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float a = bf_lo(w[k]), b = bf_hi(w[k]);
      over |= fabsf(a) > 65504.f || fabsf(b) > 65504.f;
      o[k] = (uint32_t)__half_as_ushort(__float2half_rn(a)) | ((uint32_t)__half_as_ushort(__float2half_rn(b)) << 16);
    }
    reinterpret_cast<uint4*>(dst)[i] = make_uint4(o[0], o[1], o[2], o[3]);
  }
  if (over) atomicOr(err, 2);
}

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

}  // namespace

bool encoder_tc_supported(int d, int dff, int dtype, int heads, int M) {
  if (heads < 1 || (d / heads) % 4 != 0 || (size_t)M * 3 * (d / heads) * 4 > 48 * 1024) return false;
  return dtype == Z2Z_DTYPE_BF16 && d % kNT == 0 && dff % kNT == 0 && d <= 4 * kRowThreads * kMaxVec4;
}

// Prompt-sized pass of ONE encoder (thousands of rows): the linear layers run as CTA-pair GEMMs
// that own whole output tiles, so bias, residual and GELU are applied in their epilogues; only
// attention, LayerNorm and pooling remain as separate kernels.
static cudaError_t run_encoder_pass_pair(const CbView& cb, const EncoderArgs& a, const EntryList& el, int E, int R,
                                         bool rows_mapped, Prof* prof, cudaStream_t s) {
  const int d = a.d, dff = a.dff, M = cb.M;
  const int Rt = (R + 7) / 8 * 8;
  const bool half = a.w_half != nullptr;               // fp16 copies of the linear-layer weights exist
  auto Wp = [&](int i) { return reinterpret_cast<const bf16*>(a.w[i]); };
  const int* total = el.row_off + E;                   // packed rows of this pass (device word)
  const bool narrow = d <= 4 * kRowThreads * kNarrowVec4;      // a row fits four float4 per thread: fewer registers, more CTAs per SM
  auto lnk = half ? (narrow ? k_tc_ln_rows<kNarrowVec4, true> : k_tc_ln_rows<kMaxVec4, true>)
                  : (narrow ? k_tc_ln_rows<kNarrowVec4, false> : k_tc_ln_rows<kMaxVec4, false>);
  PairGemmParams g{};
  g.cb = cb; g.el = el; g.R = R; g.Rt = Rt; g.live_rows = total; g.err = a.err;
  auto gemm = [&](const bf16* act, int K, int widx, int J, int epi, float* out, bf16* out_hl) -> cudaError_t {
    PairGemmParams p = g;
    p.J = J; p.bias = a.w[widx + 1]; p.out = out; p.out_hl = out_hl;
    ProfScope ps(prof, kProfEncGemm, 1, s);
    return launch_pair_gemm(p, act, half ? a.w_half[widx] : a.w[widx], K, epi, half, s);
  };
  cudaError_t e = cudaSuccess;
  // The q, k, v of the first layer on the distinct rows, where that can save row tiles: two of them take the
  // clusters one wave, as one does.  (The map takes 9 us instead of 3.5; 8 prompts of 2048 tokens, d = 3072,
  // 19.8 -> 18.4 ms, 16 of 8192 with their positions scored, d = 4096, single operand, 145 -> 137 ms.)
  const bool uniq = a.layers > 0 && R > 512;
  const int* row_uniq = uniq ? el.row_uniq : nullptr;
  {
    ProfScope ps(prof, kProfEncOther, uniq || !rows_mapped ? 2 : 1, s);
    if (uniq) {
      int slots = 2048;
      while (slots < 2 * R) slots *= 2;
      const size_t smem = (size_t)(slots + R) * 4;
      if ((e = cudaFuncSetAttribute(k_tc_row_map<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
      e = launch_pdl(k_tc_row_map<true>, dim3(1), dim3(1024), smem, s, cb, el, E, slots, R);
    } else if (!rows_mapped) {
      e = launch_pdl(k_tc_row_map<false>, dim3(1), dim3(1024), 0, s, cb, el, E, 0, 0);
    }
    if (e != cudaSuccess) return e;
    auto gk = half ? (narrow ? k_tc_gather_ln_packed<kNarrowVec4, true> : k_tc_gather_ln_packed<kMaxVec4, true>)
                   : (narrow ? k_tc_gather_ln_packed<kNarrowVec4, false> : k_tc_gather_ln_packed<kMaxVec4, false>);
    e = launch_pdl(gk, dim3(R), dim3(kRowThreads), 0, s, cb, el, total, row_uniq, reinterpret_cast<const bf16*>(a.table), Wp(0),
                   a.layers ? Wp(1) : Wp(0), a.layers ? Wp(2) : Wp(0), a.X, a.Ahl, d, Rt, a.layers > 0 ? 1 : 0);
    if (e != cudaSuccess) return e;
  }
  const int dh = d / a.heads;
  for (int l = 0; l < a.layers; ++l) {
    const int o = 1 + 12 * l;
    const int* at = l == 0 ? row_uniq : nullptr;
    g.live_rows = at ? at + (size_t)el.chunk * M : total;
    if ((e = gemm(a.Ahl, d, o + 2, 3 * d, kEpiStore, a.QKV, nullptr)) != cudaSuccess) return e;
    g.live_rows = total;
    {
      ProfScope ps(prof, kProfEncOther, 1, s);
      if (dh <= 128 && M <= 4) {
        auto ak = half ? k_tc_attention_rows_warp<4, true> : k_tc_attention_rows_warp<4, false>;
        e = launch_pdl(ak, dim3((E * a.heads + 7) / 8), dim3(256), 0, s, cb, el, a.QKV, at, a.Ahl, E, d, a.heads, Rt);
      } else {
        e = launch_pdl(k_tc_attention_rows, dim3(E, a.heads), dim3(32, M), (size_t)M * 3 * dh * 4, s, cb, el, a.QKV, at, a.Ahl, d,
                       a.heads, Rt, half ? 1 : 0);
      }
      if (e != cudaSuccess) return e;
    }
    if ((e = gemm(a.Ahl, d, o + 4, d, kEpiResid, a.X, nullptr)) != cudaSuccess) return e;
    if (dff > 0) {                                     // dff == 0: attention-only layer
      {
        ProfScope ps(prof, kProfEncOther, 1, s);
        if ((e = launch_pdl(lnk, dim3(R), dim3(kRowThreads), 0, s, total, a.X, Wp(o + 6), Wp(o + 7), a.Ahl, d, Rt)) != cudaSuccess) return e;
      }
      if ((e = gemm(a.Ahl, d, o + 8, dff, kEpiGelu, nullptr, a.Hhl)) != cudaSuccess) return e;
      if ((e = gemm(a.Hhl, dff, o + 10, d, kEpiResid, a.X, nullptr)) != cudaSuccess) return e;
    }
    if (l + 1 < a.layers) {
      ProfScope ps(prof, kProfEncOther, 1, s);
      if ((e = launch_pdl(lnk, dim3(R), dim3(kRowThreads), 0, s, total, a.X, Wp(o + 12), Wp(o + 13), a.Ahl, d, Rt)) != cudaSuccess) return e;
    }
  }
  ProfScope ps(prof, kProfEncOther, 1, s);
  return launch_pdl(k_tc_pool_packed, dim3(E, (d / 4 + kRowThreads - 1) / kRowThreads), dim3(kRowThreads), 0, s, cb, el,
                    a.X, a.cache, a.cache_f32, d);
}

// Bytes of fp16 copies of one encoder's linear-layer weights.
size_t encoder_half_bytes(int d, int dff, int layers) {
  return (size_t)layers * ((size_t)4 * d * d + (size_t)2 * d * dff) * 2;
}

bool encoder_rows_are_prompt_sized(int rows) { return rows >= kPromptPassRows; }

size_t encoder_result_bytes(int R, int d, int dff, int matrices) {
  return (size_t)matrices * ((R + 7) / 8 * 8) * (size_t)(3 * d > dff ? 3 * d : dff) * sizeof(float);
}

// Makes fp16 copies of the linear-layer weights of one encoder in `scratch` and fills
// half_ptrs[i] (host array, ABI tensor order) with their device addresses (nullptr elsewhere).
cudaError_t convert_encoder_weights_to_half(const void* const* w, int d, int dff, int layers, void* scratch,
                                            const void** half_ptrs, int* err_word, Prof* prof, cudaStream_t s) {
  char* dst = reinterpret_cast<char*>(scratch);
  for (int i = 0; i < 1 + 12 * layers; ++i) half_ptrs[i] = nullptr;
  const int n_sm = sm_count();
  for (int l = 0; l < layers; ++l) {
    const int o = 1 + 12 * l;
    const int idx[4] = {o + 2, o + 4, o + 8, o + 10};
    const size_t elems[4] = {(size_t)3 * d * d, (size_t)d * d, (size_t)dff * d, (size_t)d * dff};
    for (int k = 0; k < 4; ++k) {
      if (elems[k] == 0) continue;
      ProfScope ps(prof, kProfEncOther, 1, s);
      k_tc_weights_to_half<<<n_sm * 8, 256, 0, s>>>(reinterpret_cast<const bf16*>(w[idx[k]]),
                                                    reinterpret_cast<__half*>(dst), elems[k] / 8, err_word);
      half_ptrs[idx[k]] = dst;
      dst += elems[k] * 2;
    }
  }
  return cudaGetLastError();
}

// A GEMM of the prompt-sized passes costs ceil(row tiles x column tiles / CTA pairs) waves of its K, so that the
// number of rows in a pass decides how full the last wave is: with d = 3072 passes of 1024 entries (about
// 2400 rows, ten row tiles) left a fifth of the tile slots empty, passes of six or twelve row tiles a
// thirtieth; with d = 4096 nine row tiles fit.
int encoder_pass_rows(long long total, int max_rows, int M, int d, int dff) {
  const int nc = sm_count() / 2;
  const int J[4] = {3 * d, d, dff, d}, K[4] = {d, d, d, dff};
  auto cost = [&](long long rows) {                    // of one pass, in columns of K; the kernels between count too
    const long long t = (rows + 255) / 256;
    long long c = rows > 0 ? 2 * d : 0;
    for (int i = 0; i < (dff > 0 ? 4 : 2); ++i) c += (t * ((J[i] + 255) / 256) + nc - 1) / nc * K[i];
    return c;
  };
  int best = 256;
  long long best_cost = -1;
  for (int rows = 256; rows <= max_rows; rows += 256) {
    const int per = rows - (M - 1);
    const long long c = total / per * cost(rows) + cost(total % per);
    if (best_cost < 0 || c <= best_cost) { best_cost = c; best = rows; }
  }
  return best;
}

cudaError_t run_encoder_pass_tc(const CbView& cb, const EncoderArgs* grp, int ng, const EntryList& el,
                                bool rows_mapped, Prof* prof, cudaStream_t s) {
  const EncoderArgs& a0 = grp[0];
  const int d = a0.d, dff = a0.dff, M = cb.M;
  const int E = a0.entries;
  if (E > el.list || E > 1024 * kMapPerThread) return cudaErrorInvalidValue;
  const int R = a0.rows > 0 ? a0.rows : E * M;         // row capacity of this pass
  // Passes of a call that knows its rows (a0.rows) always take whole tiles in a session of prompt size: their
  // results are then the same bits whatever else is in the call, which stream-K sums are not.
  const bool whole_tiles = R >= kPromptPassRows || (a0.prompt && (a0.rows > 0 || R >= prompt_call_min_rows(d)));
  if (ng == 1 && whole_tiles) return run_encoder_pass_pair(cb, a0, el, E, R, rows_mapped, prof, s);
  const int Rt = (R + 7) / 8 * 8;                      // rows of the result matrix per group
  const int* total = el.row_off + E;                   // packed rows of this pass (device word)
  const int n_sm = sm_count();
  const bool narrow = d <= 4 * kRowThreads * kNarrowVec4;      // a row fits four float4 per thread
  const bool halves = a0.prompt;                       // the call's bits must not depend on who adds first
  const int parts2 = halves ? 2 : 1;
  // (results in four parts have at most 14 tiles of 256 columns: d <= 3584, a narrow row)
  auto rlk = [&](int parts) {
    return parts == 4 ? k_tc_reduce_resid_ln<kNarrowVec4, 4>
           : parts == 2 ? (narrow ? k_tc_reduce_resid_ln<kNarrowVec4, 2> : k_tc_reduce_resid_ln<kMaxVec4, 2>)
                        : (narrow ? k_tc_reduce_resid_ln<kNarrowVec4, 1> : k_tc_reduce_resid_ln<kMaxVec4, 1>);
  };
  float* Y = a0.part;                                  // GEMM results, all zero between GEMMs
  const size_t wide = (size_t)(3 * d > dff ? 3 * d : dff);
  const size_t hs = halves ? (size_t)ng * Rt * wide : 0;
  auto stride = [&](int parts) { return parts == 4 ? hs / 2 : hs; };       // (four matrices of d <= wide / 3 columns)
  const size_t y_bytes = encoder_result_bytes(R, d, dff, ng * (halves ? 2 : 1));
  if (y_bytes > a0.part_bytes) return cudaErrorMemoryAllocation;
  if (a0.layers > 0 && y_bytes > *a0.part_clean) {
    // a clear that is only captured into a graph leaves nothing cleared for calls outside of it
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t ce = cudaStreamIsCapturing(s, &cap);
    if (ce == cudaSuccess)
      ce = cudaMemsetAsync(reinterpret_cast<char*>(Y) + *a0.part_clean, 0, y_bytes - *a0.part_clean, s);
    if (ce != cudaSuccess) return ce;
    if (cap == cudaStreamCaptureStatusNone) *a0.part_clean = y_bytes;
  }
  auto P2 = [&](auto f) { Ptr2 p; p.p[0] = f(grp[0]); p.p[1] = ng > 1 ? f(grp[1]) : f(grp[0]); return p; };
  auto M2 = [&](auto f) { MPtr2 p; p.p[0] = f(grp[0]); p.p[1] = ng > 1 ? f(grp[1]) : f(grp[0]); return p; };
  auto W = [&](int i) { return P2([&](const EncoderArgs& a) { return a.w[i]; }); };
  const MPtr2 X = M2([](const EncoderArgs& a) { return (void*)a.X; });
  const MPtr2 Ahl = M2([](const EncoderArgs& a) { return (void*)a.Ahl; });
  const MPtr2 Hhl = M2([](const EncoderArgs& a) { return (void*)a.Hhl; });
  const MPtr2 cache = M2([](const EncoderArgs& a) { return a.cache; });
  const MPtr2 c32 = M2([](const EncoderArgs& a) { return (void*)a.cache_f32; });
  const Ptr2 table = P2([](const EncoderArgs& a) { return a.table; });

  // one GEMM: activations (hi/lo of packed row r in operand rows 2r, 2r + 1; K columns) x weight
  // [J, K], added into Y[group][Rt][J]
  const bool paired = R > kStreamSingleRows;
  const int ksb = paired ? 1 : stream_gemm_ksb(R);
  StreamGemmMaps maps;
  StreamPairMaps pair_maps;
  int gemms = 0;
  auto gemm = [&](const MPtr2& act, int K, int widx, int J, int parts) -> cudaError_t {
    auto fill = [&](auto p) {
      p.groups = ng; p.ksteps = K / (64 * ksb); p.R = R; p.out = Y; p.J = J; p.Rt = Rt;
      p.rows_dev = total; p.err = a0.err;
      return p;
    };
    auto make = [&](auto& m, auto act_maps) {
      for (int g = 0; g < ng; ++g)
        if (!act_maps(g) || !make_tmap_bf16_kblocks(&m.w[g], grp[g].w[widx], J, K, kNT, ksb)) return false;
      if (ng == 1) { m.w[1] = m.w[0]; for (int i = 0; i < 8; ++i) m.a[1][i] = m.a[0][i]; }
      return true;
    };
    ProfScope ps(prof, kProfEncGemm, 1, s);
    if (paired) {
      if (!make(pair_maps, [&](int g) { return stream_pair_act_maps(pair_maps.a[g], act.p[g], Rt, K); })) return cudaErrorInvalidValue;
      StreamPairParams p = fill(StreamPairParams{});
      p.parts = parts; p.part_stride = stride(parts);
      return launch_stream_pair(p, pair_maps, n_sm, s);
    }
    if (!make(maps, [&](int g) { return stream_gemm_act_maps(maps.a[g], act.p[g], Rt, K, R); })) return cudaErrorInvalidValue;
    StreamGemmParams p = fill(StreamGemmParams{});
    p.half_stride = hs;
    p.peek = gemms++ > 0;              // (the first one starts before the count of its pass is there)
    return launch_stream_gemm(p, maps, n_sm, s);
  };

  // parts of the results of d columns, which the two linear maps that end a half layer have
  auto parts_d = [&](int K) {
    return halves && paired ? stream_pair_parts((long long)ng * ((d + 255) / 256), n_sm / 2, K / 64, R) : parts2;
  };

  if (!rows_mapped) {
    ProfScope ps(prof, kProfEncOther, 1, s);
    launch_pdl(k_tc_row_map<false>, dim3(1), dim3(1024), 0, s, cb, el, E, 0, 0);
  }
  cudaError_t e;
  {
    ProfScope ps(prof, kProfEncOther, 1, s);
    launch_pdl(narrow ? k_tc_gather_ln<kNarrowVec4> : k_tc_gather_ln<kMaxVec4>, dim3(R, ng), dim3(kRowThreads), 0, s, cb, el, total, table, W(0), a0.layers ? W(1) : W(0),
               a0.layers ? W(2) : W(0), X, Ahl, d, a0.layers > 0 ? 1 : 0);
  }
  if (a0.layers == 0) {
    ProfScope ps(prof, kProfEncOther, 1, s);
    launch_pdl(k_tc_pool, dim3(E, ng), dim3(kRowThreads), 0, s, cb, el, X, cache, c32, d);
  }
  const int dh = d / a0.heads;
  for (int l = 0; l < a0.layers; ++l) {
    const int o = 1 + 12 * l;
    const bool last = l + 1 == a0.layers;
    if ((e = gemm(Ahl, d, o + 2, 3 * d, parts2)) != cudaSuccess) return e;
    {
      ProfScope ps(prof, kProfEncOther, 1, s);
      launch_pdl(halves ? k_tc_qkv_attention<true> : k_tc_qkv_attention<false>, dim3(E, a0.heads, ng), dim3(32, M),
                 (size_t)M * 3 * dh * 4, s, cb, el, Y, hs, W(o + 3), Ahl, d, a0.heads, Rt);
    }
    int parts = parts_d(d);
    if ((e = gemm(Ahl, d, o + 4, d, parts)) != cudaSuccess) return e;
    int last_bias = o + 5;                             // bias of the layer's last linear map
    if (dff > 0) {                                     // dff == 0: attention-only layer
      {
        ProfScope ps(prof, kProfEncOther, 1, s);
        launch_pdl(rlk(parts), dim3(R, ng), dim3(kRowThreads), 0, s, total, Y, stride(parts), W(o + 5), X, W(o + 6),
                   W(o + 7), Ahl, d, Rt);
      }
      if ((e = gemm(Ahl, d, o + 8, dff, parts2)) != cudaSuccess) return e;
      {
        ProfScope ps(prof, kProfEncOther, 1, s);
        const long long f4 = (long long)ng * R * (dff / 4);
        const int per_cta = kGeluThreads * kGeluPerThread;
        launch_pdl(halves ? k_tc_reduce_gelu<true> : k_tc_reduce_gelu<false>, dim3((unsigned)((f4 + per_cta - 1) / per_cta)),
                   dim3(kGeluThreads), 0, s, total, Y, hs, W(o + 9), Hhl, dff, R, Rt, ng);
      }
      parts = parts_d(dff);
      if ((e = gemm(Hhl, dff, o + 10, d, parts)) != cudaSuccess) return e;
      last_bias = o + 11;
    }
    {
      ProfScope ps(prof, kProfEncOther, 1, s);
      if (last)
        launch_pdl(parts == 4 ? k_tc_reduce_resid_pool<4> : parts == 2 ? k_tc_reduce_resid_pool<2> : k_tc_reduce_resid_pool<1>,
                   dim3(E, ng, (d / 4 + kRowThreads - 1) / kRowThreads), dim3(kRowThreads), 0, s, cb, el, Y, stride(parts), W(last_bias), X, cache, c32, d, Rt);
      else
        launch_pdl(rlk(parts), dim3(R, ng), dim3(kRowThreads), 0, s, total, Y, stride(parts), W(last_bias), X, W(o + 12),
                   W(o + 13), Ahl, d, Rt);
    }
  }
  return cudaGetLastError();
}

}  // namespace z2z
