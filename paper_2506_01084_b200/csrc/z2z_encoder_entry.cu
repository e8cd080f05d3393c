// Hyper-encoder pass of NARROW models on the CUDA cores (paper Section 2.2; Section 3.1): one
// cluster of four CTAs takes one codebook entry through the whole encoder, both encoders of a step
// in one launch.  Activations never leave shared memory (fp32); weights are read in their storage
// type.
//
// What bounds it: with d <= 256 the weights of a layer are a few hundred KB that stay in L2, and a
// step has at most a handful of entries, so a pass is a chain of small dependent products and not a
// stream.  As one launch per product (13 per layer and encoder, z2z_encoder.cu) that chain cost 5 to
// 11 us per link.  Here a link is: every CTA computes a quarter of the outputs for all rows of the
// entry (each weight is read by one CTA only: one SM alone would need 3 us at d = 64 and 13 us at
// d = 128 to read a layer set at its share of the L2 bandwidth), writes them into the shared memory
// of all four, and the cluster synchronises.  Decode step of the smallest configuration (V = 512,
// d = 64, two layers, both encoders): 251 us in 35 launches before, 46.5 us in 4 with this kernel.  LayerNorm and attention work on a few hundred values
// and are computed by every CTA for itself instead of being exchanged.
#include <cooperative_groups.h>

#include "z2z_common.cuh"
#include "z2z_internal.h"
#include "z2z_simt_tile.cuh"
#include "z2z_sm100.cuh"

namespace z2z {

namespace cg = cooperative_groups;

namespace {

constexpr int kEntryCtas = 4;               // CTAs of a cluster
constexpr int kEntryThreads = 256;
constexpr int kEntryMaxD = 256, kEntryMaxDff = 1024, kEntryMaxLayers = 8;

struct EntrySide {
  const void* table;
  const void* w[1 + 12 * kEntryMaxLayers];
  void* cache;
  float* cache_f32;
};
struct EntryEncoderParams {
  CbView cb;
  EntryList el;
  EntrySide side[2];
  int d, dff, heads, layers;
};

enum { kLinStore = 0, kLinGelu = 1, kLinAdd = 2 };

// out[r][j] (op)= act[r] . W[j] + bias[j] for the CTA's quarter of the J outputs, all L rows, into the
// shared memory of every CTA of the cluster (the same offset in each).  P lanes (a power of two, 4..32)
// share one output: lane p reads the weights of columns 4 p + 4 P i.
template <typename T, int OP>
__device__ __forceinline__ void entry_linear(cg::cluster_group& cluster, const float* act, int K, int L, const T* __restrict__ W,
                                             const T* __restrict__ bias, int J, float* out) {
  const int per = (J + kEntryCtas - 1) / kEntryCtas;
  const int j_lo = (int)cluster.block_rank() * per;
  const int j_hi = j_lo + per < J ? j_lo + per : J;
  int P = 32;
  while (P > 4 && (per * P > kEntryThreads || 4 * (P >> 1) >= K)) P >>= 1;
  const int p = threadIdx.x & (P - 1);
  const int groups = kEntryThreads / P;
  for (int j0 = j_lo; j0 < j_hi; j0 += groups) {              // uniform trip count: the shuffles need all lanes
    const int j = j0 + (int)threadIdx.x / P;
    const bool on = j < j_hi;
    float acc[kMaxM];
#pragma unroll
    for (int r = 0; r < kMaxM; ++r) acc[r] = 0.f;
    if (on) {
      const T* wr = W + (size_t)j * K;
#pragma unroll 4
      for (int k = p * 4; k < K; k += P * 4) {
        float w[4];
        load4<T>(wr + k, w);
#pragma unroll
        for (int r = 0; r < kMaxM; ++r) {
          if (r < L) {
            const float4 x = *reinterpret_cast<const float4*>(act + (size_t)r * K + k);
            acc[r] = fmaf(x.x, w[0], fmaf(x.y, w[1], fmaf(x.z, w[2], fmaf(x.w, w[3], acc[r]))));
          }
        }
      }
    }
    const float bj = on ? to_f32<T>(bias[j]) : 0.f;
#pragma unroll
    for (int r = 0; r < kMaxM; ++r) {
      if (r < L) {
        float v = acc[r];
        for (int o = P >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (on && p == (r & (P - 1))) {
          v += bj;
          if (OP == kLinGelu) v = 0.5f * v * (1.0f + erff(v * 0.70710678118654752440f));
          float* dst = out + (size_t)r * J + j;
          if (OP == kLinAdd) v += *dst;                        // every CTA holds the same residual
#pragma unroll
          for (int c = 0; c < kEntryCtas; ++c) *cluster.map_shared_rank(dst, c) = v;
        }
      }
    }
  }
}

// A[r] = LayerNorm(X[r]) * g + b: one warp per row.
template <typename T>
__device__ __forceinline__ void entry_layernorm(const float* X, const T* __restrict__ g, const T* __restrict__ b, float* A,
                                                int d, int L) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= L) return;
  const float* x = X + (size_t)warp * d;
  float s = 0.f;
  for (int c = lane; c < d; c += 32) s += x[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const float mean = s / (float)d;
  float q = 0.f;
  for (int c = lane; c < d; c += 32) { const float t = x[c] - mean; q += t * t; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  const float rstd = 1.0f / sqrtf(q / (float)d + kLnEps);
  float* a = A + (size_t)warp * d;
  for (int c = lane; c < d; c += 32) a[c] = (x[c] - mean) * rstd * to_f32<T>(g[c]) + to_f32<T>(b[c]);
}

// Bidirectional attention inside the entry: one warp per (head, query row).
__device__ __forceinline__ void entry_attention(const float* QKV, float* O, int d, int heads, int L) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int dh = d / heads;
  const float scale = 1.0f / sqrtf((float)dh);
  for (int item = warp; item < heads * L; item += kEntryThreads / 32) {
    const int h = item / L, i = item - h * L;
    const float* q = QKV + (size_t)i * 3 * d + h * dh;
    float s[kMaxM];
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < kMaxM; ++j) {
      s[j] = -INFINITY;
      if (j < L) {
        const float* kp = QKV + (size_t)j * 3 * d + d + h * dh;
        float t = 0.f;
        for (int c = lane; c < dh; c += 32) t = fmaf(q[c], kp[c], t);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        s[j] = t * scale;
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
        if (j < L) v = fmaf(s[j] * inv, QKV[(size_t)j * 3 * d + 2 * d + h * dh + c], v);
      O[(size_t)i * d + h * dh + c] = v;
    }
  }
}

// grid (entries * kEntryCtas, encoders), dynamic shared memory entry_smem_bytes().
template <typename T>
__global__ void __cluster_dims__(kEntryCtas, 1, 1) __launch_bounds__(kEntryThreads)
k_enc_entry(const __grid_constant__ EntryEncoderParams p) {
  extern __shared__ __align__(16) float s_act[];
  cg::cluster_group cluster = cg::this_cluster();
  sm100::pdl_trigger();
  sm100::pdl_wait();                               // the work list comes from an earlier kernel
  const CbView& cb = p.cb;
  const int d = p.d, dff = p.dff;
  const int e = blockIdx.x / kEntryCtas;
  const EntrySide& sd = p.side[blockIdx.y];
  const int L = p.el.len[e];
  if (L <= 0) return;                              // the same for all four CTAs
  auto W = [&](int i) { return reinterpret_cast<const T*>(sd.w[i]); };
  float* X = s_act;                                // [L][d]
  float* A = X + (size_t)cb.M * d;                 // [L][d]
  float* QKV = A + (size_t)cb.M * d;               // [L][3 d]
  float* H = QKV + (size_t)cb.M * 3 * d;           // [L][dff]
  const T* table = reinterpret_cast<const T*>(sd.table);
  for (int i = threadIdx.x; i < L * d; i += kEntryThreads) {
    const int r = i / d, c = i - r * d;
    X[i] = to_f32<T>(table[(size_t)p.el.tok[e * cb.M + r] * d + c]) + to_f32<T>(W(0)[(size_t)r * d + c]);
  }
  cluster.sync();                                  // all four CTAs run before anyone writes into another's memory
  for (int l = 0; l < p.layers; ++l) {
    const int o = 1 + 12 * l;
    entry_layernorm<T>(X, W(o + 0), W(o + 1), A, d, L);
    __syncthreads();
    entry_linear<T, kLinStore>(cluster, A, d, L, W(o + 2), W(o + 3), 3 * d, QKV);
    cluster.sync();
    entry_attention(QKV, A, d, p.heads, L);
    __syncthreads();
    entry_linear<T, kLinAdd>(cluster, A, d, L, W(o + 4), W(o + 5), d, X);
    cluster.sync();
    if (dff == 0) continue;                        // attention-only layer
    entry_layernorm<T>(X, W(o + 6), W(o + 7), A, d, L);
    __syncthreads();
    entry_linear<T, kLinGelu>(cluster, A, d, L, W(o + 8), W(o + 9), dff, H);
    cluster.sync();
    entry_linear<T, kLinAdd>(cluster, H, dff, L, W(o + 10), W(o + 11), d, X);
    cluster.sync();
  }
  if (cluster.block_rank() != 0) return;           // (the last cluster barrier is behind all remote writes)
  const size_t dst = ((size_t)p.el.seq[e] * cb.cap + p.el.idx[e]) * d;
  const float inv = 1.0f / (float)L;
  for (int c = threadIdx.x; c < d; c += kEntryThreads) {
    float v = 0.f;
    for (int r = 0; r < L; ++r) v += X[(size_t)r * d + c];
    v *= inv;
    reinterpret_cast<T*>(sd.cache)[dst + c] = from_f32<T>(v);
    if (sd.cache_f32) sd.cache_f32[dst + c] = v;
  }
}

size_t entry_smem_bytes(int M, int d, int dff) { return (size_t)M * (5 * d + dff) * sizeof(float); }

}  // namespace

// Narrow models: at d = 256 a layer set is 6 MB, which four SMs still read in about 13 us; wider ones
// are a stream that needs all SMs (z2z_encoder.cu, z2z_encoder_tc.cu).  And few entries: every one reads all
// weights again, so that the time grows with each wave of some 36 clusters, while the tiled kernels of
// z2z_encoder.cu take about as long for 200 entries as for one (us for 64 / 96 / 128 / 1024 entries of one
// fp32 encoder of two layers, dff = 4 d, here and there: d = 64 66 93 119 828 / 134 134 134 172, d = 128 95 138 178
// 1291 / 179 179 179 241, d = 192 156 230 301 2224 / 234 234 234 337, d = 256 195 290 380 2851 / 281 281 282 552).
bool encoder_entry_applies(int d, int dff, int layers, int entries) {
  return d <= kEntryMaxD && dff <= kEntryMaxDff && layers <= kEntryMaxLayers && entries <= (d <= 192 ? 96 : 72);
}

cudaError_t run_encoder_entries(const CbView& cb, const EncoderArgs* grp, int ng, const EntryList& el, Prof* prof,
                                cudaStream_t s) {
  const EncoderArgs& a = grp[0];
  const int E = a.entries < el.chunk ? a.entries : el.chunk;
  EntryEncoderParams p{};
  p.cb = cb; p.el = el; p.d = a.d; p.dff = a.dff; p.heads = a.heads; p.layers = a.layers;
  for (int g = 0; g < ng; ++g) {
    p.side[g].table = grp[g].table;
    for (int i = 0; i < 1 + 12 * a.layers; ++i) p.side[g].w[i] = grp[g].w[i];
    p.side[g].cache = grp[g].cache;
    p.side[g].cache_f32 = grp[g].cache_f32;
  }
  const size_t smem = entry_smem_bytes(cb.M, a.d, a.dff);
  auto kern = a.dtype == Z2Z_DTYPE_FP32 ? k_enc_entry<float> : k_enc_entry<__nv_bfloat16>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  ProfScope ps(prof, kProfEncGemm, 1, s);
  return launch_pdl(kern, dim3(E * kEntryCtas, ng), dim3(kEntryThreads), smem, s, p);
}

}  // namespace z2z
