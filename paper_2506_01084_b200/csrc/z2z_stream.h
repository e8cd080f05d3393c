// Parameters of the tcgen05 weight-streaming kernels (z2z_stream.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "z2z_common.cuh"
#include "z2z_internal.h"

namespace z2z {

constexpr int kMaxStages = 8;
constexpr int kGemmNT = 128;                    // weight rows per tile of the stream-K GEMM

constexpr int kLogitNT = 256;                   // weight rows per job of the logits kernel at most
constexpr int kLogitGran = 32;                  // scheduling granule of the logits kernel, in weight rows (TMA boxes of
                                                // fewer rows stream several times slower)
constexpr int kLogitBoxClasses = 4;             // TMA boxes of 32, 64, 128 and 256 weight rows

// Tensor maps of the logits kernel: hidden rows (all of them), W_U and U_h once per box size, and for the short jobs of
// a sequence's hypertokens a group of 8 hidden rows and boxes of 32, 64 or 128 rows of U_h with logit_short_kb k-blocks.
constexpr int kLogitShortClasses = 3;
__host__ __device__ constexpr int logit_short_kb(int cls) { return cls == 2 ? 2 : 4; }
struct LogitMaps {
  CUtensorMap h;
  CUtensorMap w[2 * kLogitBoxClasses];
  CUtensorMap h8[3];     // 1, 2 and 4 k-blocks
  CUtensorMap u[kLogitShortClasses];
  CUtensorMap h2, u2[2]; // two k-blocks of all hidden rows, and of 32 or 64 rows of U_h: for sequences with rows in several groups
};

// ---- decode logits kernel (z2z_decode_logits.cu) ---------------------------------------------
// Tensor maps, all of the form [k-block][row][64 columns]: hidden rows as one resident operand
// (h) and per stage with 1, 2 or 4 k-blocks (hk[0..2]); W_U and U_h as boxes of 64 rows x 2
// k-blocks (class 1) and 128 rows x 1 k-block (class 2): w[tensor * 2 + (class == 2)].
struct DecodeLogitMaps {
  CUtensorMap h, hk[3];
  CUtensorMap w[4];
};
struct DecodeLogitsParams {
  CbView cb;
  LogitsArgs la;
  int ksteps;            // d / 64 (a multiple of 2)
  int hid_rows;          // hidden rows held per k-block in shared memory (N rounded up to 8)
  int hid_box_kb;        // k-blocks per TMA box of the resident hidden rows
  int stages;            // stages of the load ring
  int part_stride;       // partial slots per hidden row
  int fixed_granules;    // 64-row granules of W_U every CTA owns up front
  int* counters;         // device words: [0] pool claims, [1] CTAs finished (both return to 0)
  int* err;
};
bool make_tmap_bf16_kblocks(CUtensorMap* m, const void* base, long long rows, long long cols, int box_rows,
                            int box_kb);
bool decode_logits_applies(const LogitsArgs& a);
cudaError_t run_logits_decode(const CbView& cb, const LogitsArgs& a, int* counters, int* err_word,
                              LogitsPartInfo* info, Prof* prof, cudaStream_t s);

// Stream-K GEMM over `groups` independent problems of identical shape (the two hyper-encoders).
// The unit space is (group, weight tile, k-step); CTA c of G owns units
// [floor(cU/G), floor((c+1)U/G)).  Every maximal run of units inside one tile and one CTA is one
// accumulator.  Operands are swapped with respect to the result's orientation: the 128 weight rows
// of a tile are the MMA's M, the activation rows its N, and a thread of the epilogue owns one
// output feature.
//
// The activation operand holds the hi part and the lo part of PACKED row r in rows 2r and 2r + 1
// (bf16 [2 * Rt, K]); only the first *rows_dev packed rows carry data, a count that only the device
// knows.  The TMA box and the MMA's N follow it: loads, tensor-core work and the epilogue's
// reductions grow with the number of rows that exist, not with the capacity of the pass.  The
// epilogue adds the hi and lo columns of a row in registers and reduces the sums into the fp32
// result matrix out[group][Rt][J] (lanes = consecutive features = consecutive addresses).
//
// Three or more sums that meet in one word of the result are added in the order in which they arrive, and
// their rounding depends on it.  With half_stride > 0 the two halves of K have a result matrix each and the
// work is cut so that at most two sums meet in a word (0 + a + b = 0 + b + a): the same call then
// gives the same bits.  The kernel that reads the results adds the two matrices.
// The caller fills the first block of fields, the launch the second.
struct StreamGemmParams {
  int groups, ksteps;    // ksteps = K / (64 * ksb), ksb = 64-column k-blocks per stage and TMA box
  int R;                 // row capacity of the pass
  float* out;            // [groups][Rt][J] fp32, zero before the first add
  int J, Rt;
  size_t half_stride;    // floats from the result matrix of K's first half to that of its second, or 0
  const int* rows_dev;   // device word: packed rows that carry data (<= R)
  int peek;              // look at it before the preceding kernel is done: no weights ahead when it holds 0
  int* err;

  int tiles_per_group;
  int a_box_rows, box_step;   // most operand rows of a box; boxes are multiples of box_step rows
};
struct StreamGemmMaps {
  CUtensorMap a[2][8];   // activation operand of each group, boxes of 1 .. 8 steps
  CUtensorMap w[2];      // weights of each group, 128 rows
};
// Workers (CTAs or clusters, `most` at most) for `tiles` tiles so that no part of a tile's K range is cut
// more than once: pieces no shorter than a part, or equal ones whose cuts fall into different parts (of two
// parts: 2, 3, 4 per tile; of four: 5, 6 and 8, but not 7).
inline int fixed_order_workers(long long tiles, int most, int parts) {
  if (parts * tiles >= most) return most;
  long long per = most / tiles < 2 * parts ? most / tiles : 2 * parts;
  if (parts == 4 && per == 7) per = 6;
  return (int)(tiles * per);
}
int stream_gemm_ksb(int R);
bool stream_gemm_act_maps(CUtensorMap* maps, const void* act, int Rt, int K, int R);
// At most 128 rows, one CTA per tile of 128 weight rows.
cudaError_t launch_stream_gemm(StreamGemmParams p, const StreamGemmMaps& maps, int n_sm, cudaStream_t s);

// The same product for more than 128 rows on CTA pairs (z2z_stream_pair.cu): up to 256 packed rows ride on one stream of the
// weights, and more run as blocks of 256.
struct StreamPairParams {
  int groups, ksteps;    // ksteps = K / 64
  int R;
  float* out;
  int J, Rt;
  int parts;             // result matrices: 1, or 2 or 4 for as many equal parts of K
  size_t part_stride;    // floats from one of them to the next
  const int* rows_dev;
  int* err;

  int tiles_per_group;   // tiles of 256 weight rows
  int blocks;            // blocks of 256 packed rows the capacity asks for
  int act_bytes;         // activation part of a stage
  int stages;
};
struct StreamPairMaps {
  CUtensorMap a[2][8];   // activation operand of each group, boxes of 16, 32, .. 128 rows
  CUtensorMap w[2];      // weights of each group, 128 rows
};
// Parts of K for a pass of R rows whose bits must not depend on who adds first.  Two parts keep four clusters per
// tile busy at most and four keep eight, but the kernel after the GEMM then reads and clears four matrices.
// z2z_hyper_embed bounded to R rows, us with two parts -> with four: eight clusters per tile, d = 1024 192 / 384 /
// 639 rows 138 -> 131, 198 -> 178, 288 -> 260, d = 2048 197 -> 178, 329 -> 297, 466 -> 414; six per tile, d = 3072
// 300 / 384 / 639 rows 325 -> 333, 466 -> 458, 703 -> 654.
inline int stream_pair_parts(long long tiles, int most, int ksteps, int R) {
  const int pays = R >= 384 ? 5 : 8;                             // clusters per tile from which four parts pay
  return pays * tiles <= most && ksteps % 4 == 0 ? 4 : 2;
}
bool stream_pair_act_maps(CUtensorMap* maps, const void* act, int Rt, int K);
cudaError_t launch_stream_pair(StreamPairParams p, const StreamPairMaps& maps, int n_sm, cudaStream_t s);

struct StreamLogitsParams {
  CbView cb;
  LogitsArgs la;
  int ksteps;
  int a_box_rows;
  int part_stride;       // partial slots per row
  int* err;
};

// Logits kernel for many rows (z2z_prefill_logits.cu): CTA pairs, tiles of 256 x up to 256.
constexpr int kPrefillMaxStrips = 8;            // column strips a row tile is cut into when there are many row tiles
struct PrefillLogitsParams {
  CbView cb;
  LogitsArgs la;
  int ksteps;            // d / 64
  int row_tiles;         // ceil(N / 256)
  int cta_rows;          // hidden rows per CTA (128, fewer when there are few rows in all)
  int n_static;          // 64-column granules of W_U
  int strips;            // column strips per row tile = partial reductions per hidden row
  int stages;            // of the load ring
  int32_t* tile_lo;      // [row_tiles] lowest / highest sequence owning a row of the tile
  int32_t* tile_hi;
  int32_t* tile_nh;      // [row_tiles] cost of the tile's hypertoken columns
  int* err;
};

// CTA-pair GEMM of the prompt-sized hyper-encoder passes (z2z_pair_gemm.cu).
enum { kEpiStore = 0, kEpiResid = 1, kEpiGelu = 2 };
struct PairGemmParams {
  CbView cb;
  EntryList el;
  int R, Rt;             // row capacity of the pass; rows per hi (or lo) block of the operands
  const int* live_rows;  // device word: packed rows that carry data (rows of live entries, no padding)
  int J;                 // output columns (a multiple of 128)
  const void* bias;      // [J] bf16
  float* out;            // kEpiStore / kEpiResid: fp32 [R, J]
  __nv_bfloat16* out_hl; // kEpiGelu: bf16 [2 Rt, J], hi rows then lo rows (single fp16 operand: fp16 [Rt, J])
  int ksteps, row_tiles, col_tiles;
  int tile_cols;         // columns per tile: 256, 128 or 64
  int* err;
};
cudaError_t launch_pair_gemm(const PairGemmParams& p, const void* act, const void* W, int K, int epi, bool half,
                             cudaStream_t s);

bool make_tmap_bf16(CUtensorMap* m, const void* base, long long rows, long long cols, int box_rows);

}  // namespace z2z
