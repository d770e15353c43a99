// Exact sliced-product GEMM on the tcgen05 tensor cores (ozaki.cu).
//
// An FP64 operand row is split, per block of KB consecutive K elements, into S
// integer "slices" of W bits under a common power-of-two exponent e:
//     x = 2^e sum_{s<S} a_s 2^{-W(s+1)},  a_0 in [-2^W, 2^W], |a_s| <= 2^(W-1),
// each a_s stored exactly as BF16.  A K-block sum of slice products stays within
// 2^24, so the FP32 tensor core accumulation is exact whatever its internal
// rounding.  Products with s + t = l share TMEM accumulator l; levels l < S are
// kept (error about 2^-WS of |A||B| per term), combined exactly in integers and
// added to FP64 accumulators once per K-block with scale 2^(eA + eB).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dfjk {

// Formats: S slices of W bits under one exponent per K block of KB elements.  The
// leading digit has one bit more, in [-2^W, 2^W]; KB keeps every level sum
// (l + 1 products) within 2^24.
//   OZ_36   6 x 6 bits: X = B C and K of the mixed path
//   OZ_48   8 x 6 bits: its whitening (L^-1 amplifies the rounding)
//   OZ_F64  8 x 7 bits: the dense products of the FP64 path; 56 bits below a row's
//           largest element, dropped products below 2^-57 of |A||B| per term
//           (FP64 rounds its sums to 2^-53)
enum : int { OZ_36 = 0, OZ_48 = 1, OZ_F64 = 2 };
template <int F>
struct OzFmt {
  static constexpr int S = F == OZ_36 ? 6 : 8, W = F == OZ_F64 ? 7 : 6, KB = F == OZ_F64 ? 384 : 1024;
};
inline int oz_slices(int fmt) { return fmt == OZ_36 ? 6 : 8; }
inline int oz_kblock(int fmt) { return fmt == OZ_F64 ? OzFmt<OZ_F64>::KB : OzFmt<OZ_36>::KB; }
constexpr int OZ_BM = 128, OZ_BN = 64;
constexpr int OZ_BK = 16;   // K per stage of the GEMM (operands are padded to it)

// An operand in sliced form, stored as images of the GEMM's shared-memory
// stages: [batch][row tile of R rows][K step of 16][K group of 8][slice][R rows][8]
// (BF16), so that a stage is contiguous in memory and the 8-row groups of a
// K group are the 128-byte core matrices the tensor core reads.  R is 128 for an
// A operand and 64 for a B operand; an operand that serves as both has 128.
// Exponents: [batch][rows_pad][nkb] (int32).  Rows >= rows of the last tile are
// not defined when a kernel writes `rows` rows only (their products land in
// outputs that are not stored); K beyond the operand's K is zero.
struct SlicedOp {
  __nv_bfloat16 *data = nullptr;
  int *expo = nullptr;
  int batch = 1, fmt = 0, S = 0, rows = 0, rows_pad = 0, K = 0, nks = 0, nkb = 0, row_tile = 0;
  size_t data_bytes() const { return (size_t)batch * S * rows_pad * nks * OZ_BK * sizeof(__nv_bfloat16); }
  size_t expo_bytes() const { return (size_t)batch * rows_pad * nkb * sizeof(int); }
};

// Sizes an operand (rows padded to `row_tile`, K to OZ_BK) and allocates it.
void oz_alloc(SlicedOp &op, int batch, int fmt, int rows, int K, int row_tile);
void oz_free(SlicedOp &op);
// Bytes of the slices of one batch of such an operand.
size_t oz_bytes(int fmt, int rows, int K, int row_tile);
// A view of op's buffers sized for `rows` rows and K columns (at most the
// allocated rows and K): the layout a fresh allocation of that size would
// have, placed at the start of op's buffers.  Used for the short last chunk
// of a chunked reduction without reallocating.
SlicedOp oz_view(const SlicedOp &op, int rows, int K);

// The kept partners of every AO, for the X GEMM over kept pairs only.  AOs with
// the same partners (the functions of a shell) form a group; group g's list holds
// its partners' AO indices in ascending order, padded with -1 to whole K steps
// (at least one), at list[16 gstep[g]]; AO mu's operand rows are counted by
// zstep in the same way.  All arrays are on the device.
struct PairLists {
  int fmt = OZ_36;                  // slice format of the operands built from the lists
  int ngroup = 0, nkb = 1;          // nkb: K blocks of the longest list
  int longest = 0;                  // entries of the longest list, padded
  long long steps = 0, gsteps = 0;  // K steps over all AOs, over all groups
  const int *list = nullptr, *gstep = nullptr, *zstep = nullptr, *zgroup = nullptr;
  const int *krow = nullptr;      // row of B per (AO, list entry), -1 in the padding
};
// Fills krow (16 pl.steps ints) from the lists and the row map (null: B holds every
// pair, row mu nao + nu).
void oz_krow(const PairLists &pl, const int *rowmap, int nao, int *krow, cudaStream_t st);

// Fills `op` from the FP64 view x(z, r, k) = src[z sz + r sr + k sk]
// (rows >= op.rows and k >= op.K are zero); sr or sk must be 1.
// rows_per_block: rows of a K-contiguous source per block (8, 16 or 32; 0 = the
// default, 16, or DFJK_SLICE_ROWS).
void oz_slice_f64(const double *src, long long sz, long long sr, long long sk, SlicedOp &op,
                  cudaStream_t st, int rows_per_block = 0);

// The same from rows of double-single pairs (K-contiguous, rows sr apart): the
// digits come from the two FP32 parts with integer arithmetic alone.
void oz_slice_df(const float2 *src, long long sr, SlicedOp &op, cudaStream_t st, int rows_per_block = 0);

struct OzGemmArgs {
  int M = 0, N = 0, K = 0;
  int nz = 1;            // grid z: batches, or split-K parts
  int a_batched = 0;     // A indexed by z
  int b_batched = 0;     // B indexed by z
  int kb_per_split = 0;  // >0: z selects K-blocks [z kb_per_split, (z+1) kb_per_split)
  int k_upto_n = 0;      // K limited to < end of the N tile (B lower triangular)
  int lower_only = 0;    // skip tiles strictly above the diagonal
  int mode = 0;          // 0: out[z out_bs + m ldo + n] = C;
                         // 1: row m to out[(mu nao + nu) ldo + n] and out[(nu nao +
                         //    mu) ldo + n], mu = colmu[m] (none if < 0), nu = colnu[m]
                         // 2: split-K in order, out[m ldo + n] (+)= C of split z
                         //    after splits 0..z-1
                         // 3: out[z out_bs + n ldo + m] = C (transposed)
                         // (1 to 3: persistent kernel only)
  const int *colmu = nullptr, *colnu = nullptr;
  int nao = 0;
  int *tile_seq = nullptr;  // mode 2: per (tile, drain warp) split counters
  int accumulate = 0;    // mode 2: split 0 also adds onto out (a later chunk of
                         // the reduction range, in chunk order)
  double *out = nullptr;
  long long ldo = 0, out_bs = 0;
  int *status = nullptr;       // STATUS_TIMEOUT on an expired wait
  long long timeout = 1 << 26; // polls per mbarrier wait
  int phase = -1;              // phase timer id of this launch (-1: none)
  // ragged batches (zstep != nullptr): batch z stands for AO z0 + z of the pair
  // lists; its K is its own list's, its B operand its group's (B holds the
  // groups from g0 on), and its output is out[(z0 + z) out_bs + ..]
  const int *zstep = nullptr, *zgroup = nullptr, *gstep = nullptr;
  int z0 = 0, g0 = 0;
  int *tile_ctr = nullptr;     // device int for the dynamic tile queue; oz_gemm
                               // zeroes it on the stream, so launches that can
                               // run concurrently need distinct counters
};

// B stored by rows of ldb doubles (P contiguous), one row per kept AO pair, as the
// A operand of the X GEMM: batch mu, rows P, K = mu's kept partners.
// The exponents (one per K block) for every mu and the rows P of columns [0, rows) of `B`, written
// as rows pcol.. of expo[(mu pre_rows + P) nkb + kb] (prows of them, a multiple
// of 32; 0 beyond `rows`).  B does not change between builds, so a handle
// computes them once.
void oz_expo_pairs(const double *B, long long ldb, int rows, const PairLists &pl, int nao, int prows, int pcol,
                   int pre_rows, int *expo, cudaStream_t st);
// The slices of the columns [0, rows) of `B` for all mu, with the exponents from
// oz_expo_pairs (`expo` points at the first of these rows).  Bytes of `out`:
// oz_pairs_bytes.  warps: warps per block (4, 8 or 16; 0 = the default, 8, or
// DFJK_PSLICE_ROWS).
void oz_slice_pairs(const double *B, long long ldb, int rows, const PairLists &pl, int nao, const int *expo,
                    int pre_rows, __nv_bfloat16 *out, cudaStream_t st, int warps = 0);
inline size_t oz_pairs_bytes(int fmt, long long steps, int rows) {
  return (size_t)steps * oz_slices(fmt) * OZ_BK * sizeof(__nv_bfloat16) * (size_t)((rows + OZ_BM - 1) / OZ_BM * OZ_BM);
}
// C[nu][i] = C[nu ldc + i ldi] (i < nocc) as the B operands of groups [g0, g1): op.rows =
// nocc, row tiles of 64, exponents [g - g0][rows_pad][nkb].
void oz_slice_c(const double *C, long long ldc, long long ldi, int nocc, const PairLists &pl, int g0, int g1, SlicedOp &op,
                cudaStream_t st);

// True when DFJK_OZ_SIMPLE=1 selects the one-tile-per-CTA kernel (no mode 2).
bool oz_simple_mode();
// Counters mode 2 needs for a launch of M x N (ints).
size_t oz_tile_seq_count(int M, int N);

// out = A B^T with A (M x K) and B (N x K) in sliced form, both with S slices.
void oz_gemm(const SlicedOp &A, const SlicedOp &B, const OzGemmArgs &g, cudaStream_t st);

}  // namespace dfjk
