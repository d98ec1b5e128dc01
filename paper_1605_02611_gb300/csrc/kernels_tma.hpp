// TMA-staged tensor-core grouped GEMM (tcgen05, BF16 in, FP32 accumulate) for
// the single-pass sigma vector of the group-stacked layout.
#pragma once
#include <cuda.h>  // CUtensorMap (type only; the encoder is reached through the runtime)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

namespace gbdmrg {

// Operand layout of the sigma modes (store and reduce): every BF16 matrix of rows x cols
// is kept in column groups of 8, [cols / 8][slice][rows][8], rows a multiple of 16.  Eight
// columns of consecutive rows are contiguous, so a box copy moves runs of 256 bytes
// (16 rows), lands in shared memory in the K-major layout that the tensor cores read without
// swizzle, and a warp that owns 32 rows writes 512 contiguous bytes.  The slices of a box
// follow one another like further rows, so that one instruction can multiply by several
// slices of B.  The tensor map has four dimensions, (8 columns x 16 rows, row groups, slices,
// column groups).
//
// One term of an output tile: C[128 x n] (-)= A[128 x k] B[n x k]^T (neg bit 0), where A is the
// box of rows [ay, ay + 128) and columns [ax, ax + k) of tensor map amap and B the
// rows [by, by + n) and columns [bx, bx + k) of tensor map bmap; rows outside a map's
// extent read as zero.  ay, by and k are multiples of 16, ax and bx of 8.  A piece, 16
// columns of a term, is one copy per operand that brings all its slices.  The B map's box
// height must be the tile's n.
//
// Exact mode (TM_MODE_EXACT_F64): the operands are integer slices (|x| <= 128, exact in
// BF16) of blocks scaled by powers of two, so every product sum is an exact integer in
// the FP32 accumulator.  A term stands for all slice pairs (i, j), i + j < nsl (neg
// bits 4-7; slice i of map m is map m + i), taken level by level: the pairs of level
// l = i + j form one segment, added with weight 2^(expo[ea] + expo[eb] - 7 (l + 2));
// neg bit 0 negates.  k <= 128, so that the sums stay below 2^24.
struct TmTerm {
  int amap, bmap;
  int ax, ay, bx, by;
  int k, neg;
  int ea, eb;
};

// Output tile over the terms [t0, t1).  n: MMA width (multiple of 16, <= the
// kernel's maximum).
//   store mode (X intermediates, BF16 slices): the output matrix has xrows rows and ldo
//     columns in the layout above, from element xbase.
//     Row r of the tile is its row rowmap[rowmap_off + r] (< 0: skipped), its columns are
//     out_off .. out_off + n.
//   reduce mode (sigma^T, FP32): rows r < m_valid are added (vector reductions) to
//     out + out_off + r * ldo, columns [0, n).
//   pad, nseg (reduce mode): the tile's stages and segments, ceil(products /
//     TM_SEG_PRODUCTS); each segment accumulates in tensor memory on its own and the
//     epilogue adds the segments in FP32.
struct TmTile {
  int t0, t1;
  int n, m_valid;
  int ldo, nseg;
  long out_off;
  long rowmap_off;
  long xbase, xrows;
  int nvalid, pad;  // exact mode: valid columns of the output block; reduce mode: pad = stages
};

//   exact mode (FP64): rows r < m_valid, columns c < nvalid of
//     out + out_off + r * ldo receive the sum of the tile's segments, accumulated in
//     two-float (hi + lo) registers and stored as FP64.
constexpr int TM_MODE_STORE_BF16 = 1, TM_MODE_REDUCE_F32 = 2, TM_MODE_EXACT_F64 = 3;
// bits of the slices of the exact mode
constexpr int TM_EXACT_BITS = 7;
constexpr int TM_PIECE_COLS = 16;  // columns of a piece in the sigma modes: one K=16 instruction per product
// pieces per stage of the sigma modes: several in one pass; one, with all its slices, for two or
// three slices
__host__ __device__ constexpr int tm_slots(int nsl) { return nsl == 1 ? 2 : 1; }
// K=16 products accumulated in tensor memory before the reduce-mode epilogue takes the partial
// sum over (the tensor cores round their running sum toward zero)
constexpr int TM_SEG_PRODUCTS = 64;
// CTAs per SM of a mode
constexpr int tm_ctas(int mode) { return mode == TM_MODE_EXACT_F64 ? 1 : 2; }
// ring of two or three slices: at most TM_MAX_SLOTS slots of one piece in TM_RING_BYTES
constexpr int TM_MAX_SLOTS = 12, TM_RING_BYTES = 108 * 1024;
constexpr int tm_slot_bytes(int nsl, int n) { return ((128 + n) * TM_PIECE_COLS * 2 * nsl + 1023) / 1024 * 1024; }
constexpr int tm_fit_slots(int nsl, int n) {
  return TM_RING_BYTES / tm_slot_bytes(nsl, n) < TM_MAX_SLOTS ? TM_RING_BYTES / tm_slot_bytes(nsl, n) : TM_MAX_SLOTS;
}
// most pieces of a term of two or three slices in a launch whose widest tile has n columns: what its
// ring holds and the straight-line code takes
constexpr int TM_TERM_PIECES = 6;
constexpr int tm_term_pieces(int nsl, int n) {
  return tm_fit_slots(nsl, n) < TM_TERM_PIECES ? tm_fit_slots(nsl, n) : TM_TERM_PIECES;
}
// maximum MMA width of a mode
constexpr int tm_max_n(int mode, int nsl) {
  return mode == TM_MODE_EXACT_F64 ? 64 : mode == TM_MODE_STORE_BF16 && nsl == 1 ? 256 : 128;
}

// Copy lists.  The tiles' terms are expanded before the launch into stages, each holding
// up to tma_pieces(mode, nsl) pieces.  In the sigma modes a piece is 16 columns of one term
// with all slices of both operands: the slice products i + j < nsl come from one pair of
// copies, and a term's pieces stay in the ring until all its products have been issued (slice pair
// by slice pair, each over all pieces), so a term has at most tm_term_pieces of them.
// In the exact mode a term expands into its slice pairs (i, j), i + j < nsl, in the
// order of the level l = i + j (A map amap + i, B map bmap + j), each into boxes of 64
// columns along K, one to a stage.  CTA c of a launch of `grid` CTAs takes the tiles c,
// c + grid, ... and issues the stages [cta_stage[c], cta_stage[c + 1]), stage s with the
// pieces pieces[s * tma_pieces(mode, nsl) + p], p < np.
// A piece's coordinates are columns and rows in the exact mode, column groups (8) and row
// groups (16) in the sigma modes.
struct TmPiece {  // 32 bytes, so that any run of pieces is a bulk copy of 16-byte multiples
  int amap, ax, ay, bmap, bx, by, pad[2];
};
// word: the stage word the MMA issuer reads, the instruction descriptor (negation of A in
// the exact mode) in the low half.  High half, exact mode and one slice: the K=16 instructions
// (exact) or pieces in bits 0-2, flags first of a segment (bit 3), end of a segment (4), last
// stage of the tile (5), with one slice the negation of slot p in bit 8 + p.  Two or three slices:
// the term's pieces in bits 0-7 (read from its first),
// negation (9), last term of the tile (10).  bytes: the stage's expected
// copy bytes.
struct TmStage {
  uint64_t word;
  uint32_t bytes;
  int np;
};
struct TmListsDev {  // device copies, kept alive by the caller for the launches
  int grid = 0, slots = 0, slot_bytes = 0;
  const int* cta_stage = nullptr;
  const TmStage* stages = nullptr;
  const TmPiece* pieces = nullptr;
};
// host side of a launch's lists: its grid and (two or three slices) ring, every CTA's first stage (grid + 1 entries),
// the tiles in stage order (sorder) with their first stages (sfirst), and every term's
// first piece within its tile (tpiece0; a term belongs to one tile)
struct TmListPlan {
  int grid = 0, slots = 0, slot_bytes = 0;
  long total = 0;
  std::vector<int> cta_stage;
  std::vector<int> sorder;
  std::vector<long> sfirst;
  std::vector<int> tpiece0;
};

// instruction descriptor of tcgen05.mma kind::f16: D FP32, A and B BF16, both K-major,
// M = 128, N = n; negA negates A
__host__ __device__ inline uint32_t tm_idesc_bf16(int n, bool negA) {
  uint32_t d = 0;
  d |= 1u << 4;
  d |= 1u << 7;
  d |= 1u << 10;
  if (negA) d |= 1u << 13;
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(128 >> 4) << 24;
  return d;
}

// Host: the stage counts of a launch of `mode` (operands of nsl slices) over these tiles
// (for the grid the launch will use).  The tiles are put in an order that levels the work of the
// CTAs; reduce mode: every tile's pad (its stages) and nseg are set.  Returns false if a term is malformed (k not a positive
// multiple of 16, or longer than tm_term_pieces allows), belongs to two tiles, or the lists would be too long.
bool tma_plan_lists(int mode, int nsl, std::vector<TmTile>& tiles, const std::vector<TmTerm>& terms, TmListPlan& out);
// Device: fills the copy lists (stages: total entries, pieces: total * tma_pieces(mode,
// nsl)), one thread per stage, from the tiles and terms the plan was made from and the plan's
// tpiece0, sorder and sfirst (all on the device).
cudaError_t launch_fill_lists(int mode, int nsl, const TmTile* d_tiles, int ntiles, const TmTerm* d_terms,
                              const int* d_tpiece0, const int* d_sorder, const long* d_sfirst, long total,
                              TmStage* d_stages, TmPiece* d_pieces, cudaStream_t s);
// CTAs of a launch over ntiles tiles (at most ctas per SM of the current device)
int tma_grid(int ctas, int ntiles);
int tma_pieces(int mode, int nsl);

// maps: device array of encoded tensor maps (64-byte aligned).  nsl: BF16 slices of the
// operands (1-3; store mode: also of the results, x = s0 + s1 + ... of every FP32 value).
// err: set to 1 if a bounded wait ran out (the CTA then stops, lets its copies land and frees
// its tensor memory).  lists: the copy lists of these tiles (tma_plan_lists,
// launch_fill_lists), on the device.
cudaError_t launch_gemm_slices(int mode, int nsl, const TmTile* d_tiles, int ntiles, const CUtensorMap* d_maps,
                               const long* d_rowmap, void* out, int* d_err, cudaStream_t s, const TmListsDev& lists);
// the exact mode (d_terms and d_expo: read by its epilogue)
cudaError_t launch_gemm_exact(const TmTile* d_tiles, int ntiles, const TmTerm* d_terms, const CUtensorMap* d_maps,
                              double* out, int* d_err, cudaStream_t s, const TmListsDev& lists, const int* d_expo);

// Exact splitting of FP64 blocks for the exact mode: per job, e = the smallest
// exponent with |scale * x| < 2^e over the block, then nsl (1 to 6) integer slices d_s
// with scale * x * 2^-e = sum_s d_s 2^(-7 (s + 1)) (+ remainder below 2^(-7 nsl)), each
// stored exactly as BF16 (|d_0| <= 128, |d_3| <= 72, the others <= 64), nsl slices
// slice_stride elements apart; columns
// [cols, wcols) are zero.  trans: dst[j * ldd + i] holds element (i, j) (rows of
// the source become columns).  expo[job.expo] receives e.
struct SplitJob {
  const double* src;
  __nv_bfloat16* dst;
  long slice_stride;
  int rows, cols, lds, ldd, wcols, trans, expo;
  double scale;
};
cudaError_t launch_split_exact(const SplitJob* d_jobs, int njobs, int nsl, int* d_expo, cudaStream_t s);
// Host: encode a 2D BF16 tensor map of the exact mode over a row-major matrix (rows x cols,
// leading dimension ld elements, ld * 2 a multiple of 16 bytes, base 16-byte aligned), boxes
// of 64 columns (128-byte swizzle) x box_rows rows.  Returns false on failure.
bool encode_bf16_map(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows);
// Host: encode the 4D map of a matrix in the layout of the sigma modes (rows a multiple of
// 16, cols of 8, nsl slices), boxes of box_rows rows (a multiple of 16, at
// most 256), TM_PIECE_COLS columns and all slices.  Returns false on failure.
bool encode_slice_map(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, int nsl, uint32_t box_rows);

}  // namespace gbdmrg
