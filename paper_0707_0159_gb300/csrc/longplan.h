// Work lists of the two-pass H·v, shared by dense and sector-restricted superblocks.
// Internal header.
//
// Each column-major matrix V_q (one for a dense superblock) is cut along one dimension
// only, the one the operator blocks act on:
//   pass 0 (V H_r^T): columns in segments; Y(:, c) = sum_e V(:, c_e) R_e^T over all rows;
//   pass 1 (H_l V):   rows in segments;    Y(r, :) += sum_e L_e V(r_e, :) over all columns.
// An item is some indices of one segment by a range of the long dimension.  The scalar
// tile moves run in a kernel of their own afterwards.
#pragma once
#include <cstdint>
#include <vector>

#include "common.h"

namespace dmrg2d {

constexpr int LP_ROWS = 64;  // segment indices per item
constexpr int FX_LONG = 128; // long indices per item of the split-operand kernel

struct LSeg {
  long long base;  // first element of V_q
  int ld, nlong;   // leading dimension; extent of the long dimension
  int off, dim, dim_pad;  // segment: offset, indices, indices with padding
  int kb, ke;      // operator blocks ks[kb..ke)
  int ub, ue;      // the same blocks as units[ub..ue)
  int e0;          // first entry of the segment's operator rows in opE
  int head;        // extra exponent bits of the operator side (K above 256)
};
struct LK {
  long long op;    // element offset of the block (row-major dim x kdim)
  int v_off, kdim; // first index of the source segment in V_q; its extent
};
struct LUnit {     // up to 8 consecutive K of one block
  long long op;    // element offset of row 0, first K
  int v, kdim, n;  // first index in V_q; row length of the block; K in this unit
};
struct LItem {
  int seg, s0, cnt, x0;  // segment; its indices s0 .. s0 + cnt; first long index
};
struct MoveRec {    // scalar move: first element and ld of its source
  long long src;
  int ld;
  float c32;
  double c64;
};
struct MoveItem {   // columns c_in .. c_in + ncol of a destination block
  long long dst;    // its first element
  int ld, dim, nquad;  // leading dimension, rows, fours of rows (with padding)
  int c_in, ncol, mb, me;  // moves[mb..me)
  long long group;  // blocks of one group share their sources
};

struct LongPlan {
  std::vector<LSeg> segs[2];
  std::vector<LK> ks[2];
  std::vector<MoveRec> mrec;
  std::vector<MoveItem> mitems;
  bool quads = true;  // every row of fours lies inside its matrix and is 4-aligned
  const double *op64[2] = {nullptr, nullptr};  // device blocks: [0] H_r, [1] H_l
  const float *op32[2] = {nullptr, nullptr};
  // derived (lp_finalise)
  std::vector<LUnit> units[2];
  std::vector<LItem> items[2], items32[2], fitems[2];  // FP64, FP32, FP64X
  LSeg* d_segs[2] = {nullptr, nullptr};
  LK* d_ks[2] = {nullptr, nullptr};
  LUnit* d_units[2] = {nullptr, nullptr};
  LItem *d_items[2] = {nullptr, nullptr}, *d_items32[2] = {nullptr, nullptr}, *d_fitems[2] = {nullptr, nullptr};
  int* d_opE[2] = {nullptr, nullptr};  // largest exponent field of every operator row
  MoveRec* d_mrec = nullptr;
  MoveItem* d_mitems = nullptr;
  int* err = nullptr;
  int sms = 1;
  std::vector<void*> allocs;
};

// Moves of one destination block: appends its items (columns in chunks).  A move keeps the
// block-1 and the block-4 sector, so all sources of a block lie in its `group` (one per pair
// of sectors); lp_finalise orders the items by group and chunk.
void lp_add_moves(LongPlan* L, int group, long long dst, int ld, int dim, int dim_pad, int ncols,
                  int mb, int me);
// Cuts the segments into items and uploads everything; op64 / op32 must be set.
int lp_finalise(dmrg2d_ops* ops, LongPlan* L, cudaStream_t s);
void lp_release(LongPlan* L);
int lp_read_error(const LongPlan* L, int* code);

// y = V H_r^T + H_l V by the plan (no scalar moves); the padding rows of row segments are
// written as zero.
int lp_launch_f64(const LongPlan* L, const double* v, double* y, cudaStream_t s);
int lp_launch_f32(const LongPlan* L, const float* v, float* y, cudaStream_t s);
// the same in FP64X: operands split into fixed-point FP16 digits on the tensor cores
int fx_launch(const LongPlan* L, const double* v, double* y, cudaStream_t s);
void fx_opE(LongPlan* L, cudaStream_t s);  // fills d_opE
// y += the scalar moves
int lp_moves_f64(const LongPlan* L, const double* v, double* y, cudaStream_t s);
int lp_moves_f32(const LongPlan* L, const float* v, float* y, cudaStream_t s);
int lp_moves_bf16(const LongPlan* L, const __nv_bfloat16* v, float* y, cudaStream_t s);

}  // namespace dmrg2d
