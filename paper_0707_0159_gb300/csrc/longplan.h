// Work list of the CUDA-core two-pass H·v, shared by dense and sector-restricted
// superblocks.  Internal header.
//
// Each column-major matrix V_q (one for a dense superblock) is cut along one dimension
// only, the one the operator blocks act on:
//   pass 0 (V H_r^T): columns in segments; Y(:, c) = sum_e V(:, c_e) R_e^T over all rows;
//   pass 1 (H_l V):   rows in segments;    Y(r, :) += sum_e L_e V(r_e, :) over all columns.
// An item is up to LP_ROWS indices of one segment by a range of the long dimension.
#pragma once
#include <cstdint>
#include <vector>

#include "common.h"

namespace dmrg2d {

constexpr int LP_ROWS = 64;  // segment indices per item

struct LSeg {
  long long base;  // first element of V_q
  int ld, nlong;   // leading dimension; extent of the long dimension
  int off, dim, dim_pad;  // segment: offset, indices, indices with padding
  int kb, ke;      // operator blocks ks[kb..ke)
};
struct LK {
  long long op;    // element offset of the block (row-major dim x kdim)
  int v_off, kdim; // first index of the source segment in V_q; its extent
};
struct LItem {
  int seg, s0, cnt, x0;  // segment; its indices s0 .. s0 + cnt; first long index
};

struct LongPlan {
  std::vector<LSeg> segs[2];
  std::vector<LK> ks[2];
  std::vector<LItem> items[2];
  LSeg* d_segs[2] = {nullptr, nullptr};
  LK* d_ks[2] = {nullptr, nullptr};
  LItem* d_items[2] = {nullptr, nullptr};
};

// Cuts the segments into items (host only), the most expensive first.
void lp_items(LongPlan* L);
// y = V H_r^T + H_l V by the plan; the padding rows of row segments are written as zero.
// opL / opR: the blocks the plan's offsets refer to, in the storage type of v.
int lp_launch_f64(const LongPlan* L, const double* v, double* y, const double* opL,
                  const double* opR, cudaStream_t s);
int lp_launch_f32(const LongPlan* L, const float* v, float* y, const float* opL,
                  const float* opR, cudaStream_t s);

}  // namespace dmrg2d
