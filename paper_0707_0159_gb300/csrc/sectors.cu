// Sector-restricted superblock H·v: quantum-number blocks of uneven size as one grouped
// launch (the paper's blocks carry conserved quantum numbers, but it does not describe
// their use in H·v).
//
// Packed vector layout (also in include/dmrg2d.h): for every combined left label qL
// (block-1 label + column-2 label), in increasing lexicographic order, one column-major
// matrix V_qL:
//   rows    = for i2 = 0..d-1, the block-1 sector a with label qL - q(i2) (if present),
//             its states i1 in increasing order, each segment padded to a multiple of 8
//             rows (padding is zero on input and written as zero on output);
//   columns = for i3 = 0..d-1, the block-4 sector b with label Q - qL - q(i3) (if present),
//             its states i4 in increasing order;
//   ld      = padded row count; matrices are stored one after another.
// Within each V_qL the order is the paper's (i2 slow, i1 fast) x (i3 slow, i4 fast).
//
// H_l restricted to qL couples row segment (i2, a) to (i2', a') with a' fixed by charge
// conservation; the operator sub-block is the (a, a') part of the dense block
// HL[i2, i2'].  Same for H_r on column segments.  Scalar tile moves keep a and b and may
// change qL (H_c moves charge between the columns).
#include <algorithm>
#include <array>
#include <cmath>
#include <map>

#include "common.h"
#include "grouped.h"
#include "longplan.h"

namespace dmrg2d {

namespace {

using Lab = std::array<int, 2>;
Lab add(Lab a, Lab b) { return {a[0] + b[0], a[1] + b[1]}; }
Lab sub(Lab a, Lab b) { return {a[0] - b[0], a[1] - b[1]}; }

struct RowSegD {  // device row segment
  int q, off, dim, dim_pad, k1b, k1e;
};
struct ColSegD {
  int q, off, dim, k2b, k2e;
};
struct K1D {  // phase 1: A = L sub-block, B = rows of V_q
  long long a_off;  // compact FP64/FP32 offset of the sub-block (row-major dim(a) x kdim)
  int a_pool;       // first row of the sub-block in the tensor-core pool
  int b_row;        // first row of segment (i2', a') in V_q
  int kdim;
};
struct K2D {  // phase 2: A = columns of V_q, B = R sub-block
  long long b_off;  // compact offset (row-major dim(b) x kdim)
  int b_pool;
  int a_col;        // first column of segment (i3', b') in V_q
  int kdim;
};
struct MoveDst {
  int rs, cs, mb, me;
};
struct MoveSrc {
  int rs, cs;
  double c64;
  float c32;
};
struct SecState {
  int nQ = 0;
  std::vector<long long> qbase;
  std::vector<int> qld, qcols;
  std::vector<RowSegD> rseg;
  std::vector<ColSegD> cseg;
  std::vector<K1D> k1;
  std::vector<K2D> k2;
  std::vector<MoveDst> mdst;
  std::vector<MoveSrc> msrc;
  std::vector<int> rs_i2, rs_a, cs_i3, cs_b;  // host: segment identities
  std::vector<int> a_first, b_first;          // first state of each block sector
  // device copies
  double* d_L64 = nullptr;
  float* d_L32 = nullptr;
  double* d_R64 = nullptr;
  float* d_R32 = nullptr;
  // padding rows (zeroed in solver start vectors): (offset, count) pairs
  std::vector<long long> pad_off;
  std::vector<int> pad_cnt;
  long long* d_pad_off = nullptr;
  int* d_pad_cnt = nullptr;
  std::vector<void*> allocs;
  GroupPlan plan;  // tensor-core form of the same work (pools deduplicated up to sign)
  bool gp_ok = false;
};

// ---- kernels ------------------------------------------------------------------------------
__global__ void k_zero_pad(double* __restrict__ x, const long long* __restrict__ off,
                           const int* __restrict__ cnt, int n) {
  const int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= n) return;
  for (int i = 0; i < cnt[w]; ++i) x[off[w] + i] = 0.0;
}

template <typename T>
int up(SecState* S, const std::vector<T>& h, T** d, int64_t* bytes, cudaStream_t s) {
  *d = nullptr;
  if (h.empty()) return DMRG2D_OK;
  const size_t nb = h.size() * sizeof(T);
  if (cudaMalloc((void**)d, nb) != cudaSuccess) {
    *d = nullptr;
    return set_error(DMRG2D_ENOMEM, "cudaMalloc(%zu) failed (sectors)", nb);
  }
  S->allocs.push_back(*d);
  *bytes += (int64_t)nb;
  D2_CUDA(cudaMemcpyAsync(*d, h.data(), nb, cudaMemcpyHostToDevice, s));
  return DMRG2D_OK;
}

}  // namespace

// Grouped layout of a sector superblock: 128 x 256 pieces, longest first, with the scalar moves
// in the epilogue (TF32) or in their own kernel (BF16, whose epilogue converts every source:
// 4-leg Heisenberg, m = 1024, 1.49 against 0.63 ms; TF32 0.93 against 1.01 ms).
static int grouped_cfg(int precision) {
  return precision == DMRG2D_BF16 ? gp_num_configs() + 5 : 5;
}
// The configuration before any autotuning: the segment kernels where the grouped kernel's
// stages would read more than 2.5 times their bytes (its pieces pad narrow sectors on both
// sides) and the superblock is large enough for their two passes.  Grouped / segment bytes and
// times, TF32: 4-leg Heisenberg m = 384 2.1 / 0.72 GB, 0.167 / 0.146 ms; m = 512 2.6 / 1.3 GB,
// 0.204 / 0.223 ms; 2-leg m = 256 0.05 / 0.01 GB, 0.021 / 0.032 ms; 2-leg Hubbard m = 256 2.0 /
// 0.12 GB, 0.184 / 0.049 ms; 3-leg Hubbard m = 1024 6.0 / 3.2 ms.
static int default_cfg(const GroupPlan* g, int precision) {
  double grouped, segment;
  gp_stage_bytes(g, precision == DMRG2D_BF16 ? 64 : 32, &grouped, &segment);
  return segment < 0.4 * grouped && grouped > 3e8 ? 2 * gp_num_configs() : grouped_cfg(precision);
}

int sec_build(dmrg2d_ops* ops, const dmrg2d_block* L, const dmrg2d_block* R, const int32_t* target,
              const std::vector<double>& HL, const std::vector<double>& HR, cudaStream_t s) {
  const int d = ops->d, m1 = ops->m1, m4 = ops->m4;
  const int nq = ops->kind == DMRG2D_HEISENBERG ? 1 : 2;
  if (!L->qn || !R->qn)
    return set_error(DMRG2D_EINVAL, "sector-restricted build needs qn on both blocks");
  auto lab_of = [&](const int32_t* qn, int i) -> Lab {
    return {qn[i * nq], nq == 2 ? qn[i * nq + 1] : 0};
  };
  const Lab Q = {target[0], nq == 2 ? target[1] : 0};
  // ---- block sectors: maximal runs of equal labels ----
  auto runs = [&](const dmrg2d_block* B, std::vector<Lab>& lab, std::vector<int>& off,
                  std::vector<int>& dim, std::map<Lab, int>& idx, const char* name) -> int {
    for (int i = 0; i < B->m;) {
      const Lab l = lab_of(B->qn, i);
      int j = i + 1;
      while (j < B->m && lab_of(B->qn, j) == l) ++j;
      if (idx.count(l))
        return set_error(DMRG2D_EINVAL, "%s block: states with label (%d,%d) are not contiguous",
                         name, l[0], l[1]);
      idx[l] = (int)lab.size();
      lab.push_back(l);
      off.push_back(i);
      dim.push_back(j - i);
      i = j;
    }
    return DMRG2D_OK;
  };
  std::vector<Lab> lab1, lab4;
  std::vector<int> off1, dim1, off4, dim4;
  std::map<Lab, int> idx1, idx4;
  D2_TRY(runs(L, lab1, off1, dim1, idx1, "left"));
  D2_TRY(runs(R, lab4, off4, dim4, idx4, "right"));
  std::vector<Lab> qc(d);
  for (int i = 0; i < d; ++i) qc[i] = {ops->hqc[2 * i], nq == 2 ? ops->hqc[2 * i + 1] : 0};
  auto find = [](const std::map<Lab, int>& m, Lab l) {
    auto it = m.find(l);
    return it == m.end() ? -1 : it->second;
  };
  // ---- combined left labels with a non-empty right partner ----
  std::map<Lab, int> qset;
  for (int i2 = 0; i2 < d; ++i2)
    for (size_t a = 0; a < lab1.size(); ++a) {
      const Lab qL = add(lab1[a], qc[i2]);
      bool ok = false;
      for (int i3 = 0; i3 < d && !ok; ++i3) ok = find(idx4, sub(sub(Q, qL), qc[i3])) >= 0;
      if (ok) qset[qL] = 0;
    }
  if (qset.empty()) return set_error(DMRG2D_ESHAPE, "target sector is empty");
  SecState* S = new SecState();
  ops->sec = S;
  S->a_first = off1;
  S->b_first = off4;
  std::map<std::pair<int, int>, int> rs_of, cs_of;  // (i2,a) -> row seg, (i3,b) -> col seg
  long long base = 0;
  int qi = 0;
  for (auto& kv : qset) {
    kv.second = qi;
    const Lab qL = kv.first;
    int off = 0;
    for (int i2 = 0; i2 < d; ++i2) {
      const int a = find(idx1, sub(qL, qc[i2]));
      if (a < 0) continue;
      const int pad = (dim1[a] + 7) / 8 * 8;
      rs_of[{i2, a}] = (int)S->rseg.size();
      S->rseg.push_back({qi, off, dim1[a], pad, 0, 0});
      S->rs_i2.push_back(i2);
      S->rs_a.push_back(a);
      off += pad;
    }
    const int ld = off;
    int coff = 0;
    for (int i3 = 0; i3 < d; ++i3) {
      const int b = find(idx4, sub(sub(Q, qL), qc[i3]));
      if (b < 0) continue;
      cs_of[{i3, b}] = (int)S->cseg.size();
      S->cseg.push_back({qi, coff, dim4[b], 0, 0});
      S->cs_i3.push_back(i3);
      S->cs_b.push_back(b);
      coff += dim4[b];
    }
    S->qbase.push_back(base);
    S->qld.push_back(ld);
    S->qcols.push_back(coff);
    base += (long long)ld * coff;
    ++qi;
  }
  S->nQ = qi;
  ops->n_vec = base;
  // padding positions: every column of every padded row segment
  for (size_t r = 0; r < S->rseg.size(); ++r) {
    const RowSegD& rs = S->rseg[r];
    if (rs.dim_pad == rs.dim) continue;
    for (int c = 0; c < S->qcols[rs.q]; ++c) {
      S->pad_off.push_back(S->qbase[rs.q] + rs.off + rs.dim + (long long)S->qld[rs.q] * c);
      S->pad_cnt.push_back(rs.dim_pad - rs.dim);
    }
  }
  // ---- operator sub-blocks and K lists ----
  std::vector<double> Lc, Rc;  // compact row-major sub-blocks
  double flops = 0.0;
  int poolL = 0, poolR = 0;
  std::vector<int> qvalid_rows(S->nQ, 0);
  for (const RowSegD& rs : S->rseg) qvalid_rows[rs.q] += rs.dim;
  for (size_t r = 0; r < S->rseg.size(); ++r) {
    RowSegD& rs = S->rseg[r];
    const int i2 = S->rs_i2[r], a = S->rs_a[r];
    rs.k1b = (int)S->k1.size();
    for (int e = ops->hLptr[i2]; e < ops->hLptr[i2 + 1]; ++e) {
      const int i2p = ops->hLcol[e];
      const int ap = find(idx1, sub(add(lab1[a], qc[i2]), qc[i2p]));
      if (ap < 0) continue;
      auto it = rs_of.find({i2p, ap});
      if (it == rs_of.end()) continue;
      const double* blk = HL.data() + (size_t)e * m1 * m1;
      double mx = 0.0;
      for (int i = 0; i < dim1[a]; ++i)
        for (int k = 0; k < dim1[ap]; ++k)
          mx = std::max(mx, std::fabs(blk[(size_t)(off1[a] + i) * m1 + off1[ap] + k]));
      if (mx == 0.0) continue;  // structurally zero sub-block: no work
      {
        const auto pe = S->plan.poolL.add(blk + (size_t)off1[a] * m1 + off1[ap], dim1[a],
                                          dim1[ap], m1);
        S->plan.k1.push_back({pe.first, S->rseg[it->second].off, dim1[ap], pe.second});
      }
      K1D k;
      k.a_off = (long long)Lc.size();
      k.a_pool = poolL;
      k.b_row = S->rseg[it->second].off;
      k.kdim = dim1[ap];
      for (int i = 0; i < dim1[a]; ++i)
        for (int kk = 0; kk < dim1[ap]; ++kk)
          Lc.push_back(blk[(size_t)(off1[a] + i) * m1 + off1[ap] + kk]);
      poolL += dim1[a];
      S->k1.push_back(k);
      flops += 2.0 * dim1[a] * dim1[ap] * S->qcols[rs.q];
    }
    rs.k1e = (int)S->k1.size();
  }
  for (size_t c = 0; c < S->cseg.size(); ++c) {
    ColSegD& cs = S->cseg[c];
    const int i3 = S->cs_i3[c], b = S->cs_b[c];
    cs.k2b = (int)S->k2.size();
    for (int e = ops->hRptr[i3]; e < ops->hRptr[i3 + 1]; ++e) {
      const int i3p = ops->hRcol[e];
      const int bp = find(idx4, sub(add(lab4[b], qc[i3]), qc[i3p]));
      if (bp < 0) continue;
      auto it = cs_of.find({i3p, bp});
      if (it == cs_of.end()) continue;
      const double* blk = HR.data() + (size_t)e * m4 * m4;
      double mx = 0.0;
      for (int i = 0; i < dim4[b]; ++i)
        for (int k = 0; k < dim4[bp]; ++k)
          mx = std::max(mx, std::fabs(blk[(size_t)(off4[b] + i) * m4 + off4[bp] + k]));
      if (mx == 0.0) continue;
      {
        const auto pe = S->plan.poolR.add(blk + (size_t)off4[b] * m4 + off4[bp], dim4[b],
                                          dim4[bp], m4);
        S->plan.k2.push_back({S->cseg[it->second].off, pe.first, dim4[bp], pe.second});
      }
      K2D k;
      k.b_off = (long long)Rc.size();
      k.b_pool = poolR;
      k.a_col = S->cseg[it->second].off;
      k.kdim = dim4[bp];
      for (int i = 0; i < dim4[b]; ++i)
        for (int kk = 0; kk < dim4[bp]; ++kk)
          Rc.push_back(blk[(size_t)(off4[b] + i) * m4 + off4[bp] + kk]);
      poolR += dim4[b];
      S->k2.push_back(k);
      flops += 2.0 * dim4[b] * dim4[bp] * qvalid_rows[cs.q];
    }
    cs.k2e = (int)S->k2.size();
  }
  // ---- scalar moves per destination sub-block ----
  LongPlan* lp = new LongPlan();
  ops->lp = lp;
  for (size_t r = 0; r < S->rseg.size(); ++r)
    for (size_t c = 0; c < S->cseg.size(); ++c) {
      if (S->rseg[r].q != S->cseg[c].q) continue;
      const int i2 = S->rs_i2[r], a = S->rs_a[r], i3 = S->cs_i3[c], b = S->cs_b[c];
      const int t = i2 + d * i3;
      MoveDst md{(int)r, (int)c, (int)S->msrc.size(), 0};
      for (int e = ops->hCptr[t]; e < ops->hCptr[t + 1]; ++e) {
        const int src = ops->hCsrc[e];
        const int s2 = src % d, s3 = src / d;
        auto ir = rs_of.find({s2, a});
        auto ic = cs_of.find({s3, b});
        if (ir == rs_of.end() || ic == cs_of.end()) continue;
        if (S->rseg[ir->second].q != S->cseg[ic->second].q) continue;
        S->msrc.push_back({ir->second, ic->second, ops->hCval[e], (float)ops->hCval[e]});
        flops += 2.0 * dim1[a] * dim4[b];
      }
      md.me = (int)S->msrc.size();
      if (md.me == md.mb) continue;
      S->mdst.push_back(md);
      const RowSegD& rs = S->rseg[r];
      const ColSegD& cs = S->cseg[c];
      lp_add_moves(lp, a * (int)lab4.size() + b, S->qbase[rs.q] + rs.off + (long long)S->qld[rs.q] * cs.off, S->qld[rs.q],
                   rs.dim, rs.dim_pad, cs.dim, md.mb, md.me);
    }
  for (const MoveSrc& m : S->msrc) {
    const RowSegD& sr = S->rseg[m.rs];
    const ColSegD& sc = S->cseg[m.cs];
    lp->mrec.push_back({S->qbase[sr.q] + sr.off + (long long)S->qld[sr.q] * sc.off, S->qld[sr.q],
                        m.c32, m.c64});
  }
  // ---- two-pass plan over the same segments ----
  for (const ColSegD& c : S->cseg)
    lp->segs[0].push_back({S->qbase[c.q], S->qld[c.q], S->qld[c.q], c.off, c.dim, c.dim, c.k2b,
                           c.k2e, 0, 0, 0, 0});
  for (const K2D& k : S->k2) lp->ks[0].push_back({k.b_off, k.a_col, k.kdim});
  for (const RowSegD& r : S->rseg)
    lp->segs[1].push_back({S->qbase[r.q], S->qld[r.q], S->qcols[r.q], r.off, r.dim, r.dim_pad,
                           r.k1b, r.k1e, 0, 0, 0, 0});
  for (const K1D& k : S->k1) lp->ks[1].push_back({k.a_off, k.b_row, k.kdim});
  ops->flops = flops;
  // ---- upload ----
  std::vector<float> Lc32(Lc.begin(), Lc.end()), Rc32(Rc.begin(), Rc.end());
  int64_t* nb = &ops->device_bytes;
  int st = DMRG2D_OK;
#define SUP(h, dp) \
  if (st == DMRG2D_OK) st = up(S, h, &dp, nb, s)
  SUP(Lc, S->d_L64);
  SUP(Lc32, S->d_L32);
  SUP(Rc, S->d_R64);
  SUP(Rc32, S->d_R32);
  SUP(S->pad_off, S->d_pad_off);
  SUP(S->pad_cnt, S->d_pad_cnt);
#undef SUP
  if (st == DMRG2D_OK) {
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = set_error(DMRG2D_ECUDA, "sector upload: %s", cudaGetErrorString(e));
  }
  if (st == DMRG2D_OK) {
    lp->op64[0] = S->d_R64;
    lp->op64[1] = S->d_L64;
    lp->op32[0] = S->d_R32;
    lp->op32[1] = S->d_L32;
    st = lp_finalise(ops, lp, s);
  }
  // ---- grouped tensor-core plan over the same segments ----
  if (st == DMRG2D_OK) {
    GroupPlan& g = S->plan;
    g.nQ = S->nQ;
    g.qbase = S->qbase;
    g.qld = S->qld;
    g.qcols = S->qcols;
    for (const RowSegD& r : S->rseg) g.rows.push_back({r.q, r.off, r.dim, r.dim_pad, r.k1b, r.k1e});
    for (const ColSegD& c : S->cseg) g.cols.push_back({c.q, c.off, c.dim, c.k2b, c.k2e});
    for (const MoveDst& md : S->mdst) {  // the scalar moves run in the grouped epilogue
      g.mdst.push_back({md.rs, md.cs, (int)g.moves.size(), 0});
      for (int e = md.mb; e < md.me; ++e)
        g.moves.push_back({S->msrc[e].rs, S->msrc[e].cs, S->msrc[e].c32});
      g.mdst.back().me = (int)g.moves.size();
    }
    const int gs = gp_finalise(ops, &g, s);
    if (gs == DMRG2D_OK) {
      S->gp_ok = true;
      ops->tc_ok = 1;
      for (int p = 0; p < 4; ++p) ops->tc_cfg[p] = default_cfg(&g, p);
    } else if (gs == DMRG2D_EUNSUPPORTED) {
      clear_error();  // CUDA-core path only for this sector structure
    } else {
      st = gs;
    }
  }
  return st;
}

void sec_release(dmrg2d_ops* ops) {
  SecState* S = (SecState*)ops->sec;
  if (!S) return;
  gp_release(&S->plan);
  for (void* p : S->allocs) cudaFree(p);
  delete S;
  ops->sec = nullptr;
}

int sec_apply(const dmrg2d_ops* ops, const void* v, void* y, int precision, cudaStream_t s) {
  const SecState* S = (const SecState*)ops->sec;
  if (!S) return set_error(DMRG2D_EINVAL, "not a sector-restricted ops object");
  const LongPlan* lp = ops->lp;
  // tensor-core configuration; the segment kernels store Y in 16-byte pieces, so unless they
  // were asked for, a Y off that boundary takes the grouped kernel
  const int tp = precision == DMRG2D_TF32 ? DMRG2D_TF32 : DMRG2D_BF16;
  int cfg = ops->tc_cfg[tp];
  if (cfg == 2 * gp_num_configs() && !ops->tc_chosen[tp] && ((uintptr_t)y & 15) != 0)
    cfg = grouped_cfg(tp);
  // timed kernel: the block products here; the grouped tensor-core launch times itself
  const bool simt =
      precision == DMRG2D_FP64 || precision == DMRG2D_FP32 || precision == DMRG2D_FP64X;
  auto ev = simt ? prof_slot(ops) : std::pair<cudaEvent_t, cudaEvent_t>(nullptr, nullptr);
  if (ev.first) D2_CUDA(cudaEventRecord(ev.first, s));
  if (precision == DMRG2D_FP64 || precision == DMRG2D_FP64X) {
    // FP64X: the block products on split operands, the scalar moves in FP64
    if (precision == DMRG2D_FP64)
      D2_TRY(lp_launch_f64(lp, (const double*)v, (double*)y, s));
    else
      D2_TRY(fx_launch(lp, (const double*)v, (double*)y, s));
    if (ev.second) D2_CUDA(cudaEventRecord(ev.second, s));
    D2_TRY(lp_moves_f64(lp, (const double*)v, (double*)y, s));
  } else if (precision == DMRG2D_FP32) {
    D2_TRY(lp_launch_f32(lp, (const float*)v, (float*)y, s));
    if (ev.second) D2_CUDA(cudaEventRecord(ev.second, s));
    D2_TRY(lp_moves_f32(lp, (const float*)v, (float*)y, s));
  } else if (precision == DMRG2D_BF16X3 && S->gp_ok && cfg == 2 * gp_num_configs()) {
    // segment kernels: three products, then the moves on v_hi and v_lo
    const __nv_bfloat16* vhi = (const __nv_bfloat16*)v;
    const __nv_bfloat16* vlo = vhi + ops->n_vec;
    D2_TRY(gp_launch_seg(ops, &S->plan, vhi, (float*)y, DMRG2D_BF16, s, false, false));
    D2_TRY(gp_launch_seg(ops, &S->plan, vlo, (float*)y, DMRG2D_BF16, s, false, true));
    D2_TRY(gp_launch_seg(ops, &S->plan, vhi, (float*)y, DMRG2D_BF16, s, true, true));
    D2_TRY(lp_moves_bf16(lp, vhi, (float*)y, s));
    D2_TRY(lp_moves_bf16(lp, vlo, (float*)y, s));
  } else if ((precision == DMRG2D_TF32 || precision == DMRG2D_BF16) && S->gp_ok &&
             cfg == 2 * gp_num_configs()) {
    // segment kernels (M along the long dimension of each V_q), then the scalar moves
    D2_TRY(gp_launch_seg(ops, &S->plan, v, (float*)y, precision, s));
    if (precision == DMRG2D_BF16)
      D2_TRY(lp_moves_bf16(lp, (const __nv_bfloat16*)v, (float*)y, s));
    else
      D2_TRY(lp_moves_f32(lp, (const float*)v, (float*)y, s));
  } else if (precision == DMRG2D_BF16X3 && S->gp_ok) {
    // v = [v_hi | v_lo]: H_hi v_hi + H_hi v_lo + H_lo v_hi with the layout chosen for BF16,
    // the scalar moves applied to v_hi and v_lo (in the epilogues, or their own kernel)
    const int G = gp_num_configs();
    const bool fused = cfg < G;
    const __nv_bfloat16* vhi = (const __nv_bfloat16*)v;
    const __nv_bfloat16* vlo = vhi + ops->n_vec;
    D2_TRY(gp_launch(ops, &S->plan, vhi, (float*)y, DMRG2D_BF16, cfg % G, s, fused, false, false));
    D2_TRY(gp_launch(ops, &S->plan, vlo, (float*)y, DMRG2D_BF16, cfg % G, s, fused, false, true));
    D2_TRY(gp_launch(ops, &S->plan, vhi, (float*)y, DMRG2D_BF16, cfg % G, s, false, true, true));
    if (!fused) {
      D2_TRY(lp_moves_bf16(lp, vhi, (float*)y, s));
      D2_TRY(lp_moves_bf16(lp, vlo, (float*)y, s));
    }
  } else if ((precision == DMRG2D_TF32 || precision == DMRG2D_BF16) && S->gp_ok) {
    // tc_cfg < G: one launch, the grouped kernel's epilogue adds the scalar moves;
    // G <= tc_cfg < 2G: the moves run in their own kernel after it (G tile layouts)
    const int G = gp_num_configs();
    const bool fused = cfg < G;
    D2_TRY(gp_launch(ops, &S->plan, v, (float*)y, precision, cfg % G, s, fused));
    if (!fused) {
      if (precision == DMRG2D_BF16)
        D2_TRY(lp_moves_bf16(lp, (const __nv_bfloat16*)v, (float*)y, s));
      else
        D2_TRY(lp_moves_f32(lp, (const float*)v, (float*)y, s));
    }
  } else {
    return set_error(DMRG2D_EUNSUPPORTED,
                     "sector-restricted H·v: precision %d not available here", precision);
  }
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

int sec_dense_index(const dmrg2d_ops* ops, int64_t* out) {
  const SecState* S = (const SecState*)ops->sec;
  if (!S) return set_error(DMRG2D_EINVAL, "not a sector-restricted ops object");
  const int64_t m1 = ops->m1, d = ops->d, m4 = ops->m4;
  for (int64_t p = 0; p < ops->n_vec; ++p) out[p] = -1;
  for (size_t r = 0; r < S->rseg.size(); ++r)
    for (size_t c = 0; c < S->cseg.size(); ++c) {
      const RowSegD& rs = S->rseg[r];
      const ColSegD& cs = S->cseg[c];
      if (rs.q != cs.q) continue;
      const int64_t i2 = S->rs_i2[r], i3 = S->cs_i3[c];
      const int64_t a0 = S->a_first[S->rs_a[r]], b0 = S->b_first[S->cs_b[c]];
      for (int j = 0; j < cs.dim; ++j)
        for (int i = 0; i < rs.dim; ++i) {
          const int64_t pos = S->qbase[rs.q] + rs.off + i + (int64_t)S->qld[rs.q] * (cs.off + j);
          const int64_t i1 = a0 + i, i4 = b0 + j;
          out[pos] = i1 + m1 * i2 + m1 * d * i4 + m1 * d * m4 * i3;
        }
    }
  return DMRG2D_OK;
}

int sec_diag_tables(const dmrg2d_ops* ops, std::vector<long long>& qbase, std::vector<int>& qld,
                    std::vector<int>& qcols, std::vector<double>& rowD, std::vector<int>& rowI2,
                    std::vector<double>& colD, std::vector<int>& colI3) {
  const SecState* S = (const SecState*)ops->sec;
  if (!S) return set_error(DMRG2D_EINVAL, "not a sector-restricted ops object");
  const int m1 = ops->m1, m4 = ops->m4;
  qbase = S->qbase;
  qld = S->qld;
  qcols = S->qcols;
  for (int q = 0; q < S->nQ; ++q) {
    const size_t r0 = rowD.size();
    rowD.resize(r0 + S->qld[q], 0.0);
    rowI2.resize(r0 + S->qld[q], -1);  // padding rows stay -1
    for (size_t r = 0; r < S->rseg.size(); ++r) {
      const RowSegD& rs = S->rseg[r];
      if (rs.q != q) continue;
      const int i2 = S->rs_i2[r], a0 = S->a_first[S->rs_a[r]];
      for (int i = 0; i < rs.dim; ++i) {
        rowD[r0 + rs.off + i] = ops->hdL[(size_t)(a0 + i) + (size_t)m1 * i2];
        rowI2[r0 + rs.off + i] = i2;
      }
    }
    const size_t c0 = colD.size();
    colD.resize(c0 + S->qcols[q], 0.0);
    colI3.resize(c0 + S->qcols[q], 0);
    for (size_t c = 0; c < S->cseg.size(); ++c) {
      const ColSegD& cs = S->cseg[c];
      if (cs.q != q) continue;
      const int i3 = S->cs_i3[c], b0 = S->b_first[S->cs_b[c]];
      for (int j = 0; j < cs.dim; ++j) {
        colD[c0 + cs.off + j] = ops->hdR[(size_t)(b0 + j) + (size_t)m4 * i3];
        colI3[c0 + cs.off + j] = i3;
      }
    }
  }
  return DMRG2D_OK;
}

int sec_layout(const dmrg2d_ops* ops, std::vector<long long>& qbase, std::vector<int>& qld,
               std::vector<int>& qcols, std::vector<int64_t>& row_left,
               std::vector<int64_t>& col_right) {
  const SecState* S = (const SecState*)ops->sec;
  if (!S) return set_error(DMRG2D_EINVAL, "not a sector-restricted ops object");
  const int64_t m1 = ops->m1, m4 = ops->m4;
  qbase = S->qbase;
  qld = S->qld;
  qcols = S->qcols;
  row_left.clear();
  col_right.clear();
  for (int q = 0; q < S->nQ; ++q) {
    const size_t r0 = row_left.size(), c0 = col_right.size();
    row_left.resize(r0 + S->qld[q], -1);  // padding rows stay -1
    col_right.resize(c0 + S->qcols[q], -1);
    for (size_t r = 0; r < S->rseg.size(); ++r) {
      const RowSegD& rs = S->rseg[r];
      if (rs.q != q) continue;
      const int64_t a0 = S->a_first[S->rs_a[r]], i2 = S->rs_i2[r];
      for (int i = 0; i < rs.dim; ++i) row_left[r0 + rs.off + i] = a0 + i + m1 * i2;
    }
    for (size_t c = 0; c < S->cseg.size(); ++c) {
      const ColSegD& cs = S->cseg[c];
      if (cs.q != q) continue;
      const int64_t b0 = S->b_first[S->cs_b[c]], i3 = S->cs_i3[c];
      for (int j = 0; j < cs.dim; ++j) col_right[c0 + cs.off + j] = b0 + j + m4 * i3;
    }
  }
  return DMRG2D_OK;
}

int sec_read_error(const dmrg2d_ops* ops, int* code) {
  *code = 0;
  const SecState* S = (const SecState*)ops->sec;
  if (!S || !S->gp_ok) return DMRG2D_OK;
  return gp_read_error(&S->plan, code);
}

int sec_count(const dmrg2d_ops* ops) {
  const SecState* S = (const SecState*)ops->sec;
  return S ? S->nQ : 0;
}

int sec_zero_padding(const dmrg2d_ops* ops, double* x, cudaStream_t s) {
  const SecState* S = (const SecState*)ops->sec;
  if (!S || S->pad_off.empty()) return DMRG2D_OK;
  const int n = (int)S->pad_off.size();
  k_zero_pad<<<(n + 255) / 256, 256, 0, s>>>(x, S->d_pad_off, S->d_pad_cnt, n);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

}  // namespace dmrg2d
