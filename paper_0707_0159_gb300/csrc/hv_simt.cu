// Superblock H·v on CUDA cores (FP64 DFMA or FP32 FMA), and the apply_H entry point.
//
//     Y = H_l V + V H_r^T + sum_k A_k V B_k^T        (paper, text after Eq. (dec))
//
// Dense superblocks take pieces (this file) or the two-pass kernels (hv_long.cu: V H_r^T, then
// H_l V added, then the scalar moves added), by simt_choice.h.  In pieces, one CTA computes a
// BM x BN piece of one output tile (i2, i3) in three phases that share one register accumulator:
//   1. H_l V:    for every block (i2, i2') of H_l:  acc += HL[i2,i2'] * V_tile(i2', i3)
//   2. V H_r^T:  for every block (i3, i3') of H_r:  acc += V_tile(i2, i3') * HR[i3,i3']^T
//   3. scalar moves (H_c and off-diagonal column terms): acc += c * V_tile(i2', i3')
// and writes Y once.  V is column-major with leading dimension m1*d.
#include <algorithm>

#include "common.h"
#include "longplan.h"
#include "simt_choice.h"

namespace dmrg2d {

namespace {

struct SimtParams {
  int m1, m4, d;
  int64_t ld;
  const int* Lptr;
  const int* Lcol;
  const int* Rptr;
  const int* Rcol;
  const int* Cptr;
  const int* Csrc;
};

constexpr int BM = 64, BK = 16, TX = 16, TY = 16;  // 256 threads, 4x4 outputs each

// BMt x BNt piece per CTA (64 x 64: 4 x 4 outputs per thread; smaller pieces for small
// superblocks, whose 64 x 64 grid would leave most SMs idle at GB300's FP64 rate)
template <typename T, int BMt, int BNt>
__global__ void __launch_bounds__(TX * TY)
hv_simt_kernel(const T* __restrict__ v, T* __restrict__ y, const T* __restrict__ HL,
               const T* __restrict__ HR, const T* __restrict__ Cval, SimtParams p) {
  constexpr int RA = BMt / TX, RB = BNt / TY;  // outputs per thread along rows / columns
  constexpr int NT = TX * TY;
  __shared__ T As[BK][BMt];
  __shared__ T Bs[BK][BNt];
  const int nbm = (p.m1 + BMt - 1) / BMt;
  const int nbn = (p.m4 + BNt - 1) / BNt;
  const int bm = blockIdx.x % nbm, i2 = blockIdx.x / nbm;
  const int bn = blockIdx.y % nbn, i3 = blockIdx.y / nbn;
  const int i0 = bm * BMt, j0 = bn * BNt;
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int m1 = p.m1, m4 = p.m4;
  const int64_t ld = p.ld;

  T acc[RA][RB];
#pragma unroll
  for (int a = 0; a < RA; ++a)
#pragma unroll
    for (int b = 0; b < RB; ++b) acc[a][b] = T(0);

  auto mma_tile = [&]() {
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      T av[RA], bv[RB];
#pragma unroll
      for (int a = 0; a < RA; ++a) av[a] = As[k][tx + TX * a];
#pragma unroll
      for (int b = 0; b < RB; ++b) bv[b] = Bs[k][ty + TY * b];
#pragma unroll
      for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < RB; ++b) acc[a][b] += av[a] * bv[b];
    }
  };

  // ---- phase 1: H_l V ----
  for (int e = p.Lptr[i2]; e < p.Lptr[i2 + 1]; ++e) {
    const T* A = HL + (size_t)e * m1 * m1;                    // A[i][k] = A[i*m1 + k]
    const T* B = v + (int64_t)p.Lcol[e] * m1 + ld * ((int64_t)i3 * m4);  // B[k][j] = B[k + ld*j]
    for (int k0 = 0; k0 < m1; k0 += BK) {
      if constexpr (BMt == 64 && BNt == 64) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int k = tid % BK, i = tid / BK + 16 * r;
          const int gi = i0 + i, gk = k0 + k;
          As[k][i] = (gi < m1 && gk < m1) ? A[(size_t)gi * m1 + gk] : T(0);
          const int gj = j0 + i;  // the same (k, row) mapping for B's 64 columns
          Bs[k][i] = (gk < m1 && gj < m4) ? B[gk + ld * gj] : T(0);
        }
      } else {
        for (int idx = tid; idx < BK * BMt; idx += NT) {
          const int k = idx % BK, i = idx / BK;
          const int gi = i0 + i, gk = k0 + k;
          As[k][i] = (gi < m1 && gk < m1) ? A[(size_t)gi * m1 + gk] : T(0);
        }
        for (int idx = tid; idx < BK * BNt; idx += NT) {
          const int k = idx % BK, j = idx / BK;
          const int gj = j0 + j, gk = k0 + k;
          Bs[k][j] = (gk < m1 && gj < m4) ? B[gk + ld * gj] : T(0);
        }
      }
      __syncthreads();
      mma_tile();
      __syncthreads();
    }
  }
  // ---- phase 2: V H_r^T ----
  for (int e = p.Rptr[i3]; e < p.Rptr[i3 + 1]; ++e) {
    const T* A = v + (int64_t)i2 * m1 + ld * ((int64_t)p.Rcol[e] * m4);  // A[i][k] = A[i + ld*k]
    const T* B = HR + (size_t)e * m4 * m4;                    // B[k][j] = B[j*m4 + k]
    for (int k0 = 0; k0 < m4; k0 += BK) {
      if constexpr (BMt == 64 && BNt == 64) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int i = tid % BM, k = tid / BM + 4 * r;
          const int gi = i0 + i, gk = k0 + k;
          As[k][i] = (gi < m1 && gk < m4) ? A[gi + ld * gk] : T(0);
          const int kb = tid % BK, j = tid / BK + 16 * r;
          const int gj = j0 + j, gkb = k0 + kb;
          Bs[kb][j] = (gj < m4 && gkb < m4) ? B[(size_t)gj * m4 + gkb] : T(0);
        }
      } else {
        for (int idx = tid; idx < BK * BMt; idx += NT) {
          const int i = idx % BMt, k = idx / BMt;
          const int gi = i0 + i, gk = k0 + k;
          As[k][i] = (gi < m1 && gk < m4) ? A[gi + ld * gk] : T(0);
        }
        for (int idx = tid; idx < BK * BNt; idx += NT) {
          const int kb = idx % BK, j = idx / BK;
          const int gj = j0 + j, gkb = k0 + kb;
          Bs[kb][j] = (gj < m4 && gkb < m4) ? B[(size_t)gj * m4 + gkb] : T(0);
        }
      }
      __syncthreads();
      mma_tile();
      __syncthreads();
    }
  }
  // ---- phase 3: scalar tile moves, then the single store of Y ----
  const int t = i2 + p.d * i3;
  for (int e = p.Cptr[t]; e < p.Cptr[t + 1]; ++e) {
    const int src = p.Csrc[e];
    const int s2 = src % p.d, s3 = src / p.d;
    const T c = Cval[e];
    const T* S = v + (int64_t)s2 * m1 + ld * ((int64_t)s3 * m4);
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        const int gi = i0 + tx + TX * a, gj = j0 + ty + TY * b;
        if (gi < m1 && gj < m4) acc[a][b] += c * S[gi + ld * gj];
      }
  }
  T* Yt = y + (int64_t)i2 * m1 + ld * ((int64_t)i3 * m4);
#pragma unroll
  for (int a = 0; a < RA; ++a)
#pragma unroll
    for (int b = 0; b < RB; ++b) {
      const int gi = i0 + tx + TX * a, gj = j0 + ty + TY * b;
      if (gi < m1 && gj < m4) Yt[gi + ld * gj] = acc[a][b];
    }
}

// Small pieces (TS x TS, one output per thread) for superblocks whose larger pieces leave SMs
// idle.  The next K chunk of 16 travels through registers while the current one is
// multiplied; the three phases form one sequence of chunks.  Bound by the FP64 pipe once
// every SM has the same number of pieces: on the 2-leg m = 64 superblock (V 256 x 256) 16 x
// 16 pieces without the prefetch took 66 us (256 pieces on 152 SMs: two on most, one on some),
// 8 x 8 pieces (1024: 6.7 per SM, seven on the fullest) take 47 us; 41 us is the pipe's rate.
template <typename T, int TS>
__global__ void __launch_bounds__(TS * TS)
hv_simt_small_kernel(const T* __restrict__ v, T* __restrict__ y, const T* __restrict__ HL,
                     const T* __restrict__ HR, const T* __restrict__ Cval, SimtParams p) {
  constexpr int NT = TS * TS, R = BK * TS / NT;  // elements of each operand per thread
  __shared__ T As[BK][TS + 1];
  __shared__ T Bs[BK][TS + 1];
  const int m1 = p.m1, m4 = p.m4;
  const int nbm = (m1 + TS - 1) / TS, nbn = (m4 + TS - 1) / TS;
  const int i0 = (blockIdx.x % nbm) * TS, i2 = blockIdx.x / nbm;
  const int j0 = (blockIdx.y % nbn) * TS, i3 = blockIdx.y / nbn;
  const int64_t ld = p.ld;
  const int tid = threadIdx.x, tx = tid % TS, ty = tid / TS;
  const int kk = tid % BK, kr = tid / BK;  // K and row of k-contiguous operands
  const int nL = p.Lptr[i2 + 1] - p.Lptr[i2], nR = p.Rptr[i3 + 1] - p.Rptr[i3];
  T ra[R], rb[R];
  auto fetch = [&](int e, int k0) {  // chunk k0 of block e (H_l blocks first)
    if (e < nL) {
      const int g = p.Lptr[i2] + e;
      const T* A = HL + (size_t)g * m1 * m1;
      const T* B = v + (int64_t)p.Lcol[g] * m1 + ld * ((int64_t)i3 * m4);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int q = kr + r * (NT / BK);
        const bool in = k0 + kk < m1;
        ra[r] = in && i0 + q < m1 ? A[(size_t)(i0 + q) * m1 + k0 + kk] : T(0);
        rb[r] = in && j0 + q < m4 ? B[k0 + kk + ld * (j0 + q)] : T(0);
      }
    } else {
      const int g = p.Rptr[i3] + e - nL;
      const T* A = v + (int64_t)i2 * m1 + ld * ((int64_t)p.Rcol[g] * m4);
      const T* B = HR + (size_t)g * m4 * m4;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int k = ty + r * TS, q = kr + r * (NT / BK);
        ra[r] = k0 + k < m4 && i0 + tx < m1 ? A[i0 + tx + ld * (k0 + k)] : T(0);
        rb[r] = k0 + kk < m4 && j0 + q < m4 ? B[(size_t)(j0 + q) * m4 + k0 + kk] : T(0);
      }
    }
  };
  T acc = T(0);
  int e = 0, k0 = 0;
  if (nL + nR > 0) fetch(0, 0);
  while (e < nL + nR) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int q = kr + r * (NT / BK);
      if (e < nL)
        As[kk][q] = ra[r];
      else
        As[ty + r * TS][tx] = ra[r];
      Bs[kk][q] = rb[r];
    }
    __syncthreads();
    k0 += BK;
    if (k0 >= (e < nL ? m1 : m4)) {
      k0 = 0;
      ++e;
    }
    if (e < nL + nR) fetch(e, k0);
#pragma unroll
    for (int k = 0; k < BK; ++k) acc += As[k][tx] * Bs[k][ty];
  }
  const int gi = i0 + tx, gj = j0 + ty;
  if (gi >= m1 || gj >= m4) return;
  const int t = i2 + p.d * i3;
  for (int c = p.Cptr[t]; c < p.Cptr[t + 1]; ++c) {
    const int src = p.Csrc[c];
    acc += Cval[c] * v[(int64_t)(src % p.d) * m1 + gi + ld * ((int64_t)(src / p.d) * m4 + gj)];
  }
  y[(int64_t)i2 * m1 + gi + ld * ((int64_t)i3 * m4 + gj)] = acc;
}

template <typename T>
int launch(const dmrg2d_ops* ops, const T* v, T* y, const T* HL, const T* HR, const T* C,
           cudaStream_t s) {
  SimtParams p;
  p.m1 = ops->m1;
  p.m4 = ops->m4;
  p.d = ops->d;
  p.ld = ops->ld;
  p.Lptr = ops->dev.Lptr;
  p.Lcol = ops->dev.Lcol;
  p.Rptr = ops->dev.Rptr;
  p.Rcol = ops->dev.Rcol;
  p.Cptr = ops->dev.Cptr;
  p.Csrc = ops->dev.Csrc;
  const int sms = ops->lp->sms;
  const SimtChoice c =
      sizeof(T) == 8
          ? simt_choice_f64(ops->m1, ops->m4, ops->d, sms, (int64_t)ops->lp->items[0].size())
          : simt_choice_f32(ops->m1, ops->m4, ops->d, sms, (int64_t)ops->lp->items32[0].size());
  const int tb = c.piece;
  const int64_t gx = simt_pieces(ops->m1, ops->d, tb), gy = simt_pieces(ops->m4, ops->d, tb);
  if (!c.two_pass && !simt_grid_fits(ops->m1, ops->m4, ops->d, tb))
    return set_error(DMRG2D_EUNSUPPORTED, "SIMT grid %lld x %lld too large", (long long)gx,
                     (long long)gy);
  dim3 grid((unsigned)gx, (unsigned)gy);
  auto ev = prof_slot(ops);
  if (ev.first) D2_CUDA(cudaEventRecord(ev.first, s));
  if (c.two_pass) {
    if constexpr (sizeof(T) == 8) {
      D2_TRY(lp_launch_f64(ops->lp, v, y, s));
      if (ev.second) D2_CUDA(cudaEventRecord(ev.second, s));
      return lp_moves_f64(ops->lp, v, y, s);
    } else {
      D2_TRY(lp_launch_f32(ops->lp, v, y, s));
      if (ev.second) D2_CUDA(cudaEventRecord(ev.second, s));
      return lp_moves_f32(ops->lp, v, y, s);
    }
  }
  if (tb == 64)
    hv_simt_kernel<T, 64, 64><<<grid, TX * TY, 0, s>>>(v, y, HL, HR, C, p);
  else if (tb == 32)
    hv_simt_kernel<T, 32, 32><<<grid, TX * TY, 0, s>>>(v, y, HL, HR, C, p);
  else if (tb == 16)
    hv_simt_small_kernel<T, 16><<<grid, 256, 0, s>>>(v, y, HL, HR, C, p);
  else if constexpr (sizeof(T) == 8)  // FP64 only (simt_choice.h)
    hv_simt_small_kernel<T, 8><<<grid, 64, 0, s>>>(v, y, HL, HR, C, p);
  D2_CUDA(cudaGetLastError());
  if (ev.second) D2_CUDA(cudaEventRecord(ev.second, s));
  return DMRG2D_OK;
}

int launch_fx(const dmrg2d_ops* ops, const double* v, double* y, cudaStream_t s) {
  auto ev = prof_slot(ops);
  if (ev.first) D2_CUDA(cudaEventRecord(ev.first, s));
  D2_TRY(fx_launch(ops->lp, v, y, s));
  if (ev.second) D2_CUDA(cudaEventRecord(ev.second, s));
  return lp_moves_f64(ops->lp, v, y, s);
}

}  // namespace

int launch_hv_simt_ff64(const dmrg2d_ops* ops, const double* v, double* y, cudaStream_t s) {
  if (ops->sec) return sec_apply(ops, v, y, DMRG2D_FP64X, s);
  return launch_fx(ops, v, y, s);
}

int launch_hv_simt_f64(const dmrg2d_ops* ops, const double* v, double* y, cudaStream_t s) {
  if (ops->sec) return sec_apply(ops, v, y, DMRG2D_FP64, s);
  return launch<double>(ops, v, y, ops->dev.HL64, ops->dev.HR64, ops->dev.Cval64, s);
}

int launch_hv_simt_f32(const dmrg2d_ops* ops, const float* v, float* y, cudaStream_t s) {
  if (ops->sec) return sec_apply(ops, v, y, DMRG2D_FP32, s);
  return launch<float>(ops, v, y, ops->dev.HL32, ops->dev.HR32, ops->dev.Cval32, s);
}

}  // namespace dmrg2d

using namespace dmrg2d;

extern "C" int dmrg2d_apply_H(const dmrg2d_ops* ops, const void* v, void* y, int precision,
                              void* stream) {
  if (!ops || !v || !y) return set_error(DMRG2D_EINVAL, "NULL argument to apply_H");
  cudaStream_t s = (cudaStream_t)stream;
  switch (precision) {
    case DMRG2D_FP64:
      return launch_hv_simt_f64(ops, (const double*)v, (double*)y, s);
    case DMRG2D_FP32:
      return launch_hv_simt_f32(ops, (const float*)v, (float*)y, s);
    case DMRG2D_FP64X:
      return launch_hv_simt_ff64(ops, (const double*)v, (double*)y, s);
    case DMRG2D_TF32:
    case DMRG2D_BF16:
    case DMRG2D_BF16X3:
      if (!ops->tc_ok)
        return set_error(DMRG2D_EUNSUPPORTED, "tensor-core path does not support m1=%d m4=%d",
                         ops->m1, ops->m4);
      return launch_hv_tc(ops, v, (float*)y, precision, s);
    default:
      return set_error(DMRG2D_EINVAL, "unknown precision %d", precision);
  }
}
