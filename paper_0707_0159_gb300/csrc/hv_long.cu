// Two-pass H·v on CUDA cores (FP64 DFMA, FP32 FFMA) over a LongPlan.
//
// What bounds it: the FP64 pipe (GB300: 2 DFMA per clock and SM, 1.25 TFLOP/s) or the FP32
// pipe; a warp instruction costs the same with one active lane as with 32.  So lanes run
// along the long dimension of V_q (hundreds of indices, whole warps of it skipped at the
// end), and the short side, a quantum-number segment of any size, is held in registers with
// its exact extent: each warp owns up to 8 of the item's segment indices, and the loop body
// is instantiated for 1..8 of them.  K runs over each block's exact extent.  Nothing is
// padded but the last 64 long indices.
// Measured against one 64 x 64 piece per (row segment x column segment), whose padding was
// the time (3-leg Hubbard superblock of 25 sectors, 4-leg Heisenberg of 7; moves included):
//   Hubbard m = 256     FP64 115.6 -> 4.42 ms (1.01 TFLOP/s of 1.25), FP32 7.51 -> 0.98 ms
//   Heisenberg m = 256  FP64 7.85 -> 4.13 ms,                         FP32 0.55 -> 0.51 ms
//   Heisenberg m = 1024 FP64 275 -> 218 ms (1.23 TFLOP/s),            FP32 17.8 -> 15.9 ms
#include <algorithm>

#include "longplan.h"

namespace dmrg2d {

namespace {

constexpr int LT = 256;  // threads: 8 warps = row groups x groups of 64 long indices
constexpr int TN_MAX = 512;

// row groups of an item: 8 indices per warp at most, the other warps along the long side
__host__ __device__ inline int row_groups(int cnt) {
  return cnt <= 8 ? 1 : cnt <= 16 ? 2 : cnt <= 32 ? 4 : 8;
}

template <typename T>
struct alignas(16) Vec16 {
  T v[16 / sizeof(T)];
};

// acc[a][b] += O[k][a] * V[k][c + 32 b] for the warp's RA indices
template <typename T, int RA, int OS, int VS>
__device__ __forceinline__ void mac_k(T (&acc)[8][2], const T* __restrict__ O,
                                      const T* __restrict__ V, int k) {
  constexpr int W = 16 / sizeof(T), NV = (RA + W - 1) / W;
  const T b0 = V[k * VS], b1 = V[k * VS + 32];
  Vec16<T> o[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) o[i] = *reinterpret_cast<const Vec16<T>*>(O + k * OS + i * W);
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    acc[a][0] += o[a / W].v[a % W] * b0;
    acc[a][1] += o[a / W].v[a % W] * b1;
  }
}
template <typename T, int RA, int OS, int VS>
__device__ __forceinline__ void mac(T (&acc)[8][2], const T* __restrict__ O,
                                    const T* __restrict__ V, int kk) {
  constexpr int BK = 64 / sizeof(T);
  if (kk == BK) {
#pragma unroll
    for (int k = 0; k < BK; ++k) mac_k<T, RA, OS, VS>(acc, O, V, k);
  } else {
    for (int k = 0; k < kk; ++k) mac_k<T, RA, OS, VS>(acc, O, V, k);
  }
}

// One item with RG row groups (RG x 64 / CG long indices); Os, Vs: the CTA's tiles.
template <typename T, int PASS, int RG>
__device__ __forceinline__ void long_item(const T* __restrict__ v, T* __restrict__ y,
                                          const T* __restrict__ op, const LItem& it,
                                          const LSeg& sg, const LK* __restrict__ ks,
                                          T* __restrict__ Os, T* __restrict__ Vs) {
  constexpr int BK = 64 / sizeof(T);
  constexpr int CG = 8 / RG, TN = 64 * CG;
  constexpr int OS = LP_ROWS;            // operator tile: [k][8 slots per row group]
  constexpr int NV = BK * TN / LT;       // V elements per thread and chunk
  constexpr int NO = BK * 8 * RG / LT > 0 ? BK * 8 * RG / LT : 1;
  // V tile [k][long index]; a row stride of 2 modulo the banks keeps pass 1's transposing
  // stores (consecutive threads take consecutive k) off each other's banks
  constexpr int VS = TN + 2;
  const int ra = (it.cnt + RG - 1) / RG, inv = 65536 / ra + 1;  // i / ra for i < 64
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = warp / CG, cg = warp % CG;
  const int nx = min(TN, sg.nlong - it.x0);
  const int mine = cg * 64 < nx ? max(0, min(ra, it.cnt - rg * ra)) : 0;
  const long long ld = sg.ld;

  T acc[8][2];
#pragma unroll
  for (int a = 0; a < 8; ++a) acc[a][0] = acc[a][1] = T(0);

  // the next K chunk travels through registers while the current one is multiplied
  T rv[NV], ro[NO];
  const int okx = tid % BK, oi = tid / BK;             // operator element of this thread
  const int vx = PASS == 0 ? tid % TN : tid / BK;      // V element: long index, k
  const int vk = PASS == 0 ? tid / TN : tid % BK;
  auto fetch = [&](const LK& k, int k0) {
    const int kk = min(BK, k.kdim - k0);
    const T* po = op + k.op + (long long)(it.s0 + oi) * k.kdim + k0 + okx;
#pragma unroll
    for (int r = 0; r < NO; ++r, po += (long long)(LT / BK) * k.kdim)
      ro[r] = (oi + r * (LT / BK) < it.cnt && okx < kk) ? *po : T(0);
    if (PASS == 0) {  // V(x, k): rows are contiguous
      constexpr int DX = TN > LT ? LT : 0, DK = TN > LT ? 0 : LT / TN;  // step of r
      const T* p = v + sg.base + it.x0 + vx + ld * (k.v_off + k0 + vk);
#pragma unroll
      for (int r = 0; r < NV; ++r) {
        const int x = vx + (DX ? (r & 1) * LT : 0), kx = vk + (DX ? r / 2 : r * DK);
        rv[r] = (x < nx && kx < kk) ? *p : T(0);
        p += DX ? ((r & 1) ? ld - LT : LT) : ld * DK;
      }
    } else {  // V(k, x): the k of one column are contiguous
      const T* p = v + sg.base + k.v_off + k0 + vk + ld * (it.x0 + vx);
#pragma unroll
      for (int r = 0; r < NV; ++r, p += ld * (LT / BK))
        rv[r] = (vx + r * (LT / BK) < nx && vk < kk) ? *p : T(0);
    }
  };
  auto put = [&]() {
#pragma unroll
    for (int r = 0; r < NO; ++r) {
      const int i = oi + r * (LT / BK), g = (i * inv) >> 16;
      if (i < it.cnt) Os[okx * OS + g * 8 + i - g * ra] = ro[r];
    }
#pragma unroll
    for (int r = 0; r < NV; ++r) {
      if (PASS == 0) {
        const int x = vx + (TN > LT ? (r & 1) * LT : 0);
        const int kx = vk + (TN > LT ? r / 2 : r * (TN > LT ? 0 : LT / TN));
        Vs[kx * VS + x] = rv[r];
      } else {
        Vs[vk * VS + vx + r * (LT / BK)] = rv[r];
      }
    }
  };

  int e = sg.kb, k0 = 0;
  LK k = e < sg.ke ? ks[e] : LK{0, 0, 0};
  if (e < sg.ke) fetch(k, 0);
  while (e < sg.ke) {
    const int kk = min(BK, k.kdim - k0);
    __syncthreads();
    put();
    __syncthreads();
    k0 += BK;
    if (k0 >= k.kdim) {
      k0 = 0;
      if (++e < sg.ke) k = ks[e];
    }
    if (e < sg.ke) fetch(k, k0);
    const T* O = Os + rg * 8;
    const T* V = Vs + cg * 64 + lane;
    switch (mine) {  // uniform in the warp
      case 8: mac<T, 8, OS, VS>(acc, O, V, kk); break;
      case 7: mac<T, 7, OS, VS>(acc, O, V, kk); break;
      case 6: mac<T, 6, OS, VS>(acc, O, V, kk); break;
      case 5: mac<T, 5, OS, VS>(acc, O, V, kk); break;
      case 4: mac<T, 4, OS, VS>(acc, O, V, kk); break;
      case 3: mac<T, 3, OS, VS>(acc, O, V, kk); break;
      case 2: mac<T, 2, OS, VS>(acc, O, V, kk); break;
      case 1: mac<T, 1, OS, VS>(acc, O, V, kk); break;
      default: break;
    }
  }
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int x = cg * 64 + lane + 32 * b;
    if (x >= nx) continue;
    const long long gx = it.x0 + x;
    const int j0 = sg.off + it.s0 + rg * ra;
#pragma unroll
    for (int a = 0; a < 8; ++a)
      if (a < mine) {
        if (PASS == 0)
          y[sg.base + gx + ld * (j0 + a)] = acc[a][b];
        else
          y[sg.base + j0 + a + ld * gx] += acc[a][b];
      }
    // the segment's padding rows, by the first row group of its last item
    if (PASS == 1 && rg == 0 && it.s0 + it.cnt == sg.dim)
      for (int j = sg.dim; j < sg.dim_pad; ++j) y[sg.base + sg.off + j + ld * gx] = T(0);
  }
}

template <typename T, int PASS>
__global__ void __launch_bounds__(LT, 2)
hv_long_kernel(const T* __restrict__ v, T* __restrict__ y, const T* __restrict__ op,
               const LItem* __restrict__ items, const LSeg* __restrict__ segs,
               const LK* __restrict__ ks) {
  constexpr int BK = 64 / sizeof(T);
  __shared__ __align__(16) T Os[BK * LP_ROWS];
  __shared__ __align__(16) T Vs[BK * (TN_MAX + 2)];
  const LItem it = items[blockIdx.x];
  const LSeg sg = segs[it.seg];
  switch (row_groups(it.cnt)) {
    case 1: long_item<T, PASS, 1>(v, y, op, it, sg, ks, Os, Vs); break;
    case 2: long_item<T, PASS, 2>(v, y, op, it, sg, ks, Os, Vs); break;
    case 4: long_item<T, PASS, 4>(v, y, op, it, sg, ks, Os, Vs); break;
    default: long_item<T, PASS, 8>(v, y, op, it, sg, ks, Os, Vs); break;
  }
}

template <typename T>
int launch(const LongPlan* L, const T* v, T* y, const T* opL, const T* opR, cudaStream_t s) {
  const int n0 = (int)L->items[0].size(), n1 = (int)L->items[1].size();
  if (n0)
    hv_long_kernel<T, 0><<<n0, LT, 0, s>>>(v, y, opR, L->d_items[0], L->d_segs[0], L->d_ks[0]);
  if (n1)
    hv_long_kernel<T, 1><<<n1, LT, 0, s>>>(v, y, opL, L->d_items[1], L->d_segs[1], L->d_ks[1]);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

}  // namespace

void lp_items(LongPlan* L) {
  for (int ps = 0; ps < 2; ++ps) {
    std::vector<std::pair<double, LItem>> its;
    for (size_t i = 0; i < L->segs[ps].size(); ++i) {
      const LSeg& sg = L->segs[ps][i];
      double kt = 1.0;
      for (int e = sg.kb; e < sg.ke; ++e) kt += L->ks[ps][e].kdim;
      // chunks of equal size, at most LP_ROWS
      const int nch = (sg.dim + LP_ROWS - 1) / LP_ROWS;
      for (int c = 0; c < nch; ++c) {
        const int s0 = (int)((int64_t)sg.dim * c / nch), s1 = (int)((int64_t)sg.dim * (c + 1) / nch);
        const int tn = 64 * (8 / row_groups(s1 - s0));
        for (int x = 0; x < sg.nlong; x += tn)
          its.push_back({kt * (s1 - s0) * std::min(tn, sg.nlong - x), {(int)i, s0, s1 - s0, x}});
      }
    }
    std::stable_sort(its.begin(), its.end(),
                     [](const auto& a, const auto& b) { return a.first > b.first; });
    L->items[ps].clear();
    for (const auto& p : its) L->items[ps].push_back(p.second);
  }
}

int lp_launch_f64(const LongPlan* L, const double* v, double* y, const double* opL,
                  const double* opR, cudaStream_t s) {
  return launch<double>(L, v, y, opL, opR, s);
}
int lp_launch_f32(const LongPlan* L, const float* v, float* y, const float* opL,
                  const float* opR, cudaStream_t s) {
  return launch<float>(L, v, y, opL, opR, s);
}

}  // namespace dmrg2d
