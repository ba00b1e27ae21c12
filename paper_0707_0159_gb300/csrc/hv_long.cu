// Two-pass H·v on CUDA cores over a LongPlan, in FP64 (hv_long_kernel) and FP32
// (hv_long32_kernel); the scalar moves; the plan's work lists.
//
// What bounds FP64: its pipe (GB300: 2 DFMA per clock and SM, 1.25 TFLOP/s); a warp instruction
// costs the same with one active lane as with 32.  So lanes run along the long dimension of V_q
// (hundreds of indices, whole warps of it skipped at the end), and the short side, a
// quantum-number segment of any size, is held in registers with its exact extent: each warp owns
// up to 8 of the item's segment indices, and the loop body is instantiated for 1..8 of them.  K
// runs over each block's exact extent.  Nothing is padded but the last 64 long indices.
// Measured against one 64 x 64 piece per (row segment x column segment), whose padding was
// the time (3-leg Hubbard superblock of 25 sectors, 4-leg Heisenberg of 7; moves included):
//   Hubbard m = 256     FP64 115.6 -> 4.36 ms (1.02 TFLOP/s of 1.25), FP32 7.51 -> 0.52 ms
//   Heisenberg m = 256  FP64 7.85 -> 4.10 ms,                         FP32 0.55 -> 0.20 ms
//   Heisenberg m = 1024 FP64 275 -> 218 ms (1.23 TFLOP/s),            FP32 17.8 -> 7.0 ms
#include <algorithm>

#include "longplan.h"

namespace dmrg2d {

namespace {

constexpr int LT = 256;  // threads: 8 warps = row groups x groups of 64 long indices
constexpr int TN_MAX = 512;
constexpr int BK = 8;    // K per chunk

// row groups of an item: 8 indices per warp at most, the other warps along the long side
__host__ __device__ inline int row_groups(int cnt) {
  return cnt <= 8 ? 1 : cnt <= 16 ? 2 : cnt <= 32 ? 4 : 8;
}

struct alignas(16) Vec16 {
  double v[2];
};

// acc[a][b] += O[k][a] * V[k][c + 32 b] for the warp's RA indices
template <int RA, int OS, int VS>
__device__ __forceinline__ void mac_k(double (&acc)[8][2], const double* __restrict__ O,
                                      const double* __restrict__ V, int k) {
  constexpr int W = 2, NV = (RA + W - 1) / W;
  const double b0 = V[k * VS], b1 = V[k * VS + 32];
  Vec16 o[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) o[i] = *reinterpret_cast<const Vec16*>(O + k * OS + i * W);
#pragma unroll
  for (int a = 0; a < RA; ++a) {
    acc[a][0] += o[a / W].v[a % W] * b0;
    acc[a][1] += o[a / W].v[a % W] * b1;
  }
}
template <int RA, int OS, int VS>
__device__ __forceinline__ void mac(double (&acc)[8][2], const double* __restrict__ O,
                                    const double* __restrict__ V, int kk) {
  if (kk == BK) {
#pragma unroll
    for (int k = 0; k < BK; ++k) mac_k<RA, OS, VS>(acc, O, V, k);
  } else {
    for (int k = 0; k < kk; ++k) mac_k<RA, OS, VS>(acc, O, V, k);
  }
}

// One item with RG row groups (RG x 64 / CG long indices); Os, Vs: the CTA's tiles.
template <int PASS, int RG>
__device__ __forceinline__ void long_item(const double* __restrict__ v, double* __restrict__ y,
                                          const double* __restrict__ op, const LItem& it,
                                          const LSeg& sg, const LK* __restrict__ ks,
                                          double* __restrict__ Os, double* __restrict__ Vs) {
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

  double acc[8][2];
#pragma unroll
  for (int a = 0; a < 8; ++a) acc[a][0] = acc[a][1] = 0.0;

  // the next K chunk travels through registers while the current one is multiplied
  double rv[NV], ro[NO];
  const int okx = tid % BK, oi = tid / BK;             // operator element of this thread
  const int vx = PASS == 0 ? tid % TN : tid / BK;      // V element: long index, k
  const int vk = PASS == 0 ? tid / TN : tid % BK;
  auto fetch = [&](const LK& k, int k0) {
    const int kk = min(BK, k.kdim - k0);
    const double* po = op + k.op + (long long)(it.s0 + oi) * k.kdim + k0 + okx;
#pragma unroll
    for (int r = 0; r < NO; ++r, po += (long long)(LT / BK) * k.kdim)
      ro[r] = (oi + r * (LT / BK) < it.cnt && okx < kk) ? *po : 0.0;
    if (PASS == 0) {  // V(x, k): rows are contiguous
      constexpr int DX = TN > LT ? LT : 0, DK = TN > LT ? 0 : LT / TN;  // step of r
      const double* p = v + sg.base + it.x0 + vx + ld * (k.v_off + k0 + vk);
#pragma unroll
      for (int r = 0; r < NV; ++r) {
        const int x = vx + (DX ? (r & 1) * LT : 0), kx = vk + (DX ? r / 2 : r * DK);
        rv[r] = (x < nx && kx < kk) ? *p : 0.0;
        p += DX ? ((r & 1) ? ld - LT : LT) : ld * DK;
      }
    } else {  // V(k, x): the k of one column are contiguous
      const double* p = v + sg.base + k.v_off + k0 + vk + ld * (it.x0 + vx);
#pragma unroll
      for (int r = 0; r < NV; ++r, p += ld * (LT / BK))
        rv[r] = (vx + r * (LT / BK) < nx && vk < kk) ? *p : 0.0;
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
    const double* O = Os + rg * 8;
    const double* V = Vs + cg * 64 + lane;
    switch (mine) {  // uniform in the warp
      case 8: mac<8, OS, VS>(acc, O, V, kk); break;
      case 7: mac<7, OS, VS>(acc, O, V, kk); break;
      case 6: mac<6, OS, VS>(acc, O, V, kk); break;
      case 5: mac<5, OS, VS>(acc, O, V, kk); break;
      case 4: mac<4, OS, VS>(acc, O, V, kk); break;
      case 3: mac<3, OS, VS>(acc, O, V, kk); break;
      case 2: mac<2, OS, VS>(acc, O, V, kk); break;
      case 1: mac<1, OS, VS>(acc, O, V, kk); break;
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
      for (int j = sg.dim; j < sg.dim_pad; ++j) y[sg.base + sg.off + j + ld * gx] = 0.0;
  }
}

template <int PASS>
__global__ void __launch_bounds__(LT, 2)
hv_long_kernel(const double* __restrict__ v, double* __restrict__ y, const double* __restrict__ op,
               const LItem* __restrict__ items, const LSeg* __restrict__ segs,
               const LK* __restrict__ ks) {
  __shared__ __align__(16) double Os[BK * LP_ROWS];
  __shared__ __align__(16) double Vs[BK * (TN_MAX + 2)];
  const LItem it = items[blockIdx.x];
  const LSeg sg = segs[it.seg];
  switch (row_groups(it.cnt)) {
    case 1: long_item<PASS, 1>(v, y, op, it, sg, ks, Os, Vs); break;
    case 2: long_item<PASS, 2>(v, y, op, it, sg, ks, Os, Vs); break;
    case 4: long_item<PASS, 4>(v, y, op, it, sg, ks, Os, Vs); break;
    default: long_item<PASS, 8>(v, y, op, it, sg, ks, Os, Vs); break;
  }
}

// FP32: the same passes in tiles of SEG segment indices by 2048 / SEG * 4 long ones, 8 long x
// 4 segment outputs per thread, K chunks of 16 through registers.  Bound by the FP32 pipe
// (SEG = 64: six wavefronts of shared memory per 32 FFMA of a warp) and, with narrow segments
// (SEG = 16: nine), by shared memory.  Threads of one segment group fill whole or half warps,
// so groups beyond a segment's end cost nothing.  Against the FP64 kernel's shape run in FP32
// (16 outputs per thread in 8 x 2): Hubbard sectors m = 512 6.6 -> 2.0 ms, Heisenberg m = 1024
// 15.9 -> 7.0 ms (38 TFLOP/s); dense 3-leg Hubbard m = 128, against 64 x 64 pieces, 12.4 ->
// 5.8 ms (42 TFLOP/s).
template <int PASS, int SEG>
__device__ __forceinline__ void long_item32(const float* __restrict__ v, float* __restrict__ y,
                                            const float* __restrict__ op, const LItem& it,
                                            const LSeg& sg, const LK* __restrict__ ks,
                                            float* __restrict__ Os, float* __restrict__ Vs, bool vec) {
  constexpr int BK = 16, TL = 8192 / SEG, TX = TL / 8;  // long indices, threads along them
  constexpr int NV = BK * TL / LT, NO = BK * SEG / LT;
  constexpr int VS = TL + 4, OS = SEG + 4;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int nx = min(TL, sg.nlong - it.x0);
  const bool mine = 4 * ty < it.cnt && 4 * tx < nx;  // the second four long ones: + TL / 2
  const long long ld = sg.ld;
  float acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
  float rv[NV], ro[NO];
  const int kx = tid % BK, kr = tid / BK;
  auto fetch = [&](const LK& k, int k0) {
    const int kk = min(BK, k.kdim - k0);
    const float* po = op + k.op + (long long)(it.s0 + kr) * k.kdim + k0 + kx;
#pragma unroll
    for (int r = 0; r < NO; ++r, po += (long long)(LT / BK) * k.kdim)
      ro[r] = (kr + r * (LT / BK) < it.cnt && kx < kk) ? *po : 0.f;
    if (PASS == 0) {  // V(x, k): rows are contiguous
      if constexpr (TL >= LT) {
#pragma unroll
        for (int r = 0; r < NV; ++r) {
          const int x = tid + (r % (TL / LT)) * LT, q = r / (TL / LT);
          rv[r] = (x < nx && q < kk) ? v[sg.base + it.x0 + x + ld * (k.v_off + k0 + q)] : 0.f;
        }
      } else {
        const float* p = v + sg.base + it.x0 + tid % TL + ld * (k.v_off + k0 + tid / TL);
#pragma unroll
        for (int r = 0; r < NV; ++r, p += ld * (LT / TL))
          rv[r] = (tid % TL < nx && tid / TL + r * (LT / TL) < kk) ? *p : 0.f;
      }
    } else {  // V(k, x): the k of one column are contiguous
      const float* p = v + sg.base + k.v_off + k0 + kx + ld * (it.x0 + kr);
#pragma unroll
      for (int r = 0; r < NV; ++r, p += ld * (LT / BK))
        rv[r] = (kr + r * (LT / BK) < nx && kx < kk) ? *p : 0.f;
    }
  };
  auto put = [&]() {
#pragma unroll
    for (int r = 0; r < NO; ++r) Os[kx * OS + kr + r * (LT / BK)] = ro[r];
#pragma unroll
    for (int r = 0; r < NV; ++r) {
      if (PASS == 1)
        Vs[kx * VS + kr + r * (LT / BK)] = rv[r];
      else if constexpr (TL >= LT)
        Vs[(r / (TL / LT)) * VS + tid + (r % (TL / LT)) * LT] = rv[r];
      else
        Vs[(tid / TL + r * (LT / TL)) * VS + tid % TL] = rv[r];
    }
  };
  int e = sg.kb, k0 = 0;
  LK k = e < sg.ke ? ks[e] : LK{0, 0, 0};
  if (e < sg.ke) fetch(k, 0);
  while (e < sg.ke) {
    __syncthreads();
    put();
    __syncthreads();
    k0 += BK;
    if (k0 >= k.kdim) {
      k0 = 0;
      if (++e < sg.ke) k = ks[e];
    }
    if (e < sg.ke) fetch(k, k0);
    if (mine) {
#pragma unroll
      for (int q = 0; q < BK; ++q) {
        const float4 o = *(const float4*)(Os + q * OS + 4 * ty);
        const float4 a0 = *(const float4*)(Vs + q * VS + 4 * tx);
        const float4 a1 = *(const float4*)(Vs + q * VS + TL / 2 + 4 * tx);
        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(av[a], ov[b], acc[a][b]);
      }
    }
  }
  const int j0 = sg.off + it.s0 + 4 * ty, nj = min(4, it.cnt - 4 * ty);
  if (mine) {
    if (PASS == 0) {
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int x = 4 * tx + g * (TL / 2);
          float* Y = y + sg.base + it.x0 + x + ld * (j0 + b);
          if (b < nj && vec && x + 3 < nx) {
            *(float4*)Y = make_float4(acc[4 * g][b], acc[4 * g + 1][b], acc[4 * g + 2][b],
                                      acc[4 * g + 3][b]);
          } else if (b < nj) {
#pragma unroll
            for (int a = 0; a < 4; ++a)
              if (x + a < nx) Y[a] = acc[4 * g + a][b];
          }
        }
    } else {
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const int x = 4 * tx + (a / 4) * (TL / 2) + a % 4;
        if (x >= nx) continue;
        float* Y = y + sg.base + j0 + ld * (it.x0 + x);
        if (vec && nj == 4) {
          float4 o = *(const float4*)Y;
          o.x += acc[a][0];
          o.y += acc[a][1];
          o.z += acc[a][2];
          o.w += acc[a][3];
          *(float4*)Y = o;
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (b < nj) Y[b] += acc[a][b];
        }
      }
    }
  }
  if (PASS == 1 && it.s0 + it.cnt == sg.dim)  // the segment's padding rows
    for (int x = tid; x < nx; x += LT)
      for (int j = sg.dim; j < sg.dim_pad; ++j) y[sg.base + sg.off + j + ld * (it.x0 + x)] = 0.f;
}

// long indices of an FP32 item of cnt segment indices
int long_of32(int cnt) { return cnt <= 16 ? 512 : cnt <= 32 ? 256 : 128; }

template <int PASS>
__global__ void __launch_bounds__(LT, 2)
hv_long32_kernel(const float* __restrict__ v, float* __restrict__ y, const float* __restrict__ op,
                 const LItem* __restrict__ items, const LSeg* __restrict__ segs,
                 const LK* __restrict__ ks) {
  __shared__ __align__(16) float Os[16 * (LP_ROWS + 4)];
  __shared__ __align__(16) float Vs[16 * (512 + 4)];
  const LItem it = items[blockIdx.x];
  const LSeg sg = segs[it.seg];
  // 16-byte accesses to y: first element and leading dimension multiples of four
  const bool vec = ((((uintptr_t)y >> 2) | (uintptr_t)sg.base | (uintptr_t)sg.ld |
                     (uintptr_t)(PASS == 0 ? it.x0 : sg.off + it.s0)) & 3) == 0;
  if (it.cnt <= 16)
    long_item32<PASS, 16>(v, y, op, it, sg, ks, Os, Vs, vec);
  else if (it.cnt <= 32)
    long_item32<PASS, 32>(v, y, op, it, sg, ks, Os, Vs, vec);
  else
    long_item32<PASS, 64>(v, y, op, it, sg, ks, Os, Vs, vec);
}

// Four rows of a column, n of them inside the matrix (VEC: all four, aligned).
template <typename Tout, bool VEC, typename Tin>
__device__ __forceinline__ void load4(const Tin* p, int n, Tout (&o)[4]) {
  if constexpr (VEC && sizeof(Tin) == 8) {
    const double2 a = *(const double2*)p, b = *(const double2*)(p + 2);
    o[0] = (Tout)a.x, o[1] = (Tout)a.y, o[2] = (Tout)b.x, o[3] = (Tout)b.y;
  } else if constexpr (VEC && sizeof(Tin) == 4) {
    const float4 a = *(const float4*)p;
    o[0] = (Tout)a.x, o[1] = (Tout)a.y, o[2] = (Tout)a.z, o[3] = (Tout)a.w;
  } else if constexpr (VEC) {
    const uint2 u = *(const uint2*)p;
    o[0] = (Tout)__uint_as_float(u.x << 16), o[1] = (Tout)__uint_as_float(u.x & 0xffff0000u);
    o[2] = (Tout)__uint_as_float(u.y << 16), o[3] = (Tout)__uint_as_float(u.y & 0xffff0000u);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (sizeof(Tin) == 2)
        o[i] = i < n ? (Tout)__bfloat162float(p[i]) : Tout(0);
      else
        o[i] = i < n ? (Tout)p[i] : Tout(0);
    }
  }
}

// Y(block) += sum_moves c * V(source block).  Bound by memory in FP32 and BF16, in FP64 by the
// FP64 pipe (93 .. 95 % busy): a thread takes four rows of one column (sector segments start at
// multiples of 8 rows, so the fours of an aligned vector are aligned) and walks the block's moves with their addresses precomputed.  The
// earlier form (one row per thread of 256, eight columns, three dependent table reads per
// move) left most lanes of a small sector idle: on the 4-leg Heisenberg sectors of m = 1024
// the whole BF16 H·v went from 958 to 675 us, on the 3-leg Hubbard ones in TF32 from 5.92
// to 5.33 ms (there the tile configuration with separate moves became the faster one).
// The items run group by group (all blocks that exchange elements, a few MB): every source
// comes from L2 after its first use.  In the order of the vector each of the 3-4 sources of
// an element was a read from memory: 0.89 -> 0.69 ms on the 3-leg Hubbard sectors in TF32.
constexpr int MV_THREADS = 128, MV_ITEMS = 1024;  // threads; fours of rows per block
template <typename Tin, typename Tout, bool VEC>
__global__ void __launch_bounds__(MV_THREADS)
k_moves(const Tin* __restrict__ v, Tout* __restrict__ y, const MoveRec* __restrict__ recs,
        const MoveItem* __restrict__ items) {
  const MoveItem it = items[blockIdx.x];
  for (int t = threadIdx.x; t < it.nquad * it.ncol; t += MV_THREADS) {
    const int c = it.c_in + t / it.nquad, i = 4 * (t % it.nquad), n = it.dim - i;
    Tout acc[4], x[4];
    Tout* Y = y + it.dst + i + (long long)it.ld * c;
    load4<Tout, VEC>(Y, n, acc);
#pragma unroll 4
    for (int e = it.mb; e < it.me; ++e) {
      const MoveRec m = recs[e];
      load4<Tout, VEC>(v + m.src + i + (long long)m.ld * c, n, x);
      const Tout f = sizeof(Tout) == 8 ? (Tout)m.c64 : (Tout)m.c32;
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += f * x[q];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < n) Y[q] = acc[q];
  }
}

template <typename Tin, typename Tout>
int moves(const LongPlan* L, const Tin* v, Tout* y, cudaStream_t s) {
  const int nm = (int)L->mitems.size();
  if (!nm) return DMRG2D_OK;
  // vector loads where both vectors start on a 16-byte boundary
  if (L->quads && (((uintptr_t)v | (uintptr_t)y) & 15) == 0)
    k_moves<Tin, Tout, true><<<nm, MV_THREADS, 0, s>>>(v, y, L->d_mrec, L->d_mitems);
  else
    k_moves<Tin, Tout, false><<<nm, MV_THREADS, 0, s>>>(v, y, L->d_mrec, L->d_mitems);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

// Items of one pass: chunks of equal size (rounded to `round`), at most `cap` indices, by
// width(chunk) long indices; the most expensive first.
template <typename W>
std::vector<LItem> cut(const LongPlan* L, int ps, int cap, int round, W width) {
  std::vector<std::pair<double, LItem>> its;
  for (size_t i = 0; i < L->segs[ps].size(); ++i) {
    const LSeg& sg = L->segs[ps][i];
    double kt = 1.0;
    for (int e = sg.kb; e < sg.ke; ++e) kt += L->ks[ps][e].kdim;
    const int nch = (sg.dim + cap - 1) / cap;
    const int per = ((sg.dim + nch - 1) / nch + round - 1) / round * round;
    for (int s0 = 0; s0 < sg.dim; s0 += per) {
      const int cnt = std::min(per, sg.dim - s0), tn = width(cnt);
      for (int x = 0; x < sg.nlong; x += tn)
        its.push_back({kt * cnt * std::min(tn, sg.nlong - x), {(int)i, s0, cnt, x}});
    }
  }
  std::stable_sort(its.begin(), its.end(),
                   [](const auto& a, const auto& b) { return a.first > b.first; });
  std::vector<LItem> out;
  for (const auto& p : its) out.push_back(p.second);
  return out;
}

template <typename T>
int up(LongPlan* L, const std::vector<T>& h, T** d, int64_t* bytes, cudaStream_t s) {
  *d = nullptr;
  if (h.empty()) return DMRG2D_OK;
  const size_t nb = h.size() * sizeof(T);
  if (cudaMalloc((void**)d, nb) != cudaSuccess) {
    *d = nullptr;
    return set_error(DMRG2D_ENOMEM, "cudaMalloc(%zu) failed (H·v work list)", nb);
  }
  L->allocs.push_back(*d);
  *bytes += (int64_t)nb;
  D2_CUDA(cudaMemcpyAsync(*d, h.data(), nb, cudaMemcpyHostToDevice, s));
  return DMRG2D_OK;
}

}  // namespace

void lp_add_moves(LongPlan* L, int group, long long dst, int ld, int dim, int dim_pad, int ncols,
                  int mb, int me) {
  const int nquad = (dim_pad + 3) / 4, step = std::max(1, MV_ITEMS / nquad);
  for (int c = 0; c < ncols; c += step)
    L->mitems.push_back({dst, ld, dim, nquad, c, std::min(step, ncols - c), mb, me,
                         ((long long)group << 32) + c});
}

int lp_finalise(dmrg2d_ops* ops, LongPlan* L, cudaStream_t s) {
  if (cudaDeviceGetAttribute(&L->sms, cudaDevAttrMultiProcessorCount, ops->device) != cudaSuccess)
    L->sms = 1;
  for (int ps = 0; ps < 2; ++ps) {
    int e0 = 0;
    for (LSeg& sg : L->segs[ps]) {
      sg.e0 = e0;
      e0 += sg.dim;
      sg.ub = (int)L->units[ps].size();
      int64_t kt = 0;
      for (int e = sg.kb; e < sg.ke; ++e) {
        const LK& k = L->ks[ps][e];
        kt += k.kdim;
        for (int k0 = 0; k0 < k.kdim; k0 += 8)
          L->units[ps].push_back({k.op + k0, k.v_off + k0, k.kdim, std::min(8, k.kdim - k0)});
      }
      sg.ue = (int)L->units[ps].size();
      sg.head = 0;  // 64-bit sums of K products below 2^54 each
      while ((kt >> sg.head) > 256) ++sg.head;
    }
    L->items[ps] = cut(L, ps, LP_ROWS, 1, [](int cnt) { return 64 * (8 / row_groups(cnt)); });
    L->items32[ps] = cut(L, ps, LP_ROWS, 4, long_of32);
    // narrower items where 64 indices by 128 would leave SMs without one
    for (int cap = LP_ROWS; cap >= 16; cap /= 2) {
      L->fitems[ps] = cut(L, ps, cap, 8, [](int) { return FX_LONG; });
      if ((int)L->fitems[ps].size() >= L->sms) break;
    }
    int64_t* nb = &ops->device_bytes;
    D2_TRY(up(L, L->segs[ps], &L->d_segs[ps], nb, s));
    D2_TRY(up(L, L->ks[ps], &L->d_ks[ps], nb, s));
    D2_TRY(up(L, L->units[ps], &L->d_units[ps], nb, s));
    D2_TRY(up(L, L->items[ps], &L->d_items[ps], nb, s));
    D2_TRY(up(L, L->items32[ps], &L->d_items32[ps], nb, s));
    D2_TRY(up(L, L->fitems[ps], &L->d_fitems[ps], nb, s));
    D2_TRY(up(L, std::vector<int>((size_t)e0, 0), &L->d_opE[ps], nb, s));
  }
  std::stable_sort(L->mitems.begin(), L->mitems.end(),
                   [](const MoveItem& a, const MoveItem& b) { return a.group < b.group; });
  D2_TRY(up(L, L->mrec, &L->d_mrec, &ops->device_bytes, s));
  D2_TRY(up(L, L->mitems, &L->d_mitems, &ops->device_bytes, s));
  D2_TRY(up(L, std::vector<int>(1, 0), &L->err, &ops->device_bytes, s));
  fx_opE(L, s);
  D2_CUDA(cudaGetLastError());
  D2_CUDA(cudaStreamSynchronize(s));
  return DMRG2D_OK;
}

void lp_release(LongPlan* L) {
  if (!L) return;
  for (void* p : L->allocs) cudaFree(p);
  delete L;
}

int lp_read_error(const LongPlan* L, int* code) {
  *code = 0;
  if (!L || !L->err) return DMRG2D_OK;
  D2_CUDA(cudaMemcpy(code, L->err, sizeof(int), cudaMemcpyDeviceToHost));
  if (*code) D2_CUDA(cudaMemset(L->err, 0, sizeof(int)));
  return DMRG2D_OK;
}

int lp_launch_f64(const LongPlan* L, const double* v, double* y, cudaStream_t s) {
  const int n0 = (int)L->items[0].size(), n1 = (int)L->items[1].size();
  if (n0)
    hv_long_kernel<0><<<n0, LT, 0, s>>>(v, y, L->op64[0], L->d_items[0], L->d_segs[0],
                                        L->d_ks[0]);
  if (n1)
    hv_long_kernel<1><<<n1, LT, 0, s>>>(v, y, L->op64[1], L->d_items[1], L->d_segs[1],
                                        L->d_ks[1]);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}
int lp_launch_f32(const LongPlan* L, const float* v, float* y, cudaStream_t s) {
  const int n0 = (int)L->items32[0].size(), n1 = (int)L->items32[1].size();
  if (n0)
    hv_long32_kernel<0><<<n0, LT, 0, s>>>(v, y, L->op32[0], L->d_items32[0], L->d_segs[0],
                                          L->d_ks[0]);
  if (n1)
    hv_long32_kernel<1><<<n1, LT, 0, s>>>(v, y, L->op32[1], L->d_items32[1], L->d_segs[1],
                                          L->d_ks[1]);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}
int lp_moves_f64(const LongPlan* L, const double* v, double* y, cudaStream_t s) {
  return moves(L, v, y, s);
}
int lp_moves_f32(const LongPlan* L, const float* v, float* y, cudaStream_t s) {
  return moves(L, v, y, s);
}
int lp_moves_bf16(const LongPlan* L, const __nv_bfloat16* v, float* y, cudaStream_t s) {
  return moves(L, v, y, s);
}

}  // namespace dmrg2d
