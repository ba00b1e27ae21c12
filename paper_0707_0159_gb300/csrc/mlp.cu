// Learned preconditioner for the Davidson correction: a small MLP, trained and evaluated by
// the kernels in this file (FP32 on CUDA cores).
//
// The network g maps four features of one vector component to a factor that replaces
// the Jacobi factor 1/(theta - D_i):   t_i = (r_i / s_D) * g(x_i).
//   d_i  = (D_i - theta) / s_D,  s_D = RMS over the vector of (D - theta)
//   x0 = clamp(d_i, -8, 8)
//   x1 = clamp(1/d_i, -16, 16) / 16
//   x2 = clamp((mean of D over the component's sector - theta) / s_D, -8, 8)
//   x3 = log(number of components in the sector) / 16
// (Jacobi itself is g = -1/d.)  Architecture: 4 -> H (tanh) -> H (tanh) -> 1.
// Inference: g depends on i only through d_i and its sector, so each Davidson step
// evaluates the network exactly on a grid of G values of d per sector and interpolates
// linearly per component.  Training: weighted least squares on logged Davidson steps,
//   L = 1/(2B) sum_b (w_b g(x_b) - T_b)^2,  w_b = r_i/(s_D s_t),  T_b = alpha delta_i / s_t,
// delta = x_final - (x_k . x_final) x_k, alpha = (delta . t_J)/(delta . delta) (t_J the Jacobi
// correction), s_t = RMS(t_J): the network learns the direction of the ideal correction.
#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "common.h"

struct dmrg2d_mlp {
  int H = 0;
  int np = 0;
  float* p = nullptr;   // parameters: W1[H][4], b1[H], W2[H][H], b2[H], w3[H], b3
  float* g = nullptr;   // gradient
  float* m1 = nullptr;  // Adam moments
  float* m2 = nullptr;
  int step = 0;
  int bcap = 0;         // batch scratch capacity
  float *h1 = nullptr, *h2 = nullptr, *y = nullptr;
  float *dz2 = nullptr, *dz1 = nullptr;
  float* sums = nullptr;   // partial sums of the gradient (grow)
  double* part = nullptr;  // partial sums of the loss
};

namespace dmrg2d {

namespace {

constexpr int MF = 4;       // inputs
constexpr int GRID = 1024;  // table points per sector

inline int off_b1(int H) { return H * MF; }
inline int off_W2(int H) { return H * MF + H; }
inline int off_b2(int H) { return H * MF + H + H * H; }
inline int off_w3(int H) { return H * MF + H + H * H + H; }
inline int off_b3(int H) { return H * MF + H + H * H + 2 * H; }

// ---- matrix products ----------------------------------------------------------------------
// C[M x N] = A B on the FP32 pipes, 128 x 64 per CTA in K chunks of 16, 8 x 4 per thread; the
// next chunk travels through registers while the current one is multiplied.  Bound by the
// FP32 pipe: 12 wavefronts of shared memory against 32 FFMA per warp and K pair.  blockIdx.z
// cuts K into gridDim.z ranges (partial results C + z M N): the weight gradient's M x N is a
// few tiles for a K of thousands.
//   AK: A(i,k) = A[i lda + k], else A[k lda + i];  BK: B(k,j) = B[j ldb + k], else B[k ldb + j]
//   VEC: lda, ldb, K range and the pointers allow 16-byte loads
enum { EP_RAW, EP_TANH, EP_TANHGRAD };  // C = acc; tanh(acc + aux[j]); acc (1 - aux[i N + j]^2)
constexpr int GM = 128, GN = 64, GK = 16;

template <bool AK, bool BK, bool VEC, int EP>
__global__ void __launch_bounds__(256)
k_gemm(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
       float* __restrict__ C, int M, int N, int K, const float* __restrict__ aux) {
  __shared__ __align__(16) float As[GK][GM + 4];
  __shared__ __align__(16) float Bs[GK][GN + 4];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int i0 = blockIdx.y * GM, j0 = blockIdx.x * GN;
  const int per = ((K + (int)gridDim.z - 1) / (int)gridDim.z + GK - 1) / GK * GK;
  const int kb = blockIdx.z * per, ke = min(K, kb + per);
  float acc[8][4] = {};
  float4 ra[2], rb;
  // four consecutive elements along the contiguous index of an operand
  auto quad = [&](const float* P, int ld, int o, int no, int in, int ni) -> float4 {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (o < no && in < ni) {
      const float* p = P + (long long)o * ld + in;
      if (VEC && in + 3 < ni) {
        v = *(const float4*)p;
      } else {
        v.x = p[0];
        if (in + 1 < ni) v.y = p[1];
        if (in + 2 < ni) v.z = p[2];
        if (in + 3 < ni) v.w = p[3];
      }
    }
    return v;
  };
  auto fetch = [&](int k0) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int q = tid + 256 * r;
      ra[r] = AK ? quad(A, lda, i0 + q / 4, M, k0 + 4 * (q % 4), ke)
                 : quad(A, lda, k0 + q / 32, ke, i0 + 4 * (q % 32), M);
    }
    rb = BK ? quad(B, ldb, j0 + tid / 4, N, k0 + 4 * (tid % 4), ke)
            : quad(B, ldb, k0 + tid / 16, ke, j0 + 4 * (tid % 16), N);
  };
  auto put = [&]() {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int q = tid + 256 * r;
      if (AK) {
        As[4 * (q % 4)][q / 4] = ra[r].x;
        As[4 * (q % 4) + 1][q / 4] = ra[r].y;
        As[4 * (q % 4) + 2][q / 4] = ra[r].z;
        As[4 * (q % 4) + 3][q / 4] = ra[r].w;
      } else {
        *(float4*)&As[q / 32][4 * (q % 32)] = ra[r];
      }
    }
    if (BK) {
      Bs[4 * (tid % 4)][tid / 4] = rb.x;
      Bs[4 * (tid % 4) + 1][tid / 4] = rb.y;
      Bs[4 * (tid % 4) + 2][tid / 4] = rb.z;
      Bs[4 * (tid % 4) + 3][tid / 4] = rb.w;
    } else {
      *(float4*)&Bs[tid / 16][4 * (tid % 16)] = rb;
    }
  };
  if (kb < ke) fetch(kb);
  for (int k0 = kb; k0 < ke; k0 += GK) {
    __syncthreads();
    put();
    __syncthreads();
    if (k0 + GK < ke) fetch(k0 + GK);
#pragma unroll
    for (int k = 0; k < GK; ++k) {
      const float4 a0 = *(const float4*)&As[k][ty * 8], a1 = *(const float4*)&As[k][ty * 8 + 4];
      const float4 b = *(const float4*)&Bs[k][tx * 4];
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
    }
  }
  C += (long long)blockIdx.z * M * N;
#pragma unroll
  for (int u = 0; u < 8; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int i = i0 + ty * 8 + u, j = j0 + tx * 4 + v;
      if (i < M && j < N) {
        const long long e = (long long)i * N + j;
        float z = acc[u][v];
        if (EP == EP_TANH) z = tanhf(z + aux[j]);
        if (EP == EP_TANHGRAD) z *= 1.f - aux[e] * aux[e];
        C[e] = z;
      }
    }
}

template <bool AK, bool BK, int EP>
int gemm(const float* A, int lda, const float* B, int ldb, float* C, int M, int N, int K,
         const float* aux, int splits, cudaStream_t s) {
  const dim3 grid((N + GN - 1) / GN, (M + GM - 1) / GM, splits);
  const bool vec = lda % 4 == 0 && ldb % 4 == 0 && (((uintptr_t)A | (uintptr_t)B) & 15) == 0;
  if (vec)
    k_gemm<AK, BK, true, EP><<<grid, 256, 0, s>>>(A, lda, B, ldb, C, M, N, K, aux);
  else
    k_gemm<AK, BK, false, EP><<<grid, 256, 0, s>>>(A, lda, B, ldb, C, M, N, K, aux);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

// h1 = tanh(X W1^T + b1): four products per entry, bound by the store
__global__ void __launch_bounds__(256)
k_layer1(const float* __restrict__ X, const float* __restrict__ W1, const float* __restrict__ b1,
         float* __restrict__ h1, int B, int H) {
  const long long n = (long long)B * H;
  for (long long q = (long long)blockIdx.x * 256 + threadIdx.x; q < n;
       q += (long long)gridDim.x * 256) {
    const long long b = q / H;
    const int o = (int)(q - b * H);
    float z = b1[o];
#pragma unroll
    for (int f = 0; f < MF; ++f) z = fmaf(X[b * MF + f], W1[o * MF + f], z);
    h1[q] = tanhf(z);
  }
}

// y = h2 w3 + b3, one warp per row
__device__ __forceinline__ float row_output(const float* __restrict__ h, const float* __restrict__ w3,
                                            float b3, int H, int lane) {
  float z = 0.f;
  for (int o = lane; o < H; o += 32) z = fmaf(h[o], w3[o], z);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  return z + b3;
}
__global__ void __launch_bounds__(256)
k_output(const float* __restrict__ h2, const float* __restrict__ w3, const float* __restrict__ b3,
         float* __restrict__ y, int B, int H) {
  const int lane = threadIdx.x & 31;
  for (int b = blockIdx.x * 8 + (threadIdx.x >> 5); b < B; b += gridDim.x * 8) {
    const float z = row_output(h2 + (long long)b * H, w3, *b3, H, lane);
    if (lane == 0) y[b] = z;
  }
}

// One block of rows: y, dy = (w y - T) w / B, the block's sum of (w y - T)^2,
// dz2 = dy w3 (1 - h2^2), and the block's sums for the gradients of w3, b2 and b3
// (sums[blk][2 H + 1]).  The rows of h2 are read twice, the second time from cache.
constexpr int OUT_ROWS = 128;  // rows per block at most
__global__ void __launch_bounds__(256)
k_output_back(const float* __restrict__ h2, const float* __restrict__ w3,
              const float* __restrict__ b3, const float* __restrict__ w,
              const float* __restrict__ T, float* __restrict__ dz2, int B, int H, int rows,
              float* __restrict__ sums, double* __restrict__ part) {
  __shared__ float dy[OUT_ROWS];
  __shared__ double red[8], redy[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b0 = blockIdx.x * rows, nr = min(rows, B - b0);
  double s = 0.0, sy = 0.0;
  for (int r = warp; r < nr; r += 8) {
    const float y = row_output(h2 + (long long)(b0 + r) * H, w3, *b3, H, lane);
    const float e = w[b0 + r] * y - T[b0 + r], d = e * w[b0 + r] / (float)B;
    if (lane == 0) dy[r] = d;
    s += (double)e * e;
    sy += (double)d;
  }
  if (lane == 0) {
    red[warp] = s;
    redy[warp] = sy;
  }
  __syncthreads();
  float* out = sums + (long long)blockIdx.x * (2 * H + 1);
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) {
      s += red[k];
      sy += redy[k];
    }
    part[blockIdx.x] = s;
    out[2 * H] = (float)sy;
  }
  for (int o = threadIdx.x; o < H; o += 256) {
    const float wo = w3[o];
    const float* h = h2 + (long long)b0 * H + o;
    float* dz = dz2 + (long long)b0 * H + o;
    float g3 = 0.f, g2 = 0.f;
#pragma unroll 4
    for (int r = 0; r < nr; ++r) {
      const float hv = h[(long long)r * H], z = dy[r] * wo * (1.f - hv * hv);
      g3 = fmaf(dy[r], hv, g3);
      g2 += z;
      dz[(long long)r * H] = z;
    }
    out[o] = g2;
    out[H + o] = g3;
  }
}

// One block of rows and 256 columns: the sums for the gradients of W1 and b1
// (sums[blk][5 H]: W1 as [H][4], then b1)
__global__ void __launch_bounds__(256)
k_layer1_back(const float* __restrict__ dz1, const float* __restrict__ X, int B, int H, int rows,
              float* __restrict__ sums) {
  const int o = blockIdx.y * 256 + threadIdx.x;
  const int b0 = blockIdx.x * rows, nr = min(rows, B - b0);
  if (o >= H) return;
  float g[MF + 1] = {};
#pragma unroll 4
  for (int r = 0; r < nr; ++r) {
    const float z = dz1[(long long)(b0 + r) * H + o];
#pragma unroll
    for (int f = 0; f < MF; ++f) g[f] = fmaf(z, X[(long long)(b0 + r) * MF + f], g[f]);
    g[MF] += z;
  }
  float* out = sums + (long long)blockIdx.x * (MF + 1) * H;
#pragma unroll
  for (int f = 0; f < MF; ++f) out[o * MF + f] = g[f];
  out[MF * H + o] = g[MF];
}

// the gradient from its partial sums, in order: W1, b1 (n1 blocks), W2 (n2 ranges of K),
// b2, w3, b3 (n3 blocks)
__global__ void __launch_bounds__(256)
k_grad(const float* __restrict__ s1, int n1, const float* __restrict__ s2, int n2,
       const float* __restrict__ s3, int n3, int H, int np, float* __restrict__ g) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= np) return;
  const int e1 = (MF + 1) * H, e2 = e1 + H * H;
  const float* p;
  int n, stride;
  if (i < e1)
    p = s1 + i, n = n1, stride = e1;
  else if (i < e2)
    p = s2 + (i - e1), n = n2, stride = H * H;
  else
    p = s3 + (i - e2), n = n3, stride = 2 * H + 1;
  float a = 0.f, c = 0.f;  // two chains
  int k = 0;
#pragma unroll 4
  for (; k + 1 < n; k += 2) {
    a += p[(long long)k * stride];
    c += p[(long long)(k + 1) * stride];
  }
  if (k < n) a += p[(long long)k * stride];
  g[i] = a + c;
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, int n, float lr, float c1, float c2) {
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
    const float gi = g[i];
    m1[i] = 0.9f * m1[i] + 0.1f * gi;
    m2[i] = 0.999f * m2[i] + 0.001f * gi * gi;
    p[i] -= lr * (m1[i] / c1) / (sqrtf(m2[i] / c2) + 1e-8f);
  }
}

__device__ __forceinline__ void features(double Di, double theta, double sD, float x2, float x3,
                                         float* x) {
  const double d = (Di - theta) / sD;
  x[0] = (float)fmin(fmax(d, -8.0), 8.0);
  double inv = d != 0.0 ? 1.0 / d : 16.0;
  inv = fmin(fmax(inv, -16.0), 16.0);
  x[1] = (float)(inv / 16.0);
  x[2] = x2;
  x[3] = x3;
}

// grid inputs: for sector q, point k: d = dlo_q + k (dhi_q - dlo_q)/(G-1)
__global__ void k_grid_inputs(float* __restrict__ X, const double* __restrict__ qp, int nq,
                              double theta, double sD) {
  const int q = blockIdx.x;
  const double dlo = qp[4 * q], dhi = qp[4 * q + 1];
  const float x2 = (float)qp[4 * q + 2], x3 = (float)qp[4 * q + 3];
  for (int k = threadIdx.x; k < GRID; k += blockDim.x) {
    const double d = dlo + (dhi - dlo) * k / (GRID - 1);
    features(theta + d * sD, theta, sD, x2, x3, X + ((size_t)q * GRID + k) * MF);
  }
}

__device__ __forceinline__ int sector_of(const long long* __restrict__ qstart, int nq, long long i) {
  int lo = 0, hi = nq - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (qstart[mid] <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The Jacobi factor in units of s_D: t_i = r_i / (theta - D_i) = (r_i / s_D) j(d_i),
// j(d) = -1/d, clamped like the network's input |1/d| <= 16.
__device__ __forceinline__ double jacobi_factor(double d) {
  const double inv = d != 0.0 ? 1.0 / d : 16.0;
  return -fmin(fmax(inv, -16.0), 16.0);
}

// t_i = (r_i / s_D) j(d_i) (1 + y(d_i)), y interpolated from the sector's table
__global__ void k_apply_table(double* __restrict__ t, const double* __restrict__ r,
                              const double* __restrict__ D, const float* __restrict__ table,
                              const double* __restrict__ qp, const long long* __restrict__ qstart,
                              int nq, double theta, double sD, long long n) {
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n;
       i += (long long)gridDim.x * 256) {
    const int q = sector_of(qstart, nq, i);
    const double dlo = qp[4 * q], dhi = qp[4 * q + 1];
    const double d = (D[i] - theta) / sD;
    double u = dhi > dlo ? (d - dlo) / (dhi - dlo) * (GRID - 1) : 0.0;
    u = fmin(fmax(u, 0.0), (double)(GRID - 1));
    const int k = min((int)u, GRID - 2);
    const double f = u - k;
    const float* tq = table + (size_t)q * GRID;
    const double y = (1.0 - f) * tq[k] + f * tq[k + 1];
    t[i] = r[i] / sD * jacobi_factor(d) * (1.0 + y);
  }
}

// training samples: X (features), w = r/(s_D s_t), T = alpha delta / s_t at positions idx
__global__ void k_make_batch(const double* __restrict__ xk, const double* __restrict__ rk,
                             const double* __restrict__ xf, const double* __restrict__ D,
                             const long long* __restrict__ idx, int B, double theta, double sD,
                             double proj, double alpha, double st, const double* __restrict__ qp,
                             const long long* __restrict__ qstart, int nq, float* __restrict__ X,
                             float* __restrict__ w, float* __restrict__ T) {
  for (int b = blockIdx.x * 256 + threadIdx.x; b < B; b += gridDim.x * 256) {
    const long long i = idx[b];
    const int q = sector_of(qstart, nq, i);
    features(D[i], theta, sD, (float)qp[4 * q + 2], (float)qp[4 * q + 3], X + (size_t)b * MF);
    // the preconditioner is (r/s_D) j (1 + y): w y - T with w = (r/s_D) j / s_t and
    // T = (target - (r/s_D) j) / s_t fits the correction y to plain Jacobi
    const double wj = rk[i] / sD * jacobi_factor((D[i] - theta) / sD) / st;
    w[b] = (float)wj;
    T[b] = (float)(alpha * (xf[i] - proj * xk[i]) / st - wj);
  }
}

// per-range partial statistics of D: sum, sum of squares, min, max
__global__ void k_dstats(const double* __restrict__ D, long long n, double* __restrict__ out) {
  __shared__ double s1[256], s2[256], mn[256], mx[256];
  double a = 0, b = 0, lo = 1e300, hi = -1e300;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n;
       i += (long long)gridDim.x * 256) {
    const double v = D[i];
    a += v;
    b += v * v;
    lo = fmin(lo, v);
    hi = fmax(hi, v);
  }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  mn[threadIdx.x] = lo;
  mx[threadIdx.x] = hi;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      s1[threadIdx.x] += s1[threadIdx.x + o];
      s2[threadIdx.x] += s2[threadIdx.x + o];
      mn[threadIdx.x] = fmin(mn[threadIdx.x], mn[threadIdx.x + o]);
      mx[threadIdx.x] = fmax(mx[threadIdx.x], mx[threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[4 * blockIdx.x] = s1[0];
    out[4 * blockIdx.x + 1] = s2[0];
    out[4 * blockIdx.x + 2] = mn[0];
    out[4 * blockIdx.x + 3] = mx[0];
  }
}

// out = [x_k . x_f, delta . t_J, delta . delta, t_J . t_J], delta = x_f - (x_k . x_f) x_k,
// t_J = r / (theta - D): two passes with per-block partials summed on the host
__global__ void k_dot2(const double* __restrict__ a, const double* __restrict__ b, long long n,
                       double* __restrict__ part) {
  __shared__ double red[256];
  double s = 0.0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256)
    s += a[i] * b[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_delta3(const double* __restrict__ xk, const double* __restrict__ rk,
                         const double* __restrict__ xf, const double* __restrict__ D, double theta,
                         double proj, long long n, double* __restrict__ part) {
  __shared__ double r1[256], r2[256], r3[256];
  double a = 0, b = 0, c = 0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
    double den = theta - D[i];
    if (fabs(den) < 1e-8) den = den < 0 ? -1e-8 : 1e-8;
    const double tj = rk[i] / den;
    const double dl = xf[i] - proj * xk[i];
    a += dl * tj;
    b += dl * dl;
    c += tj * tj;
  }
  r1[threadIdx.x] = a;
  r2[threadIdx.x] = b;
  r3[threadIdx.x] = c;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      r1[threadIdx.x] += r1[threadIdx.x + o];
      r2[threadIdx.x] += r2[threadIdx.x + o];
      r3[threadIdx.x] += r3[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = r1[0];
    part[3 * blockIdx.x + 1] = r2[0];
    part[3 * blockIdx.x + 2] = r3[0];
  }
}

int vec_delta_stats(const double* xk, const double* rk, const double* xf, const double* D,
                    double theta, int64_t n, double* out, cudaStream_t s) {
  double* part = nullptr;
  if (cudaMalloc((void**)&part, 3 * 256 * 8) != cudaSuccess)
    return set_error(DMRG2D_ENOMEM, "delta stats");
  std::vector<double> hp(3 * 256, 0.0);
  k_dot2<<<256, 256, 0, s>>>(xk, xf, n, part);
  cudaMemcpyAsync(hp.data(), part, 256 * 8, cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  double proj = 0.0;
  for (int i = 0; i < 256; ++i) proj += hp[i];
  k_delta3<<<256, 256, 0, s>>>(xk, rk, xf, D, theta, proj, n, part);
  cudaMemcpyAsync(hp.data(), part, 3 * 256 * 8, cudaMemcpyDeviceToHost, s);
  const cudaError_t e = cudaStreamSynchronize(s);
  cudaFree(part);
  if (e != cudaSuccess) return set_error(DMRG2D_ECUDA, "delta stats: %s", cudaGetErrorString(e));
  out[0] = proj;
  out[1] = out[2] = out[3] = 0.0;
  for (int i = 0; i < 256; ++i) {
    out[1] += hp[3 * i];
    out[2] += hp[3 * i + 1];
    out[3] += hp[3 * i + 2];
  }
  return DMRG2D_OK;
}

// how a batch of B rows is cut: blocks of rows, ranges of K of the W2 gradient
struct Cut {
  int rows, blocks, splits;
};
Cut cut_batch(int B, int H) {
  constexpr int TARGET = 152;  // blocks: one per SM
  Cut c;
  c.rows = std::min(OUT_ROWS, std::max(16, (B + TARGET - 1) / TARGET));
  c.blocks = (B + c.rows - 1) / c.rows;
  const int tiles = ((H + GM - 1) / GM) * ((H + GN - 1) / GN);
  c.splits = std::max(1, std::min(2 * TARGET / tiles, (B + 8 * GK - 1) / (8 * GK)));
  return c;
}

int grow(dmrg2d_mlp* M, int B) {
  if (B <= M->bcap) return DMRG2D_OK;
  float** bufs[] = {&M->h1, &M->h2, &M->dz2, &M->dz1, &M->y, &M->sums};
  for (float** b : bufs) {
    if (*b) cudaFree(*b);
    *b = nullptr;
  }
  if (M->part) cudaFree(M->part);
  M->part = nullptr;
  M->bcap = 0;
  const int64_t H = M->H;
  // the largest cut of any batch up to B: 152 blocks or B / OUT_ROWS, 304 / tiles ranges
  const Cut c = cut_batch(B, M->H);
  const int64_t blocks = std::max(152, c.blocks);
  const size_t sizes[] = {(size_t)B * H, (size_t)B * H, (size_t)B * H, (size_t)B * H, (size_t)B,
                          (size_t)(blocks * ((MF + 1) * H + 2 * H + 1) + c.splits * H * H)};
  for (int i = 0; i < 6; ++i)
    if (cudaMalloc((void**)bufs[i], sizes[i] * 4) != cudaSuccess) {
      *bufs[i] = nullptr;
      return set_error(DMRG2D_ENOMEM, "MLP scratch");
    }
  if (cudaMalloc((void**)&M->part, blocks * 8) != cudaSuccess) {
    M->part = nullptr;
    return set_error(DMRG2D_ENOMEM, "MLP scratch");
  }
  M->bcap = B;
  return DMRG2D_OK;
}

// h1, h2 of the hidden layers
int hidden(dmrg2d_mlp* M, const float* X, int B, cudaStream_t s) {
  const int H = M->H;
  const float* p = M->p;
  const int g1 = (int)std::min<long long>(((long long)B * H + 255) / 256, 152 * 16);
  k_layer1<<<g1, 256, 0, s>>>(X, p, p + off_b1(H), M->h1, B, H);
  D2_CUDA(cudaGetLastError());
  return gemm<true, true, EP_TANH>(M->h1, H, p + off_W2(H), H, M->h2, B, H, H, p + off_b2(H), 1, s);
}

int forward(dmrg2d_mlp* M, const float* X, int B, cudaStream_t s) {
  const int H = M->H;
  const float* p = M->p;
  D2_TRY(hidden(M, X, B, s));
  k_output<<<std::min((B + 7) / 8, 152 * 8), 256, 0, s>>>(M->h2, p + off_w3(H), p + off_b3(H), M->y,
                                                         B, H);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

// Loss and gradient of L into M->g; loss (host) optional.  Every reduction over the batch is
// cut into blocks whose sums are added in order at the end: the weight gradient's 16 tiles
// with K = 8192 on one CTA each, and the biases' sums on one to four CTAs, were 4.7 of 4.9 ms
// (batch 8192, 256 hidden units; the call is now 0.18 ms, 19 TFLOP/s, and its gradient
// closer to FP64: 7.9e-8 against 1.3e-6).
int loss_and_gradient(dmrg2d_mlp* M, const float* X, const float* w, const float* T, int B,
                      float* loss, cudaStream_t s) {
  const int H = M->H;
  const float* p = M->p;
  const Cut c = cut_batch(B, H);
  float* s1 = M->sums;
  float* s3 = s1 + (int64_t)c.blocks * (MF + 1) * H;
  float* s2 = s3 + (int64_t)c.blocks * (2 * H + 1);
  D2_TRY(hidden(M, X, B, s));
  k_output_back<<<c.blocks, 256, 0, s>>>(M->h2, p + off_w3(H), p + off_b3(H), w, T, M->dz2, B, H,
                                         c.rows, s3, M->part);
  D2_CUDA(cudaGetLastError());
  D2_TRY((gemm<false, false, EP_RAW>(M->dz2, H, M->h1, H, s2, H, H, B, nullptr, c.splits, s)));
  // dz1 = (dz2 W2) (1 - h1^2)
  D2_TRY((gemm<true, false, EP_TANHGRAD>(M->dz2, H, p + off_W2(H), H, M->dz1, B, H, H, M->h1, 1, s)));
  k_layer1_back<<<dim3(c.blocks, (H + 255) / 256), 256, 0, s>>>(M->dz1, X, B, H, c.rows, s1);
  D2_CUDA(cudaGetLastError());
  k_grad<<<(M->np + 255) / 256, 256, 0, s>>>(s1, c.blocks, s2, c.splits, s3, c.blocks, H, M->np, M->g);
  D2_CUDA(cudaGetLastError());
  if (loss) {
    double hp[1024], tot = 0;  // no host allocation: batches of any size, 1024 sums at a time
    for (int b0 = 0; b0 < c.blocks; b0 += 1024) {
      const int nb = std::min(1024, c.blocks - b0);
      D2_CUDA(cudaMemcpyAsync(hp, M->part + b0, nb * sizeof(double), cudaMemcpyDeviceToHost, s));
      D2_CUDA(cudaStreamSynchronize(s));
      for (int i = 0; i < nb; ++i) tot += hp[i];
    }
    *loss = (float)(tot / (2.0 * B));
  }
  return DMRG2D_OK;
}

// contiguous vector ranges of the sectors (dense: one range)
void ranges(const dmrg2d_ops* ops, std::vector<long long>& start, std::vector<long long>& len) {
  if (ops->sec) {
    std::vector<long long> qb;
    std::vector<int> qld, qc;
    std::vector<double> rd, cd;
    std::vector<int> ri, ci;
    sec_diag_tables(ops, qb, qld, qc, rd, ri, cd, ci);
    for (size_t q = 0; q < qb.size(); ++q) {
      start.push_back(qb[q]);
      len.push_back((long long)qld[q] * qc[q]);
    }
  } else {
    start.push_back(0);
    len.push_back(ops->n_vec);
  }
}

}  // namespace

int mlp_precond_setup(const dmrg2d_mlp* M, const dmrg2d_ops* ops, const double* D, MlpPrecond* P,
                      cudaStream_t s) {
  (void)M;
  std::vector<long long> start, len;
  ranges(ops, start, len);
  P->nq = (int)start.size();
  P->mean.assign(P->nq, 0.0);
  P->dmin.assign(P->nq, 0.0);
  P->dmax.assign(P->nq, 0.0);
  P->count.assign(P->nq, 0.0);
  double* part = nullptr;
  if (cudaMalloc((void**)&part, 4 * 128 * sizeof(double)) != cudaSuccess)
    return set_error(DMRG2D_ENOMEM, "MLP setup");
  double s1 = 0, s2 = 0, n = 0;
  std::vector<double> hp(4 * 128);
  for (int q = 0; q < P->nq; ++q) {
    k_dstats<<<128, 256, 0, s>>>(D + start[q], len[q], part);
    cudaMemcpyAsync(hp.data(), part, hp.size() * 8, cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    double a = 0, b = 0, lo = 1e300, hi = -1e300;
    for (int k = 0; k < 128; ++k) {
      a += hp[4 * k];
      b += hp[4 * k + 1];
      lo = std::min(lo, hp[4 * k + 2]);
      hi = std::max(hi, hp[4 * k + 3]);
    }
    P->mean[q] = a / std::max<long long>(len[q], 1);
    P->dmin[q] = lo;
    P->dmax[q] = hi;
    P->count[q] = (double)len[q];
    s1 += a;
    s2 += b;
    n += (double)len[q];
  }
  cudaFree(part);
  P->meanD = s1 / n;
  P->meanD2 = s2 / n;
  std::vector<long long> qs(start);
  qs.push_back(ops->n_vec);
  auto al = [&](void** p, size_t b) -> int {
    if (cudaMalloc(p, b) != cudaSuccess) return set_error(DMRG2D_ENOMEM, "MLP setup");
    return DMRG2D_OK;
  };
  D2_TRY(al((void**)&P->qstart, qs.size() * 8));
  D2_CUDA(cudaMemcpyAsync(P->qstart, qs.data(), qs.size() * 8, cudaMemcpyHostToDevice, s));
  D2_TRY(al((void**)&P->qp, (size_t)P->nq * 4 * 8));
  D2_TRY(al((void**)&P->Xg, (size_t)P->nq * GRID * MF * 4));
  D2_TRY(al((void**)&P->table, (size_t)P->nq * GRID * 4));
  P->hqp.resize((size_t)P->nq * 4);
  D2_CUDA(cudaStreamSynchronize(s));
  return DMRG2D_OK;
}

static int precond_params(MlpPrecond* P, double theta, double* sD, cudaStream_t s) {
  const double var = P->meanD2 - 2.0 * theta * P->meanD + theta * theta;
  *sD = std::sqrt(std::max(var, 1e-300));
  for (int q = 0; q < P->nq; ++q) {
    P->hqp[4 * q] = (P->dmin[q] - theta) / *sD;
    P->hqp[4 * q + 1] = (P->dmax[q] - theta) / *sD;
    P->hqp[4 * q + 2] = std::min(std::max((P->mean[q] - theta) / *sD, -8.0), 8.0);
    P->hqp[4 * q + 3] = std::log(std::max(P->count[q], 1.0)) / 16.0;
  }
  D2_CUDA(cudaMemcpyAsync(P->qp, P->hqp.data(), P->hqp.size() * 8, cudaMemcpyHostToDevice, s));
  return DMRG2D_OK;
}

int mlp_precond_apply(const dmrg2d_mlp* Mc, MlpPrecond* P, const double* r, const double* D,
                      double theta, double* t, int64_t n, cudaStream_t s) {
  dmrg2d_mlp* M = const_cast<dmrg2d_mlp*>(Mc);
  double sD = 1.0;
  D2_TRY(precond_params(P, theta, &sD, s));
  k_grid_inputs<<<P->nq, 256, 0, s>>>(P->Xg, P->qp, P->nq, theta, sD);
  D2_CUDA(cudaGetLastError());
  D2_TRY(grow(M, P->nq * GRID));
  D2_TRY(forward(M, P->Xg, P->nq * GRID, s));
  D2_CUDA(cudaMemcpyAsync(P->table, M->y, (size_t)P->nq * GRID * 4, cudaMemcpyDeviceToDevice, s));
  const int grid = (int)std::min<long long>((n + 255) / 256, 4096);
  k_apply_table<<<grid, 256, 0, s>>>(t, r, D, P->table, P->qp, P->qstart, P->nq, theta, sD, n);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

void mlp_precond_release(MlpPrecond* P) {
  for (void* p : {(void*)P->qstart, (void*)P->qp, (void*)P->Xg, (void*)P->table})
    if (p) cudaFree(p);
  P->qstart = nullptr;
  P->qp = nullptr;
  P->Xg = nullptr;
  P->table = nullptr;
}

}  // namespace dmrg2d

using namespace dmrg2d;

extern "C" int dmrg2d_mlp_create(int hidden, uint64_t seed, dmrg2d_mlp** out) {
  if (!out || hidden < 1 || hidden > 4096) return set_error(DMRG2D_EINVAL, "mlp_create: bad argument");
  *out = nullptr;
  dmrg2d_mlp* M = new dmrg2d_mlp();
  M->H = hidden;
  M->np = off_b3(hidden) + 1;
  std::vector<float> h(M->np, 0.f);
  std::mt19937_64 rng(seed);
  std::normal_distribution<float> nd(0.f, 1.f);
  const int H = hidden;
  for (int i = 0; i < H * MF; ++i) h[i] = nd(rng) / std::sqrt((float)MF);
  for (int i = 0; i < H * H; ++i) h[off_W2(H) + i] = nd(rng) / std::sqrt((float)H);
  // output layer starts at zero: y = 0 is plain Jacobi (the factor is j(d) (1 + y))
  for (int i = 0; i < H; ++i) h[off_w3(H) + i] = 0.f;
  int st = DMRG2D_OK;
  for (float** b : {&M->p, &M->g, &M->m1, &M->m2})
    if (st == DMRG2D_OK && cudaMalloc((void**)b, (size_t)M->np * 4) != cudaSuccess)
      st = set_error(DMRG2D_ENOMEM, "mlp_create");
  if (st == DMRG2D_OK) {
    cudaMemcpy(M->p, h.data(), (size_t)M->np * 4, cudaMemcpyHostToDevice);
    cudaMemset(M->m1, 0, (size_t)M->np * 4);
    cudaMemset(M->m2, 0, (size_t)M->np * 4);
    if (cudaDeviceSynchronize() != cudaSuccess) st = set_error(DMRG2D_ECUDA, "mlp_create");
  }
  if (st != DMRG2D_OK) {
    dmrg2d_mlp_free(M);
    return st;
  }
  *out = M;
  return DMRG2D_OK;
}

extern "C" void dmrg2d_mlp_free(dmrg2d_mlp* M) {
  if (!M) return;
  for (void* p : {(void*)M->p, (void*)M->g, (void*)M->m1, (void*)M->m2, (void*)M->h1, (void*)M->h2,
                  (void*)M->y, (void*)M->dz2, (void*)M->dz1, (void*)M->sums, (void*)M->part})
    if (p) cudaFree(p);
  delete M;
}

extern "C" int dmrg2d_mlp_num_params(const dmrg2d_mlp* M) { return M ? M->np : 0; }

extern "C" int dmrg2d_mlp_get_params(const dmrg2d_mlp* M, float* host) {
  if (!M || !host) return set_error(DMRG2D_EINVAL, "NULL argument");
  D2_CUDA(cudaMemcpy(host, M->p, (size_t)M->np * 4, cudaMemcpyDeviceToHost));
  return DMRG2D_OK;
}

extern "C" int dmrg2d_mlp_set_params(dmrg2d_mlp* M, const float* host) {
  if (!M || !host) return set_error(DMRG2D_EINVAL, "NULL argument");
  D2_CUDA(cudaMemcpy(M->p, host, (size_t)M->np * 4, cudaMemcpyHostToDevice));
  M->step = 0;
  D2_CUDA(cudaMemset(M->m1, 0, (size_t)M->np * 4));
  D2_CUDA(cudaMemset(M->m2, 0, (size_t)M->np * 4));
  return DMRG2D_OK;
}

extern "C" int dmrg2d_mlp_forward(dmrg2d_mlp* M, const float* X, float* Y, int B, void* stream) {
  if (!M || !X || !Y || B < 1) return set_error(DMRG2D_EINVAL, "mlp_forward: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  D2_TRY(grow(M, B));
  D2_TRY(forward(M, X, B, s));
  D2_CUDA(cudaMemcpyAsync(Y, M->y, (size_t)B * 4, cudaMemcpyDeviceToDevice, s));
  return DMRG2D_OK;
}

extern "C" int dmrg2d_mlp_loss_grad(dmrg2d_mlp* M, const float* X, const float* w, const float* T,
                                    int B, float* grad, float* loss, void* stream) {
  if (!M || !X || !w || !T || B < 1) return set_error(DMRG2D_EINVAL, "mlp_loss_grad: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  D2_TRY(grow(M, B));
  D2_TRY(loss_and_gradient(M, X, w, T, B, loss, s));
  if (grad) D2_CUDA(cudaMemcpyAsync(grad, M->g, (size_t)M->np * 4, cudaMemcpyDeviceToDevice, s));
  return DMRG2D_OK;
}

extern "C" int dmrg2d_mlp_train_step(dmrg2d_mlp* M, const float* X, const float* w, const float* T,
                                     int B, float lr, float* loss, void* stream) {
  if (!M || !X || !w || !T || B < 1) return set_error(DMRG2D_EINVAL, "mlp_train_step: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  D2_TRY(grow(M, B));
  D2_TRY(loss_and_gradient(M, X, w, T, B, loss, s));
  ++M->step;
  const float c1 = 1.f - std::pow(0.9f, (float)M->step), c2 = 1.f - std::pow(0.999f, (float)M->step);
  k_adam<<<(M->np + 255) / 256, 256, 0, s>>>(M->p, M->g, M->m1, M->m2, M->np, lr, c1, c2);
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

extern "C" int dmrg2d_mlp_make_batch(const dmrg2d_ops* ops, const double* x_k, const double* r_k,
                                     double theta, const double* x_final, const double* D,
                                     const int64_t* idx, int B, float* X, float* w, float* T,
                                     void* stream) {
  if (!ops || !x_k || !r_k || !x_final || !D || !idx || !X || !w || !T || B < 1)
    return set_error(DMRG2D_EINVAL, "mlp_make_batch: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  MlpPrecond P;
  D2_TRY(mlp_precond_setup(nullptr, ops, D, &P, s));
  double sD = 1.0;
  int st = precond_params(&P, theta, &sD, s);
  // global scalars: proj = x_k . x_f ; delta = x_f - proj x_k ; t_J = r/(theta - D)
  double sc[4] = {0, 0, 0, 0};
  if (st == DMRG2D_OK) st = vec_delta_stats(x_k, r_k, x_final, D, theta, ops->n_vec, sc, s);
  const double proj = sc[0];
  const double alpha = sc[2] > 0 ? sc[1] / sc[2] : 0.0;          // (delta.tJ)/(delta.delta)
  const double stj = std::sqrt(std::max(sc[3] / (double)ops->n_vec, 1e-300));  // RMS(t_J)
  if (st == DMRG2D_OK) {
    k_make_batch<<<(B + 255) / 256, 256, 0, s>>>(x_k, r_k, x_final, D, (const long long*)idx, B,
                                                 theta, sD, proj, alpha, stj, P.qp, P.qstart, P.nq,
                                                 X, w, T);
    if (cudaGetLastError() != cudaSuccess) st = set_error(DMRG2D_ECUDA, "make_batch launch");
  }
  if (st == DMRG2D_OK && cudaStreamSynchronize(s) != cudaSuccess)
    st = set_error(DMRG2D_ECUDA, "make_batch");
  mlp_precond_release(&P);
  return st;
}
