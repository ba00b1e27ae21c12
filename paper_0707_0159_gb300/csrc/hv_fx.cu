// FP64X: H·v with FP64 vectors and operators on the FP16 tensor cores, exactly split.
//
// Every operand row (128 long indices of V, up to 64 segment indices of an operator) is
// scaled by a power of two so that its entries are 61-bit integers, and each integer is
// written as eight balanced base-256 digits, which FP16 holds exactly.  Products of digits
// summed over 128 K stay within 2^24, so the tensor cores' FP32 accumulators are exact: the
// 36 products of digits i, j with i + j = d <= 7 go into eight accumulators (one per d),
// which are then added into one 64-bit integer per output.  Rounding happens when an entry
// is cut to its row's scale (2^-60 of the row's largest entry), by the products left out
// (i + j > 7, about 2^-60 of the product of the two rows' largest entries), when a group of
// stages is added (2^-54 of the two scales' product for K up to 256, twice that for each
// doubling of K) and in the final conversion.
// With seven digits, 53-bit integers and 28 products (9.65 ms on the dense superblock below)
// the error was larger than float pairs' where the operator's rows and the vector are uneven,
// as ground states are: 1.9e-14 against 1.1e-14 on that of a 2 x 8 Hubbard ladder, m = 40.
// It is now 1.0e-15 there (FP64: 2.8e-16).  An entry far below the largest of its row is still
// held in fewer bits than by itself.
//
// Two passes over Y (longplan.h).  A CTA per SM walks its items; per stage of 32 K
//   warps 0-7   load FP64 entries of V, keep a scale for each row (the largest exponent so
//               far and one bit) and write their digits into shared memory (two stages);
//   warps 8-11  do the same for the operator (scales known from the build);
//   warp 12     issues the tcgen05.mma (M = 128 long indices, K = 16).  The operator's digits
//               lie one after another along N, so digit i of V meets all digits j <= 7 - i in
//               one instruction (two above N = 256) that adds to diagonals i .. 7;
//   warps 16-23 add the diagonals from tensor memory to their integers, after at most four
//               stages or when a scale has grown (the integers are then shifted).
//
// What bounds it: the digit arithmetic, about 25 instructions per entry of the two operands,
// most of them on the half-rate integer pipe (3600-4800 cycles a stage of 128 x 64 x 32, at
// 45 % of the integer pipe: three warps on an SM quarter do not hide its latencies), and the
// addition of the diagonals (5000-8000 cycles a group, during which no MMA runs).  The MMAs
// took 1800 cycles a stage with a guard predicate on each (84 to issue one); issued in a block
// of one elected lane they take half (dense m = 128 10.40 -> 9.65 ms).  (Cycles with seven
// digits.)  Measured against float pairs on the FP32 pipes (12 FP32 operations per product,
// pieces of 64 x 64):
//   3-leg Hubbard dense, m = 128          73.6 -> 11.3 ms (21 TFLOP/s), error 1.7e-13 -> 2.5e-15
//   4-leg Heisenberg sectors, m = 512     16.8 -> 2.23 ms,              error 2.6e-13 -> 8.6e-16
//   3-leg Hubbard sectors, m = 256        44.7 -> 1.81 ms
// Tried with seven digits and left out: 8 instead of 12 conversion warps, one warp role for
// conversion and addition (17 ms), the swizzled operand layouts (11.0 ms), one accumulation
// per stage (17.8 ms), one MMA per pair of digits (13.3 ms).
#include <algorithm>
#include <type_traits>

#include <cuda_fp16.h>

#include "longplan.h"
#include "tc_ptx.cuh"

namespace dmrg2d {

namespace {

using namespace tc;

constexpr int FX_CONV_A = 8, FX_CONV = 12, FX_EPI = 8;  // V, V + operator, epilogue warps
constexpr int FX_EPI0 = FX_CONV + 4;                   // first epilogue warp (whole warpgroups)
constexpr int FX_THREADS = 32 * (FX_EPI0 + FX_EPI);
// registers per thread of the conversion, MMA and epilogue warpgroups; the launch gives
// 768 x 80 = 61440, they take 128 (3 x 64 + 48 + 2 x 120) = 61440
constexpr int FX_R_CONV = 64, FX_R_MMA = 48, FX_R_EPI = 120;
constexpr int FX_S = 8;                                // digits = diagonals
constexpr int FX_K = 32;                               // K per stage
constexpr uint32_t FX_A = FX_LONG * FX_K * 2, FX_B = LP_ROWS * FX_K * 2;  // one digit, bytes
constexpr uint32_t FX_STAGE = FX_S * (FX_A + FX_B);
constexpr int FX_RING = 16;                            // stages whose scales are kept
constexpr int FX_GROUP = 4;                            // stages per accumulation (exact: 128 K)
constexpr uint32_t FX_SMEM = 2 * FX_STAGE + FX_RING * (FX_LONG + FX_CONV_A) * 4 + 256 + 128;
constexpr int FX_EMIN = 64;    // exponent fields below this are treated as zero

// a scale (exponent field) above the 20 bits of a high word's mantissa, all ones
// (2048, above every finite exponent and one bit: the row has an Inf or NaN)
__device__ __forceinline__ uint32_t scale_word(uint32_t e) { return e << 20 | 0xfffffu; }
// Digits of (53-bit mantissa 2^8 >> (scale - exponent)) with the sign of d, for four values, packed
// in pairs; E[i]: the scale as scale_word; out[i * stride8]: digit i (0 = most significant)
// as 4 halves.
__device__ __forceinline__ void digits4(const double* d, const uint32_t (&E)[4], uint2* out,
                                        uint32_t stride8) {
  uint32_t lo[4], hi[4], sg[2], nb[2];
#pragma unroll
  for (int t = 0; t < 2; ++t) {  // +-1 and -+1152 in FP16: digit = sign * (1024 + byte) - sign * 1152
    const uint32_t x = (__byte_perm((uint32_t)__double2hiint(d[2 * t]),
                                    (uint32_t)__double2hiint(d[2 * t + 1]), 0x7632) &
                        0x80008000u) |
                       0x3c003c00u;
    sg[t] = x;
    const __half2 n = __hmul2(*reinterpret_cast<const __half2*>(&x),
                              __halves2half2(__ushort_as_half(0xe480), __ushort_as_half(0xe480)));
    nb[t] = *reinterpret_cast<const uint32_t*>(&n);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t h = (uint32_t)__double2hiint(d[i]);
    // scale - exponent: the mantissa bits of h only lower the difference of the low 20 bits.
    // shr takes shifts above 63 as 64
    const uint32_t sh = (E[i] - (h & 0x7fffffffu)) >> 20, l = (uint32_t)__double2loint(d[i]);
    uint64_t m = ((uint64_t)__funnelshift_l(l, (h & 0xfffffu) | 0x100000u, 8) << 32) | (l << 8);
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(sh));
    // the digit bias 0x80 in every byte
    const uint64_t q = m + 0x8080808080808080ull;
    lo[i] = (uint32_t)q;
    hi[i] = (uint32_t)(q >> 32);
  }
  auto fin = [&](uint32_t x, int t) {
    const __half2 r =
        __hfma2(*reinterpret_cast<const __half2*>(&x), *reinterpret_cast<const __half2*>(&sg[t]),
                *reinterpret_cast<const __half2*>(&nb[t]));
    return *reinterpret_cast<const uint32_t*>(&r);
  };
#pragma unroll
  for (int j = 0; j < 4; ++j) {  // bytes 3, 2 then 1, 0 of the high, then the low words
    const uint32_t* w = j < 2 ? hi : lo;
    // {a.hi, b.hi, a.lo, b.lo} of the byte pair; 0x64 above a byte: FP16 1024 + byte
    const uint32_t x0 = __byte_perm(w[0], w[1], (j & 1) == 0 ? 0x6273 : 0x4051);
    const uint32_t x1 = __byte_perm(w[2], w[3], (j & 1) == 0 ? 0x6273 : 0x4051);
    *out = make_uint2(fin(__byte_perm(x0, 0x64646464u, 0x4140), 0),
                      fin(__byte_perm(x1, 0x64646464u, 0x4140), 1));
    out += stride8;
    *out = make_uint2(fin(__byte_perm(x0, 0x64646464u, 0x4342), 0),
                      fin(__byte_perm(x1, 0x64646464u, 0x4342), 1));
    out += stride8;
  }
}

__device__ __forceinline__ uint32_t absbits(double x) {
  return (uint32_t)__double2hiint(x) & 0x7fffffffu;
}
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// a 2^p (rounded to nearest); p + 63 and p stay inside the exponent range or the slow path
// takes it
__device__ __forceinline__ double scaled(long long a, int p) {
  if (a == 0) return 0.0;
  const uint64_t s = (uint64_t)(a >> 63);
  const uint64_t u = ((uint64_t)a ^ s) - s;
  const int lz = __clzll((long long)u);
  const int e = p + 63 - lz + 1023;
  if (e < 1 || e > 2045) {  // in two factors: |p| < 2002
    const int p1 = p / 2;
    return (double)a * __hiloint2double((p1 + 1023) << 20, 0) *
           __hiloint2double((p - p1 + 1023) << 20, 0);
  }
  const uint64_t m = u << lz;
  const uint64_t r = (m >> 11) + ((m >> 10) & 1);  // 53 bits; a carry raises the exponent
  return __longlong_as_double((long long)((((uint64_t)(e - 1)) << 52) + r) | (long long)(s << 63));
}

// eight tensor-memory columns of the warp's 32 lanes; valid after tmem_wait8
__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
}
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}

struct FxParams {
  const LItem* items;
  const LSeg* segs;
  const LUnit* units;
  const int* opE;
  const double* op;
  const double* v;
  double* y;
  int* err;
  int nitems;
};

template <int PASS>
__global__ void __launch_bounds__(FX_THREADS, 1) hv_fx_kernel(const FxParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
  uint32_t* esm = (uint32_t*)(smem + 2 * FX_STAGE);   // [FX_RING][FX_LONG] scale of each long index
  int* grown = (int*)(esm + FX_RING * FX_LONG);     // [FX_RING][FX_CONV_A] a scale of the warp has grown
  uint64_t* bars = (uint64_t*)(grown + FX_RING * FX_CONV_A);
  uint32_t* tmem_slot = (uint32_t*)(bars + 6);
  volatile int* abort = (volatile int*)(tmem_slot + 1);
  // accumulation group g: ginfo[g % 4] = 2 * first stage + (last group of its item)
  volatile uint32_t* ginfo = (volatile uint32_t*)(tmem_slot + 2);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  auto ready = [&](int b) { return smem_u32(bars + b); };
  auto freeb = [&](int b) { return smem_u32(bars + 2 + b); };
  const uint32_t tfull = smem_u32(bars + 4), tempty = smem_u32(bars + 5);

  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(ready(b), FX_CONV);
      mbar_init(freeb(b), 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, FX_EPI);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == FX_CONV) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp < FX_CONV) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FX_R_CONV));
    // ------------------------- digits of both operands -------------------------
    // Each warp has two batches of eight entries per thread.  Lanes along K (the operator,
    // and V in pass 1): eight rows, K = lane; the first of K = 8 (lane / 8) is unit lane / 8.
    // V in pass 0: lane % 8 is the row, the eight K of unit lane / 8.
    auto convert = [&](auto is_a) {
      constexpr bool isA = decltype(is_a)::value, XL = PASS == 0 && isA;  // XL: lanes along rows
      const int kl = lane & 7;
      const int r0 = 16 * (isA ? warp : warp - FX_CONV_A);  // first row of batch 0
      uint32_t st = 0;                                       // stages so far
      for (int ti = blockIdx.x; ti < p.nitems; ti += gridDim.x) {
        const LItem it = p.items[ti];
        const LSeg* sg = p.segs + it.seg;
        const int ub = sg->ub, ue = sg->ue, nst = (ue - ub + 3) / 4;
        const int rows = (isA ? sg->nlong - it.x0 : it.cnt) - r0;  // valid rows from r0
        const uint32_t dig8 = isA ? FX_A / 8 : (uint32_t)((it.cnt + 15) / 16 * 16) * 8;
        const bool active = isA || r0 < (it.cnt + 15) / 16 * 16;
        const long long ld = sg->ld;
        const double* src = p.op + kl;
        if (isA) src = p.v + sg->base + (XL ? it.x0 + r0 + kl : kl + ld * (it.x0 + r0));
        // scale so far (scale_word): lane 8 h + j has that of row r0 + 8 h + j (XL: every lane of a row has
        // it, er for batch 0 and er1 for batch 1)
        uint32_t er = scale_word(FX_EMIN), er1 = scale_word(FX_EMIN);
        if (!isA && (lane & 15) < rows)
          er = scale_word(p.opE[sg->e0 + it.s0 + r0 + (lane & 15)] + sg->head);
        // this lane's entries of the next stage to load: first address, valid K, row length
        const double* q = nullptr;
        int n = 0;
        long long step = ld;
        auto unit = [&](int c) {
          const int ul = ub + 4 * c + (lane >> 3);
          n = 0;
          if (ul < ue) {
            const LUnit u = p.units[ul];
            n = XL ? u.n : kl < u.n ? rows : 0;
            if (isA) {
              q = src + (XL ? ld * u.v : u.v);
            } else {
              step = u.kdim;
              q = src + u.op + step * (it.s0 + r0);
            }
          }
        };
        auto load = [&](double (&d)[8], int h) {
          const double* a = q + (XL ? 8 : 8 * step) * h;
          const int m = XL ? (8 * h + kl < rows ? n : 0) : n - 8 * h;
#pragma unroll
          for (int j = 0; j < 8; ++j, a += step) d[j] = j < m ? *a : 0.0;
        };
        double d[8];
        if (nst > 0 && active) {
          unit(0);
          load(d, 0);
        }
        for (int c = 0; c < nst; ++c, ++st) {
          const int b = st & 1;
          // the whole warp goes on or gives up together
          if (!__all_sync(0xffffffffu, mbar_wait(freeb(b), ((st >> 1) & 1u) ^ 1u, abort))) {
            if (lane == 0) raise_abort(abort, p.err, 41);
            return;
          }
          if (active) {
            uint8_t* sa = smem + b * FX_STAGE;
            uint32_t* es = esm + (st % FX_RING) * FX_LONG + r0;
            bool up = false;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              // growth of a scale is rare (it was set one bit above its largest entry)
              if (XL) {
                uint32_t& r = h ? er1 : er;
                int g = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) g |= (int)(r - absbits(d[j]));
                if (__any_sync(0xffffffffu, g < 0)) {
                  uint32_t e = 0;
#pragma unroll
                  for (int j = 0; j < 8; ++j) e = max(e, absbits(d[j]));
                  e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
                  e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
                  if (e > r) {
                    r = scale_word((e >> 20) + 1);
                    up = true;
                  }
                }
                const int xl = 8 * h + kl;
                if (lane < 8) es[xl] = r;
                // [digit][K / 8][row][8 K]
                uint2* o = (uint2*)(sa + (lane >> 3) * (FX_LONG * 16) + (r0 + xl) * 16);
                const uint32_t ee[4] = {r, r, r, r};
                digits4(d, ee, o, dig8);
                digits4(d + 4, ee, o + 1, dig8);
              } else {
                if (isA) {
                  int g = 0;
#pragma unroll
                  for (int j = 0; j < 8; ++j)
                    g |= (int)(__shfl_sync(0xffffffffu, er, 8 * h + j) - absbits(d[j]));
                  if (__any_sync(0xffffffffu, g < 0)) {
                    uint32_t m = 0;  // lane 8 h + j: the largest of row j
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                      const uint32_t e = __reduce_max_sync(0xffffffffu, absbits(d[j]));
                      if (lane == 8 * h + j) m = e;
                    }
                    if (m > er) {
                      er = scale_word((m >> 20) + 1);
                      up = true;
                    }
                  }
                  if ((lane >> 3) == h) es[lane] = er;
                }
                // [digit][row / 8][K][8 rows]
                uint2* o = (uint2*)(sa + (isA ? 0 : FX_S * FX_A) +
                                    (uint32_t)(r0 / 8 + h) * (FX_K * 16) + lane * 16);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                  uint32_t ee[4];
#pragma unroll
                  for (int j = 0; j < 4; ++j)
                    ee[j] = __shfl_sync(0xffffffffu, er, 8 * h + 4 * k + j);
                  digits4(d + 4 * k, ee, o + k, dig8);
                }
              }
              if (h == 0) {
                load(d, 1);
                if (c + 1 < nst) unit(c + 1);
              } else if (c + 1 < nst) {
                load(d, 0);  // in flight during the wait for the next stage
              }
            }
            if (isA) {
              up = __any_sync(0xffffffffu, up);
              if (lane == 0) grown[(st % FX_RING) * FX_CONV_A + warp] = up;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(ready(b));
        }
      }
    };
    if (warp < FX_CONV_A)
      convert(std::true_type{});
    else
      convert(std::false_type{});
  } else if (warp < FX_EPI0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FX_R_MMA));
    // ------------------------------- MMA issuer ---------------------------------
    // the whole warp runs the loops, one elected lane issues
    if (warp == FX_CONV) {
      uint32_t st = 0, g = 0, next = 0, first = 0;  // g: current group
      bool ok = true;
      const uint32_t el = elect_one();
      // V: pass 0 K-major (K cores 2048 apart, row cores 128), pass 1 MN-major
      const uint64_t ah = PASS == 0 ? sdesc(0, FX_LONG * 16, 128, 0) : sdesc(0, 128, FX_K * 16, 0);
      const uint64_t bh = sdesc(0, 128, FX_K * 16, 0);
      constexpr uint32_t AK = PASS == 0 ? 2 * FX_LONG * 16 : 256;  // 16 K further on
      for (int ti = blockIdx.x; ti < p.nitems && ok; ti += gridDim.x) {
        const LItem it = p.items[ti];
        const LSeg sg = p.segs[it.seg];
        const int nst = (sg.ue - sg.ub + 3) / 4;
        const uint32_t N = (it.cnt + 15) / 16 * 16;
        // FP32 accumulate, FP16 operands, M = 128; bit 15 / 16: A / B are MN-major
        const uint32_t id = (1u << 4) | ((PASS == 0 ? 0u : 1u) << 15) | (1u << 16) |
                            ((uint32_t)(FX_LONG >> 4) << 24);
        int len = 0;  // stages in the group so far
        for (int c = 0; c < nst && ok; ++c, ++st) {
          const int b = st & 1;
          ok = __all_sync(0xffffffffu, mbar_wait(ready(b), (st >> 1) & 1u, abort));
          if (!ok) {
            if (lane == 0) raise_abort(abort, p.err, 42);
            break;
          }
          const int gr = lane < FX_CONV_A ? grown[(st % FX_RING) * FX_CONV_A + lane] : 0;
          const bool fresh = c == 0 || len == FX_GROUP || __any_sync(0xffffffffu, gr != 0);
          const bool last = c + 1 == nst;
          if (fresh) {
            if (c > 0 && el) umma_commit(tfull);  // the group before this stage is complete
            len = 0;
            first = st;
            g = next++;
            ok = __all_sync(0xffffffffu, mbar_wait(tempty, (g & 1u) ^ 1u, abort));
            if (!ok) {
              if (lane == 0) raise_abort(abort, p.err, 43);
              break;
            }
            tc_fence_after();
          }
          ++len;
          if ((fresh || last) && el) {
            ginfo[g & 3] = 2 * first + (last ? 1 : 0);
            __threadfence_block();
          }
          const uint32_t sa = smem_u32(smem) + b * FX_STAGE;
          const uint64_t a0 = ah | sdesc_addr(sa), b0 = bh | sdesc_addr(sa + FX_S * FX_A);
          uint32_t n;  // opaque: keeps the instruction descriptors out of the outer loops
          asm volatile("mov.u32 %0, %1;" : "=r"(n) : "r"(N));
          if (el) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int i = 0; i < FX_S; ++i) {
                const uint32_t w = n * (FX_S - i);  // columns of diagonals i .. 6
                const uint64_t a = a0 + ((i * FX_A + k * AK) >> 4), bb = b0 + ((k * 256) >> 4);
                const uint32_t dt = tmem + n * i, acc = k > 0 || i > 0 || !fresh;
                umma_t<1>(dt, a, bb, id | (min(w, 256u) >> 3) << 17, acc);
                if (i < 4 && w > 256)  // N = 48 or 64: the columns above 256
                  umma_t<1>(dt + 256, a, bb + ((256 / 8 * FX_K * 16) >> 4),
                            id | ((w - 256) >> 3) << 17, acc);
              }
            umma_commit(freeb(b));
            if (last) umma_commit(tfull);
          }
        }
      }
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(FX_R_EPI));
    // -------------------- integers: diagonals from tensor memory -----------------
    const int q4 = warp & 3, half = (warp - FX_EPI0) >> 2;
    const uint32_t lane_base = (uint32_t)(32 * q4) << 16;
    uint32_t g = 0;
    bool ok = true;
    // the descriptors are read again here, not kept over the accumulation
    auto put_item = [&](const LItem it, int xl, int j0, int nj, int E, const long long (&acc)[32]) {
      const LSeg sg = p.segs[it.seg];
      const long long x = it.x0 + xl;
      if (nj > 0 && x < sg.nlong) {
        const double nanv = __longlong_as_double(0x7ff8000000000000ll);
        const int j1 = sg.off + it.s0 + j0;
        if (PASS == 0) {
          double* yp = p.y + sg.base + x + (long long)sg.ld * j1;
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j < nj) {
              const int eb = p.opE[sg.e0 + it.s0 + j0 + j];
              const bool bad = E == 2048 || eb == 2047;  // Inf or NaN
              yp[(long long)sg.ld * j] =
                  bad ? nanv : scaled(acc[j], E + eb + sg.head + 68 - 2 * 1083);
            }
        } else {
          double* yp = p.y + sg.base + j1 + (long long)sg.ld * x;
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j < nj) {
              const int eb = p.opE[sg.e0 + it.s0 + j0 + j];
              const bool bad = E == 2048 || eb == 2047;  // Inf or NaN
              yp[j] += bad ? nanv : scaled(acc[j], E + eb + sg.head + 68 - 2 * 1083);
            }
          // the segment's padding rows, after its last index
          if (it.s0 + j0 + nj == sg.dim && (half == 1 || it.cnt <= 32))
            for (int j = sg.dim; j < sg.dim_pad; ++j)
              p.y[sg.base + sg.off + j + (long long)sg.ld * x] = 0.0;
        }
      }
    };
    for (int ti = blockIdx.x; ti < p.nitems && ok; ti += gridDim.x) {
      const LItem it = p.items[ti];
      const int xl = 32 * q4 + lane, j0 = 32 * half;
      const int nj = max(0, min(32, it.cnt - j0)), N = (it.cnt + 15) / 16 * 16;
      long long acc[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) acc[j] = 0;
      int E = FX_EMIN;
      bool more = p.segs[it.seg].ue > p.segs[it.seg].ub;
      for (; more && ok; ++g) {
        ok = __all_sync(0xffffffffu, mbar_wait(tfull, g & 1u, abort));
        if (!ok) {
          if (lane == 0) raise_abort(abort, p.err, 44);
          break;
        }
        tc_fence_after();
        const uint32_t gi = ginfo[g & 3];
        more = !(gi & 1u);
        const int En = (int)(esm[((gi >> 1) % FX_RING) * FX_LONG + xl] >> 20);
        if (En != E) {
          const int sh = min(En - E, 63);
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] >>= sh;
          E = En;
        }
        // eight columns of one diagonal at a time; the next eight are read meanwhile
        uint32_t r[2][8];
        const uint32_t tc = tmem + lane_base + j0;
        if (nj > 0) {
          tmem_ld8(tc, r[0]);
          tmem_wait8(r[0]);
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          if (8 * h >= nj) break;
#pragma unroll
          for (int d = 0; d < FX_S; ++d) {
            uint32_t(&cur)[8] = r[(FX_S * h + d) & 1], (&nxt)[8] = r[(FX_S * h + d + 1) & 1];
            const bool go = d + 1 < FX_S || (h < 3 && 8 * h + 8 < nj);
            if (go) tmem_ld8(d + 1 < FX_S ? tc + (d + 1) * N + 8 * h : tc + 8 * h + 8, nxt);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              // weight 2^(44 - 8 d); d = 6 and 7 are rounded to the unit.  |sum| < 2^22 for
              // d <= 2 (the leading digits are at most 33): the cheap conversion
              constexpr float magic = 12582912.f;  // 1.5 * 2^23: the integer in the low bits
              const float x = __uint_as_float(cur[j]);
              int a = d < 3 ? __float_as_int(x + magic) - 0x4B400000 : __float2int_rn(x);
              if (d == 6) a = (a + 8) >> 4;
              if (d == 7) a = (a + 2048) >> 12;
              constexpr int W[FX_S] = {0, 0, 1 << 28, 1 << 20, 1 << 12, 1 << 4, 1, 1};
              if (d < 2)
                acc[8 * h + j] += (long long)((unsigned long long)(unsigned)(a * (d == 0 ? 4096 : 16)) << 32);
              else
                asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc[8 * h + j]) : "r"(a), "r"(W[d]));
            }
            if (go) tmem_wait8(nxt);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
      if (!ok) break;
      // ---- the item's outputs ----
      put_item(p.items[ti], xl, j0, nj, E, acc);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == FX_CONV) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  }
}

// largest exponent field of every operator row of every segment; one warp per row
__global__ void __launch_bounds__(256)
k_fx_opE(const LSeg* __restrict__ segs, const LK* __restrict__ ks, const double* __restrict__ op,
         int* __restrict__ out) {
  const LSeg sg = segs[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int j = blockIdx.y * 8 + warp; j < sg.dim; j += gridDim.y * 8) {
    int e = FX_EMIN;
    for (int b = sg.kb; b < sg.ke; ++b) {
      const LK k = ks[b];
      const double* row = op + k.op + (long long)j * k.kdim;
      for (int i = lane; i < k.kdim; i += 32) e = max(e, expo(row[i]));
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) out[sg.e0 + j] = e;
  }
}

}  // namespace

void fx_opE(LongPlan* L, cudaStream_t s) {
  for (int ps = 0; ps < 2; ++ps) {
    if (L->segs[ps].empty()) continue;
    int mx = 1;
    for (const LSeg& sg : L->segs[ps]) mx = std::max(mx, sg.dim);
    const dim3 grid((unsigned)L->segs[ps].size(), (unsigned)std::min((mx + 7) / 8, 1024));
    k_fx_opE<<<grid, 256, 0, s>>>(L->d_segs[ps], L->d_ks[ps], L->op64[ps], L->d_opE[ps]);
  }
}

int fx_launch(const LongPlan* L, const double* v, double* y, cudaStream_t s) {
  for (int ps = 0; ps < 2; ++ps) {
    FxParams p;
    p.nitems = (int)L->fitems[ps].size();
    if (!p.nitems) continue;
    p.items = L->d_fitems[ps];
    p.segs = L->d_segs[ps];
    p.units = L->d_units[ps];
    p.opE = L->d_opE[ps];
    p.op = L->op64[ps];
    p.v = v;
    p.y = y;
    p.err = L->err;
    const int grid = std::min(p.nitems, L->sms);
    if (ps == 0) {
      D2_CUDA(cudaFuncSetAttribute(hv_fx_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)FX_SMEM));
      hv_fx_kernel<0><<<grid, FX_THREADS, FX_SMEM, s>>>(p);
    } else {
      D2_CUDA(cudaFuncSetAttribute(hv_fx_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)FX_SMEM));
      hv_fx_kernel<1><<<grid, FX_THREADS, FX_SMEM, s>>>(p);
    }
  }
  D2_CUDA(cudaGetLastError());
  return DMRG2D_OK;
}

}  // namespace dmrg2d
