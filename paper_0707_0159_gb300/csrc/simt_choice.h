// Which dense CUDA-core kernel a superblock takes.  Host code without CUDA; internal header.
#pragma once
#include <algorithm>
#include <cstdint>

namespace dmrg2d {

struct SimtChoice {
  int piece;      // side of the square pieces: 64, 32, 16 or 8
  bool two_pass;  // the two-pass kernel instead
};

// d x d tiles of m1 x m4 in pieces of side b
inline int64_t simt_pieces(int m, int d, int b) { return (int64_t)((m + b - 1) / b) * d; }
inline bool simt_grid_fits(int m1, int m4, int d, int b) {
  return simt_pieces(m1, d, b) <= 0x7fffffff && simt_pieces(m4, d, b) <= 65535;
}

// FP64: every kernel runs at the FP64 pipe's rate, so the time is the fullest SM's outputs times
// their padded K: pieces of 64, 32, 16 or 8, or the two-pass kernel, which pads nothing
// but takes two kernels more and 1.1 of the rate, once it has two items per SM.
// (3-leg Heisenberg 250 x 131: pieces of 64 9.63 ms, two-pass 6.13 ms; 2-leg 200 x 200:
// pieces of 64 2.53 ms, of 8 1.31 ms; 2-leg Hubbard 40 x 40: 0.99 and 0.34 ms.)
// Pieces whose grid is beyond the launch limits (of 16 at d = 256, m4 = 4096) are passed over.
inline SimtChoice simt_choice_f64(int m1, int m4, int d, int sms, int64_t items) {
  auto pad = [](int m, int b) { return (double)((m + b - 1) / b * b) / m; };
  const double kpad = std::max(pad(m1, 16), pad(m4, 16));
  double best = 0.0;
  int piece = 0;
  for (int b : {64, 32, 16, 8}) {
    if (!simt_grid_fits(m1, m4, d, b)) continue;
    const int64_t g = simt_pieces(m1, d, b) * simt_pieces(m4, d, b);
    const double cost = (double)((g + sms - 1) / sms) * b * b * kpad;
    if (!piece || cost < 0.98 * best) {
      best = cost;
      piece = b;
    }
  }
  const double n = (double)m1 * m4 * d * d;
  const bool two_pass = items >= 2 * sms && (!piece || 1.1 * n / sms < 0.98 * best);
  return {piece ? piece : 64, two_pass};
}

// FP32: the largest piece (64, 32 or 16 square) whose grid still gives every SM a CTA; the
// two-pass kernel's larger register tiles once they fill nearly half of the SMs (2-leg
// 100 x 128, 32 items: 66 us in pieces, 67 two-pass; 2-leg Hubbard 40 x 40, 80 items: 80
// and 48 us; 3-leg Heisenberg 250 x 131: 641 and 295 us; 3-leg Hubbard 128 x 128: 12.4
// and 5.8 ms).
inline SimtChoice simt_choice_f32(int m1, int m4, int d, int sms, int64_t items) {
  auto ctas = [&](int b) { return simt_pieces(m1, d, b) * simt_pieces(m4, d, b); };
  return {ctas(64) >= sms ? 64 : (ctas(32) >= sms ? 32 : 16), 5 * items >= 2 * (int64_t)sms};
}

}  // namespace dmrg2d
