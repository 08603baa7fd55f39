// How the look-ahead stream and the main stream share the GPU's SMs while a factorisation's diagonal block runs beside a
// trailing update (host code).
#pragma once

#include <stdint.h>

namespace exa {

constexpr int kDiagCtas = 104;  // CTAs of one diagonal-block launch at most

// What a 512 block takes on a grid (measured), microseconds.  Nothing is gained beyond 104 CTAs.
inline double diag_block_us(int ctas) {
  constexpr struct { int ctas; double us; } kAt[] = {{16, 1180.0}, {32, 698.0}, {64, 464.0}, {104, 426.0}};
  if (ctas <= kAt[0].ctas) return kAt[0].us * kAt[0].ctas / ctas;
  for (int i = 1; i < 4; ++i)
    if (ctas <= kAt[i].ctas) {  // linear in the reciprocal
      const double f = (1.0 / ctas - 1.0 / kAt[i].ctas) / (1.0 / kAt[i - 1].ctas - 1.0 / kAt[i].ctas);
      return kAt[i].us + f * (kAt[i - 1].us - kAt[i].us);
    }
  return kAt[3].us;
}

// CTAs of a diagonal block for which `wanted` are asked: all are resident at once, one an SM, and CTA 0 runs the leaves
// while at least one other runs the updates.
inline int diag_grid(int wanted, int sms) {
  const int grid = wanted < kDiagCtas ? wanted : kDiagCtas;
  return grid < 2 ? 2 : grid < sms ? grid : sms;
}

// The look-ahead stream's share beside a trailing update of m rows from a panel of `width` as digit products
// (m^2 width operations at 42 TFLOP/s on 152 SMs): the grid of the diagonal block with which the later of the two ends
// first.  Less than sms, so that the update has an SM left.
inline int side_share(int64_t m, int width, int sms) {
  const double update_us = (double)m * (double)m * width / 42e6 * 152.0;  // on one SM
  int best = 0;
  double best_us = 0.0;
  for (int ctas = kDiagCtas; ctas >= 16; ctas -= 8) {
    if (ctas >= sms) continue;
    const double block = diag_block_us(ctas), update = update_us / (sms - ctas);
    const double us = block > update ? block : update;
    if (best == 0 || us < best_us) {
      best_us = us;
      best = ctas;
    }
  }
  return best > 0 ? best : sms > 3 ? sms / 2 : 2;
}

}  // namespace exa
