// What the block fixed point of csrc/fixpoint.h accepts is as accurate as FP64: over rows and vectors whose entries differ
// by up to 30 orders of magnitude, every sum that has the words of fix_needed errs by less than 21 x 2^-53 of S, the sum
// of the magnitudes of its 48 products (long double reference); rough rows and vectors are taken, and sums whose S is
// below 2^E / 10 never are.
#include <cmath>
#include <cstdio>

#include "fixpoint.h"

using namespace lqcd;

static uint64_t state = 0x243f6a8885a308d3ull;
static double uniform() {  // SplitMix64
  uint64_t z = (state += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return (double)((z ^ (z >> 31)) >> 11) * (1.0 / 9007199254740992.0);
}

int main() {
  int taken = 0, rough_taken = 0, rough = 0;
  for (int t = 0; t < 60000; ++t) {
    const bool is_rough = t % 3 == 0;
    double u[8][6], v[8][6];
    // what differs in size: entry by entry, or the same three entries (a colour) in every hop
    const double su = is_rough ? 0 : 30 * uniform() * (t % 2), sv = is_rough ? 0 : 30 * uniform();
    double cu[6], cv[6];
    for (int c = 0; c < 6; ++c) cu[c] = std::pow(10, -su * uniform()), cv[c] = std::pow(10, -sv * uniform());
    for (int h = 0; h < 8; ++h) {
      double n = 0;
      for (int c = 0; c < 6; ++c) u[h][c] = (2 * uniform() - 1) * cu[c], n += u[h][c] * u[h][c];
      // row norm 1/2, or a small row of a link whose other entries hold the norm
      if (is_rough || t % 4 < 2)
        for (double& a : u[h]) a *= 0.5 / std::sqrt(n);
      else
        for (double& a : u[h]) a *= 0.2;
      for (int c = 0; c < 6; ++c) v[h][c] = (2 * uniform() - 1) * cv[c];
    }
    int w[4];
    for (int q = 0; q < 4; ++q) {
      double both[12];
      for (int k = 0; k < 12; ++k) both[k] = v[2 * q + k / 6][k % 6];
      w[q] = fix_max_word(both);
    }
    const int E = fix_block_exponent(w);
    int64_t sum = 0;
    uint32_t words = 0;
    long double exact = 0, S = 0;
    for (int q = 0; q < 4; ++q) {
      int64_t hh = 0, x = 1 << (kFixLow - 1);
      int fwd = 0;
      for (int k = 0; k < 12; ++k) {
        if (k == 6) fwd = fix_upper(hh);
        const int h = 2 * q + k / 6, c = k % 6;
        const Fix2 a = fix_link_entry(u[h][c]);
        const Fix2 b = fix_component<false>(v[h][c], E);
        fix_mac(hh, x, a.h, a.l, b);
        const long double prod = (long double)u[h][c] * v[h][c];
        exact += prod;
        S += std::fabs(prod);
      }
      const int64_t part = hh + (x >> kFixLow);
      words += fix_hop_words(fwd, fix_upper(part));
      sum += part;
    }
    const bool ok = words >= fix_needed(w, E);
    taken += ok;
    rough += is_rough;
    rough_taken += is_rough && ok;
    const long double got = std::ldexp((long double)sum, E - kFixUnit), unit = std::ldexp(1.0L, E - 1023);
    if (ok && (std::fabs(got - exact) > 21 * std::ldexp(1.0L, -53) * S || S < unit / 10)) {
      std::printf("error %.3Lg, S %.3Lg, unit %.3Lg\n", got - exact, S, unit);
      return 1;
    }
  }
  // a rough sum falls short in fewer than one case of 10^3 (eight hops of near zero)
  if (rough_taken < rough - rough / 1000 || taken == rough_taken || taken > 59000) {
    std::printf("taken %d, rough %d of %d\n", taken, rough_taken, rough);
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
