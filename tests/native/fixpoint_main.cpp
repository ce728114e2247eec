// The block fixed point of csrc/fixpoint.h on the host: one component's 48 products summed as the FP64 Dslash
// kernel sums them (four threads of two hops each), against long double (at least 64 significant bits), over
// seeded SU(3)-like rows and vectors of many scales; and the limits of the format.
//
// Bar: the digits drop less than 2^-57 of the largest component per vector component (times a link entry, 48
// terms, row norms <= 1/2: at most 8 x sqrt(6) / 2 x 2^-57), round link entries to 2^-58 (48 terms of at most the
// largest component), drop L L products below 2^-58 each (48 terms), and round H L once per thread (4 x 2^-59):
// together below 112 x 2^-58 of the largest component.
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include <limits>

#include "fixpoint.h"

using namespace lqcd;

struct C {
  double x, y;
};

static uint64_t state = 0x9e3779b97f4a7c15ull;
static uint64_t next_u64() {  // SplitMix64
  uint64_t z = (state += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static double uniform() { return (double)(next_u64() >> 11) * (1.0 / 9007199254740992.0); }
static double signed_uniform() { return 2 * uniform() - 1; }

static int fail(const char* what, double got, double want) {
  std::printf("%s: %.17g, not %.17g\n", what, got, want);
  return 1;
}

int main() {
  const double bar = 112 * std::ldexp(1.0, -58);
  for (int t = 0; t < 20000; ++t) {
    // eight rows (3 complex entries) of norm 1/2 and eight vectors
    double u[8][6], v[8][6], vmax = 0;
    const int scale = (int)(uniform() * 1400) - 700, spread = (int)(uniform() * 3) * 40;
    for (int h = 0; h < 8; ++h) {
      double n = 0;
      for (double& a : u[h]) a = signed_uniform() * (uniform() < 0.1 ? 1e-9 : 1), n += a * a;
      for (double& a : u[h]) a *= 0.5 / std::sqrt(n);
      for (double& a : v[h]) {
        a = uniform() < 0.05 ? 0.0 : std::ldexp(signed_uniform(), scale - (int)(uniform() * spread));
        vmax = std::fmax(vmax, std::fabs(a));
      }
    }
    int w[4];
    for (int q = 0; q < 4; ++q) {
      double both[12];
      for (int k = 0; k < 12; ++k) both[k] = v[2 * q + k / 6][k % 6];
      w[q] = fix_max_word(both);
    }
    const int E = fix_block_exponent(w);
    if (E < 0) return fail("exponent", E, scale);
    int64_t sum = 0;
    long double exact = 0;
    for (int q = 0; q < 4; ++q) {
      int64_t hh = 0, x = 1 << (kFixLow - 1);
      for (int k = 0; k < 12; ++k) {
        const int h = 2 * q + k / 6, c = k % 6;
        const Fix2 a = fix_link_entry(u[h][c]);
        const bool flip = (t + k) & 1;
        const Fix2 b = flip ? fix_component<true>(v[h][c], E) : fix_component<false>(v[h][c], E);
        fix_mac(hh, x, a.h, a.l, b);
        exact += (long double)u[h][c] * (flip ? -v[h][c] : v[h][c]);
      }
      sum += hh + (x >> kFixLow);
    }
    const long double got = std::ldexp((long double)sum, E - kFixUnit);
    if (!(std::fabs((double)(got - exact)) <= bar * vmax)) return fail("sum", (double)got, (double)exact);
  }
  // single digits: exact where the mantissa fits, both signs
  for (double x : {1.0, -1.0, 0.75, 1.5, 0x1.fffffffffffffp0, std::ldexp(1.0, -57), 0.0}) {
    const Fix2 d = fix_component<false>(x, 1023), n = fix_component<true>(x, 1023);
    const double back = std::ldexp(d.h * 268435456.0 + d.l, -57);
    if (x != 0x1.fffffffffffffp0 && back != x) return fail("digit", back, x);
    if (std::fabs(back - x) > std::ldexp(1.0, -57) || n.h != -d.h || n.l != -d.l) return fail("digit", back, x);
  }
  for (double x : {0.5, -0.5, 0.501, 0x1.0000000000001p-1, 0.1, 1e-300, 0.0}) {
    const Fix2 d = fix_link_entry(x);
    const double back = std::ldexp((long double)d.h * 268435456.0L + d.l, -57);
    if (std::fabs(back - x) > std::ldexp(1.0, -58)) return fail("link digit", back, x);
  }
  // the format's limits
  const double nan = std::numeric_limits<double>::quiet_NaN(), inf = std::numeric_limits<double>::infinity();
  C one[9] = {{0.5, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0.5}, {0, 0}, {0, 0}, {0, 0}, {0.3, 0.4}};
  if (!fix_link_fits(one)) return fail("SU(3) link refused", 0, 1);
  for (double bad : {0.6, -3.0, nan, inf, -inf}) {
    C l[9];
    for (int j = 0; j < 9; ++j) l[j] = one[j];
    l[5].y = bad;
    if (fix_link_fits(l)) return fail("link taken", bad, 0);
  }
  const double small = std::ldexp(1.0, -801), large = std::ldexp(1.0, 801), tiny = 4.9e-324;
  struct {
    double x;
    int want;  // E, or -1
  } limits[] = {{0.0, kFixMinE}, {1.0, 1023}, {std::ldexp(1.0, -800), kFixMinE}, {std::ldexp(1.0, 800), kFixMaxE},
                {small, -1},     {large, -1}, {tiny, -1},                        {nan, -1},
                {inf, -1},       {-inf, -1}};
  for (const auto& c : limits) {
    const double v[2] = {0.0, c.x};
    const int w[4] = {0, fix_max_word(v), 0, 0};
    if (fix_block_exponent(w) != c.want) return fail("block exponent", fix_block_exponent(w), c.want);
  }
  std::printf("ok\n");
  return 0;
}
