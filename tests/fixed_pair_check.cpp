// Host check of the fixed-point pair arithmetic (csrc/fixed.cuh): random pairs
// over its whole range (extents 2^-30 to 2^30, distances down to the close-pair
// limit, offsets up to 2^15 extents, masses over the mass rule) against
// extended precision.  Prints the largest errors in units of their bounds.
//   force: 2^-55 (largest / mass) + 4 u / r;  potential: 2^-57 (largest / mass) + 4 u / r
// where u is the unit of the coordinates (each rounded by at most u / 2, plus
// the 16-bit products of the low words: below 2^-52 r at r = 2^51 u).  With an
// exponent of its own a mass is as exact as the largest, down to the last place
// of the sums (2^-57 of the largest mass's force at the tile's extent, which is
// what the mass rule bounds: see the sums around a heavy particle below).
// Then pairs with r^2 exactly a power of four, where x = 1/4 and 1/r is at the
// top of its range: prints the largest error of both terms in units of 2^-57.
// Then the force on the heaviest particle of its tile, at the end of the mass
// rule: 127 light ones on a sphere around it; prints the largest error in units
// of 2^-53 of the sum of the terms' magnitudes.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#include "../paper_1803_01190_gb300/csrc/fixed.cuh"

using namespace nb;
typedef long double ld;

static uint32_t hi(double x) { uint64_t b; memcpy(&b, &x, 8); return (uint32_t)(b >> 32); }
static uint32_t lo(double x) { uint64_t b; memcpy(&b, &x, 8); return (uint32_t)b; }
static ld value(const fx96 &a, int e) {
  return ldexpl((ld)a.w2, e + 64) + ldexpl((ld)a.w1, e + 32) + ldexpl((ld)a.w0, e);
}

int main() {
  std::mt19937_64 g(5);
  auto U = [&] { return (double)(g() >> 11) * 0x1p-53; };
  double worst_f = 0, worst_p = 0, bias = 0;
  long used = 0, plain = 0, close = 0, wrong = 0;
  for (long t = 0; t < 600000; t++) {
    const double E = std::exp2(-30 + 60 * U());
    int e;
    frexp(E, &e);
    const int L = e - FX_BITS;
    const double eps = E * std::exp2(-20 + 20 * U()) * 0.99;
    const double off = (t & 1) ? 0.0 : E * std::exp2(20 * U() - 5) * (U() - 0.5);
    const double span = E * std::exp2(-14 * U());
    double xi[3], xj[3];
    uint64_t Xi[3], Xj[3];
    for (int c = 0; c < 3; c++) {
      xi[c] = off + 0.3 * E * (U() - 0.5);
      xj[c] = xi[c] + 0.99 * span * (U() - 0.5);
      Xi[c] = fx_coord(hi(xi[c]), lo(xi[c]), L);
      Xj[c] = fx_coord(hi(xj[c]), lo(xj[c]), L);
    }
    const double mmax = std::exp2(-20 + 40 * U());
    const int em = ilogb(mmax);
    const bool wide = t % 5 == 0, equal = t % 5 == 1;
    const int range = wide ? FX_MASS_RANGE : FX_MASS_NARROW;
    const double m = equal ? 1.0 : t % 3 ? mmax * std::exp2(-range * U()) : mmax;
    if (!equal && ilogb(m) < em - range) continue;
    const FxMass M = equal ? FxMass{0, 0, 0} : wide ? fx_mass<true>(hi(m), lo(m), em) : fx_mass<false>(hi(m), lo(m), em);
    const FxEps e2 = fx_eps2(eps * eps, L);
    const float off_seed = 1.0f + (float)((2 * U() - 1) * 0x1p-22);  // the SFU's error
    FxPair p;
    const bool ok = fx_geometry<false>(Xj, Xi, e2, [&](uint32_t x) {
      const float y = (float)(1.0 / std::sqrt((double)(float)x)) * off_seed;
      uint32_t b;
      memcpy(&b, &y, 4);
      return b;
    }, p);
    ld d[3], r2 = (ld)(eps * eps);
    for (int c = 0; c < 3; c++) {
      d[c] = (ld)xj[c] - (ld)xi[c];
      r2 += d[c] * d[c];
    }
    const ld r = sqrtl(r2), ur = ldexpl(1, L) / r;
    // the limit: |d| between sqrt(63/64) 2^51 units and 2^51 units
    const ld du = sqrtl(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) / ldexpl(1, L + 51);
    if (!ok) {
      close++;
      if (du > 1.001L) wrong++;
      continue;
    }
    if (du < 0.992L) wrong++;
    fx96 f[3] = {}, pot = {};
    if (equal)
      fx_both<false>(p, f, pot, nullptr, nullptr);
    else if (wide)
      fx_side<false, true>(p, M, f, pot);
    else
      fx_side<false, false>(p, M, f, pot);
const ld ratio = equal ? 1 : (ld)mmax / m;
    const int e_m = equal ? FX_EQ_EM : em;
    // with its own exponent: the place of the last bit of the 96-bit sums
    const ld light_f = wide ? 1 + ldexpl(ratio, -2) : ratio;
    const ld light_p = wide ? 1 + ldexpl(ratio, -12) : ratio;
    const ld rel = value(pot, fx_pot_exp(L, e_m)) * r / m - 1;
    ld err = 0;
    for (int c = 0; c < 3; c++) {
      const ld x = value(f[c], fx_force_exp(L, e_m)) * r2 / m - d[c] / r;
      err += x * x;
    }
    worst_f = std::fmax(worst_f, (double)(sqrtl(err) / (ldexpl(light_f, -55) + 4 * ur)));
    worst_p = std::fmax(worst_p, (double)(fabsl(rel) / (ldexpl(light_p, -57) + 4 * ur)));
    if (!wide) bias += (double)rel, plain++;
    used++;
  }
  double worst_4 = 0;
  for (int k = -40; k <= 3; k++)  // r = 2^k at a unit of 2^(4 - FX_BITS)
    for (int axis = 0; axis < 2; axis++)
      for (int seed = -2; seed <= 2; seed++) {
        const int L = 4 - FX_BITS;
        const double r = std::exp2(k), d = axis ? r : r / 2, eps2 = axis ? 0.0 : r * r / 4;
        if (std::exp2(51 + L) >= r) continue;
        const uint64_t Xi[3] = {0, 0, 0}, q = fx_coord(hi(d), lo(d), L);
        const uint64_t Xj[3] = {q, axis ? 0 : q, axis ? 0 : 0 - q};
        FxPair p;
        fx_geometry<false>(Xj, Xi, fx_eps2(eps2, L), [&](uint32_t x) {
          const float y = (float)(1.0 / std::sqrt((double)(float)x)) * (1.0f + (float)seed * 0x1p-23f);
          uint32_t b;
          memcpy(&b, &y, 4);
          return b;
        }, p);
        for (int form = 0; form < 3; form++) {  // equal, one exponent, an exponent each
          fx96 f[3] = {}, pot = {};
          const FxMass M = form == 1 ? fx_mass<false>(hi(1.0), 0, 0) : fx_mass<true>(hi(1.0), 0, 0);
          if (form == 0)
            fx_both<false>(p, f, pot, nullptr, nullptr);
          else if (form == 1)
            fx_side<false, false>(p, M, f, pot);
          else
            fx_side<false, true>(p, M, f, pot);
          const int em = form ? 0 : FX_EQ_EM;
          const ld ep = value(pot, fx_pot_exp(L, em)) * r - 1;
          const ld ef = value(f[0], fx_force_exp(L, em)) * r * r * r / d - 1;
          worst_4 = std::fmax(worst_4, (double)std::fmax(fabsl(ep), fabsl(ef)));
        }
      }
  double worst_heavy = 0;
  std::normal_distribution<double> N;
  for (int s = 0; s < 200; s++) {  // masses of 1 around one of 2^FX_MASS_RANGE, unit 2^(1 - FX_BITS)
    const int L = 1 - FX_BITS;
    const uint64_t Xi[3] = {0, 0, 0};
    fx96 f[3] = {}, pot = {};
    ld sum[3] = {0, 0, 0}, size = 0;
    for (int k = 0; k < 127; k++) {
      double x[3], n = 0;
      uint64_t Xj[3];
      for (double &c : x) c = N(g), n += c * c;
      for (int c = 0; c < 3; c++) {
        x[c] /= std::sqrt(n);
        Xj[c] = fx_coord(hi(x[c]), lo(x[c]), L);
      }
      FxPair p;
      fx_geometry<false>(Xj, Xi, fx_eps2(1e-4, L), [&](uint32_t v) {
        const float y = (float)(1.0 / std::sqrt((double)(float)v));
        uint32_t b;
        memcpy(&b, &y, 4);
        return b;
      }, p);
      fx_side<false, true>(p, fx_mass<true>(hi(1.0), 0, FX_MASS_RANGE), f, pot);
      ld r2 = 1e-4L, d2 = 0;
      for (double c : x) r2 += (ld)c * c, d2 += (ld)c * c;
      for (int c = 0; c < 3; c++) sum[c] += x[c] / (r2 * sqrtl(r2));
      size += sqrtl(d2) / (r2 * sqrtl(r2));
    }
    ld err = 0;
    for (int c = 0; c < 3; c++) {
      const ld v = value(f[c], fx_force_exp(L, FX_MASS_RANGE)) - sum[c];
      err += v * v;
    }
    worst_heavy = std::fmax(worst_heavy, (double)(sqrtl(err) / size));
  }
  printf("%ld %ld %ld %.4f %.4f %.3e %.3f %.3f\n", used, close, wrong, worst_f, worst_p, bias / plain,
         std::ldexp(worst_4, 57), std::ldexp(worst_heavy, 53));
  return 0;
}
