// Host-side checks of the fixed-point products of the float64 path (csrc/fix64.cuh), no GPU needed:
//   * to_fix is x 2^(56-e) rounded to the nearest integer, in slices within their ranges, for values
//     over the whole exponent range, zeros, subnormals and non-finite values (which give 0);
//   * sums of 64 products of extreme slices stay within 64 bits;
//   * a sum of K <= 64 products is within K (2^-57 + 2^-57 + 2^-58) 2^(ex + ey) + the final rounding
//     of the long double sum of the exact products, and over blocks of normal random numbers its
//     root-mean-square error is no larger than that of the float64 multiply-add loop.
// Prints "ok" and exits 0, or prints the first violations and exits 1.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_1503_03004_gb300/csrc/fix64.cuh"

using namespace sfr;

static int fails = 0;
#define CHECK(cond, ...)                      \
  do {                                        \
    if (!(cond) && fails++ < 10) {            \
      std::printf("FAIL %s: ", #cond);        \
      std::printf(__VA_ARGS__);               \
      std::printf("\n");                      \
    }                                         \
  } while (0)

static int hi_word(double x) {
  long long b;
  std::memcpy(&b, &x, sizeof b);
  return (int)(b >> 32) & 0x7fffffff;
}

static __int128 value(int2 f) { return (__int128)f.x * (1LL << 28) + f.y; }

static void check_fix(double x, int e) {
  const int2 f = fx::to_fix(x, e);
  CHECK(f.x <= (1 << 28) && f.x >= -(1 << 28) && f.y < (1 << 27) && f.y >= -(1 << 27), "%a e %d: %d %d", x, e, f.x, f.y);
  // x 2^(56-e) in 80-bit floats is exact; ties round away from zero
  const long double want = std::round(std::ldexp((long double)x, 56 - e));
  CHECK((long double)(long long)value(f) == want, "%a e %d: %lld want %Lf", x, e, (long long)value(f), want);
}

int main() {
  std::mt19937_64 g(7);
  for (int it = 0; it < 400000; ++it) {
    uint64_t b = g();
    double x;
    std::memcpy(&x, &b, sizeof x);
    if (!std::isfinite(x)) {
      const int2 f = fx::to_fix(x, 3);
      CHECK(f.x == 0 && f.y == 0, "non-finite");
      continue;
    }
    const int e = fx::exponent(hi_word(x));
    CHECK(std::fabs((long double)x) < std::ldexp(1.0L, e), "%a exponent %d", x, e);
    check_fix(x, e);
    check_fix(x, e + (int)(g() % 70));
  }
  for (double x : {0.0, -0.0, 5e-324, -5e-324, 2.2250738585072014e-308, 1.0, -1.0, 0x1.fffffffffffffp0, 1.7976931348623157e308})
    check_fix(x, fx::exponent(hi_word(x)));
  check_fix(0x1p5, 5);  // at the bound itself (a rounded bound may be met)
  CHECK(fx::exponent(hi_word(INFINITY)) == fx::kBad && fx::exponent(hi_word(NAN)) == fx::kBad, "kBad");
  CHECK(std::isnan(fx::Scale(fx::kBad + 100).c1) && std::isnan(fx::Scale(fx::kBad - 2000).c2), "NaN scale");
  for (int k = -1100; k <= 1030; ++k) CHECK(fx::pow2(k) == std::ldexp(1.0, k), "pow2 %d", k);

  // extreme slices: no overflow over kTerms products
  for (int sx : {-1, 1})
    for (int sy : {-1, 1}) {
      __int128 H = 0, C = 0;
      long long hh = 0, cx = 0;
      const int2 a = make_int2(sx * (1 << 28), -(1 << 27)), b = make_int2(sy * (1 << 28), -(1 << 27));
      for (int k = 0; k < fx::kTerms; ++k) {
        fx::mac(a, b, hh, cx);
        H += (__int128)a.x * b.x;
        C += (__int128)a.x * b.y + (__int128)a.y * b.x;
      }
      CHECK(H == hh && C == cx, "overflow");
      const __int128 t = H + ((C + (1 << 27)) >> 28);
      CHECK(t == fx::total(hh, cx), "overflow of the total");
    }

  std::normal_distribution<double> nd;
  long double rms_fix = 0, rms_f64 = 0;
  for (int it = 0; it < 20000; ++it) {
    const int K = 1 + (int)(g() % 64);
    const double sx = std::ldexp(1.0, (int)(g() % 40) - 20), sy = std::ldexp(1.0, (int)(g() % 40) - 20);
    std::vector<double> x(K), y(K);
    int hx = 0, hy = 0;
    for (int k = 0; k < K; ++k) {
      x[k] = sx * nd(g);
      y[k] = sy * nd(g);
      hx = std::max(hx, hi_word(x[k]));
      hy = std::max(hy, hi_word(y[k]));
    }
    const int ex = fx::exponent(hx), ey = fx::exponent(hy);
    long long hh = 0, cx = 0;
    long double want = 0;
    double loop = 0;
    for (int k = 0; k < K; ++k) {
      fx::mac(fx::to_fix(x[k], ex), fx::to_fix(y[k], ey), hh, cx);
      want += (long double)x[k] * y[k];
      loop = std::fma(x[k], y[k], loop);
    }
    const double got = fx::add_total(fx::total(hh, cx), fx::Scale(ex + ey), 0.0);
    const long double unit = std::ldexp(1.0L, ex + ey), err = std::fabs((long double)got - want);
    const long double bar = K * unit * (2 * 0x1p-57L + 0x1p-58L) + unit * 0x1p-57L + std::fabs(want) * (0x1p-53L + 64 * 0x1p-64L);
    CHECK(err <= bar, "K %d: error %Lg over %Lg", K, err, bar);
    rms_fix += err / unit * err / unit;
    rms_f64 += ((long double)loop - want) / unit * ((long double)loop - want) / unit;
  }
  CHECK(rms_fix <= rms_f64, "rms error %Lg against %Lg of the float64 loop", std::sqrt(rms_fix), std::sqrt(rms_f64));
  if (fails) {
    std::printf("%d violations\n", fails);
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
