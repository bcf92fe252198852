// Host-side check of the fixed-point sums of products (no GPU needed): random
// sums of four products over operand spreads from equal magnitudes to the whole
// float64 range, zeros, subnormals, infinities and NaN among them, against
// 113-bit arithmetic.
//
// Bounds.  A term is rounded to nearest, off by at most half a unit, and the
// largest term is at least 2^58 units: four terms are off by at most 2^-57 of
// the largest (and 2^-20 of that for what the product's floor drops), and the
// final rounding by 2^-53 of the result.  Without the final rounding the
// errors average out: over sums of positive terms their mean is below 2^-61 of
// the largest term (a truncation's would be 2^-57).
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_1604_07163_gb300/csrc/mg_soft64.cuh"

using namespace mgdev;

static long long check(std::mt19937_64& g, long long n, long long& declined) {
  constexpr int N = 4;
  std::uniform_real_distribution<double> U(-1, 1);
  long long bad = 0;
  for (long long t = 0; t < n; ++t) {
    S64 a[N], c[N];
    double u[N], k[N];
    __float128 exact = 0;
    double big = 0;
    bool finite = true;
    const double spread = t % 4 == 0 ? 0 : t % 4 == 1 ? 8 : t % 4 == 2 ? 60 : 1000, common = U(g);
    const double kr = t % 5 == 0 ? 190 : 20;
    for (int i = 0; i < N; ++i) {
      u[i] = (t & 8 ? common * (1 + std::ldexp(U(g), -(int)(t % 50))) : U(g)) * std::exp2(std::floor(spread * U(g)));
      k[i] = std::exp2(kr * U(g));
      if (t % 17 == i) u[i] = t & 1 ? 0.0 : -0.0;
      if (t % 1009 == i) u[i] = t & 1 ? INFINITY : NAN;
      a[i] = soft_unpack(u[i]);
      c[i] = soft_coef(k[i]);
      finite = finite && std::isfinite(u[i]);
      if (!finite) continue;
      const __float128 p = (__float128)u[i] * k[i];
      exact += p;
      big = std::fmax(big, (double)(p < 0 ? -p : p));
    }
    double out;
    if (!soft_sum4(a, c, out)) {
      ++declined;
      continue;
    }
    const __float128 d = (__float128)out - exact;
    const double err = (double)(d < 0 ? -d : d), tol = std::ldexp(big, -57) * (1 + 0x1p-20) + std::ldexp(std::fabs(out), -53);
    if (!finite || !(err <= tol)) {
      if (bad++ < 5) printf("case %lld: %a, off by %g (bound %g), finite %d\n", t, out, err, tol, finite);
    }
  }
  return bad;
}

// mean error of sums that the final rounding leaves exact: three positive terms
// and one that cancels them but for a small rest
static double mean_error(std::mt19937_64& g, int n, bool short_coefs) {
  std::uniform_real_distribution<double> U(1, 2);
  double sum = 0;
  for (int t = 0; t < n; ++t) {
    S64 a[4], c[4];
    __float128 exact = 0;
    double s = 0;
    for (int i = 0; i < 4; ++i) {
      const double k = short_coefs ? 65536.0 : 1000 * U(g), u = i < 3 ? U(g) : -(s + 1e-6) / k;
      a[i] = soft_unpack(u);
      c[i] = soft_coef(k);
      exact += (__float128)u * k;
      s += u * k;
    }
    double out;
    if (soft_sum4(a, c, out)) sum += (double)(((__float128)out - exact) / s);
  }
  return sum / n;
}

int main() {
  std::mt19937_64 g(11);
  const long long n = 1 << 23;
  long long declined = 0;
  const long long bad = check(g, n, declined);
  if (declined > n / 2) printf("declined %lld of %lld sums\n", declined, n);
  if (bad || declined > n / 2) return 1;
  for (bool b : {false, true}) {
    const double m = mean_error(g, 1 << 20, b);
    if (!(std::fabs(m) < 0x1p-61)) {
      printf("mean error %g of the largest term\n", m);
      return 1;
    }
  }
  printf("OK (%lld of %lld sums left to float64)\n", declined, n);
  return 0;
}
