// Test helper: the host forms of the digit-splitting arithmetic (kkt_oz.cuh).
// Built by the tests with the host compiler; not part of the library.
#include "../../paper_2511_00946_gb300/csrc/kkt_oz.cuh"

extern "C" {
// exponent of a row of n elements, and its digits (u[n])
int oz_row(const double* z, int n, unsigned long long* u) {
  int em = 0;
  for (int k = 0; k < n; ++k) em = em > kkt::oz::mag(kkt::oz::dbits(z[k])) ? em : kkt::oz::mag(kkt::oz::dbits(z[k]));
  const int f = kkt::oz::row_exp(em);
  if (f != kkt::oz::kFp64Row)
    for (int k = 0; k < n; ++k) u[k] = kkt::oz::encode(kkt::oz::dbits(z[k]), f);
  return f;
}
double oz_value(unsigned long long u, int f) { return kkt::oz::value(u, f); }
double oz_to_double(long long u, int e) { return kkt::oz::to_double(u, e); }
// the digit sums p[7] of two rows of digits, and their product's value
double oz_dot(const unsigned long long* a, int fa, const unsigned long long* b, int fb, int n, long long* p) {
  int q[kkt::oz::kDig];
  for (int g = 0; g < kkt::oz::kDig; ++g) p[g] = 0;
  for (int k = 0; k < n; ++k)
    for (int i = 0; i < kkt::oz::kDig; ++i)
      for (int j = kkt::oz::kLow - i; j < kkt::oz::kDig; ++j)
        p[i + j - kkt::oz::kLow] += ((long long)(a[k] >> (9 * i) & 511) - 256) * ((long long)(b[k] >> (9 * j) & 511) - 256);
  for (int g = 0; g < kkt::oz::kDig; ++g) q[g] = (int)p[g];
  return kkt::oz::to_double(kkt::oz::combine(q), fa + fb + kkt::oz::kUnit);
}
}
