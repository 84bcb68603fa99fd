// Host check of div_const (csrc/innerq_div_const.h): the correctly rounded quotient for every mantissa of the three
// divisors that need one, at the ends and in the middle of the range the quantisers see, for 0, infinity and NaN, and
// x itself for the divisor 1.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "innerq_div_const.h"

namespace {

template <int DEN> bool check() {
  const uint32_t exponents[5] = {32, 100, 127, 128, 254};      // biased; quotients of all of them are normal numbers
  for (uint32_t e : exponents)
    for (uint32_t m = 0; m < (1u << 23); ++m) {
      const uint32_t bits = (e << 23) | m;
      float x;
      std::memcpy(&x, &bits, 4);
      if (iq::div_const<DEN>(x) != x / (float)DEN) { std::printf("%a / %d: %a\n", x, DEN, iq::div_const<DEN>(x)); return false; }
      if (DEN == 1) break;
    }
  return iq::div_const<DEN>(0.f) == 0.f && iq::div_const<DEN>(INFINITY) == INFINITY && std::isnan(iq::div_const<DEN>(NAN));
}

}  // namespace

int main() {
  const bool ok = check<1>() && check<3>() && check<7>() && check<15>();
  std::puts(ok ? "ok" : "failed");
  return !ok;
}
