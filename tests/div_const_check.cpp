// Host check of div_const (innerq_quantize_prefill.cu): x / d by the rounded reciprocal and one remainder correction is
// the correctly rounded quotient for every mantissa, at the ends and in the middle of the range the quantisers see.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

int main() {
  const float divisors[3] = {3.f, 7.f, 15.f};
  const uint32_t exponents[5] = {32, 100, 127, 128, 254};      // biased; quotients of all of them are normal numbers
  for (float d : divisors)
    for (uint32_t e : exponents)
      for (uint32_t m = 0; m < (1u << 23); ++m) {
        const uint32_t bits = (e << 23) | m;
        float x;
        std::memcpy(&x, &bits, 4);
        const float r = 1.0f / d, q = x * r, q1 = std::fmaf(std::fmaf(-d, q, x), r, q);
        if (q1 != x / d) { std::printf("%a / %g: %a\n", x, d, q1); return 1; }
      }
  std::puts("ok");
  return 0;
}
