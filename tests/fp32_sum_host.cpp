// Host check of csrc/fp32_sum.cuh against exact integer sums: values m 2^(x - 40) with 24-bit m and x spread over 0..span,
// in runs of up to 256, as they are and with the largest ones cancelled later.  Prints, over all runs, the worst error of
// Fp32Sum relative to the larger of 2^-53 |sum| and 2^-66 max |value|, and how often it lies further off than the FP64 sum.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "fp32_sum.cuh"

static uint64_t state = 1708;
static uint64_t next() {  // SplitMix64
  uint64_t z = (state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

int main() {
  double worst = 0;
  long further = 0;
  const int spans[] = {0, 4, 12, 24, 38}, counts[] = {1, 2, 3, 8, 31, 32, 256};
  for (int span : spans)
    for (int n : counts)
      for (int run = 0; run < 400; ++run) {
        std::vector<int64_t> v;
        for (int i = 0; i < n; ++i) {
          const int64_t m = (int64_t)(next() >> 40) - (1 << 23);
          v.push_back(m * ((int64_t)1 << (span ? next() % (span + 1) : 0)));
        }
        if (run & 1)  // cancellation: the larger half again with the other sign
          for (int i = 0; i < n; ++i)
            if (std::llabs(v[i]) > ((int64_t)1 << (22 + span / 2))) v.push_back(-v[i]);
        __int128 exact = 0;
        cisor::Fp32Sum part[8], a;  // as the warps of a CTA sum: eight sums in turn, added in order
        double d = 0, big = 0;
        int i = 0;
        for (int64_t x : v) {
          const float f = std::ldexp((float)x, -40);  // exact: 24 significant bits
          exact += x;
          part[i++ % 8].add(f);
          d += f;
          big = std::fmax(big, std::fabs(f));
        }
        for (const auto& p : part) a.add(p);
        // errors in units of 2^-40, exactly: the sums are multiples of it below 2^80, a double's part of them exact
        const auto err = [&](double s) {
          const double hi = std::ldexp(s, 40);
          return std::fabs((double)((__int128)hi - exact) + (hi - (double)(__int128)hi)) * std::ldexp(1.0, -40);
        };
        const double ea = err(a.value()), ed = err(d), ref = std::fabs((double)exact) * std::ldexp(1.0, -40);
        worst = std::fmax(worst, ea / std::fmax(std::fmax(ref * std::ldexp(1.0, -53), big * std::ldexp(1.0, -66)), 1e-300));
        if (ea > ed) ++further;
      }
  // range: FP32 overflows, a value that is not finite stays so
  cisor::Fp32Sum o;
  for (float f : {3e38f, 3e38f, -3e38f}) o.add(f);
  std::printf("%.3f %ld %d\n", worst, further, (int)std::isfinite(o.value()));
  return 0;
}
