// CPU check of fft_stages (csrc/host_logic.h), the radices of every transform but the 16-bit prologue's:
// for each length the library takes, in the 12 stages of its plans (fft.cuh: kFftMaxStages).
#include <cstdio>

#include "host_logic.h"

int main() {
  int bad = 0;
  for (int n = 1; n <= 1024; ++n) {
    int radix[12];
    const int ns = recon::fft_stages(n, radix, 12);
    long long prod = 1;
    int twos = 0;
    bool ok = true, powers = false;   // a power of two has come
    for (int s = 0; s < ns; ++s) {
      const int r = radix[s];
      prod *= r;
      if (r == 2 || r == 4 || r == 8) {
        powers = true;
        twos += r == 2;
      } else {
        ok = ok && !powers && r >= 3;   // odd primes first, where no twiddles are due
        for (int d = 2; d < r; ++d) ok = ok && r % d;
      }
    }
    ok = ok && prod == n && twos <= 1 && (n > 1 || ns == 0);
    if (!ok) {
      std::printf("FAIL n=%d: %d stages, product %lld, %d radix 2\n", n, ns, prod, twos);
      ++bad;
    }
  }
  std::printf(bad ? "%d FAILED\n" : "OK\n", bad);
  return bad != 0;
}
