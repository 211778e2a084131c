// CPU check of plan_tc_cols (csrc/host_logic.h), the chunk of the tensor-core inversion.
#include <cstdio>

#include "host_logic.h"

int main() {
  int bad = 0;
  const int sides[] = {33, 64, 96, 128, 160, 256, 320, 416}, frames[] = {1, 2, 7, 22, 32, 128}, widths[] = {1, 2, 19, 64, 256, 1024};
  for (int ny : sides)
    for (int nt : frames)
      for (int nx : widths) {
        const double np = (ny + 31) / 32 * 32, per = 56.0 * np * np, inv = 4.0 * np * np * nx * nt;
        const int c = recon::plan_tc_cols(nx, nt, 152, per, inv);
        const double got = c * nt * per, most = 1.25 * inv > 6e8 ? 1.25 * inv : 6e8;
        bool ok = c >= 1 && c <= nx;
        ok = ok && (c == 1 || got <= most);                             // the stated limit on the scratch
        const double want = 608 * per > 2.56e8 ? 608 * per : 2.56e8;   // and no less than it allows
        ok = ok && (c == nx || got + nt * per > (want < most ? want : most));
        if (!ok) {
          std::printf("FAIL ny=%d nt=%d nx=%d: %d columns, %.0f bytes\n", ny, nt, nx, c, got);
          ++bad;
        }
      }
  std::printf(bad ? "%d FAILED\n" : "OK\n", bad);
  return bad != 0;
}
