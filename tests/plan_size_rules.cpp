// Host-only driver of the size rules of csrc/plan.h for the CPU tests: prints
// the fused radices of each length given on the command line and, for a list of
// grids, the tiles choose_pass takes. Compiled with g++; it launches nothing.
#include <cstdio>
#include <cstdlib>

#include "plan.h"

int main(int argc, char** argv) {
  std::printf("{\"fused\": {");
  for (int a = 1; a < argc; ++a) {
    const int L = std::atoi(argv[a]);
    int rad[gad::kMaxStages], rev[gad::kMaxStages];
    const int n = gad::plan_radices(L, 13, false, rad);
    gad::plan_radices(L, 13, true, rev);
    std::printf("%s\"%d\": {\"ok\": %d, \"key\": %d, \"key64\": %d, \"r\": [", a > 1 ? ", " : "", L,
                gad::fused_length(L) ? 1 : 0, gad::plan_E(L, 12, 8), gad::plan_E(L, 12, 16));
    for (int i = 0; i < n; ++i) std::printf("%s%d", i ? ", " : "", rad[i]);
    std::printf("], \"rev\": [");
    for (int i = 0; i < n; ++i) std::printf("%s%d", i ? ", " : "", rev[i]);
    std::printf("]}");
  }
  std::printf("}, \"tiles\": [");
  bool first = true;
  const int lens[] = {8, 18, 32, 48, 64, 128, 144, 256, 512, 768, 1024, 1152, 2048, 2304};
  const long long rows[] = {8, 128, 1024, 65536};
  for (int L : lens)
    for (long long nseq : rows)
      for (size_t cs : {8, 16})
        for (int t = 0; t < 2; ++t)
          for (int want : {64, 256}) {
            gad::TileShape ts;
            const int div = t ? gad::pow2_part(nseq) : 0;
            const bool ok = gad::choose_pass(L, L + 1, div, nseq, t != 0, cs, ts, want);
            int rad[gad::kMaxStages];
            const int n = ok ? gad::plan_radices(L, gad::plan_E(L, ts.E, cs), false, rad) : 0;
            std::printf("%s[%d, %lld, %d, %d, %d, %d, %d, %d, %d, %d, %zu, %d]", first ? "" : ", ", L, nseq, (int)cs, t,
                        want, ok ? 1 : 0, ts.E, ts.W, ts.T, ts.ld, ts.smem, n);
            first = false;
          }
  std::printf("]}\n");
  return 0;
}
