// Host-only driver of the per-grid tile rule of csrc/plan.h for the CPU tests:
// for each grid given on the command line as Nx,Ny,Nz,csize and a list of
// batches, the element count, width and threads of every pass. Compiled with
// g++; it launches nothing.
#include <cstdio>

#include "plan.h"

int main(int argc, char** argv) {
  std::printf("[");
  bool first = true;
  for (int a = 1; a < argc; ++a) {
    int nx = 0, ny = 0, nz = 0, cs = 0;
    if (std::sscanf(argv[a], "%d,%d,%d,%d", &nx, &ny, &nz, &cs) != 4) return 2;
    for (int batch : {1, 3, 16, 64, 1024}) {
      gad::GridTiles t;
      const bool ok = gad::grid_tiles(nx, ny, nz, batch, (size_t)cs, t);
      std::printf("%s{\"grid\": [%d, %d, %d], \"cs\": %d, \"batch\": %d, \"ok\": %d", first ? "" : ", ", nx, ny, nz, cs,
                  batch, ok ? 1 : 0);
      first = false;
      const gad::TileShape* ts[] = {&t.xf, &t.xi, &t.xi_nodots, &t.fl, &t.fl_nodots, &t.y};
      const char* name[] = {"xf", "xi", "xi_nodots", "fl", "fl_nodots", "y"};
      for (int i = 0; i < 6; ++i)
        std::printf(", \"%s\": [%d, %d, %d, %d, %zu]", name[i], ts[i]->E, ts[i]->W, ts[i]->T, ts[i]->ld, ts[i]->smem);
      std::printf("}");
    }
  }
  std::printf("]\n");
  return 0;
}
