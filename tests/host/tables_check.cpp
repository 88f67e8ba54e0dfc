// Which pointer tables may serve again (ScratchTables): prints ok, exits 1 on a failure.
#include <cstdio>

#include "acr_tables.h"

int main() {
  acr::ScratchTables t;
  char arena[64];
  int ranks[8];
  bool ok = !t.serve(-2, 0, 0, nullptr, nullptr, 0, 0, 0, 0);
  t.epoch = 3; t.nr = 2; t.pc = 4; t.scr = arena; t.rscr = ranks;
  t.stride = 1024; t.rstride = 16;   // built for 4096 bytes and 64 slots
  ok &= t.serve(3, 2, 4, arena, ranks, 512, 8, 4096, 64);
  ok &= t.serve(3, 2, 4, arena, ranks, 1024, 16, 8192, 128);
  ok &= !t.serve(3, 2, 4, arena, ranks, 512, 8, 4095, 64);    // a smaller arena at the same place
  ok &= !t.serve(3, 2, 4, arena, ranks, 512, 8, 4096, 63);
  ok &= !t.serve(3, 2, 4, arena, ranks, 1025, 8, 8192, 64);   // planes that need more
  ok &= !t.serve(3, 2, 4, arena, ranks, 512, 17, 8192, 128);
  ok &= !t.serve(4, 2, 4, arena, ranks, 512, 8, 4096, 64);
  ok &= !t.serve(3, 2, 3, arena, ranks, 512, 8, 4096, 64);
  ok &= !t.serve(3, 3, 4, arena, ranks, 512, 8, 4096, 64);
  ok &= !t.serve(3, 2, 4, arena + 1, ranks, 512, 8, 4096, 64);
  ok &= !t.serve(3, 2, 4, arena, ranks + 1, 512, 8, 4096, 64);
  std::printf(ok ? "ok\n" : "FAIL\n");
  return ok ? 0 : 1;
}
