// What a plan run's pointer tables were built for, and whether they serve the next run.
// (Host logic without CUDA; the engine keeps the tables' own copies beside it.)
#pragma once
#include <cstddef>
#include <cstdint>

namespace acr {

struct ScratchTables {
  int64_t epoch = -1;              // of the staging ring that holds them; -1: none
  int nr = 0, pc = 0;              // operand roles, planes
  const void *scr = nullptr, *rscr = nullptr;
  size_t stride = 0, rstride = 0;  // scratch bytes and rank slots per plane

  // Do they serve a run of the same shape whose planes need `bytes` and `ranks` of scratch,
  // out of an arena of `have` bytes and `have_r` slots at the same addresses?  (The arena
  // may have been given back and taken again, smaller, at the same place: the planes are
  // spread over all of the one that the tables were built for.)
  bool serve(int64_t now, int roles, int planes, const void* base, const void* rbase,
             size_t bytes, size_t ranks, size_t have, size_t have_r) const {
    return epoch == now && nr == roles && pc == planes && scr == base && rscr == rbase &&
           stride >= bytes && rstride >= ranks && stride * (size_t)pc <= have &&
           rstride * (size_t)pc <= have_r;
  }
};

}  // namespace acr
