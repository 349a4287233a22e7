// One search of a batch or serving kernel.
#pragma once

#include "search.cuh"

namespace {

// The search of one instance of a batch or of a request, on the layout the sizes ask for
// (the same for every CTA of its cluster). table_words: gather tables up to this size do
// without the int16 limits; limit_words: shared memory of the launch. False when no layout
// fits.
template <bool PEN, bool DL>
__device__ __forceinline__ bool search_instance(const KParams& P, int C, int rank, bool compact, int table_words,
                                                int limit_words) {
  const bool half = compact || make_layout(P.M, P.V, P.L, P.nt, false).total + batch_reserve(P.M, P.V) > table_words;
  Layout lay;
  const int kind = pick_search(P.M, P.V, P.L, P.nt, DL, C, blockDim.x >> 5, P.tenure, compact, half, limit_words, &lay);
  if (lay.total > limit_words) return false;
  if (kind == SEARCH_CARRY32) carry_solve<PEN, DL, CTab32>(P, lay, C, rank);
  else if (kind == SEARCH_CARRY16) carry_solve<PEN, DL, CTab16>(P, lay, C, rank);
  else if (kind == SEARCH_TABLES) solve_full<PEN, DL, false>(P, lay, C, rank, 1, 0);
  else solve_full<PEN, DL, true>(P, lay, C, rank, 1, 0);
  return true;
}

}  // namespace
