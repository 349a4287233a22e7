// One search of a batch or serving kernel.
#pragma once

#include "search.cuh"

namespace {

// The full evaluation, inlined into the kernel: as a call it took 5 to 9 % longer.
template <bool PEN, bool DL, bool RP>
__device__ __forceinline__ void full_search(const KParams& P, const Layout& lay, int kind, int C, int rank) {
  if (kind == SEARCH_TABLES) solve_one<PEN, DL, false, false, RP>(P, lay, C, rank, 1, 0);
  else solve_one<PEN, DL, false, true, RP>(P, lay, C, rank, 1, 0);
}

// The search of one instance of a batch or of a request, on the layout the sizes ask for
// (the same for every CTA of its cluster). table_words: gather tables up to this size do
// without the int16 limits; limit_words: shared memory of the launch. False when no layout
// fits.
template <bool PEN, bool DL>
__device__ __forceinline__ bool search_instance(const KParams& P, int C, int rank, bool compact, int table_words,
                                                int limit_words) {
  const bool half = compact || make_layout(P.M, P.V, P.L, P.nt, false, true).total > table_words;
  Layout lay;
  const int kind = pick_search(P.M, P.V, P.L, P.nt, DL, C, blockDim.x >> 5, P.tenure, compact, half, true,
                              limit_words, &lay);
  if (lay.total > limit_words) return false;
  if (kind == SEARCH_CARRY32) carry_solve<PEN, DL, CTab32>(P, lay, C, rank);
  else if (kind == SEARCH_CARRY16) carry_solve<PEN, DL, CTab16>(P, lay, C, rank);
  else if (!takes_quads(P.M, P.V, C, blockDim.x >> 5)) full_search<PEN, DL, false>(P, lay, kind, C, rank);
  else full_search<PEN, DL, true>(P, lay, kind, C, rank);
  return true;
}

}  // namespace
