// Radial chunks of the streaming tile kernels: host code only.
#pragma once
#include <cstdint>

namespace tn {

constexpr int kSMs = 152;

// Launch time, in layer times, of ncells cell layers in chunks of kc by `columns` tile columns with `resident` CTAs
// per SM.  A CTA sweeps its chunk plus the cell layer below it (recomputed for the carried contributions) and a
// prologue worth about half a layer, and the GPU runs the CTAs in ceil(CTAs / (SMs resident)) waves.
inline double chunk_cost(int64_t columns, int ncells, int resident, int kc) {
  const int64_t ctas = columns * ((ncells + kc - 1) / kc), slots = (int64_t)kSMs * resident;
  return (double)((ctas + slots - 1) / slots) * (kc + 1.5);
}

// Cell layers per radial chunk, at most kmax: the cheapest even split, the longest of equally cheap ones.  Small grids
// get short chunks that fill the SMs (level 4 / 17 layers FP64: 80 CTAs of 2 layers instead of 20 of 8), large ones a
// last wave that is nearly full (level 7 / 129 layers: 16 layers, the best of a sweep as well).  Runs at every launch,
// so it visits each chunk length ceil(ncells / c) once, about 2 sqrt(ncells) of them, and not each c.
inline int radial_chunk(int64_t columns, int ncells, int resident, int kmax) {
  int best = 1;
  double cost = 1e30;
  auto even = [&](int kc) { return (ncells + (ncells + kc - 1) / kc - 1) / ((ncells + kc - 1) / kc); };
  for (int kc = ncells < kmax ? ncells : kmax; kc >= 1; --kc) {
    kc = even(kc);  // as few chunks, evenly long
    const double t = chunk_cost(columns, ncells, resident, kc);
    if (t < cost) cost = t, best = kc;
  }
  return best;
}

}  // namespace tn
