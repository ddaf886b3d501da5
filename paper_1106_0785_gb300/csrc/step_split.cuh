// step_split.cuh - the step with one velocity per lane, for small grids (host interface).
#pragma once

#include "kernels.cuh"

namespace mrtlb {

// What lane l = 4 s + k of a node's 16 lanes multiplies with (see
// step_split.cu); field by field, so that the lanes' loads are consecutive.
template <typename R>
struct SplitTable {
  R mom[4][16];    // the lane's moment from the harmonics k of shells 0..3
  R inv[3][16];    // the lane's harmonic of the collision from three moments
  R full[4][16];   // the lane's harmonic from the family's four moments
  R rate[16], mod_a[16], mod_b[16];
  R lw[4][16];
  R wall[4][16];   // per side: the lane's moment of its equilibrium at unit density
  double num[4][16], e64[4][16], inv_den[4];  // per diffuse side (Walls)
};
template <typename R>
void split_table(const Coef<R>& c, const Walls& w, SplitTable<R>* t);

// Whether a grid is small enough for it (the lines are in step_split.cu).
template <typename R>
bool use_split(const Layout& L, int version);
// One step; walls and diffuse ghosts are worked out beside their nodes when
// `refill` (and written to fin too when `keep`), else read from fin.  `t`: the
// context's table on the device.
template <typename R>
void launch_step_split(const R* fin, R* fout, const Layout& L, const Coef<R>& c, const SplitTable<R>* t, bool refill,
                       bool keep, int* err, cudaStream_t st);

}  // namespace mrtlb
