// FP64 passes (fixed-point line FFTs): instantiation of hpsi_passes_tile.cuh.
#include <algorithm>

#include "hpsi_passes_tile.cuh"

namespace paro {

using Grids = TileGrids<NumF64, 27, 32, 36, 48, 54, 64, 72, 81, 96, 108>;

template <>
int passes_tile<double>(Ctx* c, const Basis& B, int nb, const cplx<double>* psi, cplx<double>* S, cplx<double>* hpsi, double shift,
                      const int* active, const double* vplane, bool acc, bool* used) {
  return Grids::passes(c, B, nb, psi, S, hpsi, shift, active, vplane, acc, used);
}
template <>
int sticks_tile<double>(Ctx* c, const Basis& B, int nb, const cplx<double>* psi, cplx<double>* S, bool* used) {
  return Grids::sticks(c, B, nb, psi, S, used);
}
template <>
int density_tile<double>(Ctx* c, const Basis& B, const cplx<double>* S, int nbands, int ngrp, int gsize, double wfac,
                       const double* wsq, double* part, bool* used) {
  return Grids::density(c, B, S, nbands, ngrp, gsize, wfac, wsq, part, used);
}

}  // namespace paro
