// FP32 passes on the cubic grids without a register form: instantiation of hpsi_passes_tile.cuh.
#include <algorithm>

#include "hpsi_passes_tile.cuh"

namespace paro {

using Grids = TileGrids<NumF32, 27, 54, 64, 81, 96, 108>;

template <>
int passes_tile<float>(Ctx* c, const Basis& B, int nb, const cplx<float>* psi, cplx<float>* S, cplx<float>* hpsi, double shift,
                      const int* active, const float* vplane, bool acc, bool* used) {
  return Grids::passes(c, B, nb, psi, S, hpsi, shift, active, vplane, acc, used);
}
template <>
int sticks_tile<float>(Ctx* c, const Basis& B, int nb, const cplx<float>* psi, cplx<float>* S, bool* used) {
  return Grids::sticks(c, B, nb, psi, S, used);
}
template <>
int density_tile<float>(Ctx* c, const Basis& B, const cplx<float>* S, int nbands, int ngrp, int gsize, double wfac,
                       const double* wsq, double* part, bool* used) {
  return Grids::density(c, B, S, nbands, ngrp, gsize, wfac, wsq, part, used);
}

}  // namespace paro
