// H psi of a batch's items on one cubic grid by the line-FFT passes of hpsi_passes_tile.cuh: the bodies of the
// per-context kernels over (stick group or plane, item), the item's problem looked up on the device. A mesh of 27
// k-points of the 8-atom cell (540 orbitals on 32^3) spent 385 of 500 us in planes whose FFT stages met at block
// barriers; these planes meet twice.
#include <algorithm>

#include "batch_prob.cuh"
#include "hpsi_passes_tile.cuh"

namespace paro {

template <typename NT> struct ProbTables;
template <> struct ProbTables<NumF32> {
  using T = float;
  static __device__ __forceinline__ const float2* tw(const ProbDev& p, int a) { return p.tw32[a]; }
};
template <> struct ProbTables<NumF64> {
  using T = double;
  static __device__ __forceinline__ const fxw* tw(const ProbDev& p, int a) { return p.twfx[a]; }
};

template <typename NT, int N>
__global__ void __launch_bounds__(256) k_batch_zinv(const int* __restrict__ gitems, const ProbDev* __restrict__ probs,
                                                    const int2* __restrict__ items,
                                                    const __grid_constant__ BatchRows<typename NT::R> rows,
                                                    typename NT::S* __restrict__ S, const int* __restrict__ active,
                                                    int CB) {
  using PT = ProbTables<NT>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 it = items[gitems[blockIdx.y]];
  const ProbDev& P = probs[it.x];
  const int c0 = blockIdx.x * CB;
  if (c0 >= P.ncol || (active != nullptr && active[P.band0 + it.y] == 0)) return;
  const typename NT::S* x = (rows.direct ? rows.px[it.x] : rows.x + P.off) + (size_t)it.y * P.npw;
  zinv_sticks<NT, N>(smem_raw, x, S + P.soff + (size_t)it.y * N * P.ncol, P.col_off, P.g_col, P.g_z, P.ncol,
                     PT::tw(P, 2), c0, CB);
}

template <typename NT, int N>
__global__ void __launch_bounds__(32 * TileWarps<N>::value, TileMinBlocks<NT, N>::value)
    k_batch_plane(const int* __restrict__ gitems, const ProbDev* __restrict__ probs, const int2* __restrict__ items,
                  typename NT::S* __restrict__ S, const int* __restrict__ active) {
  using PT = ProbTables<NT>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 it = items[gitems[blockIdx.y]];
  const ProbDev& P = probs[it.x];
  if (active != nullptr && active[P.band0 + it.y] == 0) return;
  plane_sticks<NT, N>(smem_raw, S + P.soff + ((size_t)it.y * N + blockIdx.x) * P.ncol, P.stick_of, P.xrow_c, P.nxr,
                      PT::tw(P, 0), PT::tw(P, 1), pd_v<typename NT::R>(P) + (size_t)blockIdx.x * N * N);
}

template <typename NT, int N>
__global__ void __launch_bounds__(256) k_batch_zfwd(const int* __restrict__ gitems, const ProbDev* __restrict__ probs,
                                                    const int2* __restrict__ items,
                                                    const __grid_constant__ BatchRows<typename NT::R> rows,
                                                    const typename NT::S* __restrict__ S,
                                                    const typename NT::S* __restrict__ DP,
                                                    const int* __restrict__ active, const double* __restrict__ sigma,
                                                    int shifted, int CB) {
  using PT = ProbTables<NT>;
  using R = typename NT::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int2 it = items[gitems[blockIdx.y]];
  const ProbDev& P = probs[it.x];
  const int c0 = blockIdx.x * CB;
  if (c0 >= P.ncol || (active != nullptr && active[P.band0 + it.y] == 0)) return;
  const size_t row = (size_t)it.y * P.npw;
  const typename NT::S* x = (rows.direct ? rows.px[it.x] : rows.x + P.off) + row;
  typename NT::S* y = (rows.direct ? rows.py[it.x] : rows.y + P.off) + row;
  zfwd_sticks<NT, N, false, true>(smem_raw, S + P.soff + (size_t)it.y * N * P.ncol, x, y, pd_kin<R>(P),
                                  shifted ? (R)sigma[it.x] : (R)0, P.col_off, P.g_col, P.g_z, P.ncol, PT::tw(P, 2), c0,
                                  CB, P.nproj, P.npw, pd_beta<R>(P), DP + P.dpoff + (size_t)it.y * P.nproj);
}

template <typename NT, int N>
static int batch_apply_n(Ctx* c, cudaStream_t s, const BatchGroup& g, const ProbDev* probs, const int2* items,
                         const BatchRows<typename NT::R>& rows, typename NT::S* S, const typename NT::S* DP,
                         const int* active, const double* sigma, int shifted, int phase) {
  static int done[3][64];
  int st;
  if ((st = tile_attr(c, k_batch_zinv<NT, N>, done[0])) || (st = tile_attr(c, k_batch_plane<NT, N>, done[1])) ||
      (st = tile_attr(c, k_batch_zfwd<NT, N>, done[2])))
    return st;
  const TileZ z = tile_z<NT, N>(g.max_ncol, g.nitems);
  const dim3 gz((g.max_ncol + z.cb - 1) / z.cb, g.nitems);
  constexpr int NW = TileWarps<N>::value;
  if (phase == 1)
    k_batch_zinv<NT, N><<<gz, z.threads, z.smem, s>>>(g.d_items, probs, items, rows, S, active, z.cb);
  else if (phase == 2)
    k_batch_plane<NT, N><<<dim3(N, g.nitems), 32 * NW, tile_plane_smem<NT, N>(g.max_nxr, NW), s>>>(g.d_items, probs, items,
                                                                                                  S, active);
  else
    k_batch_zfwd<NT, N><<<gz, z.threads, z.smem, s>>>(g.d_items, probs, items, rows, S, DP, active, sigma, shifted, z.cb);
  PARO_CU(c, cudaGetLastError());
  return PARO_OK;
}

template <typename NT, int... Ns> struct BatchGrids {
  static bool covers(const ProbDev& p) {
    return ((p.N1 == Ns && p.N2 == Ns && p.N3 == Ns &&
             tile_plane_smem<NT, Ns>(p.nxr, TileWarps<Ns>::value) <= kTileSmemMax) || ...);
  }
  template <typename... A> static int apply(int n, A&&... a) {
    int st = PARO_ERR_ARG;
    ((n == Ns ? (st = batch_apply_n<NT, Ns>(a...), 0) : 0), ...);
    return st;
  }
};
// Up to 72 points: batches are of small cells, and every grid more is three kernels of each type to compile; larger
// grids keep the shared-memory passes of k_batch.cu, untimed against these.
using Batch32 = BatchGrids<NumF32, 27, 32, 36, 48, 54, 64, 72>;
using Batch64 = BatchGrids<NumF64, 27, 32, 36, 48, 54, 64, 72>;

bool batch_tile_covers(const ProbDev& p, bool f64) { return f64 ? Batch64::covers(p) : Batch32::covers(p); }

template <>
int batch_tile_apply<float>(Ctx* c, cudaStream_t s, const BatchGroup& g, const ProbDev* probs, const int2* items,
                            const BatchRows<float>& rows, float2* S, const float2* DP, const int* active,
                            const double* sigma, int shifted, int phase) {
  return Batch32::apply(g.n, c, s, g, probs, items, rows, S, DP, active, sigma, shifted, phase);
}
template <>
int batch_tile_apply<double>(Ctx* c, cudaStream_t s, const BatchGroup& g, const ProbDev* probs, const int2* items,
                             const BatchRows<double>& rows, double2* S, const double2* DP, const int* active,
                             const double* sigma, int shifted, int phase) {
  return Batch64::apply(g.n, c, s, g, probs, items, rows, S, DP, active, sigma, shifted, phase);
}

}  // namespace paro
