// The problems of a batch as its kernels see them (k_batch.cu, k_tile_batch.cu).
#pragma once

#include "fft_tile.cuh"
#include "paro_ctx.h"

namespace paro {

// Per problem (one k-point of one context), device-visible.
struct ProbDev {
  int npw, ncol, nxr, nb, N1, N2, N3, nproj;
  long long off;   // first element of the problem's rows in the batch vectors
  long long soff;  // first element of the problem's stick buffers (nb x N3 x ncol)
  long long dpoff; // first element of the problem's scaled projections (nb x nproj)
  int band0;       // first band of the problem in the flat band list
  int pad;
  FftPlan plan[3];
  const int *col_x, *col_y, *col_off, *g_col, *g_z, *xrows;
  const double* kin;
  const float* kin32;
  const double* vplane;
  const float* vplane32;
  const double2* tw64[3];
  const float2* tw32[3];
  const double2* beta;
  const float2* beta32;
  const double* dvec;
  const int *stick_of, *xrow_c;  // line-FFT passes (hpsi_passes_tile.cuh)
  const fxw* twfx[3];
};

template <typename T> __device__ __forceinline__ const cplx<T>* pd_tw(const ProbDev& p, int a);
template <> __device__ __forceinline__ const double2* pd_tw<double>(const ProbDev& p, int a) { return p.tw64[a]; }
template <> __device__ __forceinline__ const float2* pd_tw<float>(const ProbDev& p, int a) { return p.tw32[a]; }
template <typename T> __device__ __forceinline__ const T* pd_kin(const ProbDev& p);
template <> __device__ __forceinline__ const double* pd_kin<double>(const ProbDev& p) { return p.kin; }
template <> __device__ __forceinline__ const float* pd_kin<float>(const ProbDev& p) { return p.kin32; }
template <typename T> __device__ __forceinline__ const T* pd_v(const ProbDev& p);
template <> __device__ __forceinline__ const double* pd_v<double>(const ProbDev& p) { return p.vplane; }
template <> __device__ __forceinline__ const float* pd_v<float>(const ProbDev& p) { return p.vplane32; }
template <typename T> __device__ __forceinline__ const cplx<T>* pd_beta(const ProbDev& p);
template <> __device__ __forceinline__ const double2* pd_beta<double>(const ProbDev& p) { return p.beta; }
template <> __device__ __forceinline__ const float2* pd_beta<float>(const ProbDev& p) { return p.beta32; }

// Rows of the batch vectors, or, with direct, the caller's own arrays (one per problem, paro_batch_apply_h), whose
// addresses travel in the kernels' parameters: 96 problems are 1.5 KB of the 4 that every kernel may have. Larger
// batches (a mesh of 5 x 5 x 5 k-points) go through the batch's vectors, two device copies a problem.
static const int kBatchDirect = 96;
template <typename T> struct BatchRows {
  const cplx<T>* x;
  cplx<T>* y;
  int direct;
  const cplx<T>* px[kBatchDirect];
  cplx<T>* py[kBatchDirect];
};

// Items of one cubic grid that the line-FFT passes cover
struct BatchGroup {
  int n = 0;           // grid edge
  int nitems = 0;
  int max_ncol = 0, max_nxr = 0;
  int* d_items = nullptr;  // indices into the batch's item list
};

// whether the line-FFT passes cover a problem (k_tile_batch.cu), and H psi of a group's items by them
bool batch_tile_covers(const ProbDev& p, bool f64);
template <typename T>
int batch_tile_apply(Ctx* c, cudaStream_t s, const BatchGroup& g, const ProbDev* probs, const int2* items,
                     const BatchRows<T>& rows, cplx<T>* S, const cplx<T>* DP, const int* active, const double* sigma,
                     int shifted, int phase);

template <>
int batch_tile_apply<float>(Ctx*, cudaStream_t, const BatchGroup&, const ProbDev*, const int2*, const BatchRows<float>&,
                            float2*, const float2*, const int*, const double*, int, int);
template <>
int batch_tile_apply<double>(Ctx*, cudaStream_t, const BatchGroup&, const ProbDev*, const int2*,
                             const BatchRows<double>&, double2*, const double2*, const int*, const double*, int, int);

}  // namespace paro
