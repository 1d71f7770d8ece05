// The three H psi passes and the density planes with the line FFTs of fft_tile.cuh, for cubic grids: FP64
// data (fixed-point butterflies) on every listed grid outside the ParO iteration, FP32 data on the grids without a register form in
// hpsi_passes_reg.cuh. The passes and their data layout are those of hpsi_passes_reg.cuh.
#pragma once

#include "fft_tile.cuh"
#include "paro_ctx.h"

namespace paro {

// warps of a plane CTA: one to three rounds of the N lines along x; twelve on the grids whose plane leaves room for
// one CTA an SM
template <int N> struct TileWarps {
  static constexpr int kRounds = (N + TileLine<N>::G - 1) / TileLine<N>::G;
  static constexpr int value = N >= 96 ? 12 : kRounds <= 8 ? kRounds : kRounds <= 16 ? (kRounds + 1) / 2 : (kRounds + 2) / 3;
};
// Resident plane CTAs the fixed-point kernels are compiled for (a register cap of 65536 / (CTAs x threads)), each
// measured: uncapped, 72 points took 211 registers, eight warps an SM and 3.30 ms for 144 orbitals, with two CTAs
// 1.97 ms; 64 points 1.43 -> 0.83 ms with three, 36 points 102 -> 49 us (23 orbitals), 32 points 38 -> 27 us (20 orbitals),
// 81 points 2.12 -> 1.70 ms (60 orbitals).
template <int N> struct TileCtas { static constexpr int value = 1; };
template <> struct TileCtas<27> { static constexpr int value = 5; };
template <> struct TileCtas<32> { static constexpr int value = 5; };
template <> struct TileCtas<36> { static constexpr int value = 3; };
template <> struct TileCtas<48> { static constexpr int value = 2; };
template <> struct TileCtas<54> { static constexpr int value = 2; };
template <> struct TileCtas<64> { static constexpr int value = 3; };
template <> struct TileCtas<72> { static constexpr int value = 2; };
template <> struct TileCtas<81> { static constexpr int value = 2; };
template <typename NT, int N> struct TileMinBlocks {
  // FP32: 32 warps an SM (64 registers): 81 points 462 -> 322 us (100 orbitals), 54 points 186 -> 151 us (144), a mesh of
  // 27 problems on 32 points 181 -> 157 us; 24 and 40 warps were within a tenth of it
  static constexpr int kF32 = 32 / TileWarps<N>::value;
  static constexpr int value = NT::kFixed ? TileCtas<N>::value : kF32 < 1 ? 1 : kF32;
};
template <int N> struct TileStride { static constexpr int value = N | 1; };

// lane -> line of the warp's group and lane of the line; lanes beyond the last whole line idle
template <int N> struct TileLane {
  int grp, p, base;
  bool ok;
  __device__ __forceinline__ TileLane(int lane) {
    using L = TileLine<N>;
    ok = lane < L::G * L::P;
    grp = ok ? lane / L::P : L::G - 1;
    p = lane % L::P;
    base = grp * L::P;
  }
};

// sticks c0 .. c0 + CB - 1 of one band: scatter, inverse transform along z, into the band's stick buffer Sb
template <typename NT, int N>
__device__ __forceinline__ void zinv_sticks(unsigned char* smem_raw, const typename NT::S* __restrict__ pp,
                                            typename NT::S* __restrict__ Sb, const int* __restrict__ col_off,
                                            const int* __restrict__ g_col, const int* __restrict__ g_z, int ncol,
                                            const typename NT::W* __restrict__ twz, int c0, int CB) {
  using L = TileLine<N>;
  using ST = typename NT::S;
  using C = typename NT::C;
  constexpr int LS = TileStride<N>::value;
  C* tiles = reinterpret_cast<C*>(smem_raw);
  ST* line = reinterpret_cast<ST*>(tiles + (blockDim.x >> 5) * L::WTILE);
  const int ncb = min(CB, ncol - c0);
  ST zero;
  zero.x = zero.y = 0;
  for (int i = threadIdx.x; i < ncb * LS; i += blockDim.x) line[i] = zero;
  __syncthreads();
  const int g0 = col_off[c0], g1 = col_off[c0 + ncb];
  for (int g = g0 + threadIdx.x; g < g1; g += blockDim.x) line[(g_col[g] - c0) * LS + g_z[g]] = pp[g];
  __syncthreads();
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const TileLane<N> t(threadIdx.x & 31);
  C* tile = tiles + warp * L::WTILE + t.grp * L::TILE;
  for (int l0 = warp * L::G; l0 < ncb; l0 += nw * L::G) {
    const int l = l0 + t.grp;
    const bool ok = t.ok && l < ncb;
    ST* ln = line + (ok ? l : 0) * LS;
    ST raw[L::Q];
#pragma unroll
    for (int q = 0; q < L::Q; ++q) raw[q] = ok ? ln[L::P * q + t.p] : zero;
    C v[L::V];
    const FxScale sc = tile_load<NT, N>(raw, v, t.base);
    tile_inv<NT, N>(v, t.p, twz, tile, t.ok);
    if (ok)
#pragma unroll
      for (int i = 0; i < L::V; ++i) {
        const int k = tile_index<N>(t.p, i);
        if (k >= 0) ln[k] = tile_out<NT>(v[i], sc);
      }
  }
  __syncthreads();
  const int sh = 31 - __clz(CB);  // CB is a power of two
  for (int i = threadIdx.x; i < N << sh; i += blockDim.x) {
    const int z = i >> sh, cc = i & (CB - 1);
    if (cc < ncb) Sb[(size_t)z * ncol + c0 + cc] = line[cc * LS + z];
  }
}

template <typename NT, int N>
__global__ void __launch_bounds__(256) k_zinv_tile(const typename NT::S* __restrict__ psi, int ldpsi,
                                                   typename NT::S* __restrict__ S, const int* __restrict__ col_off,
                                                   const int* __restrict__ g_col, const int* __restrict__ g_z,
                                                   int ncol, const typename NT::W* __restrict__ twz,
                                                   const int* __restrict__ active, int CB) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int b = blockIdx.y;
  if (active != nullptr && active[b] == 0) return;
  zinv_sticks<NT, N>(smem_raw, psi + (size_t)b * ldpsi, S + (size_t)b * N * ncol, col_off, g_col, g_z, ncol, twz,
                     blockIdx.x * CB, CB);
}

// inverse along y of the plane's stick rows, from the stick buffer into the compact plane
template <typename NT, int N>
__device__ __forceinline__ void tile_rows_inv(const typename NT::S* Sz, const int* __restrict__ stick_of, int nxr,
                                              const typename NT::W* __restrict__ twy, typename NT::C* tiles,
                                              typename NT::S* Pl) {
  using L = TileLine<N>;
  using ST = typename NT::S;
  using C = typename NT::C;
  constexpr int LS = TileStride<N>::value;
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const TileLane<N> t(threadIdx.x & 31);
  C* tile = tiles + warp * L::WTILE + t.grp * L::TILE;
  ST zero;
  zero.x = zero.y = 0;
  for (int r0 = warp * L::G; r0 < nxr; r0 += nw * L::G) {
    const int r = r0 + t.grp;
    const bool ok = t.ok && r < nxr;
    const int* so = stick_of + (size_t)(ok ? r : 0) * N;
    ST raw[L::Q];
#pragma unroll
    for (int q = 0; q < L::Q; ++q) {
      const int cs = ok ? so[L::P * q + t.p] : -1;
      raw[q] = cs >= 0 ? Sz[cs] : zero;
    }
    C v[L::V];
    const FxScale sc = tile_load<NT, N>(raw, v, t.base);
    tile_inv<NT, N>(v, t.p, twy, tile, t.ok);
    if (ok) {
      ST* row = Pl + r * LS;
#pragma unroll
      for (int i = 0; i < L::V; ++i) {
        const int k = tile_index<N>(t.p, i);
        if (k >= 0) row[k] = tile_out<NT>(v[i], sc);
      }
    }
  }
}

// v *= V over a line in the transformed layout (V at Vc[index * N])
template <typename NT, int N>
__device__ __forceinline__ void tile_times_v(typename NT::C* v, const typename NT::R* __restrict__ Vc, bool ok, int p,
                                             int base, FxScale& sc) {
  using L = TileLine<N>;
  if constexpr (NT::kFixed) {
    // the potential is read twice, for its exponent and for the product, rather than held beside the line
    int key = 0;
#pragma unroll
    for (int i = 0; i < L::V; ++i) {
      const int k = tile_index<N>(p, i);
      if (ok && k >= 0) key = max(key, __double2hiint(Vc[k * N]) & 0x7fffffff);
    }
    key = tile_max<L::P>(key, base);
    const int ex = key >> 20, e = max(ex, 1) - 1022;
    sc.nan = sc.nan || ex == 0x7ff;
    tile_normalise<NT, N, 61>(v, p, sc, base);
#pragma unroll
    for (int i = 0; i < L::V; ++i) {
      const int k = tile_index<N>(p, i);
      const FxSplit w = fx_cut(ok && k >= 0 ? fx_from<62>(Vc[k * N], e) : 0);
      v[i] = fxc{fx_mul(fx_cut(v[i].x), w), fx_mul(fx_cut(v[i].y), w)};
    }
    sc.k += e;
    tile_normalise<NT, N, 62 - L::GROW>(v, p, sc, base);
  } else {
#pragma unroll
    for (int i = 0; i < L::V; ++i) {
      const int k = tile_index<N>(p, i);
      v[i] = cscale(v[i], ok && k >= 0 ? Vc[k * N] : 0.f);
    }
  }
}

// one plane of one band: sticks Sz in and out, V its potential plane
template <typename NT, int N>
__device__ __forceinline__ void plane_sticks(unsigned char* smem_raw, typename NT::S* __restrict__ Sz,
                                             const int* __restrict__ stick_of, const int* __restrict__ xrow_c, int nxr,
                                             const typename NT::W* __restrict__ twx,
                                             const typename NT::W* __restrict__ twy,
                                             const typename NT::R* __restrict__ V) {
  using L = TileLine<N>;
  using ST = typename NT::S;
  using C = typename NT::C;
  constexpr int LS = TileStride<N>::value;
  C* tiles = reinterpret_cast<C*>(smem_raw);
  ST* Pl = reinterpret_cast<ST*>(tiles + (blockDim.x >> 5) * L::WTILE);
  int* roff = reinterpret_cast<int*>(Pl + (size_t)nxr * LS);
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const int r = xrow_c[i];
    roff[i] = r >= 0 ? r * LS : -1;
  }
  tile_rows_inv<NT, N>(Sz, stick_of, nxr, twy, tiles, Pl);
  __syncthreads();
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const TileLane<N> t(threadIdx.x & 31);
  C* tile = tiles + warp * L::WTILE + t.grp * L::TILE;
  ST zero;
  zero.x = zero.y = 0;
  for (int c0 = warp * L::G; c0 < N; c0 += nw * L::G) {  // along x: inverse, times V / N_grid, forward
    const int y = c0 + t.grp;
    const bool ok = t.ok && y < N;
    ST raw[L::Q];
#pragma unroll
    for (int q = 0; q < L::Q; ++q) {
      const int o = roff[L::P * q + t.p];
      raw[q] = ok && o >= 0 ? Pl[o + y] : zero;
    }
    C v[L::V];
    FxScale sc = tile_load<NT, N>(raw, v, t.base);
    tile_inv<NT, N>(v, t.p, twx, tile, t.ok);
    tile_times_v<NT, N>(v, V + (ok ? y : 0), ok, t.p, t.base, sc);
    tile_fwd<NT, N>(v, t.p, twx, tile, t.ok);
#pragma unroll
    for (int q = 0; q < L::Q; ++q) {
      const int o = roff[L::P * q + t.p];
      if (ok && o >= 0) Pl[o + y] = tile_out<NT>(v[q], sc);
    }
  }
  __syncthreads();
  for (int r0 = warp * L::G; r0 < nxr; r0 += nw * L::G) {  // forward along y, back into the stick buffer
    const int r = r0 + t.grp;
    const bool ok = t.ok && r < nxr;
    const ST* row = Pl + (ok ? r : 0) * LS;
    C v[L::V];
    FxScale sc{0, false};
    if constexpr (NT::kFixed) {  // the line's exponent over the transformed layout
      ST raw[L::V];
      int key = 0;
#pragma unroll
      for (int i = 0; i < L::V; ++i) {
        const int k = tile_index<N>(t.p, i);
        raw[i] = ok && k >= 0 ? row[k] : zero;
        key = max(key, fx_key(raw[i]));
      }
      key = tile_max<L::P>(key, t.base);
      const int ex = key >> 20, e = max(ex, 1) - 1022;
      sc.nan = ex == 0x7ff;
      sc.k = e - (62 - L::GROW);
#pragma unroll
      for (int i = 0; i < L::V; ++i)
        v[i] = fxc{fx_from<62 - L::GROW>(raw[i].x, e), fx_from<62 - L::GROW>(raw[i].y, e)};
    } else {
#pragma unroll
      for (int i = 0; i < L::V; ++i) {
        const int k = tile_index<N>(t.p, i);
        v[i] = ok && k >= 0 ? row[k] : zero;
      }
    }
    tile_fwd<NT, N>(v, t.p, twy, tile, t.ok);
    if (ok) {
      const int* so = stick_of + (size_t)r * N;
#pragma unroll
      for (int q = 0; q < L::Q; ++q) {
        const int cs = so[L::P * q + t.p];
        if (cs >= 0) Sz[cs] = tile_out<NT>(v[q], sc);
      }
    }
  }
}

template <typename NT, int N>
__global__ void __launch_bounds__(32 * TileWarps<N>::value, TileMinBlocks<NT, N>::value)
    k_plane_tile(typename NT::S* __restrict__ S, int ncol, const int* __restrict__ stick_of,
                 const int* __restrict__ xrow_c, int nxr, const typename NT::W* __restrict__ twx,
                 const typename NT::W* __restrict__ twy, const typename NT::R* __restrict__ vplane,
                 const int* __restrict__ active) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int z = blockIdx.x, b = blockIdx.y;
  if (active != nullptr && active[b] == 0) return;
  plane_sticks<NT, N>(smem_raw, S + ((size_t)b * N + z) * ncol, stick_of, xrow_c, nxr, twx, twy,
                      vplane + (size_t)z * N * N);
}

// sticks c0 .. of one band: forward transform along z, gather, kinetic term and shift; ACC: h += the transformed
// potential term alone; KB: the projector term sum_j beta_j(G) dp_j as well (batches)
template <typename NT, int N, bool ACC, bool KB>
__device__ __forceinline__ void zfwd_sticks(unsigned char* smem_raw, const typename NT::S* __restrict__ Sb,
                                            const typename NT::S* pp, typename NT::S* h,
                                            const typename NT::R* __restrict__ kin, typename NT::R shift,
                                            const int* __restrict__ col_off, const int* __restrict__ g_col,
                                            const int* __restrict__ g_z, int ncol,
                                            const typename NT::W* __restrict__ twz, int c0, int CB, int np = 0, int npw = 0,
                                            const typename NT::S* __restrict__ beta = nullptr,
                                            const typename NT::S* __restrict__ dp = nullptr) {
  using L = TileLine<N>;
  using ST = typename NT::S;
  using C = typename NT::C;
  constexpr int LS = TileStride<N>::value;
  C* tiles = reinterpret_cast<C*>(smem_raw);
  ST* line = reinterpret_cast<ST*>(tiles + (blockDim.x >> 5) * L::WTILE);
  const int ncb = min(CB, ncol - c0);
  const int sh = 31 - __clz(CB);  // CB is a power of two
  for (int i = threadIdx.x; i < N << sh; i += blockDim.x) {
    const int z = i >> sh, cc = i & (CB - 1);
    if (cc < ncb) line[cc * LS + z] = Sb[(size_t)z * ncol + c0 + cc];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const TileLane<N> t(threadIdx.x & 31);
  C* tile = tiles + warp * L::WTILE + t.grp * L::TILE;
  ST zero;
  zero.x = zero.y = 0;
  for (int l0 = warp * L::G; l0 < ncb; l0 += nw * L::G) {
    const int l = l0 + t.grp;
    const bool ok = t.ok && l < ncb;
    ST* ln = line + (ok ? l : 0) * LS;
    C v[L::V];
    FxScale sc{0, false};
    if constexpr (NT::kFixed) {
      ST raw[L::V];
      int key = 0;
#pragma unroll
      for (int i = 0; i < L::V; ++i) {
        const int k = tile_index<N>(t.p, i);
        raw[i] = ok && k >= 0 ? ln[k] : zero;
        key = max(key, fx_key(raw[i]));
      }
      key = tile_max<L::P>(key, t.base);
      const int ex = key >> 20, e = max(ex, 1) - 1022;
      sc.nan = ex == 0x7ff;
      sc.k = e - (62 - L::GROW);
#pragma unroll
      for (int i = 0; i < L::V; ++i)
        v[i] = fxc{fx_from<62 - L::GROW>(raw[i].x, e), fx_from<62 - L::GROW>(raw[i].y, e)};
    } else {
#pragma unroll
      for (int i = 0; i < L::V; ++i) {
        const int k = tile_index<N>(t.p, i);
        v[i] = ok && k >= 0 ? ln[k] : zero;
      }
    }
    tile_fwd<NT, N>(v, t.p, twz, tile, t.ok);
    if (ok)
#pragma unroll
      for (int q = 0; q < L::Q; ++q) ln[L::P * q + t.p] = tile_out<NT>(v[q], sc);
  }
  __syncthreads();
  const int g0 = col_off[c0], g1 = col_off[c0 + ncb];
  for (int g = g0 + threadIdx.x; g < g1; g += blockDim.x) {
    const ST v = line[(g_col[g] - c0) * LS + g_z[g]];
    if (ACC) {
      h[g] = cadd(h[g], v);
    } else {
      const ST cc = pp[g];
      const typename NT::R tk = kin[g] - shift;
      ST o;
      o.x = v.x + tk * cc.x;
      o.y = v.y + tk * cc.y;
      if constexpr (KB)
        for (int j = 0; j < np; ++j) {
          const ST bv = beta[(size_t)j * npw + g], d = dp[j];
          o.x += bv.x * d.x - bv.y * d.y;
          o.y += bv.x * d.y + bv.y * d.x;
        }
      h[g] = o;
    }
  }
}

template <typename NT, int N, bool ACC>
__global__ void __launch_bounds__(256) k_zfwd_tile(const typename NT::S* __restrict__ S,
                                                   const typename NT::S* __restrict__ psi, int ldpsi,
                                                   typename NT::S* __restrict__ hpsi, int ldh,
                                                   const typename NT::R* __restrict__ kin, typename NT::R shift,
                                                   const int* __restrict__ col_off, const int* __restrict__ g_col,
                                                   const int* __restrict__ g_z, int ncol,
                                                   const typename NT::W* __restrict__ twz,
                                                   const int* __restrict__ active, int CB) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int b = blockIdx.y;
  if (active != nullptr && active[b] == 0) return;
  zfwd_sticks<NT, N, ACC, false>(smem_raw, S + (size_t)b * N * ncol, psi + (size_t)b * ldpsi, hpsi + (size_t)b * ldh, kin,
                                 shift, col_off, g_col, g_z, ncol, twz, blockIdx.x * CB, CB);
}

// Density planes: per (z-plane, band group) the inverse transforms of each band, |psi(r)|^2 summed in FP64
// in shared memory and written to part.
template <typename NT, int N>
__global__ void __launch_bounds__(32 * TileWarps<N>::value)
    k_density_tile(const typename NT::S* __restrict__ S, int ncol, int nbands, int gsize,
                   const int* __restrict__ stick_of, const int* __restrict__ xrow_c, int nxr,
                   const typename NT::W* __restrict__ twx, const typename NT::W* __restrict__ twy, double wfac,
                   const double* __restrict__ wsq, double* __restrict__ part) {
  using L = TileLine<N>;
  using ST = typename NT::S;
  using C = typename NT::C;
  constexpr int LS = TileStride<N>::value;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tiles = reinterpret_cast<C*>(smem_raw);
  ST* Pl = reinterpret_cast<ST*>(tiles + (blockDim.x >> 5) * L::WTILE);
  double* acc = reinterpret_cast<double*>(Pl + (size_t)nxr * LS);
  int* roff = reinterpret_cast<int*>(acc + N * N);
  const int z = blockIdx.x, grp_b = blockIdx.y;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const int r = xrow_c[i];
    roff[i] = r >= 0 ? r * LS : -1;
  }
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) acc[i] = 0.0;
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const TileLane<N> t(threadIdx.x & 31);
  C* tile = tiles + warp * L::WTILE + t.grp * L::TILE;
  ST zero;
  zero.x = zero.y = 0;
  const int b0 = grp_b * gsize, b1 = min(nbands, b0 + gsize);
  for (int b = b0; b < b1; ++b) {
    const ST* Sz = S + ((size_t)b * N + z) * ncol;
    __syncthreads();  // the plane of the band before has been read
    tile_rows_inv<NT, N>(Sz, stick_of, nxr, twy, tiles, Pl);
    __syncthreads();
    const double wb = wsq ? wsq[b] * wsq[b] : 1.0;  // the band's occupation weight
    for (int c0 = warp * L::G; c0 < N; c0 += nw * L::G) {
      const int y = c0 + t.grp;
      const bool ok = t.ok && y < N;
      ST raw[L::Q];
#pragma unroll
      for (int q = 0; q < L::Q; ++q) {
        const int o = roff[L::P * q + t.p];
        raw[q] = ok && o >= 0 ? Pl[o + y] : zero;
      }
      C v[L::V];
      const FxScale sc = tile_load<NT, N>(raw, v, t.base);
      tile_inv<NT, N>(v, t.p, twx, tile, t.ok);
      if (ok)
#pragma unroll
        for (int i = 0; i < L::V; ++i) {
          const int k = tile_index<N>(t.p, i);
          if (k < 0) continue;
          const ST o = tile_out<NT>(v[i], sc);
          const double re = o.x, im = o.y;
          acc[k * N + y] += wb * (re * re + im * im);
        }
    }
  }
  __syncthreads();
  double* out = part + ((size_t)grp_b * N + z) * N * N;
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) out[i] = acc[i] * wfac;
}

// ---- host side ----
template <typename NT> struct TileTables;  // twiddles, potential and kinetic table of a context
template <> struct TileTables<NumF32> {
  static const float2* tw(const Ctx* c, int ax) { return c->d_tw32[ax]; }
  static const float* v(const Ctx* c) { return c->d_vplane32; }
  static const float* kin(const Basis& b) { return b.d_kin32; }
};
template <> struct TileTables<NumF64> {
  static const fxw* tw(const Ctx* c, int ax) { return static_cast<const fxw*>(c->d_twfx[ax]); }
  static const double* v(const Ctx* c) { return c->d_vplane; }
  static const double* kin(const Basis& b) { return b.d_kin; }
};

static const size_t kTileSmemMax = 227 * 1024;

template <typename K> static int tile_attr(Ctx* c, K kernel, int* done) {
  int dev = 0;
  PARO_CU(c, cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && done[dev]) return PARO_OK;
  PARO_CU(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmemMax));
  PARO_CU(c, cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  if (dev >= 0 && dev < 64) done[dev] = 1;
  return PARO_OK;
}

// z-pass launch shape: 32 sticks per CTA, fewer while that leaves SMs without a CTA; a warp per G lines
struct TileZ {
  int cb, threads;
  size_t smem;
};
template <typename NT, int N> static TileZ tile_z(int ncol, int nb) {
  using L = TileLine<N>;
  TileZ z;
  z.cb = 32;
  while (z.cb > 8 && (long long)((ncol + z.cb - 1) / z.cb) * nb < 304) z.cb /= 2;
  const int w = std::min(8, (z.cb + L::G - 1) / L::G);
  z.threads = 32 * w;
  z.smem = (size_t)w * L::WTILE * sizeof(typename NT::C) + (size_t)z.cb * TileStride<N>::value * sizeof(typename NT::S);
  return z;
}

template <typename NT, int N> static size_t tile_plane_smem(int nxr, int warps) {
  using L = TileLine<N>;
  return (size_t)warps * L::WTILE * sizeof(typename NT::C) +
         (size_t)nxr * TileStride<N>::value * sizeof(typename NT::S) + N * sizeof(int);
}

template <typename NT, int N>
static int tile_passes(Ctx* c, const Basis& B, int nb, const typename NT::S* psi, typename NT::S* S,
                       typename NT::S* hpsi, double shift, const int* active, const typename NT::R* vplane, bool acc) {
  static int done[4][64];
  using TT = TileTables<NT>;
  const bool f64 = NT::kFixed;
  int st;
  if ((st = tile_attr(c, k_zinv_tile<NT, N>, done[0])) || (st = tile_attr(c, k_plane_tile<NT, N>, done[1])) ||
      (st = tile_attr(c, k_zfwd_tile<NT, N, false>, done[2])) || (st = tile_attr(c, k_zfwd_tile<NT, N, true>, done[3])))
    return st;
  const TileZ z = tile_z<NT, N>(B.ncol, nb);
  const dim3 gz((B.ncol + z.cb - 1) / z.cb, nb);
  cudaEvent_t ev = prof_begin(c);
  k_zinv_tile<NT, N><<<gz, z.threads, z.smem, c->stream>>>(psi, B.npw, S, B.d_col_off, B.d_g_col, B.d_g_z, B.ncol,
                                                           TT::tw(c, 2), active, z.cb);
  PARO_LAUNCH(c, "k_zinv_tile");
  prof_end(c, f64 ? "k_zpass_inv<f64>" : "k_zpass_inv<f32>", ev);
  ev = prof_begin(c);
  constexpr int NW = TileWarps<N>::value;
  k_plane_tile<NT, N><<<dim3(N, nb), 32 * NW, tile_plane_smem<NT, N>(B.nxr, NW), c->stream>>>(
      S, B.ncol, B.d_stick_of, B.d_xrow_c, B.nxr, TT::tw(c, 0), TT::tw(c, 1), vplane ? vplane : TT::v(c), active);
  PARO_LAUNCH(c, "k_plane_tile");
  prof_end(c, f64 ? "k_plane<f64>" : "k_plane<f32>", ev);
  ev = prof_begin(c);
  if (acc)
    k_zfwd_tile<NT, N, true><<<gz, z.threads, z.smem, c->stream>>>(S, psi, B.npw, hpsi, B.npw, TT::kin(B),
                                                                   (typename NT::R)shift, B.d_col_off, B.d_g_col,
                                                                   B.d_g_z, B.ncol, TT::tw(c, 2), active, z.cb);
  else
    k_zfwd_tile<NT, N, false><<<gz, z.threads, z.smem, c->stream>>>(S, psi, B.npw, hpsi, B.npw, TT::kin(B),
                                                                    (typename NT::R)shift, B.d_col_off, B.d_g_col,
                                                                    B.d_g_z, B.ncol, TT::tw(c, 2), active, z.cb);
  PARO_LAUNCH(c, "k_zfwd_tile");
  prof_end(c, f64 ? "k_zpass_fwd<f64>" : "k_zpass_fwd<f32>", ev);
  return PARO_OK;
}

template <typename NT, int N>
static int tile_sticks(Ctx* c, const Basis& B, int nb, const typename NT::S* psi, typename NT::S* S) {
  static int done[64];
  if (int st = tile_attr(c, k_zinv_tile<NT, N>, done)) return st;
  const TileZ z = tile_z<NT, N>(B.ncol, nb);
  k_zinv_tile<NT, N><<<dim3((B.ncol + z.cb - 1) / z.cb, nb), z.threads, z.smem, c->stream>>>(
      psi, B.npw, S, B.d_col_off, B.d_g_col, B.d_g_z, B.ncol, TileTables<NT>::tw(c, 2), nullptr, z.cb);
  PARO_LAUNCH(c, "k_zinv_tile");
  return PARO_OK;
}

// warps of the density CTA: as many of the plane pass's as fit beside the accumulator (0: none)
template <typename NT, int N> static int tile_density_warps(int nxr) {
  for (int w = TileWarps<N>::value; w >= 2; --w)
    if (tile_plane_smem<NT, N>(nxr, w) + (size_t)N * N * sizeof(double) + 16 <= kTileSmemMax) return w;
  return 0;
}

template <typename NT, int N>
static int tile_density(Ctx* c, const Basis& B, const typename NT::S* S, int nbands, int ngrp, int gsize, double wfac,
                        const double* wsq, double* part, bool* used) {
  static int done[64];
  const int w = tile_density_warps<NT, N>(B.nxr);
  *used = w > 0;
  if (!w) return PARO_OK;
  if (int st = tile_attr(c, k_density_tile<NT, N>, done)) return st;
  const size_t smem = tile_plane_smem<NT, N>(B.nxr, w) + (size_t)N * N * sizeof(double) + 16;
  k_density_tile<NT, N><<<dim3(N, ngrp), 32 * w, smem, c->stream>>>(S, B.ncol, nbands, gsize, B.d_stick_of, B.d_xrow_c,
                                                                    B.nxr, TileTables<NT>::tw(c, 0),
                                                                    TileTables<NT>::tw(c, 1), wfac, wsq, part);
  PARO_LAUNCH(c, "k_density_tile");
  return PARO_OK;
}

// The passes of one number type over its list of grids (cubic; the plane must fit in shared memory); *used =
// false for other grids.
template <typename NT, int... Ns> struct TileGrids {
  template <int N> static bool fits(const Ctx* c, const Basis& B) {
    return c->N[0] == N && c->N[1] == N && c->N[2] == N &&
           tile_plane_smem<NT, N>(B.nxr, TileWarps<N>::value) <= kTileSmemMax;
  }
  static int passes(Ctx* c, const Basis& B, int nb, const typename NT::S* psi, typename NT::S* S,
                    typename NT::S* hpsi, double shift, const int* active, const typename NT::R* vplane, bool acc,
                    bool* used) {
    int st = PARO_OK;
    *used = false;
    ((!*used && fits<Ns>(c, B)
          ? (*used = true, st = tile_passes<NT, Ns>(c, B, nb, psi, S, hpsi, shift, active, vplane, acc), 0)
          : 0),
     ...);
    return st;
  }
  static int sticks(Ctx* c, const Basis& B, int nb, const typename NT::S* psi, typename NT::S* S, bool* used) {
    int st = PARO_OK;
    *used = false;
    ((!*used && fits<Ns>(c, B) ? (*used = true, st = tile_sticks<NT, Ns>(c, B, nb, psi, S), 0) : 0), ...);
    return st;
  }
  static int density(Ctx* c, const Basis& B, const typename NT::S* S, int nbands, int ngrp, int gsize, double wfac,
                     const double* wsq, double* part, bool* used) {
    int st = PARO_OK;
    bool hit = false;
    *used = false;
    ((!hit && fits<Ns>(c, B)
          ? (hit = true, st = tile_density<NT, Ns>(c, B, S, nbands, ngrp, gsize, wfac, wsq, part, used), 0)
          : 0),
     ...);
    return st;
  }
};

}  // namespace paro
