// Line FFTs of N = Q P points held by P lanes of a warp, Q values each, with both factors transformed inside
// the lanes: n = P q + p, k = k1 + Q k2,
//   A  Q-point DFT over q in every lane,
//   B  twiddle W_N^{p k1},
//   exchange through a Q x P tile in shared memory (row k1 = the P lanes' values of that k1),
//   C  P-point DFTs of the rows k1 = p, p + P, .. in lane p.
// Natural layout: lane p holds v[q] = x[P q + p]. Transformed layout: lane p holds v[j P + k2] = X[k1 + Q k2],
// k1 = p + P j (slots with k1 >= Q, where P does not divide Q, are unused). The forward transform runs the mirror
// image and takes the transformed layout back to the natural one. P need not be a power of two: a warp takes
// 32 / P lines and the lanes left over idle.
//
// Two number types: float, and 64-bit fixed point for FP64 data. The FP64 pipe of this chip issues one
// instruction in 32 cycles of a quarter SM (1/64 of the FP32 rate), a 64-bit integer addition is two
// instructions of the full-rate integer pipe and a product with a 62-bit constant about a dozen, so the
// butterflies of FP64 lines run in integers: a line is brought to the exponent of its largest value with
// the headroom of its growth (N sqrt 2), transformed, and converted back to FP64 with its exponent. The error is
// that of an FP64 transform, relative to the line: values are multiples of 2^-(62 - GROW) of the power of two above
// the line's largest (2^-56 up to 45 points, 2^-55 up to 90, 2^-54 above), so that elements far below it keep fewer
// bits than FP64 would, sums are exact, products are rounded to that unit, and the constants are doubles scaled by
// 2^62 (the twiddles to 2^-54; sqrt 3 / 2, 1 / sqrt 2 and t_root's series to 6.5 x 2^-56). Results below the normal
// range of FP64 become zero.
#pragma once

#include "paro_common.cuh"

namespace paro {

// ---- 64-bit fixed point ----
struct fxc {
  long long x, y;
};
struct __align__(16) fxw {  // twiddle: Q62 parts as hi 2^32 + lo, lo signed
  int rh, rl, ih, il;
};

struct FxSplit {
  int h, l;
};
__host__ __device__ __forceinline__ constexpr FxSplit fx_split(long long v) {
  return {(int)((v - (long long)(int)(unsigned)(v & 0xffffffffll)) >> 32), (int)(unsigned)(v & 0xffffffffll)};
}
__device__ __forceinline__ FxSplit fx_cut(long long v) {
  FxSplit s;
  s.l = (int)v;
  s.h = (int)(v >> 32) + (int)((unsigned)s.l >> 31);
  return s;
}
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
// (x w) 2^-62, |x| < 2^62, |w| <= 2^62 (the product of the low words is below the last bit)
__device__ __forceinline__ long long fx_mul(FxSplit x, FxSplit w) {
  const long long q = fx_mad(x.l, w.h, fx_mad(x.h, w.l, 1ll << 29));
  return (fx_mad(x.h, w.h, 0) << 2) + (q >> 30);
}
__device__ __forceinline__ fxc fx_cmul(fxc z, int rh, int rl, int ih, int il) {
  const FxSplit a = fx_cut(z.x), b = fx_cut(z.y);
  fxc r;
  const long long qx = fx_mad(b.l, -ih, fx_mad(b.h, -il, fx_mad(a.l, rh, fx_mad(a.h, rl, 1ll << 29))));
  r.x = (fx_mad(b.h, -ih, fx_mad(a.h, rh, 0)) << 2) + (qx >> 30);
  const long long qy = fx_mad(b.l, rh, fx_mad(b.h, rl, fx_mad(a.l, ih, fx_mad(a.h, il, 1ll << 29))));
  r.y = (fx_mad(b.h, rh, fx_mad(a.h, ih, 0)) << 2) + (qy >> 30);
  return r;
}

// ---- number types of a line ----
struct NumF32 {
  using S = float2;  // as stored
  using R = float;
  using C = float2;  // in registers
  using W = float2;  // twiddle table entry
  static constexpr bool kFixed = false;
};
struct NumF64 {
  using S = double2;
  using R = double;
  using C = fxc;
  using W = fxw;
  static constexpr bool kFixed = true;
};

__device__ __forceinline__ float2 t_zero(float2) { return make_float2(0.f, 0.f); }
__device__ __forceinline__ fxc t_zero(fxc) { return fxc{0, 0}; }
__device__ __forceinline__ float2 t_half(float2 a) { return make_float2(0.5f * a.x, 0.5f * a.y); }
__device__ __forceinline__ fxc t_half(fxc a) { return fxc{(a.x + 1) >> 1, (a.y + 1) >> 1}; }
__device__ __forceinline__ float2 t_real(float2 a, double c) { return make_float2(a.x * (float)c, a.y * (float)c); }
__device__ __forceinline__ fxc t_real(fxc a, double c) {
  const FxSplit w = fx_split((long long)(c * 4611686018427387904.0));
  return fxc{fx_mul(fx_cut(a.x), w), fx_mul(fx_cut(a.y), w)};
}
__device__ __forceinline__ float2 t_const(float2 a, double c, double s) {
  return cmul(a, make_float2((float)c, (float)s));
}
__device__ __forceinline__ fxc t_const(fxc a, double c, double s) {
  const FxSplit r = fx_split((long long)(c * 4611686018427387904.0)), i = fx_split((long long)(s * 4611686018427387904.0));
  return fx_cmul(a, r.h, r.l, i.h, i.l);
}
template <bool INV> __device__ __forceinline__ float2 t_tw(float2 a, float2 w) { return cmul(a, INV ? cconj(w) : w); }
template <bool INV> __device__ __forceinline__ fxc t_tw(fxc a, fxw w) {
  return INV ? fx_cmul(a, w.rh, w.rl, -w.ih, -w.il) : fx_cmul(a, w.rh, w.rl, w.ih, w.il);
}

// cos and sin of 2 pi m / R for constant m (after unrolling), by reduction to an angle up to pi / 4
struct TRoot {
  double c, s;
};
__host__ __device__ __forceinline__ constexpr TRoot t_root(int m, int R) {
  m %= R;
  const int oct = 8 * m / R;  // octant 0..7
  // angle to the nearest multiple of pi / 2 below or above: 2 pi a / R with a in [-R/8, R/8]
  const int quad = (oct + 1) / 2;
  const double x = 6.283185307179586476925286766559 * ((double)(4 * m - quad * R) / (4.0 * R));
  const double z = x * x;
  const double s = x * (1 + z * (-1.0 / 6 + z * (1.0 / 120 + z * (-1.0 / 5040 + z * (1.0 / 362880 + z * (-1.0 / 39916800 +
                   z * (1.0 / 6227020800.0 + z * (-1.0 / 1307674368000.0))))))));
  const double c = 1 + z * (-0.5 + z * (1.0 / 24 + z * (-1.0 / 720 + z * (1.0 / 40320 + z * (-1.0 / 3628800 +
                   z * (1.0 / 479001600.0 + z * (-1.0 / 87178291200.0 + z * (1.0 / 20922789888000.0))))))));
  return quad % 4 == 0 ? TRoot{c, s} : quad % 4 == 1 ? TRoot{-s, c} : quad % 4 == 2 ? TRoot{-c, -s} : TRoot{s, -c};
}
// z exp(-+ 2 pi i m / R)
template <bool INV, int R, typename C> __device__ __forceinline__ C t_rotate(C z, int m) {
  m %= R;
  if (m == 0) return z;
  if (4 * m == R) return rot90<INV>(z);
  if (2 * m == R) return csub(t_zero(z), z);
  if (4 * m == 3 * R) return rot90<!INV>(z);
  if (8 * m == R) {  // (1 -+ i) / sqrt 2
    return t_real(cadd(z, rot90<INV>(z)), 0.70710678118654752440);
  }
  if (8 * m == 3 * R) return t_real(csub(rot90<INV>(z), z), 0.70710678118654752440);
  const TRoot w = t_root(m, R);
  return t_const(z, w.c, INV ? w.s : -w.s);
}

// ---- R-point DFTs in registers ----
template <int R, bool INV> struct TDft;
template <bool INV> struct TDft<2, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) {
    const C a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};
template <bool INV> struct TDft<3, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) {
    const C a = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const C m = csub(v[0], t_half(a)), jd = t_real(rot90<INV>(d), 0.86602540378443864676);
    v[0] = cadd(v[0], a);
    v[1] = cadd(m, jd);
    v[2] = csub(m, jd);
  }
};
template <bool INV> struct TDft<4, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) {
    const C a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = rot90<INV>(csub(v[1], v[3]));
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = cadd(b, d);
    v[3] = csub(b, d);
  }
};
// R = A B: input q = B a + b, output k = k1 + A k2
template <int A, int B, bool INV, typename C> __device__ __forceinline__ void t_dft_2f(C* v) {
  C w[A * B];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    C t[A];
#pragma unroll
    for (int a = 0; a < A; ++a) t[a] = v[B * a + b];
    TDft<A, INV>::run(t);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) w[k1 * B + b] = t_rotate<INV, A * B>(t[k1], b * k1);
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    C u[B];
#pragma unroll
    for (int b = 0; b < B; ++b) u[b] = w[k1 * B + b];
    TDft<B, INV>::run(u);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = u[k2];
  }
}
template <bool INV> struct TDft<6, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) { t_dft_2f<2, 3, INV>(v); }
};
template <bool INV> struct TDft<8, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) { t_dft_2f<4, 2, INV>(v); }
};
template <bool INV> struct TDft<9, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) { t_dft_2f<3, 3, INV>(v); }
};
template <bool INV> struct TDft<12, INV> {
  template <typename C> static __device__ __forceinline__ void run(C* v) { t_dft_2f<4, 3, INV>(v); }
};

// ---- line shapes ----
// Few values a lane keep the fixed-point kernels below 128 registers: 54 = 9 x 6 took 1.22 ms a plane pass of 144
// orbitals where 18 x 3 (255 registers) took 3.03, 36 = 6 x 6 52 us (23 orbitals) where 12 x 3 took 71, 96 = 12 x 8
// 3.3 ms (60 orbitals) where 16 x 6 took 3.7; 72 = 8 x 9 was no better than 12 x 6 (2.07 and 1.97 ms, 144 orbitals).
template <int N> struct TileShape;
template <> struct TileShape<27> { static constexpr int Q = 9, P = 3; };
template <> struct TileShape<32> { static constexpr int Q = 8, P = 4; };
template <> struct TileShape<36> { static constexpr int Q = 6, P = 6; };
template <> struct TileShape<48> { static constexpr int Q = 12, P = 4; };
template <> struct TileShape<54> { static constexpr int Q = 9, P = 6; };
template <> struct TileShape<64> { static constexpr int Q = 8, P = 8; };
template <> struct TileShape<72> { static constexpr int Q = 12, P = 6; };
template <> struct TileShape<81> { static constexpr int Q = 9, P = 9; };
template <> struct TileShape<96> { static constexpr int Q = 12, P = 8; };
template <> struct TileShape<108> { static constexpr int Q = 12, P = 9; };

template <int N> struct TileLine {
  static constexpr int Q = TileShape<N>::Q, P = TileShape<N>::P;
  static constexpr int J = (Q + P - 1) / P;       // P-point DFTs per lane
  static constexpr int V = J * P > Q ? J * P : Q;  // register slots
  static constexpr int G = 32 / P;                 // lines per warp
  static constexpr int TS = P | 1;                 // tile row stride: odd, so a column of rows meets no bank twice
  static constexpr int TILE = Q * TS;              // elements of one line's tile
  static constexpr int WTILE = G * TILE;
  // headroom bits: |X| <= N max|x| sqrt 2
  static constexpr int GROW = N <= 45 ? 6 : N <= 90 ? 7 : 8;
};

// the grid point of slot i of the transformed layout (-1: unused slot)
template <int N> __device__ __forceinline__ int tile_index(int p, int i) {
  using L = TileLine<N>;
  const int k1 = p + L::P * (i / L::P);
  return k1 < L::Q ? k1 + L::Q * (i % L::P) : -1;
}

template <typename NT, int N>
__device__ __forceinline__ void tile_inv(typename NT::C* v, int p, const typename NT::W* tw, typename NT::C* tile,
                                         bool lane_ok) {
  using L = TileLine<N>;
  using C = typename NT::C;
  TDft<L::Q, true>::run(v);
  __syncwarp();  // the tile's earlier readers are done
#pragma unroll
  for (int k1 = 0; k1 < L::Q; ++k1) {
    const C t = k1 ? t_tw<true>(v[k1], tw[p * k1]) : v[k1];
    if (lane_ok) tile[k1 * L::TS + p] = t;
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < L::J; ++j) {
    const int k1 = p + L::P * j;
    C u[L::P];
#pragma unroll
    for (int i = 0; i < L::P; ++i) u[i] = tile[(k1 < L::Q ? k1 : 0) * L::TS + i];
    TDft<L::P, true>::run(u);
#pragma unroll
    for (int i = 0; i < L::P; ++i) v[j * L::P + i] = u[i];
  }
}

template <typename NT, int N>
__device__ __forceinline__ void tile_fwd(typename NT::C* v, int p, const typename NT::W* tw, typename NT::C* tile,
                                         bool lane_ok) {
  using L = TileLine<N>;
  using C = typename NT::C;
  __syncwarp();
#pragma unroll
  for (int j = 0; j < L::J; ++j) {
    const int k1 = p + L::P * j;
    C u[L::P];
#pragma unroll
    for (int i = 0; i < L::P; ++i) u[i] = v[j * L::P + i];
    TDft<L::P, false>::run(u);
    if (lane_ok && k1 < L::Q)
#pragma unroll
      for (int i = 0; i < L::P; ++i) tile[k1 * L::TS + i] = u[i];
  }
  __syncwarp();
#pragma unroll
  for (int k1 = 0; k1 < L::Q; ++k1) {
    const C t = tile[k1 * L::TS + p];
    v[k1] = k1 ? t_tw<false>(t, tw[p * k1]) : t;
  }
  TDft<L::Q, false>::run(v);
}

// ---- conversions ----
// maximum over the P lanes of a line (every lane of the warp calls it; base: first lane of the line)
template <int P> __device__ __forceinline__ int tile_max(int x, int base) {
  if constexpr ((P & (P - 1)) == 0) {
#pragma unroll
    for (int h = P / 2; h >= 1; h >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, h));
    return x;
  } else {
    int m = x;
#pragma unroll
    for (int i = 0; i < P; ++i) m = max(m, __shfl_sync(0xffffffffu, x, base + i));
    return m;
  }
}
// exponent state of a line in fixed point: value = F 2^k; nan: the line holds Inf or NaN
struct FxScale {
  int k;
  bool nan;
};
__device__ __forceinline__ long long fx_shift(long long v, int s) {  // v 2^s, rounded
  return s >= 0 ? v << s : (v + (1ll << (-s - 1))) >> -s;
}
// x 2^(B - e) for |x| < 2^e, B <= 62
template <int B> __device__ __forceinline__ long long fx_from(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  unsigned long long u = ((unsigned long long)(hi & 0xfffff) << 32) | (unsigned)__double2loint(x);
  if (ex) u |= 1ull << 52;
  const int s = max(ex, 1) - 1075 + B - e;
  if (s >= 0) u <<= min(s, 63);
  else u = s < -54 ? 0ull : (u + (1ull << (-s - 1))) >> -s;
  return hi < 0 ? -(long long)u : (long long)u;
}
__device__ __forceinline__ double fx_to(long long v, int k) {  // v 2^k
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll((long long)a);
  const unsigned long long m = a << (z & 63);
  const int ex = 63 - z + k + 1023;
  const unsigned long long q = (m >> 11) + ((m >> 10) & 1ull);
  unsigned long long bits = ((unsigned long long)(unsigned)(ex - 1) << 52) + q;
  if (a == 0 || ex <= 0) bits = 0;  // results below the normal range vanish
  if (ex >= 2047) bits = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(bits | ((unsigned long long)v & 0x8000000000000000ull)));
}
__device__ __forceinline__ int fx_key(double2 v) {
  return max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
}

// Q raw values of a line -> registers in the line's number type
template <typename NT, int N>
__device__ __forceinline__ FxScale tile_load(const typename NT::S* raw, typename NT::C* v, int base) {
  using L = TileLine<N>;
  FxScale sc{0, false};
  if constexpr (NT::kFixed) {
    int key = 0;
#pragma unroll
    for (int q = 0; q < L::Q; ++q) key = max(key, fx_key(raw[q]));
    key = tile_max<L::P>(key, base);
    const int ex = key >> 20, e = max(ex, 1) - 1022;
    sc.nan = ex == 0x7ff;
    sc.k = e - (62 - L::GROW);
#pragma unroll
    for (int q = 0; q < L::Q; ++q)
      v[q] = fxc{fx_from<62 - L::GROW>(raw[q].x, e), fx_from<62 - L::GROW>(raw[q].y, e)};
  } else {
#pragma unroll
    for (int q = 0; q < L::Q; ++q) v[q] = raw[q];
  }
  return sc;
}
// shifts the line so that its largest component is just below 2^B
template <typename NT, int N, int B>
__device__ __forceinline__ void tile_normalise(typename NT::C* v, int p, FxScale& sc, int base) {
  using L = TileLine<N>;
  int h = 0;
#pragma unroll
  for (int i = 0; i < L::V; ++i) {
    if (L::V != L::Q && tile_index<N>(p, i) < 0) continue;
    const int a = (int)(v[i].x >> 32), b = (int)(v[i].y >> 32);
    h = max(h, max(a ^ (a >> 31), b ^ (b >> 31)));
  }
  h = tile_max<L::P>(h, base);
  const int s = B - 64 + __clz(h);
  sc.k -= s;
  if (s >= 0) {
#pragma unroll
    for (int i = 0; i < L::V; ++i) v[i] = fxc{v[i].x << s, v[i].y << s};
  } else {
#pragma unroll
    for (int i = 0; i < L::V; ++i) v[i] = fxc{fx_shift(v[i].x, s), fx_shift(v[i].y, s)};
  }
}
template <typename NT>
__device__ __forceinline__ typename NT::S tile_out(typename NT::C v, const FxScale& sc) {
  if constexpr (NT::kFixed) {
    if (sc.nan) return make_double2(NAN, NAN);
    return make_double2(fx_to(v.x, sc.k), fx_to(v.y, sc.k));
  } else {
    return v;
  }
}

}  // namespace paro
