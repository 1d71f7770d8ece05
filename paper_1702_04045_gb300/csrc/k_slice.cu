// Complex GEMMs with FP64 (or better than FP32) accuracy on the bf16 tensor cores, by error-free slicing
// (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix multiplication", Numer. Algorithms 59,
// 2012; the tensor-core form of Mukunoki, Ozaki, Ogita, Imamura, ISC 2020): the FP64 pipe of this chip does
// 1.25 TFLOP/s, its bf16 tensor cores about 2 PFLOP/s.
//
// Every operand row is brought to a common exponent (|x| < 2^e), rounded to an integer of 8 L - 2 bits and
// sign and written in L balanced base-256 digits, d_i in [-128, 127], which bf16 holds exactly:
//   x = 2^(e + 2) sum_i d_i 256^-i.
// A product of rows is sum over (i, j) of 256^-(i+j) (d_i . d'_j). The digit products are integers of at most
// 2^14, and a chunk of K values is short enough that the sums of all (i, j) with one i + j = g stay below
// 2^24, so the tensor core's FP32 accumulation of each group g is exact. After every chunk the groups are
// read from tensor memory and added into 64-bit integers at their weights; floating point appears only in
// the final conversion. Groups up to g = PMAX are kept:
//   L = 7, PMAX = 9 (34 digit products): operands rounded to 2^-55 of the row's largest power of two, groups
//     dropped below that: FP64 results, more accurate than FP64 sums of the same length;
//   L = 4, PMAX = 5 (10 products): operands rounded to 2^-31, for FP32 operands outside the inner solves.
//
// Measured on the 64-atom cell (N_pw = 23847): V_nl of 144 FP64 orbitals 17.7 -> 0.57 ms, Cholesky
// orthonormalisation of 288 rows 31.8 -> 1.88 ms (0.8 ms of it the factorisation); the error against extended
// precision is 3e-17 of the rows' norms where FP64 sums have 3e-15. A stage (16 K values) of a 128 x 32 tile takes
// 1.8 us, 53 cycles per MMA of 64 columns against 48 for its operands' shared-memory traffic: the tensor
// pipe's operand feed bounds the FP64 projections (the tensor-core pipe is active 85 % of the cycles and multiplies in
// 54 %, shared memory is at 82 %; DRAM at 20 %), the loads (79 KB a stage) and the sums are hidden. The update (68 % and
// 44 %) and the FP32 form (55 % and 45 %) lose more to the start, drain and conversion of their shorter tiles.
// Rows keep an accuracy relative to their largest value: elements far below it keep fewer bits.
//
// C[m][n] = sum_k conj(a_m,k) b_n,k with planes of real and imaginary digits: the A tile holds 128 rows, the
// B tile NC rows three times (b_r; b_i; -b_r), so that a_r meets (b_r | b_i) and a_i meets (b_i | -b_r) as
// one MMA of 2 NC columns each: Re and Im side by side in tensor memory.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "paro_ctx.h"
#include "tc_sm100.cuh"

namespace paro {

static const int kSliceM = 128;           // rows of the A tile (TMEM lanes)
static const int kSliceK = 16;            // complex K values per stage (one MMA K step per plane)
static const int kSliceThreads = 320;     // producer warp, MMA warp, eight epilogue warps
static const uint32_t kSlicePolls = 1u << 24;
// Polls after which a wait of the kernel's roles gives up: kSlicePolls, or PARO_SLICE_POLLS of the environment (0: at
// once), which lets a test run the time-out path. The waits that drain the kernel keep kSlicePolls.
static uint32_t slice_polls() {
  static const uint32_t n = [] {
    const char* e = std::getenv("PARO_SLICE_POLLS");
    return e && e[0] ? (uint32_t)std::min<unsigned long>(std::strtoul(e, nullptr, 10), kSlicePolls) : kSlicePolls;
  }();
  return n;
}

// NC: columns of an output tile (2 NC accumulator columns per group, at most 512 in tensor memory): 32 for
// L = 7, 64 or 48 for L = 4, whichever pads less;
// CH: stages per exact chunk: 2 (planes) * 16 CH * 2^14 * (most pairs in a group) <= 2^24; NS: stage buffers
template <int L> struct SliceCfg;
template <> struct SliceCfg<7> { static constexpr int PMAX = 9, CH = 4, NS = 2; };
template <> struct SliceCfg<4> { static constexpr int PMAX = 5, CH = 8, NS = 3; };

template <int L> __host__ __device__ constexpr int slice_a_bytes() { return L * 2 * kSliceM * kSliceK * 2; }
template <int L> __host__ __device__ constexpr int slice_b_bytes(int nc) { return L * 3 * nc * kSliceK * 2; }
template <int L> static int slice_nc(int n) { return L == 7 ? 32 : (n + 47) / 48 * 48 < (n + 63) / 64 * 64 ? 48 : 64; }

// ------------------------------------------------------------------------------------------------
// digits
// ------------------------------------------------------------------------------------------------
// key: bits whose integer order is that of |x| (the high word for doubles); ex: biased exponent
__device__ __forceinline__ int slice_key(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int slice_key(float x) { return __float_as_int(x) & 0x7fffffff; }
template <typename T> __device__ __forceinline__ int slice_key_exp(int key) { return sizeof(T) == 8 ? key >> 20 : key >> 23; }
// the row exponent e (|x| < 2^e for every x of the row) from the row's largest key; bad: Inf or NaN inside
template <typename T> __device__ __forceinline__ int slice_exponent(int key, bool* bad) {
  const int ex = slice_key_exp<T>(key);
  *bad = ex == (sizeof(T) == 8 ? 0x7ff : 0xff);
  return max(ex, 1) - (sizeof(T) == 8 ? 1022 : 126);
}
// the integer of a value: round(x 2^(8 L - 2 - e)), halves away from zero; 30 bits fit 32-bit arithmetic
template <int L> struct SliceInt { using t = long long; };
template <> struct SliceInt<4> { using t = int; };
template <int L> __device__ __forceinline__ typename SliceInt<L>::t slice_fixed(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  unsigned long long u = ((unsigned long long)(hi & 0xfffff) << 32) | (unsigned)__double2loint(x);
  if (ex) u |= 1ull << 52;
  const int s = max(ex, 1) - 1075 + 8 * L - 2 - e;
  if (s >= 0) u <<= min(s, 63);
  else u = s < -55 ? 0ull : (u + (1ull << (-s - 1))) >> -s;
  const typename SliceInt<L>::t f = (typename SliceInt<L>::t)u;
  return hi < 0 ? -f : f;
}
template <int L> __device__ __forceinline__ typename SliceInt<L>::t slice_fixed(float x, int e) {
  const int b = __float_as_int(x), ex = (b >> 23) & 0xff;
  unsigned u = (unsigned)(b & 0x7fffff);
  if (ex) u |= 1u << 23;
  const int s = max(ex, 1) - 150 + 8 * L - 2 - e;
  if (s >= 0) u <<= min(s, 31);
  else u = s < -25 ? 0u : (u + (1u << (-s - 1))) >> -s;
  return b < 0 ? -(int)u : (int)u;
}
// balanced digits of F, most significant first, as bf16 bits in the upper half of d[i]: with 128 added to
// every low byte the bytes hold the digits + 128 (the top one as a signed byte), and a byte b under the
// exponent of 2^23 is the float 2^23 + b
__device__ __forceinline__ uint32_t slice_digit(uint32_t word, int byte) {
  return __float_as_uint(__uint_as_float(__byte_perm(word, 0x4B000000u, 0x7540 | byte)) - 8388736.0f);
}
template <int L> __device__ __forceinline__ void slice_digits(typename SliceInt<L>::t F, uint32_t d[L]) {
  if constexpr (L == 4) {
    const uint32_t t = ((uint32_t)F + 0x00808080u) ^ 0x80000000u;
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = slice_digit(t, 3 - i);
  } else {
    static_assert(L == 7, "digit layouts");
    const long long t = F + 0x0000808080808080ll;
    const uint32_t lo = (uint32_t)t, hi = (uint32_t)(t >> 32) ^ 0x00800000u;
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] = slice_digit(hi, 2 - i);
#pragma unroll
    for (int i = 3; i < 7; ++i) d[i] = slice_digit(lo, 6 - i);
  }
}
__device__ __forceinline__ uint32_t slice_pack(uint32_t d0, uint32_t d1) { return __byte_perm(d0, d1, 0x7632); }

// result scale of a row: 2^(e + 2 - 4 PMAX) (a result is the integer sum times the scales of its two rows)
template <int L> __device__ __forceinline__ int slice_scale(int e) { return e + 2 - 4 * SliceCfg<L>::PMAX; }
static const int kSliceBad = 1 << 20;  // scale of a row with Inf or NaN: its results are NaN

// eight consecutive k of one row (|v_j| < 2^e_j) -> its 16-byte core-matrix rows of every slice and plane
template <int L, typename T>
__device__ __forceinline__ void slice_store(const cplx<T>* v, const int* e, bool conj_a, unsigned char* a_dst,
                                            unsigned char* b_dst, int nc) {
  const int NCB = nc * kSliceK * 2;
  uint32_t wr[L][4], wi[L][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t d0[L], d1[L];
    slice_digits<L>(slice_fixed<L>(v[2 * q].x, e[2 * q]), d0);
    slice_digits<L>(slice_fixed<L>(v[2 * q + 1].x, e[2 * q + 1]), d1);
#pragma unroll
    for (int i = 0; i < L; ++i) wr[i][q] = slice_pack(d0[i], d1[i]);
    slice_digits<L>(slice_fixed<L>(v[2 * q].y, e[2 * q]), d0);
    slice_digits<L>(slice_fixed<L>(v[2 * q + 1].y, e[2 * q + 1]), d1);
#pragma unroll
    for (int i = 0; i < L; ++i) wi[i][q] = slice_pack(d0[i], d1[i]);
  }
#pragma unroll
  for (int i = 0; i < L; ++i) {
    const uint4 r = make_uint4(wr[i][0], wr[i][1], wr[i][2], wr[i][3]);
    const uint4 m = make_uint4(wi[i][0], wi[i][1], wi[i][2], wi[i][3]);
    const uint32_t neg = 0x80008000u;  // sign of both bf16 values
    if (a_dst) {
      *reinterpret_cast<uint4*>(a_dst + (size_t)(2 * i) * kSliceM * kSliceK * 2) = r;
      *reinterpret_cast<uint4*>(a_dst + (size_t)(2 * i + 1) * kSliceM * kSliceK * 2) =
          conj_a ? make_uint4(m.x ^ neg, m.y ^ neg, m.z ^ neg, m.w ^ neg) : m;
    }
    if (b_dst) {
      unsigned char* p = b_dst + (size_t)i * 3 * NCB;
      *reinterpret_cast<uint4*>(p) = r;
      *reinterpret_cast<uint4*>(p + NCB) = m;
      *reinterpret_cast<uint4*>(p + 2 * NCB) = make_uint4(r.x ^ neg, r.y ^ neg, r.z ^ neg, r.w ^ neg);
    }
  }
}

// byte offset of (row r of the tile, k8 of the stage) in a plane: 8-row x 16-byte core matrices
__device__ __forceinline__ size_t slice_core(int r, int c) { return (size_t)((r >> 3) * 2 + c) * 128 + (r & 7) * 16; }

template <int L>
__device__ __forceinline__ unsigned char* slice_a_at(unsigned char* img, int nstage, int row, int k8) {
  return img + ((size_t)(row / kSliceM) * nstage + (k8 >> 1)) * slice_a_bytes<L>() + slice_core(row % kSliceM, k8 & 1);
}
template <int L>
__device__ __forceinline__ unsigned char* slice_b_at(unsigned char* img, int nstage, int nc, int row, int k8) {
  return img + ((size_t)(row / nc) * nstage + (k8 >> 1)) * slice_b_bytes<L>(nc) + slice_core(row % nc, k8 & 1);
}

// Largest key of every row (rowkey cleared by the caller); finite: of its finite values only.
template <typename T>
__global__ void __launch_bounds__(256) k_slice_rowkey(int N, const cplx<T>* __restrict__ x, int ld,
                                                      int finite, int* __restrict__ rowkey) {
  const cplx<T>* xr = x + (size_t)blockIdx.y * ld;
  int key = 0;
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < N; n += gridDim.x * blockDim.x) {
    const cplx<T> v = xr[n];
    const int a = slice_key(v.x), b = slice_key(v.y);
    if (!finite || slice_key_exp<T>(a) != (sizeof(T) == 8 ? 0x7ff : 0xff)) key = max(key, a);
    if (!finite || slice_key_exp<T>(b) != (sizeof(T) == 8 ? 0x7ff : 0xff)) key = max(key, b);
  }
  key = __reduce_max_sync(0xffffffffu, key);
  if ((threadIdx.x & 31) == 0) atomicMax(&rowkey[blockIdx.y], key);
}
// Rows along contiguous k (orbitals, projectors): 8 rows x one K slice per CTA. Exponents are those of the
// slice (es[z][row], ld rows_pad), or with rowkey those of the whole rows (es[row]). a_img, b_img: either may be null. The slice is staged in shared memory,
// read coalesced (a thread's own eight values are 64 or 128 bytes apart from its neighbour's) and once when it
// fits the stage's 32 KB, else in pieces after a first pass for the exponents.
template <typename T> struct SliceStage { static constexpr int value = sizeof(T) == 8 ? 256 : 512; };
template <typename T, int L>
__global__ void __launch_bounds__(256) k_slice_rows(int rows, int rows_a, int rows_b, int K, int kslice, int nstage,
                                                    const cplx<T>* __restrict__ x, int ld, int conj_a,
                                                    unsigned char* __restrict__ a_img,
                                                    unsigned char* __restrict__ b_img, int* __restrict__ es,
                                                    int rows_pad, int stage, const int* __restrict__ rowkey, int nc) {
  extern __shared__ __align__(16) unsigned char smem_dyn[];
  cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_dyn);  // 8 x (stage + 1): columns of eight rows meet no bank twice
  __shared__ int skey[8];
  const int z = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = z * kslice, k1 = min(nstage * kSliceK, k0 + kslice);  // padded K: zeros past K
  const int lds = stage + 1;
  const bool once = k1 - k0 <= stage;
  if (once || !rowkey) {  // warp w: row w
    const int row = blockIdx.x * 8 + warp;
    const cplx<T>* xr = x + (size_t)min(row, rows - 1) * ld;
    int key = 0;
    for (int k = k0 + lane; k < k1; k += 32) {
      const cplx<T> v = row < rows && k < K ? xr[k] : mk<T>(0, 0);
      key = max(key, max(slice_key(v.x), slice_key(v.y)));
      if (once) buf[warp * lds + k - k0] = v;
    }
    key = __reduce_max_sync(0xffffffffu, key);
    if (rowkey) key = row < rows ? rowkey[row] : 0;
    if (lane == 0) skey[warp] = key;
  } else if (lane == 0) {
    const int row = blockIdx.x * 8 + warp;
    skey[warp] = row < rows ? rowkey[row] : 0;
  }
  __syncthreads();
  const int r = threadIdx.x & 7, row = blockIdx.x * 8 + r;
  bool bad;
  const int e = slice_exponent<T>(skey[r], &bad);
  if (threadIdx.x < 8 && (!rowkey || z == 0)) es[(size_t)z * rows_pad + row] = bad ? kSliceBad : slice_scale<L>(e);
  int ev[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) ev[j] = e;
  for (int p0 = k0; p0 < k1; p0 += stage) {
    const int p1 = min(k1, p0 + stage);
    if (!once) {
      __syncthreads();
      const int rw = blockIdx.x * 8 + warp;
      const cplx<T>* xr = x + (size_t)min(rw, rows - 1) * ld;
      for (int k = p0 + lane; k < p1; k += 32) buf[warp * lds + k - p0] = rw < rows && k < K ? xr[k] : mk<T>(0, 0);
      __syncthreads();
    }
    for (int k8 = p0 / 8 + (threadIdx.x >> 3); k8 < p1 / 8; k8 += 32) {
      cplx<T> v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = buf[r * lds + 8 * k8 - p0 + j];
      slice_store<L, T>(v, ev, conj_a != 0, a_img && row < rows_a ? slice_a_at<L>(a_img, nstage, row, k8) : nullptr,
                        b_img && row < rows_b ? slice_b_at<L>(b_img, nstage, nc, row, k8) : nullptr, nc);
    }
  }
}

// An update sums over the rows of X, whose sizes may differ widely (orbitals beside small corrections): the
// digits are taken of X[k][n] 2^-c_k and W(k, m) 2^c_k with c_k the exponent of row k, so that every row
// keeps its own accuracy. c_k = 0 without row keys (the projectors, all of one size).
template <typename T> __device__ __forceinline__ int slice_rowshift(const int* rowkey, int k) {
  if (!rowkey) return 0;
  const int key = rowkey[k];
  return key ? max(slice_key_exp<T>(key), 1) - (sizeof(T) == 8 ? 1022 : 126) : 0;
}
// running maximum of the exponents of v 2^-shift; Inf and NaN beat every number
static const int kSliceNonfinite = 1 << 16;
template <typename T> __device__ __forceinline__ int slice_top(cplx<T> v, int shift) {
  const int key = max(slice_key(v.x), slice_key(v.y));
  const int ex = slice_key_exp<T>(key);
  if (ex == (sizeof(T) == 8 ? 0x7ff : 0xff)) return kSliceNonfinite;
  return key ? max(ex, 1) - (sizeof(T) == 8 ? 1022 : 126) - shift : -kSliceNonfinite;
}

// Columns of X[k][n] as A rows (row n, K = the K rows of X), conjugated (the GEMM conjugates them back):
// 32 columns per CTA, eight warps over k.
template <typename T, int L>
__global__ void __launch_bounds__(256) k_slice_cols(int N, int K, int nstage, const cplx<T>* __restrict__ x, int ld,
                                                    const int* __restrict__ rowkey,
                                                    unsigned char* __restrict__ a_img, int* __restrict__ es) {
  __shared__ int stop[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = blockIdx.x * 32 + lane;
  if (threadIdx.x < 32) stop[threadIdx.x] = -kSliceNonfinite;
  __syncthreads();
  int top = -kSliceNonfinite;
  if (n < N)
    for (int k = warp; k < K; k += 8) top = max(top, slice_top<T>(x[(size_t)k * ld + n], slice_rowshift<T>(rowkey, k)));
  atomicMax(&stop[lane], top);
  __syncthreads();
  const bool bad = stop[lane] == kSliceNonfinite;
  const int e = stop[lane] == -kSliceNonfinite ? 0 : stop[lane];
  if (warp == 0) es[n] = bad ? kSliceBad : slice_scale<L>(e);
  for (int k8 = warp; k8 < 2 * nstage; k8 += 8) {
    cplx<T> v[8];
    int ev[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = 8 * k8 + j;
      v[j] = n < N && k < K ? x[(size_t)k * ld + n] : mk<T>(0, 0);
      ev[j] = e + (k < K ? slice_rowshift<T>(rowkey, k) : 0);
    }
    slice_store<L, T>(v, ev, true, slice_a_at<L>(a_img, nstage, n, k8), nullptr, 0);
  }
}

// The small matrix of an update as B rows: row m, value s_k W(k, m) 2^c_k (element (k, m) at W[k ldw + m], or
// at W[m ldw + k] when wt); 8 rows per CTA. TX: type of X, whose row keys give c_k.
template <int L, typename TX>
__global__ void __launch_bounds__(256) k_slice_w(int M, int K, int nstage, const double2* __restrict__ W, int ldw,
                                                 int wt, const double* __restrict__ s,
                                                 const int* __restrict__ rowkey, unsigned char* __restrict__ b_img,
                                                 int* __restrict__ es, int nc) {
  __shared__ int stop[8];
  const int r = threadIdx.x & 7, m = blockIdx.x * 8 + r;
  if (threadIdx.x < 8) stop[threadIdx.x] = -kSliceNonfinite;
  __syncthreads();
  auto at = [&](int k) {
    if (m >= M || k >= K) return make_double2(0.0, 0.0);
    const double2 w = wt ? W[(size_t)m * ldw + k] : W[(size_t)k * ldw + m];
    return s ? cscale(w, s[k]) : w;
  };
  int top = -kSliceNonfinite;
  for (int k = threadIdx.x >> 3; k < K; k += 32) top = max(top, slice_top<double>(at(k), -slice_rowshift<TX>(rowkey, k)));
  atomicMax(&stop[r], top);
  __syncthreads();
  const bool bad = stop[r] == kSliceNonfinite;
  const int e = stop[r] == -kSliceNonfinite ? 0 : stop[r];
  if (threadIdx.x < 8) es[m] = bad ? kSliceBad : slice_scale<L>(e);
  for (int k8 = threadIdx.x >> 3; k8 < 2 * nstage; k8 += 32) {
    double2 v[8];
    int ev[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = 8 * k8 + j;
      v[j] = at(k);
      ev[j] = e - (k < K ? slice_rowshift<TX>(rowkey, k) : 0);
    }
    slice_store<L, double>(v, ev, false, nullptr, slice_b_at<L>(b_img, nstage, nc, m, k8), nc);
  }
}

// ------------------------------------------------------------------------------------------------
// integer sums -> floating point
// ------------------------------------------------------------------------------------------------
// (hi 2^32 + lo) 2^k, rounded to nearest, by integer instructions (the FP64 pipe issues 1/64 of their rate)
__device__ __forceinline__ double slice_to_double(long long hi, long long lo, int k) {
  // 128-bit sum, two's complement
  const unsigned long long h0 = (unsigned long long)hi << 32;
  long long t1 = hi >> 32;
  unsigned long long t0 = h0 + (unsigned long long)lo;
  t1 += (lo >> 63) + (t0 < h0 ? 1 : 0);
  const bool neg = t1 < 0;
  if (neg) {
    t0 = 0ull - t0;
    t1 = ~t1 + (t0 == 0 ? 1 : 0);
  }
  if ((t1 | (long long)t0) == 0) return 0.0;
  // the leading 64 bits m (bit 63 set), value m 2^sh, the rest into a sticky bit
  int sh = 0;
  unsigned long long m;
  if (t1) {
    const int z = __clzll(t1);
    sh = 64 - z;
    m = z ? ((unsigned long long)t1 << z) | (t0 >> (64 - z)) : (unsigned long long)t1;
    if (z < 64 && (t0 << z)) m |= 1ull;
  } else {
    const int z = __clzll((long long)t0);
    sh = -z;
    m = t0 << z;
  }
  int ex = sh + k + 63 + 1023;  // biased exponent of the leading bit
  if (ex >= 2047) return neg ? -INFINITY : INFINITY;
  int drop = 11;
  if (ex <= 0) {  // denormal result
    drop = 12 - ex;
    ex = 0;
    if (drop > 64) return neg ? -0.0 : 0.0;
  }
  unsigned long long q = drop < 64 ? m >> drop : 0ull;
  const unsigned long long rem = drop < 64 ? m << (64 - drop) : m;
  if (rem > (1ull << 63) || (rem == (1ull << 63) && (q & 1ull))) ++q;
  // q holds the leading bit at 52 for normal results: the carry of rounding moves into the exponent
  const unsigned long long bits = ex > 0 ? ((unsigned long long)(ex - 1) << 52) + q : q;
  return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}
// lo 2^k in FP32 (one rounding of the sum's leading 24 bits, one more only for results below 2^-126)
__device__ __forceinline__ float slice_to_float(long long lo, int k) { return ldexpf(__ll2float_rn(lo), k); }

// ------------------------------------------------------------------------------------------------
// the GEMM
// ------------------------------------------------------------------------------------------------
namespace tc {
// Instruction descriptor of kind::f16 with bf16 operands: D FP32, both K-major, M x N tile.
__host__ __device__ constexpr uint32_t idesc_bf16(uint32_t M, uint32_t N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}
// 1 in one lane of a converged warp, 0 in the others. The compiler knows the result for what it is and keeps
// the operands of the instructions it guards in uniform registers: 53 instead of 78 cycles per MMA here.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "elect.sync _|p, 0xffffffff;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(r));
  return r;
}
// executed by a whole warp, issued by the lane whose leader is nonzero
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate, uint32_t leader) {
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.u32 p, %4, 0;\n"
      "setp.ne.u32 q, %5, 0;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
      : "memory");
}
// no-swizzle K-major descriptor (smem_desc with lbo 128, sbo 256) from its low word
__device__ __forceinline__ uint64_t desc_lo(uint32_t lo) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"((256u >> 4) | 1u << 14));
  return d;
}
// 32 lanes x 16 columns, not waited for
__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_x8_async(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
}  // namespace tc

// acc += v * W (one wide multiply-add)
template <int W> __device__ __forceinline__ void slice_acc(long long& acc, int v) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(v), "n"(W));
}

// MODE 0: part[z][m][n] = C over K slice z (complex double; M x N), herm: tiles wholly left of the diagonal
// are left out. MODE 1: Y[n][m] (+)= C[m][n] (the update: A rows are the long axis of Y), OUT = double or float;
// lower: B is lower triangular and the stages past a tile's last row are left out.
// Persistent: a CTA takes the tiles blockIdx.x, + gridDim.x, .. (column tiles fastest, so that CTAs in flight
// share the long operand's tile in L2). The roles run ahead of each other across tiles: while the eight
// epilogue warps convert and store a tile from their registers, the next tile's operands and MMAs are under way.
struct SliceTiles {
  int nt, mt, nz;        // column tiles, row tiles, K slices
  int nstage, kstages;   // stages in all, stages per K slice
  int herm, lower;
  int per_z;             // tiles of one K slice (Hermitian: those not wholly left of the diagonal)
};
template <int NC> struct SliceTile {
  int nt, mt, z, st0, nst;
  __device__ __forceinline__ SliceTile(const SliceTiles& g, int t) {
    z = t / g.per_z;
    int r = t - z * g.per_z;
    if (g.herm) {  // row tile mt starts at the column tile of its first row
      for (mt = 0;; ++mt) {
        const int n0 = mt * kSliceM / NC;
        if (r < g.nt - n0) {
          nt = n0 + r;
          break;
        }
        r -= g.nt - n0;
      }
    } else {
      mt = r / g.nt;
      nt = r - mt * g.nt;
    }
    st0 = z * g.kstages;
    nst = max(0, min(g.kstages, g.nstage - st0));
    if (g.lower) nst = min(nst, (nt * NC + NC + kSliceK - 1) / kSliceK);  // b_n,k = 0 for k > n
  }
};

template <int L, int NC, int MODE, typename OUT>
__global__ void __launch_bounds__(kSliceThreads, 1)
    k_slice_gemm(int M, int N, SliceTiles geo, const unsigned char* __restrict__ a_img, const int* __restrict__ ea,
                 int ea_ld, const unsigned char* __restrict__ b_img, const int* __restrict__ eb, int eb_ld,
                 cplx<OUT>* __restrict__ out, int ldo, int accum, uint32_t polls, int* __restrict__ err) {
  using Cfg = SliceCfg<L>;
  constexpr int PMAX = Cfg::PMAX, CH = Cfg::CH, NS = Cfg::NS, NG = PMAX - 1;
  constexpr int AB = slice_a_bytes<L>(), BB = slice_b_bytes<L>(NC), BUF = AB + BB;
  constexpr int HC = NC / 2;                 // columns per epilogue thread
  constexpr int NSUM = NG > 4 ? 2 : 1;       // 64-bit sums per value (four groups each)
  static_assert(2 * NC * NG <= 512 && HC % 8 == 0, "tensor memory columns");
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  unsigned char* smem = tc_align1024(smem_dyn);
  __shared__ uint64_t full[NS], freeb[NS], gfull[NG], gfree[NG], done;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail, s_last_copy[NS];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int ntiles = geo.per_z * geo.nz;
  if (tid == 0) {
    for (int b = 0; b < NS; ++b) {
      tc::mbar_init(&full[b], 1);
      tc::mbar_init(&freeb[b], 1);
      s_last_copy[b] = -1;
    }
    for (int g = 0; g < NG; ++g) {
      tc::mbar_init(&gfull[g], 1);
      tc::mbar_init(&gfree[g], kSliceThreads - 64);
    }
    tc::mbar_init(&done, 1);
    s_fail = 0;
    tc::fence_mbar_init();
  }
  if (warp == 1) {
    tc::tmem_alloc(&tmem_base, 512u);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
  volatile int* vfail = &s_fail;
  // sg: stages so far (buffer sg % NS), cg: chunks so far (parity of the group barriers); every role counts alike
  if (tid == 0) {  // operand tiles: two bulk copies per stage
    int sg = 0;
    for (int t = blockIdx.x; t < ntiles && !*vfail; t += gridDim.x) {
      const SliceTile<NC> tl(geo, t);
      for (int s = 0; s < tl.nst && !*vfail; ++s, ++sg) {
        const int b = sg % NS;
        if (sg >= NS && !tc::mbar_wait(&freeb[b], (uint32_t)(sg / NS - 1) & 1u, polls)) {
          *vfail = 1;
          break;
        }
        tc::mbar_arrive_expect_tx(&full[b], (uint32_t)BUF);
        tc::bulk_g2s(smem + b * BUF, a_img + ((size_t)tl.mt * geo.nstage + tl.st0 + s) * AB, (uint32_t)AB, &full[b]);
        tc::bulk_g2s(smem + b * BUF + AB, b_img + ((size_t)tl.nt * geo.nstage + tl.st0 + s) * BB, (uint32_t)BB,
                     &full[b]);
        s_last_copy[b] = sg;
      }
    }
  } else if (warp == 1) {  // the MMAs: group by group, so that a chunk's first groups drain while its last are formed
    const uint32_t leader = tc::elect_one();
    constexpr uint32_t idesc = tc::idesc_bf16(128, 2 * NC);
    int sg = 0, cg = 0;
    bool okg = true;
    for (int t = blockIdx.x; t < ntiles && okg; t += gridDim.x) {
      const SliceTile<NC> tl(geo, t);
      for (int s = 0; s < tl.nst && okg; ++s, ++sg) {
        const int b = sg % NS, ch = cg + s / CH;
        const bool first = s % CH == 0, last = s % CH == CH - 1 || s == tl.nst - 1;
        // votes keep the loop's control flow, and with it the descriptors, uniform over the warp
        okg = __all_sync(0xffffffffu, !*vfail && tc::mbar_wait(&full[b], (uint32_t)(sg / NS) & 1u, polls));
        if (!okg) break;
        tc::tc_fence_after();
        // descriptors by their low words: the stage's base plus constant offsets (in 16 bytes); the issuing
        // warp's instructions per MMA are what the tensor pipe would otherwise wait for
        const uint32_t a0 = (tc::smem_addr(smem + b * BUF) >> 4) | (128u >> 4) << 16, b0 = a0 + (uint32_t)(AB >> 4);
#pragma unroll
        for (int g = 2; g <= PMAX; ++g) {
          if (first && ch > 0 && okg) {
            okg = __all_sync(0xffffffffu, tc::mbar_wait(&gfree[g - 2], (uint32_t)(ch - 1) & 1u, polls));
            tc::tc_fence_after();
          }
          if (okg) {
            const uint32_t d = tm + (uint32_t)((g - 2) * 2 * NC);
#pragma unroll
            for (int i = g > L ? g - L : 1; i <= (g > L ? L : g - 1); ++i) {
              const uint32_t ai = a0 + (uint32_t)((i - 1) * 2 * (kSliceM * kSliceK * 2) >> 4);
              const uint32_t bj = b0 + (uint32_t)((g - i - 1) * 3 * (NC * kSliceK * 2) >> 4);
              tc::mma_bf16(d, tc::desc_lo(ai), tc::desc_lo(bj), idesc, first && i == (g > L ? g - L : 1) ? 0u : 1u,
                           leader);
              tc::mma_bf16(d, tc::desc_lo(ai + (kSliceM * kSliceK * 2 >> 4)),
                           tc::desc_lo(bj + (NC * kSliceK * 2 >> 4)), idesc, 1u, leader);
            }
            if (last && leader) tc::mma_commit(&gfull[g - 2]);
          }
        }
        if (!okg) break;
        if (leader) tc::mma_commit(&freeb[b]);
      }
      cg += (tl.nst + CH - 1) / CH;
    }
    // every MMA issued so far, those of a stage that was given up among them
    if (leader) tc::mma_commit(&done);
    if (!okg) *vfail = 1;
  } else if (warp >= 2) {  // the sums: TMEM lanes 32 (warp % 4) .., columns HC half .. of Re and of Im
    constexpr int PC = HC % 16 == 0 ? 16 : 8;  // columns per read
    const uint32_t base = tm + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(((warp - 2) >> 2) * HC);
    int cg = 0;
    bool okc = true;
    for (int t = blockIdx.x; t < ntiles && okc; t += gridDim.x) {
      const SliceTile<NC> tl(geo, t);
      const int nchunk = (tl.nst + CH - 1) / CH;
      long long acc[NSUM][2][HC];
#pragma unroll
      for (int q = 0; q < NSUM; ++q)
#pragma unroll
        for (int j = 0; j < HC; ++j) acc[q][0][j] = acc[q][1][j] = 0;
      for (int ch = 0; ch < nchunk && okc; ++ch, ++cg) {
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          if (okc && (*vfail || !tc::mbar_wait(&gfull[g], (uint32_t)cg & 1u, polls))) okc = false;
          okc = __all_sync(0xffffffffu, okc);
          if (!okc) continue;
          tc::tc_fence_after();
#pragma unroll
          for (int c0 = 0; c0 < HC; c0 += PC) {
            uint32_t re[PC], im[PC];
            if constexpr (PC == 16) {
              tc::tmem_ld_x16(base + (uint32_t)(g * 2 * NC + c0), re);
              tc::tmem_ld_x16(base + (uint32_t)(g * 2 * NC + NC + c0), im);
            } else {
              tc::tmem_ld_x8_async(base + (uint32_t)(g * 2 * NC + c0), re);
              tc::tmem_ld_x8_async(base + (uint32_t)(g * 2 * NC + NC + c0), im);
            }
            tc::tmem_ld_wait();
            if (c0 + PC == HC) {
              tc::tc_fence_before();
              tc::mbar_arrive(&gfree[g]);
            }
#pragma unroll
            for (int j = 0; j < PC; ++j) {
              // weight 256^(PMAX - g): four groups per 64-bit sum
              constexpr int kW[4] = {1 << 24, 1 << 16, 1 << 8, 1};
              const int ir = __float2int_rn(__uint_as_float(re[j])), ii = __float2int_rn(__uint_as_float(im[j]));
              long long &ar = acc[NSUM == 2 ? g / 4 : 0][0][c0 + j], &ai = acc[NSUM == 2 ? g / 4 : 0][1][c0 + j];
              if (g % 4 == 0) { slice_acc<kW[0]>(ar, ir); slice_acc<kW[0]>(ai, ii); }
              if (g % 4 == 1) { slice_acc<kW[1]>(ar, ir); slice_acc<kW[1]>(ai, ii); }
              if (g % 4 == 2) { slice_acc<kW[2]>(ar, ir); slice_acc<kW[2]>(ai, ii); }
              if (g % 4 == 3) { slice_acc<kW[3]>(ar, ir); slice_acc<kW[3]>(ai, ii); }
            }
          }
        }
      }
      const int row = tl.mt * kSliceM + 32 * (warp & 3) + lane, n0 = tl.nt * NC + ((warp - 2) >> 2) * HC;
      const int sa = row < M ? ea[(size_t)tl.z * ea_ld + row] : 0;
      const int* ebz = eb + (size_t)tl.z * eb_ld;
      constexpr int JB = sizeof(OUT) == 8 ? 4 : 8;  // loads in flight before their first store
      if (okc && row < M)
#pragma unroll
      for (int j0 = 0; j0 < HC; j0 += JB) {
        cplx<OUT> old[JB];
        if constexpr (MODE == 1) {
#pragma unroll
          for (int j = 0; j < JB; ++j) {
            const int n = n0 + j0 + j;
            old[j] = accum && n < N ? out[(size_t)n * ldo + row] : mk<OUT>(0, 0);
          }
        }
#pragma unroll
        for (int j = 0; j < JB; ++j) {
          const int n = n0 + j0 + j, i = j0 + j;
          if (n >= N) continue;
          const int sb = ebz[n];
          cplx<OUT> v;
          if (sa == kSliceBad || sb == kSliceBad) v = mk<OUT>(NAN, NAN);
          else if constexpr (std::is_same<OUT, float>::value)
            v = mk<OUT>(slice_to_float(acc[0][0][i], sa + sb), slice_to_float(acc[0][1][i], sa + sb));
          else if constexpr (NSUM == 2)
            v = mk<OUT>(slice_to_double(acc[0][0][i], acc[NSUM - 1][0][i], sa + sb),
                        slice_to_double(acc[0][1][i], acc[NSUM - 1][1][i], sa + sb));
          else
            v = mk<OUT>(slice_to_double(0, acc[0][0][i], sa + sb), slice_to_double(0, acc[0][1][i], sa + sb));
          if constexpr (MODE == 0) out[((size_t)tl.z * M + row) * N + n] = v;
          else out[(size_t)n * ldo + row] = accum ? cadd(old[j], v) : v;
        }
      }
      __syncwarp();
    }
    if (!okc) *vfail = 1;
  }
  __syncthreads();
  // every MMA has read its operands and written tensor memory, and every copy has landed, before the CTA gives
  // either up (after a time-out too)
  int ok = !*vfail;
  if (!tc::mbar_wait(&done, 0u, kSlicePolls)) ok = 0;
  if (tid == 0)
    for (int b = 0; b < NS; ++b)
      if (s_last_copy[b] >= 0 && !tc::mbar_wait(&full[b], (uint32_t)(s_last_copy[b] / NS) & 1u, kSlicePolls)) ok = 0;
  ok = __syncthreads_and(ok);
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem_base, 512u);
  }
  if (!ok && tid == 0) atomicExch(err, 1);
}

// C[m][n] = sum of the slices' partials; elements whose tile was skipped are the conjugate of their mirror
__global__ void k_slice_reduce(int M, int N, int nz, const double2* __restrict__ part, double2* __restrict__ C,
                               int ldc, int herm, int nc) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= M * N) return;
  const int m = idx / N, n = idx - m * N;
  const bool mirror = herm && n / nc * nc + nc - 1 < m / kSliceM * kSliceM;
  const size_t off = mirror ? (size_t)n * N + m : (size_t)m * N + n;
  double2 s = make_double2(0.0, 0.0);
  for (int z = 0; z < nz; ++z) s = cadd(s, part[(size_t)z * M * N + off]);
  C[(size_t)m * ldc + n] = mirror ? cconj(s) : s;
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
static const int kSliceSms = 152;  // one CTA per SM (its tensor memory is full)
template <typename T> struct SliceL { static constexpr int value = sizeof(T) == 8 ? 7 : 4; };

template <int L, int NC, int MODE, typename OUT>
static int slice_launch_nc(Ctx* c, int M, int N, const SliceTiles& geo, const unsigned char* a, const int* ea, int ea_ld,
                           const unsigned char* b, const int* eb, int eb_ld, cplx<OUT>* out, int ldo, bool accum) {
  int* err = tc_err_flag(c);
  if (!err) return PARO_ERR_CUDA;
  const size_t sm = (size_t)SliceCfg<L>::NS * (slice_a_bytes<L>() + slice_b_bytes<L>(NC)) + 1024;
  static int attr_dev = -1;
  int dev = 0;
  PARO_CU(c, cudaGetDevice(&dev));
  if (attr_dev != dev) {
    PARO_CU(c, cudaFuncSetAttribute(k_slice_gemm<L, NC, MODE, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sm));
    attr_dev = dev;
  }
  const int tiles = geo.per_z * geo.nz;
  k_slice_gemm<L, NC, MODE, OUT><<<std::min(tiles, kSliceSms), kSliceThreads, sm, c->stream>>>(
      M, N, geo, a, ea, ea_ld, b, eb, eb_ld, out, ldo, accum, slice_polls(), err);
  PARO_LAUNCH(c, "k_slice_gemm");
  return PARO_OK;
}
template <int L, int MODE, typename OUT>
static int slice_launch(Ctx* c, int nc, int M, int N, const SliceTiles& geo, const unsigned char* a, const int* ea,
                        int ea_ld, const unsigned char* b, const int* eb, int eb_ld, cplx<OUT>* out, int ldo,
                        bool accum) {
  if constexpr (L == 7) {
    return slice_launch_nc<7, 32, MODE, OUT>(c, M, N, geo, a, ea, ea_ld, b, eb, eb_ld, out, ldo, accum);
  } else {
    if (nc == 48) return slice_launch_nc<4, 48, MODE, OUT>(c, M, N, geo, a, ea, ea_ld, b, eb, eb_ld, out, ldo, accum);
    return slice_launch_nc<4, 64, MODE, OUT>(c, M, N, geo, a, ea, ea_ld, b, eb, eb_ld, out, ldo, accum);
  }
}

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

template <typename T, int L>
static int slice_rows(Ctx* c, int rows, int rows_a, int rows_b, int pad, int K, int kslice, int nz, int nstage,
                      const cplx<T>* x, int ld, unsigned char* a_img, unsigned char* b_img, int* es,
                      const int* rowkey = nullptr, int nc = 64) {
  const int stage = std::min(kslice, SliceStage<T>::value);
  k_slice_rows<T, L><<<dim3(pad / 8, nz), 256, (size_t)8 * (stage + 1) * sizeof(cplx<T>), c->stream>>>(
      rows, rows_a, rows_b, K, kslice, nstage, x, ld, 0, a_img, b_img, es, pad, stage, rowkey, nc);
  PARO_LAUNCH(c, "k_slice_rows");
  return PARO_OK;
}

template <typename T>
static int slice_rowkeys(Ctx* c, int rows, int n, const cplx<T>* x, int ld, bool finite, int* rowkey) {
  PARO_CU(c, cudaMemsetAsync(rowkey, 0, (size_t)rows * sizeof(int), c->stream));
  const int seg = std::max(1, std::min((n + 1023) / 1024, 2048 / rows));
  k_slice_rowkey<T><<<dim3(seg, rows), 256, 0, c->stream>>>(n, x, ld, finite, rowkey);
  PARO_LAUNCH(c, "k_slice_rowkey");
  return PARO_OK;
}

// K slices of the long-K product: the count that minimises waves of 152 CTAs times (stages + the stages' worth
// of a CTA's start and a tile's conversion, about 4)
static int slice_split_k(int tiles, int nstage) {
  int best_nz = 1;
  long long best = -1;
  for (int nz = 1; nz <= std::max(1, nstage / 4); ++nz) {
    const int ks = (nstage + nz - 1) / nz, z = (nstage + ks - 1) / ks;
    const long long cost = ((long long)tiles * z + 151) / 152 * (ks + 4) * 64 + z;  // ties: fewer slices
    if (best < 0 || cost < best) {
      best = cost;
      best_nz = z;
    }
  }
  return best_nz;
}

// C = conj(A) B^T with A given as an image (scales ea[row], the same for every K slice) or as rows
template <typename T>
static int slice_cn(Ctx* c, int M, int N, int K, const cplx<T>* A, int lda, const unsigned char* a_img, const int* ea,
                    const cplx<T>* B, int ldb, double2* C, int ldc, bool herm) {
  constexpr int L = SliceL<T>::value;
  const int NC = slice_nc<L>(N);
  const int mt = (M + kSliceM - 1) / kSliceM, nt = (N + NC - 1) / NC, nstage = (K + kSliceK - 1) / kSliceK;
  int tiles = mt * nt;
  if (herm)
    for (int i = 0; i < mt; ++i) tiles -= std::min(nt, i * kSliceM / NC);
  int nz = slice_split_k(tiles, nstage);
  const int ks = (nstage + nz - 1) / nz;
  nz = (nstage + ks - 1) / ks;
  const int ma = mt * kSliceM, nb = nt * NC;
  const bool same = !a_img && A == B && lda == ldb && M == N;
  const int pad = same ? std::max(ma, nb) : nb;
  OptionalInUse use(c);
  unsigned char* bi = static_cast<unsigned char*>(ws_try(c, "slice_b", (size_t)nt * nstage * slice_b_bytes<L>(NC)));
  int* eb = static_cast<int*>(ws_try(c, "slice_eb", (size_t)nz * pad * sizeof(int)));
  double2* part = static_cast<double2*>(ws_try(c, "gemm_parts", (size_t)nz * M * N * sizeof(double2)));
  if (!bi || !eb || !part) return kNoMemory;
  unsigned char* ai = nullptr;
  int* ean = nullptr;
  if (!a_img) {
    ai = static_cast<unsigned char*>(ws_try(c, "slice_a", (size_t)mt * nstage * slice_a_bytes<L>()));
    ean = same ? eb : static_cast<int*>(ws_try(c, "slice_ea", (size_t)nz * ma * sizeof(int)));
    if (!ai || !ean) return kNoMemory;
  }
  cudaEvent_t ev = prof_begin(c);
  int st;
  if (!a_img && !same && (st = slice_rows<T, L>(c, M, ma, 0, ma, K, ks * kSliceK, nz, nstage, A, lda, ai, nullptr, ean)))
    return st;
  if ((st = slice_rows<T, L>(c, N, same ? ma : 0, nb, pad, K, ks * kSliceK, nz, nstage, B, ldb, same ? ai : nullptr, bi, eb,
                             nullptr, NC)))
    return st;
  prof_end(c, sizeof(T) == 8 ? "k_slice_rows<f64>" : "k_slice_rows<f32>", ev);
  ev = prof_begin(c);
  const SliceTiles geo{nt, mt, nz, nstage, ks, herm ? 1 : 0, 0, tiles};
  st = slice_launch<L, 0, double>(c, NC, M, N, geo, a_img ? a_img : ai, a_img ? ea : ean,
                                  a_img ? 0 : (same ? pad : ma), bi, eb, pad, part, 0, false);
  if (st) return st;
  prof_end(c, sizeof(T) == 8 ? "k_slice_gemm_cn<f64>" : "k_slice_gemm_cn<f32>", ev);
  k_slice_reduce<<<(M * N + 255) / 256, 256, 0, c->stream>>>(M, N, nz, part, C, ldc, herm, NC);
  PARO_LAUNCH(c, "k_slice_reduce");
  return PARO_OK;
}

template <typename T>
int gemm_cn_slice(Ctx* c, int M, int N, int K, const cplx<T>* A, int lda, const cplx<T>* B, int ldb, double2* C,
                  int ldc, bool herm) {
  return slice_cn<T>(c, M, N, K, A, lda, nullptr, nullptr, B, ldb, C, ldc, herm);
}

// Y (+)= sum_k s_k W(k, m) X[k][n] with X given as rows or as an image of its columns
template <typename T>
static int slice_wx(Ctx* c, int M, int N, int K, const double2* W, int ldw, bool wt, const double* s, const cplx<T>* X,
                    int ldx, const unsigned char* a_img, const int* ea, cplx<T>* Y, int ldy, bool accum, bool lower) {
  constexpr int L = SliceL<T>::value;
  const int NC = slice_nc<L>(M);
  const int at = (N + kSliceM - 1) / kSliceM, bt = (M + NC - 1) / NC, nstage = (K + kSliceK - 1) / kSliceK;
  OptionalInUse use(c);
  unsigned char* bi = static_cast<unsigned char*>(ws_try(c, "slice_b", (size_t)bt * nstage * slice_b_bytes<L>(NC)));
  int* eb = static_cast<int*>(ws_try(c, "slice_eb", (size_t)bt * NC * sizeof(int)));
  if (!bi || !eb) return kNoMemory;
  unsigned char* ai = nullptr;
  int *ean = nullptr, *rowkey = nullptr;
  if (!a_img) {
    ai = static_cast<unsigned char*>(ws_try(c, "slice_a", (size_t)at * nstage * slice_a_bytes<L>()));
    ean = static_cast<int*>(ws_try(c, "slice_ea", (size_t)at * kSliceM * sizeof(int)));
    rowkey = static_cast<int*>(ws_try(c, "slice_rowkey", (size_t)std::max(K, 1) * sizeof(int)));
    if (!ai || !ean || !rowkey) return kNoMemory;
  }
  cudaEvent_t ev = prof_begin(c);
  if (!a_img) {
    if (int st = slice_rowkeys<T>(c, K, N, X, ldx, true, rowkey)) return st;
    k_slice_cols<T, L><<<at * kSliceM / 32, 256, 0, c->stream>>>(N, K, nstage, X, ldx, rowkey, ai, ean);
    PARO_LAUNCH(c, "k_slice_cols");
    a_img = ai;
    ea = ean;
  }
  k_slice_w<L, T><<<bt * NC / 8, 256, 0, c->stream>>>(M, K, nstage, W, ldw, wt ? 1 : 0, s, rowkey, bi, eb, NC);
  PARO_LAUNCH(c, "k_slice_w");
  prof_end(c, sizeof(T) == 8 ? "k_slice_cols<f64>" : "k_slice_cols<f32>", ev);
  ev = prof_begin(c);
  const SliceTiles geo{bt, at, 1, nstage, nstage, 0, lower ? 1 : 0, bt * at};
  int st = slice_launch<L, 1, T>(c, NC, N, M, geo, a_img, ea, 0, bi, eb, 0, Y, ldy, accum);
  if (st) return st;
  prof_end(c, sizeof(T) == 8 ? "k_slice_gemm_wx<f64>" : "k_slice_gemm_wx<f32>", ev);
  return PARO_OK;
}

template <typename T>
int gemm_wx_slice(Ctx* c, int M, int N, int K, const double2* W, int ldw, bool wt, const double* s, const cplx<T>* X,
                  int ldx, cplx<T>* Y, int ldy, bool accum, bool lower) {
  return slice_wx<T>(c, M, N, K, W, ldw, wt, s, X, ldx, nullptr, nullptr, Y, ldy, accum, lower);
}

// ---- the projectors as the fixed operand: their images change only with the atom positions ----
// 32 bytes an entry of the projectors' table in FP32, 56 in FP64 (512 atoms in FP32: 9 GB beside a table of 2.2).
template <typename T> static const cplx<T>* slice_beta(const Basis& b);
template <> const double2* slice_beta<double>(const Basis& b) { return b.d_beta; }
template <> const float2* slice_beta<float>(const Basis& b) { return b.d_beta32; }

template <typename T>
static int slice_form_beta(Ctx* c, const Basis& B, const SliceImages& im, int* rowkey, int ma, int na, int scn,
                           int swx) {
  constexpr int L = SliceL<T>::value;
  const int np = c->nproj, npw = B.npw;
  int st = slice_rowkeys<T>(c, np, npw, slice_beta<T>(B), npw, false, rowkey);
  if (st) return st;
  const int nzi = std::max(1, std::min((npw + 511) / 512, 1216 / (ma / 8)));
  const int ksi = (scn + nzi - 1) / nzi;
  if ((st = slice_rows<T, L>(c, np, ma, 0, ma, npw, ksi * kSliceK, (scn + ksi - 1) / ksi, scn, slice_beta<T>(B), npw,
                             im.cn, nullptr, im.ecn, rowkey)))
    return st;
  k_slice_cols<T, L><<<na / 32, 256, 0, c->stream>>>(npw, np, swx, slice_beta<T>(B), npw, nullptr, im.wx,
                                                        im.ewx);
  PARO_LAUNCH(c, "k_slice_cols");
  return PARO_OK;
}

template <typename T>
static int slice_beta_images(Ctx* c, int ik) {
  constexpr int L = SliceL<T>::value, q = sizeof(T) == 8 ? 1 : 0;
  Basis& B = c->bases[ik];
  if (B.beta_slices[q].cn) return PARO_OK;
  const int np = c->nproj, npw = B.npw;
  const int ma = round_up(np, kSliceM), na = round_up(npw, kSliceM);
  const int scn = (npw + kSliceK - 1) / kSliceK, swx = (np + kSliceK - 1) / kSliceK;
  const size_t bcn = (size_t)(ma / kSliceM) * scn * slice_a_bytes<L>();
  const size_t bwx = (size_t)(na / kSliceM) * swx * slice_a_bytes<L>();
  int* rowkey = static_cast<int*>(ws_try(c, "slice_rowkey", (size_t)np * sizeof(int)));
  unsigned char* p = nullptr;  // [cn image | wx image | cn scales | wx scales]
  if (!rowkey || cudaMalloc(&p, bcn + bwx + (size_t)(ma + na) * sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return kNoMemory;
  }
  SliceImages im;
  im.cn = p;
  im.wx = p + bcn;
  im.ecn = reinterpret_cast<int*>(p + bcn + bwx);
  im.ewx = im.ecn + ma;
  if (int st = slice_form_beta<T>(c, B, im, rowkey, ma, na, scn, swx)) {
    cudaStreamSynchronize(c->stream);
    cudaFree(p);
    return st;
  }
  B.beta_slices[q] = im;  // marks the images as formed
  return PARO_OK;
}

template <typename T>
int kb_project_slice(Ctx* c, int ik, int nb, const cplx<T>* psi, double2* P) {
  OptionalInUse use(c);
  int st = slice_beta_images<T>(c, ik);
  if (st) return st;
  const Basis& B = c->bases[ik];
  const SliceImages& im = B.beta_slices[sizeof(T) == 8 ? 1 : 0];
  return slice_cn<T>(c, c->nproj, nb, B.npw, nullptr, 0, im.cn, im.ecn, psi, B.npw, P, nb, false);
}

template <typename T>
int kb_update_slice(Ctx* c, int ik, int nb, const double2* P, cplx<T>* hpsi) {
  OptionalInUse use(c);
  int st = slice_beta_images<T>(c, ik);
  if (st) return st;
  const Basis& B = c->bases[ik];
  const SliceImages& im = B.beta_slices[sizeof(T) == 8 ? 1 : 0];
  return slice_wx<T>(c, nb, B.npw, c->nproj, P, nb, false, c->d_dvec, nullptr, 0, im.wx, im.ewx, hpsi, B.npw, true,
                     false);
}

template int gemm_cn_slice<double>(Ctx*, int, int, int, const double2*, int, const double2*, int, double2*, int, bool);
template int gemm_wx_slice<double>(Ctx*, int, int, int, const double2*, int, bool, const double*, const double2*, int,
                                   double2*, int, bool, bool);
template int kb_project_slice<double>(Ctx*, int, int, const double2*, double2*);
template int kb_project_slice<float>(Ctx*, int, int, const float2*, double2*);
template int kb_update_slice<double>(Ctx*, int, int, const double2*, double2*);
template int kb_update_slice<float>(Ctx*, int, int, const double2*, float2*);

}  // namespace paro
