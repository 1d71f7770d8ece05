// Complex FP32 products on the tensor cores (tcgen05, kind::tf32) with the 3xTF32 split: every FP32
// operand x = hi + lo (hi, lo TF32), a b ~ ah bh + ah bl + al bh accumulated in FP32 in tensor memory;
// the dropped al bl and the rounding of lo keep the product within a few FP32 ulps.
//
// Complex arithmetic as real products on the interleaved storage: a row of complex values
// (re0, im0, re1, im1, ...) is a real row of twice the length, so for C = conj(A) B^T
//   Re C = A' . B'              (A', B' the interleaved rows)
//   Im C = A'' . B',  A'' = (-im0, re0, -im1, re1, ...)
// The products are those with the projectors as the fixed operand (k_tc_beta.cu). This file holds what they share: the
// presplit of the small matrix, the K split and the reduction of its parts.
#include <algorithm>

#include "paro_ctx.h"
#include "tc_sm100.cuh"

namespace paro {

static const int kTcM = 128;       // rows of A per CTA = TMEM lanes

static const int kCnKC = 8;

// C[m][n] = sum over z of part[z][m][n] in a fixed order, added into an FP32 two-sum pair (no FP64 pipe)
__global__ void k_reduce_parts32(int M, int N, int nz, const float2* __restrict__ part, double2* __restrict__ C,
                                 int ldc) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= M * N) return;
  float hx = 0.f, lx = 0.f, hy = 0.f, ly = 0.f;
  for (int z = 0; z < nz; ++z) {
    const float2 v = part[(size_t)z * M * N + idx];
    two_sum_acc(hx, lx, v.x);
    two_sum_acc(hy, ly, v.y);
  }
  const int m = idx / N, n = idx - m * N;
  C[(size_t)m * ldc + n] = make_double2((double)hx + (double)lx, (double)hy + (double)ly);
}

// The small matrix of the update product B[m][k] = s_k W(k, m) (W(k, m) at W[k ldw + m], or W[m ldw + k] when wt) as
// the four tiles of every stage, Re D = A' . (Br, -Bi)' and Im D = A' . (Bi, Br)', split once per call.
__global__ void k_wx_presplit(int M, int K, int NT, int KC, const double2* __restrict__ W, int ldw, int wt,
                              const double* __restrict__ sc, float4* __restrict__ Wp) {
  const int ch = KC / 2, nstage = (K + KC - 1) / KC;
  const int mt = blockIdx.y;  // M tile
  const size_t tile = (size_t)NT * ch;  // float4 per variant per stage
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < (size_t)nstage * tile;
       i += (size_t)gridDim.x * blockDim.x) {
    const int st = (int)(i / tile);
    const int rem = (int)(i - (size_t)st * tile);
    const int r = rem / ch, c = rem - r * ch;
    const int gm = mt * NT + r, k0 = st * KC + 2 * c;
    float2 b0 = make_float2(0.f, 0.f), b1 = b0;
    if (gm < M) {
      if (k0 < K) {
        const double2 w = wt ? W[(size_t)gm * ldw + k0] : W[(size_t)k0 * ldw + gm];
        const double f = sc ? sc[k0] : 1.0;
        b0 = make_float2((float)(f * w.x), (float)(f * w.y));
      }
      if (k0 + 1 < K) {
        const double2 w = wt ? W[(size_t)gm * ldw + k0 + 1] : W[(size_t)(k0 + 1) * ldw + gm];
        const double f = sc ? sc[k0 + 1] : 1.0;
        b1 = make_float2((float)(f * w.x), (float)(f * w.y));
      }
    }
    float4 h, l;
    tc_split(b0, b1, h, l);
    const size_t base = (((size_t)mt * nstage + st) * 4) * tile;
    const uint32_t o = tc_off(r, c, ch) / 16;  // float4 index within a variant tile
    Wp[base + 0 * tile + o] = make_float4(h.x, -h.y, h.z, -h.w);  // Re, hi
    Wp[base + 1 * tile + o] = make_float4(l.x, -l.y, l.z, -l.w);  // Re, lo
    Wp[base + 2 * tile + o] = make_float4(h.y, h.x, h.w, h.z);    // Im, hi
    Wp[base + 3 * tile + o] = make_float4(l.y, l.x, l.w, l.z);    // Im, lo
  }
}

// K split of the tensor-core product: one CTA per SM, the slice count minimising waves x stages per
// slice (at least 4 stages per slice), and no slice longer than 8192 complex terms, so the FP32 sum in
// tensor memory stays short (slices are added in an FP32 two-sum pair).
void tc_cn_plan(int M, int N, int K, int* nz_out, int* kslice_out) {
  const int ntiles = (N + 255) / 256;
  const int mtiles = (M + kTcM - 1) / kTcM;
  const int tiles = mtiles * ntiles;
  const int kc = kCnKC;
  const int steps = (K + kc - 1) / kc;
  const int maxz = std::max(1, steps / 4);
  const int minz = (steps + 8192 / kc - 1) / (8192 / kc);
  int best_nz = minz;
  long long best = -1;
  for (int z = std::min(minz, maxz); z <= std::min(std::max(maxz, minz), 1024); ++z) {
    const int s = (steps + z - 1) / z;
    const int zz = (steps + s - 1) / s;
    const long long cost = (long long)((tiles * zz + 151) / 152) * s;
    if (best < 0 || cost < best) {
      best = cost;
      best_nz = zz;
    }
  }
  const int kslice = ((steps + best_nz - 1) / best_nz) * kc;
  *kslice_out = kslice;
  *nz_out = std::max(1, (K + kslice - 1) / kslice);
}

int reduce_parts32(Ctx* c, int M, int N, int nz, const float2* part, double2* C, int ldc) {
  k_reduce_parts32<<<(M * N + 255) / 256, 256, 0, c->stream>>>(M, N, nz, part, C, ldc);
  PARO_LAUNCH(c, "k_reduce_parts32");
  return PARO_OK;
}

int wx_presplit(Ctx* c, int M, int K, int NT, int KC, const double2* W, int ldw, bool wt, const double* s,
                float4* Wp) {
  const int mtiles = (M + NT - 1) / NT;
  k_wx_presplit<<<dim3(64, mtiles), 256, 0, c->stream>>>(M, K, NT, KC, W, ldw, wt ? 1 : 0, s, Wp);
  PARO_LAUNCH(c, "k_wx_presplit");
  return PARO_OK;
}

}  // namespace paro
