// Per-voxel pieces of the tangent passes (cg.cu, tangent_rows.cu): the
// matrix-free FP32 tangents from H = F - I and the dot-product accumulator.
#pragma once

#include "launch.h"

namespace {

// Per-thread dot-product accumulator: exact FP32 products (two-product by FMA)
// summed with Neumaier compensation in FP32; the thread totals are then
// combined in FP64.  FP64 arithmetic per element would cost as much as the
// whole pass on a part whose FP64 rate is 1/57 of its FP32 rate.
struct Dot32 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add_term(float v) {
    const float t = s + v;
    c += (fabsf(s) >= fabsf(v)) ? ((s - t) + v) : ((v - t) + s);
    s = t;
  }
  __device__ __forceinline__ void add_prod(float a, float b) {
    const float p = a * b;
    add_term(p);
    add_term(fmaf(a, b, -p));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

__device__ __forceinline__ constexpr int vgt(int i, int j) {
  return i == j ? i : (i + j == 3 ? 3 : (i + j == 2 ? 4 : 5));
}

// t = K : q for St Venant-Kirchhoff from H = F - I and a 6x6 Voigt stiffness.
__device__ __forceinline__ void svk_apply(const float (&h)[9], const float* __restrict__ C,
                                          const float (&q)[9], float (&t)[9]) {
  float e6[6], d6[6];
  // E = (H + H^T + H^T H)/2 in Voigt form with engineering shears
  float E[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      E[a][b] = 0.5f * (h[3 * a + b] + h[3 * b + a] + h[a] * h[b] + h[3 + a] * h[3 + b] + h[6 + a] * h[6 + b]);
  e6[0] = E[0][0]; e6[1] = E[1][1]; e6[2] = E[2][2];
  e6[3] = 2.f * E[1][2]; e6[4] = 2.f * E[0][2]; e6[5] = 2.f * E[0][1];
  // dE = sym(F^T q), F = I + H
  float D[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
      D[a][b] = q[3 * a + b] + h[a] * q[b] + h[3 + a] * q[3 + b] + h[6 + a] * q[6 + b];  // (F^T q)_ab
  d6[0] = D[0][0]; d6[1] = D[1][1]; d6[2] = D[2][2];
  d6[3] = D[1][2] + D[2][1]; d6[4] = D[0][2] + D[2][0]; d6[5] = D[0][1] + D[1][0];
  float sv[6], dv[6];
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int J = 0; J < 6; ++J) { a += C[6 * I + J] * e6[J]; b += C[6 * I + J] * d6[J]; }
    sv[I] = a; dv[I] = b;
  }
  // t = q S + F dS
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      float acc = dv[vgt(i, j)];
#pragma unroll
      for (int k = 0; k < 3; ++k) acc += q[3 * i + k] * sv[vgt(k, j)] + h[3 * i + k] * dv[vgt(k, j)];
      t[3 * i + j] = acc;
    }
}

// t = K : q for the neo-Hookean law from H = F - I.
__device__ __forceinline__ void neohooke_apply(const float (&h)[9], float mu, float lam,
                                               const float (&q)[9], float (&t)[9]) {
  const float f0 = 1.f + h[0], f4 = 1.f + h[4], f8 = 1.f + h[8];
  const float c00 = f4 * f8 - h[5] * h[7];
  const float c01 = h[5] * h[6] - h[3] * f8;
  const float c02 = h[3] * h[7] - f4 * h[6];
  // J - 1 without cancellation: tr H + (tr^2 H - tr H^2)/2 + det H
  const float trH = h[0] + h[4] + h[8];
  const float tr2 = h[0] * h[0] + h[4] * h[4] + h[8] * h[8] +
                    2.f * (h[1] * h[3] + h[2] * h[6] + h[5] * h[7]);
  const float detH = h[0] * (h[4] * h[8] - h[5] * h[7]) - h[1] * (h[3] * h[8] - h[5] * h[6]) +
                     h[2] * (h[3] * h[7] - h[4] * h[6]);
  const float Jm1 = trH + 0.5f * (trH * trH - tr2) + detH;
  const float J = 1.f + Jm1;
  const float iJ = 1.f / J;
  float G[9];
  G[0] = c00 * iJ; G[1] = c01 * iJ; G[2] = c02 * iJ;
  G[3] = (h[2] * h[7] - h[1] * f8) * iJ;
  G[4] = (f0 * f8 - h[2] * h[6]) * iJ;
  G[5] = (h[1] * h[6] - f0 * h[7]) * iJ;
  G[6] = (h[1] * h[5] - h[2] * f4) * iJ;
  G[7] = (h[2] * h[3] - f0 * h[5]) * iJ;
  G[8] = (f0 * f4 - h[1] * h[3]) * iJ;
  const float lnJ = log1pf(Jm1);
  const float c3 = mu - lam * lnJ;
  float gq = 0.f;
#pragma unroll
  for (int c = 0; c < 9; ++c) gq += G[c] * q[c];
  // (G q^T G)_ij = sum_kl G_il q_kl G_kj
  float M[3][3];   // M_lj = sum_k q_kl G_kj = (q^T G)_lj
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int j = 0; j < 3; ++j) M[l][j] = q[l] * G[j] + q[3 + l] * G[3 + j] + q[6 + l] * G[6 + j];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float gqg = G[3 * i] * M[0][j] + G[3 * i + 1] * M[1][j] + G[3 * i + 2] * M[2][j];
      t[3 * i + j] = mu * q[3 * i + j] + lam * gq * G[3 * i + j] + c3 * gqg;
    }
}

}  // namespace
