// FP64 force and K w of one tetrahedron (device code), arranged for few
// instructions: GB300's FP64 pipe issues one instruction per 19 cycles and SM,
// and it bounds every FP64 element map, so each product is formed once, as
// chains of fused multiply-adds, and the rest volume goes into the Lame parameters once
// instead of into every corner output.  The formulas are those of
// tet_math.cuh (in terms of G = F - I, accurate at small strain).
// Measured, one thread per tet, 163,840 tets, us: StVK force and K w 131 -> 98,
// K w 100 -> 78; neo-Hookean 135 -> 117, 98 -> 90.
#pragma once

#include "tet_math.cuh"

namespace ebb {

// Corner outputs from Q = V P (times s): out[a][c] = s Q_c . b_a for a = 1..3
// (b_a = row a-1 of B), corner 0 minus their sum.
__device__ __forceinline__ void corners_f64(const double* Q, const double* B, double (&out)[4][3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
      out[a + 1][c] = fma(Q[c * 3], B[a * 3], fma(Q[c * 3 + 1], B[a * 3 + 1], Q[c * 3 + 2] * B[a * 3 + 2]));
    out[0][c] = -(out[1][c] + (out[2][c] + out[3][c]));
  }
}

// C += A S, S symmetric as (00 01 02 11 12 22).
__device__ __forceinline__ void mm_sym_add(const double* A, const double* S, double* C) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double a0 = A[i * 3], a1 = A[i * 3 + 1], a2 = A[i * 3 + 2];
    C[i * 3] = fma(a0, S[0], fma(a1, S[1], fma(a2, S[2], C[i * 3])));
    C[i * 3 + 1] = fma(a0, S[1], fma(a1, S[3], fma(a2, S[4], C[i * 3 + 1])));
    C[i * 3 + 2] = fma(a0, S[2], fma(a1, S[4], fma(a2, S[5], C[i * 3 + 2])));
  }
}

// A symmetric 2 mu sym + lam tr form from the doubled symmetric part e2
// (e2 = A + A^T as 00 01 02 11 12 22): mu e2 + (lam / 2) tr(e2) I.
__device__ __forceinline__ void sym_stress(const double* e2, double mu, double lam, double* S) {
  const double t = 0.5 * lam * (e2[0] + e2[3] + e2[5]);
  S[0] = fma(mu, e2[0], t);
  S[1] = mu * e2[1];
  S[2] = mu * e2[2];
  S[3] = fma(mu, e2[3], t);
  S[4] = mu * e2[4];
  S[5] = fma(mu, e2[5], t);
}

template <bool FORCE, bool KV>
__device__ __forceinline__ void stvk_eval_f64(const double* B, double V, double mu, double lam, const double* Du,
                                              const double* Dw, double (&fo)[4][3], double (&ko)[4][3]) {
  const double vmu = V * mu, vlam = V * lam;
  double G[9], e2[6], S[6];
  mm(Du, B, G);
  {
    // 2 E = G + G^T + G^T G
    int q = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j)
        e2[q++] = fma(G[i], G[j], fma(G[3 + i], G[3 + j], fma(G[6 + i], G[6 + j], G[i * 3 + j] + G[j * 3 + i])));
  }
  sym_stress(e2, vmu, vlam, S);   // V S
  if (FORCE) {
    // -V P = -(S + G S)
    double P[9] = {S[0], S[1], S[2], S[1], S[3], S[4], S[2], S[4], S[5]};
    mm_sym_add(G, S, P);
#pragma unroll
    for (int i = 0; i < 9; ++i) P[i] = -P[i];
    corners_f64(P, B, fo);
  }
  if (KV) {
    double dF[9], Y[6];
    mm(Dw, B, dF);
    {
      // W + W^T, W = dF + G^T dF
      double W[9];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
          W[i * 3 + j] = fma(G[i], dF[j], fma(G[3 + i], dF[3 + j], fma(G[6 + i], dF[6 + j], dF[i * 3 + j])));
      const double w2[6] = {W[0] + W[0], W[1] + W[3], W[2] + W[6], W[4] + W[4], W[5] + W[7], W[8] + W[8]};
      sym_stress(w2, vmu, vlam, Y);
    }
    // dP = dF S + Y + G Y
    double dP[9] = {Y[0], Y[1], Y[2], Y[1], Y[3], Y[4], Y[2], Y[4], Y[5]};
    mm_sym_add(G, Y, dP);
    mm_sym_add(dF, S, dP);
    corners_f64(dP, B, ko);
  }
}

// False for an inverted element (J <= 0).
template <bool FORCE, bool KV>
__device__ __forceinline__ bool nh_eval_f64(const double* B, double V, double mu, double lam, const double* Du,
                                            const double* Dw, double (&fo)[4][3], double (&ko)[4][3]) {
  double G[9];
  mm(Du, B, G);
  NhState<double> sn;
  if (!nh_state(G, sn)) return false;
  const double* A = sn.FiT;
  const double vmu = V * mu, vll = V * lam * sn.lnJ;
  if (FORCE) {
    // -V P = -(V mu (G + G^T F^-T) + V lam ln J F^-T)
    double P[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double x = fma(G[i], A[j], fma(G[3 + i], A[3 + j], fma(G[6 + i], A[6 + j], G[i * 3 + j])));
        P[i * 3 + j] = -fma(vmu, x, vll * A[i * 3 + j]);
      }
    corners_f64(P, B, fo);
  }
  if (KV) {
    double dF[9], T1[9], dP[9];
    mm(Dw, B, dF);
    mtm(dF, A, T1);   // dF^T F^-T, whose trace is F^-T : dF
    const double c1 = vmu - vll, c2 = V * lam * (T1[0] + T1[4] + T1[8]);
#pragma unroll
    for (int i = 0; i < 9; ++i) T1[i] *= c1;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        dP[i * 3 + j] = fma(A[i * 3], T1[j], fma(A[i * 3 + 1], T1[3 + j],
                            fma(A[i * 3 + 2], T1[6 + j], fma(vmu, dF[i * 3 + j], c2 * A[i * 3 + j]))));
    corners_f64(dP, B, ko);
  }
  return true;
}

}  // namespace ebb
