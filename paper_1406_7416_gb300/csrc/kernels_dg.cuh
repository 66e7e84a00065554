// ADER-DG kernels: space-time predictor (Sec. 2.2 Eq. pde.nc.dg2), DG face
// fluxes and corrector (Sec. 2.3 Eq. pde.nc.gw2) fused with the a-posteriori
// detector (Sec. 4.3 Eqs. positivity, dmp, relax).
#pragma once

#include <climits>

#include "adg_internal.h"
#include "fixed.cuh"

namespace adg {

template <int D, int N>
struct Dims {
  static constexpr int n = N + 1;
  static constexpr int NV = D + 2;
  static constexpr int ND = ipow(n, D);          // spatial nodes per cell
  static constexpr int NST = ipow(n, D + 1);     // space-time nodes per cell
  static constexpr int NF = ipow(n, D - 1);      // tangential nodes per face
  static constexpr int NT = NF * n;              // tangential x time nodes per face
  static constexpr int Ns = 2 * N + 1;
  static constexpr int NSD = ipow(Ns, D);        // subcells per cell
  static constexpr int NSF = ipow(Ns, D - 1);    // sub-faces per cell face
  static constexpr int L = Ns + 6;               // limiter patch width (3 ghost layers)
  static constexpr int LD = ipow(L, D);
  static constexpr int NE = Ns + 2;              // reconstructed block -1..Ns
  static constexpr int NED = ipow(NE, D);
  static constexpr int NST3 = ipow(3, D + 1);    // subcell space-time nodes
  static constexpr int ND3 = ipow(3, D);
};

// Predictor block shape.  The mixed kernel at high 2D degrees is latency
// bound with one 128-thread block per SM (measured: 4 warps per SM, FP64 pipe
// 41% busy at N = 9); 256 threads capped at 128 registers, two blocks per SM,
// hide the FP32 and FP64 latencies.  Below N = 6 the 2D mixed kernel runs 128
// threads capped at 102 registers, five blocks per SM (measured against four
// blocks at N = 4 and 5: 8% and 4% faster; 160 threads: 17% slower at N = 4;
// 256 threads: 40% slower), the 3D mixed kernel 160 threads, four blocks per
// SM (9% faster than 128 at N = 3).
template <int D, int N, bool MIXED>
struct PredShape {
  static constexpr bool wide = MIXED && D == 2 && N >= 6;
  static constexpr bool narrow3 = MIXED && D == 3;
  static constexpr int threads = wide ? 256 : (narrow3 ? 160 : 128);   // launched per block
  static constexpr int bound = (MIXED && !wide) ? threads : 256;       // __launch_bounds__ maximum
  // registers: <= 102 for the narrow mixed kernels (five 128- or four
  // 160-thread blocks per SM), <= 128 for the wide ones (two 256-thread or four
  // 128-thread blocks); <= 64 in FP64 up to N = 5, where the phases' barriers
  // want more blocks beside each other; no cap above (no difference).  Measured
  // (GB300, us per launch, FP64, the better block width, at most 64 / 80 / 128
  // registers): 200^2 N = 1 191 / 191 / 180, N = 2 441 / 460 / 531, N = 3 807 /
  // 819 / 904, N = 4 1958 / 2019 / 2240, N = 5 3899 / 4076 / 4523; 24^3 N = 1 117 /
  // 118 / 126, N = 2 494 / 513 / 562, N = 3 1784 / 1834 / 1829.  The short phases
  // of 2D N = 1 want the registers.
  static constexpr int min_blocks =
      narrow3 ? 4
              : ((MIXED && !wide) ? 5
                                  : (MIXED ? 2 : ((D == 2 && N >= 6) ? 1 : (D == 2 && N == 1 ? 2 : 4))));
};

// ---------------------------------------------------------------------------
// Picard phases on one space-time block of n^(D+1) nodes (Eq. pde.nc.dg2):
//   q <- u (x) 1 - Ktau x_tau sum_k c_k D x_k f_k(q),  c_k = dt / dx_k.
// Work items are spread over threads tid .. (step nth).
// ---------------------------------------------------------------------------
template <int D, int n, typename T>
__device__ __forceinline__ void picard_flux(const T* __restrict__ q, T* __restrict__ F, T gm1,
                                            int tid, int nth) {
  constexpr int NV = D + 2, NST = ipow(n, D + 1);
  for (int l = tid; l < NST; l += nth) {
    T Q[NV];
    T Fl[D][D + 2];
#pragma unroll
    for (int v = 0; v < NV; ++v) Q[v] = q[v * NST + l];
    euler_fluxes<D, T>(Q, gm1, Fl);
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int v = 0; v < NV; ++v) F[(k * NV + v) * NST + l] = Fl[k][v];
  }
}

template <int D, int n, typename T>
__device__ __forceinline__ void picard_deriv(const T* __restrict__ F, T* __restrict__ S,
                                             const T* __restrict__ Dm, const T* c, int tid,
                                             int nth) {
  constexpr int NV = D + 2, NST = ipow(n, D + 1);
  for (int e = tid; e < NV * NST; e += nth) {
    const int v = e / NST, l = e - v * NST;
    T s = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
      const int ak = (l / st) % n;
      const T* f = F + (k * NV + v) * NST + (l - ak * st);
      const T* dr = Dm + ak * n;
      T acc = T(0);
#pragma unroll
      for (int j = 0; j < n; ++j) acc += dr[j] * f[j * st];
      s += c[k] * acc;
    }
    S[e] = s;
  }
}

template <int D, int n, typename T, typename UT>
__device__ __forceinline__ void picard_time(T* __restrict__ q, const UT* __restrict__ u,
                                            const T* __restrict__ Kt, int tid, int nth) {
  constexpr int NV = D + 2, ND = ipow(n, D), NST = ipow(n, D + 1);
  for (int e = tid; e < NV * ND; e += nth) {
    const int v = e / ND, i = e - v * ND;
    T Sl[n];
#pragma unroll
    for (int m = 0; m < n; ++m) Sl[m] = q[v * NST + i + m * ND];
    const T u0 = (T)u[v * ND + i];
#pragma unroll
    for (int m = 0; m < n; ++m) {
      T acc = T(0);
#pragma unroll
      for (int j = 0; j < n; ++j) acc += Kt[m * n + j] * Sl[j];
      q[v * NST + i + m * ND] = u0 - acc;
    }
  }
}

// FP64 sweep phases with the contractions on the integer pipes (fixed.cuh).  The
// FP64 pipe bounds an FP64 sweep: per node its fluxes take 16 operations in 2D
// and a division, its contractions (D + 1) n + D + 1 per variable, more than
// four times as many at n = 6.  The FP64 pipe keeps the fluxes and the sums over
// the axes; the phases run by lines, each line read and converted once for its
// n outputs, and the derivative phase works in place, so that the axes need no
// barrier between them.  Measured (GB300, predictor phase per step): 256^2
// N = 5 FP64 17.1 -> 6.4 ms, 67 x 53 N = 6 FP64 1.93 -> 0.77 ms, 33 x 29 x 30
// N = 3 FP64 7.75 -> 3.68 ms, 200^2 N = 9 mixed (nine FP32 sweeps and this one)
// 17.0 -> 11.4 ms.
//
// Fluxes of `nodes` space-time nodes (all NST, or the ND of time node 0).
template <int D, int n>
__device__ __forceinline__ void flux_fx(const double* __restrict__ q, double* __restrict__ F, double gm1,
                                        int nodes, int qstride, int tid, int nth) {
  constexpr int NV = D + 2, NST = ipow(n, D + 1);
  for (int l = tid; l < nodes; l += nth) {
    double Q[NV], Fl[D][D + 2];
#pragma unroll
    for (int v = 0; v < NV; ++v) Q[v] = q[v * qstride + l];
    euler_fluxes_sym<D>(Q, gm1, Fl);
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int v = 0; v < NV; ++v) F[(k * NV + v) * NST + l] = Fl[k][v];
  }
}

// Derivative phase, F_k <- (c_k D) x_k F_k in place for every axis: one thread
// per line of n nodes (cD[k n n ..] is c_k D with scale exponent gD[k]; coef and
// Dm its factors).  NL lines per variable (those of all time nodes, or of time
// node 0).
template <int D, int n, int NL>
__device__ __forceinline__ void deriv_fx(double* F, const FxOp* cD, const int* gD,
                                         const double* __restrict__ coef, const double* __restrict__ Dm,
                                         int tid, int nth) {
  constexpr int NV = D + 2, NST = ipow(n, D + 1);
  for (int e = tid; e < D * NV * NL; e += nth) {
    const int kv = e / NL, r = e - kv * NL;
    const int k = kv / NV;
    const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
    double* f = F + kv * NST + n * r - (n - 1) * (r % st);
    double x[n];
#pragma unroll
    for (int j = 0; j < n; ++j) x[j] = f[j * st];
    fx_apply<n, n, false>(x, cD + k * (n * n), gD[k], FxRows{Dm, coef[k]}, [&](int a, double y) { f[a * st] = y; });
  }
}

// Time phase, q <- u - Ktau S with S = sum_k of the derivative phase's F_k.
template <int D, int n>
__device__ __forceinline__ void time_fx(const double* F, double* q, const double* u, const FxOp* Kt,
                                        int gK, const double* __restrict__ Ktd, int tid, int nth) {
  constexpr int NV = D + 2, ND = ipow(n, D), NST = ipow(n, D + 1);
  for (int e = tid; e < NV * ND; e += nth) {
    const int v = e / ND, i = e - v * ND;
    double S[n];
#pragma unroll
    for (int m = 0; m < n; ++m) {
      double s = F[v * NST + i + m * ND];
#pragma unroll
      for (int k = 1; k < D; ++k) s += F[(k * NV + v) * NST + i + m * ND];
      S[m] = s;
    }
    const double u0 = u[e];
    double* qv = q + v * NST + i;
    // (no look for steep lines: S itself is rounded at 2^-53 of the fluxes, which
    // differ little between the time nodes, and lines of rounding noise, a uniform
    // flow's, are as steep as a shock's)
    fx_apply<n, n, true>(S, Kt, gK, FxRows{Ktd, 1.0}, [&](int m, double y) { qv[m * ND] = u0 - y; });
  }
}

// FP32 Picard operators D and Ktau of every degree N (index N) in constant
// memory, one copy per translation unit (filled by upload_picard_constants):
// with the loops unrolled every operator entry is a constant-bank operand of
// its FMA, so the FP32 sweeps load only their data from shared memory.
static __constant__ float c_Dmf[MAXN][MAXN * MAXN];
static __constant__ float c_Ktf[MAXN][MAXN * MAXN];
// the projection P of every degree
static __constant__ float c_P1f[MAXN][MAXNS * MAXN];
// the degree-2 subcell predictor's operators (3 nodes), likewise
static __constant__ float c_D3f[9];
static __constant__ float c_K3f[9];

// Derivative and time phases of an FP32 sweep of the subcell predictor with
// its operators from constant memory; one output per work item and no
// barrier inside (the caller's thread groups run them under a condition).
// Operation order as in picard_deriv / picard_time.
template <int D>
__device__ __forceinline__ void picard_deriv_sub(const float* __restrict__ F, float* __restrict__ S,
                                                 const float* c, int tid, int nth) {
  constexpr int n = 3, NV = D + 2, NST = ipow(n, D + 1);
  for (int e = tid; e < NV * NST; e += nth) {
    const int v = e / NST, l = e - v * NST;
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
      const int ak = (l / st) % n;
      const float* f = F + (k * NV + v) * NST + (l - ak * st);
      float x[n];
#pragma unroll
      for (int j = 0; j < n; ++j) x[j] = f[j * st];
      // row ak of D3 from constant memory (ak is 0, 1 or 2)
      const float d0 = ak == 0 ? c_D3f[0] : (ak == 1 ? c_D3f[3] : c_D3f[6]);
      const float d1 = ak == 0 ? c_D3f[1] : (ak == 1 ? c_D3f[4] : c_D3f[7]);
      const float d2 = ak == 0 ? c_D3f[2] : (ak == 1 ? c_D3f[5] : c_D3f[8]);
      float acc = 0.0f;
      acc += d0 * x[0];
      acc += d1 * x[1];
      acc += d2 * x[2];
      s += c[k] * acc;
    }
    S[e] = s;
  }
}

template <int D>
__device__ __forceinline__ void picard_time_sub(float* __restrict__ q, const float* __restrict__ u,
                                                int tid, int nth) {
  constexpr int n = 3, NV = D + 2, ND = ipow(n, D), NST = ipow(n, D + 1);
  for (int e = tid; e < NV * ND; e += nth) {
    const int v = e / ND, i = e - v * ND;
    float Sl[n];
#pragma unroll
    for (int m = 0; m < n; ++m) Sl[m] = q[v * NST + i + m * ND];
    const float u0 = u[v * ND + i];
#pragma unroll
    for (int m = 0; m < n; ++m) {
      float acc = 0.0f;
#pragma unroll
      for (int j = 0; j < n; ++j) acc += c_K3f[m * n + j] * Sl[j];
      q[v * NST + i + m * ND] = u0 - acc;
    }
  }
}

// Derivative phase of an FP32 sweep, S = sum_k c_k D x_k F_k, one thread per
// line of n nodes along axis k: the line's n fluxes are loaded once and give
// n outputs (n independent FMA chains).  The axes run one after the other
// (S is written for k = 0 and accumulated after), with the same operation
// order per output as picard_deriv.
template <int D, int N>
__device__ __forceinline__ void picard_deriv_lines(const float* __restrict__ F, float* __restrict__ S,
                                                   const float* c, int tid, int nth) {
  constexpr int n = N + 1, NV = D + 2, NST = ipow(n, D + 1), NL = NST / n;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
    const float ck = c[k];
    for (int e = tid; e < NV * NL; e += nth) {
      const int v = e / NL, r = e - v * NL;
      const int base = r % st + (r / st) * (st * n);
      const float* f = F + (k * NV + v) * NST + base;
      float x[n];
#pragma unroll
      for (int j = 0; j < n; ++j) x[j] = f[j * st];
      float* sl = S + v * NST + base;
#pragma unroll
      for (int a = 0; a < n; ++a) {
        float acc = 0.0f;
#pragma unroll
        for (int j = 0; j < n; ++j) acc += c_Dmf[N][a * n + j] * x[j];
        if (k == 0) sl[a * st] = ck * acc;
        else sl[a * st] += ck * acc;
      }
    }
    if (k + 1 < D) __syncthreads();
  }
}

// Time phase of an FP32 sweep, q <- u - Ktau S, with Ktau from constant memory.
template <int D, int N>
__device__ __forceinline__ void picard_time_cf(float* __restrict__ q, const float* __restrict__ u,
                                               int tid, int nth) {
  constexpr int n = N + 1, NV = D + 2, ND = ipow(n, D), NST = ipow(n, D + 1);
  for (int e = tid; e < NV * ND; e += nth) {
    const int v = e / ND, i = e - v * ND;
    float Sl[n];
#pragma unroll
    for (int m = 0; m < n; ++m) Sl[m] = q[v * NST + i + m * ND];
    const float u0 = u[v * ND + i];
#pragma unroll
    for (int m = 0; m < n; ++m) {
      float acc = 0.0f;
#pragma unroll
      for (int j = 0; j < n; ++j) acc += c_Ktf[N][m * n + j] * Sl[j];
      q[v * NST + i + m * ND] = u0 - acc;
    }
  }
}

// The time phase of the last FP32 Picard sweep when no FP64 sweep follows:
// only the space-time correction dq = q - u = -Ktau S is formed (FP32, from
// the sweep's S = sum_k c_k D x_k f_k(q)); the final stage adds it to the
// FP64 u term by term (face traces, fluxes), so q carries no FP32 rounding of
// u itself (the dominant error of a plain FP32 sweep).
template <int D, int N>
__device__ __forceinline__ void picard_time_dq(const float* __restrict__ S,
                                               float* __restrict__ dq, int tid, int nth) {
  constexpr int n = N + 1, NV = D + 2, ND = ipow(n, D), NST = ipow(n, D + 1);
  for (int e = tid; e < NV * ND; e += nth) {
    const int v = e / ND, i = e - v * ND;
    float Sl[n];
#pragma unroll
    for (int m = 0; m < n; ++m) Sl[m] = S[v * NST + i + m * ND];
#pragma unroll
    for (int m = 0; m < n; ++m) {
      float acc = 0.0f;
#pragma unroll
      for (int j = 0; j < n; ++j) acc += c_Ktf[N][m * n + j] * Sl[j];
      dq[v * NST + i + m * ND] = -acc;
    }
  }
}

// Euler flux difference F_k(U + dQ) - F_k(U), k = 0..D-1, in FP32 and in a
// form where every term carries a factor of dQ (velocity change
// dv = (dm - v drho) / (rho + drho), pressure change
// dp = (gamma - 1)(dE - d(m.v)/2) with d(m.v) = sum_j dm_j (v_j + dv_j) + m_j dv_j),
// so its rounding error is relative to the change, not to the flux: with
// F(U) in FP64 the sum equals F(U + dQ) to FP32 rounding of the correction.
template <int D>
__device__ __forceinline__ void euler_flux_delta(const float* U, const float* dQ, float gm1,
                                                 float (*G)[D + 2]) {
  const float r = 1.0f / U[0];
  const float r1 = 1.0f / (U[0] + dQ[0]);
  float v[D], dv[D];
  float mv = 0.0f, dmv = 0.0f;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    v[j] = U[1 + j] * r;
    mv += U[1 + j] * v[j];
    dv[j] = (dQ[1 + j] - v[j] * dQ[0]) * r1;
  }
#pragma unroll
  for (int j = 0; j < D; ++j) dmv += dQ[1 + j] * (v[j] + dv[j]) + U[1 + j] * dv[j];
  const float Ep = U[D + 1] + gm1 * (U[D + 1] - 0.5f * mv);
  const float dp = gm1 * (dQ[D + 1] - 0.5f * dmv);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float vk1 = v[k] + dv[k];
    G[k][0] = dQ[1 + k];
#pragma unroll
    for (int j = 0; j < D; ++j) G[k][1 + j] = dQ[1 + j] * vk1 + U[1 + j] * dv[k];
    G[k][1 + k] += dp;
    G[k][D + 1] = (dQ[D + 1] + dp) * vk1 + Ep * dv[k];
  }
}

// Apply a matrix along axis k of a (nv, e0, e1, e2) tensor (x fastest):
// out[v][.., r, ..] = sum_c M[r * cols + c] in[v][.., c, ..].
// ein: extents of `in`; out has extent `rows` along k.
template <int D>
__device__ __forceinline__ void apply_axis(const double* __restrict__ in, double* __restrict__ out,
                                           const double* __restrict__ M, int rows, int cols, int k,
                                           const int* ein, int nv, int tid, int nth) {
  int eout[3] = {1, 1, 1};
  int insz = 1, outsz = 1;
  for (int j = 0; j < D; ++j) {
    eout[j] = (j == k) ? rows : ein[j];
    insz *= ein[j];
    outsz *= eout[j];
  }
  int stride = 1;
  for (int j = 0; j < k; ++j) stride *= ein[j];
  for (int e = tid; e < nv * outsz; e += nth) {
    const int v = e / outsz;
    int r = e - v * outsz;
    int idx[3] = {0, 0, 0};
    for (int j = 0; j < D; ++j) {
      idx[j] = r % eout[j];
      r /= eout[j];
    }
    int off = 0, s = 1;
    for (int j = 0; j < D; ++j) {
      off += (j == k ? 0 : idx[j]) * s;
      s *= ein[j];
    }
    const double* src = in + v * insz + off;
    const double* mr = M + idx[k] * cols;
    double acc = 0.0;
    for (int c = 0; c < cols; ++c) acc += mr[c] * src[c * stride];
    out[e] = acc;
  }
}

// Tensor projection / reconstruction of all variables of one cell through two
// buffers: NV variables, NI -> NO points per axis, matrix M[NO][NI]; every
// index division is by a constant.
template <int D, int NV, int NI, int NO, int K, typename T = double>
__device__ __forceinline__ void apply_pass_ct(const T* __restrict__ in, T* __restrict__ out,
                                              const T* __restrict__ M, int tid, int nth) {
  constexpr int I0 = (0 < K) ? NO : NI, I1 = (1 < K) ? NO : NI, I2 = (2 < K) ? NO : NI;
  constexpr int O0 = (0 <= K) ? NO : NI, O1 = (1 <= K) ? NO : NI, O2 = (2 <= K) ? NO : NI;
  constexpr int E1 = (D > 1) ? 1 : 0, E2 = (D > 2) ? 1 : 0;
  constexpr int ISZ = I0 * (E1 ? I1 : 1) * (E2 ? I2 : 1);
  constexpr int OSZ = O0 * (E1 ? O1 : 1) * (E2 ? O2 : 1);
  constexpr int STRIDE = (K == 0) ? 1 : (K == 1 ? I0 : I0 * I1);
  for (int e = tid; e < NV * OSZ; e += nth) {
    const int v = e / OSZ;
    int r = e - v * OSZ;
    const int x0 = r % O0;
    r /= O0;
    const int x1 = E1 ? r % O1 : 0;
    const int x2 = E2 ? r / O1 : 0;
    const int xk = (K == 0) ? x0 : (K == 1 ? x1 : x2);
    const int off = (K == 0 ? 0 : x0) + I0 * ((K == 1 ? 0 : x1) + I1 * (K == 2 ? 0 : x2));
    const T* src = in + v * ISZ + off;
    const T* mr = M + xk * NI;
    T acc = T(0);
#pragma unroll
    for (int c = 0; c < NI; ++c) acc += mr[c] * src[c * STRIDE];
    out[e] = acc;
  }
}

// One pass of the FP32 projection P of the step's change: one thread per line of
// n nodes along axis K, its Ns outputs' operator entries from constant memory
// (the sums in the order of apply_pass_ct).  One thread per output loaded 2 n
// operands for n FMAs.  With it the detector's scan reads and updates the kept
// averages itself (no copy of them in shared memory, one barrier fewer) and
// reduces its extremes by warp_max_key: 5022 -> 3774 instructions per 2D N = 5
// cell.  Measured (GB300), corrector and detector per step, mixed: 512^2 N = 5
// 2.14 -> 1.91 ms, 200^2 N = 9 1.65 -> 1.32, 64^3 N = 3 10.1 -> 8.4.
template <int D, int N, int K>
__device__ __forceinline__ void project_pass_f(const float* in, float* out, int tid, int nth) {
  constexpr int NV = D + 2, NI = N + 1, NO = 2 * N + 1;
  constexpr int I0 = (0 < K) ? NO : NI, I1 = (D < 2) ? 1 : ((1 < K) ? NO : NI), I2 = (D < 3) ? 1 : NI;
  constexpr int ISZ = I0 * I1 * I2, LINES = ISZ / NI, OSZ = LINES * NO;
  constexpr int S = (K == 0) ? 1 : (K == 1 ? I0 : I0 * I1);       // stride along K, in and out
  for (int e = tid; e < NV * LINES; e += nth) {
    const int v = e / LINES, r = e - v * LINES;
    const int lo = r % S, hi = r / S;
    const float* src = in + v * ISZ + lo + hi * (S * NI);
    float* dst = out + v * OSZ + lo + hi * (S * NO);
    float x[NI];
#pragma unroll
    for (int j = 0; j < NI; ++j) x[j] = src[j * S];
#pragma unroll
    for (int a = 0; a < NO; ++a) {
      float acc = 0.0f;
#pragma unroll
      for (int j = 0; j < NI; ++j) acc += c_P1f[N][a * NI + j] * x[j];
      dst[a * S] = acc;
    }
  }
}

template <int D, int N, bool WARP>
__device__ __forceinline__ const float* project_f(float* a, float* b, int tid, int nth) {
  auto sync = [] {
    if (WARP) __syncwarp();
    else __syncthreads();
  };
  project_pass_f<D, N, 0>(a, b, tid, nth);
  sync();
  project_pass_f<D, N, 1>(b, a, tid, nth);
  sync();
  if (D == 2) return a;
  project_pass_f<D, N, 2>(a, b, tid, nth);
  sync();
  return b;
}

// Tensor reconstruction R of one cell in FP64 (few cells: the FMA chain, whose
// DOFs the FP32 subcell and predictor kernels round from).
template <int D, int N>
__device__ __forceinline__ double* reconstruct(double* a, double* b, const double* R1, int tid, int nth) {
  constexpr int NV = D + 2, n = N + 1, Ns = 2 * N + 1;
  apply_pass_ct<D, NV, Ns, n, 0, double>(a, b, R1, tid, nth);
  __syncthreads();
  apply_pass_ct<D, NV, Ns, n, 1, double>(b, a, R1, tid, nth);
  __syncthreads();
  if (D == 2) return a;
  apply_pass_ct<D, NV, Ns, n, 2, double>(a, b, R1, tid, nth);
  __syncthreads();
  return b;
}

// The FP64 projection operator: its fixed-point entries (shared memory) with
// their scale exponent, and its doubles.
struct FxMat {
  const FxOp* x;
  int g;
  const double* d;
};

// One pass of apply_ct in FP64 on the integer pipes (fixed.cuh): one thread per
// line of NI points along axis K.  Lines of two points (N = 1) stay on the FP64
// pipe: the conversions cost more there than the two FMAs of each output (and
// at N = 3 already half of the FMAs').
template <int D, int NV, int NI, int NO, int K>
__device__ __forceinline__ void apply_pass_fx(const double* in, double* out, const FxMat& M, int tid,
                                              int nth) {
  if constexpr (NI < 3) {
    apply_pass_ct<D, NV, NI, NO, K, double>(in, out, M.d, tid, nth);
  } else {
    constexpr int I0 = (0 < K) ? NO : NI, I1 = (D < 2) ? 1 : ((1 < K) ? NO : NI), I2 = (D < 3) ? 1 : NI;
    constexpr int ISZ = I0 * I1 * I2, LINES = ISZ / NI, OSZ = LINES * NO;
    constexpr int S = (K == 0) ? 1 : (K == 1 ? I0 : I0 * I1);     // stride along K, in and out
    for (int e = tid; e < NV * LINES; e += nth) {
      const int v = e / LINES, r = e - v * LINES;
      const int lo = r % S, hi = r / S;                           // places below and above axis K
      const double* src = in + v * ISZ + lo + hi * (S * NI);
      double* dst = out + v * OSZ + lo + hi * (S * NO);
      double x[NI];
#pragma unroll
      for (int j = 0; j < NI; ++j) x[j] = src[j * S];
      fx_apply<NI, NO, false>(x, M.x, M.g, FxRows{M.d, 1.0}, [&](int a, double y) { dst[a * S] = y; });
    }
  }
}

// Tensor projection in FP64 through two buffers, by a block or (WARP) a warp.
template <int D, int NV, int NI, int NO, bool WARP = false>
__device__ __forceinline__ double* apply_fx(double* a, double* b, const FxMat& M, int tid, int nth) {
  auto sync = [] {
    if (WARP) __syncwarp();
    else __syncthreads();
  };
  apply_pass_fx<D, NV, NI, NO, 0>(a, b, M, tid, nth);
  sync();
  if (D == 1) return b;
  apply_pass_fx<D, NV, NI, NO, 1>(b, a, M, tid, nth);
  sync();
  if (D == 2) return a;
  apply_pass_fx<D, NV, NI, NO, 2>(a, b, M, tid, nth);
  sync();
  return b;
}

// Block-wide reductions of per-thread values (blockDim a multiple of 32).
__device__ __forceinline__ double block_reduce_max(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v = nanmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  double r = red[0];
  for (int i = 1; i < nw; ++i) r = nanmax(r, red[i]);
  __syncthreads();
  return r;
}

__device__ __forceinline__ double block_reduce_min(double v, double* red) {
  return -block_reduce_max(-v, red);
}

// Trace element e of a cell, laid out [k][side][v][ts + NF * m] (face axis k,
// side s, variable v, tangential node ts, time node m): returns v and sets the
// space-time node offset `base` of the line of n nodes across axis k, its
// stride `stk` and the side s.
template <int D, int n>
__device__ __forceinline__ int trace_index(int e, int& base, int& stk, int& s) {
  constexpr int NV = D + 2, ND = ipow(n, D), NF = ipow(n, D - 1), NT = NF * n;
  const int k = e / (2 * NV * NT);
  int r = e - k * (2 * NV * NT);
  s = r / (NV * NT);
  r -= s * (NV * NT);
  const int v = r / NT, tt = r - v * NT;
  const int m = tt / NF;
  int ts = tt - m * NF;
  int st = 1;
  base = m * ND;
  stk = 1;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    if (j == k) {
      stk = st;
    } else {
      base += (ts % n) * st;
      ts /= n;
    }
    st *= n;
  }
  return v;
}

// ---------------------------------------------------------------------------
// K1 predictor: one cell per block.  Writes the candidate's volume part
// u + sum_k c_k Mvol x_k fbar_k into Unext and the space-time face traces.
// ---------------------------------------------------------------------------
template <int D, int N, bool MIXED>
__host__ __device__ constexpr size_t predictor_smem_bytes() {
  using DM = Dims<D, N>;
  // u, q, F, fbar, the integer-pipe operators (cD, cM, Ktx, kapx, wx, phx of
  // k_predictor), w and phi
  size_t d = (size_t)DM::NV * DM::ND + (size_t)DM::NV * DM::NST + (size_t)D * DM::NV * DM::NST +
             (size_t)D * DM::NV * DM::ND + (2 * D + 1) * DM::n * DM::n + 4 * DM::n + 3 * DM::n;
  // the FP32 sweep arrays qf, Ff live inside the FP64 flux array F (unused
  // until the FP32 sweeps are over); u and the trace weights in FP32 stay
  // apart (the FP32 sweep operators are in constant memory)
  size_t f = MIXED ? ((size_t)DM::NV * DM::ND + 2 * DM::n) : 0;
  return d * sizeof(double) + f * sizeof(float);
}

template <int D, int N, bool MIXED>
__global__ void __launch_bounds__(PredShape<D, N, MIXED>::bound, PredShape<D, N, MIXED>::min_blocks)
    k_predictor(Batch bt) {
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, NST = DM::NST, NF = DM::NF, NT = DM::NT;
  extern __shared__ double sm[];
  double* u = sm;
  double* q = u + NV * ND;
  double* F = q + NV * NST;
  double* fbar = F + D * NV * NST;
  // integer-pipe operators: c_k D and c_k Mvol per axis (of the state in hand),
  // Ktau, its row sums, the time weights and the two traces
  FxOp* cD = reinterpret_cast<FxOp*>(fbar + D * NV * ND);
  FxOp* cM = cD + D * n * n;
  FxOp* Ktx = cM + D * n * n;
  FxOp* kapx = Ktx + n * n;         // row sums of Ktau
  FxOp* wx = kapx + n;
  FxOp* phx = wx + n;               // [2][n]
  double* w = reinterpret_cast<double*>(phx + 2 * n);
  double* ph0 = w + n;
  double* ph1 = ph0 + n;
  // FP32 sweep arrays inside F: (1 + D) NV NST floats fit in D NV NST doubles
  float* qf = reinterpret_cast<float*>(F);
  float* Ff = qf + NV * NST;
  float* uf = reinterpret_cast<float*>(ph1 + n);
  float* ph0f = uf + NV * ND;
  float* ph1f = ph0f + n;
  __shared__ double s_rs[5];        // largest row sums: D, Mvol, Ktau, w, phi
  __shared__ int gD[3], gM[3];      // scale exponents of cD, cM

  const int tid = threadIdx.x, nth = blockDim.x;
  const Ops* o = bt.pps[0]->ops;      // every state of a batch has degree N
  for (int i = tid; i < n; i += nth) {
    w[i] = o->w[i];
    ph0[i] = o->phi0[i];
    ph1[i] = o->phi1[i];
    if (MIXED) {
      ph0f[i] = (float)o->phi0[i];
      ph1f[i] = (float)o->phi1[i];
    }
  }
  if (tid < 32) {
    double rs[5] = {};
    if (tid < n) {
      for (int j = 0; j < n; ++j) {
        rs[0] += fabs(o->D[tid * n + j]);
        rs[1] += fabs(o->Mvol[tid * n + j]);
        rs[2] += fabs(o->Kt[tid * n + j]);
        rs[3] += fabs(o->w[j]);
        rs[4] += fabs(tid & 1 ? o->phi1[j] : o->phi0[j]);
      }
    }
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      for (int d = 16; d > 0; d >>= 1) rs[r] = fmax(rs[r], __shfl_xor_sync(0xffffffffu, rs[r], d));
      if (tid == 0) s_rs[r] = rs[r];
    }
  }
  __syncthreads();
  const int gK = fx_scale(s_rs[2]), gw = fx_scale(s_rs[3]), gph = fx_scale(s_rs[4]);
  for (int i = tid; i < n * n; i += nth) Ktx[i] = fx_op(o->Kt[i], gK);
  for (int i = tid; i < n; i += nth) {
    double ks = 0.0;
    for (int j = 0; j < n; ++j) ks += o->Kt[i * n + j];
    kapx[i] = fx_op(ks, gK);
    wx[i] = fx_op(o->w[i], gw);
    phx[i] = fx_op(o->phi0[i], gph);
    phx[n + i] = fx_op(o->phi1[i], gph);
  }
  int state = -1;
  for (long long g = blockIdx.x; g < bt.pre[bt.n]; g += gridDim.x) {
    const int sidx = batch_state(bt, g);
    const Params& p = *bt.pps[sidx];
    const long long cell = g - bt.pre[sidx];
    const double dt = *p.b.dt;
    if (!(dt > 0.0)) continue;          // state idle this step (block-uniform)
    double c[3];
#pragma unroll
    for (int k = 0; k < D; ++k) c[k] = p.b.coef[k];
    const double gm1 = p.gamma - 1.0;
    const double* Uc = p.b.U[p.cur] + cell * (NV * ND);
    for (int i = tid; i < NV * ND; i += nth) u[i] = Uc[i];
    if (sidx != state) {
      // the operators of this state's step, scaled by c_k
      state = sidx;
      if (tid < D) {
        gD[tid] = fx_scale(p.b.coef[tid] * s_rs[0]);
        gM[tid] = fx_scale(p.b.coef[tid] * s_rs[1]);
      }
      for (int i = tid; i < D * n * n; i += nth) {
        const int k = i / (n * n), r = i - k * (n * n);
        const double ck = p.b.coef[k];
        cD[i] = fx_op(ck * o->D[r], fx_scale(ck * s_rs[0]));
        cM[i] = fx_op(ck * o->Mvol[r], fx_scale(ck * s_rs[1]));
      }
    }
    __syncthreads();
    int it0 = 0;
    const int n32 = p.iters - p.fp64_sweeps;    // sweeps in FP32
    // with no FP64 sweep the traces split into trace(u) (FP64, once per face
    // node) + trace(q - u) (FP32, per space-time node): the same sum, with
    // FP32 rounding only on the small correction
    const bool split = MIXED && n32 > 0 && p.fp64_sweeps == 0;
    double* tr = p.b.trace + cell * (size_t)(D * 2 * NV * NT);
    if (MIXED && n32 > 0) {
      float cf[3];
#pragma unroll
      for (int k = 0; k < D; ++k) cf[k] = (float)c[k];
      for (int e = tid; e < NV * ND; e += nth) uf[e] = (float)u[e];
      __syncthreads();
      for (int e = tid; e < NV * NST; e += nth) {
        const int v = e / NST, l = e - v * NST;
        qf[e] = uf[v * ND + (l % ND)];
      }
      __syncthreads();
      const bool last64 = p.fp64_sweeps == 0;     // no FP64 sweep: close on the FP64 u
      for (int it = 0; it < n32; ++it) {
        picard_flux<D, n, float>(qf, Ff, (float)gm1, tid, nth);
        __syncthreads();
        picard_deriv_lines<D, N>(Ff, qf, cf, tid, nth);
        __syncthreads();
        if (last64 && it == n32 - 1) picard_time_dq<D, N>(qf, Ff, tid, nth);
        else picard_time_cf<D, N>(qf, uf, tid, nth);
        __syncthreads();
      }
      if (!last64)
        for (int e = tid; e < NV * NST; e += nth) q[e] = widen_f32_any(qf[e]);
      it0 = n32;
    } else {
      // the first sweep starts from u (x) 1, whose fluxes and derivatives S are
      // the same at every time node: it runs on the n^d spatial nodes, and
      // q_m = u - kappa_m S with kappa = Ktau 1
      flux_fx<D, n>(u, F, gm1, ND, ND, tid, nth);
      __syncthreads();
      deriv_fx<D, n, ND / n>(F, cD, gD, p.b.coef, o->D, tid, nth);
      __syncthreads();
      for (int e = tid; e < NV * ND; e += nth) {
        const int v = e / ND, i = e - v * ND;
        double S = F[v * NST + i];
#pragma unroll
        for (int k = 1; k < D; ++k) S += F[(k * NV + v) * NST + i];
        const double u0 = u[e];
        double* qv = q + v * NST + i;
        fx_apply<1, n, true>(&S, kapx, gK, FxSums<n>{o->Kt}, [&](int m, double y) { qv[m * ND] = u0 - y; });
      }
      it0 = 1;
    }
    __syncthreads();
    for (int it = it0; it < p.iters; ++it) {
      flux_fx<D, n>(q, F, gm1, NST, NST, tid, nth);
      __syncthreads();
      deriv_fx<D, n, NST / n>(F, cD, gD, p.b.coef, o->D, tid, nth);
      __syncthreads();
      time_fx<D, n>(F, q, u, Ktx, gK, o->Kt, tid, nth);
      __syncthreads();
    }
    if (split) {
      // final stage on u (FP64) + dq (FP32): fbar_k = F_k(u) + sum_m w_m
      // (F_k(u + dq_m) - F_k(u)); the face traces stay split, trace(u) in FP64
      // and trace(dq) in FP32 (split trace layout, see k_faceflux)
      const float* dq = Ff;
      float* dF = qf + 2 * NV * NST;      // [D][NV][NST] weighted flux differences
      for (int i = tid; i < ND; i += nth) {
        double Q[NV], Fl[D][D + 2];
#pragma unroll
        for (int v = 0; v < NV; ++v) Q[v] = u[v * ND + i];
        euler_fluxes<D, double>(Q, gm1, Fl);
#pragma unroll
        for (int k = 0; k < D; ++k)
#pragma unroll
          for (int v = 0; v < NV; ++v) fbar[(k * NV + v) * ND + i] = Fl[k][v];
      }
      for (int e = tid; e < D * 2 * NV * NF; e += nth) {
        int base, stk, s;
        const int v = trace_index<D, n>((e / NF) * NT + e % NF, base, stk, s);   // time node 0
        const double* ph = s ? ph1 : ph0;
        double acc = 0.0;
#pragma unroll
        for (int a = 0; a < n; ++a) acc += ph[a] * u[v * ND + base + a * stk];
        tr[(e / (NV * NF)) * (NV * NT) + e % (NV * NF)] = acc;
      }
      for (int l = tid; l < NST; l += nth) {
        const int i = l % ND, m = l / ND;
        float U[NV], dQ[NV], G[D][D + 2];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          U[v] = uf[v * ND + i];
          dQ[v] = dq[v * NST + l];
        }
        euler_flux_delta<D>(U, dQ, (float)gm1, G);
        const float wm = (float)w[m];
#pragma unroll
        for (int k = 0; k < D; ++k)
#pragma unroll
          for (int v = 0; v < NV; ++v) dF[(k * NV + v) * NST + l] = wm * G[k][v];
      }
      __syncthreads();
      for (int e = tid; e < D * 2 * NV * NT; e += nth) {
        int base, stk, s;
        const int v = trace_index<D, n>(e, base, stk, s);
        const float* ph = s ? ph1f : ph0f;
        const float* d = dq + v * NST + base;
        float acc = 0.0f;
#pragma unroll
        for (int a = 0; a < n; ++a) acc += ph[a] * d[a * stk];
        const int blk = e / (NV * NT);
        reinterpret_cast<float*>(tr + blk * (NV * NT) + NV * NF)[e - blk * (NV * NT)] = acc;
      }
      for (int e = tid; e < D * NV * ND; e += nth) {
        const int kv = e / ND, i = e - kv * ND;
        float acc = 0.0f;
#pragma unroll
        for (int m = 0; m < n; ++m) acc += dF[kv * NST + i + m * ND];
        fbar[e] += (double)acc;
      }
      __syncthreads();
    } else {
      // corrector volume term from the time-averaged nodal fluxes
      flux_fx<D, n>(q, F, gm1, NST, NST, tid, nth);
      __syncthreads();
      for (int e = tid; e < D * NV * ND; e += nth) {
        const int kv = e / ND, i = e - kv * ND;
        double x[n];
#pragma unroll
        for (int m = 0; m < n; ++m) x[m] = F[kv * NST + i + m * ND];
        fx_apply<n, 1, true>(x, wx, gw, FxRows{w, 1.0}, [&](int, double y) { fbar[e] = y; });
      }
      __syncthreads();
    }
    // c_k Mvol x_k fbar_k in place, by lines, then the sum with u
    for (int e = tid; e < D * NV * NF; e += nth) {
      const int kv = e / NF, r = e - kv * NF;
      const int k = kv / NV;
      const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
      double* f = fbar + kv * ND + n * r - (n - 1) * (r % st);
      double x[n];
#pragma unroll
      for (int j = 0; j < n; ++j) x[j] = f[j * st];
      fx_apply<n, n, false>(x, cM + k * (n * n), gM[k], FxRows{o->Mvol, p.b.coef[k]}, [&](int a, double y) { f[a * st] = y; });
    }
    // space-time traces on the faces, trace[cell][k][side][v][ts + NF * m], by
    // lines: the n nodes of a line along axis k give both faces normal to k, and
    // the line's index within its variable is the trace's index ts + NF m
    if (!split)
      for (int e = tid; e < D * NV * NT; e += nth) {
        const int k = e / (NV * NT), vr = e - k * (NV * NT);
        const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
        const double* f = q + n * vr - (n - 1) * (vr % st);
        double x[n];
#pragma unroll
        for (int j = 0; j < n; ++j) x[j] = f[j * st];
        double* t = tr + (2 * k) * (NV * NT) + vr;
        fx_apply<n, 2, false>(x, phx, gph, FxRows{ph0, 1.0}, [&](int side, double y) { t[side * (NV * NT)] = y; });
      }
    __syncthreads();
    double* Uo = p.b.U[1 - p.cur] + cell * (NV * ND);
    for (int e = tid; e < NV * ND; e += nth) {
      double acc = u[e];
#pragma unroll
      for (int k = 0; k < D; ++k) acc += fbar[k * (NV * ND) + e];
      Uo[e] = acc;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// K2 face flux: the time-averaged numerical flux at every tangential node of
// every face normal to axis k.
// ---------------------------------------------------------------------------
// Whether a state's predictor leaves its face traces split: per (cell, axis,
// side) block of NV x NT doubles, trace(u) [NV][NF] in FP64 followed by
// trace(dq) [NV][NT] in FP32 (mixed precision with no FP64 Picard sweep).
__device__ __forceinline__ bool split_traces(const Params& p) {
  return p.prec == ADG_PREC_MIXED_FP32 && p.fp64_sweeps == 0 && p.iters > 0;
}

// Space-time trace value at tangential node ts, time node m of one block.
template <int D, int n>
__device__ __forceinline__ void load_trace(const double* blk, int ts, int m, bool split, double* Q) {
  constexpr int NV = D + 2, NF = ipow(n, D - 1), NT = NF * n;
  if (split) {
    const float* d = reinterpret_cast<const float*>(blk + NV * NF);
#pragma unroll
    for (int v = 0; v < NV; ++v) Q[v] = blk[v * NF + ts] + (double)d[v * NT + ts + NF * m];
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v) Q[v] = blk[v * NT + ts + NF * m];
  }
}

// Euler flux along axis k (FP64); RCP: 1 / rho from rcp_newton (the
// mixed-precision path's split face flux).
template <int D, bool RCP = false>
__device__ __forceinline__ void euler_flux_k(const double* Q, double gm1, int k, double* F) {
  const double r = RCP ? rcp_newton(Q[0]) : 1.0 / Q[0];
  double kin = 0.0;
#pragma unroll
  for (int j = 0; j < D; ++j) kin += Q[1 + j] * Q[1 + j];
  const double p = gm1 * (Q[D + 1] - 0.5 * kin * r);
  const double vk = Q[1 + k] * r;
  F[0] = Q[1 + k];
#pragma unroll
  for (int j = 0; j < D; ++j) F[1 + j] = Q[1 + j] * vk;
  F[1 + k] += p;
  F[D + 1] = vk * (Q[D + 1] + p);
}

// F_k(U + dQ) - F_k(U) in FP32, every term carrying a factor of dQ (the
// along-axis-k part of euler_flux_delta).
template <int D>
__device__ __forceinline__ void euler_flux_delta_k(const float* U, const float* dQ, float gm1, int k,
                                                   float* G) {
  const float r = 1.0f / U[0];
  const float r1 = 1.0f / (U[0] + dQ[0]);
  float v[D], dv[D];
  float mv = 0.0f, dmv = 0.0f;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    v[j] = U[1 + j] * r;
    mv += U[1 + j] * v[j];
    dv[j] = (dQ[1 + j] - v[j] * dQ[0]) * r1;
  }
#pragma unroll
  for (int j = 0; j < D; ++j) dmv += dQ[1 + j] * (v[j] + dv[j]) + U[1 + j] * dv[j];
  const float Ep = U[D + 1] + gm1 * (U[D + 1] - 0.5f * mv);
  const float dp = gm1 * (dQ[D + 1] - 0.5f * dmv);
  const float vk1 = v[k] + dv[k];
  G[0] = dQ[1 + k];
#pragma unroll
  for (int j = 0; j < D; ++j) G[1 + j] = dQ[1 + j] * vk1 + U[1 + j] * dv[k];
  G[1 + k] += dp;
  G[D + 1] = (dQ[D + 1] + dp) * vk1 + Ep * dv[k];
}

// |v_k| + c of U + dQ in FP32, with rho p = (gamma - 1)(E rho - |m|^2 / 2)
// taken as the FP64 value rpU of U plus its change, which carries a factor of
// dQ; NaN for an inadmissible state.
template <int D>
__device__ __forceinline__ float speed_split(const float* U, const float* dQ, float rpU, float gamma,
                                             float gm1, int k) {
  float drp = U[D + 1] * dQ[0] + (U[0] + dQ[0]) * dQ[D + 1];
#pragma unroll
  for (int j = 0; j < D; ++j) drp -= (U[1 + j] + 0.5f * dQ[1 + j]) * dQ[1 + j];
  const float r = 1.0f / (U[0] + dQ[0]);
  return fabsf(U[1 + k] + dQ[1 + k]) * r + sqrtf(gamma * (rpU + gm1 * drp)) * r;
}

// Time-averaged Rusanov flux of an interior face from split traces:
//   G = (F_k(uL) + F_k(uR)) / 2 + sum_m w_m (dF_L,m + dF_R,m) / 2
//       - (uR - uL) sum_m w_m s_m / 2 - sum_m w_m s_m (dqR_m - dqL_m) / 2,
// F_k(u) in FP64 once per face node, the per-time-node parts in FP32.
template <int D, int n>
__device__ __forceinline__ void face_split_rusanov(const double* bL, const double* bR, int ts, int k,
                                                   double gamma, const float* wf, float gf,
                                                   float gm1f, double* G) {
  constexpr int NV = D + 2, NF = ipow(n, D - 1), NT = NF * n;
  const float* dL = reinterpret_cast<const float*>(bL + NV * NF);
  const float* dR = reinterpret_cast<const float*>(bR + NV * NF);
  const double gm1 = gamma - 1.0;
  double uL[NV], uR[NV], FL[NV], FR[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    uL[v] = bL[v * NF + ts];
    uR[v] = bR[v * NF + ts];
  }
  euler_flux_k<D, true>(uL, gm1, k, FL);
  euler_flux_k<D, true>(uR, gm1, k, FR);
  double kinL = 0.0, kinR = 0.0;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    kinL += uL[1 + j] * uL[1 + j];
    kinR += uR[1 + j] * uR[1 + j];
  }
  // the FP32 copies of the FP64 terms, narrowed on the integer pipe (toward
  // zero: they are the base states of the FP32 per-time-node corrections)
  const float rpL = narrow_f64_rz(gm1 * (uL[D + 1] * uL[0] - 0.5 * kinL));
  const float rpR = narrow_f64_rz(gm1 * (uR[D + 1] * uR[0] - 0.5 * kinR));
  float ULf[NV], URf[NV], sumD[NV], sumJ[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    ULf[v] = narrow_f64_rz(uL[v]);
    URf[v] = narrow_f64_rz(uR[v]);
    sumD[v] = 0.0f;
    sumJ[v] = 0.0f;
  }
  float S = 0.0f;
#pragma unroll 1
  for (int m = 0; m < n; ++m) {
    float qL[NV], qR[NV], GL[NV], GR[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      qL[v] = dL[v * NT + ts + NF * m];
      qR[v] = dR[v * NT + ts + NF * m];
    }
    euler_flux_delta_k<D>(ULf, qL, gm1f, k, GL);
    euler_flux_delta_k<D>(URf, qR, gm1f, k, GR);
    const float sL = speed_split<D>(ULf, qL, rpL, gf, gm1f, k);
    const float sR = speed_split<D>(URf, qR, rpR, gf, gm1f, k);
    const float s = (sL > sR || sL != sL) ? sL : sR;     // NaN propagates
    const float wm = wf[m];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      sumD[v] += wm * (GL[v] + GR[v]);
      sumJ[v] += wm * s * (qR[v] - qL[v]);
    }
    S += wm * s;
  }
  const double Sd = widen_f32(S);
#pragma unroll
  for (int v = 0; v < NV; ++v)
    G[v] = 0.5 * (FL[v] + FR[v]) + 0.5 * widen_f32(sumD[v]) -
           0.5 * ((uR[v] - uL[v]) * Sd + widen_f32(sumJ[v]));
}

// One face node (a face normal to axis k, its tangential node ts) of a state:
// the trace blocks on both sides and which sides are inside the domain.
template <int D, int N>
struct FaceNode {
  using DM = Dims<D, N>;
  int ijk[3];                // the face's index along k, its cell's along the others
  int ts;
  long long face;
  bool hasL, hasR;
  const double *trL, *trR;   // (a missing side takes the other's)

  __device__ __forceinline__ FaceNode(const Params& p, int k, const int* at, int tsn) : ts(tsn) {
    constexpr int NV = DM::NV, NT = DM::NT;
    const Geo& g = p.geo;
    int L[3], R[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) L[j] = R[j] = ijk[j] = at[j];
    const int f = ijk[k];
    hasL = hasR = true;
    if (f == 0) {
      if (g.periodic[k]) L[k] = g.n[k] - 1; else hasL = false;
    } else {
      L[k] = f - 1;
    }
    if (f == g.n[k]) {
      if (g.periodic[k]) R[k] = 0; else hasR = false;
    }
    face = face_index<D>(g, ijk, k, f);
    const size_t csz = (size_t)D * 2 * NV * NT;
    trL = hasL ? p.b.trace + cell_index<D>(L, g) * csz + ((size_t)k * 2 + 1) * NV * NT : nullptr;
    trR = hasR ? p.b.trace + cell_index<D>(R, g) * csz + ((size_t)k * 2 + 0) * NV * NT : nullptr;
    if (!hasL) trL = trR;
    if (!hasR) trR = trL;
  }
  __device__ __forceinline__ bool inside() const { return hasL && hasR; }

  // The numerical flux at time node m; at a domain boundary the missing side
  // is the ghost state of the face's kind (boundary_ghost).
  template <bool OSHER>
  __device__ __forceinline__ void flux(const Params& p, int k, int m, bool split, double* Gm) const {
    constexpr int n = DM::n, NV = DM::NV;
    const Geo& g = p.geo;
    double QL[NV], QR[NV];
    load_trace<D, n>(trL, ts, m, split, QL);
    load_trace<D, n>(trR, ts, m, split, QR);
    if (!hasL || !hasR) {
      const int side = 2 * k + (hasL ? 1 : 0);
      double pos = 0.0, t = 0.0;
      if (g.bc[side] == ADG_BC_FRONT) {
        // the node's coordinate along the front's axis, and its time
        const int j = g.front_axis[side];
        int a = 0, tt = ts;
#pragma unroll
        for (int jj = 0; jj < D; ++jj)
          if (jj != k) {
            if (jj == j) a = tt % n;
            tt /= n;
          }
        pos = g.x0[j] + (ijk[j] + p.ops->xi[a]) * g.dx[j];
        t = *p.b.tstart + p.ops->xi[m] * *p.b.dt;
      }
      if (!hasL) boundary_ghost<D>(g, side, QR, QL, pos, t);
      else boundary_ghost<D>(g, side, QL, QR, pos, t);
    }
    face_flux<D>(OSHER ? ADG_FLUX_OSHER : ADG_FLUX_RUSANOV, QL, QR, k, p.gamma, Gm,
                 p.prec == ADG_PREC_MIXED_FP32);
  }
};

// Time-averaged numerical flux at every face node normal to axis k.  Past the
// first `wide_blocks` blocks, one thread takes a node inside the domain and
// steps through its time nodes.  The first blocks take n lanes per node, one
// per time node, and add the n fluxes in order from one lane to the next (the
// same operations: the same bits): the nodes on the domain's boundary, whose
// ghost states and FP64 fluxes at n time nodes in a row kept one warp busy long
// after the other faces were done, or with `wide` (few nodes: waiting for one
// thread's n fluxes is then the whole kernel) every node that is not a split
// Rusanov one, whose time nodes are FP32.
// Measured (GB300), face fluxes per step with the axes side by side: 32^2 N = 3
// mixed, transmissive, 49 -> 17 us; 350 x 100 N = 5 mixed (inflow, wall, fronts)
// 178 -> 74 us; 64^3 N = 3 mixed 2.63 -> 1.92 ms; 256^2 N = 5 FP64 0.77 -> 0.66.
//
// KIND: FACE_OSHER, FACE_RUSANOV, or FACE_LEAN for launches whose nodes are all
// split Rusanov ones inside the domain (mixed precision, periodic axis): without
// the general path's registers more warps hide that path's load latency.
// K: the axis at compile time (-1: taken from `axis`; the Osher-type flux only),
// so that the states' and fluxes' k-th components are registers and not an
// indexed array in local memory.  512^2 N = 5 mixed (lean): 0.71 -> 0.38 ms per
// step at three blocks per SM, 0.35 at four, 0.51 at two.
enum FaceKind { FACE_RUSANOV, FACE_OSHER, FACE_LEAN };

template <int D, int N, int KIND, int K>
__global__ void __launch_bounds__(256, KIND == FACE_OSHER ? 2 : (KIND == FACE_LEAN ? 6 - D : (D == 2 && N >= 6 ? 2 : 3)))
    k_faceflux(Batch bt, int axis, int wide_blocks, int wide) {
  const int k = K >= 0 ? K : axis;
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, NF = DM::NF;
  if ((int)blockIdx.x >= wide_blocks) {
    for (long long eg = (long long)(blockIdx.x - wide_blocks) * blockDim.x + threadIdx.x; eg < bt.pre[bt.n];
         eg += (long long)(gridDim.x - wide_blocks) * blockDim.x) {
      const int sidx = batch_state(bt, eg);
      const Params& p = *bt.pps[sidx];
      if (!(*p.b.dt > 0.0)) continue;
      const long long e = eg - bt.pre[sidx];
      const Geo& g = p.geo;
      const long long face = e / NF;
      int ijk[3] = {0, 0, 0};
      // (32-bit divisions as in cell_coords: faces along an axis < 2^32)
      unsigned r = (unsigned)face;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        if (j + 1 < D) {
          const unsigned ext = (unsigned)((j == k) ? g.n[j] + 1 : g.n[j]), t = r / ext;
          ijk[j] = (int)(r - t * ext);
          r = t;
        } else {
          ijk[j] = (int)r;
        }
      }
      if (KIND != FACE_LEAN && !g.periodic[k] && (ijk[k] == 0 || ijk[k] == g.n[k])) continue;
      const bool split = KIND == FACE_LEAN || split_traces(p);
      const bool fp32 = split && KIND != FACE_OSHER;
      if (KIND != FACE_LEAN && wide && !fp32) continue;
      const FaceNode<D, N> fn(p, k, ijk, (int)(e - face * NF));
      double* G = p.b.G[k] + face * (NV * NF) + fn.ts;
      double acc[NV];
      if (KIND == FACE_LEAN || fp32) {
        face_split_rusanov<D, n>(fn.trL, fn.trR, fn.ts, k, p.gamma, p.ops->wf, p.b.coef_f[7],
                                 p.b.coef_f[6], acc);
      } else {
        const double* w = p.ops->w;
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = 0.0;
        for (int m = 0; m < n; ++m) {
          double Gm[NV];
          fn.template flux<KIND == FACE_OSHER>(p, k, m, split, Gm);
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] += w[m] * Gm[v];
        }
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) G[v * NF] = acc[v];
    }
    return;
  }
  if constexpr (KIND != FACE_LEAN) {
  constexpr int GPW = 32 / n;                            // nodes per warp
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int grp = lane / n < GPW ? lane / n : GPW - 1;   // (idle lanes repeat the last node's)
  const int m = lane / n < GPW ? lane - grp * n : n - 1;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long stride = (long long)wide_blocks * (blockDim.x >> 5) * GPW;
  for (long long q0 = warp * GPW;; q0 += stride) {       // (uniform over the warp)
    // node q: the q-th of all (wide), or of the boundary nodes of state after state
    long long q = q0 + grp;
    const Params* pp = nullptr;
    int ijk[3] = {0, 0, 0}, ts = 0;
    if (wide) {
      if (q0 >= bt.pre[bt.n]) break;
      if (q < bt.pre[bt.n]) {
        const int s = batch_state(bt, q);
        pp = bt.pps[s];
        q -= bt.pre[s];
        ts = (int)(q % NF);
        q /= NF;
#pragma unroll
        for (int j = 0; j < D; ++j) {
          const int ext = (j == k) ? pp->geo.n[j] + 1 : pp->geo.n[j];
          ijk[j] = (int)(q % ext);
          q /= ext;
        }
      }
    } else {
      long long left = q;
      for (int s = 0; s < bt.n && !pp; ++s) {
        const Geo& g = bt.pps[s]->geo;
        if (g.periodic[k]) continue;
        const long long cnt = 2 * (g.cells / g.n[k]) * NF;
        if (left < cnt) {
          pp = bt.pps[s];
          ts = (int)(left % NF);
          left /= NF;
          ijk[k] = (left & 1) ? g.n[k] : 0;
          left >>= 1;
#pragma unroll
          for (int j = 0; j < D; ++j)
            if (j != k) {
              ijk[j] = (int)(left % g.n[j]);
              left /= g.n[j];
            }
        } else {
          left -= cnt;
        }
      }
      if (!__any_sync(FULL, pp != nullptr)) break;
    }
    double Gm[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Gm[v] = 0.0;
    double* G = nullptr;
    if (pp && *pp->b.dt > 0.0) {
      const Params& p = *pp;
      const FaceNode<D, N> fn(p, k, ijk, ts);
      const bool split = split_traces(p);
      if (!fn.inside() || !split || KIND == FACE_OSHER) {
        fn.template flux<KIND == FACE_OSHER>(p, k, m, split, Gm);
        G = p.b.G[k] + fn.face * (NV * NF) + ts;
      }
    }
    const double* w = bt.pps[0]->ops->w;                 // (every state of a batch has degree N)
    __syncwarp();
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      double acc = 0.0;
#pragma unroll
      for (int i = 0; i < n; ++i) acc += w[i] * __shfl_sync(FULL, Gm[v], grp * n + i);
      if (G && m == v % n && lane < GPW * n) G[v * NF] = acc;
    }
  }
  }
}

// Tangential node index of spatial node i for the faces normal to axis k.
template <int D, int n>
__device__ __forceinline__ int tangential(int i, int k) {
  int ts = 0, mul = 1;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const int a = i % n;
    i /= n;
    if (j != k) {
      ts += a * mul;
      mul *= n;
    }
  }
  return ts;
}

// Order-preserving map of a double onto a signed 64-bit key (x < y <=> key(x)
// < key(y) for non-NaN x, y; +NaN above +inf), so that min / max reductions
// run on the integer pipe instead of the FP64 pipe.
__device__ __forceinline__ long long ord_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double ord_val(long long k) {
  return __longlong_as_double(k >= 0 ? k : (k ^ 0x7fffffffffffffffLL));
}
// max(a, b) of two doubles that are not negative (+0 included) and not NaN:
// their bit patterns order as signed integers
__device__ __forceinline__ double max_nonneg(double a, double b) {
  return __double_as_longlong(a) >= __double_as_longlong(b) ? a : b;
}
// Bulk prefetch of `bytes` (a multiple of 16, 16-byte aligned) into L2 by the
// TMA unit (cp.async.bulk.prefetch): no shared memory, nothing to wait for.
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// Bulk prefetch into L2 of the 16-byte-aligned part of [src, src + bytes), in
// pieces of at most 4 KB (the bytes outside it, at most 15 at each end, are
// left to the loads).
__device__ __forceinline__ void prefetch_range_l2(const void* src, size_t bytes) {
  const uintptr_t a = (reinterpret_cast<uintptr_t>(src) + 15) & ~(uintptr_t)15;
  const uintptr_t e = (reinterpret_cast<uintptr_t>(src) + bytes) & ~(uintptr_t)15;
  for (uintptr_t x = a; x < e; x += 4096) {
    const uintptr_t len = (e - x < 4096) ? (e - x) : 4096;
    bulk_prefetch_l2(reinterpret_cast<const void*>(x), (unsigned)len);
  }
}

// Key of a wave speed for a max-reduction: a NaN of either sign (an
// inadmissible state) is the largest key, so the cell's speed is NaN and the
// CFL step reports the state (ord_key alone would order a NaN with its sign
// bit set below every speed).
__device__ __forceinline__ long long speed_key(double s) {
  return isnan_f64(s) ? LLONG_MAX : ord_key(s);
}

// Key of an interval's end for the test on keys, key(x) >= key(lo) && key(x) <=
// key(hi): exactly the FP64 comparisons (a zero of either sign is the lower
// zero below and the upper zero above; a NaN end fails every x but NaN, which
// fails at the other end).  FP64 comparisons run on the FP64 pipe, once for
// every warp here.
__device__ __forceinline__ long long bound_key(double x, bool high) {
  if (isnan_f64(x)) return high ? LLONG_MIN : LLONG_MAX;
  const long long b = __double_as_longlong(x);
  if ((b << 1) == 0) return high ? 0 : -1;
  return ord_key(x);
}

// Detector bounds over the Voronoi neighbourhood (3^d block) from per-cell
// min/max, then the relaxed DMP interval [m - delta, M + delta] (Eq. relax
// with a relative floor).  Threads v < nvar write the keys of its ends
// (bound_key), lohi[2v], lohi[2v+1].
template <int D>
__device__ __forceinline__ void dmp_interval_lane(const Params& p, const double* __restrict__ cmm,
                                                  const int* ijk, long long* lohi, int v);

template <int D>
__device__ __forceinline__ void dmp_interval(const Params& p, const double* __restrict__ cmm,
                                             const int* ijk, long long* lohi) {
  if ((int)threadIdx.x < D + 2) dmp_interval_lane<D>(p, cmm, ijk, lohi, threadIdx.x);
}

// The interval of variable v (one thread per variable).
template <int D>
__device__ __forceinline__ void dmp_interval_lane(const Params& p, const double* __restrict__ cmm,
                                                  const int* ijk, long long* lohi, int v) {
  const int NV = D + 2;
  const Geo& g = p.geo;
  // min / max on order-preserving integer keys (the integer pipe), NaNs
  // skipped as fmin / fmax skip them
  long long kmn = LLONG_MAX, kmx = LLONG_MIN;
  const int nb3 = ipow(3, D);
  for (int o = 0; o < nb3; ++o) {
    int c[3] = {0, 0, 0}, oo = o;
    bool in = true, flip = false;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      int cj = ijk[j] + (oo % 3) - 1;
      oo /= 3;
      if (cj < 0 || cj >= g.n[j]) {
        const int kind = g.bc[2 * j + (cj < 0 ? 0 : 1)];
        if (kind == ADG_BC_PERIODIC) {
          cj = (cj + g.n[j]) % g.n[j];
        } else if (kind == ADG_BC_REFLECTIVE) {
          // mirror image of the boundary cell: its wall-normal momentum
          // bounds negate and swap
          cj = cj < 0 ? 0 : g.n[j] - 1;
          if (v == 1 + j) flip = !flip;
        } else {
          in = false;
        }
      }
      c[j] = cj;
    }
    if (!in) continue;
    const long long nb = cell_index<D>(c, g);
    const double lo = cmm[(nb * NV + v) * 2 + 0], hi = cmm[(nb * NV + v) * 2 + 1];
    // the mirror image's bounds: negated (sign bit) and swapped
    const double l2 = flip ? __longlong_as_double(__double_as_longlong(hi) ^ LLONG_MIN) : lo;
    const double h2 = flip ? __longlong_as_double(__double_as_longlong(lo) ^ LLONG_MIN) : hi;
    if (!isnan_f64(l2)) kmn = min(kmn, ord_key(l2));
    if (!isnan_f64(h2)) kmx = max(kmx, ord_key(h2));
  }
  const double mn = kmn == LLONG_MAX ? INFINITY : ord_val(kmn);
  const double mx = kmx == LLONG_MIN ? -INFINITY : ord_val(kmx);
  // fmax of non-negative doubles as integer compares of their bit patterns
  // (the same result; the FP64 pipe runs fmax)
  const double scale = max_nonneg(1.0, max_nonneg(fabs(mx), fabs(mn)));
  const double delta = max_nonneg(p.eps * (mx - mn), p.floor * scale);
  lohi[2 * v] = bound_key(mn - delta, false);
  lohi[2 * v + 1] = bound_key(mx + delta, true);
}

// The largest of the warp's 64-bit keys, in every lane: the largest high words
// by one 32-bit reduction, then the largest low word among the lanes that have
// it (a shuffle tree of 64-bit maxima takes five times as many instructions).
__device__ __forceinline__ long long warp_max_key(long long k) {
  const int h = __reduce_max_sync(0xffffffffu, (int)(k >> 32));
  const unsigned l = __reduce_max_sync(0xffffffffu, (int)(k >> 32) == h ? (unsigned)k : 0u);
  return ((long long)h << 32) | l;
}

// Max-reduces K integer keys per thread over the block (blockDim a multiple of
// 32, at most 256 threads); the results land in red[nw * K + j].
template <int K>
__device__ __forceinline__ const long long* block_max_keys(long long* r, long long* red) {
#pragma unroll
  for (int j = 0; j < K; ++j) r[j] = warp_max_key(r[j]);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int j = 0; j < K; ++j) red[w * K + j] = r[j];
  __syncthreads();
  if (threadIdx.x < K) {
    long long x = red[threadIdx.x];
    for (int i = 1; i < nw; ++i) x = max(x, red[i * K + threadIdx.x]);
    red[nw * K + threadIdx.x] = x;
  }
  __syncthreads();
  return red + nw * K;
}

// Checks of the subcell data of one cell, value(v, s) (called once per variable
// and subcell):
//   PAD: rho > 0 and rho E - |m|^2 / 2 > 0 on every subcell (for rho > 0 the
//        second test is p > 0 without a division; NaN in any component fails);
//   per-variable extremes and, with `speed`, the largest wave speed
//        max_k |v_k| + c (FP32 speeds with f32speed) as keys in
//        r[2 v] = ~min, r[2 v + 1] = max, r[2 nvar].
// Returns whether PAD failed on a subcell of this thread.
template <int D, typename Value>
__device__ __forceinline__ bool scan_subcells(Value value, int nsub, double gamma, bool speed,
                                              bool f32speed, float g2f, int tid, int nth,
                                              long long* r) {
  constexpr int NV = D + 2, K = 2 * NV + 1;
  bool bad = false;
#pragma unroll
  for (int j = 0; j < K; ++j) r[j] = LLONG_MIN;
  for (int s = tid; s < nsub; s += nth) {
    double Q[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Q[v] = value(v, s);
      const long long k = ord_key(Q[v]);
      r[2 * v] = max(r[2 * v], ~k);          // ~k reverses the order: max of ~k = ~min k
      r[2 * v + 1] = max(r[2 * v + 1], k);
    }
    double kin = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) kin += Q[1 + k] * Q[1 + k];
    const double pe = Q[D + 1] * Q[0] - 0.5 * kin;
    // the two PAD comparisons as exact integer tests
    bad = bad || !(positive_f64(Q[0]) && positive_f64(pe));
    if (speed)
      r[2 * NV] = max(r[2 * NV], speed_key(f32speed ? wave_speed_f<D>(Q, pe, g2f) : wave_speed<D>(Q, gamma)));
  }
  return bad;
}

// Block version: the scan, the DMP test (lohi != null: the keys of the interval
// [lo_v, hi_v], tested exactly on the per-variable extremes) and the results:
// min / max to mm[2v], mm[2v+1], the largest speed to *lam (lam != null).
// Returns (block-uniform) whether any check failed.  `red` needs
// (blockDim/32 + 1) * (2 nvar + 1) doubles.
template <int D, typename Value>
__device__ __forceinline__ bool check_values(Value value, int nsub, const long long* lohi, double gamma,
                                             double* mm, double* lam, double* red, bool f32speed,
                                             float g2f) {
  constexpr int NV = D + 2, K = 2 * NV + 1;
  long long r[K];
  bool bad = scan_subcells<D>(value, nsub, gamma, lam != nullptr, f32speed, g2f, threadIdx.x, blockDim.x, r);
  bad = __syncthreads_or(bad);
  const long long* res = block_max_keys<K>(r, reinterpret_cast<long long*>(red));
  if (lohi) {
#pragma unroll
    for (int v = 0; v < NV; ++v) bad = bad || !(~res[2 * v] >= lohi[2 * v] && res[2 * v + 1] <= lohi[2 * v + 1]);
  }
  if (threadIdx.x < 2 * NV) mm[threadIdx.x] = ord_val(threadIdx.x & 1 ? res[threadIdx.x] : ~res[threadIdx.x]);
  if (threadIdx.x == 0 && lam) *lam = ord_val(res[2 * NV]);
  return bad;
}

template <int D>
__device__ __forceinline__ bool check_subcells(const double* __restrict__ vs, int nsub,
                                               const long long* lohi, double gamma, double* mm,
                                               double* lam, double* red, bool f32speed = false,
                                               float g2f = 0.0f) {
  return check_values<D>([vs, nsub](int v, int s) { return vs[v * nsub + s]; }, nsub, lohi, gamma, mm,
                         lam, red, f32speed, g2f);
}

// ---------------------------------------------------------------------------
// K3 + K4 corrector and detector: one cell per block.
// ---------------------------------------------------------------------------
// Stages of the projection per variable: u (n^D), after the x pass (Ns
// n^(D-1)), after the y pass, after the z pass.  The two buffers hold the even
// and the odd ones, in FP64 or (the step's change) in FP32.
template <int D, int N>
struct ProjStages {
  using DM = Dims<D, N>;
  static constexpr int S0 = DM::ND, S1 = DM::Ns * ipow(DM::n, D - 1);
  static constexpr int S2 = (D >= 2) ? DM::Ns * DM::Ns * ipow(DM::n, D - 2) : 0;
  static constexpr int S3 = (D == 3) ? DM::NSD : 0;
  static constexpr int SA = S0 > S2 ? S0 : S2, SB = S1 > S3 ? S1 : S3;
};

template <int D, int N>
__host__ __device__ constexpr size_t correct_smem_bytes() {
  using DM = Dims<D, N>;
  // the two stages, P1 (fixed point), the DMP interval, extremes, reductions
  // and the face terms' weights (2 d n doubles)
  return (size_t)(DM::NV * (ProjStages<D, N>::SA + ProjStages<D, N>::SB) + DM::Ns * DM::n + 4 * DM::NV +
                  128 + 2 * D * DM::n) *
         sizeof(double);
}

// (at most 64 registers, eight blocks per SM: 5-12% faster than the 72 the
// compiler takes unbounded)
template <int D, int N>
__global__ void __launch_bounds__(128, 8) k_correct_detect(Batch bt) {
  using DM = Dims<D, N>;
  using ST = ProjStages<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, NF = DM::NF, Ns = DM::Ns, NSD = DM::NSD;
  extern __shared__ double sm[];
  double* A = sm;                     // NV * SA
  double* B = A + NV * ST::SA;        // NV * SB
  FxOp* P1x = reinterpret_cast<FxOp*>(B + NV * ST::SB);            // Ns * n
  long long* lohi = reinterpret_cast<long long*>(P1x + Ns * n);    // 2 NV
  double* mm = reinterpret_cast<double*>(lohi + 2 * NV);           // 2 NV
  double* red = mm + 2 * NV;          // 128
  double* cw = red + 128;             // 2 D n: [k][side][a] dt/dx_k phi_side(a) / w_a
  const int tid = threadIdx.x, nth = blockDim.x;
  const Ops* o = bt.pps[0]->ops;
  for (int i = tid; i < Ns * n; i += nth) P1x[i] = o->P1x[i];
  const FxMat P1m = {P1x, o->gP1, o->P1};
  __syncthreads();
  for (long long g = blockIdx.x; g < bt.pre[bt.n]; g += gridDim.x) {
    const int sidx = batch_state(bt, g);
    const Params& p = *bt.pps[sidx];
    const long long cell = g - bt.pre[sidx];
    if (tid == 0) {
      // the next cell's DOF blocks and kept averages, into L2 while this one runs
      const long long gn = g + gridDim.x;
      if (gn < bt.pre[bt.n]) {
        const int sn = batch_state(bt, gn);
        const Params* pn = bt.pps[sn];
        const long long cn = gn - bt.pre[sn];
        prefetch_range_l2(pn->b.U[1 - pn->cur] + cn * (NV * ND), NV * ND * sizeof(double));
        if (pn->b.vstar) {
          prefetch_range_l2(pn->b.U[pn->cur] + cn * (NV * ND), NV * ND * sizeof(double));
          prefetch_range_l2(pn->b.vstar + cn * (size_t)(NV * NSD), NV * NSD * sizeof(double));
        }
      }
    }
    const double dt = *p.b.dt;
    if (!(dt > 0.0)) continue;
    double c[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < D; ++k) c[k] = p.b.coef[k];
    const int nxt = 1 - p.cur;
    int ijk[3];
    cell_coords<D>(cell, p.geo, ijk);
    double* Uo = p.b.U[nxt] + cell * (NV * ND);
    // mixed precision: P(u*) = P(u^n) (kept) + P(u* - u^n) in FP32 where P(u^n)
    // is known, except every 16th step (bounds the drift of the kept values)
    double* vkeep = p.b.vstar ? p.b.vstar + cell * (size_t)(NV * NSD) : nullptr;
    const bool delta = vkeep && p.b.vok[cell] && (p.stamp & 15) != 0;
    const double* Un = p.b.U[p.cur] + cell * (NV * ND);
    float* dA = reinterpret_cast<float*>(A);          // FP32 change, then its projection
    float* dB = reinterpret_cast<float*>(B);
    // the face terms' weights of this cell's step, one product each (the
    // previous cell's readers passed several barriers since)
    for (int q = tid; q < 2 * D * n; q += nth) {
      const int k = q / (2 * n), r = q - k * 2 * n;
      const double ck = k == 0 ? c[0] : (k == 1 ? c[1] : c[2]);
      cw[q] = ck * (r < n ? o->phi0w[r] : o->phi1w[r - n]);
    }
    __syncthreads();
    for (int e = tid; e < NV * ND; e += nth) {
      const int v = e / ND, i = e - v * ND;
      double acc = Uo[e];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
        const int ak = (i / st) % n;
        const int ts = tangential<D, n>(i, k);
        const long long flo = face_index<D>(p.geo, ijk, k, ijk[k]);
        const long long fhi = face_index<D>(p.geo, ijk, k, ijk[k] + 1);
        const double Glo = p.b.G[k][(flo * NV + v) * NF + ts];
        const double Ghi = p.b.G[k][(fhi * NV + v) * NF + ts];
        // u* -= dt/dx_k (phi1(a)/w_a Ghi - phi0(a)/w_a Glo), as two FMAs
        acc = fma(-cw[(2 * k + 1) * n + ak], Ghi, acc);
        acc = fma(cw[2 * k * n + ak], Glo, acc);
      }
      Uo[e] = acc;
      if (delta) dA[e] = narrow_f64_rz(acc - Un[e]);    // (integer pipe; toward zero)
      else A[e] = acc;
    }
    dmp_interval<D>(p, p.b.cmm[p.cur], ijk, lohi);
    __syncthreads();
    double lam = 0.0;
    bool bad;
    if (delta) {
      // the projected change is added to the kept averages as the scan reads them
      const float* dv = project_f<D, N, false>(dA, dB, tid, nth);
      auto value = [vkeep, dv](int v, int s) {
        const int e = v * NSD + s;
        const double x = vkeep[e] + widen_f32(dv[e]);
        vkeep[e] = x;
        return x;
      };
      bad = check_values<D>(value, NSD, lohi, p.gamma, mm, p.lam_mode ? &lam : nullptr, red,
                            p.prec == ADG_PREC_MIXED_FP32, p.gam2f);
    } else {
      const double* vs = apply_fx<D, NV, n, Ns>(A, B, P1m, tid, nth);
      auto value = [vkeep, vs](int v, int s) {
        const int e = v * NSD + s;
        const double x = vs[e];
        if (vkeep) vkeep[e] = x;
        return x;
      };
      bad = check_values<D>(value, NSD, lohi, p.gamma, mm, p.lam_mode ? &lam : nullptr, red,
                            p.prec == ADG_PREC_MIXED_FP32, p.gam2f);
    }
    if (tid == 0) {
      int slot = -1;
      if (bad || p.force) {
        slot = atomicAdd(&p.b.counters[CNT_TROUBLED0 + nxt], 1);
        if (slot < p.cap) {
          p.b.list[nxt][slot] = (int)cell;
        } else {
          // no subcell slot left: the cell keeps its candidate, the step is
          // reported as failed (ADG_ERR_CAPACITY) by the next status query
          atomicOr(&p.b.counters[CNT_STATUS], 1);
          slot = -1;
        }
      }
      p.b.beta[nxt][cell] = (uint8_t)(slot >= 0);
      p.b.slot[nxt][cell] = slot;
      if (p.lam_mode) p.b.lam[cell] = lam;
      if (vkeep) p.b.vok[cell] = 1;       // reset by any later change of the cell's DOFs
    }
    if (tid < 2 * NV) p.b.cmm[nxt][cell * 2 * NV + tid] = mm[tid];
    __syncthreads();
  }
}

}  // namespace adg

namespace adg {

// ---------------------------------------------------------------------------
// K3 + K4 with one warp per cell: the same per-item arithmetic as
// k_correct_detect (face terms, projection, kept averages, PAD, DMP on the
// extremes, integer-key reductions), synchronised by __syncwarp and reduced
// with warp shuffles instead of block barriers; W cells per block.
// ---------------------------------------------------------------------------
constexpr int CD_WARPS = 4;

// Warp version of check_values; every lane returns the extremes mm, *lam and
// whether a check failed.
template <int D, typename Value>
__device__ __forceinline__ bool check_values_warp(Value value, int nsub, const long long* lohi,
                                                  double gamma, double* mm, double* lam, bool f32speed,
                                                  int lane, float g2f) {
  constexpr int NV = D + 2, K = 2 * NV + 1;
  long long r[K];
  bool bad = scan_subcells<D>(value, nsub, gamma, lam != nullptr, f32speed, g2f, lane, 32, r);
#pragma unroll
  for (int j = 0; j < K; ++j) r[j] = warp_max_key(r[j]);
  bad = __any_sync(0xffffffffu, bad);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    bad = bad || !(~r[2 * v] >= lohi[2 * v] && r[2 * v + 1] <= lohi[2 * v + 1]);
    mm[2 * v] = ord_val(~r[2 * v]);
    mm[2 * v + 1] = ord_val(r[2 * v + 1]);
  }
  if (lam) *lam = ord_val(r[2 * NV]);
  return bad;
}

template <int D, int N>
struct CdLayout {
  using DM = Dims<D, N>;
  using ST = ProjStages<D, N>;
  // per warp: the two stages of the projection, face weights [2 D][n], the keys
  // of the DMP interval [2 NV]
  static constexpr int A_DBL = DM::NV * ST::SA, B_DBL = DM::NV * ST::SB;
  static constexpr int CW_DBL = 2 * D * DM::n;
  static constexpr int WARP_DBL = A_DBL + B_DBL + CW_DBL + 2 * DM::NV;
  // per block: P1 (fixed point)
  static constexpr int OPS_DBL = DM::Ns * DM::n;
};

template <int D, int N>
__host__ __device__ constexpr size_t correct_warp_smem_bytes() {
  return (size_t)(CdLayout<D, N>::OPS_DBL + CD_WARPS * CdLayout<D, N>::WARP_DBL) * sizeof(double);
}

template <int D, int N>
__global__ void __launch_bounds__(32 * CD_WARPS) k_correct_detect_w(Batch bt) {
  using DM = Dims<D, N>;
  using LY = CdLayout<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, NF = DM::NF, Ns = DM::Ns, NSD = DM::NSD;
  extern __shared__ double sm[];
  FxOp* P1x = reinterpret_cast<FxOp*>(sm);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* A = sm + LY::OPS_DBL + w * LY::WARP_DBL;
  double* B = A + LY::A_DBL;
  double* cw = B + LY::B_DBL;          // [k][side][a]: dt/dx_k phi_side(a) / w_a
  long long* lohi = reinterpret_cast<long long*>(cw + LY::CW_DBL);
  const Ops* o = bt.pps[0]->ops;
  for (int i = threadIdx.x; i < Ns * n; i += 32 * CD_WARPS) P1x[i] = o->P1x[i];
  const FxMat P1m = {P1x, o->gP1, o->P1};
  __syncthreads();
  const long long total = bt.pre[bt.n];
  for (long long g = (long long)blockIdx.x * CD_WARPS + w; g < total;
       g += (long long)gridDim.x * CD_WARPS) {
    const int sidx = batch_state(bt, g);
    const Params& p = *bt.pps[sidx];
    const long long cell = g - bt.pre[sidx];
    if (lane == 0) {
      // the next cell's DOF blocks and kept averages, into L2 while this one runs
      const long long gn = g + (long long)gridDim.x * CD_WARPS;
      if (gn < total) {
        const int sn = batch_state(bt, gn);
        const Params* pn = bt.pps[sn];
        const long long cn = gn - bt.pre[sn];
        constexpr unsigned UB = NV * ND * sizeof(double), VB = NV * NSD * sizeof(double);
        static_assert(UB % 16 == 0 && VB % 16 == 0, "bulk prefetch sizes are multiples of 16 bytes");
        bulk_prefetch_l2(pn->b.U[1 - pn->cur] + cn * (NV * ND), UB);
        if (pn->b.vstar) {
          bulk_prefetch_l2(pn->b.U[pn->cur] + cn * (NV * ND), UB);
          bulk_prefetch_l2(pn->b.vstar + cn * (size_t)(NV * NSD), VB);
        }
      }
    }
    const double dt = *p.b.dt;
    if (!(dt > 0.0)) continue;          // (warp-uniform)
    double c[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < D; ++k) c[k] = p.b.coef[k];
    const int nxt = 1 - p.cur;
    int ijk[3];
    cell_coords<D>(cell, p.geo, ijk);
    double* Uo = p.b.U[nxt] + cell * (NV * ND);
    double* vkeep = p.b.vstar ? p.b.vstar + cell * (size_t)(NV * NSD) : nullptr;
    const bool delta = vkeep && p.b.vok[cell] && (p.stamp & 15) != 0;
    const double* Un = p.b.U[p.cur] + cell * (NV * ND);
    float* dA = reinterpret_cast<float*>(A);
    float* dB = reinterpret_cast<float*>(B);
    // the face terms' weights of this cell's step, one product each
    for (int q = lane; q < 2 * D * n; q += 32) {
      const int k = q / (2 * n), r = q - k * 2 * n;
      const double ck = k == 0 ? c[0] : (k == 1 ? c[1] : c[2]);   // (registers, not a local array)
      cw[q] = ck * (r < n ? o->phi0w[r] : o->phi1w[r - n]);
    }
    __syncwarp();
    for (int e = lane; e < NV * ND; e += 32) {
      const int v = e / ND, i = e - v * ND;
      double acc = Uo[e];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
        const int ak = (i / st) % n;
        const int ts = tangential<D, n>(i, k);
        const long long flo = face_index<D>(p.geo, ijk, k, ijk[k]);
        const long long fhi = face_index<D>(p.geo, ijk, k, ijk[k] + 1);
        const double Glo = p.b.G[k][(flo * NV + v) * NF + ts];
        const double Ghi = p.b.G[k][(fhi * NV + v) * NF + ts];
        // u* -= dt/dx_k (phi1(a)/w_a Ghi - phi0(a)/w_a Glo), as two FMAs
        acc = fma(-cw[(2 * k + 1) * n + ak], Ghi, acc);
        acc = fma(cw[2 * k * n + ak], Glo, acc);
      }
      Uo[e] = acc;
      if (delta) dA[e] = narrow_f64_rz(acc - Un[e]);
      else A[e] = acc;
    }
    if (lane < NV) dmp_interval_lane<D>(p, p.b.cmm[p.cur], ijk, lohi, lane);
    __syncwarp();
    double lam = 0.0, mm[2 * NV];
    bool bad;
    if (delta) {
      // the projected change is added to the kept averages as the scan reads them
      const float* dv = project_f<D, N, true>(dA, dB, lane, 32);
      auto value = [vkeep, dv](int v, int s) {
        const int e = v * NSD + s;
        const double x = vkeep[e] + widen_f32(dv[e]);
        vkeep[e] = x;
        return x;
      };
      bad = check_values_warp<D>(value, NSD, lohi, p.gamma, mm, p.lam_mode ? &lam : nullptr,
                                 p.prec == ADG_PREC_MIXED_FP32, lane, p.gam2f);
    } else {
      const double* vs = apply_fx<D, NV, n, Ns, true>(A, B, P1m, lane, 32);
      auto value = [vkeep, vs](int v, int s) {
        const int e = v * NSD + s;
        const double x = vs[e];
        if (vkeep) vkeep[e] = x;
        return x;
      };
      bad = check_values_warp<D>(value, NSD, lohi, p.gamma, mm, p.lam_mode ? &lam : nullptr,
                                 p.prec == ADG_PREC_MIXED_FP32, lane, p.gam2f);
    }
    if (lane == 0) {
      int slot = -1;
      if (bad || p.force) {
        slot = atomicAdd(&p.b.counters[CNT_TROUBLED0 + nxt], 1);
        if (slot < p.cap) {
          p.b.list[nxt][slot] = (int)cell;
        } else {
          atomicOr(&p.b.counters[CNT_STATUS], 1);
          slot = -1;
        }
      }
      p.b.beta[nxt][cell] = (uint8_t)(slot >= 0);
      p.b.slot[nxt][cell] = slot;
      if (p.lam_mode) p.b.lam[cell] = lam;
      if (vkeep) p.b.vok[cell] = 1;
    }
#pragma unroll
    for (int j = 0; j < 2 * NV; ++j)
      if (lane == j) p.b.cmm[nxt][cell * 2 * NV + j] = mm[j];
    __syncwarp();
  }
}

}  // namespace adg
