// Subcell limiter kernels (Sec. 4.3-4.4): gather of the subcell patch from
// Eq. (ader.icbc), dimension-by-dimension WENO3 reconstruction, degree-2
// space-time predictor per subcell, sub-face Rusanov fluxes, finite volume
// update A (Eq. aderweno), reconstruction R (Eq. subcell.r) and the flux
// correction of unlimited face neighbours.  All work runs over the compacted
// troubled-cell list, in chunks of `chunk` cells that share the scratch.
#pragma once

#include "fixed.cuh"
#include "kernels_dg.cuh"

namespace adg {

__host__ __device__ __forceinline__ int ipow3(int k) { return k == 0 ? 1 : (k == 1 ? 3 : (k == 2 ? 9 : 27)); }

// Troubled cells handled by limiter pass `pass` of one state (0 past the end,
// and 0 for a state idle this step).  Pass c covers list entries
// [c * chunk, (c + 1) * chunk).
__device__ __forceinline__ int pass_len(const Params& p, int pass) {
  if (!(*p.b.dt > 0.0)) return 0;
  int nT = p.b.counters[CNT_TROUBLED0 + (1 - p.cur)];
  if (nT > p.cap) nT = p.cap;
  const int len = nT - pass * p.chunk;
  return len < 0 ? 0 : (len > p.chunk ? p.chunk : len);
}

// The pass a limiter kernel works on: its argument, or for the pass loop
// sized on the device (argument < 0) the pass stored after the prefix.
__device__ __forceinline__ int lim_pass(const Batch& bt, int pass) {
  return pass >= 0 ? pass : (int)bt.pre[bt.n + 1];
}

// Item t (a troubled cell of the current pass, counted over the batch) ->
// state index and the cell's position j within its state's pass.
struct LimItem {
  int s;
  int j;
};
__device__ __forceinline__ LimItem lim_item(const Batch& bt, long long t) {
  LimItem it;
  it.s = batch_state(bt, t);
  it.j = (int)(t - bt.pre[it.s]);
  return it;
}

// v^n at one subcell of cell `o` (Eq. ader.icbc): the stored subgrid data of a
// troubled cell, else the projection P(u^n) evaluated at that subcell.
template <int D, int N>
__device__ __forceinline__ void subcell_value(const Params& p, long long o, const int* s,
                                              const double* __restrict__ P1, double* out) {
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, Ns = DM::Ns, NSD = DM::NSD;
  if (p.b.beta[p.cur][o]) {
    const int slot = p.b.slot[p.cur][o];
    const int sidx = s[0] + Ns * (s[1] + (D == 3 ? Ns * s[2] : 0));
    const double* st = p.b.store[p.cur] + (size_t)slot * NV * NSD;
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v] = st[v * NSD + sidx];
    return;
  }
  const double* U = p.b.U[p.cur] + o * (NV * ND);
  const double* px = P1 + s[0] * n;
  const double* py = P1 + s[1] * n;
  const double* pz = P1 + (D == 3 ? s[2] : 0) * n;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const double* Uv = U + v * ND;
    double acc = 0.0;
    for (int c = 0; c < (D == 3 ? n : 1); ++c) {
      double accb = 0.0;
      for (int b = 0; b < n; ++b) {
        double acca = 0.0;
#pragma unroll
        for (int a = 0; a < n; ++a) acca += px[a] * Uv[a + n * (b + n * c)];
        accb += py[b] * acca;
      }
      acc += (D == 3 ? pz[c] : 1.0) * accb;
    }
    out[v] = acc;
  }
}

// v^n at local subcell loc[k] (may lie outside the cell, up to three
// layers) around cell ijk, with the ghost rules of the boundary kinds: a
// global subcell index outside the domain wraps (periodic), is clamped
// (transmissive: constant extrapolation), is mirrored with the wall-normal
// momentum negated (reflective: -1 - g below, 2 n - 1 - g above), or takes
// the face's fixed state (inflow).  The per-axis transforms apply in axis
// order.
template <int D, int N>
__device__ __forceinline__ void patch_value(const Params& p, const int* ijk, const int* loc,
                                            const double* __restrict__ P1, double* val) {
  using DM = Dims<D, N>;
  constexpr int NV = DM::NV, Ns = DM::Ns;
  const Geo& g = p.geo;
  int own[3] = {0, 0, 0}, sub[3] = {0, 0, 0}, mode[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const int ng = g.n[k] * Ns;
    int gi = ijk[k] * Ns + loc[k];
    if (gi < 0 || gi >= ng) {
      const int face = 2 * k + (gi < 0 ? 0 : 1);
      int kind = g.bc[face];
      int part = -1;
      if (kind == ADG_BC_FRONT) {
        // the ghost subcell's centre along the front's axis (unmapped index)
        const int j = g.front_axis[face];
        const double h = g.dx[j] / Ns;
        const double pos = g.x0[j] + ((ijk[j] * Ns + loc[j]) + 0.5) * h;
        part = front_part(g, face, pos, *p.b.tstart);
        kind = g.front_kind[face][part];
      }
      if (kind == ADG_BC_PERIODIC) {
        gi = (gi % ng + ng) % ng;
      } else {
        if (kind == ADG_BC_REFLECTIVE) {
          gi = gi < 0 ? -1 - gi : 2 * ng - 1 - gi;
          mode[k] = 1;
        } else if (kind == ADG_BC_INFLOW) {
          // which fixed state: 2 + 2 face an inflow face's, 14 + 2 face + part a front part's
          mode[k] = (part < 0) ? 2 + 2 * face : 14 + 2 * face + part;
        }
        gi = gi < 0 ? 0 : (gi >= ng ? ng - 1 : gi);
      }
    }
    own[k] = gi / Ns;
    sub[k] = gi - own[k] * Ns;
  }
  subcell_value<D, N>(p, cell_index<D>(own, g), sub, P1, val);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    if (mode[k] == 1) {
      val[1 + k] = -val[1 + k];
    } else if (mode[k] >= 2) {
      // 2 + 2 face: the inflow face's state; 14 + 2 face + part: a front part's
      const int m = mode[k] - 2;
      const double* q = (m < 12) ? g.bstate[m / 2] : g.front_state[(m - 12) / 2][(m - 12) % 2];
#pragma unroll
      for (int v = 0; v < NV; ++v) val[v] = q[v];
    }
  }
}

// L0: patch[j][v][L^d], local subcell -3..Ns+2 per axis around troubled cell
// list[chunk0 + j], ghosts by patch_value.
// Offset of local subcell loc (-3 .. Ns+2 per axis) in a limiter patch.
template <int D, int L>
__device__ __forceinline__ int patch_offset(const int* loc) {
  int off = 0, m = 1;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    off += (loc[k] + 3) * m;
    m *= L;
  }
  return off;
}

// Position j2 in the current pass of the troubled neighbour of cell ijk across
// its face on side `side` (-1, +1) of axis k, or -1.  The neighbour's interior
// subcells next to that face are the cell's ghost subcells there: the same
// level-n averages (both patches take them by global subcell index) and the
// same reconstruction, hence the same predictor bit for bit, so the
// neighbour's is used and the ghosts are not computed again.  (A moving front
// cuts its face by the unwrapped coordinate, which a periodic image does not
// share: with one, periodic neighbours are left out.)  A 3D N = 3 cell has 294
// face ghosts beside its 343 subcells.  The patch kernel writes the table nbr
// of the pass (looking the neighbour up in the predictor cost more than the
// ghosts it saved where troubled cells lie scattered).  Measured, the limiter
// per step: closed box 37 x 30 x 26 N = 2 mixed 4.10 -> 3.44 ms, 3D explosion
// 64^3 N = 3 mixed (noise, scattered cells) 79.3 -> 76.8 ms, 512^2 N = 5 mixed
// 1.54 -> 1.44 ms.
template <int D>
__device__ __forceinline__ int find_shared(const Params& p, int pass, const int* ijk, int k, int side) {
  const Geo& g = p.geo;
  int nb[3];
  if (!face_neighbour<D>(g, ijk, k, side, nb)) return -1;
  if (nb[k] != ijk[k] + side) {
    for (int f = 0; f < 2 * D; ++f)
      if (g.bc[f] == ADG_BC_FRONT) return -1;
  }
  const int slot = p.b.slot[1 - p.cur][cell_index<D>(nb, g)];
  if (slot < 0) return -1;
  const int j2 = slot - pass * p.chunk;
  return j2 >= 0 && j2 < pass_len(p, pass) ? j2 : -1;
}

// The table's entry of item j (-1 everywhere for the patches of the
// no-allocation entry point, which has no table).
template <int D>
__device__ __forceinline__ int shared_neighbour(const Params& p, long long j, int k, int side) {
  return p.b.nbr ? p.b.nbr[j * (2 * D) + 2 * k + (side > 0 ? 1 : 0)] : -1;
}

// Limiter patch of each troubled cell: v^n on L^D subcells (the cell and
// three layers around it, Eq. ader.icbc), each value as patch_value gives it
// and in the same operation order, gathered by neighbour boxes.  The patch
// splits into 3^D boxes, one per neighbour offset o in {-1, 0, 1}^D (per axis
// the 3 subcell layers below the cell, its Ns subcells, or the 3 layers
// above).  A box whose owner is one cell reached without a boundary ghost
// rule (an interior or periodic neighbour) is copied from that cell's stored
// subcell data when it was troubled at level n, else projected from its DOFs
// by tensor passes of P, axis by axis over the box (about n FMA per value and
// axis instead of n^D per value); other boxes take patch_value per subcell.
// One block per (troubled cell, box).
template <int D, int N>
__global__ void __launch_bounds__(128) k_lim_patch(Batch bt, int pass) {
  pass = lim_pass(bt, pass);
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, Ns = DM::Ns, NSD = DM::NSD, L = DM::L, LD = DM::LD;
  constexpr int NB = ipow(3, D), NR = ipow(n, D - 1);
  __shared__ double P1[Ns * n];
  __shared__ double Us[NV * ND];
  __shared__ double T1[NV * Ns * NR];                     // after the x pass
  __shared__ double T2[(D == 3) ? NV * Ns * Ns * n : 1];  // after the y pass (3D)
  for (int i = threadIdx.x; i < Ns * n; i += blockDim.x) P1[i] = bt.pps[0]->ops->P1[i];
  for (long long item = blockIdx.x; item < bt.pre[bt.n] * NB; item += gridDim.x) {
    __syncthreads();
    const long long t = item / NB;
    const int b = (int)(item - t * NB);
    const LimItem it = lim_item(bt, t);
    const Params& p = *bt.pps[it.s];
    const Geo& g = p.geo;
    const int j = it.j;
    const long long cell = p.b.list[1 - p.cur][pass * p.chunk + j];
    int ijk[3];
    cell_coords<D>(cell, g, ijk);
    int o[3] = {0, 0, 0}, lo[3] = {0, 0, 0}, R[3] = {1, 1, 1}, own[3] = {0, 0, 0};
    bool simple = true;
    {
      int bb = b;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        o[k] = bb % 3 - 1;
        bb /= 3;
        lo[k] = o[k] < 0 ? -3 : (o[k] == 0 ? 0 : Ns);
        R[k] = o[k] == 0 ? Ns : 3;
        int c = ijk[k] + o[k];
        if (c < 0 || c >= g.n[k]) {
          if (g.periodic[k]) c = (c + g.n[k]) % g.n[k];
          else simple = false;
        }
        own[k] = c;
      }
    }
    const int nbox = R[0] * R[1] * R[2];
    double* dst = p.b.patch + (size_t)j * NV * LD;
    if (threadIdx.x == 0) {
      // a face neighbour's box: the table of shared ghosts
      int k = 0, faces = 0;
#pragma unroll
      for (int x = 0; x < D; ++x)
        if (o[x] != 0) {
          k = x;
          ++faces;
        }
      const int side = k == 0 ? o[0] : (k == 1 ? o[1] : o[2]);
      if (faces == 1) p.b.nbr[(long long)j * (2 * D) + 2 * k + (side > 0 ? 1 : 0)] = find_shared<D>(p, pass, ijk, k, side);
    }
    if (!simple) {
      // a ghost rule applies along some axis: per subcell
      for (int e = threadIdx.x; e < nbox; e += blockDim.x) {
        int r = e, loc[3] = {0, 0, 0};
#pragma unroll
        for (int k = 0; k < D; ++k) {
          loc[k] = lo[k] + r % R[k];
          r /= R[k];
        }
        double val[NV];
        patch_value<D, N>(p, ijk, loc, P1, val);
        const int off = patch_offset<D, L>(loc);
#pragma unroll
        for (int v = 0; v < NV; ++v) dst[v * LD + off] = val[v];
      }
      continue;
    }
    const long long oc = cell_index<D>(own, g);
    if (p.b.beta[p.cur][oc]) {
      // the owner's subcell data of level n
      const double* st = p.b.store[p.cur] + (size_t)p.b.slot[p.cur][oc] * NV * NSD;
      for (int e = threadIdx.x; e < NV * nbox; e += blockDim.x) {
        const int v = e / nbox;
        int r = e - v * nbox, loc[3] = {0, 0, 0}, sidx = 0, m = 1;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          loc[k] = lo[k] + r % R[k];
          r /= R[k];
          sidx += (loc[k] - o[k] * Ns) * m;
          m *= Ns;
        }
        dst[v * LD + patch_offset<D, L>(loc)] = st[v * NSD + sidx];
      }
      continue;
    }
    // P(u^n) of the owner over the box, by tensor passes (x, y[, z])
    const double* U = p.b.U[p.cur] + oc * (NV * ND);
    for (int e = threadIdx.x; e < NV * ND; e += blockDim.x) Us[e] = U[e];
    __syncthreads();
    for (int e = threadIdx.x; e < NV * R[0] * NR; e += blockDim.x) {
      const int v = e / (R[0] * NR);
      const int r = e - v * (R[0] * NR);
      const int sx = r % R[0], rest = r / R[0];
      const double* px = P1 + (lo[0] + sx - o[0] * Ns) * n;
      const double* u = Us + v * ND + rest * n;
      double acc = 0.0;
#pragma unroll
      for (int a = 0; a < n; ++a) acc += px[a] * u[a];
      T1[(v * R[0] + sx) * NR + rest] = acc;
    }
    __syncthreads();
    if (D == 2) {
      for (int e = threadIdx.x; e < NV * R[0] * R[1]; e += blockDim.x) {
        const int v = e / (R[0] * R[1]);
        const int r = e - v * (R[0] * R[1]);
        const int sx = r % R[0], sy = r / R[0];
        const double* py = P1 + (lo[1] + sy - o[1] * Ns) * n;
        const double* t1 = T1 + (v * R[0] + sx) * NR;
        double accb = 0.0;
#pragma unroll
        for (int bb = 0; bb < n; ++bb) accb += py[bb] * t1[bb];
        const int loc[3] = {lo[0] + sx, lo[1] + sy, 0};
        dst[v * LD + patch_offset<D, L>(loc)] = 0.0 + accb;   // as 0 + 1 * accb in subcell_value
      }
    } else {
      for (int e = threadIdx.x; e < NV * R[0] * R[1] * n; e += blockDim.x) {
        const int v = e / (R[0] * R[1] * n);
        int r = e - v * (R[0] * R[1] * n);
        const int sx = r % R[0];
        r /= R[0];
        const int sy = r % R[1], c = r / R[1];
        const double* py = P1 + (lo[1] + sy - o[1] * Ns) * n;
        const double* t1 = T1 + (v * R[0] + sx) * NR + c * n;
        double accb = 0.0;
#pragma unroll
        for (int bb = 0; bb < n; ++bb) accb += py[bb] * t1[bb];
        T2[((v * R[0] + sx) * R[1] + sy) * n + c] = accb;
      }
      __syncthreads();
      for (int e = threadIdx.x; e < NV * nbox; e += blockDim.x) {
        const int v = e / nbox;
        int r = e - v * nbox;
        const int sx = r % R[0];
        r /= R[0];
        const int sy = r % R[1], sz = r / R[1];
        const double* pz = P1 + (lo[2] + sz - o[2] * Ns) * n;
        const double* t2 = T2 + ((v * R[0] + sx) * R[1] + sy) * n;
        double acc = 0.0;
#pragma unroll
        for (int c = 0; c < n; ++c) acc += pz[c] * t2[c];
        const int loc[3] = {lo[0] + sx, lo[1] + sy, lo[2] + sz};
        dst[v * LD + patch_offset<D, L>(loc)] = acc;
      }
    }
  }
}


// 1D WENO3 on five consecutive subcell averages u[0..4] (target subcell u[2]):
// values of the reconstruction at the 3 GL nodes x = 1/2, 1/2 -+ y of the
// target subcell, y^2 = 3/20.
//
// The FP64 pipe bounds the sweeps, so the stencils are written in the first
// and second differences they share.  The parabola of stencil k has the average
// u[2] over the target, the slope b_k at its middle and the second derivative
// s_k (the stencil's second difference):
//   p_k(x) = u[2] + b_k (x - 1/2) + s_k ((x - 1/2)^2 / 2 - 1/24),
//   sigma_k = int_0^1 (p')^2 + (p'')^2 = b_k^2 + 13/12 s_k^2,
// and the interface slopes d1 = u[2] - u[1], d2 = u[3] - u[2] give
//   b = d1 + s_0 / 2, d1 + s_1 / 2, d2 - s_2 / 2.
// About 54 FP64 operations, the division among them; in the monomials of each
// stencil they were about 97.
//
// Weights w_k = lambda_k / (sigma_k + eps)^8, normalised: with t_k the
// sigma_k + eps over the power of two of the smallest and a_k = lambda_k
// prod_{j != k} t_j^8 they are a_k / sum a, one division.  t_k is cut at 2^50, so
// that no product overflows whatever the data's magnitude, and a stencil that far
// from the smoothest has no weight (below 2^-370 of the largest: what it would
// add lies under the last place of the smoothest one's differences).
//
// Measured (GB300, 3D explosion 33 x 29 x 30, N = 3): the three sweeps of 5611
// troubled cells 30.2 ms; in the monomial form 46.1 ms for 4883 (means of two
// launches).  2D N = 5, 146 patches: 94 -> 60 us.
// (t over the power of two with the exponent bits emin, by integer operations on
// a positive number's bits; compared before the rebias, which can wrap)
__device__ __forceinline__ double weno_scaled(double t, int emin, bool* far) {
  const int up = __double2hiint(t) - emin, one = 1023 << 20, cut = 50 << 20;
  *far = up >= cut;
  return up >= cut ? __hiloint2double(one + cut, 0) : __hiloint2double(one + up, __double2loint(t));
}

__device__ __forceinline__ void weno3(const double* u, const Ops* __restrict__ o, double* out) {
  const double d0 = u[1] - u[0], d1 = u[2] - u[1], d2 = u[3] - u[2], d3 = u[4] - u[3];
  const double s[3] = {d1 - d0, d2 - d1, d3 - d2};
  const double b[3] = {fma(0.5, s[0], d1), fma(0.5, s[1], d1), fma(-0.5, s[2], d2)};
  double t[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) t[k] = fma(b[k], b[k], fma((13.0 / 12.0) * s[k], s[k], WENO_EPS));
  // over the smallest's power of two (t >= eps > 0; NaN stays in b and s)
  const int h0 = __double2hiint(t[0]), h1 = __double2hiint(t[1]), h2 = __double2hiint(t[2]);
  const int emin = min(h0, min(h1, h2)) & 0x7ff00000;
  bool far[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double x = weno_scaled(t[k], emin, &far[k]);
    x = x * x;
    x = x * x;
    t[k] = x * x;
  }
  const double a0 = far[0] ? 0.0 : t[1] * t[2];
  const double a1 = far[1] ? 0.0 : WENO_LAMBDA_C * (t[0] * t[2]);
  const double a2 = far[2] ? 0.0 : t[0] * t[1];
  const double inv = 1.0 / (a0 + a1 + a2);
  const double B = (a0 * b[0] + a1 * b[1] + a2 * b[2]) * inv;
  const double S = (a0 * s[0] + a1 * s[1] + a2 * s[2]) * inv;
  const double y = 0.5 - o->xi3[0];
  const double side = fma(1.0 / 30.0, S, u[2]);       // y^2 / 2 - 1/24 = 1/30
  out[0] = fma(-y, B, side);
  out[1] = fma(-1.0 / 24.0, S, u[2]);
  out[2] = fma(y, B, side);
}

// FP32 form of weno3 (mixed precision).  (sigma_k + eps)^8 underflows in FP32
// for smooth data, so every t_k is divided by the smallest:
// t_k = ((sigma_min + eps) / (sigma_k + eps))^8 lies in [0, 1] and the weights
// lambda_k t_k / sum_j lambda_j t_j are those of weno3 (an underflow to 0 is
// the exact limit).  The nodal values come straight from the stencil
// averages (Wf = E C per stencil).
__device__ __forceinline__ void weno3f(const float* u, const Ops* __restrict__ o, float* out) {
  float sg[3], v[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float* C = o->Cf[k];
    const float c1 = C[0] * u[k] + C[1] * u[k + 1] + C[2] * u[k + 2];
    const float c2 = C[3] * u[k] + C[4] * u[k + 1] + C[5] * u[k + 2];
    sg[k] = c1 * (c1 + 2.0f * c2) + (16.0f / 3.0f) * c2 * c2 + (float)WENO_EPS;
    const float* W = o->Wf[k];
#pragma unroll
    for (int a = 0; a < 3; ++a) v[k][a] = W[a * 3] * u[k] + W[a * 3 + 1] * u[k + 1] + W[a * 3 + 2] * u[k + 2];
  }
  const float smin = fminf(sg[0], fminf(sg[1], sg[2]));
  float wt[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float r = smin / sg[k];
    r = r * r;
    r = r * r;
    wt[k] = r * r * (k == 1 ? (float)WENO_LAMBDA_C : 1.0f);
  }
  const float inv = 1.0f / (wt[0] + wt[1] + wt[2]);
#pragma unroll
  for (int a = 0; a < 3; ++a) out[a] = (wt[0] * v[0][a] + wt[1] * v[1][a] + wt[2] * v[2][a]) * inv;
}

// L1..L3: sweep along axis K.  Input extents (L or Ns+2 per axis) with NNIN
// nodal values per element; the output has extent Ns+2 along K and 3 NNIN
// nodes (the new nodal index is the slowest digit).
// T: the sweeps' precision (double; float for the mixed-precision FP32
// reconstruction); the patch (input of the x sweep) is always FP64.
//
// One thread takes sweep_run neighbouring targets along K: their stencils share
// all but one value each, and index arithmetic was 100 of the 234 instructions
// that one FP32 target took by itself.  Measured (GB300), x / y / z: 40^3 N = 3
// mixed 566 / 972 / 1982 -> 366 / 716 / 1840 us, 33 x 29 x 30 N = 3 FP64 4.1 / 8.5
// / 17.6 -> 3.6 / 7.5 / 16.0 ms.  In 2D FP64, bound by the FP64 pipe with a
// hundredth of the targets per cell, one target per thread stays: 146 patches
// at N = 5 take 22 + 37 us, in runs of three 25 + 53.
template <int D, typename T>
constexpr int sweep_run = (D == 3 || sizeof(T) == sizeof(float)) ? 3 : 1;

template <int D, int N, int K, typename T>
__global__ void __launch_bounds__(256) k_lim_sweep(Batch bt, int pass) {
  using DM = Dims<D, N>;
  constexpr int NV = DM::NV, L = DM::L, NE = DM::NE, R = sweep_run<D, T>, NR = (NE + R - 1) / R;
  constexpr int I0 = (0 < K) ? NE : L, I1 = (1 < K) ? NE : L, I2 = (D < 3) ? 1 : ((2 < K) ? NE : L);
  constexpr int O0 = (0 <= K) ? NE : L, O1 = (1 <= K) ? NE : L, O2 = (D < 3) ? 1 : ((2 <= K) ? NE : L);
  constexpr int NNIN = ipow(3, K);
  constexpr int INSZ = I0 * I1 * I2 * NNIN;
  constexpr int OUTSZ = O0 * O1 * O2 * NNIN;          // elements, each producing 3 values
  constexpr int RUNS = OUTSZ / NE * NR;               // runs of targets
  constexpr int R0 = K == 0 ? NR : O0, R1 = K == 1 ? NR : O1;
  constexpr int STRIDE = ((K == 0) ? 1 : (K == 1 ? I0 : I0 * I1)) * NNIN;       // input, along K
  constexpr int OSTRIDE = ((K == 0) ? 1 : (K == 1 ? O0 : O0 * O1)) * NNIN * 3;  // output
  const Ops* ops = bt.pps[0]->ops;
  for (long long eg = blockIdx.x * (long long)blockDim.x + threadIdx.x;
       eg < bt.pre[bt.n] * (NV * RUNS); eg += (long long)gridDim.x * blockDim.x) {
    const long long t = eg / (NV * RUNS);
    const LimItem it = lim_item(bt, t);
    const Params& p = *bt.pps[it.s];
    int r = (int)(eg - t * (NV * RUNS));
    const int v = r / RUNS;
    r -= v * RUNS;
    const long long jv = (long long)it.j * NV + v;
    const int node = r % NNIN;
    r /= NNIN;
    int x0 = r % R0;
    r /= R0;
    int x1 = r % R1;
    int x2 = r / R1;
    const int first = R * (K == 0 ? x0 : (K == 1 ? x1 : x2));
    if (K == 0) x0 = first;
    if (K == 1) x1 = first;
    if (K == 2) x2 = first;
    // input element whose axis-K index equals the output's (stencil x_K .. x_K + 4)
    const size_t src_off = jv * INSZ + (size_t)(x0 + I0 * (x1 + I1 * x2)) * NNIN + node;
    T u[R + 4];
    if (K == 0) {
      const double* src = p.b.patch + src_off;
#pragma unroll
      for (int q = 0; q < R + 4; ++q) u[q] = (T)(first + q < NE + 4 ? src[q * STRIDE] : 0.0);
    } else {
      const T* src = reinterpret_cast<const T*>(p.b.sweep[K > 0 ? K - 1 : 0]) + src_off;
#pragma unroll
      for (int q = 0; q < R + 4; ++q) u[q] = first + q < NE + 4 ? src[q * STRIDE] : T(0);
    }
    T* dst = reinterpret_cast<T*>(p.b.sweep[K]) + jv * (size_t)OUTSZ * 3 +
             (size_t)(x0 + O0 * (x1 + O1 * x2)) * NNIN * 3 + node;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (first + i >= NE) break;
      T res[3];
      if constexpr (sizeof(T) == sizeof(double)) weno3(u + i, ops, res);
      else weno3f(u + i, ops, res);
#pragma unroll
      for (int a = 0; a < 3; ++a) dst[i * OSTRIDE + a * NNIN] = res[a];
    }
  }
}

// L4: degree-2 space-time predictor (Eq. pde.nc.dg2 with 3 GL nodes per axis
// and in time, 3 Picard sweeps) on the subcells whose traces the sub-face
// fluxes use: the Ns^d interior subcells and the Ns^(d-1) ghost subcells
// facing each of the 2d cell faces.
constexpr int SUBS_PER_BLOCK_2D = 4;
constexpr int SUBS_PER_BLOCK_3D = 2;

// index in the (Ns+2)^d block (array index = local + 1) of the r-th subcell
// of the interior + face-ghost set
template <int D, int Ns>
__device__ __forceinline__ int cross_subcell(int r) {
  constexpr int NE = Ns + 2, NSD = ipow(Ns, D), NSF = ipow(Ns, D - 1);
  int c[3] = {0, 0, 0};
  if (r < NSD) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      c[k] = r % Ns + 1;
      r /= Ns;
    }
  } else {
    r -= NSD;
    const int k = r / (2 * NSF);
    r -= k * 2 * NSF;
    const int side = r / NSF;
    int t = r - side * NSF;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (a == k) {
        c[a] = side ? Ns + 1 : 0;
      } else {
        c[a] = t % Ns + 1;
        t /= Ns;
      }
    }
  }
  return c[0] + NE * (c[1] + NE * c[2]);
}

// Whether subcell r of an item's interior + face-ghost set (cross_subcell) is a
// ghost that a troubled neighbour of the pass computes.
template <int D, int Ns>
__device__ __forceinline__ bool ghost_elsewhere(const Params& p, long long j, int r) {
  constexpr int NSD = ipow(Ns, D), NSF = ipow(Ns, D - 1);
  if (r < NSD) return false;
  r -= NSD;
  const int k = r / (2 * NSF);
  const int side = (r - k * 2 * NSF) / NSF;
  return shared_neighbour<D>(p, j, k, side ? 1 : -1) >= 0;
}

// L4 in mixed precision with some sweeps in each precision: n32 (1..3) of the
// three run in FP32, the others in FP64 after them (the same n32 for the whole
// launch, so every block takes the same barriers).  WT: the element type of
// the reconstruction.
template <int D, int N, typename WT>
__global__ void __launch_bounds__(256) k_lim_predict(Batch bt, int pass, int n32) {
  using DM = Dims<D, N>;
  constexpr int NV = DM::NV, NST3 = DM::NST3, ND3 = DM::ND3, NED = DM::NED, Ns = DM::Ns;
  constexpr int NCROSS = DM::NSD + 2 * D * DM::NSF;
  constexpr int SPB = (D == 2) ? SUBS_PER_BLOCK_2D : SUBS_PER_BLOCK_3D;
  __shared__ double su[SPB][NV * ND3];
  __shared__ double sq[SPB][NV * NST3];
  __shared__ double sF[SPB][D * NV * NST3];
  __shared__ float suf[SPB][NV * ND3];
  __shared__ float sqf[SPB][NV * NST3];
  __shared__ float sFf[SPB][D * NV * NST3];
  __shared__ double D3[9], K3[9];
  __shared__ float D3f[9], K3f[9];
  if (threadIdx.x < 9) {
    const Ops* o = bt.pps[0]->ops;
    D3[threadIdx.x] = o->D3[threadIdx.x];
    K3[threadIdx.x] = o->Kt3[threadIdx.x];
    D3f[threadIdx.x] = (float)o->D3[threadIdx.x];
    K3f[threadIdx.x] = (float)o->Kt3[threadIdx.x];
  }
  const int grp = threadIdx.x / NST3, lt = threadIdx.x - grp * NST3;
  const bool active_thread = grp < SPB;
  const long long total = bt.pre[bt.n] * NCROSS;
  for (long long base = (long long)blockIdx.x * SPB; base < total;
       base += (long long)gridDim.x * SPB) {
    const long long item = base + grp;
    const bool live = active_thread && item < total;
    const long long tg = live ? item / NCROSS : 0;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j = it.j;
    const int sc = live ? cross_subcell<D, Ns>((int)(item - tg * NCROSS)) : 0;
    double c[3];
    float cf[3];
    {
#pragma unroll
      for (int k = 0; k < D; ++k) {
        c[k] = p.b.coef[3 + k];
        cf[k] = (float)c[k];
      }
    }
    const double gm1 = p.gamma - 1.0;
    const WT* W = reinterpret_cast<const WT*>(p.b.sweep[D - 1]);   // [j][v][NED][ND3]
    __syncthreads();
    if (live) {
      for (int e = lt; e < NV * ND3; e += NST3) {
        const int v = e / ND3, i = e - v * ND3;
        su[grp][e] = (double)W[((j * NV + v) * NED + sc) * ND3 + i];
      }
    }
    __syncthreads();
    if (live) {
      for (int e = lt; e < NV * ND3; e += NST3) suf[grp][e] = (float)su[grp][e];
      for (int e = lt; e < NV * NST3; e += NST3) {
        const int v = e / NST3, l = e - v * NST3;
        sqf[grp][e] = (float)su[grp][v * ND3 + (l % ND3)];
      }
    }
    __syncthreads();
    for (int it = 0; it < n32; ++it) {
      if (live) picard_flux<D, 3, float>(sqf[grp], sFf[grp], (float)gm1, lt, NST3);
      __syncthreads();
      if (live) picard_deriv<D, 3, float>(sFf[grp], sqf[grp], D3f, cf, lt, NST3);
      __syncthreads();
      if (live) picard_time<D, 3, float>(sqf[grp], suf[grp], K3f, lt, NST3);
      __syncthreads();
    }
    if (live)
      for (int e = lt; e < NV * NST3; e += NST3) sq[grp][e] = (double)sqf[grp][e];
    __syncthreads();
    for (int it = n32; it < 3; ++it) {
      if (live) picard_flux<D, 3, double>(sq[grp], sF[grp], gm1, lt, NST3);
      __syncthreads();
      if (live) picard_deriv<D, 3, double>(sF[grp], sq[grp], D3, c, lt, NST3);
      __syncthreads();
      if (live) picard_time<D, 3, double>(sq[grp], su[grp], K3, lt, NST3);
      __syncthreads();
    }
    if (live) {
      double* dst = p.b.qsub + ((size_t)j * NED + sc) * (size_t)(NV * NST3);
      for (int e = lt; e < NV * NST3; e += NST3) dst[e] = sq[grp][e];
    }
  }
}

// The FP64 subcell predictor of a warp's subcells with its contractions on the
// FP64 pipe (lanes, lines and operators as in k_lim_predict_i): x[v] the lane's
// reconstruction on entry, x[m NV + v] its three time nodes on return.  For
// magnitudes outside the fixed-point range, which are rare: out of line, rolled.
template <int D>
__device__ __noinline__ void sub_predict_fp64(double* x, const double* ck, double gm1, const Ops* o, int sx,
                                              int sy, int sz, int a, int b, int c) {
  constexpr int NV = D + 2;
  constexpr unsigned FULL = 0xffffffffu;
  double u[NV], S[3][NV];
  for (int v = 0; v < NV; ++v) {
    u[v] = x[v];
    x[NV + v] = x[2 * NV + v] = u[v];
  }
#pragma unroll 1
  for (int it = 0; it < 3; ++it) {
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {
      double Q[NV], F[D][D + 2];
#pragma unroll
      for (int v = 0; v < NV; ++v) Q[v] = x[m * NV + v];
      euler_fluxes_sym<D>(Q, gm1, F);
#pragma unroll 1
      for (int v = 0; v < NV; ++v) {
        double s = 0.0;
#pragma unroll 1
        for (int k = 0; k < D; ++k) {
          const int base = k == 0 ? sx : (k == 1 ? sy : sz), st = k == 0 ? 1 : (k == 1 ? 3 : 9);
          const double* row = o->D3 + 3 * (k == 0 ? a : (k == 1 ? b : c));
          double t = 0.0;
          for (int j = 0; j < 3; ++j) t = fma(row[j], __shfl_sync(FULL, F[k][v], base + j * st), t);
          s = fma(ck[k], t, s);
        }
        S[m][v] = s;
      }
    }
#pragma unroll 1
    for (int m = 0; m < 3; ++m)
      for (int v = 0; v < NV; ++v) {
        double t = 0.0;
        for (int j = 0; j < 3; ++j) t = fma(o->Kt3[3 * m + j], S[j][v], t);
        x[m * NV + v] = u[v] - t;
      }
  }
}

// L4 in FP64: the subcell predictor in registers with its contractions on the
// integer pipes (fixed.cuh).  What bounds the FP64 limiter is the FP64 pipe (two
// operations per clock and multiprocessor): of the 22 FP64 operations that a
// 3D space-time node and variable cost per sweep, 16 were the contractions.
//
// Lane l works on spatial node l (3D: 27 nodes of one subcell; 2D: 9 nodes of
// each of three subcells) and holds its three time nodes.  The fluxes F_k of a
// time node are put on one scale per subcell and variable (the largest
// magnitude over its nodes and axes; a smooth subcell's values lie within the
// 6 bits that scale keeps below FP64's), the three operands of each line come
// from the lanes on it as integers by shuffles, and S = sum_k (c_k D) x_k F_k
// is one exact integer sum over the axes: c_k is folded into the operator once
// per state.  The time solve acts on the lane's own S, brought to the largest
// of its three scales, and only its result becomes a double again:
// q = u - Ktau S.  The first sweep starts from u (x) 1: one space term, and
// q_m = u - kappa_m S with kappa = Ktau 1.  FP64 operations per sweep, node and
// variable: the flux (4.4 in 3D, 4.1 in 2D) and one subtraction.
//
// Measured (GB300, 3D explosion 33 x 29 x 30, N = 3): 47 ms for 4883 troubled
// cells (mean of two launches; 3.1 million subcells, FP64 pipe 63% busy), the
// former kernel with FP64 contractions from shared memory 174 ms; 2D N = 5, 146
// patches: 351 -> 113 us.
template <int D, int N, typename WT>
__global__ void __launch_bounds__(128) k_lim_predict_i(Batch bt) {
  using DM = Dims<D, N>;
  constexpr int NV = DM::NV, NST3 = DM::NST3, ND3 = DM::ND3, NED = DM::NED, Ns = DM::Ns;
  constexpr int NCROSS = DM::NSD + 2 * D * DM::NSF;
  constexpr int SPW = D == 2 ? 3 : 1;                   // subcells per warp
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ FxOp K3[9], kap[3];                        // Ktau and its row sums
  __shared__ int s_gK;
  const Ops* o = bt.pps[0]->ops;                        // (the subcell operators do not depend on N)
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    // scale exponents from the row sums, then one entry per lane
    double ks = 0.0;
    for (int m = 0; m < 3; ++m) {
      const double r = fabs(o->Kt3[3 * m]) + fabs(o->Kt3[3 * m + 1]) + fabs(o->Kt3[3 * m + 2]);
      ks = r > ks ? r : ks;
    }
    const int gK = fx_scale(ks);
    if (lane < 9) K3[lane] = fx_op(o->Kt3[lane], gK);
    else if (lane < 12) {
      const double* r = o->Kt3 + 3 * (lane - 9);
      kap[lane - 9] = fx_op(r[0] + r[1] + r[2], gK);
    }
    if (lane == 0) s_gK = gK;
  }
  __syncthreads();
  const int gK = s_gK;
  const int l = lane < 27 ? lane : 26;                  // idle lanes mirror lane 26
  const int grp = D == 2 ? l / 9 : 0, node = l - grp * ND3;
  const int a = node % 3, b = (node / 3) % 3, c = D == 3 ? node / 9 : 0;
  const int sx = l - a, sy = l - 3 * b, sz = l - 9 * c; // first lanes of this node's lines
  FxOp row[D][3] = {};                                  // this node's rows of c_k D3
  int gD = 0, state = -1;
  const int wpb = blockDim.x >> 5;
  const long long total = bt.pre[bt.n] * NCROSS;
  const long long groups = (total + SPW - 1) / SPW;
  for (long long gi = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); gi < groups;
       gi += (long long)gridDim.x * wpb) {
    const long long item = gi * SPW + grp;
    const long long tg = item < total ? item / NCROSS : bt.pre[bt.n] - 1;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j0 = it.j;
    const int r = item < total ? (int)(item - tg * NCROSS) : 0;
    const bool needed = item < total && !ghost_elsewhere<D, Ns>(p, it.j, r);
    if (!__any_sync(FULL, needed)) continue;
    const bool live = needed && lane < 27;
    const int sc = cross_subcell<D, Ns>(r);
    if (__any_sync(FULL, it.s != state)) {
      // the rows of c_k D3 of this lane's state (they change with its step)
      state = it.s;
      double cs = 0.0, rs = 0.0;
#pragma unroll
      for (int k = 0; k < D; ++k) cs += p.b.coef[3 + k];
      for (int m = 0; m < 3; ++m) {
        const double r = fabs(o->D3[3 * m]) + fabs(o->D3[3 * m + 1]) + fabs(o->D3[3 * m + 2]);
        rs = r > rs ? r : rs;
      }
      gD = fx_scale(cs * rs);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const int ak = k == 0 ? a : (k == 1 ? b : c);
#pragma unroll
        for (int j = 0; j < 3; ++j) row[k][j] = fx_op(p.b.coef[3 + k] * o->D3[ak * 3 + j], gD);
      }
    }
    const double gm1 = p.gamma - 1.0;
    const WT* W = reinterpret_cast<const WT*>(p.b.sweep[D - 1]);   // [j][v][NED][ND3]
    double u[NV], q[3][NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = (double)W[((j0 * NV + v) * NED + sc) * ND3 + node];
    // outside the range of the fixed-point products: fluxes by FX_E_MAX, results by
    // FX_B_MIN and FX_B_MAX, and fluxes of a variable below 2^-900 (not zero), which
    // may be below FX_E_MIN
    bool far = false;
#pragma unroll
    for (int v = 0; v < NV; ++v)
      far = far || (fx_key(u[v]) < ((1023u - 900u) << 21) && (fx_key(u[v]) | (unsigned)__double2loint(u[v])) != 0u);
    // S = sum_k c_k D x_k F_k(Q) at this node: Sv[v] 2^64 on the scale es[v]
    auto space_term = [&](const double* Q, long long* Sv, unsigned* es) {
      double F[D][D + 2];
      euler_fluxes_sym<D>(Q, gm1, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        unsigned key = fx_key(F[0][v]);
#pragma unroll
        for (int k = 1; k < D; ++k) key = max(key, fx_key(F[k][v]));
        unsigned e;
        if constexpr (D == 3) {
          e = __reduce_max_sync(FULL, key) >> 21;
        } else {
          const unsigned e0 = __reduce_max_sync(FULL, grp == 0 ? key : 0u);
          const unsigned e1 = __reduce_max_sync(FULL, grp == 1 ? key : 0u);
          const unsigned e2 = __reduce_max_sync(FULL, grp == 2 ? key : 0u);
          e = (grp == 0 ? e0 : (grp == 1 ? e1 : e2)) >> 21;
        }
        const unsigned ec = max(e, FX_E_MIN);
        FxAcc acc;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const int base = k == 0 ? sx : (k == 1 ? sy : sz);
          const int st = k == 0 ? 1 : (k == 1 ? 3 : 9);
          const FxVal f = fx_val(F[k][v], ec);
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            FxVal x;
            x.h = __shfl_sync(FULL, f.h, base + j * st);
            x.l = __shfl_sync(FULL, f.l, base + j * st);
            acc.add(x, row[k][j]);
          }
        }
        Sv[v] = acc.sum().r;
        es[v] = ec;
      }
    };
    // u - (R as a double), R on the scale of a dot product of S by Ktau
    auto close = [&](double u0, FxSum R, unsigned e) {
      const int bf = (int)e + gD + gK + 6;
      far = far || e >= FX_E_MAX || bf > FX_B_MAX || (bf < FX_B_MIN && R.r != 0);
      const double x = fx_double(R, bf);
      return u0 - (bf < FX_B_MIN ? 0.0 : x);
    };
    {
      long long S[NV];
      unsigned es[NV];
      space_term(u, S, es);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        FxVal x;
        x.l = (int)S[v];
        x.h = (int)((S[v] - x.l) >> 32);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          FxAcc acc;
          acc.add(x, kap[m]);
          q[m][v] = close(u[v], acc.sum(), es[v]);
        }
      }
    }
#pragma unroll 1
    for (int sweep = 1; sweep < 3; ++sweep) {
      long long S[3][NV];
      unsigned es[3][NV];
#pragma unroll
      for (int m = 0; m < 3; ++m) space_term(q[m], S[m], es[m]);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const unsigned e = max(max(es[0][v], es[1][v]), es[2][v]);
        FxVal x[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const unsigned sh = e - es[m][v];
          const long long s = S[m][v] >> (sh < 63u ? sh : 63u);
          x[m].l = (int)s;
          x[m].h = (int)((s - x[m].l) >> 32);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          FxAcc acc;
#pragma unroll
          for (int j = 0; j < 3; ++j) acc.add(x[j], K3[m * 3 + j]);
          q[m][v] = close(u[v], acc.sum(), e);
        }
      }
    }
    if (__any_sync(FULL, far)) {
      double x[3 * NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) x[v] = u[v];
      sub_predict_fp64<D>(x, p.b.coef + 3, gm1, o, sx, sy, sz, a, b, c);
      const bool own = D == 3 || (__ballot_sync(FULL, far) >> (9 * grp) & 0x1ffu) != 0u;
#pragma unroll
      for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (own) q[m][v] = x[m * NV + v];
    }
    if (live) {
      double* dst = p.b.qsub + ((size_t)j0 * NED + sc) * (size_t)(NV * NST3);
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int m = 0; m < 3; ++m) dst[v * NST3 + m * ND3 + node] = q[m][v];
    }
  }
}

// L4 in mixed precision with the whole subcell predictor in FP32 (the default
// of the FP32 subcell scheme): one warp per subcell, W subcells per block,
// each warp synchronised by __syncwarp alone.  The blocks loop over the pass's subcells.
template <int D>
struct LimWarps {
  static constexpr int W = (D == 2) ? 8 : 4;     // subcells per block (static shared memory)
};

template <int D, int N>
__global__ void __launch_bounds__(32 * LimWarps<D>::W) k_lim_predict_w(Batch bt) {
  using DM = Dims<D, N>;
  constexpr int NV = DM::NV, NST3 = DM::NST3, ND3 = DM::ND3, NED = DM::NED, Ns = DM::Ns;
  constexpr int NCROSS = DM::NSD + 2 * D * DM::NSF;
  constexpr int W = LimWarps<D>::W;
  __shared__ float suf[W][NV * ND3];
  __shared__ float sqf[W][NV * NST3];
  __shared__ float sFf[W][D * NV * NST3];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* u = suf[w];
  float* q = sqf[w];
  float* F = sFf[w];
  const long long total = bt.pre[bt.n] * NCROSS;
  for (long long item = (long long)blockIdx.x * W + w; item < total;
       item += (long long)gridDim.x * W) {
    const long long tg = item / NCROSS;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j = it.j;
    const int sc = cross_subcell<D, Ns>((int)(item - tg * NCROSS));
    float cf[3];
#pragma unroll
    for (int k = 0; k < D; ++k) cf[k] = p.b.coef_f[3 + k];
    const float gm1 = p.b.coef_f[6];
    const float* Wr = reinterpret_cast<const float*>(p.b.sweep[D - 1]);   // [j][v][NED][ND3]
    for (int e = lane; e < NV * ND3; e += 32) {
      const int v = e / ND3, i = e - v * ND3;
      u[e] = Wr[((j * NV + v) * NED + sc) * ND3 + i];
    }
    __syncwarp();
    for (int e = lane; e < NV * NST3; e += 32) {
      const int v = e / NST3, l = e - v * NST3;
      q[e] = u[v * ND3 + (l % ND3)];
    }
    __syncwarp();
    for (int sweep = 0; sweep < 3; ++sweep) {
      picard_flux<D, 3, float>(q, F, gm1, lane, 32);
      __syncwarp();
      picard_deriv_sub<D>(F, q, cf, lane, 32);
      __syncwarp();
      picard_time_sub<D>(q, u, lane, 32);
      __syncwarp();
    }
    float* dst = reinterpret_cast<float*>(p.b.qsub) + ((size_t)j * NED + sc) * (size_t)(NV * NST3);
    for (int e = lane; e < NV * NST3; e += 32) dst[e] = q[e];
    __syncwarp();
  }
}

// Face traces of the 2D subcell predictor, the input of k_lim_flux_t2: for
// each troubled cell j, axis k, sub-face e normal to k (the enumeration of
// k_lim_flux) and side (0: the left subcell's trace at its high end, 1: the
// right subcell's at its low end), 9 points times 4 variables, the point
// t = (tangential node digit) + 3 (time node).
template <int N>
struct SubTraces2 {
  static constexpr int Ns = 2 * N + 1, NFK = (Ns + 1) * Ns, NP = 9;
  static constexpr long long per_cell = 2LL * NFK * 2 * 4 * NP;     // floats
  __host__ __device__ static constexpr long long offset(int k, int e, int side) {
    return ((long long)(k * NFK + e) * 2 + side) * 4 * NP;
  }
};

// The same subcell predictor in 2D in registers, three subcells per warp:
// lane l < 27 works on subcell l / 9 of the warp's three and holds its spatial
// node (a, b) = (l % 3, (l / 3) % 3) with the three time nodes.  The space
// derivatives take their three operands from the lanes on the node's line by
// warp shuffles; the time solve (Ktau) runs on the lane's own time nodes; the
// first sweep, from u (x) 1, forms the space term once for the three time
// nodes.  The operation order of every output is that of picard_flux /
// picard_deriv_sub / picard_time_sub.  TRACES: the subcell's traces on the
// sub-faces of the flux kernels (SubTraces2), each evaluated as k_lim_flux
// evaluates it from the nodal values, instead of the nodal values.
// Bound by instruction issue and the shuffles.  The traces go through shared
// memory, one lane to a line and both its ends: by shuffles, with a third of
// the lanes storing single floats under branches, they were 40% of the
// instructions.  463 cells at N = 5: 68.1 -> 44.0 us (128 registers, two
// blocks per SM; 80 registers 46.7, 64 registers 50.1); 512^2 limiter 1.36 ->
// 1.10 ms per step.
template <int N, bool TRACES>
__global__ void __launch_bounds__(256) k_lim_predict_s2(Batch bt) {
  using DM = Dims<2, N>;
  constexpr int NV = 4, NST3 = 27, ND3 = 9, NED = DM::NED, Ns = DM::Ns;
  constexpr int NCROSS = DM::NSD + 4 * DM::NSF;
  const int lane = threadIdx.x & 31;
  const int l = lane < 27 ? lane : 26;                  // idle lanes mirror lane 26
  const int g = l / 9, node = l - 9 * g;                 // subcell slot, spatial node
  const int a = node % 3, b = node / 3;
  float da[3], db[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    da[j] = c_D3f[a * 3 + j];
    db[j] = c_D3f[b * 3 + j];
  }
  const int sx = l - a, sy = l - 3 * b;                 // first lanes of this node's lines
  // the trace weights in FP32, converted once per thread
  float ph0[3], ph1[3];
  {
    const Ops* o = bt.pps[0]->ops;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      ph0[j] = (float)o->phi03[j];
      ph1[j] = (float)o->phi13[j];
    }
  }
  constexpr int QS = NV * NST3 + 29;                    // the three subcells' nodes in different banks
  __shared__ float nodal[TRACES ? 8 : 1][TRACES ? 3 * QS : 1];
  __shared__ __align__(16) float* ends[TRACES ? 8 : 1][12];   // [subcell][axis][high, low end]
  const int wpb = blockDim.x >> 5;
  const long long total = bt.pre[bt.n] * NCROSS;
  const long long groups = (total + 2) / 3;
  for (long long grp = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); grp < groups;
       grp += (long long)gridDim.x * wpb) {
    const long long item = grp * 3 + g;
    const long long tg = item < total ? item / NCROSS : 0;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j0 = it.j;
    const int r = (int)(item - tg * NCROSS);
    const bool needed = item < total && !ghost_elsewhere<2, Ns>(p, it.j, r);
    if (!__any_sync(0xffffffffu, needed)) continue;
    const bool live = needed && lane < 27;
    const int sc = item < total ? cross_subcell<2, Ns>(r) : 0;
    const float cx = p.b.coef_f[3], cy = p.b.coef_f[4];
    const float gm1 = p.b.coef_f[6];
    const float* Wr = reinterpret_cast<const float*>(p.b.sweep[1]);   // [j][v][NED][ND3]
    float u[NV], q[3][NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = item < total ? Wr[((j0 * NV + v) * NED + sc) * ND3 + node] : 1.0f;
    // S = cx D x F_x + cy D y F_y at this lane's node (picard_deriv_sub's order)
    auto space_term = [&](const float* Q, float* Sv) {
      float F[2][4];
      euler_fluxes<2, float>(Q, gm1, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float s = 0.0f;
        {
          const float x0 = __shfl_sync(0xffffffffu, F[0][v], sx);
          const float x1 = __shfl_sync(0xffffffffu, F[0][v], sx + 1);
          const float x2 = __shfl_sync(0xffffffffu, F[0][v], sx + 2);
          float acc = 0.0f;
          acc += da[0] * x0;
          acc += da[1] * x1;
          acc += da[2] * x2;
          s += cx * acc;
        }
        {
          const float x0 = __shfl_sync(0xffffffffu, F[1][v], sy);
          const float x1 = __shfl_sync(0xffffffffu, F[1][v], sy + 3);
          const float x2 = __shfl_sync(0xffffffffu, F[1][v], sy + 6);
          float acc = 0.0f;
          acc += db[0] * x0;
          acc += db[1] * x1;
          acc += db[2] * x2;
          s += cy * acc;
        }
        Sv[v] = s;
      }
    };
#pragma unroll 1
    for (int sweep = 0; sweep < 3; ++sweep) {
      float S[3][NV];
      if (sweep == 0) {
        space_term(u, S[0]);
#pragma unroll
        for (int v = 0; v < NV; ++v) S[1][v] = S[2][v] = S[0][v];
      } else {
#pragma unroll
        for (int m = 0; m < 3; ++m) space_term(q[m], S[m]);
      }
#pragma unroll
      for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          float acc = 0.0f;
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) acc += c_K3f[m * 3 + jj] * S[jj][v];
          q[m][v] = u[v] - acc;
        }
    }
    if constexpr (!TRACES) {
      if (live) {
        float* dst = reinterpret_cast<float*>(p.b.qsub) + ((size_t)j0 * NED + sc) * (size_t)(NV * NST3);
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int m = 0; m < 3; ++m) dst[v * NST3 + m * ND3 + node] = q[m][v];
      }
    } else {
      // the nodal values through shared memory; then a lane takes a whole line
      // (its subcell gs, axis k and row w = point + 9 v, v its variable) and
      // both its ends
      using TR = SubTraces2<N>;
      float* sq = nodal[threadIdx.x >> 5];
      float** dst = ends[threadIdx.x >> 5];
      if (lane < 27) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int m = 0; m < 3; ++m) sq[g * QS + v * NST3 + m * ND3 + node] = q[m][v];
        if (node < 2) {
          const int ck = node == 0 ? sc % (Ns + 2) : sc / (Ns + 2);
          const int co = node == 0 ? sc / (Ns + 2) : sc % (Ns + 2);
          const bool faces = live && co >= 1 && co <= Ns;
          const int ft = (co - 1) * (node == 0 ? Ns + 1 : 1), kmul = node == 0 ? 1 : Ns;
          float* trc = reinterpret_cast<float*>(p.b.qsub) + (size_t)j0 * TR::per_cell;
          dst[2 * (2 * g + node)] = faces && ck <= Ns ? trc + TR::offset(node, ft + ck * kmul, 0) : nullptr;
          dst[2 * (2 * g + node) + 1] = faces && ck >= 1 ? trc + TR::offset(node, ft + (ck - 1) * kmul, 1) : nullptr;
        }
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 7; ++i) {
        const int li = i * 32 + lane;
        if (li < 216) {
          const int gk = li / 36, w = li - 36 * gk, r3 = w / 3, k = gk & 1;
          const float* x = sq + (gk >> 1) * QS + (k == 0 ? 3 * w : 9 * r3 + (w - 3 * r3));
          const int st = k == 0 ? 1 : 3;
          float* hi = dst[2 * gk];
          float* lo = dst[2 * gk + 1];
          const float x0 = x[0], x1 = x[st], x2 = x[2 * st];
          if (hi) hi[w] = ph1[0] * x0 + ph1[1] * x1 + ph1[2] * x2;
          if (lo) lo[w] = ph0[0] * x0 + ph0[1] * x1 + ph0[2] * x2;
        }
      }
      __syncwarp();
    }
  }
}

// Sub-face fluxes normal to axis k from the face traces of k_lim_predict_s2
// (2D, FP32 subcell scheme, Rusanov): three sub-faces per warp, lane
// 9 f + t evaluating the flux at point t of sub-face f from two contiguous
// trace rows, then the GL-weighted sum over each sub-face's 9 points in point
// order, as k_lim_flux accumulates it.  The result is stored in FP64.
template <int N, int k>
__global__ void __launch_bounds__(256) k_lim_flux_t2(Batch bt, int pass) {
  pass = lim_pass(bt, pass);
  using TR = SubTraces2<N>;
  constexpr int NV = 4, Ns = TR::Ns, NFK = TR::NFK, NP = TR::NP;
  constexpr int WPB = 8;
  __shared__ float wts[NP];
  __shared__ float gsum[WPB][3][NV][NP + 1];
  const Ops* o = bt.pps[0]->ops;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x < NP) {
    // the point's weight, formed in k_lim_flux's order (tangential digit, then time)
    const int d = threadIdx.x % 3, mt = threadIdx.x / 3;
    float wt = 1.0f;
    wt *= (float)o->w3[d];
    wt *= (float)o->w3[mt];
    wts[threadIdx.x] = wt;
  }
  __syncthreads();
  const int fl = lane < 27 ? lane / 9 : 2, t = lane < 27 ? lane % 9 : 8;   // idle lanes mirror lane 26
  const long long total = bt.pre[bt.n] * NFK;
  const long long groups = (total + 2) / 3;
  for (long long grp = (long long)blockIdx.x * WPB + w; grp < groups; grp += (long long)gridDim.x * WPB) {
    const long long f = grp * 3 + fl;
    const bool live = f < total;
    const long long tg = live ? f / NFK : 0;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j = it.j;
    const int e = live ? (int)(f - tg * NFK) : 0;
    const int fck = k == 0 ? e % (Ns + 1) : e / Ns;     // the face's index along k
    int wall = 0;
    const bool lo_wall = fck == 0 && p.geo.bc[2 * k] == ADG_BC_REFLECTIVE;
    const bool hi_wall = fck == Ns && p.geo.bc[2 * k + 1] == ADG_BC_REFLECTIVE;
    if (live && (lo_wall || hi_wall)) {
      const long long cell = p.b.list[1 - p.cur][pass * p.chunk + j];
      int ijk[3];
      cell_coords<2>(cell, p.geo, ijk);
      if (lo_wall && ijk[k] == 0) wall = -1;
      if (hi_wall && ijk[k] == p.geo.n[k] - 1) wall = 1;
    }
    float G[NV] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (live) {
      const float* tr = reinterpret_cast<const float*>(p.b.qsub) + (size_t)j * TR::per_cell;
      const float* tl = tr + TR::offset(k, e, 0);
      const float* trr = tr + TR::offset(k, e, 1);
      if (fck == 0 || fck == Ns) {
        // the ghost's side from the neighbour that computed it as its interior
        const int j2 = shared_neighbour<2>(p, j, k, fck == 0 ? -1 : 1);
        constexpr int across = Ns * (k == 0 ? 1 : Ns);
        const float* t2 = reinterpret_cast<const float*>(p.b.qsub) + (long long)j2 * TR::per_cell;
        if (j2 >= 0 && fck == 0) tl = t2 + TR::offset(k, e + across, 0);
        if (j2 >= 0 && fck == Ns) trr = t2 + TR::offset(k, e - across, 1);
      }
      float QL[NV], QR[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        QL[v] = tl[v * NP + t];
        QR[v] = trr[v * NP + t];
      }
      if (wall < 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) QL[v] = QR[v];
        QL[1 + k] = -QR[1 + k];
      } else if (wall > 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) QR[v] = QL[v];
        QR[1 + k] = -QL[1 + k];
      }
      rusanov_f<2>(QL, QR, k, p.b.coef_f[7], G);
    }
    if (lane < 27) {
#pragma unroll
      for (int v = 0; v < NV; ++v) gsum[w][fl][v][t] = G[v];
    }
    __syncwarp();
    if (lane < 3 * NV) {
      const int ff = lane / NV, v = lane - ff * NV;
      const long long fo = grp * 3 + ff;
      if (fo < total) {
        const long long tgo = fo / NFK;
        const LimItem ito = lim_item(bt, tgo);
        const Params& po = *bt.pps[ito.s];
        const int eo = (int)(fo - tgo * NFK);
        float acc = 0.0f;
#pragma unroll
        for (int q = 0; q < NP; ++q) acc += wts[q] * gsum[w][ff][v][q];
        po.b.fsub[k][((size_t)ito.j * NV + v) * NFK + eo] = (double)acc;
      }
    }
    __syncwarp();
  }
}

// Face traces of the 3D subcell predictor, the input of k_lim_flux_t: for
// each troubled cell j, axis k, sub-face e normal to k (the enumeration of
// k_lim_flux: digits over the axes, Ns + 1 values along k and Ns along the
// others) and side (0: the trace of the left subcell at its high end, 1: of
// the right subcell at its low end), 27 points times NV variables, where the
// point t enumerates the node digits of the two tangential axes (lower axis
// fastest) and then the time node.
template <int N>
struct SubTraces {
  static constexpr int Ns = 2 * N + 1, NSF = Ns * Ns, NFK = (Ns + 1) * NSF, NP = 27;
  static constexpr long long per_cell = 3LL * NFK * 2 * 5 * NP;     // floats
  __host__ __device__ static constexpr long long offset(int k, int e, int side) {
    return ((long long)(k * NFK + e) * 2 + side) * 5 * NP;
  }
};

// The 3D subcell predictor in registers: lane l < 27 holds spatial node
// (a, b, c) = (l % 3, (l / 3) % 3, l / 9) of the subcell and its three time
// nodes.  The space derivatives take their three operands per axis from the
// lanes on the node's line by warp shuffles; the time contraction
// (Ktau) runs on the lane's own three time nodes, so it needs no exchange at
// all, and the first sweep, from the time-constant u (x) 1, forms the space
// term once for the three time nodes.  A
// sweep uses no shared memory and no synchronisation.  The operation order of
// every output is that of picard_flux / picard_deriv_sub / picard_time_sub.
// The subcell's traces on the sub-faces the flux kernels use are written in
// place of its nodal values (SubTraces), each evaluated as k_lim_flux
// evaluates it from the nodal values.  They go through shared memory: every
// lane takes lines of three nodes and writes the traces on both ends, 32
// neighbouring values at a time, where shuffles left 18 lanes of 32 with
// something to write and took three per value (the LSU, 63% busy with
// shuffles, and the issue slots bound this kernel).  40^3 N = 3, the larger of
// two passes: 12.4 -> 9.3 ms (1840 -> 1450 instructions per subcell; five
// blocks of four warps per SM at 96 registers, 1% faster than 128 registers).
template <int N>
__global__ void __launch_bounds__(128, 5) k_lim_predict_s3(Batch bt) {
  using DM = Dims<3, N>;
  constexpr int NV = 5, NST3 = 81, ND3 = 27, NED = DM::NED, Ns = DM::Ns;
  constexpr int NCROSS = DM::NSD + 6 * DM::NSF;
  __shared__ float s_q[4][NV * NST3];
  const int lane = threadIdx.x & 31;
  float* sq = s_q[threadIdx.x >> 5];
  const int l = lane < ND3 ? lane : ND3 - 1;            // idle lanes mirror node 26
  const int a = l % 3, b = (l / 3) % 3, c = l / 9;
  float da[3], db[3], dc[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    da[j] = c_D3f[a * 3 + j];
    db[j] = c_D3f[b * 3 + j];
    dc[j] = c_D3f[c * 3 + j];
  }
  const int sx = l - a, sy = l - 3 * b, sz = l - 9 * c;   // first lanes of this node's lines
  // the trace weights in FP32, converted once per thread (FP64 -> FP32
  // conversions run on the narrow FP64 pipe)
  float ph0[3], ph1[3];
  {
    const Ops* o = bt.pps[0]->ops;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      ph0[j] = (float)o->phi03[j];
      ph1[j] = (float)o->phi13[j];
    }
  }
  const int wpb = blockDim.x >> 5;
  const long long total = bt.pre[bt.n] * NCROSS;
  for (long long item = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); item < total;
       item += (long long)gridDim.x * wpb) {
    const long long tg = item / NCROSS;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j0 = it.j;
    const int r = (int)(item - tg * NCROSS);
    if (ghost_elsewhere<3, Ns>(p, it.j, r)) continue;      // (uniform over the warp)
    const int sc = cross_subcell<3, Ns>(r);
    const float cf[3] = {p.b.coef_f[3], p.b.coef_f[4], p.b.coef_f[5]};
    const float gm1 = p.b.coef_f[6];
    const float* Wr = reinterpret_cast<const float*>(p.b.sweep[2]);   // [j][v][NED][ND3]
    float u[NV], q[3][NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      u[v] = Wr[((j0 * NV + v) * NED + sc) * ND3 + l];
#pragma unroll
      for (int m = 0; m < 3; ++m) q[m][v] = u[v];
    }
    // S = sum_k c_k D x_k f_k(Q) at this lane's node, in picard_deriv_sub's order
    auto space_term = [&](const float* Q, float* Sv) {
      float F[3][5];
      euler_fluxes<3, float>(Q, gm1, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const int base = k == 0 ? sx : (k == 1 ? sy : sz);
          const int st = k == 0 ? 1 : (k == 1 ? 3 : 9);
          const float* dr = k == 0 ? da : (k == 1 ? db : dc);
          const float x0 = __shfl_sync(0xffffffffu, F[k][v], base);
          const float x1 = __shfl_sync(0xffffffffu, F[k][v], base + st);
          const float x2 = __shfl_sync(0xffffffffu, F[k][v], base + 2 * st);
          float acc = 0.0f;
          acc += dr[0] * x0;
          acc += dr[1] * x1;
          acc += dr[2] * x2;
          s += cf[k] * acc;
        }
        Sv[v] = s;
      }
    };
#pragma unroll 1
    for (int sweep = 0; sweep < 3; ++sweep) {
      float S[3][NV];
      if (sweep == 0) {
        // the first sweep starts from u (x) 1: its three time nodes carry the
        // same values, hence the same space term
        space_term(u, S[0]);
#pragma unroll
        for (int v = 0; v < NV; ++v) S[1][v] = S[2][v] = S[0][v];
      } else {
#pragma unroll
        for (int m = 0; m < 3; ++m) space_term(q[m], S[m]);
      }
#pragma unroll
      for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          float acc = 0.0f;
#pragma unroll
          for (int j = 0; j < 3; ++j) acc += c_K3f[m * 3 + j] * S[j][v];
          q[m][v] = u[v] - acc;
        }
    }
    // traces, from the nodal values in the warp's shared memory [v][m][node]
    __syncwarp();
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int m = 0; m < 3; ++m)
        if (lane < ND3) sq[(v * 3 + m) * ND3 + l] = q[m][v];
    __syncwarp();
    // the subcell's block coordinates (local + 1, 0 .. Ns + 1 per axis)
    using TR = SubTraces<N>;
    float* trc = reinterpret_cast<float*>(p.b.qsub) + (size_t)j0 * TR::per_cell;
    const int cc[3] = {sc % (Ns + 2), (sc / (Ns + 2)) % (Ns + 2), sc / ((Ns + 2) * (Ns + 2))};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      // a subcell has faces normal to k in the set when its other coordinates are interior
      bool inner = true;
#pragma unroll
      for (int x = 0; x < 3; ++x)
        if (x != k && (cc[x] < 1 || cc[x] > Ns)) inner = false;
      if (!inner) continue;                                 // uniform over the warp
      constexpr int ST[3] = {1, 3, 9};
      const int st = ST[k];
      // the face's tangential index
      int ft = 0, mul = 1;
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const int ext = (x == k) ? Ns + 1 : Ns;
        if (x != k) ft += (cc[x] - 1) * mul;
        mul *= ext;
      }
      const int kmul = k == 0 ? 1 : (k == 1 ? Ns : Ns * Ns);   // place of fc[k] in e
      // left of face cc[k] (high-end trace), right of face cc[k] - 1 (low-end trace)
      const bool wr_hi = cc[k] <= Ns, wr_lo = cc[k] >= 1;
      float* hi = trc + TR::offset(k, ft + cc[k] * kmul, 0);
      float* lo = trc + TR::offset(k, ft + (cc[k] - 1) * kmul, 1);
      // value o = v 27 + t, t = (tangential digits, lower axis first) + 9 m: both
      // ends of one line of three nodes, which starts at node 27 (o / 9) + (the
      // line's place among the 9 tangential nodes)
#pragma unroll
      for (int i = 0; i < (NV * 27 + 31) / 32; ++i) {
        const int o = lane + 32 * i;
        if (o < NV * 27) {
          const int d = o % 9;
          const float* x = sq + (o / 9) * ND3 + (k == 0 ? 3 * d : (k == 1 ? d % 3 + 9 * (d / 3) : d));
          const float x0 = x[0], x1 = x[st], x2 = x[2 * st];
          if (wr_hi) hi[o] = ph1[0] * x0 + ph1[1] * x1 + ph1[2] * x2;
          if (wr_lo) lo[o] = ph0[0] * x0 + ph0[1] * x1 + ph0[2] * x2;
        }
      }
    }
  }
}

// Sub-face fluxes normal to axis k from the face traces of k_lim_predict_s3
// (3D, FP32 subcell scheme, Rusanov): one warp per sub-face, lane t < 27
// evaluates the flux at point t of the face (its two traces are contiguous
// across the lanes).  A warp takes FLUX_TURN sub-faces and then forms their
// GL-weighted sums, one lane per (sub-face, variable), each over its 27 points
// in point order, as k_lim_flux accumulates it (after every sub-face the 27
// terms would run on five lanes: 892 -> 700 us per axis at 40^3, N = 3).  The
// result is stored in FP64.
constexpr int FLUX_TURN = 6;

template <int N, int k>
__global__ void __launch_bounds__(256) k_lim_flux_t(Batch bt, int pass) {
  pass = lim_pass(bt, pass);
  using TR = SubTraces<N>;
  constexpr int NV = 5, Ns = TR::Ns, NFK = TR::NFK, NP = TR::NP;
  constexpr int WPB = 8;
  __shared__ float wts[NP];
  __shared__ float gsum[WPB][FLUX_TURN * NV][NP + 1];
  const Ops* o = bt.pps[0]->ops;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x < NP) {
    // the point's weight, formed in k_lim_flux's order
    int tt = threadIdx.x;
    float wt = 1.0f;
#pragma unroll
    for (int x = 0; x < 3; ++x)
      if (x != k) {
        wt *= (float)o->w3[tt % 3];
        tt /= 3;
      }
    wt *= (float)o->w3[tt];
    wts[threadIdx.x] = wt;
  }
  __syncthreads();
  const int t = lane < NP ? lane : NP - 1;                 // idle lanes mirror point 26
  const long long total = bt.pre[bt.n] * NFK;
  const long long turns = (total + FLUX_TURN - 1) / FLUX_TURN;
  for (long long turn = (long long)blockIdx.x * WPB + w; turn < turns; turn += (long long)gridDim.x * WPB) {
#pragma unroll 1
  for (int rd = 0; rd < FLUX_TURN; ++rd) {
    const long long item = turn * FLUX_TURN + rd;
    if (item >= total) break;
    const long long tg = item / NFK;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j = it.j;
    const int e = (int)(item - tg * NFK);
    // the face's index along k (e = fc0 + ext0 (fc1 + ext1 fc2))
    const int fck = k == 0 ? e % (Ns + 1) : (k == 1 ? (e / Ns) % (Ns + 1) : e / (Ns * Ns));
    // reflecting walls: as in k_lim_flux
    int wall = 0;
    const bool lo_wall = fck == 0 && p.geo.bc[2 * k] == ADG_BC_REFLECTIVE;
    const bool hi_wall = fck == Ns && p.geo.bc[2 * k + 1] == ADG_BC_REFLECTIVE;
    if (lo_wall || hi_wall) {
      const long long cell = p.b.list[1 - p.cur][pass * p.chunk + j];
      int ijk[3];
      cell_coords<3>(cell, p.geo, ijk);
      if (lo_wall && ijk[k] == 0) wall = -1;
      if (hi_wall && ijk[k] == p.geo.n[k] - 1) wall = 1;
    }
    const float* tr = reinterpret_cast<const float*>(p.b.qsub) + (size_t)j * TR::per_cell;
    const float* tl = tr + TR::offset(k, e, 0);
    const float* trr = tr + TR::offset(k, e, 1);
    if (fck == 0 || fck == Ns) {
      // the ghost's side from the neighbour that computed it as its interior
      const int j2 = shared_neighbour<3>(p, j, k, fck == 0 ? -1 : 1);
      constexpr int across = Ns * (k == 0 ? 1 : (k == 1 ? Ns : Ns * Ns));
      const float* t2 = reinterpret_cast<const float*>(p.b.qsub) + (long long)j2 * TR::per_cell;
      if (j2 >= 0 && fck == 0) tl = t2 + TR::offset(k, e + across, 0);
      if (j2 >= 0 && fck == Ns) trr = t2 + TR::offset(k, e - across, 1);
    }
    float QL[NV], QR[NV], G[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      QL[v] = tl[v * NP + t];
      QR[v] = trr[v * NP + t];
    }
    if (wall < 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) QL[v] = QR[v];
      QL[1 + k] = -QR[1 + k];
    } else if (wall > 0) {
#pragma unroll
      for (int v = 0; v < NV; ++v) QR[v] = QL[v];
      QR[1 + k] = -QL[1 + k];
    }
    rusanov_f<3>(QL, QR, k, p.b.coef_f[7], G);
    if (lane < NP) {
#pragma unroll
      for (int v = 0; v < NV; ++v) gsum[w][rd * NV + v][lane] = G[v];
    }
  }
    __syncwarp();
    const long long item = turn * FLUX_TURN + lane / NV;
    if (lane < FLUX_TURN * NV && item < total) {
      const long long tg = item / NFK;
      const LimItem it = lim_item(bt, tg);
      float acc = 0.0f;
#pragma unroll
      for (int q = 0; q < NP; ++q) acc += wts[q] * gsum[w][lane][q];
      bt.pps[it.s]->b.fsub[k][((size_t)it.j * NV + lane % NV) * NFK + (int)(item - tg * NFK)] = (double)acc;
    }
    __syncwarp();
  }
}

// L5: sub-face fluxes normal to axis k: Rusanov at the 3^(d-1) x 3
// tangential x time GL points, averaged with the GL weights.  Faces f = 0..Ns
// along k (between local subcells f-1 and f), tangential subcells 0..Ns-1.
// T: the flux precision (double; float for the mixed-precision FP32 subcell
// scheme, Rusanov only); the result is stored in FP64.
// QT: the element type of the stored subcell predictor (float when it ran
// wholly in FP32).  Launched as (float, float) without the register form of that
// predictor, (float, double) with some of its sweeps in FP64, and (double, float)
// with the Osher-type flux; (double, double) is k_lim_flux_d.
template <int D, int N, int k, typename T, typename QT>
__global__ void __launch_bounds__(256) k_lim_flux(Batch bt, int pass) {
  pass = lim_pass(bt, pass);
  using DM = Dims<D, N>;
  constexpr int NV = DM::NV, NST3 = DM::NST3, ND3 = DM::ND3, NE = DM::NE, NED = DM::NED,
                Ns = DM::Ns;
  constexpr int NFK = (Ns + 1) * DM::NSF;
  const Ops* o = bt.pps[0]->ops;
  constexpr int stk = (k == 0) ? 1 : (k == 1 ? 3 : 9);   // node stride of axis k
  // the GL weights and trace weights in T, converted once per thread
  T w3t[3], p0t[3], p1t[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    w3t[q] = (T)o->w3[q];
    p0t[q] = (T)o->phi03[q];
    p1t[q] = (T)o->phi13[q];
  }
  for (long long eg = blockIdx.x * (long long)blockDim.x + threadIdx.x; eg < bt.pre[bt.n] * NFK;
       eg += (long long)gridDim.x * blockDim.x) {
    const long long tg = eg / NFK;
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const long long j = it.j;
    const long long e = j * NFK + (eg - tg * NFK);
    int r = (int)(e - j * NFK);
    int fc[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int ext = (a == k) ? Ns + 1 : Ns;
      fc[a] = r % ext;
      r /= ext;
    }
    // left / right subcells in the (Ns+2)^d block (array index = local + 1)
    int sl = 0, sr = 0, mul = 1;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int il = (a == k) ? fc[a] : fc[a] + 1;
      const int ir = (a == k) ? fc[a] + 1 : fc[a] + 1;
      sl += il * mul;
      sr += ir * mul;
      mul *= NE;
    }
    size_t jL = j, jR = j;
    if (fc[k] == 0 || fc[k] == Ns) {
      // the ghost's side from the neighbour that computed it as its interior
      const int j2 = shared_neighbour<D>(p, j, k, fc[k] == 0 ? -1 : 1);
      constexpr int across = Ns * ((k == 0) ? 1 : (k == 1 ? NE : NE * NE));
      if (j2 >= 0 && fc[k] == 0) {
        jL = j2;
        sl += across;
      }
      if (j2 >= 0 && fc[k] == Ns) {
        jR = j2;
        sr -= across;
      }
    }
    const QT* qL = reinterpret_cast<const QT*>(p.b.qsub) + (jL * NED + sl) * NV * NST3;
    const QT* qR = reinterpret_cast<const QT*>(p.b.qsub) + (jR * NED + sr) * NV * NST3;
    // a sub-face on a reflecting wall takes its flux between the interior
    // trace and its mirror image (no mass or energy through the wall)
    int wall = 0;                          // -1: low wall (ghost left), +1: high wall (ghost right)
    const bool lo_wall = fc[k] == 0 && p.geo.bc[2 * k] == ADG_BC_REFLECTIVE;
    const bool hi_wall = fc[k] == Ns && p.geo.bc[2 * k + 1] == ADG_BC_REFLECTIVE;
    if (lo_wall || hi_wall) {
      const long long cell = p.b.list[1 - p.cur][pass * p.chunk + j];
      int ijk[3];
      cell_coords<D>(cell, p.geo, ijk);
      if (lo_wall && ijk[k] == 0) wall = -1;
      if (hi_wall && ijk[k] == p.geo.n[k] - 1) wall = 1;
    }
    T acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = T(0);
    const float gf = p.b.coef_f[7];
    // tangential x time nodes: digits over axes != k, then time
    for (int t = 0; t < ND3; ++t) {
      int base = 0, tt = t;
      T wt = T(1);
      int st = 1;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        if (a != k) {
          const int dg = tt % 3;
          tt /= 3;
          base += dg * st;
          wt *= dg == 0 ? w3t[0] : (dg == 1 ? w3t[1] : w3t[2]);   // (registers, not a local array)
        }
        st *= 3;
      }
      const int m = tt;                 // remaining digit: time node
      wt *= m == 0 ? w3t[0] : (m == 1 ? w3t[1] : w3t[2]);
      base += m * ND3;
      T QL[NV], QR[NV], G[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const QT* a = qL + v * NST3 + base;
        const QT* b = qR + v * NST3 + base;
        QL[v] = p1t[0] * (T)a[0] + p1t[1] * (T)a[stk] + p1t[2] * (T)a[2 * stk];
        QR[v] = p0t[0] * (T)b[0] + p0t[1] * (T)b[stk] + p0t[2] * (T)b[2 * stk];
      }
      if (wall < 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) QL[v] = QR[v];
        QL[1 + k] = -QR[1 + k];
      } else if (wall > 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) QR[v] = QL[v];
        QR[1 + k] = -QL[1 + k];
      }
      if constexpr (sizeof(T) == sizeof(double)) face_flux<D>(p.flux, QL, QR, k, p.gamma, G);
      else rusanov_f<D>(QL, QR, k, gf, G);
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += wt * G[v];
    }
    double* dst = p.b.fsub[k] + (size_t)j * NV * NFK + (e - j * NFK);
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[v * NFK] = (double)acc[v];
  }
}

// L5 in FP64: the same sub-face fluxes from FP64 nodal values, one lane per
// point (3D: the 27 points of one sub-face; 2D: the 9 of each of three), so
// that a warp reads a subcell's nodal values together.  A warp takes a few
// rounds of sub-faces and then adds their points, one lane per (sub-face,
// variable) in point order: added after each sub-face, the sums would be 26
// dependent FP64 operations on five lanes.
//
// The FP64 pipe bounds this kernel (88% busy in the thread-per-sub-face form,
// 107 operations per point in 3D): the traces, 30 of them, go to the integer
// pipes (fixed.cuh), and with the Rusanov flux each side's flux and the
// dissipation enter the point's value by FMAs with its weight folded in
// instead of being formed first (27 operations instead of 35), the larger
// speed by an integer comparison.
//
// Measured (GB300): 33 x 29 x 30 N = 3, 5611 troubled cells, 12.4 -> 10.8 ms
// per axis (84% FP64 pipe, 75 operations per point); 2D N = 5, 146 patches,
// 72 -> 42 us per axis.
template <int D>
struct FluxPoints {
  static constexpr int SPR = D == 3 ? 1 : 3;            // sub-faces per round
  static constexpr int ROUNDS = D == 3 ? 6 : 2;         // 30 or 24 sums of a turn, one per lane
  static constexpr int FACES = SPR * ROUNDS;            // sub-faces of one warp's turn
};

template <int D, int N, int k, bool OSHER>
__global__ void __launch_bounds__(128) k_lim_flux_d(Batch bt, int pass) {
  pass = lim_pass(bt, pass);
  using DM = Dims<D, N>;
  using FP = FluxPoints<D>;
  constexpr int NV = DM::NV, NST3 = DM::NST3, ND3 = DM::ND3, NE = DM::NE, NED = DM::NED, Ns = DM::Ns;
  constexpr int NFK = (Ns + 1) * DM::NSF;
  constexpr int stk = (k == 0) ? 1 : (k == 1 ? 3 : 9);    // node stride of axis k
  __shared__ FxOp ph[2][3];         // the traces at the high and low ends
  __shared__ double hw[ND3];        // half the weight of each point
  __shared__ double s_pt[4][FP::FACES * NV][ND3 + 1];
  __shared__ int s_g;
  const Ops* o = bt.pps[0]->ops;
  if (threadIdx.x < 32) {
    const int i = threadIdx.x;
    double s0 = 0.0, s1 = 0.0;
    for (int q = 0; q < 3; ++q) {
      s0 += fabs(o->phi03[q]);
      s1 += fabs(o->phi13[q]);
    }
    const int g = fx_scale(fmax(s0, s1));
    if (i < 6) ph[i / 3][i % 3] = fx_op(i < 3 ? o->phi13[i] : o->phi03[i - 3], g);
    if (i == 0) s_g = g;
    if (i < ND3) hw[i] = 0.5 * o->w3[i % 3] * o->w3[(i / 3) % 3] * (D == 3 ? o->w3[i / 9] : 1.0);
  }
  __syncthreads();
  const int g = s_g;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int pl = lane < 27 ? lane : 26;                   // idle lanes mirror lane 26
  const int fi = pl / ND3, t = pl - fi * ND3;
  // first node of the point's line: its digits over the tangential axes, then
  // the time node
  const int m = D == 3 ? t / 9 : t / 3;
  const int d0 = t % 3, d1 = D == 3 ? (t / 3) % 3 : 0;
  const int base = m * ND3 + (k == 0 ? 3 * d0 + 9 * d1 : (k == 1 ? d0 + 9 * d1 : d0 + 3 * d1));
  const double h = hw[t];
  const long long total = bt.pre[bt.n] * NFK;
  const long long turns = (total + FP::FACES - 1) / FP::FACES;
  for (long long turn = (long long)blockIdx.x * 4 + w; turn < turns; turn += (long long)gridDim.x * 4) {
#pragma unroll 1
    for (int rd = 0; rd < FP::ROUNDS; ++rd) {
      const int ff = rd * FP::SPR + fi;
      const long long f = turn * FP::FACES + ff;
      if (turn * FP::FACES + rd * FP::SPR >= total) break;     // (uniform over the warp)
      const long long fe = f < total ? f : total - 1;
      const long long tg = fe / NFK;
      const LimItem it = lim_item(bt, tg);
      const Params& p = *bt.pps[it.s];
      const long long j = it.j;
      int fck = 0, sl = 0, sr = 0;
      {
        int r = (int)(fe - tg * NFK), mul = 1;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const int ext = (a == k) ? Ns + 1 : Ns;
          const int c = r % ext;
          r /= ext;
          if (a == k) fck = c;
          // left / right subcells in the (Ns+2)^d block (array index = local + 1)
          sl += ((a == k) ? c : c + 1) * mul;
          sr += (c + 1) * mul;
          mul *= NE;
        }
      }
      int wall = 0;                          // -1: low wall (ghost left), +1: high wall (ghost right)
      long long jL = j, jR = j;
      if (fck == 0 || fck == Ns) {
        // the ghost's side from the neighbour that computed it as its interior
        const int j2 = shared_neighbour<D>(p, j, k, fck == 0 ? -1 : 1);
        constexpr int across = Ns * ((k == 0) ? 1 : (k == 1 ? NE : NE * NE));
        if (j2 >= 0 && fck == 0) {
          jL = j2;
          sl += across;
        } else if (j2 >= 0) {
          jR = j2;
          sr -= across;
        }
        // reflecting walls: as in k_lim_flux (the list of troubled cells is read
        // only where the face can be a wall: the no-allocation entry point runs
        // this kernel with periodic kinds, no list and no table of neighbours)
        const int side = fck == 0 ? 0 : 1;
        if (p.geo.bc[2 * k + side] == ADG_BC_REFLECTIVE) {
          const long long cell = p.b.list[1 - p.cur][pass * p.chunk + j];
          int ijk[3];
          cell_coords<D>(cell, p.geo, ijk);
          if (side == 0 && ijk[k] == 0) wall = -1;
          if (side == 1 && ijk[k] == p.geo.n[k] - 1) wall = 1;
        }
      }
      const double* qL = p.b.qsub + (jL * NED + sl) * (size_t)(NV * NST3) + base;
      const double* qR = p.b.qsub + (jR * NED + sr) * (size_t)(NV * NST3) + base;
      double QL[NV], QR[NV], G[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const double* a = qL + v * NST3;
        const double* b = qR + v * NST3;
        const double xa[3] = {a[0], a[stk], a[2 * stk]}, xb[3] = {b[0], b[stk], b[2 * stk]};
        fx_apply<3, 1, true>(xa, ph[0], g, FxRows{o->phi13, 1.0}, [&](int, double y) { QL[v] = y; });
        fx_apply<3, 1, true>(xb, ph[1], g, FxRows{o->phi03, 1.0}, [&](int, double y) { QR[v] = y; });
      }
      if (wall < 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) QL[v] = QR[v];
        QL[1 + k] = -QR[1 + k];
      } else if (wall > 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v) QR[v] = QL[v];
        QR[1 + k] = -QL[1 + k];
      }
      if constexpr (OSHER) {
        face_flux<D>(ADG_FLUX_OSHER, QL, QR, k, p.gamma, G);
#pragma unroll
        for (int v = 0; v < NV; ++v) G[v] *= 2.0 * h;
      } else {
        // h (F_k(QL) + F_k(QR) - s (QR - QL)), s the larger |v_k| + c (as bits:
        // not negative, and a NaN of either sign is above every number)
        const double gm1 = p.gamma - 1.0;
        unsigned long long s = 0;
#pragma unroll
        for (int v = 0; v < NV; ++v) G[v] = 0.0;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const double* Q = side ? QR : QL;
          const double r = 1.0 / Q[0];
          double kin = 0.0;
#pragma unroll
          for (int a = 0; a < D; ++a) kin += Q[1 + a] * Q[1 + a];
          const double pr = gm1 * (Q[D + 1] - 0.5 * kin * r);
          const double vk = Q[1 + k] * r, hv = h * vk;
          G[0] += h * Q[1 + k];
#pragma unroll
          for (int a = 0; a < D; ++a) G[1 + a] += hv * Q[1 + a];
          G[1 + k] += h * pr;
          G[D + 1] += hv * (Q[D + 1] + pr);
          const double sp = fabs(vk) + sqrt(p.gamma * pr * r);
          const unsigned long long b = (unsigned long long)__double_as_longlong(sp);
          s = b > s ? b : s;
        }
        const double hs = h * __longlong_as_double((long long)s);
#pragma unroll
        for (int v = 0; v < NV; ++v) G[v] -= hs * (QR[v] - QL[v]);
      }
      if (lane < 27) {
#pragma unroll
        for (int v = 0; v < NV; ++v) s_pt[w][ff * NV + v][t] = G[v];
      }
    }
    __syncwarp();
    for (int q = lane; q < FP::FACES * NV; q += 32) {
      const int ff = q / NV, v = q - ff * NV;
      const long long f = turn * FP::FACES + ff;
      if (f < total) {
        const long long tg = f / NFK;
        const LimItem it = lim_item(bt, tg);
        double acc = s_pt[w][q][0];
#pragma unroll
        for (int i = 1; i < ND3; ++i) acc += s_pt[w][q][i];
        bt.pps[it.s]->b.fsub[k][((size_t)it.j * NV + v) * NFK + (int)(f - tg * NFK)] = acc;
      }
    }
    __syncwarp();
  }
}

// L6: finite volume update, storage of v^{n+1}, reconstruction R, per-cell
// min/max and wave speed, sub-face fluxes of the cell faces, and marking of
// unlimited face neighbours for the flux correction.  One block per cell.
template <int D, int N>
__global__ void __launch_bounds__(128) k_lim_update(Batch bt, int pass) {
  pass = lim_pass(bt, pass);
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, Ns = DM::Ns, NSD = DM::NSD, L = DM::L,
                LD = DM::LD, NSF = DM::NSF;
  constexpr int NFK = (Ns + 1) * NSF;
  extern __shared__ double sm[];
  double* A = sm;                 // NV * NSD
  double* B = A + NV * NSD;       // NV * NSD
  double* R1 = B + NV * NSD;        // n * Ns
  double* mm = R1 + n * Ns;         // 2 NV
  double* red = mm + 2 * NV;      // 128
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < n * Ns; i += nth) R1[i] = bt.pps[0]->ops->R1[i];
  for (long long tg = blockIdx.x; tg < bt.pre[bt.n]; tg += gridDim.x) {
    const LimItem it = lim_item(bt, tg);
    const Params& p = *bt.pps[it.s];
    const int j = it.j;
    const int nxt = 1 - p.cur;
    double c[3];
    {
#pragma unroll
      for (int k = 0; k < D; ++k) c[k] = p.b.coef[3 + k];
    }
    const int t = pass * p.chunk + j;
    const long long cell = p.b.list[nxt][t];
    const double* pt = p.b.patch + (size_t)j * NV * LD;
    double* st = p.b.store[nxt] + (size_t)t * NV * NSD;
    __syncthreads();
    for (int e = tid; e < NV * NSD; e += nth) {
      const int v = e / NSD;
      int s = e - v * NSD;
      int sc[3] = {0, 0, 0};
#pragma unroll
      for (int a = 0; a < D; ++a) {
        sc[a] = s % Ns;
        s /= Ns;
      }
      int poff = 0, pm = 1;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        poff += (sc[a] + 3) * pm;
        pm *= L;
      }
      double val = pt[v * LD + poff];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        int flo = 0, mul = 1;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          flo += sc[a] * mul;
          mul *= (a == k) ? Ns + 1 : Ns;
        }
        const int kst = (k == 0) ? 1 : (k == 1 ? Ns : Ns * Ns);   // stride of axis k
        const double* F = p.b.fsub[k] + ((size_t)j * NV + v) * NFK;
        val -= c[k] * (F[flo + kst] - F[flo]);
      }
      A[e] = val;
      st[e] = val;
    }
    __syncthreads();
    double lam = 0.0;
    const bool bad = check_subcells<D>(A, NSD, nullptr, p.gamma, mm, p.lam_mode ? &lam : nullptr, red,
                                       p.prec == ADG_PREC_MIXED_FP32, p.gam2f);
    if (tid == 0) {
      if (p.lam_mode) p.b.lam[cell] = lam;
      if (bad && p.cascade) {
        // first-order layer: recomputed by k_lim_fallback after all passes
        const int i = atomicAdd(&p.b.counters[CNT_FB], 1);
        p.b.fblist[i] = t;
        p.b.fbflag[t] = p.stamp;
        atomicAdd(&p.b.counters[CNT_FB_TOTAL], 1);
      } else if (bad) {
        atomicAdd(&p.b.counters[CNT_INADM], 1);
      }
    }
    if (tid < 2 * NV) p.b.cmm[nxt][cell * 2 * NV + tid] = mm[tid];
    // sub-face fluxes on the faces of the cell: edge[t][k][side][v][NSF]
    for (int e = tid; e < D * 2 * NV * NSF; e += nth) {
      const int k = e / (2 * NV * NSF);
      int r = e - k * (2 * NV * NSF);
      const int side = r / (NV * NSF);
      r -= side * NV * NSF;
      const int v = r / NSF, ts = r - v * NSF;
      int tc[2] = {ts % Ns, ts / Ns};
      int fidx = 0, mul = 1, q = 0;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const int cc = (a == k) ? (side ? Ns : 0) : tc[q++];
        fidx += cc * mul;
        mul *= (a == k) ? Ns + 1 : Ns;
      }
      p.b.edge[(size_t)t * D * 2 * NV * NSF + e] = p.b.fsub[k][((size_t)j * NV + v) * NFK + fidx];
    }
    // reconstruction R of the new subcell data
    __syncthreads();
    double* u = reconstruct<D, N>(A, B, R1, tid, nth);
    double* Uo = p.b.U[nxt] + cell * (NV * ND);
    for (int e = tid; e < NV * ND; e += nth) Uo[e] = u[e];
    if (tid == 0 && p.b.vok) p.b.vok[cell] = 0;     // P(R(v)) is not v: recompute next step
    // unlimited face neighbours get the flux correction
    if (tid < 2 * D) {
      const int k = tid >> 1, side = (tid & 1) ? 1 : -1;
      int ijk[3], nb[3];
      cell_coords<D>(cell, p.geo, ijk);
      if (face_neighbour<D>(p.geo, ijk, k, side, nb)) {
        const long long nc = cell_index<D>(nb, p.geo);
        if (!p.b.beta[nxt][nc]) {
          const int old = atomicExch(&p.b.fixstamp[nc], p.stamp);
          if (old != p.stamp) {
            const int idx = atomicAdd(&p.b.counters[CNT_FIX], 1);
            p.b.fixlist[idx] = (int)nc;
          }
        }
      }
    }
  }
}

// L7: flux correction of unlimited cells with troubled face neighbours
// (Sec. 4.4): on each such face the DG flux Gbar is replaced by the sub-face
// fluxes integrated against the test functions,
//   Fsub_b = (1/W_b) sum_e Fbar_e prod P1[e][b] / Ns^(d-1).
template <int D, int N>
__global__ void __launch_bounds__(128) k_lim_fix(Batch bt) {
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, NF = DM::NF, Ns = DM::Ns, NSD = DM::NSD,
                NSF = DM::NSF;
  extern __shared__ double sm[];
  double* U = sm;                      // NV * ND
  double* A = U + NV * ND;             // NV * max(NSD, ...)
  double* B = A + NV * NSD;
  double* Mt = B + NV * NSD;           // n * Ns
  FxOp* P1x = reinterpret_cast<FxOp*>(Mt + n * Ns);         // Ns * n
  double* mm = reinterpret_cast<double*>(P1x + Ns * n);
  double* red = mm + 2 * NV;
  const int tid = threadIdx.x, nth = blockDim.x;
  const Ops* o = bt.pps[0]->ops;
  for (int i = tid; i < n * Ns; i += nth) {
    Mt[i] = o->Mt[i];
    P1x[i] = o->P1x[i];
  }
  const FxMat P1m = {P1x, o->gP1, o->P1};
  for (long long fg = blockIdx.x; fg < bt.pre[bt.n]; fg += gridDim.x) {
    const int sidx = batch_state(bt, fg);
    const Params& p = *bt.pps[sidx];
    const long long f = fg - bt.pre[sidx];
    const int nxt = 1 - p.cur;
    const long long cell = p.b.fixlist[f];
    int ijk[3];
    cell_coords<D>(cell, p.geo, ijk);
    double* Uo = p.b.U[nxt] + cell * (NV * ND);
    __syncthreads();
    for (int e = tid; e < NV * ND; e += nth) U[e] = Uo[e];
    for (int k = 0; k < D; ++k) {
      const double ck = p.b.coef[k];
      for (int side = -1; side <= 1; side += 2) {
        int nb[3];
        if (!face_neighbour<D>(p.geo, ijk, k, side, nb)) continue;
        const long long nc = cell_index<D>(nb, p.geo);
        if (!p.b.beta[nxt][nc]) continue;
        const int slot = p.b.slot[nxt][nc];
        if (slot < 0) continue;
        // the neighbour's face that touches this cell
        const int eside = (side > 0) ? 0 : 1;
        const double* Fs = p.b.edge + (size_t)slot * D * 2 * NV * NSF + ((size_t)k * 2 + eside) * NV * NSF;
        __syncthreads();
        // project the Ns^(d-1) sub-face fluxes on the n^(d-1) tangential nodes
        for (int e = tid; e < NV * NSF; e += nth) A[e] = Fs[e];
        __syncthreads();
        double* Fp = A;
        if (D == 2) {
          int ext[3] = {Ns, 1, 1};
          apply_axis<1>(A, B, Mt, n, Ns, 0, ext, NV, tid, nth);
          Fp = B;
        } else {
          int ext[3] = {Ns, Ns, 1};
          apply_axis<2>(A, B, Mt, n, Ns, 0, ext, NV, tid, nth);
          __syncthreads();
          ext[0] = n;
          apply_axis<2>(B, A, Mt, n, Ns, 1, ext, NV, tid, nth);
          Fp = A;
        }
        __syncthreads();
        const long long face = face_index<D>(p.geo, ijk, k, side > 0 ? ijk[k] + 1 : ijk[k]);
        const double* Gd = p.b.G[k] + face * NV * NF;
        for (int e = tid; e < NV * ND; e += nth) {
          const int v = e / ND, i = e - v * ND;
          const int st = (k == 0) ? 1 : (k == 1 ? n : n * n);
          const int ak = (i / st) % n;
          const int ts = tangential<D, n>(i, k);
          const double diff = Fp[v * NF + ts] - Gd[v * NF + ts];
          if (side > 0) U[e] -= ck * p.ops->phi1w[ak] * diff;
          else U[e] += ck * p.ops->phi0w[ak] * diff;
        }
      }
    }
    __syncthreads();
    for (int e = tid; e < NV * ND; e += nth) {
      Uo[e] = U[e];
      A[e] = U[e];
    }
    __syncthreads();
    double* vs = apply_fx<D, NV, n, Ns>(A, B, P1m, tid, nth);
    if (p.b.vstar) {
      // the corrected DOFs' projection, kept for the next step's detector
      double* vk = p.b.vstar + cell * (size_t)(NV * NSD);
      for (int e = tid; e < NV * NSD; e += nth) vk[e] = vs[e];
    }
    double lam = 0.0;
    check_subcells<D>(vs, NSD, nullptr, p.gamma, mm, p.lam_mode ? &lam : nullptr, red,
                      p.prec == ADG_PREC_MIXED_FP32, p.gam2f);
    if (tid == 0 && p.lam_mode) p.b.lam[cell] = lam;
    if (tid < 2 * NV) p.b.cmm[nxt][cell * 2 * NV + tid] = mm[tid];
  }
}

// Cascade layer (Sec. 6, Fig. algo2), part 1: each troubled cell whose WENO3
// result failed PAD is recomputed from v^n by one first-order Rusanov step on
// its subgrid: sub-face fluxes between the piecewise-constant subcell data,
// ghost data from Eq. (ader.icbc) as for the WENO3 patch (wrapped or clamped
// global subcell index).  Writes v^{n+1}, min / max, wave speed, u = R(v) and
// the cell-face fluxes (the flux correction of unlimited neighbours uses
// them), and lists the WENO3 face neighbours, which must take the
// first-order flux on the shared face (part 2).  One block per cell.
template <int D, int N>
__global__ void __launch_bounds__(128) k_lim_fallback(Batch bt) {
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, Ns = DM::Ns, NSD = DM::NSD, NSF = DM::NSF;
  constexpr int NE = Ns + 2;                          // local subcells -1..Ns per axis
  constexpr int NB = (D == 3) ? NE * NE * NE : NE * NE;
  constexpr int NFK = (Ns + 1) * NSF;
  extern __shared__ double sm[];
  double* blk = sm;                 // NV * NB   v^n with one ghost layer
  double* A = blk + NV * NB;        // NV * NSD
  double* B = A + NV * NSD;         // NV * NSD
  double* F = B + NV * NSD;         // NV * NFK  sub-face fluxes of one axis
  double* R1 = F + NV * NFK;        // n * Ns
  double* P1 = R1 + n * Ns;         // Ns * n
  double* mm = P1 + Ns * n;         // 2 NV
  double* red = mm + 2 * NV;        // 128
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < n * Ns; i += nth) {
    R1[i] = bt.pps[0]->ops->R1[i];
    P1[i] = bt.pps[0]->ops->P1[i];
  }
  for (long long fg = blockIdx.x; fg < bt.pre[bt.n]; fg += gridDim.x) {
    const int sidx = batch_state(bt, fg);
    const Params& p = *bt.pps[sidx];
    const long long f = fg - bt.pre[sidx];
    const int nxt = 1 - p.cur;
    const Geo& g = p.geo;
    const int t = p.b.fblist[f];
    const long long cell = p.b.list[nxt][t];
    int ijk[3];
    cell_coords<D>(cell, g, ijk);
    __syncthreads();
    for (int e = tid; e < NB; e += nth) {
      int r = e;
      int loc[3] = {0, 0, 0};
#pragma unroll
      for (int k = 0; k < D; ++k) {
        loc[k] = r % NE - 1;
        r /= NE;
      }
      double val[NV];
      patch_value<D, N>(p, ijk, loc, P1, val);
#pragma unroll
      for (int v = 0; v < NV; ++v) blk[v * NB + e] = val[v];
    }
    __syncthreads();
    for (int e = tid; e < NV * NSD; e += nth) {
      const int v = e / NSD;
      int s = e - v * NSD, bi = 0, mul = 1;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        bi += (s % Ns + 1) * mul;
        s /= Ns;
        mul *= NE;
      }
      A[e] = blk[v * NB + bi];
    }
    for (int k = 0; k < D; ++k) {
      const double ck = p.b.coef[3 + k];
      __syncthreads();
      // faces c_k = 0..Ns between local subcells c_k - 1 and c_k
      for (int e = tid; e < NFK; e += nth) {
        int r = e, bl = 0, mul = 1, stk = 1;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const int ext = (a == k) ? Ns + 1 : Ns;
          const int c = r % ext;
          r /= ext;
          bl += (a == k ? c : c + 1) * mul;
          if (a == k) stk = mul;
          mul *= NE;
        }
        double QL[NV], QR[NV], G[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          QL[v] = blk[v * NB + bl];
          QR[v] = blk[v * NB + bl + stk];
        }
        rusanov<D>(QL, QR, k, p.gamma, G);
#pragma unroll
        for (int v = 0; v < NV; ++v) F[v * NFK + e] = G[v];
      }
      __syncthreads();
      const int kst = (k == 0) ? 1 : (k == 1 ? Ns : Ns * Ns);   // stride of axis k
      for (int e = tid; e < NV * NSD; e += nth) {
        const int v = e / NSD;
        int s = e - v * NSD, flo = 0, mul = 1;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          flo += (s % Ns) * mul;
          s /= Ns;
          mul *= (a == k) ? Ns + 1 : Ns;
        }
        A[e] -= ck * (F[v * NFK + flo + kst] - F[v * NFK + flo]);
      }
      // cell-face fluxes: edge[t][k][side][v][NSF]
      for (int e = tid; e < 2 * NV * NSF; e += nth) {
        const int side = e / (NV * NSF);
        const int r = e - side * NV * NSF;
        const int v = r / NSF, ts = r - v * NSF;
        const int tc[2] = {ts % Ns, ts / Ns};
        int fidx = 0, mul = 1, q = 0;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const int cc = (a == k) ? (side ? Ns : 0) : tc[q++];
          fidx += cc * mul;
          mul *= (a == k) ? Ns + 1 : Ns;
        }
        p.b.edge[((size_t)t * D * 2 + (size_t)k * 2 + side) * NV * NSF + r] = F[v * NFK + fidx];
      }
    }
    __syncthreads();
    double* st = p.b.store[nxt] + (size_t)t * NV * NSD;
    for (int e = tid; e < NV * NSD; e += nth) st[e] = A[e];
    double lam = 0.0;
    const bool bad = check_subcells<D>(A, NSD, nullptr, p.gamma, mm, p.lam_mode ? &lam : nullptr, red,
                                       p.prec == ADG_PREC_MIXED_FP32, p.gam2f);
    if (tid == 0) {
      if (p.lam_mode) p.b.lam[cell] = lam;
      if (bad) atomicAdd(&p.b.counters[CNT_INADM], 1);
    }
    if (tid < 2 * NV) p.b.cmm[nxt][cell * 2 * NV + tid] = mm[tid];
    __syncthreads();
    double* u = reconstruct<D, N>(A, B, R1, tid, nth);
    double* Uo = p.b.U[nxt] + cell * (NV * ND);
    for (int e = tid; e < NV * ND; e += nth) Uo[e] = u[e];
    if (tid == 0 && p.b.vok) p.b.vok[cell] = 0;     // P(R(v)) is not v: recompute next step
    if (tid < 2 * D) {
      const int k = tid >> 1, side = (tid & 1) ? 1 : -1;
      int nb[3];
      if (face_neighbour<D>(g, ijk, k, side, nb)) {
        const long long nc = cell_index<D>(nb, g);
        if (p.b.beta[nxt][nc]) {
          const int sl = p.b.slot[nxt][nc];
          // fixstamp marks unlimited cells for k_lim_fix; troubled cells are
          // never in that list, so it marks the WENO3 neighbours here
          if (sl >= 0 && p.b.fbflag[sl] != p.stamp) {
            const int old = atomicExch(&p.b.fixstamp[nc], p.stamp);
            if (old != p.stamp) {
              const int idx = atomicAdd(&p.b.counters[CNT_REFIX], 1);
              p.b.refixlist[idx] = (int)nc;
            }
          }
        }
      }
    }
  }
}

// Cascade layer, part 2: a WENO3 cell with fallback face neighbours takes
// their first-order flux on each shared face.  Its subcells next to such a
// face change by -+(dt/h_k)(F_first - F_weno), applied in the order axis 0
// low, axis 0 high, axis 1 low, ...; then min / max, wave speed and u = R(v)
// again.  One block per cell.
template <int D, int N>
__global__ void __launch_bounds__(128) k_lim_refix(Batch bt) {
  using DM = Dims<D, N>;
  constexpr int n = DM::n, NV = DM::NV, ND = DM::ND, Ns = DM::Ns, NSD = DM::NSD, NSF = DM::NSF;
  constexpr size_t EDGE = (size_t)D * 2 * NV * NSF;
  extern __shared__ double sm[];
  double* A = sm;                   // NV * NSD
  double* B = A + NV * NSD;         // NV * NSD
  double* R1 = B + NV * NSD;        // n * Ns
  double* mm = R1 + n * Ns;         // 2 NV
  double* red = mm + 2 * NV;        // 128
  __shared__ int fbslot[6];         // slot of the fallback neighbour per face, -1: none
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < n * Ns; i += nth) R1[i] = bt.pps[0]->ops->R1[i];
  for (long long fg = blockIdx.x; fg < bt.pre[bt.n]; fg += gridDim.x) {
    const int sidx = batch_state(bt, fg);
    const Params& p = *bt.pps[sidx];
    const long long f = fg - bt.pre[sidx];
    const int nxt = 1 - p.cur;
    const Geo& g = p.geo;
    const long long cell = p.b.refixlist[f];
    const int t = p.b.slot[nxt][cell];
    int ijk[3];
    cell_coords<D>(cell, g, ijk);
    __syncthreads();
    if (tid < 2 * D) {
      const int k = tid >> 1, side = (tid & 1) ? 1 : -1;
      int nb[3], fs = -1;
      if (face_neighbour<D>(g, ijk, k, side, nb)) {
        const long long nc = cell_index<D>(nb, g);
        if (p.b.beta[nxt][nc]) {
          const int sl = p.b.slot[nxt][nc];
          if (sl >= 0 && p.b.fbflag[sl] == p.stamp) fs = sl;
        }
      }
      fbslot[tid] = fs;
    }
    double* st = p.b.store[nxt] + (size_t)t * NV * NSD;
    __syncthreads();
    const double* Et = p.b.edge + (size_t)t * EDGE;
    for (int e = tid; e < NV * NSD; e += nth) {
      const int v = e / NSD;
      int s = e - v * NSD;
      int sc[3] = {0, 0, 0};
#pragma unroll
      for (int a = 0; a < D; ++a) {
        sc[a] = s % Ns;
        s /= Ns;
      }
      double val = st[e];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const double ck = p.b.coef[3 + k];
        int ts = 0, mul = 1;
#pragma unroll
        for (int a = 0; a < D; ++a)
          if (a != k) {
            ts += sc[a] * mul;
            mul *= Ns;
          }
#pragma unroll
        for (int own = 0; own < 2; ++own) {
          const int fs = fbslot[2 * k + own];
          if (fs < 0 || sc[k] != (own ? Ns - 1 : 0)) continue;
          const double Fnew = p.b.edge[(size_t)fs * EDGE + ((size_t)k * 2 + (1 - own)) * NV * NSF + v * NSF + ts];
          const double Fold = Et[((size_t)k * 2 + own) * NV * NSF + v * NSF + ts];
          const double diff = ck * (Fnew - Fold);
          if (own) val -= diff;
          else val += diff;
        }
      }
      A[e] = val;
      st[e] = val;
    }
    __syncthreads();
    double lam = 0.0;
    const bool bad = check_subcells<D>(A, NSD, nullptr, p.gamma, mm, p.lam_mode ? &lam : nullptr, red,
                                       p.prec == ADG_PREC_MIXED_FP32, p.gam2f);
    if (tid == 0) {
      if (p.lam_mode) p.b.lam[cell] = lam;
      if (bad) atomicAdd(&p.b.counters[CNT_INADM], 1);
    }
    if (tid < 2 * NV) p.b.cmm[nxt][cell * 2 * NV + tid] = mm[tid];
    __syncthreads();
    double* u = reconstruct<D, N>(A, B, R1, tid, nth);
    double* Uo = p.b.U[nxt] + cell * (NV * ND);
    for (int e = tid; e < NV * ND; e += nth) Uo[e] = u[e];
    if (tid == 0 && p.b.vok) p.b.vok[cell] = 0;     // P(R(v)) is not v: recompute next step
  }
}

}  // namespace adg
