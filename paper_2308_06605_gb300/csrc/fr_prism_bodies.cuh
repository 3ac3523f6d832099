// Device bodies of the FR residual on the prisms of mixed hexahedral/prismatic meshes (arXiv 2308.06605,
// section "FR Algorithm", Eq. 1-3; the paper's solver handles prisms alongside hexahedra).
//
// A prism of order p carries Nt = N(N+1)/2 triangle nodes times N = p + 1 Gauss-Legendre points
// along its axis, point index m = q + Nt k.  With reference normals N_f (faces 0/1: zeta = -1/+1,
// triangles whose flux points are the triangle nodes; faces 2/3/4: s = -1, r + s = 0, r = -1,
// quadrilaterals with N x N Gauss points in (edge parameter, zeta)), the DG-equivalent correction
// (c = 0) is the lifting C_f = M^-1 E_f with the exact mass matrix, which factorises:
//   triangles:       C_f = h_-/+ (x) I_Nt        (h = the 1D correction divergence of the line)
//   quadrilaterals:  C_f = I_N (x) LQ_e,  LQ_e = M_T^-1 E_e^T diag(w)   (e = f - 2)
// and the traces are L_f = l(-1/+1) (x) I_Nt, resp. I_N (x) E_e (triangle interpolation to the
// edge's Gauss points).  The residual is R = -|J|^-1 [sum_d D~_d F^_d + sum_f C_f F^I_f] with the
// own-flux part of the correction folded into D~ (Drt, Dst, D1t of the operator table); BR2 uses
// grad Q = J^-T (D Q + sum_f N_f C_f (Q^I - Q_f)) and face gradients L_f (grad_unc + eta r_f),
// r_f = J^-T N_f C_f (Q^I - Q_f).  Interfaces, boundary states, common fluxes and the RK update
// are shared with the hexahedra (slot stride N^2; a triangular interface uses its first Nt slots).
//
// Templated on the order and on the element arithmetic T (double, or df32 on the mixed path),
// like the hexahedral kernels.
//
// The bodies are shared by the per-mesh prism kernels (fr_prism.cu) and the batched persistent
// stage kernel (fr_batch_kernel.cu); everything here has internal linkage.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "df32.cuh"
#include "fr_device.hpp"
#include "fr_point.cuh"

namespace frx {
namespace {


template <int N>
__host__ __device__ constexpr int prism_points() { return N * (N + 1) / 2 * N; }
template <int N>
__host__ __device__ constexpr int prism_threads() { return ((prism_points<N>() + 31) / 32) * 32; }
// Resident blocks the register budget must allow, per order and arithmetic (checked with ptxas):
// up to 64 threads, for double-float at 96 threads and at 128 threads (p = 5) about 170
// registers per thread without spills; FP64 at 96 threads fits 4 blocks unbounded; the larger
// blocks are bound by shared memory.
template <int N, typename T>
__host__ __device__ constexpr int prism_min_blocks() {
  return prism_threads<N>() <= 32 ? 12 : (prism_threads<N>() <= 64 ? 6 :
         (prism_threads<N>() <= 96 ? (std::is_same<T, df32>::value ? 4 : 2) : (prism_threads<N>() <= 128 ? 3 : 1)));
}
// Shared-memory values (of T) of the volume kernel: Q 5, grad 15, flux 15, BR2 weights 15, quad
// lifts 15 (per point) and the jumps of 5 faces x 5 variables x N^2 slots.
template <int N>
__host__ __device__ constexpr int prism_smem_values() { return 65 * prism_points<N>() + 25 * N * N; }


// Interface slot of local flux point r of prism face f for a packed face word.
template <int N>
__device__ __forceinline__ int prism_slot(int f, int r, int code, const int32_t *__restrict__ tri_slot) {
  constexpr int Nt = N * (N + 1) / 2;
  return f < 2 ? tri_slot[code * Nt + r] : orient_slot(code, r % N, r / N, N);
}

// ------------------------------------------------------------------------------------------
// 1. Solution traces.  Thread per (prism, face, flux point); triangular faces use r < Nt.
// ------------------------------------------------------------------------------------------
template <int N, typename T>
__device__ __forceinline__ void prism_interp_body(int64_t t, const T *__restrict__ Q, const int32_t *__restrict__ ef_p,
                                                  const T *__restrict__ tab, const int32_t *__restrict__ tri_slot,
                                                  T *__restrict__ Qtr, int64_t Ep) {
  constexpr int Nt = N * (N + 1) / 2, Np = Nt * N, Nf = N * N;
  constexpr PrismTab L = prism_tab(N);
  if (t >= Ep * 5 * Nf) return;
  const int r = (int)(t % Nf);
  const int64_t eff = t / Nf;
  const int f = (int)(eff % 5);
  const int64_t e = eff / 5;
  if (f < 2 && r >= Nt) return;
  const T *q = Q + e * Np * 5;
  Dot<T> acc[5];
  if (f < 2) {
    const T *l = tab + (f ? L.lp : L.lm);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const T lk = l[k];
      const T *qk = q + (r + Nt * k) * 5;
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v].add(lk, qk[v]);
    }
  } else {
    const int a = r % N, b = r / N;
    const T *Ea = tab + L.E + (f - 2) * N * Nt + a;
#pragma unroll 4
    for (int j = 0; j < Nt; ++j) {
      const T ej = Ea[j * N];
      const T *qj = q + (j + Nt * b) * 5;
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v].add(ej, qj[v]);
    }
  }
  const int packed = ef_p[eff];
  const int64_t I = packed >> 4;
  const int side = (packed >> 3) & 1;
  T *dst = Qtr + (I * 2 + side) * 5 * Nf + prism_slot<N>(f, r, packed & 7, tri_slot);
#pragma unroll
  for (int v = 0; v < 5; ++v) dst[v * Nf] = acc[v].get();
}

// ------------------------------------------------------------------------------------------
// 2. Volume kernel.  One block per prism, one thread per solution point.
// Bound by FP32 issue (double-float) or the FP64 pipe.  Operator entries are read with consecutive
// threads on consecutive addresses and once for the five variables (row-major tables cost 15 L1
// wavefronts per load at p = 4, and were read per variable).  On the cascade passage (72 case: 25 200
// hexahedra, 10 080 prisms, p = 4) the two volume kernels together 1.505 -> 1.279 ms in double-float, 5.06 ->
// 4.60 ms in FP64.
// ------------------------------------------------------------------------------------------
// One prism e handled by `nth` threads of the block (thread index tid in [0, nth)); every thread
// of the block calls this together (it contains block barriers); inactive sub-blocks
// (active = false) only take part in the barriers.
template <int N, typename T>
__device__ __forceinline__ void prism_volume_body(int64_t e, int tid, int nth, bool active, double *sm_raw,
                                                  const T *__restrict__ Q, const T *__restrict__ metrics,
                                                  const int32_t *__restrict__ ef_p, const T *__restrict__ Qtr,
                                                  const T *__restrict__ tab, const int32_t *__restrict__ tri_slot,
                                                  T *__restrict__ Gtr, T *__restrict__ Rpart, const DevPhys &dph,
                                                  const int8_t *__restrict__ if_up, int64_t n_interior) {
  constexpr int Nt = N * (N + 1) / 2, Np = Nt * N, Nf = N * N;
  constexpr PrismTab L = prism_tab(N);
  T *sm = reinterpret_cast<T *>(sm_raw);
  T *sQ = sm;                 // [5][Np]
  T *sG = sQ + 5 * Np;        // [15][Np] uncorrected physical gradient, index j*5+v
  T *sH = sG + 15 * Np;       // [15][Np] transformed flux, index d*5+v
  T *sW = sH + 15 * Np;       // [5][3][Np] eta (N_f . S[.][j]) / |J|: BR2 lifting to physical space
  T *sL = sW + 15 * Np;       // [3][5][Np] C_f (Q^I - Q_f) of the quadrilateral faces
  T *sdQ = sL + 15 * Np;      // [5][5][Nf] Q^I - Q_own at the flux points
  const PhysT<T> &ph = phys_of<T>(dph);
  const bool viscous = dph.viscous != 0;
  if (active && viscous)
    for (int t = tid; t < 5 * Np; t += nth) sQ[(t % 5) * Np + t / 5] = Q[e * Np * 5 + t];
  if (viscous && active) {
    for (int t = tid; t < 5 * Nf; t += nth) {
      const int f = t / Nf, r = t % Nf;
      if (f < 2 && r >= Nt) continue;
      const int packed = ef_p[e * 5 + f];
      const int64_t I = packed >> 4;
      const int side = (packed >> 3) & 1;
      const int slot = prism_slot<N>(f, r, packed & 7, tri_slot);
      const T *own = Qtr + (I * 2 + side) * 5 * Nf + slot;
      const T *oth = Qtr + (I * 2 + (1 - side)) * 5 * Nf + slot;
      // Q^I - Q_own: BR2 (other - own)/2; LDG 0 on the supplying side, other - own on the other.
      float w = 0.5f;
      if (dph.ldg && I < n_interior) w = side == (if_up[I] ? 0 : 1) ? 0.f : 1.f;
#pragma unroll
      for (int v = 0; v < 5; ++v) sdQ[(f * 5 + v) * Nf + r] = scale2(oth[v * Nf] - own[v * Nf], w);
    }
  }
  __syncthreads();
  const bool pt = active && tid < Np;
  const int m = tid < Np ? tid : 0, q = m % Nt, k = m / Nt;
  if (pt) {
    T S[9], invJ, qv[5], G[15];
    const T *met = metrics + e * 10 * Np + m;
#pragma unroll
    for (int c = 0; c < 9; ++c) S[c] = met[c * Np];
    invJ = met[9 * Np];
#pragma unroll
    for (int v = 0; v < 5; ++v) qv[v] = Q[(e * Np + m) * 5 + v];
    if (viscous) {
      T sj[9];   // S[d][jj] / |J|
#pragma unroll
      for (int c = 0; c < 9; ++c) sj[c] = S[c] * invJ;
      // Reference gradient, uncorrected (sG) and corrected (sH), in this thread's own entries, which
      // only it writes before the next barrier.  Lifted jumps of the quadrilateral faces first (edge
      // f - 2); sum_f N_f C_f dQ_f with N = (0,0,-1), (0,0,1), (0,-1,0), (1,1,0), (-1,0,0).
#pragma unroll 1
      for (int f = 0; f < 3; ++f) {
        const T *lq = tab + L.LQ + f * N * Nt + q, *dq = sdQ + (2 + f) * 5 * Nf + N * k;
        T c[N];
#pragma unroll
        for (int a = 0; a < N; ++a) c[a] = lq[a * Nt];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          Dot<T> s(c[0], dq[v * Nf]);
#pragma unroll
          for (int a = 1; a < N; ++a) s.add(c[a], dq[v * Nf + a]);
          sL[(f * 5 + v) * Np + m] = s.raw();
        }
      }
      {
        const T *D1 = tab + L.D1 + k * N;
        const T hmk = -tab[L.hm + k], hpk = tab[L.hp + k];
        T c[N];
#pragma unroll
        for (int a = 0; a < N; ++a) c[a] = D1[a];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const T jlo = sdQ[v * Nf + q], jhi = sdQ[(5 + v) * Nf + q];
          Dot<T> s(c[0], sQ[v * Np + q]);
#pragma unroll
          for (int a = 1; a < N; ++a) s.add(c[a], sQ[v * Np + q + Nt * a]);
          sG[(10 + v) * Np + m] = s.raw();
          s.add(hmk, jlo);
          s.add(hpk, jhi);
          sH[(10 + v) * Np + m] = s.raw();
        }
      }
      {
        // Both triangle derivatives of the five variables together: an operator entry is read once.
        const T *Dr = tab + L.Dr + q, *Ds = tab + L.Ds + q, *sq = sQ + Nt * k;
        Dot<T> a0[5], a1[5];
#pragma unroll 3
        for (int j = 0; j < Nt; ++j) {
          const T dr = Dr[j * Nt], ds = Ds[j * Nt];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            const T x = sq[v * Np + j];
            a0[v].add(dr, x);
            a1[v].add(ds, x);
          }
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          const T g0 = a0[v].raw(), g1 = a1[v].raw();
          sG[v * Np + m] = g0;
          sG[(5 + v) * Np + m] = g1;
          const T L2 = sL[v * Np + m], L3 = sL[(5 + v) * Np + m], L4 = sL[(10 + v) * Np + m];
          Dot<T> c0(g0), c1(g1);
          c0.plus(L3);
          c0.plus(-L4);
          c1.plus(L3);
          c1.plus(-L2);
          sH[v * Np + m] = c0.raw();
          sH[(5 + v) * Np + m] = c1.raw();
        }
      }
#pragma unroll 1
      for (int v = 0; v < 5; ++v) {
        T gu[3], gc[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          gu[d] = sG[(d * 5 + v) * Np + m];
          gc[d] = sH[(d * 5 + v) * Np + m];
        }
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) {
          const T du = dot3(sj[jj], gu[0], sj[3 + jj], gu[1], sj[6 + jj], gu[2]);
          const T dc = dot3(sj[jj], gc[0], sj[3 + jj], gc[1], sj[6 + jj], gc[2]);
          sH[(jj * 5 + v) * Np + m] = dc;
          sG[(jj * 5 + v) * Np + m] = dph.ldg ? dc : du;   // LDG: corrected
        }
      }
#pragma unroll
      for (int c = 0; c < 15; ++c) G[c] = sH[c * Np + m];
#pragma unroll
      for (int jj = 0; jj < 3; ++jj) {
        const T ej = ph.eta * invJ;
        sW[(0 * 3 + jj) * Np + m] = -(ej * S[2 * 3 + jj]);
        sW[(1 * 3 + jj) * Np + m] = ej * S[2 * 3 + jj];
        sW[(2 * 3 + jj) * Np + m] = -(ej * S[1 * 3 + jj]);
        sW[(3 * 3 + jj) * Np + m] = ej * (S[0 * 3 + jj] + S[1 * 3 + jj]);
        sW[(4 * 3 + jj) * Np + m] = -(ej * S[0 * 3 + jj]);
      }
    }
    {
      // Physical flux, then its three transforms.
      const T ri = reciprocal(qv[0]);
      const T u[3] = {qv[1] * ri, qv[2] * ri, qv[3] * ri};
      const T p = ph.gm1 * (qv[4] - scale2(dot3(qv[1], u[0], qv[2], u[1], qv[3], u[2]), 0.5f));
      T tau[6], hq[3], mom[6], en[3];
      bool formed = false;
      if constexpr (std::is_same<T, double>::value)
        if (!viscous) {
          formed = true;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            double f[5];
            inviscid_transformed(qv, u, p, S + 3 * d, f);
#pragma unroll
            for (int v = 0; v < 5; ++v) sH[(d * 5 + v) * Np + m] = f[v];
          }
        }
      if (!formed) {
        if (viscous) viscous_stress<T>(qv, u, ri, G, ph, visc_of(ph), tau, hq);
        physical_flux<T>(qv, u, p, viscous, tau, hq, mom, en);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          T f[5];
          transformed_flux<T>(qv, mom, en, p, S + 3 * d, f);
#pragma unroll
          for (int v = 0; v < 5; ++v) sH[(d * 5 + v) * Np + m] = f[v];
        }
      }
    }
  }
  __syncthreads();
  if (viscous) {
    // Gradient traces: interpolated uncorrected gradient + eta * own lifting.  Triangular faces: one item
    // per (gradient component jj, face point).
    if (active)
      for (int t = tid; t < 6 * Nt; t += nth) {
        const int jj = t / (2 * Nt), f = t / Nt % 2, r = t % Nt;
        const int packed = ef_p[e * 5 + f];
        const int64_t I = packed >> 4;
        T *dst = Gtr + (I * 2 + ((packed >> 3) & 1)) * 15 * Nf + prism_slot<N>(f, r, packed & 7, tri_slot) + jj * 5 * Nf;
        const T *hh = tab + (f ? L.hp : L.hm);
        T l[N];
#pragma unroll
        for (int c = 0; c < N; ++c) l[c] = tab[(f ? L.lp : L.lm) + c];
        Dot<T> lf;
#pragma unroll
        for (int c = 0; c < N; ++c) lf.add(l[c] * hh[c], sW[(f * 3 + jj) * Np + r + Nt * c]);
        const T lfac = lf.raw();
#pragma unroll 1
        for (int v = 0; v < 5; ++v) {
          const T *g = sG + (jj * 5 + v) * Np + r;
          const T jump = sdQ[(f * 5 + v) * Nf + r];
          Dot<T> acc(l[0], g[0]);
#pragma unroll
          for (int c = 1; c < N; ++c) acc.add(l[c], g[Nt * c]);
          acc.add(lfac, jump);
          dst[v * Nf] = acc.raw();
        }
      }
    __syncthreads();
    // Quadrilateral faces, one after the other: every point adds the face's lifting to its gradient (kept in
    // registers), the sum replaces the gradient in sG, and the face points interpolate it.  (Interpolating
    // gradient and lifting by themselves took a product and two sums per term: 2.4 times the
    // instructions.)
    T g[15];
    if (pt) {
#pragma unroll
      for (int c = 0; c < 15; ++c) g[c] = sG[c * Np + m];
    }
#pragma unroll 1
    for (int f = 2; f < 5; ++f) {
      if (pt) {
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) {
          const T w = sW[(f * 3 + jj) * Np + m];
#pragma unroll
          for (int v = 0; v < 5; ++v)
            sG[(jj * 5 + v) * Np + m] = muladd(g[jj * 5 + v], w, sL[((f - 2) * 5 + v) * Np + m]);
        }
      }
      __syncthreads();
      if (active)
        for (int t = tid; t < 3 * Nf; t += nth) {
          const int jj = t / Nf, r = t % Nf, a = r % N, b = r / N;
          const int packed = ef_p[e * 5 + f];
          const int64_t I = packed >> 4;
          T *dst = Gtr + (I * 2 + ((packed >> 3) & 1)) * 15 * Nf + prism_slot<N>(f, r, packed & 7, tri_slot) + jj * 5 * Nf;
          const T *Ea = tab + L.E + (f - 2) * N * Nt + a, *x = sG + jj * 5 * Np + Nt * b;
          Dot<T> acc[5];
#pragma unroll 3
          for (int j = 0; j < Nt; ++j) {
            const T ej = Ea[j * N];
#pragma unroll
            for (int v = 0; v < 5; ++v) acc[v].add(ej, x[v * Np + j]);
          }
#pragma unroll
          for (int v = 0; v < 5; ++v) dst[v * Nf] = acc[v].raw();
        }
      if (f < 4) __syncthreads();
    }
  }
  if (pt) {
    const T *Drt = tab + L.Drt + q, *Dst = tab + L.Dst + q, *D1t = tab + L.D1t + k * N;
    const T *h0 = sH + Nt * k, *h1 = h0 + 5 * Np, *h2 = sH + 10 * Np + q;
    // The line's sum and the triangle's are kept apart until the end: each holds the large pressure part of some
    // momentum component, on top of which the other's terms would lose their last bits.  With the line's terms
    // first in one sum the error of the momentum component along the prisms' axis was 3.4 times as large (p = 7,
    // Ma 0.1), with the triangle's first that of the other two 1.2 times.
    Dot<T> acc[5], line[5];
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const T dc = D1t[c];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        if (c == 0)
          line[v] = Dot<T>(dc, h2[v * Np]);
        else
          line[v].add(dc, h2[v * Np + Nt * c]);
      }
    }
#pragma unroll 3
    for (int j = 0; j < Nt; ++j) {
      const T dr = Drt[j * Nt], ds = Dst[j * Nt];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        acc[v].add(dr, h0[v * Np + j]);
        acc[v].add(ds, h1[v * Np + j]);
      }
    }
    T *out = Rpart + (e * Np + m) * 5;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      acc[v].join(line[v]);
      out[v] = acc[v].raw();
    }
  }
}

// ------------------------------------------------------------------------------------------
// 4. Correction by the common flux, scaling and output / RK44 update.  Thread per prism point.
// ------------------------------------------------------------------------------------------
// Lifted common fluxes of the five faces at point m of prism e.  FP64: on top of the partial residual rp, in r,
// and `line` stays empty.  Double-float (rp null, the residual is added later): the quadrilaterals' in r and the
// triangles' in `line`, which joins r after the residual, for the reason given at the divergence.
template <int N, typename T>
__device__ __forceinline__ void prism_correct_lift(int64_t e, int m, const T *__restrict__ FI,
                                                   const int32_t *__restrict__ ef_p, const T *__restrict__ tab,
                                                   const int32_t *__restrict__ tri_slot, const T *rp, Dot<T> r[5],
                                                   Dot<T> line[5]) {
  if (rp)
#pragma unroll
    for (int v = 0; v < 5; ++v) r[v] = Dot<T>(rp[v]);
  constexpr int Nt = N * (N + 1) / 2, Nf = N * N;
  constexpr PrismTab L = prism_tab(N);
  const int q = m % Nt, k = m / Nt;
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const int packed = ef_p[e * 5 + f];
    const int64_t I = packed >> 4;
    const int side = (packed >> 3) & 1;
    const T h = tab[(f ? L.hp : L.hm) + k];
    const T w = side ? -h : h;
    const T *src = FI + I * 5 * Nf + tri_slot[(packed & 7) * Nt + q];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      if (rp)
        r[v].add(w, src[v * Nf]);
      else if (f == 0)
        line[v] = Dot<T>(w, src[v * Nf]);
      else
        line[v].add(w, src[v * Nf]);
    }
  }
#pragma unroll
  for (int f = 2; f < 5; ++f) {
    const int packed = ef_p[e * 5 + f];
    const int64_t I = packed >> 4;
    const int side = (packed >> 3) & 1;
    const T *lq = tab + L.LQ + (f - 2) * Nt * N + q;
    const T *src = FI + I * 5 * Nf;
#pragma unroll
    for (int a = 0; a < N; ++a) {
      const T w = side ? -lq[a * Nt] : lq[a * Nt];
      const int slot = orient_slot(packed & 7, a, k, N);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        if (f == 2 && a == 0 && !rp)
          r[v] = Dot<T>(w, src[v * Nf + slot]);
        else
          r[v].add(w, src[v * Nf + slot]);
      }
    }
  }
}

// Thread per point (batched stage).
template <int N, typename T>
__device__ __forceinline__ void prism_correct_body(int64_t t, const T *__restrict__ Rpart, const T *__restrict__ FI,
                                                   const int32_t *__restrict__ ef_p, const T *__restrict__ metrics,
                                                   const T *__restrict__ tab, const int32_t *__restrict__ tri_slot,
                                                   int64_t Ep, int64_t first_point, const StageCoef &sc,
                                                   double *__restrict__ Rout, double *__restrict__ Q,
                                                   T *__restrict__ Qc, double *__restrict__ Un, T *__restrict__ Unc,
                                                   double *__restrict__ acc, int *__restrict__ flag,
                                                   const DevPhys &dph) {
  constexpr int Np = N * (N + 1) / 2 * N;
  if (t >= Ep * Np) return;
  const int64_t e = t / Np;
  const int m = (int)(t % Np);
  Dot<T> r[5], line[5];
  prism_correct_lift<N, T>(e, m, FI, ef_p, tab, tri_slot, kGatherFirst<T> ? nullptr : Rpart + t * 5, r, line);
  T rv[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    if constexpr (kGatherFirst<T>) {
      r[v].plus(Rpart[t * 5 + v]);
      r[v].join(line[v]);
    }
    rv[v] = r[v].get();
  }
  finish_point<T>(first_point + t, rv, -metrics[(e * 10 + 9) * Np + m], sc, Rout, Q, Qc, Un, Unc, acc,
                  flag, dph);
}

}  // namespace
}  // namespace frx
