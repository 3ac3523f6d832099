// Hexahedral volume kernel with two elements per thread, in packed arithmetic: the inviscid flux and its
// divergence in double-float, the viscous branch in FP32 (FR_PREC_MIXED_VF32).
//
// With two elements per thread the loads, addresses and loop overhead, a quarter of the scalar kernel's
// instructions, fill the issue slots that the packed arithmetic (fr_f32x2.cuh) leaves.
#pragma once

#include "fr_bodies.cuh"

namespace frx {
namespace {

__device__ __forceinline__ f2 to_f2(d2 x) { return padd(x.hi, x.lo); }
__device__ __forceinline__ d2 from_f2(f2 x) { return d2{x, dupf(0.f)}; }
__device__ __forceinline__ f2 dup_f2(df32 x) { return to_f2(dup(x)); }

__device__ __forceinline__ PhysT<f2> pair_phys(const PhysT<df32> &p) {
  PhysT<f2> r;
  r.cT = dup_f2(p.cT);
  r.mu = dup_f2(p.mu);
  r.m2mu3 = dup_f2(p.m2mu3);
  r.kappa = dup_f2(p.kappa);
  return r;
}

// Bytes of shared memory per pair of elements: state perturbation 5, gradient 15 (FP32) and flux 15 (double-float) per
// point, jumps 30 per N^2; an inviscid run keeps the flux only.
template <int N, bool VISC>
constexpr int pair_smem() {
  constexpr int Np = N * N * N, Nf = N * N;
  return VISC ? 20 * Np * 8 + 15 * Np * 16 + 30 * Nf * 8 : 15 * Np * 16;
}
template <int N, bool VISC>
constexpr int pair_blocks() {
  // By shared memory (227 KB per SM), and not below 128 registers per thread.
  constexpr int by_smem = 227 * 1024 / (pair_smem<N, VISC>() + 1024);
  constexpr int by_regs = 512 / volume_threads<N>();
  return by_smem < by_regs ? by_smem : (by_regs > 0 ? by_regs : 1);
}

// Orders it is built for, and what the volume kernel takes per launch against the scalar one (GB300).  It halves the
// warps of an SM for the same shared memory, so it gains where enough of them remain: FP32 viscous branch
// 40^3 p = 3 0.638 -> 0.571 ms, 4800 elements p = 4 0.106 -> 0.097, p = 5 0.193 -> 0.170, p = 7 0.562 -> 0.493 (not
// p = 2: 0.324 -> 0.331 at 40^3, p = 6: 0.912 -> 0.946 at 24^3); inviscid 40^3 p = 2 0.098 -> 0.086, p = 3 0.209 ->
// 0.191, 4800 elements p = 4 0.042 -> 0.041.  With the viscous branch in double-float it was slower at every size (40^3
// p = 2 0.445 -> 0.460, p = 3 0.938 -> 0.960, 48^3 p = 4 3.09 -> 3.51).
template <int N, bool VISC>
constexpr bool pair_built() {
  return VISC ? N == 4 || N == 5 || N == 6 || N == 8 : N >= 3 && N <= 5;
}

// Element counts it pays at.  A block of it lasts longer than one of the scalar kernel, and there are half as many, so
// on meshes of a few elements per SM (152) the scalar kernel is through first; where exactly depends on how
// the blocks of either fill the SMs.  Volume launch, pair / scalar, us:
//   FP32 viscous p = 3:  308 elements 14.5 / 13.6, 800 17.8 / 16.4, 1200 18.5 / 18.5, 1600 22.4 / 24.8
//     (2400: 33.4 / 33.0), 4800 53.8 / 57.6;
//   p = 4:  153 14.6 / 14.0, 308 18.4 / 16.3, 400 18.6 / 16.4, 500 18.6 / 18.4, 600 18.6 / 18.7, 800 22.7 / 26.1;
//   p = 5:  100 16.5 / 14.5, 153 16.7 / 18.4, 250 16.7 / 18.8, 308 24.6 / 23.0, 400 25.0 / 24.4, 500 25.4 / 29.8;
//   p = 7:  100 31.4 / 20.9, 153 31.6 / 35.1, 250 32.2 / 37.0, 308 56.2 / 51.2, 400 58.5 / 52.1, 500 60.6 / 69.0;
//   inviscid p = 2:  100 7.9 / 6.8, 600 8.1 / 7.9, 1200 8.3 / 8.3, 1600 8.8 / 8.3, 2400 9.0 / 10.1;
//   p = 3:  100 8.0 / 7.5, 308 8.3 / 8.1, 800 9.7 / 8.5, 1200 10.0 / 10.2, 1600 11.3 / 12.2;
//   p = 4:  100 8.3 / 7.9, 308 10.2 / 9.2, 400 10.4 / 9.8, 500 10.4 / 10.4, 600 10.3 / 10.8, 1200 14.5 / 14.9.
// At p = 5 and 7 one pair block per SM beats the second scalar block, two do not beat the third.
template <int N, bool VISC>
bool pair_pays(int64_t E) {
  if (VISC && N >= 6) return E > 152 && (E <= 2 * 152 || E > 3 * 152);
  return E > 152 * (VISC ? (N == 4 ? 8 : 4) : (N == 3 ? 12 : (N == 4 ? 8 : 3)));
}

// One thread per solution point of the elements e0 and e1; the operations of volume_body in its order.  An odd
// mesh's last block holds one element twice: both lanes then store the same values.
template <int N, bool VISC>
__global__ void __launch_bounds__(volume_threads<N>(), pair_blocks<N, VISC>())
    k_volume_pair(const df32 *__restrict__ Q, const df32 *__restrict__ metrics, const int32_t *__restrict__ ef,
                  const df32 *__restrict__ Qtr, const df32 *__restrict__ liftfac, df32 *__restrict__ Gtr,
                  df32 *__restrict__ Rpart, DevPhys dph, const int8_t *__restrict__ if_up, int64_t n_interior,
                  int64_t E) {
  extern __shared__ float4 sm_pair[];
  constexpr int Np = N * N * N, Nf = N * N, nth = volume_threads<N>();
  d2 *sH = reinterpret_cast<d2 *>(sm_pair);                    // [15][Np] transformed flux, index d*5+v
  f2 *sQ = reinterpret_cast<f2 *>(sH + 15 * Np);               // [5][Np] perturbation from the first point
  f2 *sG = sQ + 5 * Np;                                        // [15][Np] uncorrected gradient, j*5+v
  f2 *sdQ = sG + 15 * Np;                                      // [6][5][Nf] Q^I - Q_own at the flux points
  const int64_t e0 = (int64_t)blockIdx.x * 2, e1 = e0 + 1 < E ? e0 + 1 : e0;
  const int tid = threadIdx.x;
  const BasisT<df32> &B = cbasis<df32>(N);
  const bool pt = tid < Np;
  const int m = pt ? tid : 0, i = m % N, j = (m / N) % N, k = m / (N * N);
  const df32 *Q0 = Q + e0 * Np * 5, *Q1 = Q + e1 * Np * 5;
  d2 S[9], invJ, q[5];
  if (pt) {
    const df32 *m0 = metrics + e0 * 10 * Np + m, *m1 = metrics + e1 * 10 * Np + m;
#pragma unroll
    for (int c = 0; c < 9; ++c) S[c] = pack(m0[c * Np], m1[c * Np]);
    invJ = pack(m0[9 * Np], m1[9 * Np]);
  }
  if constexpr (VISC) {
    for (int t = tid; t < 5 * Np; t += nth)
      sQ[(t % 5) * Np + t / 5] = to_f2(pack(Q0[t], Q1[t]) - pack(Q0[t % 5], Q1[t % 5]));
    for (int t = tid; t < 6 * Nf; t += nth) {
      const int f = t / Nf, r = t % Nf;
      const df32 *own[2], *oth[2];
      float w[2];
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        const int packed = ef[(l ? e1 : e0) * 6 + f];
        const int64_t I = packed >> 4;
        const int side = (packed >> 3) & 1, slot = slot_of(packed & 7, r % N, r / N, N);
        own[l] = Qtr + (I * 2 + side) * 5 * Nf + slot;
        oth[l] = Qtr + (I * 2 + (1 - side)) * 5 * Nf + slot;
        w[l] = 0.5f;
        if (dph.ldg && I < n_interior) w[l] = side == (if_up[I] ? 0 : 1) ? 0.f : 1.f;
      }
#pragma unroll
      for (int v = 0; v < 5; ++v)
        sdQ[(f * 5 + v) * Nf + r] = to_f2(scale2(
            pack(oth[0][v * Nf], oth[1][v * Nf]) - pack(own[0][v * Nf], own[1][v * Nf]), mkf2(w[0], w[1])));
    }
  }
  __syncthreads();
  f2 G[15];
  if (pt) {
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = pack(Q0[m * 5 + v], Q1[m * 5 + v]);
    if constexpr (VISC) {
      f2 sj[9];   // S[d][jj] / |J|
#pragma unroll
      for (int c = 0; c < 9; ++c) sj[c] = to_f2(S[c] * invJ);
      constexpr int R = sizeof(d2) / sizeof(f2);
      f2 *sGc = reinterpret_cast<f2 *>(sH);
      auto gslot = [&](int c) { return ((c / R) * Np + m) * R + c % R; };
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int row = d == 0 ? i : (d == 1 ? j : k), st = axis_stride<N>(d), at = m - row * st;
        const int r = d == 0 ? j + N * k : (d == 1 ? i + N * k : i + N * j);
        f2 c[N];
#pragma unroll
        for (int a = 0; a < N; ++a) c[a] = dup_f2(B.D[row * N + a]);
        const f2 hlo = -dup_f2(B.hm[row]), hhi = dup_f2(B.hp[row]);
        const f2 *dq = sdQ + d * 10 * Nf + r;
#pragma unroll 1
        for (int v = 0; v < 5; ++v) {
          const f2 jlo = dq[v * Nf], jhi = dq[(5 + v) * Nf];
          Dot<f2> s(c[0], sQ[v * Np + at]);
#pragma unroll
          for (int a = 1; a < N; ++a) s.add(c[a], sQ[v * Np + at + a * st]);
          sG[(d * 5 + v) * Np + m] = s.raw();
          s.add(hlo, jlo);
          s.add(hhi, jhi);
          sGc[gslot(d * 5 + v)] = s.raw();
        }
      }
#pragma unroll 1
      for (int v = 0; v < 5; ++v) {
        f2 gu[3], gc[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          gu[d] = sG[(d * 5 + v) * Np + m];
          gc[d] = sGc[gslot(d * 5 + v)];
        }
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) {
          const f2 du = dot3(sj[jj], gu[0], sj[3 + jj], gu[1], sj[6 + jj], gu[2]);
          const f2 dc = dot3(sj[jj], gc[0], sj[3 + jj], gc[1], sj[6 + jj], gc[2]);
          sGc[gslot(jj * 5 + v)] = dc;
          // Face-gradient source: BR2 the uncorrected gradient (+ eta r_f), LDG the corrected one.
          sG[(jj * 5 + v) * Np + m] = dph.ldg ? dc : du;
        }
      }
#pragma unroll
      for (int c = 0; c < 15; ++c) G[c] = sGc[gslot(c)];
    }
    const d2 ri = reciprocal(q[0]);
    const d2 u[3] = {q[1] * ri, q[2] * ri, q[3] * ri};
    const d2 p = dup(dph.f.gm1) * (q[4] - scale2(dot3(q[1], u[0], q[2], u[1], q[3], u[2]), 0.5f));
    d2 tau[6], hq[3], mom[6], en[3];
    if constexpr (VISC) {
      const PhysT<f2> pg = pair_phys(dph.f);
      f2 qg[5], ug[3], taug[6], hqg[3], rig;
#pragma unroll
      for (int v = 0; v < 5; ++v) qg[v] = to_f2(q[v]);
      rig = reciprocal(qg[0]);
#pragma unroll
      for (int c = 0; c < 3; ++c) ug[c] = qg[1 + c] * rig;
      viscous_stress<f2>(qg, ug, rig, G, pg, visc_of(pg), taug, hqg);
#pragma unroll
      for (int a = 0; a < 3; ++a) hq[a] = from_f2(hqg[a]);
#pragma unroll
      for (int a = 0; a < 6; ++a) tau[a] = from_f2(taug[a]);
    }
    physical_flux<d2>(q, u, p, VISC, tau, hq, mom, en);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      d2 f[5];
      transformed_flux<d2>(q, mom, en, p, S + 3 * d, f);
#pragma unroll
      for (int v = 0; v < 5; ++v) sH[(d * 5 + v) * Np + m] = f[v];
    }
  }
  __syncthreads();
  if constexpr (VISC) {
    for (int t = tid; t < 9 * Nf; t += nth) {
      const int jj = t / (3 * Nf), dr = t - jj * 3 * Nf;
      const int d = dr / Nf, r = dr % Nf;
      int base, sd;
      face_line<N>(2 * d, r, base, sd);
      df32 *dst[2][2];
      f2 lj[2];
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int f = 2 * d + s;
#pragma unroll
        for (int l = 0; l < 2; ++l) {
          const int packed = ef[(l ? e1 : e0) * 6 + f];
          const int64_t I = packed >> 4;
          dst[s][l] = Gtr + (I * 2 + ((packed >> 3) & 1)) * 15 * Nf + slot_of(packed & 7, r % N, r / N, N) + jj * 5 * Nf;
        }
        lj[s] = to_f2(dup(dph.f.eta) *
                          pack(liftfac[((e0 * 6 + f) * 3 + jj) * Nf + r], liftfac[((e1 * 6 + f) * 3 + jj) * Nf + r]));
      }
#pragma unroll 1
      for (int v = 0; v < 5; ++v) {
        const f2 *sg = sG + (jj * 5 + v) * Np + base;
        f2 x[N];
#pragma unroll
        for (int c = 0; c < N; ++c) x[c] = sg[c * sd];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          auto l = [&](int c) { return dup_f2(s ? B.lp[c] : B.lm[c]); };
          const f2 jump = sdQ[((2 * d + s) * 5 + v) * Nf + r];
          Dot<f2> acc(l(0), x[0]);
#pragma unroll
          for (int c = 1; c < N; ++c) acc.add(l(c), x[c]);
          acc.add(lj[s], jump);
          const d2 g = from_f2(acc.raw());
          dst[s][0][v * Nf] = lane0(g);
          dst[s][1][v * Nf] = lane1(g);
        }
      }
    }
  }
  if (pt) {
    df32 *out0 = Rpart + (e0 * Np + m) * 5, *out1 = Rpart + (e1 * Np + m) * 5;
#pragma unroll 1
    for (int v = 0; v < 5; ++v) {
      const d2 *h0 = sH + (0 * 5 + v) * Np, *h1 = sH + (1 * 5 + v) * Np, *h2 = sH + (2 * 5 + v) * Np;
      Dot<d2> acc(dup(B.Dt[i * N]), h0[N * j + N * N * k]);
      acc.add(dup(B.Dt[j * N]), h1[i + N * N * k]);
      acc.add(dup(B.Dt[k * N]), h2[i + N * j]);
#pragma unroll
      for (int a = 1; a < N; ++a) {
        acc.add(dup(B.Dt[i * N + a]), h0[a + N * j + N * N * k]);
        acc.add(dup(B.Dt[j * N + a]), h1[i + N * a + N * N * k]);
        acc.add(dup(B.Dt[k * N + a]), h2[i + N * j + N * N * a]);
      }
      const d2 o = acc.raw();
      out0[v] = lane0(o);
      out1[v] = lane1(o);
    }
  }
}

}  // namespace
}  // namespace frx
