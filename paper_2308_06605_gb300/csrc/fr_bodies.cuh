// Device bodies of the hexahedral FR kernels, shared by the per-mesh kernels (fr_kernels.cu)
// and the batched persistent stage kernel (fr_batch_kernel.cu).  Everything here has internal
// linkage: each translation unit that includes it holds its own copy, including the constant-
// memory basis tables, which each unit uploads through its upload_basis_local().
//
// Kernels of the FR residual and the RK44 stage update (arXiv 2308.06605, section "FR
// Algorithm", Eq. 1-3).  One residual evaluation is four launches (plus two for boundary faces):
//   interp_faces : Q -> solution traces at the flux points of every face (interface slots)
//   bc_prepare   : boundary faces: common solution Q^I and ghost traces
//   volume       : per element, BR2-corrected gradients, physical + transformed fluxes at the
//                  solution points, gradient traces at the flux points, and the divergence of
//                  the transformed flux including the own-flux part of the correction
//   iface_flux   : per interface flux point, Rusanov + BR2 common normal flux (bc_flux for
//                  boundary faces)
//   correct      : per solution point, adds the common-flux correction, scales by -1/|J| and
//                  writes R or applies the RK44 stage update (always FP64).
//
// Every kernel is a template on the scalar type T of its element arithmetic and of the arrays it
// exchanges: T = double is the FP64 path; T = df32 (FP32 hi + lo pairs on the FP32 pipe) is the
// mixed path, in which the Riemann flux's pressure/energy recovery, the boundary states and the
// RK update stay FP64.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include <cuda_bf16.h>

#include "df32.cuh"
#include "fr_device.hpp"
#include "fr_f32x2.cuh"
#include "fr_point.cuh"
#include "fr_prism_bodies.cuh"

namespace frx {
namespace {

template <typename T>
struct BasisT {
  T D[kMaxN * kMaxN];    // D[i*N + a] = l_a'(x_i)
  T Dt[kMaxN * kMaxN];   // D - hp (x) lp + hm (x) lm: divergence with the own-flux correction
  T lm[kMaxN], lp[kMaxN], hm[kMaxN], hp[kMaxN];
  double w[kMaxN];       // Gauss-Legendre weights (closure's element means)
};

__constant__ BasisT<double> c_basis_d[kMaxN];   // index N - 1
__constant__ BasisT<df32> c_basis_f[kMaxN];

template <typename T> __device__ __forceinline__ const BasisT<T> &cbasis(int N);
template <> __device__ __forceinline__ const BasisT<double> &cbasis<double>(int N) { return c_basis_d[N - 1]; }
template <> __device__ __forceinline__ const BasisT<df32> &cbasis<df32>(int N) { return c_basis_f[N - 1]; }

// 1D tables of one order in both element arithmetics.
inline void fill_basis(const Basis1D &b, BasisT<double> &d, BasisT<df32> &f) {
  const int N = b.N;
  d = BasisT<double>{};
  f = BasisT<df32>{};
  for (int i = 0; i < N; ++i) {
    d.lm[i] = b.lm[i];
    d.lp[i] = b.lp[i];
    d.hm[i] = b.hm[i];
    d.hp[i] = b.hp[i];
    d.w[i] = b.w[i];
    for (int a = 0; a < N; ++a) {
      d.D[i * N + a] = b.D[i * N + a];
      d.Dt[i * N + a] = b.D[i * N + a] - b.hp[i] * b.lp[a] + b.hm[i] * b.lm[a];
    }
  }
  for (int i = 0; i < kMaxN; ++i) {
    f.lm[i] = df_split_host(d.lm[i]);
    f.lp[i] = df_split_host(d.lp[i]);
    f.hm[i] = df_split_host(d.hm[i]);
    f.hp[i] = df_split_host(d.hp[i]);
    f.w[i] = d.w[i];
  }
  for (int i = 0; i < kMaxN * kMaxN; ++i) {
    f.D[i] = df_split_host(d.D[i]);
    f.Dt[i] = df_split_host(d.Dt[i]);
  }
}

// Upload of this translation unit's copy of the 1D basis tables (constant memory is per unit);
// DG-equivalent correction.
cudaError_t upload_basis_local() {
  BasisT<double> hd[kMaxN] = {};
  BasisT<df32> hf[kMaxN] = {};
  for (int p = 1; p < kMaxN; ++p) fill_basis(make_basis(p), hd[p], hf[p]);
  cudaError_t e = cudaMemcpyToSymbol(c_basis_d, hd, sizeof(hd));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_basis_f, hf, sizeof(hf));
}

// Tables of the kernels: the constant-memory DG-equivalent ones, or (VC) the mesh's own copy in
// global memory for a correction function c != 0 of the energy-stable family.
template <int N, typename T, bool VC>
__device__ __forceinline__ const BasisT<T> &basis_ref(const DevPhys &dph) {
  if constexpr (VC)
    return *reinterpret_cast<const BasisT<T> *>(dph.vc_basis);
  else
    return cbasis<T>(N);
}

// Strides of the reference axes in the point index m = i + N j + N^2 k.
template <int N>
__device__ __forceinline__ int axis_stride(int a) {
  return a == 0 ? 1 : (a == 1 ? N : N * N);
}

// Flux point r = a + N b of face f: base index of its normal line and the stride along it.
template <int N>
__device__ __forceinline__ void face_line(int f, int r, int &base, int &sd) {
  const int d = f >> 1;
  const int t0 = (d == 0) ? 1 : 0, t1 = (d == 2) ? 1 : 2;
  const int a = r % N, b = r / N;
  base = a * axis_stride<N>(t0) + b * axis_stride<N>(t1);
  sd = axis_stride<N>(d);
}

__device__ __forceinline__ int slot_of(int code, int a, int b, int N) {
  if (code & 4) { int t = a; a = b; b = t; }
  if (code & 1) a = N - 1 - a;
  if (code & 2) b = N - 1 - b;
  return a + N * b;
}

// Eddy-viscosity network for one element, evaluated by one warp (lane = 0..31): BF16 weights,
// FP32 activations and accumulation.  x: the 11 raw features; buf: 128 floats of shared memory.
// Returns nu_t = s_out Delta^2 softplus(z) (Delta = x[10]).
__device__ __forceinline__ float closure_mlp(const DevPhys &dph, const float x_raw[11], float *buf, int lane) {
  const __nv_bfloat16 *W = static_cast<const __nv_bfloat16 *>(dph.cw);
  const float *sc = dph.cscale;
  float x[11];
#pragma unroll
  for (int c = 0; c < 11; ++c) x[c] = (x_raw[c] - sc[c]) / sc[11 + c];
  const __nv_bfloat16 *W1 = W, *b1 = W1 + 64 * 11, *W2 = b1 + 64, *b2 = W2 + 64 * 64, *W3 = b2 + 64,
                      *b3 = W3 + 64 * 64, *w4 = b3 + 64, *b4 = w4 + 64;
  // Lane l owns neurons 2 l and 2 l + 1.  The device copy of W1, W2, W3 is stored input-major ([input][64], see
  // fr_set_closure), so the 32 lanes read one 128-byte row per input; with the rows output-major every
  // such load touched 32 lines (8200 L1 wavefronts per element).  FP64 24^3 p = 2 with the closure: 0.68 ->
  // 0.45 ms per volume launch.
  auto row = [lane](const __nv_bfloat16 *w, int c) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(w + c * 64 + 2 * lane));
  };
  auto gelu = [](float a) { return 0.5f * a * (1.f + erff(a * 0.70710678118654752f)); };
  float *hA = buf, *hB = buf + 64;
  {
    float2 a = row(b1, 0);
#pragma unroll
    for (int c = 0; c < 11; ++c) {
      const float2 w = row(W1, c);
      a.x = fmaf(w.x, x[c], a.x);
      a.y = fmaf(w.y, x[c], a.y);
    }
    hA[2 * lane] = gelu(a.x);
    hA[2 * lane + 1] = gelu(a.y);
  }
  __syncwarp();
  const __nv_bfloat16 *Ws[2] = {W2, W3}, *bs[2] = {b2, b3};
  float *hin = hA, *hout = hB;
#pragma unroll
  for (int layer = 0; layer < 2; ++layer) {
    float2 a = row(bs[layer], 0);
#pragma unroll 16
    for (int c = 0; c < 64; ++c) {
      const float2 w = row(Ws[layer], c);
      const float h = hin[c];
      a.x = fmaf(w.x, h, a.x);
      a.y = fmaf(w.y, h, a.y);
    }
    hout[2 * lane] = gelu(a.x);
    hout[2 * lane + 1] = gelu(a.y);
    __syncwarp();
    float *t = hin;
    hin = hout;
    hout = t;
  }
  float z = __bfloat162float(w4[lane]) * hin[lane] + __bfloat162float(w4[lane + 32]) * hin[lane + 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  z += __bfloat162float(b4[0]);
  const float sp = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));
  __syncwarp();
  return sc[22] * x_raw[10] * x_raw[10] * sp;
}

// ------------------------------------------------------------------------------------------
// 1. Solution traces.  Thread per (element, face, flux point).
// ------------------------------------------------------------------------------------------
template <int N, typename T>
__device__ __forceinline__ void interp_body(int64_t t, const T *__restrict__ Q, const int32_t *__restrict__ ef,
                                            T *__restrict__ Qtr, int64_t E) {
  constexpr int Np = N * N * N, Nf = N * N;
  if (t >= E * 6 * Nf) return;
  const int r = (int)(t % Nf);
  const int64_t eff = t / Nf;
  const int f = (int)(eff % 6);
  const int64_t e = eff / 6;
  const BasisT<T> &B = cbasis<T>(N);
  const T *l = (f & 1) ? B.lp : B.lm;
  int base, sd;
  face_line<N>(f, r, base, sd);
  const T *q = Q + e * Np * 5;
  Dot<T> acc[5];
#pragma unroll
  for (int c = 0; c < N; ++c) {
    const T lc = l[c];
    const T *qc = q + (base + c * sd) * 5;
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v].add(lc, qc[v]);
  }
  const int packed = ef[eff];
  const int64_t I = packed >> 4;
  const int side = (packed >> 3) & 1;
  const int slot = slot_of(packed & 7, r % N, r / N, N);
  T *dst = Qtr + (I * 2 + side) * 5 * Nf + slot;
#pragma unroll
  for (int v = 0; v < 5; ++v) dst[v * Nf] = acc[v].get();
}

template <int N, typename T>
__global__ void k_interp_faces(const T *__restrict__ Q, const int32_t *__restrict__ ef,
                               T *__restrict__ Qtr, int64_t E) {
  interp_body<N, T>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, Q, ef, Qtr, E);
}

// The same interpolation for double-float, with the elements' states staged through shared memory: a
// block loads interp_epb<N>() consecutive elements with coalesced reads (the point-major [pt][v] layout
// of consecutive elements is one contiguous range), then one thread per line of points and pair of
// opposite faces interpolates to both of its ends from one set of values.  Elements per block fill whole
// warps with 3 N^2 lines each (p = 4: 375 of 384 threads).  Bound by FP32 issue and by 88 bytes per point of
// traffic (0.18 ms at 48^3 p = 4): 0.357 -> 0.276 ms per launch against one thread per face
// point, 20^3 p = 7 0.144 -> 0.080 ms.
template <int N>
__host__ __device__ constexpr int interp_epb() {
  return N == 2 ? 16 : (N == 3 ? 7 : (N == 4 ? 4 : (N == 5 ? 5 : (N == 8 ? 1 : 2))));
}
template <int N>
__host__ __device__ constexpr int interp_threads() { return (3 * N * N * interp_epb<N>() + 31) / 32 * 32; }

template <int N, typename T>
__global__ void __launch_bounds__(interp_threads<N>())
    k_interp_faces_smem(const T *__restrict__ Q, const int32_t *__restrict__ ef, T *__restrict__ Qtr, int64_t E) {
  constexpr int Np = N * N * N, Nf = N * N, EPB = interp_epb<N>(), NT = interp_threads<N>();
  __shared__ T sq[EPB * 5 * Np];     // [element][point][v], as in memory
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int ne = (int)(E - e0 < EPB ? E - e0 : EPB);
  const T *src = Q + e0 * Np * 5;
  for (int idx = threadIdx.x; idx < ne * Np * 5; idx += NT) sq[idx] = src[idx];
  __syncthreads();
  const int le = threadIdx.x / (3 * Nf), dr = threadIdx.x - le * 3 * Nf;
  if (le >= ne) return;
  const BasisT<T> &B = cbasis<T>(N);
  const int d = dr / Nf, r = dr % Nf;
  int base, sd;
  face_line<N>(2 * d, r, base, sd);
  T *dst[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int packed = ef[(e0 + le) * 6 + 2 * d + s];
    const int64_t I = packed >> 4;
    dst[s] = Qtr + (I * 2 + ((packed >> 3) & 1)) * 5 * Nf + slot_of(packed & 7, r % N, r / N, N);
  }
  const T *q = sq + (le * Np + base) * 5;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    Dot<T> lo(B.lm[0], q[v]), hi(B.lp[0], q[v]);
#pragma unroll
    for (int c = 1; c < N; ++c) {
      const T x = q[c * sd * 5 + v];
      lo.add(B.lm[c], x);
      hi.add(B.lp[c], x);
    }
    dst[0][v * Nf] = lo.get();
    dst[1][v * Nf] = hi.get();
  }
}

// ------------------------------------------------------------------------------------------
// 2. Volume kernel.  One block per element, one thread per solution point.
// ------------------------------------------------------------------------------------------
template <int N>
__host__ __device__ constexpr int volume_threads() { return ((N * N * N + 31) / 32) * 32; }
// Resident blocks the register budget must allow (smem allows at least this many).
template <int N>
constexpr int volume_min_blocks() {
  // Measured on GB300: 16 warps per SM (128 registers) is fastest for the 32- and 64-thread
  // blocks of p = 2, 3 and for the 128-thread blocks of p = 4 (4 blocks; 3 blocks of 168 registers were
  // 3 % slower); p = 1 keeps 8 blocks (16 would spill).
  return N == 2 ? 8 : (N == 5 ? 4 : (volume_threads<N>() <= 128 ? 512 / volume_threads<N>()
                                                                 : (volume_threads<N>() <= 256 ? 2 : 1)));
}

// Shared-memory values (of T) one element needs in the volume kernel.
template <int N>
__host__ __device__ constexpr int volume_smem_values() { return 35 * N * N * N + 30 * N * N; }

// Shared memory of the closure's features and activations, and the block's elements: element e0 + l of
// l < n has closure_floats<N>() floats at red + l * closure_floats<N>().
struct ClosureSpace {
  float *red;
  int64_t e0;
  int n, mine;         // elements of the block, and the calling thread's
};
template <int N>
__host__ __device__ constexpr int closure_floats() { return 10 * N * N * N + 1 + 128; }

// One element e handled by `nth` threads of the block (thread index tid in [0, nth)); every
// thread of the block calls this together (it contains block barriers); inactive sub-blocks
// (active = false) only take part in the barriers.
// VISC: 1 viscous, 0 inviscid (only the transformed flux lives in shared memory), 2 decided at run time.
// SPLIT: five groups of volume_threads<N>() threads, one per variable in the gradient and the divergence.
template <int N, typename T, bool VC, bool FP32V, int VISC, bool SPLIT = false>
__device__ __forceinline__ void volume_body(int64_t e, int tid, int nth, bool active, double *sm_raw,
                                            const T *__restrict__ Q, const T *__restrict__ metrics,
                                            const int32_t *__restrict__ ef, const T *__restrict__ Qtr,
                                            const T *__restrict__ liftfac, T *__restrict__ Gtr,
                                            T *__restrict__ Rpart, const DevPhys &dph,
                                            const double *__restrict__ hel, float *__restrict__ nu_out,
                                            const int8_t *__restrict__ if_up, int64_t n_interior,
                                            const ClosureSpace &cs) {
  constexpr int Np = N * N * N, Nf = N * N;
  using TG = typename GradOf<T, FP32V>::type;   // arithmetic of the viscous branch
  constexpr bool kPert = !std::is_same<TG, T>::value;
  T *sm = reinterpret_cast<T *>(sm_raw);
  T *sQ = sm;                                                // [5][Np]
  TG *sG = reinterpret_cast<TG *>(sQ + 5 * Np);              // [15][Np] uncorrected physical gradient, j*5+v
  T *sH = VISC == 0 ? sm : sQ + 20 * Np;                     // [15][Np] transformed flux, index d*5+v
  TG *sdQ = reinterpret_cast<TG *>(sH + 15 * Np);            // [6][5][Nf] Q^I - Q_own at the flux points
  // FP32 viscous branch: Q minus the element's first point, in FP32, in the upper half of the
  // gradient buffer (the FP32 gradient uses only its lower half).
  TG *sQg = kPert ? reinterpret_cast<TG *>(sQ + 5 * Np) + 15 * Np : nullptr;   // [5][Np]
  const PhysT<T> &ph = phys_of<T>(dph);
  const PhysT<TG> &phg = phys_of<TG>(dph);
  const BasisT<T> &B = basis_ref<N, T, VC>(dph);
  // Sums of products end with raw(): the compensated sum renormalised by one fast_two_sum only (an
  // error of the order of 2^-48 of the sum of the terms' magnitudes).  All of them are compensated sums
  // (Dot).  Summing the gradient and its traces on top of a large offset instead (7 FP32 instructions per
  // term for 12) took 3 % off this kernel at 48^3 p = 4 (3.13 -> 3.05 ms), but a variable of zero mean lost up to
  // three bits: at p = 7 and Re 0.1 the momentum residual's error grew from 1.4e-11 to 5.0e-11 on hexahedra and
  // from 2.0e-11 to 1.8e-10 on prisms.  Transform and traces use packed instructions in double-float (48^3 p = 4 3.09 -> 3.00 ms,
  // 28^3 p = 5 1.174 -> 1.154, but 24^3 p = 6 1.30 -> 1.315 with its spills; packing the gradient's and the flux's
  // variables in pairs as well measured 3.03).  The kernel is bound by FP32 issue.
  const bool viscous = VISC == 2 ? dph.viscous != 0 : VISC == 1;
  const int grp = SPLIT ? tid / volume_threads<N>() : 0, tp = SPLIT ? tid % volume_threads<N>() : tid;
  const int v0 = SPLIT ? grp : 0, v1 = SPLIT ? grp + 1 : 5;     // this thread's variables
  const bool mine = active && tp < Np, pt = mine && grp == 0;
  const int m = tp < Np ? tp : 0, i = m % N, j = (m / N) % N, k = m / (N * N);
  // The point's metric terms are loaded before the staging loops so that their latency overlaps them.
  T S[9], invJ, q[5];
  if (mine) {
    const T *met = metrics + e * 10 * Np + m;
#pragma unroll
    for (int c = 0; c < 9; ++c) S[c] = met[c * Np];
    invJ = met[9 * Np];
  }
  // The state goes through shared memory for the gradient only.
  if (active && viscous)
    for (int t = tid; t < 5 * Np; t += nth) {
      const T x = Q[e * Np * 5 + t];
      sQ[(t % 5) * Np + t / 5] = x;
      if constexpr (kPert) sQg[(t % 5) * Np + t / 5] = to_g<TG>(x - Q[e * Np * 5 + t % 5]);
    }
  if (viscous && active) {
    for (int t = tid; t < 6 * Nf; t += nth) {
      const int f = t / Nf, r = t % Nf;
      const int packed = ef[e * 6 + f];
      const int64_t I = packed >> 4;
      const int side = (packed >> 3) & 1;
      const int slot = slot_of(packed & 7, r % N, r / N, N);
      const T *own = Qtr + (I * 2 + side) * 5 * Nf + slot;
      const T *oth = Qtr + (I * 2 + (1 - side)) * 5 * Nf + slot;
      // Q^I - Q_own.  BR2: (other - own)/2 (a boundary's other slot holds 2 Q^I - Q-).  LDG: 0 on
      // the side that supplies Q^I, other - own on the other; boundaries as BR2.
      float w = 0.5f;
      if (dph.ldg && I < n_interior) w = side == (if_up[I] ? 0 : 1) ? 0.f : 1.f;
#pragma unroll
      for (int v = 0; v < 5; ++v) sdQ[(f * 5 + v) * Nf + r] = to_g<TG>(scale2(oth[v * Nf] - own[v * Nf], w));
    }
  }
  __syncthreads();
  TG G[15];
  // The reference gradient, uncorrected and corrected, goes through shared memory, in this thread's own
  // entries of the gradient and transformed-flux buffers, which only this thread writes before the next
  // barrier (R gradient values of type TG per entry of type T).
  constexpr int R = sizeof(T) / sizeof(TG);
  TG *sGc = reinterpret_cast<TG *>(sH);
  auto gslot = [&](int c) { return ((c / R) * Np + m) * R + c % R; };
  if (mine) {
    if (pt)
#pragma unroll
      for (int v = 0; v < 5; ++v) q[v] = viscous ? sQ[v * Np + m] : Q[(e * Np + m) * 5 + v];
    if (viscous) {
      // S[d][jj] / |J|.  Double-float transforms the uncorrected and the corrected gradient as the two lanes
      // of packed instructions (their parts wait in shared memory lane by lane: (hi, hi) in sG, (lo, lo) in sGc).
      constexpr bool kPack = std::is_same<TG, df32>::value;
      typename std::conditional<kPack, d2, TG>::type sj[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        if constexpr (kPack)
          sj[c] = dup(S[c] * invJ);
        else
          sj[c] = to_g<TG>(S[c] * invJ);
      }
      const TG *sq;
      if constexpr (kPert)
        sq = sQg;
      else
        sq = sQ;
      // One reference direction at a time: its row of D (indexed by the lane's own i, j or k, so every
      // read of it from constant memory is a divergent one) is loaded once for the five variables.  With the
      // variables outside, the three rows were re-read for each of them (address-divergence unit 37 %
      // busy): double-float 48^3 p = 4 3.43 -> 3.27 ms per launch, 20^3 p = 7 1.56 -> 1.25 ms, 28^3 p = 5 1.30 ->
      // 1.17 ms; FP64 unchanged.  At p = 7 the five variables are unrolled (one block per SM: more loads in
      // flight; 1.270 -> 1.248 ms), below they stay rolled.
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int row = d == 0 ? i : (d == 1 ? j : k), st = axis_stride<N>(d), at = m - row * st;
        const int r = d == 0 ? j + N * k : (d == 1 ? i + N * k : i + N * j);
        TG c[N];
#pragma unroll
        for (int a = 0; a < N; ++a) c[a] = to_g<TG>(B.D[row * N + a]);
        const TG hlo = -to_g<TG>(B.hm[row]), hhi = to_g<TG>(B.hp[row]);
        const TG *dq = sdQ + d * 10 * Nf + r;
#pragma unroll(N == 8 ? 5 : 1)
        for (int v = v0; v < v1; ++v) {
          // Derivative along the point's line, then the two faces' correction added to the same sum.
          const TG jlo = dq[v * Nf], jhi = dq[(5 + v) * Nf];
          Dot<TG> s(c[0], sq[v * Np + at]);
#pragma unroll
          for (int a = 1; a < N; ++a) s.add(c[a], sq[v * Np + at + a * st]);
          const TG gu = s.raw();
          s.add(hlo, jlo);
          s.add(hhi, jhi);
          const TG gc = s.raw();
          if constexpr (kPack) {
            sG[(d * 5 + v) * Np + m] = df(gu.hi, gc.hi);
            sGc[gslot(d * 5 + v)] = df(gu.lo, gc.lo);
          } else {
            sG[(d * 5 + v) * Np + m] = gu;
            sGc[gslot(d * 5 + v)] = gc;
          }
        }
      }
#pragma unroll 1
      for (int v = v0; v < v1; ++v) {
        TG du[3], dc[3];
        if constexpr (kPack) {
          d2 g[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const df32 h = sG[(d * 5 + v) * Np + m], l = sGc[gslot(d * 5 + v)];
            g[d] = d2{mkf2(h.hi, h.lo), mkf2(l.hi, l.lo)};
          }
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) {
            const d2 r = dot3(sj[jj], g[0], sj[3 + jj], g[1], sj[6 + jj], g[2]);
            du[jj] = lane0(r);
            dc[jj] = lane1(r);
          }
        } else {
          TG gu[3], gc[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            gu[d] = sG[(d * 5 + v) * Np + m];
            gc[d] = sGc[gslot(d * 5 + v)];
          }
#pragma unroll
          for (int jj = 0; jj < 3; ++jj) {
            du[jj] = dot3(sj[jj], gu[0], sj[3 + jj], gu[1], sj[6 + jj], gu[2]);
            dc[jj] = dot3(sj[jj], gc[0], sj[3 + jj], gc[1], sj[6 + jj], gc[2]);
          }
        }
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) {
          sGc[gslot(jj * 5 + v)] = dc[jj];
          // Face-gradient source: BR2 the uncorrected gradient (+ eta r_f), LDG the corrected one.
          sG[(jj * 5 + v) * Np + m] = dph.ldg ? dc[jj] : du[jj];
        }
      }
      if constexpr (!SPLIT)
#pragma unroll
        for (int c = 0; c < 15; ++c) G[c] = sGc[gslot(c)];
    }
  }
  if constexpr (SPLIT) {
    __syncthreads();
    if (pt)
#pragma unroll
      for (int c = 0; c < 15; ++c) G[c] = sGc[gslot(c)];
  }
  T rho_nu = ph.zero;
  if (viscous && dph.closure) {
    // Eddy-viscosity closure: quadrature-weighted element mean of the corrected velocity
    // gradient, then one warp per element evaluates the network (BF16 weights, FP32 accumulation).
    float *red = cs.red + cs.mine * closure_floats<N>();
    if (pt) {
      const double ri = 1.0 / to_double(q[0]);
      const double w = (double)B.w[i] * B.w[j] * B.w[k] / to_double(invJ);
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const double dudx = (to_double(G[b * 5 + 1 + a]) - to_double(q[1 + a]) * ri * to_double(G[b * 5])) * ri;
          red[(a * 3 + b) * Np + m] = (float)(w * dudx);
        }
      red[9 * Np + m] = (float)w;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int l = threadIdx.x >> 5; l < cs.n; l += blockDim.x >> 5) {
      float *rl = cs.red + l * closure_floats<N>();
      float acc[10];
#pragma unroll
      for (int c = 0; c < 10; ++c) {
        float sacc = 0.f;
        for (int mm = lane; mm < Np; mm += 32) sacc += rl[c * Np + mm];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sacc += __shfl_xor_sync(0xffffffffu, sacc, o);
        acc[c] = sacc;
      }
      float x[11];
      float ss = 0.f;
#pragma unroll
      for (int c = 0; c < 9; ++c) x[c] = acc[c] / acc[9];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const float sab = 0.5f * (x[a * 3 + b] + x[b * 3 + a]);
          ss += sab * sab;
        }
      x[9] = sqrtf(2.f * ss);
      x[10] = (float)(hel[cs.e0 + l] / N);
      const float nu = closure_mlp(dph, x, rl + 10 * Np + 1, lane);
      if (lane == 0) {
        rl[10 * Np] = nu;
        if (nu_out) nu_out[cs.e0 + l] = nu;
      }
    }
    __syncthreads();
    if (pt) rho_nu = q[0] * from_double<T>((double)red[10 * Np]);
  }
  if (pt) {
    // Physical flux (symmetric momentum tensor and energy vector), then its three transforms.
    const T ri = reciprocal(q[0]);
    const T u[3] = {q[1] * ri, q[2] * ri, q[3] * ri};
    const T p = ph.gm1 * (q[4] - scale2(dot3(q[1], u[0], q[2], u[1], q[3], u[2]), 0.5f));
    T tau[6], hq[3], mom[6], en[3];
    bool formed = false;
    if constexpr (std::is_same<T, double>::value && VISC != 1)
      if (!viscous) {
        formed = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          double f[5];
          inviscid_transformed(q, u, p, S + 3 * d, f);
#pragma unroll
          for (int v = 0; v < 5; ++v) sH[(d * 5 + v) * Np + m] = f[v];
        }
      }
    if (viscous) {
      if constexpr (kPert) {
        TG qg[5], ug[3], taug[6], hqg[3];
#pragma unroll
        for (int v = 0; v < 5; ++v) qg[v] = to_g<TG>(q[v]);
        const TG rig = reciprocal(qg[0]);
#pragma unroll
        for (int c = 0; c < 3; ++c) ug[c] = qg[1 + c] * rig;
        viscous_stress<TG>(qg, ug, rig, G, phg, visc_with(phg, to_g<TG>(rho_nu), dph), taug, hqg);
#pragma unroll
        for (int a = 0; a < 3; ++a) hq[a] = from_g<T>(hqg[a]);
#pragma unroll
        for (int a = 0; a < 6; ++a) tau[a] = from_g<T>(taug[a]);
      } else {
        viscous_stress<T>(q, u, ri, G, ph, visc_with(ph, rho_nu, dph), tau, hq);
      }
    }
    if (!formed) {
      physical_flux<T>(q, u, p, viscous, tau, hq, mom, en);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        T f[5];
        transformed_flux<T>(q, mom, en, p, S + 3 * d, f);
#pragma unroll
        for (int v = 0; v < 5; ++v) sH[(d * 5 + v) * Np + m] = f[v];
      }
    }
  }
  __syncthreads();
  if (viscous && active) {
    // Gradient traces: uncorrected gradient interpolated to the face + eta * own lifting.
    // df32 and FP32: one item per (gradient component jj, line normal to a face pair), whose two end
    // points share the line's values.  FP64: one item per (jj, face point), because the FP64 pipe is the
    // bound there and 18 Nf single items fill its warps better than 9 Nf double ones (p = 4: 15 against 16
    // warp passes).
    constexpr int S = std::is_same<T, double>::value ? 1 : 2, kF = 6 / S;
    for (int t = tid; t < 3 * kF * Nf; t += nth) {
      const int jj = t / (kF * Nf), fr_ = t - jj * kF * Nf;
      const int f0 = fr_ / Nf * S, r = fr_ % Nf;
      int base, sd;
      face_line<N>(f0, r, base, sd);
      T *dst[S];
      TG lj[S];
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const int packed = ef[e * 6 + f0 + s];
        const int64_t I = packed >> 4;
        dst[s] = Gtr + (I * 2 + ((packed >> 3) & 1)) * 15 * Nf + slot_of(packed & 7, r % N, r / N, N) + jj * 5 * Nf;
        lj[s] = to_g<TG>(ph.eta * liftfac[((e * 6 + f0 + s) * 3 + jj) * Nf + r]);
      }
      const T *l0 = (S == 1 && (f0 & 1)) ? B.lp : B.lm;
      TG lg[N];
#pragma unroll
      for (int c = 0; c < N; ++c) lg[c] = to_g<TG>(l0[c]);
      if constexpr (std::is_same<TG, df32>::value) {
        // Double-float: the two ends are the lanes of packed instructions.
        d2 lc[N];
#pragma unroll
        for (int c = 0; c < N; ++c) lc[c] = pack(lg[c], lg[N - 1 - c]);
        const d2 lw = pack(lj[0], lj[S - 1]);
#pragma unroll 1
        for (int v = 0; v < 5; ++v) {
          const TG *sg = sG + (jj * 5 + v) * Np + base;
          const d2 jump = pack(sdQ[(f0 * 5 + v) * Nf + r], sdQ[((f0 + 1) * 5 + v) * Nf + r]);
          Dot<d2> acc(lc[0], dup(sg[0]));
#pragma unroll
          for (int c = 1; c < N; ++c) acc.add(lc[c], dup(sg[c * sd]));
          acc.add(lw, jump);
          const d2 g = acc.raw();
          dst[0][v * Nf] = lane0(g);
          dst[S - 1][v * Nf] = lane1(g);
        }
      } else {
#pragma unroll 1
        for (int v = 0; v < 5; ++v) {
          const TG *sg = sG + (jj * 5 + v) * Np + base;
          TG x[N];
#pragma unroll
          for (int c = 0; c < N; ++c) x[c] = sg[c * sd];
#pragma unroll
          for (int s = 0; s < S; ++s) {
            // l(+1) is l(-1) mirrored.
            auto l = [&](int c) { return s ? lg[N - 1 - c] : lg[c]; };
            const TG jump = sdQ[((f0 + s) * 5 + v) * Nf + r];
            Dot<TG> acc(l(0), x[0]);
#pragma unroll
            for (int c = 1; c < N; ++c) acc.add(l(c), x[c]);
            acc.add(lj[s], jump);
            dst[s][v * Nf] = from_g<T>(acc.raw());
          }
        }
      }
    }
  }
  if (mine) {
    T *out = Rpart + (e * Np + m) * 5;
#pragma unroll 1
    for (int v = v0; v < v1; ++v) {
      const T *h0 = sH + (0 * 5 + v) * Np, *h1 = sH + (1 * 5 + v) * Np, *h2 = sH + (2 * 5 + v) * Np;
      Dot<T> acc(B.Dt[i * N], h0[N * j + N * N * k]);
      acc.add(B.Dt[j * N], h1[i + N * N * k]);
      acc.add(B.Dt[k * N], h2[i + N * j]);
#pragma unroll
      for (int a = 1; a < N; ++a) {
        acc.add(B.Dt[i * N + a], h0[a + N * j + N * N * k]);
        acc.add(B.Dt[j * N + a], h1[i + N * a + N * N * k]);
        acc.add(B.Dt[k * N + a], h2[i + N * j + N * N * a]);
      }
      out[v] = acc.raw();
    }
  }
}

// Resident blocks per order and arithmetic, each measured (GB300).  p = 5 and 6: 3 blocks of 224 and
// (double-float) 2 of 352 threads at 80 registers, with some spills, beat the register-limited 2 and
// 1; FP64 p = 6 keeps 1 block.  Double-float at p = 2, 3, 4: 20, 10 and 5 blocks (96 registers, 8
// to 24 bytes of spills at p = 2 and 4) beat 16, 8 and 4, since the gradient holds one row of D instead of three: 40^3 p = 2 0.485 -> 0.463
// ms per launch, 40^3 p = 3 1.023 -> 0.985 ms, 48^3 p = 4 3.27 -> 3.09 ms.  With the viscous branch in FP32 the
// same counts (6 and 12 at p = 4 and 3 measure the same).
template <int N, typename T>
constexpr int volume_min_blocks_of() {
  if (std::is_same<T, double>::value) return N == 6 ? 3 : volume_min_blocks<N>();
  return N == 3 ? 20 : (N == 4 ? 10 : (N == 5 ? 5 : (N == 6 ? 3 : (N == 7 ? 2 : volume_min_blocks<N>()))));
}

// Elements per block: one, but 16 (128 threads) at p = 1, whose 8 points would fill a quarter of a warp
// (double-float 48^3: 0.89 -> 0.295 ms per launch).  At p = 2 (27 of 32 lanes) 7 elements in 192 threads or 9
// in 256 measured slower than one warp per element (FP64 with the closure 0.470 and 0.459 against 0.448 ms).
template <int N>
__host__ __device__ constexpr int volume_epb() { return N == 2 ? 16 : 1; }
// The same at p = 1 on viscous meshes up to this many elements: one element per warp, as long as such blocks (8 per
// SM) are resident at once.  A thread of the 16-element block does four times as much of the staging and the traces,
// which the idle lanes do not pay back before the SMs fill.  Volume launch, one element / 16 elements per block:
// FP64 200 elements 21.4 / 30.7 us, 800 26.5 / 30.6, 1200 31.5 / 31.0, 1600 41.2 / 30.9; with the closure 28.8 /
// 45.3, 32.9 / 45.3, 41.2 / 46.8, 48.6 / 47.4; double-float 12.5 / 16.9, 13.7 / 16.6, 14.2 / 17.1, 16.6 / 17.0; FP32
// viscous branch 10.3 / 14.8, 10.9 / 15.1, 11.5 / 15.2, 12.4 / 15.3.
constexpr int64_t kSingleMax = 8 * 152;
template <int N, int EPB = volume_epb<N>()>
__host__ __device__ constexpr int volume_block() {
  return EPB == 1 ? volume_threads<N>() : (EPB * N * N * N + 31) / 32 * 32;
}

// Euler runs (VISC = 0): 15 N^3 values of shared memory instead of 35 N^3 + 30 N^2 and no gradient
// registers, so 1024 threads per SM at 64 registers (704 at p = 6).
template <int N, typename T, int VISC, int EPB>
constexpr int volume_blocks() {
  return VISC == 0 ? (N == 7 ? 2 : (N == 3 ? 32 : 1024 / volume_block<N>()))
                   : (EPB == 16 ? 4 : volume_min_blocks_of<N, T>());
}

// Dynamic shared memory of a block.
template <int N, typename T, int EPB = volume_epb<N>()>
size_t volume_smem(bool viscous, bool closure) {
  return EPB * (viscous ? sizeof(T) * volume_smem_values<N>() + (closure ? sizeof(float) * closure_floats<N>() : 0)
                        : sizeof(T) * 15 * N * N * N);
}

// Few elements: five groups of threads per element, one per variable in the gradient and the divergence (one of
// them also forms the fluxes).  With one or two elements per SM the kernel above is a chain of one warp's
// instructions (an FP64 one issues every 64 cycles per scheduler, and the other schedulers idle): FP64
// 64 elements at p = 2 28.8 -> 16.4 us per launch, 125 at p = 3 29.3 -> 18.6, 125 at p = 4 30.7 -> 26.6;
// double-float 64 at p = 2 18.5 -> 10.4, 216 at p = 3 18.5 -> 12.3, 64 at p = 4 14.8 -> 14.5.  Limits: where the SMs
// fill up it costs an extra barrier and the four groups' idle time at the fluxes (FP64 p = 2 18.7 against
// 28.7 us at 216 elements but 34.3 against 29.2 at 512, p = 3 25.0 against 30.0 and 44.6 against 41.5, p = 4
// 47.5 against 43.6 at 216), so two elements per SM at p = 2 and 3 and one at p = 4.  p = 1 has a quarter of a warp
// per element, p >= 5 seven warps and more.
template <int N>
constexpr int64_t volume_split_max() { return N == 3 || N == 4 ? 2 * 152 : (N == 5 ? 152 : 0); }

template <int N, typename T, bool FP32V>
__global__ void __launch_bounds__(5 * volume_threads<N>())
    k_volume_split(const T *__restrict__ Q, const T *__restrict__ metrics, const int32_t *__restrict__ ef,
                   const T *__restrict__ Qtr, const T *__restrict__ liftfac, T *__restrict__ Gtr, T *__restrict__ Rpart,
                   DevPhys dph, const double *__restrict__ hel, float *__restrict__ nu_out,
                   const int8_t *__restrict__ if_up, int64_t n_interior) {
  extern __shared__ double sm_raw[];
  const ClosureSpace cs{reinterpret_cast<float *>(sm_raw + volume_smem_values<N>()), blockIdx.x, 1, 0};
  volume_body<N, T, false, FP32V, 1, true>(blockIdx.x, threadIdx.x, 5 * volume_threads<N>(), true, sm_raw, Q, metrics, ef,
                                           Qtr, liftfac, Gtr, Rpart, dph, hel, nu_out, if_up, n_interior, cs);
}

template <int N, typename T, bool FP32V, int VISC, int EPB = volume_epb<N>()>
__global__ void __launch_bounds__(volume_block<N, EPB>(), volume_blocks<N, T, VISC, EPB>())
    k_volume(const T *__restrict__ Q, const T *__restrict__ metrics, const int32_t *__restrict__ ef,
             const T *__restrict__ Qtr, const T *__restrict__ liftfac, T *__restrict__ Gtr, T *__restrict__ Rpart,
             DevPhys dph, const double *__restrict__ hel, float *__restrict__ nu_out,
             const int8_t *__restrict__ if_up, int64_t n_interior, int64_t E) {
  extern __shared__ double sm_raw[];
  constexpr int VALS = VISC == 0 ? 15 * N * N * N : volume_smem_values<N>();
  constexpr int NTH = EPB == 1 ? volume_threads<N>() : N * N * N;
  const int64_t e0 = (int64_t)blockIdx.x * EPB;
  const int le = EPB == 1 ? 0 : (int)threadIdx.x / NTH, tid = EPB == 1 ? (int)threadIdx.x : (int)threadIdx.x % NTH;
  const int n = EPB == 1 ? 1 : (int)(E - e0 < EPB ? E - e0 : EPB);
  const int mine = EPB == 1 || le < n ? le : 0;
  const ClosureSpace cs{reinterpret_cast<float *>(sm_raw + EPB * VALS), e0, n, mine};
  volume_body<N, T, false, FP32V, VISC>(e0 + mine, tid, NTH, EPB == 1 || le < n, sm_raw + mine * VALS, Q, metrics, ef,
                                        Qtr, liftfac, Gtr, Rpart, dph, hel, nu_out, if_up, n_interior, cs);
}

// ------------------------------------------------------------------------------------------
// 3. Common normal flux at the flux points of two-sided interfaces (Rusanov + BR2).  The
// inviscid part (pressure/energy recovery) is FP64 in both paths.
// ------------------------------------------------------------------------------------------
template <int N, typename T, bool FP32V, bool ROE>
__device__ __forceinline__ void iface_body(int64_t t, const T *__restrict__ Qtr, const T *__restrict__ Gtr,
                                           const T *__restrict__ normals, T *__restrict__ FI, int64_t n_if,
                                           const DevPhys &dph, const int32_t *__restrict__ if_elem,
                                           const float *__restrict__ nu, const int8_t *__restrict__ if_up) {
  constexpr int Nf = N * N;
  if (t >= n_if * Nf) return;
  const int64_t I = t / Nf;
  const int q = (int)(t % Nf);
  const PhysT<T> &ph = phys_of<T>(dph);
  T qL[5], qR[5], nT[3];
  const T nn = normals[(I * 4 + 3) * Nf + q];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    qL[v] = Qtr[(I * 2 + 0) * 5 * Nf + v * Nf + q];
    qR[v] = Qtr[(I * 2 + 1) * 5 * Nf + v * Nf + q];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) nT[c] = normals[(I * 4 + c) * Nf + q];
  T F[5];
  if constexpr (ROE) {
    double a[5], b[5], nd[3], Fd[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      a[v] = to_double(qL[v]);
      b[v] = to_double(qR[v]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) nd[c] = to_double(nT[c]);
    roe_flux(a, b, nd, to_double(nn), dph.gamma, Fd);
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = from_double<T>(Fd[v]);
  } else {
    T fL[5], fR[5], sL, sR;
    normal_inviscid(qL, nT, nn, dph, fL, sL);
    normal_inviscid(qR, nT, nn, dph, fR, sR);
    const T ms = -fmax(sL, sR);
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = scale2(muladd(fL[v] + fR[v], ms, qR[v] - qL[v]), 0.5f);
  }
  if (dph.viscous) {
    // BR2: the mean state and gradient (their sums, see viscous_normal); LDG: the supplying side's
    // solution and the other side's gradient.  FR_PREC_MIXED_VF32 forms the whole viscous part in FP32
    // (the gradient traces written by the volume kernel's FP32 branch are exact FP32 values).
    using TG = typename GradOf<T, FP32V>::type;
    const PhysT<TG> &phg = phys_of<TG>(dph);
    const int sup = (dph.ldg && if_up[I]) ? 0 : 1;
    TG qc[5], ng[3], tn[3], en;
#pragma unroll
    for (int v = 0; v < 5; ++v)
      qc[v] = dph.ldg ? to_g<TG>(sup == 0 ? qL[v] : qR[v]) : to_g<TG>(qL[v]) + to_g<TG>(qR[v]);
#pragma unroll
    for (int c = 0; c < 3; ++c) ng[c] = to_g<TG>(nT[c]);
    TG rho_nu = phg.zero;
    if (dph.closure)
      rho_nu = scale2(qc[0], dph.ldg ? 1.f : 0.5f) *
               from_double<TG>(0.5 * ((double)nu[if_elem[2 * I]] + (double)nu[if_elem[2 * I + 1]]));
    const Visc<TG> vc = visc_with(phg, rho_nu, dph);
    const T *g0 = Gtr + (I * 2 + 0) * 15 * Nf + q, *g1 = g0 + 15 * Nf;
    if (dph.ldg) {
      const T *gs = sup == 0 ? g1 : g0;
      viscous_normal<TG>(qc, [&](int c) { return to_g<TG>(gs[c * Nf]); }, ng, phg, vc, tn, en);
    } else {
      viscous_normal<TG>(qc, [&](int c) { return to_g<TG>(g0[c * Nf]) + to_g<TG>(g1[c * Nf]); }, ng, phg, vc, tn, en);
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) F[1 + v] -= from_g<T>(tn[v]);
    F[4] -= from_g<T>(en);
    if (dph.ldg) {
      const T tp = ph.tau * nn;
#pragma unroll
      for (int v = 0; v < 5; ++v) F[v] = muladd(F[v], tp, qL[v] - qR[v]);
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) FI[(I * 5 + v) * Nf + q] = F[v];
}

// 5 resident blocks of 128 threads (96 registers, no spills with the Rusanov flux; the Roe flux is an
// instantiation of its own, which would otherwise set the registers of both), 6 with the FP32 viscous
// part.  Measured at 5 / 6 blocks: double-float 48^3 p = 4 0.682 / 0.747 ms (0.691 since the FP32 to FP64
// conversions moved to the integer pipe), FP64 32^3 p = 4 0.843 / 0.857 ms, FP32 viscous 40^3 p = 3 0.231 / 0.220 ms
// (0.199 with the same conversions).  The double-float Roe instantiations spill 80 to 196 bytes.  Before the viscous flux was formed along the normal and
// the Roe branch split off: 0.869, 1.072 and 0.232 ms (memory floor 0.48 ms at 48^3; FP64 is bound by its
// pipe: 185 operations per point instead of 240, Roe 330 instead of 500).
template <bool FP32V>
constexpr int iface_blocks() { return FP32V ? 6 : 5; }

template <int N, typename T, bool FP32V, bool ROE>
__global__ void __launch_bounds__(128, iface_blocks<FP32V>())
    k_iface_flux(const T *__restrict__ Qtr, const T *__restrict__ Gtr, const T *__restrict__ normals, T *__restrict__ FI,
                 int64_t n_if, DevPhys dph, const int32_t *__restrict__ if_elem, const float *__restrict__ nu,
                 const int8_t *__restrict__ if_up) {
  iface_body<N, T, FP32V, ROE>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, Qtr, Gtr, normals, FI, n_if, dph,
                               if_elem, nu, if_up);
}

// ------------------------------------------------------------------------------------------
// 3b. Boundary faces.  Side 0 of a boundary interface is the element; its side-1 slot holds
// 2 Q^I - Q- so that the volume kernel's (other - own)/2 equals Q^I - Q- for the BR2 jump.
// Boundary states are FP64 in both paths.
// ------------------------------------------------------------------------------------------
// Ghost state (for the Rusanov flux) and boundary common solution Q^I from the interior trace.
__device__ void boundary_states(const double qm[5], const double n[3], double nn, const fr_bc &bc,
                                const DevPhys &ph, double ghost[5], double qi[5]) {
  const double g = ph.gamma, Rg = ph.R;
  const double ri = 1.0 / qm[0];
  const double u[3] = {qm[1] * ri, qm[2] * ri, qm[3] * ri};
  const double p = (g - 1.0) * (qm[4] - 0.5 * (qm[1] * u[0] + qm[2] * u[1] + qm[3] * u[2]));
  if (bc.kind == FR_BC_DIRICHLET) {
    for (int v = 0; v < 5; ++v) ghost[v] = qi[v] = bc.params[v];
    return;
  }
  if (bc.kind == FR_BC_WALL_ISOTHERMAL) {
    ghost[0] = qm[0]; ghost[1] = -qm[1]; ghost[2] = -qm[2]; ghost[3] = -qm[3]; ghost[4] = qm[4];
    qi[0] = qm[0]; qi[1] = qi[2] = qi[3] = 0.0;
    qi[4] = qm[0] * Rg * bc.params[0] / (g - 1.0);
    return;
  }
  const double nh[3] = {n[0] / nn, n[1] / nn, n[2] / nn};
  const double un = u[0] * nh[0] + u[1] * nh[1] + u[2] * nh[2];
  const double c = sqrt(g * p * ri);
  const double Rp = un + 2.0 * c / (g - 1.0);          // outgoing Riemann invariant
  double rb, ub[3], pb;
  if (bc.kind == FR_BC_CHAR_OUTFLOW) {
    pb = bc.params[0];
    const double sent = p / pow(qm[0], g);
    rb = pow(pb / sent, 1.0 / g);
    const double unb = Rp - 2.0 * sqrt(g * pb / rb) / (g - 1.0);
    for (int c3 = 0; c3 < 3; ++c3) ub[c3] = u[c3] + (unb - un) * nh[c3];
  } else {  // FR_BC_CHAR_INFLOW: total pressure, total temperature, direction
    const double p0 = bc.params[0], T0 = bc.params[1];
    double d[3] = {bc.params[2], bc.params[3], bc.params[4]};
    const double dn = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    for (int c3 = 0; c3 < 3; ++c3) d[c3] /= dn;
    const double a = nh[0] * d[0] + nh[1] * d[1] + nh[2] * d[2];
    const double k = 2.0 / (g - 1.0);
    const double A = a * a + k, B = -2.0 * a * Rp, C = Rp * Rp - k * k * g * Rg * T0;
    const double V = (-B + sqrt(B * B - 4.0 * A * C)) / (2.0 * A);
    const double cp = g * Rg / (g - 1.0);
    const double Tb = T0 - V * V / (2.0 * cp);
    pb = p0 * pow(Tb / T0, g / (g - 1.0));
    rb = pb / (Rg * Tb);
    for (int c3 = 0; c3 < 3; ++c3) ub[c3] = V * d[c3];
  }
  qi[0] = rb;
  qi[1] = rb * ub[0];
  qi[2] = rb * ub[1];
  qi[3] = rb * ub[2];
  qi[4] = pb / (g - 1.0) + 0.5 * rb * (ub[0] * ub[0] + ub[1] * ub[1] + ub[2] * ub[2]);
  for (int v = 0; v < 5; ++v) ghost[v] = qi[v];
}

template <int N, typename T>
__device__ __forceinline__ void bc_prepare_body(int64_t t, T *__restrict__ Qtr, const T *__restrict__ normals,
                                                const int32_t *__restrict__ if_bc, const fr_bc *__restrict__ bcs,
                                                int64_t first, int64_t count, const DevPhys &ph) {
  constexpr int Nf = N * N;
  if (t >= count * Nf) return;
  const int64_t I = first + t / Nf;
  const int q = (int)(t % Nf);
  double qm[5], n[3], gh[5], qi[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) qm[v] = to_double(Qtr[(I * 2 + 0) * 5 * Nf + v * Nf + q]);
#pragma unroll
  for (int c = 0; c < 3; ++c) n[c] = to_double(normals[(I * 4 + c) * Nf + q]);
  boundary_states(qm, n, to_double(normals[(I * 4 + 3) * Nf + q]), bcs[if_bc[I]], ph, gh, qi);
#pragma unroll
  for (int v = 0; v < 5; ++v) Qtr[(I * 2 + 1) * 5 * Nf + v * Nf + q] = from_double<T>(2.0 * qi[v] - qm[v]);
}

template <int N, typename T>
__global__ void k_bc_prepare(T *__restrict__ Qtr, const T *__restrict__ normals,
                             const int32_t *__restrict__ if_bc, const fr_bc *__restrict__ bcs,
                             int64_t first, int64_t count, DevPhys ph) {
  bc_prepare_body<N, T>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, Qtr, normals, if_bc, bcs, first, count, ph);
}

template <int N, typename T>
__device__ __forceinline__ void bc_flux_body(int64_t t, const T *__restrict__ Qtr, const T *__restrict__ Gtr,
                                             const T *__restrict__ normals, const int32_t *__restrict__ if_bc,
                                             const fr_bc *__restrict__ bcs, T *__restrict__ FI, int64_t first,
                                             int64_t count, const DevPhys &dph,
                                             const int32_t *__restrict__ if_elem, const float *__restrict__ nu) {
  constexpr int Nf = N * N;
  if (t >= count * Nf) return;
  const int64_t I = first + t / Nf;
  const int q = (int)(t % Nf);
  double qm[5], n[3], gh[5], qi[5];
  T nT[3];
#pragma unroll
  for (int v = 0; v < 5; ++v) qm[v] = to_double(Qtr[(I * 2 + 0) * 5 * Nf + v * Nf + q]);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    nT[c] = normals[(I * 4 + c) * Nf + q];
    n[c] = to_double(nT[c]);
  }
  const double nn = to_double(normals[(I * 4 + 3) * Nf + q]);
  boundary_states(qm, n, nn, bcs[if_bc[I]], dph, gh, qi);
  T F[5];
  if (dph.inviscid == FR_ROE) {
    double Fd[5];
    roe_flux(qm, gh, n, nn, dph.gamma, Fd);
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = from_double<T>(Fd[v]);
  } else {
    double fL[5], fR[5], sL, sR;
    normal_inviscid(qm, n, nn, dph.gamma, fL, sL);
    normal_inviscid(gh, n, nn, dph.gamma, fR, sR);
    const double lam = fmax(sL, sR);
#pragma unroll
    for (int v = 0; v < 5; ++v) F[v] = from_double<T>(0.5 * (fL[v] + fR[v]) - 0.5 * lam * (gh[v] - qm[v]));
  }
  if (dph.viscous) {
    const PhysT<T> &ph = phys_of<T>(dph);
    T qiT[5], tn[3], en;
#pragma unroll
    for (int v = 0; v < 5; ++v) qiT[v] = from_double<T>(qi[v]);
    T rho_nu = ph.zero;
    if (dph.closure) rho_nu = qiT[0] * from_double<T>((double)nu[if_elem[2 * I]]);
    const T *g0 = Gtr + (I * 2 + 0) * 15 * Nf + q;
    viscous_normal<T>(qiT, [&](int c) { return g0[c * Nf]; }, nT, ph, visc_with(ph, rho_nu, dph), tn, en);
#pragma unroll
    for (int v = 0; v < 3; ++v) F[1 + v] -= tn[v];
    F[4] -= en;
    if (dph.ldg) {
#pragma unroll
      for (int v = 0; v < 5; ++v) F[v] += from_double<T>(dph.ldg_tau * nn * (qm[v] - qi[v]));
    }
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) FI[(I * 5 + v) * Nf + q] = F[v];
}

template <int N, typename T>
__global__ void k_bc_flux(const T *__restrict__ Qtr, const T *__restrict__ Gtr, const T *__restrict__ normals,
                          const int32_t *__restrict__ if_bc, const fr_bc *__restrict__ bcs, T *__restrict__ FI,
                          int64_t first, int64_t count, DevPhys dph, const int32_t *__restrict__ if_elem,
                          const float *__restrict__ nu) {
  bc_flux_body<N, T>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, Qtr, Gtr, normals, if_bc, bcs, FI, first, count,
                     dph, if_elem, nu);
}

// ------------------------------------------------------------------------------------------
// 4. Correction by the common flux, scaling, and output / RK44 stage update (FP64).
// ------------------------------------------------------------------------------------------
// Lifted common fluxes of the six faces at point m of element e, on top of the partial residual rp (may be
// null): the bracket of Eq. 3.
template <int N, typename T, bool VC>
__device__ __forceinline__ void correct_lift(int64_t e, int m, const T *__restrict__ FI, const int32_t *__restrict__ ef,
                                             const DevPhys &dph, const T *rp, Dot<T> r[5]) {
  if (rp)
#pragma unroll
    for (int v = 0; v < 5; ++v) r[v] = Dot<T>(rp[v]);
  constexpr int Nf = N * N;
  const int i = m % N, j = (m / N) % N, k = m / (N * N);
  const BasisT<T> &B = basis_ref<N, T, VC>(dph);
  // Faces: (weight, local flux point (a, b)).
  const int fa[6] = {j, j, i, i, i, i};
  const int fb[6] = {k, k, k, k, j, j};
  const T wts[6] = {B.hm[i], B.hp[i], B.hm[j], B.hp[j], B.hm[k], B.hp[k]};
  // Double-float adds the partial residual after the faces: the xi faces come last, so that in either order
  // each direction's large pressure parts meet soon after one another.
#pragma unroll
  for (int g = 0; g < 6; ++g) {
    const int f = kGatherFirst<T> ? 5 - g : g;
    const int packed = ef[e * 6 + f];
    const int64_t I = packed >> 4;
    const int side = (packed >> 3) & 1;
    const int slot = slot_of(packed & 7, fa[f], fb[f], N);
    const T w = side ? -wts[f] : wts[f];
    const T *src = FI + I * 5 * Nf + slot;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      if (g == 0 && !rp)
        r[v] = Dot<T>(w, src[v * Nf]);
      else
        r[v].add(w, src[v * Nf]);
    }
  }
}

// Thread per point (small meshes and the batched stage).
template <int N, typename T, bool VC = false>
__device__ __forceinline__ void correct_body(int64_t t, const T *__restrict__ Rpart, const T *__restrict__ FI,
                                             const int32_t *__restrict__ ef, const T *__restrict__ metrics,
                                             int64_t E, const StageCoef &sc, double *__restrict__ Rout,
                                             double *__restrict__ Q, T *__restrict__ Qc, double *__restrict__ Un,
                                             T *__restrict__ Unc, double *__restrict__ acc, int *__restrict__ flag,
                                             const DevPhys &dph) {
  constexpr int Np = N * N * N;
  if (t >= E * Np) return;
  const int64_t e = t / Np;
  const int m = (int)(t % Np);
  Dot<T> r[5];
  correct_lift<N, T, VC>(e, m, FI, ef, dph, kGatherFirst<T> ? nullptr : Rpart + t * 5, r);
  T rv[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    if constexpr (kGatherFirst<T>) r[v].plus(Rpart[t * 5 + v]);
    rv[v] = r[v].get();
  }
  finish_point<T>(t, rv, -metrics[(e * 10 + 9) * Np + m], sc, Rout, Q, Qc, Un, Unc, acc, flag, dph);
}

// Up to 256 points per SM (one block of the kernel below on each): one thread per point in blocks of one
// warp, which spreads the chain of loads and FP64 instructions over more schedulers and has no
// staging barriers.  FP64 8^3 p = 3 12.6 -> 10.6 us per launch, 4^3 p = 2 10.4 -> 8.6, double-float 8^3 p = 3 10.9 ->
// 9.3; at 64000 points 14.4 against 14.7 us, and at 32^3 p = 4 0.398 ms staged against 0.431.
constexpr int64_t kCorrectPointMax = 152 * 256;

template <int N, typename T, bool VC>
__global__ void __launch_bounds__(32)
    k_correct_point(const T *__restrict__ Rpart, const T *__restrict__ FI, const int32_t *__restrict__ ef,
                    const T *__restrict__ metrics, int64_t E, StageCoef sc, double *__restrict__ Rout,
                    double *__restrict__ Q, T *__restrict__ Qc, double *__restrict__ Un, T *__restrict__ Unc,
                    double *__restrict__ acc, int *__restrict__ flag, DevPhys dph) {
  correct_body<N, T, VC>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, Rpart, FI, ef, metrics, E, sc, Rout, Q, Qc, Un,
                         Unc, acc, flag, dph);
}

template <int N, typename T, bool VC, bool SRC>
__global__ void __launch_bounds__(kCorrectThreads, std::is_same<T, double>::value ? 6 : 5)
    k_correct(const T *__restrict__ Rpart, const T *__restrict__ FI, const int32_t *__restrict__ ef,
              const T *__restrict__ metrics, int64_t E, StageCoef sc, double *__restrict__ Rout, double *__restrict__ Q,
              T *__restrict__ Qc, double *__restrict__ Un, T *__restrict__ Unc, double *__restrict__ acc,
              int *__restrict__ flag, DevPhys dph) {
  extern __shared__ double sm_raw[];
  constexpr int Np = N * N * N;
  const CorrectSmem sm(sm_raw);
  const int64_t first = (int64_t)blockIdx.x * kCorrectThreads;
  const int n = (int)(E * Np - first < kCorrectThreads ? E * Np - first : kCorrectThreads);
  const StageIn in = stage_inputs<T>(sc, Q, Un, Unc, acc);
  stage_begin<T>(sm, Rpart + first * 5, first * 5, n, in);
  Dot<T> r[5];
  T s{};
  if constexpr (!kGatherFirst<T>) stage_arrive();
  if ((int)threadIdx.x < n) {
    const int64_t t = first + threadIdx.x, e = t / Np;
    const int m = (int)(t % Np);
    correct_lift<N, T, VC>(e, m, FI, ef, dph,
                           kGatherFirst<T> ? nullptr : reinterpret_cast<const T *>(sm.r) + threadIdx.x * 5, r);
    s = -metrics[(e * 10 + 9) * Np + m];
  }
  finish_block<T, SRC>(first, n, sm, r, nullptr, s, sc, in, Rout, Q, Qc, Un, Unc, acc, flag, dph);
}

// Meshes with prisms: a triangular interface uses only the first N(N+1)/2 of its N^2 slots;
// these wrappers skip the others before running the interface bodies.
template <int N>
__device__ __forceinline__ bool unused_tri_slot(int64_t t, int64_t first, int64_t count, const int8_t *if_tri) {
  constexpr int Nf = N * N, Nt = N * (N + 1) / 2;
  if (t >= count * Nf) return false;     // out of range: the body's own bound check returns
  return if_tri[first + t / Nf] && (int)(t % Nf) >= Nt;
}

template <int N, typename T, bool ROE>
__global__ void __launch_bounds__(128, iface_blocks<false>())
    k_iface_flux_tri(const T *__restrict__ Qtr, const T *__restrict__ Gtr, const T *__restrict__ normals,
                     T *__restrict__ FI, int64_t n_if, DevPhys dph, const int32_t *__restrict__ if_elem,
                     const float *__restrict__ nu, const int8_t *__restrict__ if_tri, const int8_t *__restrict__ if_up) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (unused_tri_slot<N>(t, 0, n_if, if_tri)) return;
  iface_body<N, T, false, ROE>(t, Qtr, Gtr, normals, FI, n_if, dph, if_elem, nu, if_up);
}

template <int N, typename T>
__global__ void k_bc_prepare_tri(T *__restrict__ Qtr, const T *__restrict__ normals, const int32_t *__restrict__ if_bc,
                                 const fr_bc *__restrict__ bcs, int64_t first, int64_t count, DevPhys ph,
                                 const int8_t *__restrict__ if_tri) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (unused_tri_slot<N>(t, first, count, if_tri)) return;
  bc_prepare_body<N, T>(t, Qtr, normals, if_bc, bcs, first, count, ph);
}

template <int N, typename T>
__global__ void k_bc_flux_tri(const T *__restrict__ Qtr, const T *__restrict__ Gtr, const T *__restrict__ normals,
                              const int32_t *__restrict__ if_bc, const fr_bc *__restrict__ bcs, T *__restrict__ FI,
                              int64_t first, int64_t count, DevPhys dph, const int32_t *__restrict__ if_elem,
                              const float *__restrict__ nu, const int8_t *__restrict__ if_tri) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (unused_tri_slot<N>(t, first, count, if_tri)) return;
  bc_flux_body<N, T>(t, Qtr, Gtr, normals, if_bc, bcs, FI, first, count, dph, if_elem, nu);
}

// ------------------------------------------------------------------------------------------
// Batched persistent stage: one cooperative launch runs every phase of one RK stage for all
// cases of a ragged ensemble.  Phases are separated by a grid barrier whose waits are bounded:
// a wait that exceeds the spin limit sets the error word and every block returns.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ bool batch_grid_sync(BatchSync *sy, long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned *gen = &sy->bar_gen;
    volatile int *err = &sy->err;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(&sy->bar_count, 1u) == gridDim.x - 1) {
      atomicExch(&sy->bar_count, 0u);
      __threadfence();
      atomicAdd(&sy->bar_gen, 1u);
    } else {
      long long it = 0;
      while (*gen == g) {
        if (*err) break;
        if (++it > limit) {
          atomicExch(&sy->err, 1);
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *(volatile int *)&sy->err == 0;
}

template <typename T, int N>
__device__ __forceinline__ void batch_task(const BatchTask &tk, const BatchCase &c, const BatchLaunch &L,
                                           double *smem) {
  const DevMesh &m = c.m;
  const T *Qin = reinterpret_cast<const T *>(m.mixed ? m.Qc : m.Q);
  T *Qtr = reinterpret_cast<T *>(m.Qtr), *Gtr = reinterpret_cast<T *>(m.Gtr), *FI = reinterpret_cast<T *>(m.FI);
  T *Rpart = reinterpret_cast<T *>(m.Rpart);
  const T *met = reinterpret_cast<const T *>(m.metrics), *lift = reinterpret_cast<const T *>(m.liftfac);
  const T *nrm = reinterpret_cast<const T *>(m.normals);
  const int64_t pts = m.E * m.Np * 5;               // first prism value in per-point arrays
  const T *ptab = reinterpret_cast<const T *>(m.ptab), *pmet = reinterpret_cast<const T *>(m.metrics_p);
  const int64_t idx = tk.begin + threadIdx.x < tk.end ? tk.begin + threadIdx.x : (int64_t)1 << 62;
  switch (tk.kind) {
    case TASK_INTERP:
      interp_body<N, T>(tk.begin + threadIdx.x < tk.end ? tk.begin + threadIdx.x : (int64_t)1 << 62, Qin, m.ef, Qtr,
                        m.E);
      break;
    case TASK_BC_PREPARE:
      if (m.if_tri && unused_tri_slot<N>(idx, m.n_interior, m.n_if - m.n_interior, m.if_tri)) break;
      bc_prepare_body<N, T>(idx, Qtr, nrm, m.if_bc, m.bcs, m.n_interior, m.n_if - m.n_interior, c.ph);
      break;
    case TASK_VOLUME: {
      // Sub-blocks of nth threads, one element each; threads past the last full sub-block idle.
      const int tpe = ((N * N * N + 31) / 32) * 32;
      const int nth = tpe >= (int)blockDim.x ? (int)blockDim.x : tpe;
      const int epb = batch_elems_per_block(N, (int)blockDim.x);
      const int le = (int)threadIdx.x / nth;
      const int tid = (int)threadIdx.x % nth;
      const int64_t e = tk.begin + le;
      const bool active = le < epb && e < tk.end;
      volume_body<N, T, false, false, 2>(e, tid, nth, active, smem + (size_t)(le < epb ? le : 0) * volume_smem_values<N>(),
                                         Qin, met, m.ef, Qtr, lift, Gtr, Rpart, c.ph, m.h, nullptr, m.if_up, m.n_interior,
                                         ClosureSpace{nullptr, 0, 0, 0});
      break;
    }
    case TASK_IFACE:
      if (m.if_tri && unused_tri_slot<N>(idx, 0, m.n_interior, m.if_tri)) break;
      if (c.ph.inviscid == FR_ROE)
        iface_body<N, T, false, true>(idx, Qtr, Gtr, nrm, FI, m.n_interior, c.ph, m.if_elem, m.nu, m.if_up);
      else
        iface_body<N, T, false, false>(idx, Qtr, Gtr, nrm, FI, m.n_interior, c.ph, m.if_elem, m.nu, m.if_up);
      break;
    case TASK_BC_FLUX:
      if (m.if_tri && unused_tri_slot<N>(idx, m.n_interior, m.n_if - m.n_interior, m.if_tri)) break;
      bc_flux_body<N, T>(idx, Qtr, Gtr, nrm, m.if_bc, m.bcs, FI, m.n_interior, m.n_if - m.n_interior, c.ph, m.if_elem,
                         m.nu);
      break;
    case TASK_PRISM_INTERP:
      prism_interp_body<N, T>(idx, Qin + pts, m.ef_p, ptab, m.tri_slot, Qtr, m.Ep);
      break;
    case TASK_PRISM_VOLUME: {
      const int tpe = ((N * (N + 1) / 2 * N + 31) / 32) * 32;
      const int nth = tpe >= (int)blockDim.x ? (int)blockDim.x : tpe;
      const int epb = batch_prism_elems_per_block(N, (int)blockDim.x);
      const int le = (int)threadIdx.x / nth;
      const int tid = (int)threadIdx.x % nth;
      const int64_t e = tk.begin + le;
      const bool active = le < epb && e < tk.end;
      prism_volume_body<N, T>(e, tid, nth, active, smem + (size_t)(le < epb ? le : 0) * prism_smem_values<N>(),
                              Qin + pts, pmet, m.ef_p, Qtr, ptab, m.tri_slot, Gtr, Rpart + pts, c.ph, m.if_up,
                              m.n_interior);
      break;
    }
    case TASK_PRISM_CORRECT:
      prism_correct_body<N, T>(idx, Rpart + pts, FI, m.ef_p, pmet, ptab, m.tri_slot, m.Ep, m.E * m.Np,
                               stage_coef(MODE_RK, L.stage, L.dts[tk.cs]), nullptr, m.Q,
                               m.mixed ? reinterpret_cast<T *>(m.Qc) : nullptr, m.Un, reinterpret_cast<T *>(m.Unc), m.acc,
                               &L.sync->nonfinite, c.ph);
      break;
    case TASK_CORRECT:
      correct_body<N, T>(tk.begin + threadIdx.x < tk.end ? tk.begin + threadIdx.x : (int64_t)1 << 62, Rpart, FI, m.ef,
                         met, m.E, stage_coef(MODE_RK, L.stage, L.dts[tk.cs]), nullptr, m.Q,
                         m.mixed ? reinterpret_cast<T *>(m.Qc) : nullptr, m.Un, reinterpret_cast<T *>(m.Unc), m.acc,
                         &L.sync->nonfinite, c.ph);
      break;
  }
}

template <typename T, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1) k_batch_stage(BatchLaunch L) {
  extern __shared__ double smem[];
  __shared__ int s_task;
  if (L.debug_skip_block == (int)blockIdx.x) return;     // never arrives: the others time out
  for (int ph = 0; ph < L.n_phases; ++ph) {
    if (ph > 0 && !batch_grid_sync(L.sync, L.spin_limit)) return;
    const int t0 = L.phase_begin[ph], t1 = L.phase_begin[ph + 1];
    while (true) {
      __syncthreads();
      if (threadIdx.x == 0) s_task = t0 + (int)atomicAdd(&L.sync->counters[ph], 1u);
      __syncthreads();
      const int ti = s_task;
      if (ti >= t1) break;
      const BatchTask tk = L.tasks[ti];
      const BatchCase &c = L.cases[tk.cs];
      switch (c.m.N) {
        case 2: batch_task<T, 2>(tk, c, L, smem); break;
        case 3: batch_task<T, 3>(tk, c, L, smem); break;
        case 4: batch_task<T, 4>(tk, c, L, smem); break;
        case 5: batch_task<T, 5>(tk, c, L, smem); break;
        case 6: batch_task<T, 6>(tk, c, L, smem); break;
        case 7: if (BLOCK >= 352) batch_task<T, 7>(tk, c, L, smem); break;
        case 8: if (BLOCK >= 512) batch_task<T, 8>(tk, c, L, smem); break;
      }
    }
  }
}

}  // namespace
}  // namespace frx
