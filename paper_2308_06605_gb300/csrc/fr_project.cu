// Projection of a solution between orders (include/fr.h, fr_project_state).  The paper starts its
// runs at low order and switches to a higher one; the state is carried over by the L2 projection
// onto the target space in reference coordinates: Legendre modal coefficients on each hexahedron
// axis (truncated or zero-padded), the orthonormal triangle modes times Legendre on the prism.
// FP64, one axis at a time through shared memory, operators from the host as kernel parameters.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "fr_device.hpp"

namespace frx {
namespace {

// [q+1][p+1]: the line transfer through the Gauss points, with the exact discrete orthogonality
// of the Legendre polynomials on the order-p Gauss rule (c_k = (2k+1)/2 sum_j w_j P_k(x_j) f_j).
void line_transfer(int p, int q, std::vector<double> &T) {
  const Basis1D bp = make_basis(p), bq = make_basis(q);
  const int m = (p < q ? p : q) + 1;
  auto legendre = [](long double x, int n, long double *P) {
    P[0] = 1.0L;
    if (n > 0) P[1] = x;
    for (int k = 1; k < n; ++k) P[k + 1] = ((2 * k + 1) * x * P[k] - k * P[k - 1]) / (k + 1);
  };
  T.assign((size_t)(q + 1) * (p + 1), 0.0);
  long double Pp[kMaxN + 1], Pq[kMaxN + 1];
  for (int i = 0; i <= q; ++i) {
    legendre((long double)bq.x[i], kMaxN, Pq);
    for (int j = 0; j <= p; ++j) {
      legendre((long double)bp.x[j], kMaxN, Pp);
      long double acc = 0.0L;
      for (int k = 0; k < m; ++k) acc += Pq[k] * (2 * k + 1) / 2.0L * (long double)bp.w[j] * Pp[k];
      T[(size_t)i * (p + 1) + j] = (double)acc;
    }
  }
}

// Operators of one projection, passed by value as a kernel parameter (no device allocation or copy).
struct LineOp {
  double L[kMaxN * kMaxN];                          // [Nd][Ns]
};
constexpr int kMaxNt = kMaxN * (kMaxN + 1) / 2;
struct PrismOp {
  double L[kMaxN * kMaxN], T[kMaxNt * kMaxNt];      // line [Nd][Ns], triangle [Ntd][Nts]
};

// The projected state starts a new step: Q and U_n, and on the mixed path their double-float copies.
struct StateOut {
  double *Q, *Un;
  df32 *Qc, *Unc;                                   // null on the FP64 path
  __device__ __forceinline__ void put(int64_t o, double x) const {
    Q[o] = x;
    Un[o] = x;
    if (Qc) Qc[o] = Unc[o] = df_from(x);
  }
};

// One axis of ns -> ND values: item = lo + INNER (i + ND o), lo running over the values in front of the
// axis (variables and faster axes), o over those behind it; in has the axis at c INNER within blocks of
// ns INNER.  The target size is a template parameter, so the index arithmetic divides by constants.
template <int ND, int INNER>
__device__ __forceinline__ double along(const double *M, const double *in, int item, int ns) {
  const int lo = item % INNER, r = item / INNER, i = r % ND, o = r / ND;
  const double *x = in + o * ns * INNER + lo, *w = M + i * ns;
  double acc = w[0] * x[0];
  for (int c = 1; c < ns; ++c) acc = fma(w[c], x[c * INNER], acc);
  return acc;
}

constexpr int kProjectThreads = 256;

// Hexahedra, epb elements per block, one axis after the other through shared memory: out(i, j, k) =
// sum_c L[k][c] sum_b L[j][b] sum_a L[i][a] in(a, b, c).  Bound by the FP64 pipe and then by memory: the
// direct triple sum takes 160 operations per target point at p = 2 -> 4, the three passes 30.  GB300, 32^3
// elements p = 2 -> 4, set_state of the source and the call: 1.30 ms with the triple sum, device allocations
// for the operators and the registers set by further copies, 0.37 ms now, of which this kernel takes 0.30.
template <int Nd>
__global__ void __launch_bounds__(kProjectThreads)
    k_project_hex(const double *__restrict__ src, StateOut out, const __grid_constant__ LineOp op, int64_t E, int Ns,
                  int epb) {
  extern __shared__ double sm[];
  __shared__ double L[kMaxN * kMaxN];
  const int n0 = Ns * Ns * Ns * 5, n1 = Nd * Ns * Ns * 5, n2 = Nd * Nd * Ns * 5, n3 = Nd * Nd * Nd * 5;
  const int64_t e0 = (int64_t)blockIdx.x * epb;
  const int ne = (int)(E - e0 < epb ? E - e0 : epb);
  double *a = sm, *b = sm + (size_t)epb * (n0 > n2 ? n0 : n2);
  for (int i = threadIdx.x; i < Ns * Nd; i += kProjectThreads) L[i] = op.L[i];
  for (int i = threadIdx.x; i < ne * n0; i += kProjectThreads) a[i] = src[e0 * n0 + i];
  __syncthreads();
  for (int i = threadIdx.x; i < ne * n1; i += kProjectThreads) b[i] = along<Nd, 5>(L, a, i, Ns);
  __syncthreads();
  for (int i = threadIdx.x; i < ne * n2; i += kProjectThreads) a[i] = along<Nd, 5 * Nd>(L, b, i, Ns);
  __syncthreads();
  for (int i = threadIdx.x; i < ne * n3; i += kProjectThreads)
    out.put(e0 * n3 + i, along<Nd, 5 * Nd * Nd>(L, a, i, Ns));
}

// Prisms: out(t, k) = sum_c L[k][c] sum_s T[t][s] in(s, c).
template <int Nd>
__global__ void __launch_bounds__(kProjectThreads)
    k_project_prism(const double *__restrict__ src, StateOut out, const __grid_constant__ PrismOp op, int64_t E, int Ns,
                    int epb) {
  extern __shared__ double sm[];
  constexpr int Ntd = Nd * (Nd + 1) / 2;
  const int Nts = Ns * (Ns + 1) / 2;
  const int n0 = Nts * Ns * 5, n1 = Ntd * Ns * 5, n2 = Ntd * Nd * 5;
  const int64_t e0 = (int64_t)blockIdx.x * epb;
  const int ne = (int)(E - e0 < epb ? E - e0 : epb);
  double *T = sm, *L = T + Nts * Ntd, *a = L + Ns * Nd, *b = a + (size_t)epb * n0;
  for (int i = threadIdx.x; i < Ns * Nd; i += kProjectThreads) L[i] = op.L[i];
  for (int i = threadIdx.x; i < Nts * Ntd; i += kProjectThreads) T[i] = op.T[i];
  for (int i = threadIdx.x; i < ne * n0; i += kProjectThreads) a[i] = src[e0 * n0 + i];
  __syncthreads();
  for (int i = threadIdx.x; i < ne * n1; i += kProjectThreads) b[i] = along<Ntd, 5>(T, a, i, Nts);
  __syncthreads();
  for (int i = threadIdx.x; i < ne * n2; i += kProjectThreads)
    out.put(e0 * n2 + i, along<Nd, 5 * Ntd>(L, b, i, Ns));
}

// Elements per block: about four items per thread at the larger of the two orders.
constexpr int project_epb(int values) { return std::min(16, std::max(1, 4 * kProjectThreads / values)); }

// Shared memory of a block of k_project_prism from Ns to Nd points per line.
constexpr size_t project_prism_smem(int Ns, int Nd) {
  const int Nts = Ns * (Ns + 1) / 2, Ntd = Nd * (Nd + 1) / 2;
  const int epb = project_epb(std::max(Nts * Ns, Ntd * Nd) * 5);
  return sizeof(double) * ((size_t)Nts * Ntd + Ns * Nd + 5 * (size_t)epb * Ns * (Nts + Ntd));
}
// No pair of orders needs more than the 48 KB that a launch may ask for without raising the kernel's limit, which
// two threads' calls would set to different sizes.
constexpr size_t project_prism_smem_max() {
  size_t most = 0;
  for (int s = 2; s <= kMaxN; ++s)
    for (int d = 2; d <= kMaxN; ++d) most = std::max(most, project_prism_smem(s, d));
  return most;
}
static_assert(project_prism_smem_max() <= 48 * 1024, "k_project_prism launches without a raised limit");

template <int Nd>
cudaError_t launch_project(const DevMesh &a, const DevMesh &b, const std::vector<double> &L,
                           const std::vector<double> &Tt, cudaStream_t st) {
  df32 *Qc = b.mixed ? reinterpret_cast<df32 *>(b.Qc) : nullptr;
  df32 *Unc = b.mixed ? reinterpret_cast<df32 *>(b.Unc) : nullptr;
  if (a.E > 0) {
    LineOp op;
    std::memcpy(op.L, L.data(), L.size() * sizeof(double));
    const int epb = project_epb(std::max(a.Np, b.Np) * 5);
    const size_t n0 = (size_t)a.Np, n1 = (size_t)b.N * a.N * a.N, n2 = (size_t)b.N * b.N * a.N;
    const size_t smem = sizeof(double) * 5 * epb * (std::max(n0, n2) + n1);
    k_project_hex<Nd><<<(unsigned)((a.E + epb - 1) / epb), kProjectThreads, smem, st>>>(
        a.Q, StateOut{b.Q, b.Un, Qc, Unc}, op, a.E, a.N, epb);
  }
  if (a.Ep > 0) {
    PrismOp op;
    std::memcpy(op.L, L.data(), L.size() * sizeof(double));
    std::memcpy(op.T, Tt.data(), Tt.size() * sizeof(double));
    const int epb = project_epb(std::max(a.Npp, b.Npp) * 5);
    const size_t smem = project_prism_smem(a.N, b.N);
    const int64_t os = a.E * a.Np * 5, od = b.E * b.Np * 5;
    k_project_prism<Nd><<<(unsigned)((a.Ep + epb - 1) / epb), kProjectThreads, smem, st>>>(
        a.Q + os, StateOut{b.Q + od, b.Un + od, Qc ? Qc + od : nullptr, Unc ? Unc + od : nullptr}, op, a.Ep, a.N, epb);
  }
  return cudaGetLastError();
}

}  // namespace
}  // namespace frx

using namespace frx;

extern "C" fr_status fr_transfer_matrix(int32_t kind, int32_t p, int32_t q, double *T) {
  if (!T || p < 1 || p > 7 || q < 1 || q > 7 || (kind != 0 && kind != 1)) return FR_EINVAL;
  std::vector<double> M;
  if (kind == 0)
    line_transfer(p, q, M);
  else if (!tri_transfer(p, q, M))
    return FR_EINVAL;
  for (size_t i = 0; i < M.size(); ++i) T[i] = M[i];
  return FR_OK;
}

extern "C" fr_status fr_project_state(fr_mesh *src, fr_mesh *dst) {
  DevMesh a, b;
  DevPhys pa, pb;
  cudaStream_t sa, sb;
  int da = 0, db = 0;
  fr_status st = frx_mesh_view(src, &a, &pa, &sa, &da);
  if (st != FR_OK) return st;
  st = frx_mesh_view(dst, &b, &pb, &sb, &db);
  if (st != FR_OK) return st;
  if (da != db) return frx_mesh_fail(dst, FR_EINVAL, "fr_project_state: meshes on different devices");
  if (a.E != b.E || a.Ep != b.Ep)
    return frx_mesh_fail(dst, FR_EINVAL, "fr_project_state: the meshes must have the same elements");
  std::vector<double> L, Tt;
  line_transfer(a.p, b.p, L);
  if (a.Ep > 0 && !tri_transfer(a.p, b.p, Tt))
    return frx_mesh_fail(dst, FR_EMESH, "fr_project_state: triangle transfer failed");
  cudaError_t e = sa == sb ? cudaSuccess : cudaStreamSynchronize(sa);   // the source state is complete
  if (e == cudaSuccess) {
    switch (b.N) {
      case 2: e = launch_project<2>(a, b, L, Tt, sb); break;
      case 3: e = launch_project<3>(a, b, L, Tt, sb); break;
      case 4: e = launch_project<4>(a, b, L, Tt, sb); break;
      case 5: e = launch_project<5>(a, b, L, Tt, sb); break;
      case 6: e = launch_project<6>(a, b, L, Tt, sb); break;
      case 7: e = launch_project<7>(a, b, L, Tt, sb); break;
      case 8: e = launch_project<8>(a, b, L, Tt, sb); break;
      default: e = cudaErrorInvalidValue;
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(sb);
  if (e != cudaSuccess) return frx_mesh_fail(dst, FR_ECUDA, std::string("fr_project_state: ") + cudaGetErrorString(e));
  return FR_OK;
}
