// Pseudofermion force of the temporally preconditioned operator: the link outer products.
//
// S = phi^dag (M-hat^dag M-hat)^-1 phi, X = (M-hat^dag M-hat)^-1 phi, Y = M-hat X and
// dS = -2 Re(Y^dag dM-hat X) with M-hat = 1 - gamma_f^-2 C_L^o D^oe C_R^e C_L^e D^eo C_R^o
// (§II.B, Eq. TPrecFull; the paper defers the HMC force to later work, §IV). The host
// builds the right chain v_k and the left chain w_k (applications of C_L, C_R, D_s and their
// adjoints); these kernels turn pairs of chain vectors into, per link, the 3x3 matrix Z with
// dS/d eps_a = 2 gamma_f^-2 Re Tr[i T_a Z] for U -> exp(i eps T_a) U, T_a = lambda_a / 2:
//   temporal link U_t(t) of a line, from a C_L factor (pair a, b: P_- halves) and a C_R factor
//   (pair c, e: P_+ halves):
//     Z = s(t) sum_{P_- spins} (U_t(t) b(t+1)) a(t)^dag - s(t) sum_{P_+ spins} e(t) (U_t(t) c(t+1))^dag
//   spatial link U_k(x), from the two D_s factors:
//     Z = sum_spins (U_k v(x+k)) (P^-_k w(x))^dag - v'(x) (U_k P^+_k w'(x+k))^dag
// In the axial frame the kernels work with the rotated links and return Z to the caller's
// gauge with the rotation of the link's base site: Z <- g(x)^dag Z g(x).
#include "wf_internal.h"
#include "wf_line.cuh"

namespace wf {


__device__ __forceinline__ Vec3<double> fvec(const Cx<double>* f, size_t line_base, int comp0, int tp, int sl) {
  return ldvec(f + line_base + (size_t)comp0 * tp, tp, sl);
}

// acc += x y^dag
__device__ __forceinline__ void outer_acc(Mat3<double>& Z, const Vec3<double>& x, const Vec3<double>& y) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Z.e[3 * i + j] = cfmaconj(Z.e[3 * i + j], y.c[j], x.c[i]);  // x_i conj(y_j)
}

// F^a = coef Re Tr[i T_a Z] = -coef Im Tr[T_a Z], T_a = lambda_a / 2 (Gell-Mann)
__device__ __forceinline__ void project(const Mat3<double>& Z, double coef, double* out) {
  const Cx<double>* z = Z.e;
  auto im = [](Cx<double> v) { return v.im; };
  auto re = [](Cx<double> v) { return v.re; };
  // Tr[T_a Z] for the eight generators; only the imaginary part of i * (.) is needed
  const double t1 = im(z[3] + z[1]) * 0.5;
  const double t2 = (re(z[1]) - re(z[3])) * 0.5;   // Im((-i z10 + i z01)/2)
  const double t3 = im(z[0] - z[4]) * 0.5;
  const double t4 = im(z[6] + z[2]) * 0.5;
  const double t5 = (re(z[2]) - re(z[6])) * 0.5;
  const double t6 = im(z[7] + z[5]) * 0.5;
  const double t7 = (re(z[5]) - re(z[7])) * 0.5;
  const double t8 = (im(z[0]) + im(z[4]) - 2.0 * im(z[8])) / (2.0 * sqrt(3.0));
  out[0] = -coef * t1;
  out[1] = -coef * t2;
  out[2] = -coef * t3;
  out[3] = -coef * t4;
  out[4] = -coef * t5;
  out[5] = -coef * t6;
  out[6] = -coef * t7;
  out[7] = -coef * t8;
}

__device__ __forceinline__ Mat3<double> to_caller_gauge(const Mat3<double>& Z, const ForceArgs& A, int l, int sl) {
  if (!A.axial) return Z;
  const Mat3<double> G = ldmat(A.ut + (size_t)l * 9 * A.g.tp, A.g.tp, sl);
  return matmul(dagger(G), matmul(Z, G));
}

__device__ __forceinline__ size_t lex_site(const Geom& g, int x, int y, int z, int t) {
  return (size_t)x + g.L * ((size_t)y + g.L * ((size_t)z + (size_t)g.L * t));
}

__device__ __forceinline__ Mat3<double> force_temporal(const ForceArgs& A, int l, int t, int sl) {
  const Geom& g = A.g;
  const int tp = g.tp;
  const int tn = t == g.T - 1 ? 0 : t + 1;
  const int sln = slot_of(g, tn);
  const double sg = t == g.T - 1 ? A.bc : 1.0;
  const size_t lb = (size_t)l * NSPIN_C * tp;
  Mat3<double> U;
  bool unit = false;
  if (A.axial) {
    if (t == g.T - 1)
      U = ldmat(A.pl + (size_t)l * 9, 1, 0);
    else
      unit = true;
  } else {
    U = ldmat(A.ut + (size_t)l * 9 * tp, tp, sl);
  }
  Mat3<double> Zl, Zr;
#pragma unroll
  for (int k = 0; k < 9; ++k) Zl.e[k] = Zr.e[k] = czero<double>();
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    // C_L factor: spins 2, 3 (P_-)
    const Vec3<double> bn = fvec(A.b, lb, 6 + 3 * s, tp, sln);
    outer_acc(Zl, unit ? bn : matvec(U, bn), fvec(A.a, lb, 6 + 3 * s, tp, sl));
    // C_R factor: spins 0, 1 (P_+)
    const Vec3<double> cn = fvec(A.c, lb, 3 * s, tp, sln);
    outer_acc(Zr, fvec(A.e, lb, 3 * s, tp, sl), unit ? cn : matvec(U, cn));
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) Zl.e[k] = sg * (Zl.e[k] - Zr.e[k]);
  return Zl;
}

// upper components of u +- i sigma_k d (sg = 1, -1), the rest of (1 -+ gamma_k) psi following from them
__device__ __forceinline__ void half_of(const Cx<double>* f, size_t lb, int tp, int sl, int k, double sg, Vec3<double> (&h)[2]) {
  isigma(k, fvec(f, lb, 6, tp, sl), fvec(f, lb, 9, tp, sl), h[0], h[1]);
#pragma unroll
  for (int s = 0; s < 2; ++s) h[s] = vaxpy(sg, h[s], fvec(f, lb, 3 * s, tp, sl));
}

// sum_spins x (P y)^dag = 1/2 sum_{two spins} h_x h_y^dag for a projector P = (1 -+ gamma_k) / 2 (the lower
// spins are a unitary matrix times the upper ones)
__device__ __forceinline__ Mat3<double> force_spatial(const ForceArgs& A, int l, int sl, int k) {
  const Geom& g = A.g;
  const int tp = g.tp;
  int nb[6];
  neighbour_lines(g, A.parity, l, nb);
  const size_t lb = (size_t)l * NSPIN_C * tp, nbb = (size_t)nb[2 * k] * NSPIN_C * tp;
  const Mat3<double> U = ldmat(A.us_p + ((size_t)k * g.Nl + l) * NLINK_C * tp, tp, sl);
  Mat3<double> Z, Zr;
#pragma unroll
  for (int e = 0; e < 9; ++e) Z.e[e] = Zr.e[e] = czero<double>();
  Vec3<double> x[2], y[2];
  half_of(A.v, nbb, tp, sl, k, 1.0, x);
  half_of(A.w, lb, tp, sl, k, 1.0, y);
#pragma unroll
  for (int s = 0; s < 2; ++s) outer_acc(Z, matvec(U, x[s]), y[s]);
  half_of(A.vr, lb, tp, sl, k, -1.0, x);
  half_of(A.wr, nbb, tp, sl, k, -1.0, y);
#pragma unroll
  for (int s = 0; s < 2; ++s) outer_acc(Zr, x[s], matvec(U, y[s]));
#pragma unroll
  for (int e = 0; e < 9; ++e) Z.e[e] = 0.5 * (Z.e[e] - Zr.e[e]);
  return Z;
}

struct ForcePair {
  ForceArgs p[2];
};
// One thread per link: blockIdx.y its direction (3: temporal), blockIdx.z its base site's parity. Bound by
// latency and the FP64 pipe (8^3 x 32: 88 us; one thread per site and parity, with all four spins of the
// projected spinors, took 274 for the two parities)
__global__ void __launch_bounds__(64) k_force(const ForcePair F) {
  const ForceArgs& A = F.p[blockIdx.z];
  const Geom& g = A.g;
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= (size_t)g.Nl * g.T) return;
  const int t = (int)(i % g.T), l = (int)(i / g.T), mu = blockIdx.y;
  const int sl = slot_of(g, t);
  const Mat3<double> Z = to_caller_gauge(mu == 3 ? force_temporal(A, l, t, sl) : force_spatial(A, l, sl, mu), A, l, sl);
  int x, y, z;
  line_coords(g, A.parity, l, x, y, z);
  project(Z, A.coef, A.F + (lex_site(g, x, y, z, t) * 4 + mu) * 8);
}

void launch_force(const ForceArgs (&a)[2], cudaStream_t s) {
  ForcePair f;
  f.p[0] = a[0];
  f.p[1] = a[1];
  const unsigned blocks = (unsigned)(((size_t)a[0].g.Nl * a[0].g.T + 63) / 64);
  k_force<<<dim3(blocks, 4, 2), 64, 0, s>>>(f);
  WF_CUDA(cudaGetLastError());
}

}  // namespace wf
