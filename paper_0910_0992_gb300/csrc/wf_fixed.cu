// FP64 kernels whose spatial hops run in block fixed point (wf_fixed.cuh), one thread per site of
// the line layout: the hop alone (k_hop_fx; a time-line operation follows in place, wf_kernels.cu)
// and the Wilson matrix (k_apply_M_fx).
#include <algorithm>

#include "wf_fixed.cuh"
#include "wf_internal.h"

namespace wf {

namespace {

// direction d of line l's site (parity, source rhs, slot sl) in the line layout
struct LineDir {
  const Geom& g;
  int x, y, z, rhs, l, sl;
  const Cx<double>*src_up, *src_lo, *us_out, *us_nbr;
  const int4 *fx_out, *fx_nbr;
  __device__ __forceinline__ LineDir(const Geom& gg, int parity, int r, int ll, int s, const Cx<double>* up,
                                     const Cx<double>* lo, const int4* fo, const int4* fn, const Cx<double>* uo,
                                     const Cx<double>* un)
      : g(gg), rhs(r), l(ll), sl(s), src_up(up), src_lo(lo), us_out(uo), us_nbr(un), fx_out(fo), fx_nbr(fn) {
    line_coords(g, parity, l, x, y, z);
  }
  __device__ __forceinline__ HopDir operator()(int d) const {
    const int k = d >> 1, st = d & 1 ? g.L - 1 : 1;
    int nx = x + (k == 0 ? st : 0), ny = y + (k == 1 ? st : 0), nz = z + (k == 2 ? st : 0);
    nx -= nx >= g.L ? g.L : 0;
    ny -= ny >= g.L ? g.L : 0;
    nz -= nz >= g.L ? g.L : 0;
    const int ln = line_of(g, nx, ny, nz);
    const size_t sb = (size_t)(rhs * g.Nl + ln) * NSPIN_C * g.tp + sl;
    const size_t lk = (size_t)(k * g.Nl + (d & 1 ? ln : l)) * 9 * g.tp + sl;
    HopDir q;
    q.up = src_up + sb;
    q.lo = src_lo + sb;
    q.fx = (d & 1 ? fx_nbr : fx_out) + lk;
    q.u = (d & 1 ? us_nbr : us_out) + lk;
    return q;
  }
};

// site -> (source, line, slot), slots fastest, in the line kernels' traversal
__device__ __forceinline__ bool site_at(const Geom& g, size_t i, int nrhs, int& rhs, int& l, int& sl, int& t) {
  const int lg = (int)(i / g.tp);
  sl = (int)(i - (size_t)lg * g.tp);
  const bool in = lg < nrhs * g.Nl;
  line_rhs(in ? lg : 0, nrhs, g, rhs, l);
  t = (sl % g.lpl) * g.n + sl / g.lpl;
  return in;
}

// out = v, v = xpre + apre D_s src (xpre null: D_s src), with the spin halves exchanged if swap_out;
// post: out = xpost + apost v. Padding slots zero (post: xpost).
// (3 CTAs per SM, without spills: 4 % slower; 24^3 x 128, 12 sources)
template <int S>
__global__ void __launch_bounds__(FxShape<S>::threads, FxShape<S>::blocks)
    k_hop_fx(const LineArgs<double> A, int post) {
  grid_dep();
  const Geom& g = A.g;
  int rhs, l, sl, t;
  bool in = site_at(g, fx_site<S>(), A.nrhs, rhs, l, sl, t);
  if (A.active && g.lpw == 1 && !A.active[rhs]) in = false;  // as the line kernels skip them
  const int tp = g.tp;
  const size_t base = ((size_t)rhs * g.Nl + l) * NSPIN_C * tp;
  Vec3<double> h[4];
  double unit[4] = {0.0, 0.0, 0.0, 0.0};
  const bool site = in && t < g.T;
  hop_fx<S>(LineDir(g, A.parity, rhs, l, sl, A.src_up, A.src_lo, A.fx_out, A.fx_nbr, A.us_out, A.us_nbr), tp, tp, site,
            A.fx_out != nullptr, h, unit);
  if (!in || (S > 1 && threadIdx.x >= 32)) return;
  if (!site) {
#pragma unroll
    for (int s = 0; s < 4; ++s) h[s] = vzero<double>();
  }
  if (A.xpre && t < g.T) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      h[s] = vaxpy(A.apre * unit[s], h[s], ldvec(A.xpre + base + 3 * s * tp, tp, sl));
      unit[s] = 1.0;
    }
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int so = A.swap_out ? (s + 2) % 4 : s;
    Vec3<double> v;
    if (post && A.xpost)
      v = vaxpy(A.apost * unit[s], h[s], ldvec(A.xpost + base + 3 * so * tp, tp, sl));
    else
      v = vscale(unit[s], h[s]);
    stvec(A.out + base + 3 * so * tp, tp, sl, v);
  }
}

// The Wilson matrix on the output parity (k_apply_M of wf_line_kernels.cuh), one thread per site
template <bool AX, int S>
__global__ void __launch_bounds__(FxShape<S>::threads, FxShape<S>::blocks) k_apply_M_fx(const MArgs<double> A) {
  grid_dep();
  const Geom& g = A.g;
  int rhs, l, sl, t;
  const bool in = site_at(g, fx_site<S>(), A.nrhs, rhs, l, sl, t);
  const int tp = g.tp, T = g.T;
  const size_t base = ((size_t)rhs * g.Nl + l) * NSPIN_C * tp;
  const bool site = in && t < T;
  const Cx<double>* pp = A.psi_p + base;
  Vec3<double> h[4];
  const Cx<double>* up = A.psi_q + (A.swap ? 6 * tp : 0);
  const Cx<double>* lo = A.psi_q + (A.swap ? 0 : 6 * tp);
  double unit[4];
  hop_fx<S>(LineDir(g, A.parity, rhs, l, sl, up, lo, A.fx_out, A.fx_nbr, A.us_out, A.us_nbr), tp, tp, site,
            A.fx_out != nullptr, h, unit);
  if (S > 1 && threadIdx.x >= 32) return;
  // axial frame: spins 0-1 at t = 0 need P^dag psi(T - 1), spins 2-3 at t = T - 1 P psi(0)
  Vec3<double> wr[2];
  wr[0] = wr[1] = vzero<double>();
  if (AX) {
    const Cx<double>* P = A.pl + (size_t)l * 9;
    warp_link_product(site && t == 0, P, pp + (A.swap ? 6 * tp : 0) + slot_of(g, T - 1), tp, true, wr);
    warp_link_product(site && t == T - 1, P, pp + (A.swap ? 0 : 6 * tp) + slot_of(g, 0), tp, false, wr);
  }
  if (!in) return;
  const Cx<double>* ut_line = AX ? nullptr : A.ut + (size_t)l * NLINK_C * tp;
  const int slf = slot_of(g, t >= T - 1 ? 0 : t + 1), slb = slot_of(g, t == 0 ? T - 1 : t >= T ? 0 : t - 1);
  const double sf = t == T - 1 ? A.bc : 1.0, sb = t == 0 ? A.bc : 1.0;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int sr = A.swap ? (s + 2) % 4 : s;  // spin read for result spin s, and its place in the result
    Vec3<double> val = vzero<double>();
    if (site) {
      Vec3<double> dt;
      if (AX && t == (s < 2 ? 0 : T - 1)) {
        dt = wr[s & 1];
      } else {
        dt = ldvec(pp + 3 * sr * tp, tp, s < 2 ? slb : slf);
        if (!AX) dt = s < 2 ? matvec_dag(ldmat(ut_line, tp, slb), dt) : matvec(ldmat(ut_line, tp, sl), dt);
      }
      val = vscale(A.mu, ldvec(pp + 3 * sr * tp, tp, sl));
      val = vaxpy(s < 2 ? -sb : -sf, dt, val);
      val = vaxpy(-A.inv_gf * unit[s], h[s], val);
    }
    if (A.x) val = vaxpy(A.a, val, ldvec(A.x + base + 3 * sr * tp, tp, sl));
    stvec(A.out + base + 3 * sr * tp, tp, sl, val);
  }
}

__global__ void k_links_fx(const Cx<double>* __restrict__ in, int4* __restrict__ out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int2 r = link_limbs(in[i].re), m = link_limbs(in[i].im);
    out[i] = make_int4(r.x, r.y, m.x, m.y);
  }
}

}  // namespace

void launch_links_fx(const Cx<double>* in, int4* out, size_t n, cudaStream_t s) {
  const unsigned b = (unsigned)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, kSMs * 16));
  k_links_fx<<<b, 256, 0, s>>>(in, out, n);
  WF_CUDA(cudaGetLastError());
}

void launch_hop_fx(const LineArgs<double>& a, bool post, cudaStream_t s) {
  fx_launch((size_t)a.nrhs * a.g.Nl * a.g.tp, [&](auto S, unsigned b, int th, size_t smem) {
    fx_allow(k_hop_fx<S.value>, smem);
    launch_dep(k_hop_fx<S.value>, b, th, smem, s, a, post ? 1 : 0);
  });
  WF_CUDA(cudaGetLastError());
}

void launch_apply_M_fx(const MArgs<double>& a, bool axial, cudaStream_t s) {
  fx_launch((size_t)a.nrhs * a.g.Nl * a.g.tp, [&](auto S, unsigned b, int th, size_t smem) {
    auto* k = axial ? k_apply_M_fx<true, S.value> : k_apply_M_fx<false, S.value>;
    fx_allow(k, smem);
    launch_dep(k, b, th, smem, s, a);
  });
  WF_CUDA(cudaGetLastError());
}

}  // namespace wf
