// FP64 kernels whose spatial hops run in block fixed point (wf_fixed.cuh), one thread per site of
// the line layout: the hop alone (k_hop_fx; a time-line operation follows in place, wf_kernels.cu)
// and the Wilson matrix (k_apply_M_fx).
#include <algorithm>

#include "wf_fixed.cuh"
#include "wf_internal.h"

namespace wf {

namespace {

constexpr int kFxThreads = 128;
constexpr int kFxMinBlocks = 4;  // CTAs per SM (3, without spills: 4 % slower; 24^3 x 128, 12 sources)

// D_s at one site in FP64 (with its factor 1/2): the form of the rare sites whose neighbours are out of
// the fixed-point range (NaN, infinities, exponents near the ends of FP64's). Out of line and rolled.
__device__ __noinline__ void hop_site_fp64(const Geom& g, int parity, const Cx<double>* src_up,
                                           const Cx<double>* src_lo, const Cx<double>* us_out,
                                           const Cx<double>* us_nbr, int rhs, int l, int sl, double* out) {
  const int tp = g.tp;
  int nb[6];
  neighbour_lines(g, parity, l, nb);
  Vec3<double> h[4];
  for (int s = 0; s < 4; ++s) h[s] = vzero<double>();
#pragma unroll 1
  for (int d = 0; d < 6; ++d) {
    const int k = d >> 1, dir = d & 1, ln = nb[d];
    const size_t sb = (size_t)(rhs * g.Nl + ln) * NSPIN_C * tp;
    Mat3<double> U = ldmat(dir == 0 ? us_out + (size_t)(k * g.Nl + l) * 9 * tp : us_nbr + (size_t)(k * g.Nl + ln) * 9 * tp, tp, sl);
    if (dir) U = dagger(U);
    Vec3<double> s0, s1;
    isigma(k, ldvec(src_lo + sb, tp, sl), ldvec(src_lo + sb + 3 * tp, tp, sl), s0, s1);
    if (dir) {
      s0 = vneg(s0);
      s1 = vneg(s1);
    }
    const Vec3<double> w0 = matvec(U, vadd(ldvec(src_up + sb, tp, sl), s0));
    const Vec3<double> w1 = matvec(U, vadd(ldvec(src_up + sb + 3 * tp, tp, sl), s1));
    h[0] = vadd(h[0], w0);
    h[1] = vadd(h[1], w1);
    isigma(k, w0, w1, s0, s1);
    if (!dir) {
      s0 = vneg(s0);
      s1 = vneg(s1);
    }
    h[2] = vadd(h[2], s0);
    h[3] = vadd(h[3], s1);
  }
  for (int s = 0; s < 4; ++s)
    for (int c = 0; c < 3; ++c) {
      out[2 * (3 * s + c)] = 0.5 * h[s].c[c].re;
      out[2 * (3 * s + c) + 1] = 0.5 * h[s].c[c].im;
    }
}

// 16 bytes of device memory into shared memory, asynchronously
__device__ __forceinline__ void fx_copy(int4* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))),
               "l"(__cvta_generic_to_global(src))
               : "memory");
}
// shared memory of a warp: 12 spinor and 9 link entries per lane. A lane reads only what it copied, so
// the copies need no barrier: a direction's spinor arrives while the one before multiplies its link, its
// link while it is projected.
constexpr int kFxStage = 21 * 32;

// h unit = D_s at one site: unit times the integer-valued h (so that the scale joins the next
// multiply-add). stage: the lane's first entry
__device__ __forceinline__ double hop_site_fx(const Geom& g, int parity, const Cx<double>* __restrict__ src_up,
                                              const Cx<double>* __restrict__ src_lo, const int4* __restrict__ fx_out,
                                              const int4* __restrict__ fx_nbr, const Cx<double>* us_out,
                                              const Cx<double>* us_nbr, int rhs, int l, int sl, int4* stage,
                                              Vec3<double> (&h)[4]) {
  const int tp = g.tp, L = g.L;
  int x, y, z;
  line_coords(g, parity, l, x, y, z);
  FxAcc f;
  fx_clear(f);
  // direction d's neighbour and link into the thread's own places of shared memory
  auto neighbour = [&](int d) {
    const int k = d >> 1, st = d & 1 ? L - 1 : 1;
    int nx = x + (k == 0 ? st : 0), ny = y + (k == 1 ? st : 0), nz = z + (k == 2 ? st : 0);
    nx -= nx >= L ? L : 0;
    ny -= ny >= L ? L : 0;
    nz -= nz >= L ? L : 0;
    return line_of(g, nx, ny, nz);
  };
  auto fetch_spinor = [&](int ln) {
    const size_t sb = (size_t)(rhs * g.Nl + ln) * NSPIN_C * tp + sl;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      fx_copy(stage + 32 * c, src_up + sb + c * tp);
      fx_copy(stage + 32 * (6 + c), src_lo + sb + c * tp);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto fetch_link = [&](int d, int ln) {
    const int k = d >> 1;
    const int4* lk = (d & 1 ? fx_nbr + (size_t)(k * g.Nl + ln) * 9 * tp : fx_out + (size_t)(k * g.Nl + l) * 9 * tp) + sl;
#pragma unroll
    for (int e = 0; e < 9; ++e) fx_copy(stage + 32 * (12 + e), lk + e * tp);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  int ln = neighbour(0);
  fetch_spinor(ln);
  fetch_link(0, ln);
#pragma unroll 1
  for (int d = 0; d < 6; ++d) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    FxHalf q;
    {
      Vec3<double> v[4];
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) v[s].c[c] = *reinterpret_cast<const Cx<double>*>(stage + 32 * (3 * s + c));
      fx_project(f, q, d, v);
    }
    if (d < 5) {
      ln = neighbour(d + 1);
      fetch_spinor(ln);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    fx_multiply(f, q, d, stage + 32 * 12, 32);
    if (d < 5) fetch_link(d + 1, ln);
  }
  if (f.wide) {
    double o[24];
    hop_site_fp64(g, parity, src_up, src_lo, us_out, us_nbr, rhs, l, sl, o);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) h[s].c[c] = mk<double>(o[2 * (3 * s + c)], o[2 * (3 * s + c) + 1]);
    return 1.0;
  }
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) h[s].c[c] = mk<double>((double)f.a[s][c][0], (double)f.a[s][c][1]);
  return fx_unit(f);
}

__device__ __forceinline__ int4* fx_stage() {
  extern __shared__ int4 fx_shared[];
  return fx_shared + (threadIdx.x >> 5) * kFxStage + (threadIdx.x & 31);
}

// thread -> (source, line, slot), slots fastest, in the line kernels' traversal
__device__ __forceinline__ bool site_at(const Geom& g, int nrhs, int& rhs, int& l, int& sl, int& t) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const int lg = (int)(i / g.tp);
  sl = (int)(i - (size_t)lg * g.tp);
  const bool in = lg < nrhs * g.Nl;
  line_rhs(in ? lg : 0, nrhs, g, rhs, l);
  t = (sl % g.lpl) * g.n + sl / g.lpl;
  return in;
}

// out = v, v = xpre + apre D_s src (xpre null: D_s src), with the spin halves exchanged if swap_out;
// post: out = xpost + apost v. Padding slots zero (post: xpost).
__global__ void __launch_bounds__(kFxThreads, kFxMinBlocks) k_hop_fx(const LineArgs<double> A, int post) {
  const Geom& g = A.g;
  int rhs, l, sl, t;
  if (!site_at(g, A.nrhs, rhs, l, sl, t)) return;
  if (A.active && g.lpw == 1 && !A.active[rhs]) return;  // as the line kernels skip them
  const int tp = g.tp;
  const size_t base = ((size_t)rhs * g.Nl + l) * NSPIN_C * tp;
  Vec3<double> h[4];
  double unit = 0.0;
  if (t < g.T) {
    unit = hop_site_fx(g, A.parity, A.src_up, A.src_lo, A.fx_out, A.fx_nbr, A.us_out, A.us_nbr, rhs, l, sl, fx_stage(), h);
  } else {
#pragma unroll
    for (int s = 0; s < 4; ++s) h[s] = vzero<double>();
  }
  if (A.xpre && t < g.T) {
#pragma unroll
    for (int s = 0; s < 4; ++s) h[s] = vaxpy(A.apre * unit, h[s], ldvec(A.xpre + base + 3 * s * tp, tp, sl));
    unit = 1.0;
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int so = A.swap_out ? (s + 2) % 4 : s;
    Vec3<double> v;
    if (post && A.xpost)
      v = vaxpy(A.apost * unit, h[s], ldvec(A.xpost + base + 3 * so * tp, tp, sl));
    else
      v = vscale(unit, h[s]);
    stvec(A.out + base + 3 * so * tp, tp, sl, v);
  }
}

// The Wilson matrix on the output parity (k_apply_M of wf_line_kernels.cuh), one thread per site. The
// wrap's P (axial frame) is applied by six lanes of the warp, one result component each: as one
// lane's two 3x3 products it would hold the FP64 pipe for the whole warp as long as the site's
// other FP64 operations together.
template <bool AX>
__global__ void __launch_bounds__(kFxThreads, kFxMinBlocks) k_apply_M_fx(const MArgs<double> A) {
  const Geom& g = A.g;
  int rhs, l, sl, t;
  const bool in = site_at(g, A.nrhs, rhs, l, sl, t);
  const int tp = g.tp, T = g.T;
  const size_t base = ((size_t)rhs * g.Nl + l) * NSPIN_C * tp;
  const bool site = in && t < T;
  const Cx<double>* pp = A.psi_p + base;
  Vec3<double> h[4];
  double unit = 0.0;
  if (site) {
    unit = hop_site_fx(g, A.parity, A.psi_q + (A.swap ? 6 * tp : 0), A.psi_q + (A.swap ? 0 : 6 * tp), A.fx_out, A.fx_nbr,
                       A.us_out, A.us_nbr, rhs, l, sl, fx_stage(), h);
  }
  // axial frame: spins 0-1 at t = 0 need P^dag psi(T - 1), spins 2-3 at t = T - 1 P psi(0)
  Vec3<double> wr[2];
  wr[0] = wr[1] = vzero<double>();
  if (AX) {
    const int lane = threadIdx.x & 31;
    const int q = lane < 6 ? lane : 0, qs = q / 3, qr = q - 3 * (q / 3);
#pragma unroll
    for (int end = 0; end < 2; ++end) {
      unsigned m = __ballot_sync(0xffffffffu, site && t == (end ? T - 1 : 0));
      const int from = slot_of(g, end ? 0 : T - 1);  // the slot read
      while (m) {
        const int w = __ffs(m) - 1;
        m &= m - 1;
        const int wl = __shfl_sync(0xffffffffu, l, w), wk = __shfl_sync(0xffffffffu, rhs, w);
        // spins of the result half, read from the other half's place if the halves are exchanged
        const int sr = ((end ? 2 : 0) + qs + (A.swap ? 2 : 0)) % 4;
        const Cx<double>* x = A.psi_p + (((size_t)wk * g.Nl + wl) * NSPIN_C + 3 * sr) * tp + from;
        const Cx<double>* P = A.pl + (size_t)wl * 9;
        Cx<double> v = czero<double>();
#pragma unroll
        for (int b = 0; b < 3; ++b)
          v = end ? cfma(v, P[3 * qr + b], x[(size_t)b * tp]) : cfmaconj(v, P[3 * b + qr], x[(size_t)b * tp]);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const Cx<double> u = shfl_idx(v, i, 32);
          if (lane == w) wr[i / 3].c[i % 3] = u;
        }
      }
    }
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
      val = vaxpy(-A.inv_gf * unit, h[s], val);
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

// CTA size: one warp where the lattice is too small to give every SM four
int fx_threads(size_t sites) { return sites < (size_t)152 * kFxThreads ? 32 : kFxThreads; }

size_t fx_smem(int threads) { return (size_t)threads / 32 * kFxStage * sizeof(int4); }

}  // namespace

void launch_links_fx(const Cx<double>* in, int4* out, size_t n, cudaStream_t s) {
  const unsigned b = (unsigned)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 152 * 16));
  k_links_fx<<<b, 256, 0, s>>>(in, out, n);
  WF_CUDA(cudaGetLastError());
}

void launch_hop_fx(const LineArgs<double>& a, bool post, cudaStream_t s) {
  if (!a.fx_out || !a.fx_nbr) throw Error(1, "FP64 hop: no fixed-point links");
  const size_t sites = (size_t)a.nrhs * a.g.Nl * a.g.tp;
  const int th = fx_threads(sites);
  k_hop_fx<<<(unsigned)((sites + th - 1) / th), th, fx_smem(th), s>>>(a, post ? 1 : 0);
  WF_CUDA(cudaGetLastError());
}

void launch_apply_M_fx(const MArgs<double>& a, bool axial, cudaStream_t s) {
  if (!a.fx_out || !a.fx_nbr) throw Error(1, "FP64 Wilson matrix: no fixed-point links");
  const size_t sites = (size_t)a.nrhs * a.g.Nl * a.g.tp;
  const int th = fx_threads(sites);
  const unsigned b = (unsigned)((sites + th - 1) / th);
  if (axial)
    k_apply_M_fx<true><<<b, th, fx_smem(th), s>>>(a);
  else
    k_apply_M_fx<false><<<b, th, fx_smem(th), s>>>(a);
  WF_CUDA(cudaGetLastError());
}

}  // namespace wf
