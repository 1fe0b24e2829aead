// FP64 spatial hops in block fixed point.
//
// GB300 issues two FP64 multiply-adds per clock and SM, but 64 32 x 32 -> 64-bit integer ones: the 648
// FP64 operations of a spatial hop cost 324 clocks per site and SM, the same hop in 64-bit fixed point
// about 100 (M, both parities, 24^3 x 128, 12 sources: 30.4 -> 9.7 ms; 12^3 x 48, 4 sources: 548 -> 209
// us). The direction d of a site's stencil is a half-spinor of 12 real numbers times one SU(3) link, and
//   * a direction makes two result spins of each pair of the neighbour's spins (axes x, y: 0 and 3 of
//     spins 0 and 3, 1 and 2 of 1 and 2; z: 0 and 2, 1 and 3). Every result spin r has an exponent E_r,
//     the largest of the numbers that made it so far; a pair is taken as v = x 2^(57 - F), F the smaller
//     exponent of its two results, |v| < 2^58: an exact shift of the 53-bit mantissa but for bits below
//     2^(F - 57);
//   * links are stored beside their FP64 form as u = U 2^57 in two 32-bit limbs (|U| <= 1);
//   * projections are integer sums (< 2^59); a product takes three limb products, accumulated over the six
//     of a matrix row in two 64-bit sums: H of the high limbs' products and X of the mixed ones (the low
//     limbs' products, each below one unit of H, are left out), w = H + X / 2^28 in units of 2^(F - 58);
//   * w is shifted to units of 2^(E_r - 57) of each of its two results, and the six directions add up in 64
//     bits (|sum| < 2^62.9).
//
// Accuracy. A result component (one spin and colour) is a sum over directions and colours of a link entry
// times two spinor components; S is the sum of the terms' absolute values, the scale of FP64 arithmetic's
// error. Here the roundings (of v, U 2^57, the low products left out, X / 2^28 and the shift: 21 units of
// 2^(E_r - 57) a direction) are below 7.9 x 2^-53 2^E_r, so the form is used only where S is not far below
// 2^E_r (fx_accurate): either some direction brings result spin r a pair of spins all of whose three
// colours reach 2^(E_r - 4) (the moduli in a row of a unitary link add up to 1 or more, so then S >=
// 2^(E_r - 4) for each colour, whatever the link), or every colour's result itself has reached
// 2^(E_r - 4). Other sites take the FP64 form (hop_dir_fp64), as do sites whose result spins differ by
// more than 2^30 and spinors with a NaN, an infinity or exponents near the ends of FP64's range. Errors in
// units of 2^-53 S, root mean square over the sites that pass, fixed point : FP64 arithmetic (emulated
// against products in 113 bits): Gaussian spinors on random links 0.09 : 0.25, on links of unity 0.14 :
// 0.31; two spins 2^-20 of the others 0.17 : 0.41; components scaled at random over 2^6 0.14 : 0.39, over
// 2^30 0.33 : 0.72; colours 2^-5 of each other on links of unity 0.25 : 0.31; one component alone 0.29 :
// 0.51. Largest 4.7 : 4.9. With 2^(E_r - 5) colours 2^-6 of each other would lose (0.49 : 0.31); with
// 2^(E_r - 2) some Gaussian sites would go to the FP64 form, and the whole launch of a small lattice waits
// for one (8^3 x 32, FP64 solve 4.9 -> 7.9 ms).
#pragma once

#include <type_traits>

#include "wf_internal.h"
#include "wf_line.cuh"

namespace wf {

// one real number of a link: limbs of U 2^57, hi 2^28 + lo, 0 <= lo < 2^28
__device__ __forceinline__ int2 link_limbs(double u) {
  const long long v = llrint(u * 144115188075855872.0);  // 2^57
  return make_int2((int)(v >> 28), (int)(v & 0xfffffff));
}

// acc + a b (a limb of each sign; left to the compiler, the products with the limbs it knows to be
// non-negative became full 64-bit multiplications)
__device__ __forceinline__ void fx_mac(long long& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

constexpr int kFxMinExp = 80, kFxMaxExp = 2030;  // biased exponents served
constexpr int kFxSpread = 4;                     // of 2^(E_r - 4) above

struct FxAcc {
  long long a[4][3][2];  // [spin][colour][re, im], in units of 2^(E_r - 1023 - 57)
  // per result spin 2^16 E_r (biased) + the largest over the directions of the exponent of the smallest
  // colour of the pair that made it (1 at least; 0: nothing but zeros so far)
  unsigned eq[4];
  bool wide;             // some spinor was out of range: the result is not valid
  __device__ __forceinline__ int E(int r) const { return (int)(eq[r] >> 16); }
};

__device__ __forceinline__ void fx_clear(FxAcc& f) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
#pragma unroll
    for (int c = 0; c < 3; ++c) f.a[s][c][0] = f.a[s][c][1] = 0;
    f.eq[s] = (unsigned)kFxMinExp << 16;
  }
  f.wide = false;
}

// whether the sums are as accurate as FP64 arithmetic's would be (above)
__device__ __forceinline__ bool fx_accurate(const FxAcc& f) {
  bool ok = !f.wide;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int q = (int)(f.eq[s] & 0xffffu);
    if (q == 0 || q >= f.E(s) - kFxSpread) continue;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const long long re = f.a[s][c][0], im = f.a[s][c][1];
      ok = ok && max(re < 0 ? -re : re, im < 0 ? -im : im) >= 1LL << (57 - kFxSpread);
    }
  }
  return ok;
}

// x as v = x 2^(52 + B - E) (E >= x's exponent, B <= 10; zero and subnormal x: 0)
template <int B>
__device__ __forceinline__ long long fx_from(double x, int E) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const int s = min(E - (int)((hw >> 20) & 0x7ff), 63);
  const unsigned mh = (hw & 0xfffff) | 0x100000;
  unsigned long long m = ((unsigned long long)__funnelshift_l(lw, mh, B) << 32) | (lw << B);
  m >>= s;
  const long long neg = (long long)((int)hw >> 31);
  return ((long long)m ^ neg) - neg;
}
// v >> s, 0 <= s <= 31
__device__ __forceinline__ long long fx_shift(long long v, int s) {
  const int hi = (int)(v >> 32);
  return ((long long)(hi >> s) << 32) | __funnelshift_r((unsigned)v, (unsigned)hi, s);
}

// One direction d = 2 k + dir of D_s (without its factor 1/2): axis k, dir 0: (1 - gamma_k) U x,
// 1: (1 + gamma_k) U^dag x, x the neighbour spinor. The directions share one copy of this code (d is
// uniform; only the spin algebra branches on it): unrolled six times, the kernel missed the instruction
// cache on 45 % of its issue slots.
struct FxHalf {  // the half-spinor in limbs
  int hh[2][3][2], hl[2][3][2];
  int up[2], lo[2];  // shifts of the products of its two spins on their way to the upper and the lower result spin
};
__device__ __forceinline__ void fx_project(FxAcc& f, FxHalf& q, int d, const Vec3<double> (&x)[4]) {
  const bool z = d >= 4;
  // per pair p the largest high word, and the smallest over the colours of the larger of its two spins
  unsigned mx[2] = {0, 0}, mn[2] = {~0u, ~0u};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    unsigned m[4];
#pragma unroll
    for (int s = 0; s < 4; ++s)
      m[s] = max((unsigned)__double2hiint(x[s].c[c].re) & 0x7fffffffu, (unsigned)__double2hiint(x[s].c[c].im) & 0x7fffffffu);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const unsigned e = max(m[p], z ? m[2 + p] : m[3 - p]);
      mx[p] = max(mx[p], e);
      mn[p] = min(mn[p], e);
    }
  }
  unsigned pk[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const unsigned e = mx[p] >> 20;
    pk[p] = mx[p] ? (e << 16) | max(mn[p] >> 20, 1u) : 0;
    f.wide = f.wide || (mx[p] != 0 && (e < (unsigned)kFxMinExp || e >= (unsigned)kFxMaxExp));
    if (mx[p] == 0) {  // zeros, or numbers below 2^-1042
      unsigned low = 0;
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int s = 0; s < 4; ++s)
          if (s == p || s == (z ? 2 + p : 3 - p))
            low |= (unsigned)__double2loint(x[s].c[c].re) | (unsigned)__double2loint(x[s].c[c].im);
      f.wide = f.wide || low != 0;
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const unsigned n = __vmaxu2(f.eq[r], r < 2 ? pk[r] : z ? pk[r - 2] : pk[3 - r]);
    const int s = min((int)(n >> 16) - f.E(r), 63);
    f.eq[r] = n;
    if (s) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        f.a[r][c][0] >>= s;
        f.a[r][c][1] >>= s;
      }
    }
  }
  int F[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int eu = f.E(p), el = z ? f.E(2 + p) : f.E(3 - p);
    F[p] = min(eu, el);
    f.wide = f.wide || (mx[p] != 0 && max(eu, el) - F[p] > 30);
    q.up[p] = min(eu - F[p], 30) + 1;  // from units of 2^(F - 1023 - 58)
    q.lo[p] = min(el - F[p], 30) + 1;
  }
  // h = u +- i sigma_k d (isigma of wf_line.cuh)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    long long u[2][2], v[2][2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int G = z ? F[s] : F[1 - s];
      u[s][0] = fx_from<5>(x[s].c[c].re, F[s]);
      u[s][1] = fx_from<5>(x[s].c[c].im, F[s]);
      v[s][0] = fx_from<5>(x[2 + s].c[c].re, G);
      v[s][1] = fx_from<5>(x[2 + s].c[c].im, G);
    }
    switch (d) {
      case 0: u[0][0] -= v[1][1]; u[0][1] += v[1][0]; u[1][0] -= v[0][1]; u[1][1] += v[0][0]; break;
      case 1: u[0][0] += v[1][1]; u[0][1] -= v[1][0]; u[1][0] += v[0][1]; u[1][1] -= v[0][0]; break;
      case 2: u[0][0] += v[1][0]; u[0][1] += v[1][1]; u[1][0] -= v[0][0]; u[1][1] -= v[0][1]; break;
      case 3: u[0][0] -= v[1][0]; u[0][1] -= v[1][1]; u[1][0] += v[0][0]; u[1][1] += v[0][1]; break;
      case 4: u[0][0] -= v[0][1]; u[0][1] += v[0][0]; u[1][0] += v[1][1]; u[1][1] -= v[1][0]; break;
      default: u[0][0] += v[0][1]; u[0][1] -= v[0][0]; u[1][0] -= v[1][1]; u[1][1] += v[1][0]; break;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        q.hh[s][c][p] = (int)(u[s][p] >> 28);
        q.hl[s][c][p] = (int)u[s][p] & 0xfffffff;
      }
  }
}
// acc += the link times the half-spinor and its lower spins; lk[e * stride]: the link's entries as
// {re.hi, re.lo, im.hi, im.lo}
__device__ __forceinline__ void fx_multiply(FxAcc& f, const FxHalf& q, int d, const int4* __restrict__ lk, int stride) {
  // w = V h, V = U or U^dag (entry (a, b) at a sa + b sb, imaginary limbs with sign sg)
  const int dir = d & 1, sg = -dir;
  const int sa = (dir ? 1 : 3) * stride, sb = (dir ? 3 : 1) * stride;
  constexpr long long half = 1LL << 27;  // of X / 2^28, whose shift rounds down
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    long long H[2][2] = {}, X[2][2] = {{half, half}, {half, half}};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      int4 U = lk[a * sa + b * sb];
      U.z = (U.z ^ sg) - sg;
      U.w = (U.w ^ sg) - sg;
      const int nz = -U.z, nw = -U.w;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int rh = q.hh[s][b][0], rl = q.hl[s][b][0], ih = q.hh[s][b][1], il = q.hl[s][b][1];
        fx_mac(H[s][0], U.x, rh);
        fx_mac(X[s][0], U.x, rl);
        fx_mac(X[s][0], U.y, rh);
        fx_mac(H[s][0], nz, ih);
        fx_mac(X[s][0], nz, il);
        fx_mac(X[s][0], nw, ih);
        fx_mac(H[s][1], U.x, ih);
        fx_mac(X[s][1], U.x, il);
        fx_mac(X[s][1], U.y, ih);
        fx_mac(H[s][1], U.z, rh);
        fx_mac(X[s][1], U.z, rl);
        fx_mac(X[s][1], U.w, rh);
      }
    }
    long long w[2][2];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const long long v = H[s][p] + (X[s][p] >> 28);
        f.a[s][a][p] += fx_shift(v, q.up[s]);
        w[s][p] = fx_shift(v, q.lo[s]);
      }
    long long(&l0)[2] = f.a[2][a], (&l1)[2] = f.a[3][a];  // lower spins: -+ i sigma_k w
    switch (d) {
      case 0: l0[0] += w[1][1]; l0[1] -= w[1][0]; l1[0] += w[0][1]; l1[1] -= w[0][0]; break;
      case 1: l0[0] -= w[1][1]; l0[1] += w[1][0]; l1[0] -= w[0][1]; l1[1] += w[0][0]; break;
      case 2: l0[0] -= w[1][0]; l0[1] -= w[1][1]; l1[0] += w[0][0]; l1[1] += w[0][1]; break;
      case 3: l0[0] += w[1][0]; l0[1] += w[1][1]; l1[0] -= w[0][0]; l1[1] -= w[0][1]; break;
      case 4: l0[0] += w[0][1]; l0[1] -= w[0][0]; l1[0] -= w[1][1]; l1[1] += w[1][0]; break;
      default: l0[0] -= w[0][1]; l0[1] += w[0][0]; l1[0] += w[1][1]; l1[1] -= w[1][0]; break;
    }
  }
}

// 2^(E_r - 1023 - 58): a unit of the accumulators of spin r times the projectors' factor 1/2 (E_r >= kFxMinExp)
__device__ __forceinline__ double fx_unit(const FxAcc& f, int r) { return __hiloint2double((f.E(r) - 58) << 20, 0); }

// ----------------------------------------------------------------------------
// D_s at one site. dir(d) names direction d's operands (HopDir).
// ----------------------------------------------------------------------------
struct HopDir {
  const Cx<double>* up;  // the neighbour's components that supply spins 0-1, and
  const Cx<double>* lo;  // spins 2-3, cs elements apart
  const int4* fx;        // the link in fixed point (if there) and in FP64, entries ls elements apart
  const Cx<double>* u;
};

// one direction in FP64, added to acc (out of line: sites that fx_accurate refuses)
static __device__ __noinline__ void hop_dir_fp64(int d, HopDir q, int cs, int ls, double* acc) {
  const int k = d >> 1, dir = d & 1;
  Mat3<double> U = ldmat(q.u, ls, 0);
  if (dir) U = dagger(U);
  Vec3<double> s[2], w[2];
  isigma(k, ldvec(q.lo, cs, 0), ldvec(q.lo + 3 * cs, cs, 0), s[0], s[1]);
  for (int i = 0; i < 2; ++i) w[i] = matvec(U, vaxpy(dir ? -1.0 : 1.0, s[i], ldvec(q.up + 3 * i * cs, cs, 0)));
  isigma(k, w[0], w[1], s[0], s[1]);
  for (int i = 0; i < 2; ++i)
    for (int c = 0; c < 3; ++c) {
      acc[6 * i + 2 * c] += w[i].c[c].re;
      acc[6 * i + 2 * c + 1] += w[i].c[c].im;
      acc[12 + 6 * i + 2 * c] += dir ? s[i].c[c].re : -s[i].c[c].re;
      acc[12 + 6 * i + 2 * c + 1] += dir ? s[i].c[c].im : -s[i].c[c].im;
    }
}

// dynamic shared memory of a warp: 12 spinor and 9 link entries per lane. A lane reads only what it
// copied, so the copies need no barrier: a direction's spinor arrives while the one before multiplies its
// link, its link while it is projected.
constexpr int kFxStage = 21 * 32;
inline size_t fx_smem(int threads) { return (size_t)threads / 32 * kFxStage * sizeof(int4); }

// CTA size, resident CTAs per SM (128 registers a thread) and the thread's site for a hop split over S warps
// (S = 1: one thread per site)
template <int S>
struct FxShape {
  static constexpr int threads = S == 1 ? 128 : 32 * S, blocks = S == 1 ? 4 : 16 / S;
};
template <int S>
__device__ __forceinline__ size_t fx_site() {
  return S == 1 ? blockIdx.x * (size_t)blockDim.x + threadIdx.x : blockIdx.x * (size_t)32 + (threadIdx.x & 31);
}

// D_s = unit[s] h[s] for spin s (so that the scale joins the next multiply-add). With S > 1 the S warps
// of a CTA take 6 / S directions each of the same 32 sites and warp 0 adds them up (integers: exactly,
// but for the shift to a common exponent that the six directions of one thread see as well); the others
// have no result. Called by every thread of the CTA; site: whether the thread has one; fixed: whether there are
// fixed-point links (else FP64 arithmetic).
template <int S, class Dir>
__device__ __forceinline__ void hop_fx(const Dir& dir, int cs, int ls, bool site, bool fixed, Vec3<double> (&h)[4],
                                       double (&unit)[4]) {
  extern __shared__ int4 fx_shared[];
  int4* stage = fx_shared + (threadIdx.x >> 5) * kFxStage + (threadIdx.x & 31);
  constexpr int N = 6 / S;
  const int d0 = S == 1 ? 0 : (threadIdx.x >> 5) * N;
  FxAcc f;
  fx_clear(f);
  auto fetch_spinor = [&](const HopDir& q) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      cp_async16(stage + 32 * c, q.up + (size_t)c * cs);
      cp_async16(stage + 32 * (6 + c), q.lo + (size_t)c * cs);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto fetch_link = [&](const HopDir& q) {
#pragma unroll
    for (int e = 0; e < 9; ++e) cp_async16(stage + 32 * (12 + e), q.fx + (size_t)e * ls);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  f.wide = !fixed;
  if (site && fixed) {
    HopDir next = dir(d0);
    fetch_spinor(next);
    fetch_link(next);
#pragma unroll 1
    for (int d = d0; d < d0 + N; ++d) {
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
      if (d < d0 + N - 1) {
        next = dir(d + 1);
        fetch_spinor(next);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      fx_multiply(f, q, d, stage + 32 * 12, 32);
      if (d < d0 + N - 1) fetch_link(next);
    }
  }
  if constexpr (S > 1) {  // the stage is free: each lane's sums there, then warp 0 collects them
    longlong2* box = reinterpret_cast<longlong2*>(stage);
    if (d0) {
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) box[32 * (3 * s + c)] = make_longlong2(f.a[s][c][0], f.a[s][c][1]);
      stage[32 * 12] = make_int4((int)f.eq[0], (int)f.eq[1], (int)f.eq[2], (int)f.eq[3]);
      stage[32 * 13].x = f.wide;
    }
    __syncthreads();
    if (d0) return;
#pragma unroll
    for (int p = 1; p < S; ++p) f.wide = f.wide || stage[p * kFxStage + 32 * 13].x;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      unsigned o[S], n = f.eq[s];
#pragma unroll
      for (int p = 1; p < S; ++p) {
        o[p] = reinterpret_cast<const unsigned*>(stage + p * kFxStage + 32 * 12)[s];
        n = __vmaxu2(n, o[p]);
      }
      const int E = (int)(n >> 16), s0 = min(E - f.E(s), 63);
      f.eq[s] = n;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        f.a[s][c][0] >>= s0;
        f.a[s][c][1] >>= s0;
#pragma unroll
        for (int p = 1; p < S; ++p) {
          const longlong2 v = box[p * kFxStage + 32 * (3 * s + c)];
          const int sp = min(E - (int)(o[p] >> 16), 63);
          f.a[s][c][0] += v.x >> sp;
          f.a[s][c][1] += v.y >> sp;
        }
      }
    }
  }
  if (!site) return;
  if (!fx_accurate(f)) {
    double o[24];
    for (int i = 0; i < 24; ++i) o[i] = 0.0;
#pragma unroll 1
    for (int d = 0; d < 6; ++d) hop_dir_fp64(d, dir(d), cs, ls, o);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
#pragma unroll
      for (int c = 0; c < 3; ++c) h[s].c[c] = mk<double>(o[2 * (3 * s + c)], o[2 * (3 * s + c) + 1]);
      unit[s] = 0.5;
    }
    return;
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
#pragma unroll
    for (int c = 0; c < 3; ++c) h[s].c[c] = mk<double>((double)f.a[s][c][0], (double)f.a[s][c][1]);
    unit[s] = fx_unit(f, s);
  }
}

// Launch shape of a hop over `sites`: run(S, blocks, threads, dynamic shared memory) with the directions
// split over as many warps S (std::integral_constant) as still leaves every CTA resident at once; the
// chain of six spinor and link fetches is what bounds few sites. The Wilson matrix on one parity, us with
// S = 1, 2, 3, 6 (32-site warps): 16 warps 30, 23, 21, 17; 256 28, 22, 21, 18; 512 29, 25, 23, 30;
// 768 36, 29, 35, 42; 1024 36, 34, 39, 52; 1536 45, 48, 52, 72.
template <class Run>
inline void fx_launch(size_t sites, Run&& run) {
  const size_t warps = (sites + 31) / 32;
  auto go = [&](auto S) {
    constexpr int th = FxShape<S.value>::threads, per = S.value == 1 ? th : 32;
    run(S, (unsigned)((sites + per - 1) / per), th, fx_smem(th));
  };
  if (warps <= kSMs * FxShape<6>::blocks)
    go(std::integral_constant<int, 6>{});
  else if (warps <= kSMs * FxShape<3>::blocks)
    go(std::integral_constant<int, 3>{});
  else if (warps <= kSMs * FxShape<2>::blocks)
    go(std::integral_constant<int, 2>{});
  else
    go(std::integral_constant<int, 1>{});
}
// lets kernel k have more dynamic shared memory than a launch may by default (48 KB)
template <class K>
inline void fx_allow(K* k, size_t smem) {
  if (smem > 48 * 1024) WF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
}

// For the lanes with flag set: out = P x (dag: P^dag x) of two colour vectors, x's six components cs elements
// apart. Six lanes of the warp form one component each: as one lane's two products, the wrap of the
// axial frame would hold the FP64 pipe for the whole warp as long as the rest of a site's FP64
// operations. Warp-collective.
__device__ __forceinline__ void warp_link_product(bool flag, const Cx<double>* P, const Cx<double>* x, int cs, bool dag,
                                                  Vec3<double> (&out)[2]) {
  const int lane = threadIdx.x & 31;
  const int q = lane < 6 ? lane : 0, row = q % 3;
  unsigned m = __ballot_sync(0xffffffffu, flag);
  while (m) {
    const int w = __ffs(m) - 1;
    m &= m - 1;
    const Cx<double>* Pw = reinterpret_cast<const Cx<double>*>(__shfl_sync(0xffffffffu, (unsigned long long)P, w));
    const Cx<double>* xw = reinterpret_cast<const Cx<double>*>(__shfl_sync(0xffffffffu, (unsigned long long)x, w));
    xw += (size_t)(q - row) * cs;
    Cx<double> v = czero<double>();
#pragma unroll
    for (int b = 0; b < 3; ++b)
      v = dag ? cfmaconj(v, Pw[3 * b + row], xw[(size_t)b * cs]) : cfma(v, Pw[3 * row + b], xw[(size_t)b * cs]);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const Cx<double> u = shfl_idx(v, i, 32);
      if (lane == w) out[i / 3].c[i % 3] = u;
    }
  }
}

}  // namespace wf
