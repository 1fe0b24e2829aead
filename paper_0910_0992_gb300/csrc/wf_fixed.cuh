// FP64 spatial hops in block fixed point.
//
// GB300 issues two FP64 multiply-adds per clock and SM, but 64 32 x 32 -> 64-bit integer ones: the
// 648 FP64 operations of a spatial hop cost 324 clocks per site and SM, the same hop in 64-bit fixed
// point about 90 (M, both parities, 24^3 x 128, 12 sources: 30.4 -> 8.9 ms; 12^3 x 48, 4 sources: 548 ->
// 188 us). The direction d of a site's stencil is a half-spinor of 12 real numbers times one
// SU(3) link, and
//   * the 24 real numbers of the neighbour spinor share an exponent E (the largest of theirs, and of
//     the directions before): v = x 2^(55 - E), |v| < 2^56, an exact shift of the 53-bit mantissa but
//     for bits below 2^(E - 55), a quarter of half an ulp of the largest number;
//   * links are stored beside their FP64 form as u = U 2^58 in two 32-bit limbs (|U| <= 1);
//   * projections are integer sums (< 2^57); a product takes three limb products, accumulated over
//     the six of a matrix row in two 64-bit sums: H of the high limbs' products and X of the mixed ones
//     (the low limbs' product is below 1/4 of a unit of v), w = H + X / 2^28 in units of v / 4;
//   * the six directions add up in 64 bits (|sum| < 2^(56 + 6.9)).
// So the only roundings are those of v, U 2^58 and X / 2^28, each below an FP64 rounding of the
// largest term: the result is at least as close to the exact one as FP64 arithmetic's (measured on
// 12^3 x 48, M against 64-bit reference arithmetic: relative error 3.5e-15 either way). Spinors with a NaN,
// an infinity or exponents near the ends of FP64's range take the FP64 form (hop_dir_fp64).
#pragma once

#include <type_traits>

#include "wf_internal.h"
#include "wf_line.cuh"

namespace wf {

// one real number of a link: limbs of U 2^58, hi 2^28 + lo, 0 <= lo < 2^28
__device__ __forceinline__ int2 link_limbs(double u) {
  const long long v = llrint(u * 288230376151711744.0);  // 2^58
  return make_int2((int)(v >> 28), (int)(v & 0xfffffff));
}

// acc + a b (a limb of each sign; left to the compiler, the products with the limbs it knows to be
// non-negative became full 64-bit multiplications)
__device__ __forceinline__ void fx_mac(long long& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

struct FxAcc {
  long long a[4][3][2];  // [spin][colour][re, im], in units of 2^(E - 1023 - 57)
  int E;                 // biased FP64 exponent
  bool wide;             // some spinor was out of range: the result is not valid
};

constexpr int kFxMinExp = 80, kFxMaxExp = 2030;  // biased exponents served

__device__ __forceinline__ void fx_clear(FxAcc& f) {
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) f.a[s][c][0] = f.a[s][c][1] = 0;
  f.E = kFxMinExp;
  f.wide = false;
}

// x as v = x 2^(55 - E) (E >= x's exponent; zero and subnormal x: 0)
__device__ __forceinline__ long long fx_from(double x, int E) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const int s = min(E - (int)((hw >> 20) & 0x7ff), 63);
  const unsigned mh = (hw & 0xfffff) | 0x100000;
  unsigned long long m = ((unsigned long long)__funnelshift_l(lw, mh, 3) << 32) | (lw << 3);
  m >>= s;
  const long long neg = (long long)((int)hw >> 31);
  return ((long long)m ^ neg) - neg;
}

// One direction d = 2 k + dir of D_s (without its factor 1/2): axis k, dir 0: (1 - gamma_k) U x,
// 1: (1 + gamma_k) U^dag x, x the neighbour spinor. The directions share one copy of this code (d is
// uniform; only the spin algebra branches on it): unrolled six times, the kernel missed the instruction
// cache on 45 % of its issue slots.
struct FxHalf {  // the half-spinor in limbs; nh, nl: minus the imaginary part's
  int hh[2][3][2], hl[2][3][2], nh[2][3], nl[2][3];
};
__device__ __forceinline__ void fx_project(FxAcc& f, FxHalf& q, int d, const Vec3<double> (&x)[4]) {
  unsigned mx = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      mx = max(mx, (unsigned)__double2hiint(x[s].c[c].re) & 0x7fffffffu);
      mx = max(mx, (unsigned)__double2hiint(x[s].c[c].im) & 0x7fffffffu);
    }
  const int e = (int)(mx >> 20);
  f.wide = f.wide || (mx != 0 && (e < kFxMinExp || e >= kFxMaxExp));
  if (e > f.E) {
    const int s = min(e - f.E, 63);
    f.E = e;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        f.a[i][c][0] >>= s;
        f.a[i][c][1] >>= s;
      }
  }
  // h = u +- i sigma_k d (isigma of wf_line.cuh)
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    long long u[2][2], v[2][2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      u[s][0] = fx_from(x[s].c[c].re, f.E);
      u[s][1] = fx_from(x[s].c[c].im, f.E);
      v[s][0] = fx_from(x[2 + s].c[c].re, f.E);
      v[s][1] = fx_from(x[2 + s].c[c].im, f.E);
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
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      q.nh[s][c] = -q.hh[s][c][1];
      q.nl[s][c] = -q.hl[s][c][1];
    }
  }
}
// acc += the link times the half-spinor and its lower spins; lk[e * stride]: the link's entries as
// {re.hi, re.lo, im.hi, im.lo}
__device__ __forceinline__ void fx_multiply(FxAcc& f, const FxHalf& q, int d, const int4* __restrict__ lk, int stride) {
  // w = V h, V = U or U^dag (entry (a, b) at a sa + b sb, imaginary limbs with sign sg)
  const int dir = d & 1, sg = -dir;
  const int sa = (dir ? 1 : 3) * stride, sb = (dir ? 3 : 1) * stride;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    long long H[2][2] = {}, X[2][2] = {};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      int4 U = lk[a * sa + b * sb];
      U.z = (U.z ^ sg) - sg;
      U.w = (U.w ^ sg) - sg;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int rh = q.hh[s][b][0], rl = q.hl[s][b][0], ih = q.hh[s][b][1], il = q.hl[s][b][1];
        fx_mac(H[s][0], U.x, rh);
        fx_mac(X[s][0], U.x, rl);
        fx_mac(X[s][0], U.y, rh);
        fx_mac(H[s][0], U.z, q.nh[s][b]);
        fx_mac(X[s][0], U.z, q.nl[s][b]);
        fx_mac(X[s][0], U.w, q.nh[s][b]);
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
        w[s][p] = H[s][p] + (X[s][p] >> 28);
        f.a[s][a][p] += w[s][p];
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

// 2^(E - 1023 - 58): a unit of the accumulators times the projectors' factor 1/2 (E >= kFxMinExp)
__device__ __forceinline__ double fx_unit(const FxAcc& f) { return __hiloint2double((f.E - 58) << 20, 0); }

// ----------------------------------------------------------------------------
// D_s at one site. dir(d) names direction d's operands (HopDir).
// ----------------------------------------------------------------------------
struct HopDir {
  const Cx<double>* up;  // the neighbour's components that supply spins 0-1, and
  const Cx<double>* lo;  // spins 2-3, cs elements apart
  const int4* fx;        // the link in fixed point and in FP64, entries ls elements apart
  const Cx<double>* u;
};

// one direction in FP64, added to acc (out of line: sites whose neighbours are out of the
// fixed-point range)
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

// 16 bytes of device memory into shared memory, asynchronously
__device__ __forceinline__ void fx_copy(int4* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<unsigned>(__cvta_generic_to_shared(dst))),
               "l"(__cvta_generic_to_global(src))
               : "memory");
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

// returns unit, with unit h = D_s (so that the scale joins the next multiply-add). With S > 1 the S warps
// of a CTA take 6 / S directions each of the same 32 sites and warp 0 adds them up (integers: exactly,
// but for the shift to a common exponent that the six directions of one thread see as well); the others
// have no result. Called by every thread of the CTA; site: whether the thread has one.
template <int S, class Dir>
__device__ __forceinline__ double hop_fx(const Dir& dir, int cs, int ls, bool site, Vec3<double> (&h)[4]) {
  extern __shared__ int4 fx_shared[];
  int4* stage = fx_shared + (threadIdx.x >> 5) * kFxStage + (threadIdx.x & 31);
  constexpr int N = 6 / S;
  const int d0 = S == 1 ? 0 : (threadIdx.x >> 5) * N;
  FxAcc f;
  fx_clear(f);
  auto fetch_spinor = [&](const HopDir& q) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      fx_copy(stage + 32 * c, q.up + (size_t)c * cs);
      fx_copy(stage + 32 * (6 + c), q.lo + (size_t)c * cs);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto fetch_link = [&](const HopDir& q) {
#pragma unroll
    for (int e = 0; e < 9; ++e) fx_copy(stage + 32 * (12 + e), q.fx + (size_t)e * ls);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (site) {
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
      stage[32 * 12] = make_int4(f.E, f.wide, 0, 0);
    }
    __syncthreads();
    if (d0) return 0.0;
    int E[S];
    E[0] = f.E;
#pragma unroll
    for (int p = 1; p < S; ++p) {
      const int4 o = stage[p * kFxStage + 32 * 12];
      E[p] = o.x;
      f.E = max(f.E, o.x);
      f.wide = f.wide || o.y;
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int s0 = min(f.E - E[0], 63);
        f.a[s][c][0] >>= s0;
        f.a[s][c][1] >>= s0;
#pragma unroll
        for (int p = 1; p < S; ++p) {
          const longlong2 o = box[p * kFxStage + 32 * (3 * s + c)];
          const int sp = min(f.E - E[p], 63);
          f.a[s][c][0] += o.x >> sp;
          f.a[s][c][1] += o.y >> sp;
        }
      }
  }
  if (!site) return 0.0;
  if (f.wide) {
    double o[24];
    for (int i = 0; i < 24; ++i) o[i] = 0.0;
#pragma unroll 1
    for (int d = 0; d < 6; ++d) hop_dir_fp64(d, dir(d), cs, ls, o);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) h[s].c[c] = mk<double>(o[2 * (3 * s + c)], o[2 * (3 * s + c) + 1]);
    return 0.5;
  }
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int c = 0; c < 3; ++c) h[s].c[c] = mk<double>((double)f.a[s][c][0], (double)f.a[s][c][1]);
  return fx_unit(f);
}

// Launch shape of a hop over `sites`: run(S, blocks, threads, dynamic shared memory) with the directions
// split over as many warps S (std::integral_constant) as still leaves every CTA resident at once; the
// chain of six spinor and link fetches is what bounds few sites. The Wilson matrix on one parity, us with
// S = 1, 2, 3, 6 (32-site warps): 16 warps 28, 22, 20, 17; 256 27, 21, 19, 17; 512 27, 23, 23, 29;
// 768 34, 27, 34, 40; 1024 33, 32, 37, 49; 1536 42, 44, 49, 68.
template <class Run>
inline void fx_launch(size_t sites, Run&& run) {
  const size_t warps = (sites + 31) / 32;
  auto go = [&](auto S) {
    constexpr int th = FxShape<S.value>::threads, per = S.value == 1 ? th : 32;
    run(S, (unsigned)((sites + per - 1) / per), th, fx_smem(th));
  };
  if (warps <= 152 * FxShape<6>::blocks)
    go(std::integral_constant<int, 6>{});
  else if (warps <= 152 * FxShape<3>::blocks)
    go(std::integral_constant<int, 3>{});
  else if (warps <= 152 * FxShape<2>::blocks)
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
