// Layout conversions between the C-ABI's lexicographic complex128 arrays and the
// internal line layout, gauge ingest, and the per-line wrap-around matrices Lambda.
#include <algorithm>

#include "wf_fixed.cuh"
#include "wf_internal.h"

namespace wf {

constexpr int kThreads = 256;

static inline int nblocks(size_t n, int threads = kThreads) {
  size_t b = (n + threads - 1) / threads;
  return (int)(b > 0x7fffffff ? 0x7fffffff : b);
}

// site index (t, z, y, x) lexicographic with x fastest
__device__ __forceinline__ void site_coords(const Geom& g, size_t site, int& x, int& y, int& z, int& t) {
  x = (int)(site % g.L);
  size_t r = site / g.L;
  y = (int)(r % g.L);
  r /= g.L;
  z = (int)(r % g.L);
  t = (int)(r / g.L);
}

// ----------------------------------------------------------------------------
// Spinor import / export: between the caller's complex128 arrays, [rhs][t][z][y][x][12] (both
// parities) or [rhs][t][l][12] (one parity, "compact"), and the line layout [rhs][l][12][slot] in
// precision R, with the axial frame's colour rotation per site (import psi' = g psi, export
// psi = g^dag psi') and optionally gamma_5 = -[[0, 1], [1, 0]] (spin s <- -(spin s +- 2)).
//
// A caller's site is 192 contiguous bytes, a layout run is consecutive slots of one component, so
// each side wants another thread order. A CTA therefore takes a tile of `tl` lines x `J` lane
// groups (n J consecutive times) x all 12 components through shared memory: the caller's side
// moves as 16-byte pieces, 12 consecutive threads to a site; on the layout's side one thread holds
// one site and consecutive threads consecutive slots (runs of J elements). The rotation of a site
// stays in registers for all sources the CTA loops over. Shared-memory rows of 13 elements keep
// both orders free of bank conflicts.
//
// The rotation's 144 multiply-adds per site would bound these kernels (GB300: two FP64 FMAs per clock
// and SM): FP64 fields rotate in fixed point (rotate3_fx; full field of 24^3 x 128 x
// 12 sources, import 5.1 -> 2.5 ms, export 5.1 -> 2.9; 12^3 x 48 x 4 0.10 -> 0.063 and 0.069 ms), FP32 fields with
// rotate3_split instead, whose products are exact FP32 ones (below). Spins one after another and six
// CTAs per SM: the loads of one CTA overlap the arithmetic of the others (unrolled, at 4 CTAs per SM,
// 1.4 times slower). Measured, one odd field of 24^3 x 128 x 12 sources to and from FP32 (3.1 GB,
// 0.45 ms at the copy bandwidth): import 1.01 ms, export 1.02 ms; 6.39 and 4.34 ms with one thread
// per spin, its scattered elements and the rotation in FP64. One source of 16^3 x 128: 43 and 38 us,
// from 88 and 86.
// ----------------------------------------------------------------------------
constexpr int kTileThreads = 128;
constexpr int kTileMinBlocks = 6;      // resident CTAs per SM
constexpr int kTileRow = NSPIN_C + 1;  // shared-memory elements per site

// Tile of an import / export launch (host: tile_of)
struct SpinorTile {
  int J;      // lane groups per tile (a divisor of lpl)
  int nJ;     // times per tile, n J
  int tl;     // lines per tile (1, 2, 4 or 8)
  int nch;    // time chunks per line, lpl / J
  int ntl;    // line tiles per parity
  int rper;   // sources per CTA
};

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---- FP32 rotation with exact products.
// d = f + lo for a double of magnitude in [2^-80, 2^100) or zero, by integer operations (the
// conversions between FP64 and FP32 run at the FP64 rate): f its sign, exponent and leading 20
// fraction bits, lo the next 23. Returns false (f, lo unset) outside that range.
__device__ __forceinline__ bool split_double(double d, float& f, float& lo) {
  const unsigned hw = (unsigned)__double2hiint(d), lw = (unsigned)__double2loint(d);
  const unsigned a = hw & 0x7fffffffu, sg = hw & 0x80000000u;
  const bool zero = (a | lw) == 0;
  if (!zero && a - (943u << 20) >= (180u << 20)) return false;
  const float sc = __uint_as_float(sg | (((a >> 20) - 939u) << 23));
  f = zero ? 0.f : __uint_as_float(sg | ((a - 0x38000000u) << 3));
  lo = zero ? 0.f : (__uint_as_float(0x4b000000u | (lw >> 9)) - 8388608.f) * sc;
  return true;
}
// exact FP64 value of a finite float by integer operations; subnormal values give zero
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
  const bool z = a < 0x00800000u;
  return __hiloint2double(z ? 0 : (int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), z ? 0 : (int)(b << 29));
}

// A rotation matrix split as h + l, h a multiple of 2^-10 (|g| <= 1: 11 bits)
struct SplitMat {
  Cx<float> h[9], l[9];
};
__device__ __forceinline__ void split_unit(double g, float& h, float& l) {
  float f, lo;
  if (!split_double(g, f, lo)) f = lo = 0.f;  // below 2^-80
  h = (f + 12288.f) - 12288.f;
  l = (f - h) + lo;
}
__device__ __forceinline__ void load_rotation(const Cx<double>* __restrict__ gl, int tp, int sl, SplitMat& G) {
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const Cx<double> e = gl[(size_t)k * tp + sl];
    split_unit(e.re, G.h[k].re, G.l[k].re);
    split_unit(e.im, G.h[k].im, G.l[k].im);
  }
}
// A rotation matrix in fixed point (wf_fixed.cuh): limbs of g 2^58
struct FxMat {
  int2 re[9], im[9];
  bool one;  // the unit matrix (t = 0 of every line): vectors pass unchanged
};
__device__ __forceinline__ int2 fx_limbs(long long v) { return make_int2((int)(v >> 28), (int)v & 0xfffffff); }
__device__ __forceinline__ void load_rotation(const Cx<double>* __restrict__ gl, int tp, int sl, FxMat& G) {
  G.one = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const Cx<double> e = gl[(size_t)k * tp + sl];
    G.re[k] = fx_limbs(fx_from<6>(e.re, 1023));  // |g| <= 1 + 1e-6: exponents up to 1023
    G.im[k] = fx_limbs(fx_from<6>(e.im, 1023));
    G.one = G.one && e.re == (k % 4 ? 0.0 : 1.0) && e.im == 0.0;
  }
}
// w = g v (DAG: g^dag v), the six numbers of v sharing one exponent E. Four spins of a site: about 1100
// integer instructions and 24 conversions against 144 FP64 multiply-adds, i.e. some 20 clocks per site
// and SM against 72. The roundings (v to 2^(E - 57), g to 2^-58, the low limbs' products left out,
// X / 2^28) are below 0.63 x 2^-53 2^E; a component whose terms add up to S in absolute value therefore needs
// S not far below 2^E, as in the hops: all three colours of v reach 2^(E - 4) (then S does, whatever g
// is), or all of w's have. False (w unset) otherwise and outside the fixed-point range. Emulated, errors
// in units of 2^-53 S, root mean square, fixed point : FP64 arithmetic: Gaussian vectors 0.28 : 0.53
// (with v to 2^(E - 55), g to 2^-55 and X / 2^28 rounded down 0.81, half an ulp of it one-sided); colours
// scattered over 2^20, g random 0.39 : 0.72, g near 1 0.48 : 0.75; 2^-4 of each other, g diagonal
// 0.46 : 0.52. With 2^(E - 5) the last would lose (0.59 : 0.53).
constexpr int kRotSpread = 4;
// the larger of two magnitudes' high words
__device__ __forceinline__ unsigned fx_word(double a, double b) {
  return max((unsigned)__double2hiint(a) & 0x7fffffffu, (unsigned)__double2hiint(b) & 0x7fffffffu);
}
template <bool DAG>
__device__ __forceinline__ bool rotate3_fx(const FxMat& G, const double (&v)[6], double (&w)[6]) {
  if (G.one) {
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = v[i];
    return true;
  }
  unsigned mx = 0, mn = ~0u;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const unsigned m = fx_word(v[2 * c], v[2 * c + 1]);
    mx = max(mx, m);
    mn = min(mn, m);
  }
  const int E = (int)(mx >> 20);
  if (mx == 0) {  // zeros, or numbers below 2^-1042
    unsigned low = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      low |= (unsigned)__double2loint(v[i]);
      w[i] = 0.0;
    }
    return low == 0;
  }
  if (E < kFxMinExp || E >= kFxMaxExp) return false;
  int2 h[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) h[i] = fx_limbs(fx_from<5>(v[i], E));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    constexpr long long half = 1LL << 27;  // of X / 2^28, whose shift rounds down
    long long H[2] = {}, X[2] = {half, half};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int2 r = G.re[DAG ? 3 * b + a : 3 * a + b], i = G.im[DAG ? 3 * b + a : 3 * a + b];
      // re: gr vr -+ gi vi, im: gr vi +- gi vr
      const int2 vr = h[2 * b], vi = h[2 * b + 1], m = make_int2(-i.x, -i.y), ir = DAG ? i : m, ii = DAG ? m : i;
      fx_mac(H[0], r.x, vr.x);
      fx_mac(X[0], r.x, vr.y);
      fx_mac(X[0], r.y, vr.x);
      fx_mac(H[0], ir.x, vi.x);
      fx_mac(X[0], ir.x, vi.y);
      fx_mac(X[0], ir.y, vi.x);
      fx_mac(H[1], r.x, vi.x);
      fx_mac(X[1], r.x, vi.y);
      fx_mac(X[1], r.y, vi.x);
      fx_mac(H[1], ii.x, vr.x);
      fx_mac(X[1], ii.x, vr.y);
      fx_mac(X[1], ii.y, vr.x);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      // g v = (H 2^56 + X 2^28) 2^-58 in units of 2^(E - 1023 - 57): H + X / 2^28 in units of 2^(E - 1082)
      const double x = (double)(H[q] + (X[q] >> 28));
      const int hi = __double2hiint(x);
      w[2 * a + q] = __hiloint2double(hi ? hi + ((E - 1082) << 20) : 0, __double2loint(x));
    }
  }
  const int least = E - kRotSpread;
  if ((int)(mn >> 20) >= least) return true;
  bool large = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) large = large && (int)(fx_word(w[2 * c], w[2 * c + 1]) >> 20) >= least;
  return large;
}

// s + c = g v (DAG: g^dag v) for a vector v = f + lo (lo of relative size 2^-20 at most, or zero):
// f is split again at 2^-10 of the vector's largest exponent E, so that each h-h product is an
// integer multiple of one power of two that fits FP32 and their sums are exact; the other
// products, 2^-10 of those, are summed in FP32. The error is about 2^-34 of |v|, against
// 2^-25 for the rounding of an FP32 result: false where that would show, i.e. unless all three colours of v,
// or all of g v, reach 2^(E - 6). Emulated, error of the FP32 result against an FP64 rotation's, root mean
// square: Gaussian vectors +0.0004 %, colours scattered over 2^20 +0.03 % (without the rule, colours
// 2^-10 of each other and g diagonal +57 %).
constexpr int kSplitSpread = 6;
template <bool DAG>
__device__ __forceinline__ bool rotate3_split(const SplitMat& G, const float (&f)[6], const float (&lo)[6],
                                              float (&s)[6], float (&c)[6]) {
  auto word = [](float a, float b) { return max(__float_as_uint(a) & 0x7fffffffu, __float_as_uint(b) & 0x7fffffffu); };
  unsigned mx = 0, mn = ~0u;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const unsigned m = word(f[2 * i], f[2 * i + 1]);
    mx = max(mx, m);
    mn = min(mn, m);
  }
  const unsigned e = mx & 0x7f800000u;
  const float M = e ? __uint_as_float(e + (13u << 23) + 0x00400000u) : 0.f;  // 1.5 x 2^(E + 13)
  float vh[6], vl[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    vh[i] = __fadd_rn(__fadd_rn(f[i], M), -M);
    vl[i] = (f[i] - vh[i]) + lo[i];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float sr = 0.f, si = 0.f, cr = 0.f, ci = 0.f;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const Cx<float> H = DAG ? G.h[3 * b + a] : G.h[3 * a + b], L = DAG ? G.l[3 * b + a] : G.l[3 * a + b];
      const float hi = DAG ? -H.im : H.im, li = DAG ? -L.im : L.im;
      sr = fmaf(H.re, vh[2 * b], sr);
      sr = fmaf(-hi, vh[2 * b + 1], sr);
      si = fmaf(H.re, vh[2 * b + 1], si);
      si = fmaf(hi, vh[2 * b], si);
      const float xr = vh[2 * b] + vl[2 * b], xi = vh[2 * b + 1] + vl[2 * b + 1];
      cr = fmaf(H.re, vl[2 * b], cr);
      cr = fmaf(-hi, vl[2 * b + 1], cr);
      cr = fmaf(L.re, xr, cr);
      cr = fmaf(-li, xi, cr);
      ci = fmaf(H.re, vl[2 * b + 1], ci);
      ci = fmaf(hi, vl[2 * b], ci);
      ci = fmaf(L.re, xi, ci);
      ci = fmaf(li, xr, ci);
    }
    s[2 * a] = sr;
    s[2 * a + 1] = si;
    c[2 * a] = cr;
    c[2 * a + 1] = ci;
  }
  const unsigned least = e ? e - ((unsigned)kSplitSpread << 23) : 0;  // nonzero numbers here are 2^-80 or more
  if (mn >= least) return true;
  bool large = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) large = large && word(s[2 * a], s[2 * a + 1]) >= least;
  return large;
}

// One spin of a site on import: in (shared memory, 3 FP64 elements, negated for gamma_5) rotated by G
// into out (components os elements apart). The _wide forms are the rotation in FP64, out of line, for
// extreme magnitudes, infinities and NaN.
template <typename R>
__device__ __noinline__ void import_spin_wide(const Cx<double>* gl, int tp, const Cx<double>* in, bool neg, Cx<R>* out,
                                              int os) {
  for (int a = 0; a < 3; ++a) {
    Cx<double> w = czero<double>();
    for (int b = 0; b < 3; ++b) w = cfma(w, gl[(size_t)(3 * a + b) * tp], neg ? mk<double>(-in[b].re, -in[b].im) : in[b]);
    out[(size_t)a * os] = mk<R>((R)w.re, (R)w.im);
  }
}
__device__ __forceinline__ void import_spin(const FxMat& G, const Cx<double>* gl, int tp, int sl, const Cx<double>* in,
                                            bool neg, Cx<double>* out, int os) {
  double v[6], w[6];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    v[2 * c] = neg ? -in[c].re : in[c].re;
    v[2 * c + 1] = neg ? -in[c].im : in[c].im;
  }
  if (!rotate3_fx<false>(G, v, w)) {
    import_spin_wide<double>(gl + sl, tp, in, neg, out, os);
    return;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) out[(size_t)c * os] = mk<double>(w[2 * c], w[2 * c + 1]);
}
__device__ __forceinline__ void import_spin(const SplitMat& G, const Cx<double>* gl, int tp, int sl,
                                            const Cx<double>* in, bool neg, Cx<float>* out, int os) {
  float f[6], lo[6];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const Cx<double> v = in[k];
    ok &= split_double(neg ? -v.re : v.re, f[2 * k], lo[2 * k]);
    ok &= split_double(neg ? -v.im : v.im, f[2 * k + 1], lo[2 * k + 1]);
  }
  float s[6], c[6];
  if (!ok || !rotate3_split<false>(G, f, lo, s, c)) {
    import_spin_wide<float>(gl + sl, tp, in, neg, out, os);
    return;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) out[(size_t)k * os] = mk<float>(s[2 * k] + c[2 * k], s[2 * k + 1] + c[2 * k + 1]);
}
// One spin of a site on export: v = in (components os elements apart) rotated by G^dag into out (shared
// memory, 3 FP64 elements)
template <typename R>
__device__ __noinline__ void export_spin_wide(const Cx<double>* gl, int tp, const Cx<R>* in, int os, bool neg,
                                              Cx<double>* out) {
  for (int a = 0; a < 3; ++a) {
    Cx<double> w = czero<double>();
    for (int b = 0; b < 3; ++b) {
      const Cx<R> v = in[(size_t)b * os];
      w = cfmaconj(w, gl[(size_t)(3 * b + a) * tp], mk<double>((double)v.re, (double)v.im));
    }
    out[a] = neg ? mk<double>(-w.re, -w.im) : w;
  }
}
__device__ __forceinline__ void export_spin(const FxMat& G, const Cx<double>* gl, int tp, int sl, const Cx<double>* in,
                                            int os, bool neg, Cx<double>* out) {
  double x[6], w[6];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Cx<double> v = in[(size_t)c * os];
    x[2 * c] = neg ? -v.re : v.re;
    x[2 * c + 1] = neg ? -v.im : v.im;
  }
  if (!rotate3_fx<true>(G, x, w)) {
    export_spin_wide<double>(gl + sl, tp, in, os, neg, out);
    return;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c] = mk<double>(w[2 * c], w[2 * c + 1]);
}
__device__ __forceinline__ void export_spin(const SplitMat& G, const Cx<double>* gl, int tp, int sl,
                                            const Cx<float>* in, int os, bool neg, Cx<double>* out) {
  float f[6];
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const Cx<float> v = in[(size_t)(k >> 1) * os];
    f[k] = k & 1 ? v.im : v.re;
    const unsigned a = __float_as_uint(f[k]) & 0x7fffffffu;
    ok &= a == 0 || (a >= (47u << 23) && a < (227u << 23));  // [2^-80, 2^100)
  }
  const float lo[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  float s[6], c[6];
  if (!ok || !rotate3_split<true>(G, f, lo, s, c)) {
    export_spin_wide<float>(gl + sl, tp, in, os, neg, out);
    return;
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double w = widen(neg ? -s[k] : s[k]) + widen(neg ? -c[k] : c[k]);
    if (k & 1)
      out[k >> 1].im = w;
    else
      out[k >> 1].re = w;
  }
}

template <typename R>
struct RotationOf {
  typedef SplitMat type;
};
template <>
struct RotationOf<double> {
  typedef FxMat type;
};

// Block and thread of a tile launch -> parity, lines and times. Caller's side: thread q < 96 moves
// component q % 12 of the tile's sites s = q / 12, s + 8, ..., site s = tt tl + li; layout's side:
// thread k + (128 / SPL) h holds spins h, h + SPL, .. of row k: line li = k / nJ, slot m lpl + j0 + jj with
// (m, jj) = (k % nJ) / J, % J. SPL = 1 (a thread holds the site), or 4 where the lattice is so small
// that the rotation's serial chain, not the memory, is what a launch waits for.
// EO: the 4-D even-odd fields [rhs][L^3][12][T/2] of wf_eo4d.cu instead of the line layout; "lines" are
// then all L^3 spatial sites, p the 4-D parity, m = 0 and slot h holds t = 2 h + t0.
struct TileAt {
  int p, l0, j0, r0, r1;
  __device__ __forceinline__ TileAt(const SpinorTile& t, int npar, int par, int nrhs) {
    int b = blockIdx.x;
    p = npar == 2 ? b & 1 : par;
    b /= npar;
    l0 = (b % t.ntl) * t.tl;
    j0 = (b / t.ntl) * t.J;
    r0 = blockIdx.y * t.rper;
    r1 = min(nrhs, r0 + t.rper);
  }
};
// one line's places: the caller's site at time t is (origin + t stride) / div
template <bool EO>
struct TileLine {
  size_t origin, stride;
  int t0;             // EO: first time
  int p3, l3;         // 3-D parity and line of the line layout (rotation)
  __device__ __forceinline__ TileLine(const Geom& g, int compact, int p, int l) {
    int x, y, z;
    if (EO) {
      x = l % g.L;
      y = (l / g.L) % g.L;
      z = l / (g.L * g.L);
      t0 = (p + x + y + z) & 1;
      p3 = (x + y + z) & 1;
      l3 = line_of(g, x, y, z);
    } else {
      line_coords(g, p, l, x, y, z);
      t0 = 0;
      p3 = p;
      l3 = l;
    }
    if (!EO && compact) {
      origin = (size_t)l;
      stride = (size_t)g.Nl;
    } else {
      origin = (size_t)x + g.L * ((size_t)y + (size_t)g.L * z);
      stride = (size_t)g.L * g.L * g.L;
    }
  }
  __device__ __forceinline__ size_t site(int compact, int t) const {
    const size_t i = origin + stride * t;
    return EO && compact ? i / 2 : i;
  }
};
template <bool EO>
__device__ __forceinline__ size_t caller_sites(const Geom& g, int compact) {
  const size_t V = (size_t)g.L * g.L * g.L * g.T;
  return compact ? V / 2 : V;
}

// compact: 0 full arrays, 1 arrays of one parity (par: which)
template <typename R, int SPL, bool EO>
__global__ void __launch_bounds__(kTileThreads, kTileMinBlocks)
    k_import_spinor(const Geom g, const SpinorTile t, int compact, int par, const Cx<double>* __restrict__ lex, Cx<R>* even,
                    Cx<R>* odd, int nrhs, int g5, const Cx<double>* g_e, const Cx<double>* g_o) {
  grid_dep();
  __shared__ __align__(16) Cx<double> buf[kTileThreads / SPL * kTileRow];
  const TileAt at(t, compact ? 1 : 2, par, nrhs);
  Cx<R>* dst = at.p ? odd : even;
  if (!dst) return;
  const int q = threadIdx.x, nl = EO ? 2 * g.Nl : g.Nl, os = EO ? g.T / 2 : g.tp;
  const size_t ns = caller_sites<EO>(g, compact);
  // layout's side
  const int row = q % (kTileThreads / SPL), sp0 = q / (kTileThreads / SPL);
  const int li = row / t.nJ, mj = row - li * t.nJ, m = mj / t.J, jj = mj - m * t.J;
  const int l = at.l0 + li, sl = EO ? at.j0 + jj : m * g.lpl + at.j0 + jj;
  const TileLine<EO> mine_at(g, compact, at.p, l < nl ? l : 0);
  const int time = EO ? 2 * sl + mine_at.t0 : (at.j0 + jj) * g.n + m;
  const bool mine = li < t.tl && l < nl && (!EO || sl < os);
  const bool valid = mine && time < g.T;
  const Cx<double>* gr = mine_at.p3 ? g_o : g_e;
  const Cx<double>* gl = gr ? gr + (size_t)mine_at.l3 * 9 * g.tp : nullptr;
  const int gsl = EO ? slot_of(g, valid ? time : 0) : sl;
  typename RotationOf<R>::type G;
  if (valid && gr) load_rotation(gl, g.tp, gsl, G);
  // caller's side
  const int cc = q % 12, cs = q / 12, cli = cs & (t.tl - 1), step = 8 / t.tl;
  const bool mover = q < 96 && at.l0 + cli < nl;
  const TileLine<EO> from(g, compact, at.p, mover ? at.l0 + cli : 0);

  for (int rhs = at.r0; rhs < at.r1; ++rhs) {
    if (mover) {
      const Cx<double>* src = lex + (size_t)rhs * ns * NSPIN_C + cc;
      for (int tt = cs / t.tl; tt < t.nJ; tt += step) {
        const int tm = EO ? 2 * (at.j0 + tt) + from.t0 : at.j0 * g.n + tt;
        if (tm >= g.T) break;
        const int j = EO ? tt : tt / g.n;
        const int to = EO ? cli * t.J + tt : (cli * g.n + (tt - j * g.n)) * t.J + j;  // its row
        cp_async16(&buf[to * kTileRow + cc], src + from.site(compact, tm) * NSPIN_C);
      }
    }
    cp_async_wait_all();
    __syncthreads();
    if (mine) {
      Cx<R>* out = dst + ((size_t)rhs * nl + l) * NSPIN_C * os + sl;
#pragma unroll 1
      for (int i = 0; i < 4 / SPL; ++i) {
        const int sp = sp0 + i * SPL;
        Cx<R>* o = out + (size_t)sp * 3 * os;
        const Cx<double>* in = buf + row * kTileRow + (g5 ? (sp + 2) % 4 : sp) * 3;
        if (valid && gr) {
          import_spin(G, gl, g.tp, gsl, in, g5 != 0, o, os);
        } else {  // the caller's gauge, or padding slots: zero
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const Cx<double> v = valid ? in[c] : czero<double>();
            o[(size_t)c * os] = g5 ? mk<R>((R)-v.re, (R)-v.im) : mk<R>((R)v.re, (R)v.im);
          }
        }
      }
    }
    __syncthreads();
  }
}

template <typename R, int SPL, bool EO>
__global__ void __launch_bounds__(kTileThreads, kTileMinBlocks)
    k_export_spinor(const Geom g, const SpinorTile t, int compact, int par, const Cx<R>* even, const Cx<R>* odd,
                    Cx<double>* __restrict__ lex, int nrhs, int g5, const Cx<double>* g_e, const Cx<double>* g_o) {
  grid_dep();
  __shared__ __align__(16) Cx<double> buf[kTileThreads / SPL * kTileRow];
  const TileAt at(t, compact ? 1 : 2, par, nrhs);
  const Cx<R>* src = at.p ? odd : even;  // null: that parity's sites are zero
  const int q = threadIdx.x, nl = EO ? 2 * g.Nl : g.Nl, os = EO ? g.T / 2 : g.tp;
  const size_t ns = caller_sites<EO>(g, compact);
  const int row = q % (kTileThreads / SPL), sp0 = q / (kTileThreads / SPL);
  const int li = row / t.nJ, mj = row - li * t.nJ, m = mj / t.J, jj = mj - m * t.J;
  const int l = at.l0 + li, sl = EO ? at.j0 + jj : m * g.lpl + at.j0 + jj;
  const TileLine<EO> mine_at(g, compact, at.p, l < nl ? l : 0);
  const int time = EO ? 2 * sl + mine_at.t0 : (at.j0 + jj) * g.n + m;
  const bool valid = li < t.tl && l < nl && (!EO || sl < os) && time < g.T;
  const Cx<double>* gr = mine_at.p3 ? g_o : g_e;
  const Cx<double>* gl = gr ? gr + (size_t)mine_at.l3 * 9 * g.tp : nullptr;
  const int gsl = EO ? slot_of(g, valid ? time : 0) : sl;
  typename RotationOf<R>::type G;
  if (valid && gr && src) load_rotation(gl, g.tp, gsl, G);
  const int cc = q % 12, cs = q / 12, cli = cs & (t.tl - 1), step = 8 / t.tl;
  const bool mover = q < 96 && at.l0 + cli < nl;
  const TileLine<EO> to(g, compact, at.p, mover ? at.l0 + cli : 0);

  for (int rhs = at.r0; rhs < at.r1; ++rhs) {
    if (valid) {
      const Cx<R>* in = src ? src + ((size_t)rhs * nl + l) * NSPIN_C * os + sl : nullptr;
#pragma unroll 1
      for (int i = 0; i < 4 / SPL; ++i) {
        const int sp = sp0 + i * SPL, ss = g5 ? (sp + 2) % 4 : sp;
        Cx<double>* out = buf + row * kTileRow + sp * 3;
        const Cx<R>* from = in + (size_t)ss * 3 * os;
        if (src && gr) {
          export_spin(G, gl, g.tp, gsl, from, os, g5 != 0, out);
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const Cx<R> v = src ? from[(size_t)c * os] : czero<R>();
            const Cx<double> w = mk<double>((double)v.re, (double)v.im);
            out[c] = g5 ? mk<double>(-w.re, -w.im) : w;
          }
        }
      }
    }
    __syncthreads();
    if (mover) {
      Cx<double>* dst = lex + (size_t)rhs * ns * NSPIN_C + cc;
      for (int tt = cs / t.tl; tt < t.nJ; tt += step) {
        const int tm = EO ? 2 * (at.j0 + tt) + to.t0 : at.j0 * g.n + tt;
        if (tm >= g.T) break;
        const int j = EO ? tt : tt / g.n;
        const int from = EO ? cli * t.J + tt : (cli * g.n + (tt - j * g.n)) * t.J + j;
        dst[to.site(compact, tm) * NSPIN_C] = buf[from * kTileRow + cc];
      }
    }
    __syncthreads();
  }
}

// gauge field U[t][z][y][x][mu][row][col] -> U_t per parity [l][9][tp] and forward
// spatial links per parity [mu][l][9][tp]
__global__ void k_import_gauge(const Geom g, const Cx<double>* __restrict__ lex, Cx<double>* ut0, Cx<double>* ut1,
                               Cx<double>* us0, Cx<double>* us1) {
  const size_t V = (size_t)g.L * g.L * g.L * g.T;
  const size_t total = V * 4 * 9;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int k = (int)(i % 9);
    const int mu = (int)((i / 9) % 4);
    const size_t site = i / 36;
    int x, y, z, t;
    site_coords(g, site, x, y, z, t);
    const int p = (x + y + z) & 1;
    const int l = line_of(g, x, y, z);
    const int sl = slot_of(g, t);
    if (mu == 3) {
      Cx<double>* ut = p ? ut1 : ut0;
      ut[((size_t)l * 9 + k) * g.tp + sl] = lex[i];
    } else {
      Cx<double>* us = p ? us1 : us0;
      us[(((size_t)mu * g.Nl + l) * 9 + k) * g.tp + sl] = lex[i];
    }
  }
}

__device__ __forceinline__ Mat3<double> ldmat_d(const Cx<double>* base, int tp, int slot) {
  Mat3<double> U;
#pragma unroll
  for (int k = 0; k < 9; ++k) U.e[k] = base[k * tp + slot];
  return U;
}

// 3x3 inverse by the adjugate; returns |det|
__device__ double inv3(const Mat3<double>& A, Mat3<double>& Ai) {
  const Cx<double>* a = A.e;
  Cx<double> c00 = cmul(a[4], a[8]) - cmul(a[5], a[7]);
  Cx<double> c01 = cmul(a[5], a[6]) - cmul(a[3], a[8]);
  Cx<double> c02 = cmul(a[3], a[7]) - cmul(a[4], a[6]);
  Cx<double> det = cmul(a[0], c00) + cmul(a[1], c01) + cmul(a[2], c02);
  double d2 = det.re * det.re + det.im * det.im;
  Cx<double> id = mk<double>(det.re / d2, -det.im / d2);
  Cx<double> adj[9];
  adj[0] = c00;
  adj[3] = c01;
  adj[6] = c02;
  adj[1] = cmul(a[2], a[7]) - cmul(a[1], a[8]);
  adj[4] = cmul(a[0], a[8]) - cmul(a[2], a[6]);
  adj[7] = cmul(a[1], a[6]) - cmul(a[0], a[7]);
  adj[2] = cmul(a[1], a[5]) - cmul(a[2], a[4]);
  adj[5] = cmul(a[2], a[3]) - cmul(a[0], a[5]);
  adj[8] = cmul(a[0], a[4]) - cmul(a[1], a[3]);
  for (int k = 0; k < 9; ++k) Ai.e[k] = cmul(adj[k], id);
  return sqrt(d2);
}

// Per line: Lambda_b = (I - s mu^-N_t P)^-1, P = U_t(0) U_t(1) ... U_t(N_t-1), closes T^-1;
// Lambda_f = (I - s mu^-N_t Q)^-1, Q = U_t^dag(N_t-2) ... U_t^dag(0) U_t^dag(N_t-1), closes
// T^-dag in the lane-scan formulation (§II.A step 1; X(0) = -s mu^-N_t P).
__global__ void k_tline_init(const Geom g, const Cx<double>* __restrict__ ut, Cx<double>* lamb, Cx<double>* lamf,
                             int* singular) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= g.Nl) return;
  const int T = g.T;
  const Cx<double>* line = ut + (size_t)l * 9 * g.tp;
  Mat3<double> P = ident<double>();
  for (int t = T - 1; t >= 0; --t) P = matmul(ldmat_d(line, g.tp, slot_of(g, t)), P);
  Mat3<double> Q = dagger(ldmat_d(line, g.tp, slot_of(g, T - 1)));
  for (int t = 1; t < T; ++t) Q = matmul(dagger(ldmat_d(line, g.tp, slot_of(g, t - 1))), Q);
  const double f = g.bc * pow(g.mu, -(double)T);
  Mat3<double> Ab, Af, Ib, If;
  for (int k = 0; k < 9; ++k) {
    const double id = (k % 4 == 0) ? 1.0 : 0.0;
    Ab.e[k] = mk<double>(id - f * P.e[k].re, -f * P.e[k].im);
    Af.e[k] = mk<double>(id - f * Q.e[k].re, -f * Q.e[k].im);
  }
  const double db = inv3(Ab, Ib);
  const double df = inv3(Af, If);
  if (!(db > 1e-12) || !(df > 1e-12)) atomicExch(singular, 1);
  for (int k = 0; k < 9; ++k) {
    lamb[(size_t)l * 9 + k] = Ib.e[k];
    lamf[(size_t)l * 9 + k] = If.e[k];
  }
}

// Axial (temporal) frame (§II.C; App. C): per line, g(t) = U_t(0) U_t(1) ... U_t(t-1), g(0) = 1,
// so that U_t'(t) = g(t) U_t(t) g(t+1)^dag = 1 for t < N_t - 1 and U_t'(N_t - 1) = g(N_t - 1) U_t(N_t - 1)
// = P, the Polyakov product; P, Lambda = (1 - s mu^-N_t P)^-1 and the wrap matrix K = P Lambda per
// line, in FP64 and FP32. Lambda is a function of P, so K = Lambda P as well and K^dag = Lambda^dag P^dag
// closes T^-dag. A line's lanes multiply their n sites and scan the products (one thread per
// line took a chain of N_t loads and products, and the links six passes: with them a load of 8^3 x 32 took
// 453 us instead of 135, of 24^3 x 128 8.2 ms instead of 6.1).
__global__ void __launch_bounds__(32) k_axial_frame(const Geom g, const Cx<double>* __restrict__ lex, const AxialOut o,
                                                    int* singular) {
  const int p = blockIdx.y, lane = threadIdx.x, jj = lane % g.lpl, n = g.n, T = g.T;
  const int l_raw = blockIdx.x * g.lpw + lane / g.lpl;
  const bool in = l_raw < g.Nl;
  const int l = in ? l_raw : 0;  // idle lanes still join the shuffles
  int x, y, z;
  line_coords(g, p, l, x, y, z);
  const size_t V3 = (size_t)g.L * g.L * g.L;
  const Cx<double>* u0 = lex + (((size_t)x + g.L * ((size_t)y + (size_t)g.L * z)) * 4 + 3) * 9;
  auto link = [&](int t) {
    Mat3<double> U;
#pragma unroll
    for (int k = 0; k < 9; ++k) U.e[k] = u0[t * V3 * 36 + k];
    return U;
  };
  Mat3<double> c = ident<double>();
  for (int m = 0; m < n; ++m)
    if (jj * n + m < T) c = matmul(c, link(jj * n + m));
  for (int dd = 1; dd < g.lpl; dd <<= 1) {
    Mat3<double> q;
#pragma unroll
    for (int k = 0; k < 9; ++k)
      q.e[k] = mk<double>(shfl_up_r(c.e[k].re, dd, g.lpl), shfl_up_r(c.e[k].im, dd, g.lpl));
    if (jj >= dd) c = matmul(q, c);
  }
  Mat3<double> run;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    run.e[k] = mk<double>(shfl_up_r(c.e[k].re, 1, g.lpl), shfl_up_r(c.e[k].im, 1, g.lpl));
    if (jj == 0) run.e[k] = mk<double>(k % 4 == 0 ? 1.0 : 0.0, 0.0);
  }
  if (!in) return;
  Cx<double>* line = o.g[p] + (size_t)l * 9 * g.tp;
  for (int m = 0; m < n; ++m) {
    if (jj * n + m >= T) break;
#pragma unroll
    for (int k = 0; k < 9; ++k) line[k * g.tp + m * g.lpl + jj] = run.e[k];
    if (m + 1 < n && jj * n + m + 1 < T) run = matmul(run, link(jj * n + m));
  }
  if (jj != g.lpl - 1) return;  // the last lane has the product of the line
  const double f = g.bc * pow(g.mu, -(double)T);
  Mat3<double> A, Ai;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double id = (k % 4 == 0) ? 1.0 : 0.0;
    A.e[k] = mk<double>(id - f * c.e[k].re, -f * c.e[k].im);
  }
  const double det = inv3(A, Ai);
  if (!(det > 1e-12)) atomicExch(singular, 1);
  const Mat3<double> K = matmul(c, Ai);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const size_t at = (size_t)l * 9 + k;
    o.pl[p][at] = c.e[k];
    o.lamb[p][at] = Ai.e[k];
    o.wrap[p][at] = K.e[k];
    o.pl32[p][at] = mk<float>((float)c.e[k].re, (float)c.e[k].im);
    o.lamb32[p][at] = mk<float>((float)Ai.e[k].re, (float)Ai.e[k].im);
    o.wrap32[p][at] = mk<float>((float)K.e[k].re, (float)K.e[k].im);
  }
}

// Spatial links in the axial frame, U_k'(x) = g(x) U_k(x) g(x + k)^dag, from the lexicographic field into the
// three stored forms (FP64, FP32 rows 0 and 1, fixed point): one thread per link and slot, so that the stores
// are contiguous; padding slots zero
__global__ void __launch_bounds__(128) k_axial_links(const Geom g, const Cx<double>* __restrict__ lex, const AxialOut o) {
  const int p = blockIdx.y;
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= (size_t)3 * g.Nl * g.tp) return;
  const int sl = (int)(i % g.tp), l = (int)((i / g.tp) % g.Nl), k = (int)(i / g.tp / g.Nl);
  const int t = (sl % g.lpl) * g.n + sl / g.lpl;
  int x, y, z;
  line_coords(g, p, l, x, y, z);
  Mat3<double> r;
#pragma unroll
  for (int e = 0; e < 9; ++e) r.e[e] = czero<double>();
  if (t < g.T) {
    const Cx<double>* u = lex + (((size_t)x + g.L * ((size_t)y + g.L * ((size_t)z + (size_t)g.L * t))) * 4 + k) * 9;
#pragma unroll
    for (int e = 0; e < 9; ++e) r.e[e] = u[e];
    const int ln = line_of(g, k == 0 ? (x + 1) % g.L : x, k == 1 ? (y + 1) % g.L : y, k == 2 ? (z + 1) % g.L : z);
    r = matmul(ldmat_d(o.g[p] + (size_t)l * 9 * g.tp, g.tp, sl), r);
    r = matmul(r, dagger(ldmat_d(o.g[1 - p] + (size_t)ln * 9 * g.tp, g.tp, sl)));
  }
  const size_t lk = (size_t)k * g.Nl + l;
  constexpr int NC = SpatialLinkNC<float>::value;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    o.us[p][(lk * 9 + e) * g.tp + sl] = r.e[e];
    if (o.usfx[p]) {
      const int2 re = link_limbs(r.e[e].re), im = link_limbs(r.e[e].im);
      o.usfx[p][(lk * 9 + e) * g.tp + sl] = make_int4(re.x, re.y, im.x, im.y);
    }
    if (e < NC) o.us32[p][(lk * NC + e) * g.tp + sl] = mk<float>((float)r.e[e].re, (float)r.e[e].im);
  }
}

__global__ void k_d2f(const Cx<double>* __restrict__ in, Cx<float>* __restrict__ out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = mk<float>((float)in[i].re, (float)in[i].im);
}

static int grid_for(size_t n) {
  int b = nblocks(n);
  return b > kSMs * 16 ? kSMs * 16 : (b < 1 ? 1 : b);
}

// Tile of an import / export over npar parities: about 32 times (runs of 4 to 32 slots) of up to 8
// lines, 128 sites at most; 32 sites with four threads each where that leaves fewer than two CTAs per
// SM (then as few as one line), and all sources of a tile in one CTA (its rotation is then read
// once) only where the tiles alone fill the chip
static SpinorTile tile_of(const Geom& g, int npar, int nrhs, bool eo, dim3& grid, bool& split) {
  SpinorTile t;
  if (eo) {
    t.J = std::min(32, g.T / 2);
    t.nJ = t.J;
    t.nch = (g.T / 2 + t.J - 1) / t.J;
  } else {
    t.J = g.n == 1 ? 32 : g.n == 2 ? 16 : g.n <= 4 ? 8 : 4;
    if (t.J > g.lpl) t.J = g.lpl;
    t.nJ = g.n * t.J;
    t.nch = g.lpl / t.J;
  }
  const int nl = eo ? 2 * g.Nl : g.Nl;
  auto lines = [&](int sites) {
    t.tl = 8;
    while (t.tl > 1 && t.tl * t.nJ > sites) t.tl >>= 1;
    t.ntl = (nl + t.tl - 1) / t.tl;
    return (long long)npar * t.ntl * t.nch;
  };
  long long blocks = lines(kTileThreads);
  split = blocks * nrhs < 2 * kSMs;
  if (split) blocks = lines(kTileThreads / 4);
  long long rgroups = std::min<long long>(nrhs, (8 * kSMs + blocks - 1) / blocks);
  t.rper = (int)((nrhs + rgroups - 1) / rgroups);
  grid = dim3((unsigned)blocks, (unsigned)((nrhs + t.rper - 1) / t.rper));
  return t;
}

// par: -1 full arrays, else arrays of that parity (line layout: the caller's pointers choose it)
template <typename R, bool EO>
static void launch_import_tiles(const Geom& g, int par, const Cx<double>* in, Cx<R>* even, Cx<R>* odd, int nrhs, int g5,
                                const Cx<double>* g_e, const Cx<double>* g_o, cudaStream_t s) {
  dim3 grid;
  bool split;
  const int compact = par >= 0;
  const SpinorTile t = tile_of(g, compact ? 1 : 2, nrhs, EO, grid, split);
  if (split)
    launch_dep(k_import_spinor<R, 4, EO>, grid, kTileThreads, 0, s, g, t, compact, par, in, even, odd, nrhs, g5, g_e, g_o);
  else
    launch_dep(k_import_spinor<R, 1, EO>, grid, kTileThreads, 0, s, g, t, compact, par, in, even, odd, nrhs, g5, g_e, g_o);
  WF_CUDA(cudaGetLastError());
}
template <typename R, bool EO>
static void launch_export_tiles(const Geom& g, int par, const Cx<R>* even, const Cx<R>* odd, Cx<double>* out, int nrhs,
                                int g5, const Cx<double>* g_e, const Cx<double>* g_o, cudaStream_t s) {
  dim3 grid;
  bool split;
  const int compact = par >= 0;
  const SpinorTile t = tile_of(g, compact ? 1 : 2, nrhs, EO, grid, split);
  if (split)
    launch_dep(k_export_spinor<R, 4, EO>, grid, kTileThreads, 0, s, g, t, compact, par, even, odd, out, nrhs, g5, g_e, g_o);
  else
    launch_dep(k_export_spinor<R, 1, EO>, grid, kTileThreads, 0, s, g, t, compact, par, even, odd, out, nrhs, g5, g_e, g_o);
  WF_CUDA(cudaGetLastError());
}

template <typename R>
void launch_import_spinor(const Geom& g, const Cx<double>* lex, Cx<R>* even, Cx<R>* odd, int nrhs, int g5,
                          const Cx<double>* g_e, const Cx<double>* g_o, cudaStream_t s) {
  launch_import_tiles<R, false>(g, -1, lex, even, odd, nrhs, g5, g_e, g_o, s);
}
template <typename R>
void launch_export_spinor(const Geom& g, const Cx<R>* even, const Cx<R>* odd, Cx<double>* lex, int nrhs, int g5,
                          const Cx<double>* g_e, const Cx<double>* g_o, cudaStream_t s) {
  launch_export_tiles<R, false>(g, -1, even, odd, lex, nrhs, g5, g_e, g_o, s);
}
template <typename R>
void launch_import_compact(const Geom& g, const Cx<double>* cmp, Cx<R>* half, int nrhs, int g5,
                           const Cx<double>* gr, cudaStream_t s) {
  launch_import_tiles<R, false>(g, 0, cmp, half, nullptr, nrhs, g5, gr, nullptr, s);
}
template <typename R>
void launch_export_compact(const Geom& g, const Cx<R>* half, Cx<double>* cmp, int nrhs, int g5,
                           const Cx<double>* gr, cudaStream_t s) {
  launch_export_tiles<R, false>(g, 0, half, nullptr, cmp, nrhs, g5, gr, nullptr, s);
}
// 4-D even-odd fields; compact_par < 0: full lexicographic arrays
template <typename R>
void launch_import_eo(const Geom& g, const Cx<double>* lex, Cx<R>* even, Cx<R>* odd, int nrhs, const Cx<double>* g0,
                      const Cx<double>* g1, int compact_par, cudaStream_t s) {
  launch_import_tiles<R, true>(g, compact_par, lex, even, odd, nrhs, 0, g0, g1, s);
}
template <typename R>
void launch_export_eo(const Geom& g, const Cx<R>* even, const Cx<R>* odd, Cx<double>* lex, int nrhs,
                      const Cx<double>* g0, const Cx<double>* g1, int compact_par, cudaStream_t s) {
  launch_export_tiles<R, true>(g, compact_par, even, odd, lex, nrhs, 0, g0, g1, s);
}
#define WF_INST(R)                                                                                          \
  template void launch_import_spinor<R>(const Geom&, const Cx<double>*, Cx<R>*, Cx<R>*, int, int,             \
                                        const Cx<double>*, const Cx<double>*, cudaStream_t);                \
  template void launch_export_spinor<R>(const Geom&, const Cx<R>*, const Cx<R>*, Cx<double>*, int, int,      \
                                        const Cx<double>*, const Cx<double>*, cudaStream_t);                \
  template void launch_import_compact<R>(const Geom&, const Cx<double>*, Cx<R>*, int, int, const Cx<double>*, \
                                         cudaStream_t);                                                     \
  template void launch_export_compact<R>(const Geom&, const Cx<R>*, Cx<double>*, int, int, const Cx<double>*, \
                                         cudaStream_t);                                                     \
  template void launch_import_eo<R>(const Geom&, const Cx<double>*, Cx<R>*, Cx<R>*, int, const Cx<double>*,   \
                                    const Cx<double>*, int, cudaStream_t);                                  \
  template void launch_export_eo<R>(const Geom&, const Cx<R>*, const Cx<R>*, Cx<double>*, int,               \
                                    const Cx<double>*, const Cx<double>*, int, cudaStream_t);
WF_INST(float)
WF_INST(double)
#undef WF_INST

void launch_import_gauge(const Geom& g, const Cx<double>* lex, Cx<double>* ut[2], Cx<double>* us[2], cudaStream_t s) {
  size_t n = (size_t)g.L * g.L * g.L * g.T * 36;
  k_import_gauge<<<grid_for(n), kThreads, 0, s>>>(g, lex, ut[0], ut[1], us[0], us[1]);
  WF_CUDA(cudaGetLastError());
}

void launch_tline_init(const Geom& g, const Cx<double>* ut, Cx<double>* lamb, Cx<double>* lamf, int* singular,
                       cudaStream_t s) {
  k_tline_init<<<(g.Nl + 127) / 128, 128, 0, s>>>(g, ut, lamb, lamf, singular);
  WF_CUDA(cudaGetLastError());
}

void launch_axial_frame(const Geom& g, const Cx<double>* lex, const AxialOut& o, int* singular, cudaStream_t s) {
  k_axial_frame<<<dim3((g.Nl + g.lpw - 1) / g.lpw, 2), 32, 0, s>>>(g, lex, o, singular);
  WF_CUDA(cudaGetLastError());
  const size_t n = (size_t)3 * g.Nl * g.tp;
  k_axial_links<<<dim3((unsigned)((n + 127) / 128), 2), 128, 0, s>>>(g, lex, o);
  WF_CUDA(cudaGetLastError());
}

// FP32 spatial links: rows 0 and 1 of every FP64 link ([3][Nl][9][tp] -> [3][Nl][6][tp])
__global__ void k_d2f_links(const Cx<double>* __restrict__ in, Cx<float>* __restrict__ out, size_t nlinks, int tp) {
  constexpr int NC = SpatialLinkNC<float>::value;
  const size_t total = nlinks * NC * (size_t)tp;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t sl = i % tp;
    const size_t e = (i / tp) % NC;
    const size_t lk = i / ((size_t)tp * NC);
    const Cx<double> v = in[(lk * 9 + e) * tp + sl];
    out[i] = mk<float>((float)v.re, (float)v.im);
  }
}

void launch_d2f_links(const Cx<double>* in, Cx<float>* out, size_t nlinks, int tp, cudaStream_t s) {
  k_d2f_links<<<grid_for(nlinks * SpatialLinkNC<float>::value * (size_t)tp), kThreads, 0, s>>>(in, out, nlinks, tp);
  WF_CUDA(cudaGetLastError());
}

// Gauge-field check at load: every link must be finite and in SU(3) (the FP32 kernels rebuild a
// link's third row from the first two, which holds only for det U = 1 and U^dag U = 1). One
// thread per link; flag |= 1 for a non-finite entry, |= 2 for max |(U^dag U - 1)_ij| or
// |det U - 1| above tol.
__global__ void k_check_links(const Cx<double>* __restrict__ U, size_t nlinks, double tol, int* flag) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= nlinks) return;
  Mat3<double> A;
  bool finite = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    A.e[k] = U[i * 9 + k];
    finite = finite && isfinite(A.e[k].re) && isfinite(A.e[k].im);
  }
  if (!finite) {
    atomicOr(flag, 1);
    return;
  }
  double dev = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      Cx<double> s = czero<double>();  // (U^dag U)_ab = sum_c conj(U_ca) U_cb
#pragma unroll
      for (int c = 0; c < 3; ++c) s = cfmaconj(s, A.e[3 * c + a], A.e[3 * c + b]);
      if (a == b) s.re -= 1.0;
      dev = fmax(dev, fmax(fabs(s.re), fabs(s.im)));
    }
  // det U by cofactors along the first row
  const Cx<double>* e = A.e;
  const Cx<double> m0 = cmul(e[4], e[8]) - cmul(e[5], e[7]);
  const Cx<double> m1 = cmul(e[3], e[8]) - cmul(e[5], e[6]);
  const Cx<double> m2 = cmul(e[3], e[7]) - cmul(e[4], e[6]);
  const Cx<double> det = cmul(e[0], m0) - cmul(e[1], m1) + cmul(e[2], m2);
  dev = fmax(dev, fmax(fabs(det.re - 1.0), fabs(det.im)));
  if (!(dev <= tol)) atomicOr(flag, 2);
}

void launch_check_links(const Cx<double>* U, size_t nlinks, double tol, int* flag, cudaStream_t s) {
  const int threads = 256;
  k_check_links<<<(unsigned)((nlinks + threads - 1) / threads), threads, 0, s>>>(U, nlinks, tol, flag);
  WF_CUDA(cudaGetLastError());
}

void launch_d2f(const Cx<double>* in, Cx<float>* out, size_t n, cudaStream_t s) {
  k_d2f<<<grid_for(n), kThreads, 0, s>>>(in, out, n);
  WF_CUDA(cudaGetLastError());
}

}  // namespace wf
