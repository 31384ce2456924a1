// gm_factor64.cuh -- class sums of one region for the integrands that are
// products of one factor per axis (exponentials and the product peak) or the
// real part of such a product (the cosine): node values from per-axis
// factors.  Shared by the single-integral and the batched FP64 rule kernels.
//
// Bound: the FP64 pipe (one warp instruction in 76 cycles per SM quarter;
// integer and shared-memory instructions beside it are nearly free), so the
// design counts FP64 instructions.  With S = S_0 + Delta_j (+ Delta_k) an
// exponential node is f = F e_j (e_k): F = f(centre), e = exp(-Delta) one of
// six factors per axis (c +- lambda h for three generators), formed once per
// region, and every node's value is one product, formed and added in one go:
// 401 nodes at d = 8 cost 368 products and 49 exponentials instead of 401
// exponentials, 401 chain steps and 401 adds.  The product peak's factors are
// ratios of its per-axis denominators (a reciprocal each); the cosine's are
// rotations (cos Delta, sin Delta), two products per node.  Exponentials, sines
// and class sums run in fixed point on the integer pipes (gmq_families.cuh,
// Limbs below).  Measured at d = 8, 2^20 regions, one thread per region, against
// the outer function at every node: C0 8.14 -> 0.94 ms (4080 -> 278 FP64
// instructions a region), Gaussian 8.25 -> 1.04, product peak 4.71 -> 1.12,
// cosine 10.99 -> 1.42; with factors and FP64 sums and functions they took 2.23,
// 2.34, 2.00 and 3.31 ms.  What is left on the FP64 pipe (46-82 % active) is the
// coordinates, the chains and the weights; twelve warps an SM, as many as the
// workspaces in shared memory let.
//
// Accuracy: F is a common factor of every node, so its error scales the
// region's value and is not amplified by the rule's weights of both signs
// (sum |w| is 5.8 at d = 8), and it is formed beyond FP64 (Centre); the factors
// carry an error near 2^-53 each, whatever their size.  Against 113-bit arithmetic
// (d = 2..16, slopes 0.5 to 300, random boxes and the whole domain) the rms error of
// I7 is 0.01 (cosine) to 1.4 times the separable form's, or, where both are below 2^-53 of
// the terms, up to 1.9 times.
//
// Factors may over- or underflow where f does not (a factor is relative to
// the centre): regions whose factors' exponents do not leave room are
// evaluated by region_sums64, decided from the region alone, so that every
// lane mapping takes the same path.
//
// Classes 4 and 5 (368 of the 401 nodes at d = 8) add their products in fixed
// point on the integer pipes (Limbs below); classes 2 and 3 stay in FP64, one
// leaf per axis (the sum of its two nodes) of the adjacent-pairwise tree, which
// T lanes share in bit-reversed order as in gm_region64.cuh.  Integer sums are
// exact and the tree is fixed, so every lane mapping gives the same bits.
#pragma once

#include <type_traits>

#include "gm_fixed64.cuh"
#include "gm_region64.cuh"

namespace gmq {

// How an integrand factors: kReal: f = F prod e_k (e() below); kRotation:
// f = Re(F prod (cos Delta_k + i sin Delta_k)); kNone: not at all.
enum FacKind { kNone = 0, kReal = 1, kRotation = 2 };

template <int FAM>
struct Fac {
  static constexpr int kind = kNone;
};

// Relative to the centre's, the factor of coordinate c + lam h on axis j is, for
// the product peak, fc over arg(P, j, c, h, lam); for the others, whose phi at the
// centre is fc, it is the exponential of a difference z(lam), |lam| < 1, which is
// formed in fixed point: rounded relative to its own size it would put a factor
// far from 1 (and the F that makes up for it) further from f than the node's own
// inner sum, small where f is large, does.  terms<q>: what z takes from the axis,
// in units of 2^-q (m) and 2^-(q+1) (lin, quad), each an FP64 value and its
// rounding error (low: that of fc); z<q>(x, l): z in units of 2^-q, l = |lam|
// 2^63, neg: lam < 0.  size: the two values whose size limits q.
// Differences c - u enter as they are rounded: no rounding of c + lam h.
struct FacTerms {
  i64 m, lin, quad;
  bool neg, aneg;  // c < u, a < 0 (the kink)
};

// a l 2^-64 for 0 <= l < 2^63; within 1 unit for q = 54, 3 for q = 58
template <int q>
__device__ __forceinline__ i64 lam_mul(i64 a, u64 l) {
  if constexpr (q < 58) return __mul64hi(a, (i64)l);
  return fixed_mul_signed(a, l);
}
template <int q>
__device__ __forceinline__ i64 to_fixed2(double hi, double lo) {
  return to_fixed(hi, q) + to_fixed(lo, q);
}

// z = a |t| - a |t + lam h|
template <>
struct Fac<GMQ_C0> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double low(const PT& P, int j, double c, double fc) {
    return fma(P.a[j], fabs(__dsub_rn(c, P.u[j])), -fc);
  }
  template <class PT>
  __device__ __forceinline__ static void size(const PT& P, int j, double, double h, double fc,
                                              double& x, double& y) {
    x = fc;
    y = __dmul_rn(P.a[j], h);
  }
  template <int q, class PT>
  __device__ __forceinline__ static FacTerms terms(const PT& P, int j, double c, double h,
                                                   double fc) {
    FacTerms t;
    const double ah = __dmul_rn(P.a[j], h);
    t.m = to_fixed2<q>(fc, low(P, j, c, fc));
    t.lin = to_fixed2<q + 1>(ah, fma(P.a[j], h, -ah));
    t.neg = __double2hiint(__dsub_rn(c, P.u[j])) < 0;
    t.aneg = __double2hiint(P.a[j]) < 0;
    return t;
  }
  template <int q>
  __device__ __forceinline__ static i64 z(const FacTerms& t, u64 l, bool neg) {
    const i64 g = lam_mul<q>(t.lin, l);
    i64 v = (t.neg ? -t.m : t.m) + (neg ? -g : g);  // a (t + lam h)
    if ((v < 0) != t.aneg) v = -v;                  // a |t + lam h|
    return t.m - v;
  }
};

// z = -b ((t + lam h)^2 - t^2) = -(lam 2 b h t + lam^2 b h^2), t = c - u
template <>
struct Fac<GMQ_GAUSSIAN> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double low(const PT& P, int j, double c, double fc) {
    const double t = __dsub_rn(c, P.u[j]), t2 = __dmul_rn(t, t);
    return fma(P.b[j], fma(t, t, -t2), fma(P.b[j], t2, -fc));
  }
  template <class PT>
  __device__ __forceinline__ static void size(const PT& P, int j, double c, double h, double,
                                              double& x, double& y) {
    const double t = __dsub_rn(c, P.u[j]), bh = __dmul_rn(P.b[j], h);
    x = __dmul_rn(__dadd_rn(t, t), bh);
    y = __dmul_rn(bh, h);
  }
  template <int q, class PT>
  __device__ __forceinline__ static FacTerms terms(const PT& P, int j, double c, double h,
                                                   double) {
    FacTerms t;
    const double t1 = __dsub_rn(c, P.u[j]), tt = __dadd_rn(t1, t1);
    const double bh = __dmul_rn(P.b[j], h), bl = fma(P.b[j], h, -bh);
    const double x = __dmul_rn(tt, bh), y = __dmul_rn(bh, h);
    t.lin = to_fixed2<q + 1>(x, fma(tt, bl, fma(tt, bh, -x)));
    t.quad = to_fixed2<q + 1>(y, fma(bl, h, fma(bh, h, -y)));
    return t;
  }
  template <int q>
  __device__ __forceinline__ static i64 z(const FacTerms& t, u64 l, bool neg) {
    const i64 g = lam_mul<q>(t.lin, l);
    const i64 s = lam_mul<q>(t.quad, (u64)__umul64hi(l, l) << 1);
    return (neg ? g : -g) - s;
  }
};

// z = lam a h
template <>
struct Fac<GMQ_DISCONTINUOUS> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double low(const PT& P, int j, double c, double fc) {
    return fma(P.a[j], c, -fc);
  }
  template <class PT>
  __device__ __forceinline__ static void size(const PT& P, int j, double, double h, double,
                                              double& x, double& y) {
    x = y = __dmul_rn(P.a[j], h);
  }
  template <int q, class PT>
  __device__ __forceinline__ static FacTerms terms(const PT& P, int j, double, double h, double) {
    FacTerms t;
    const double ah = __dmul_rn(P.a[j], h);
    t.lin = to_fixed2<q + 1>(ah, fma(P.a[j], h, -ah));
    return t;
  }
  template <int q>
  __device__ __forceinline__ static i64 z(const FacTerms& t, u64 l, bool neg) {
    const i64 g = lam_mul<q>(t.lin, l);
    return neg ? -g : g;
  }
};

template <>
struct Fac<GMQ_PRODUCT_PEAK> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double arg(const PT& P, int j, double c, double h,
                                               double lam) {
    const double t = fma(lam, h, __dsub_rn(c, P.u[j]));
    return fma(t, t, P.b[j]);
  }
};

template <>
struct Fac<GMQ_OSCILLATORY> {
  static constexpr int kind = kRotation;
  template <class PT>
  __device__ __forceinline__ static double low(const PT& P, int j, double c, double fc) {
    return fma(P.a[j], c, -fc);
  }
};

static __device__ __noinline__ double rcp_any(double x) { return gm_rcp(x); }

template <int FAM, class PT>
__device__ __forceinline__ i64 low_fixed(const PT& P, int k, double c, double fc) {
  return to_fixed(Fac<FAM>::low(P, k, c, fc), 58);
}

// |lam| in units of 2^-63
__device__ __forceinline__ u64 lam_fixed(double lam) { return (u64)to_fixed(fabs(lam), 63); }

// |x| < 256, tested on the high word
__device__ __forceinline__ bool below_256(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) < 0x40700000u;
}
// The largest |z| of an axis' six factors, from the values of size(), in FP32.
template <int FAM>
__device__ __forceinline__ float largest_z(double x, double y) {
  constexpr float l3 = 0.9486833f;
  if constexpr (FAM == GMQ_GAUSSIAN) return l3 * (abs_f32(x) + l3 * abs_f32(y));
  return l3 * abs_f32(y);
}

// The factors of N coordinates c + lam[i] h.  Which form they take is decided
// for the axis, not for a factor: one test, so that the instructions of N
// exponentials interleave (a test for each kept them one after the other), and a
// factor does not depend on which others it is formed with.
template <int FAM, class PT, int N>
__device__ __forceinline__ void factors(const PT& P, int k, double c, double h, double fc,
                                        const double (&lam)[N], double (&e)[N]) {
  using F = Fac<FAM>;
  if constexpr (Sep<FAM>::kMul) {
    double z[N];
    bool near = true;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      z[i] = F::arg(P, k, c, h, lam[i]);
      near = near && rcp_near(z[i]);
    }
    if (near) {
#pragma unroll
      for (int i = 0; i < N; ++i) e[i] = __dmul_rn(fc, rcp_refined(z[i]));
      return;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) e[i] = __dmul_rn(fc, rcp_any(z[i]));
  } else {
    double x, y;
    F::size(P, k, c, h, fc, x, y);
    if (sincos_near(x) && sincos_near(y)) {  // both below 16: |z| < 31
      const FacTerms t = F::template terms<58>(P, k, c, h, fc);
#pragma unroll
      for (int i = 0; i < N; ++i)
        e[i] = exp_fixed(F::template z<58>(t, lam_fixed(lam[i]), __double2hiint(lam[i]) < 0));
      return;
    }
    // Beyond exp(+-345) = 2^+-498 the axis has no exponent room (kFacExpRoom): 0
    // says so, without an exponential.  In units of 2^-54 below 256; what is left
    // has an exponent near the limit, and its size is all that matters.
    const bool none = !(largest_z<FAM>(x, y) < 345.0f);
    const bool wide = below_256(x) && below_256(y);
    FacTerms t{};
    if (wide) t = F::template terms<54>(P, k, c, h, fc);
#pragma unroll 1
    for (int i = 0; i < N; ++i) {
      double v = 0.0;
      if (wide) {
        const i64 z = F::template z<54>(t, lam_fixed(lam[i]), __double2hiint(lam[i]) < 0);
        v = exp_wide(z << 4, round_shifted(z));
      } else if (!none) {
        const double p = Sep<FAM>::phi(P, k, fma(lam[i], h, c));
        v = gm_exp(FAM == GMQ_DISCONTINUOUS ? __dsub_rn(p, fc) : __dsub_rn(fc, p));
      }
      e[i] = none ? 0.0 : v;
    }
  }
}

// The six factors of an axis: c +- lambda2 h, c +- lambda3 h, c +- lambda5 h.
template <int FAM, class PT>
__device__ __forceinline__ void axis_factors(const PT& P, int k, double c, double h, double fc,
                                             double lam2, double lam3, double lam5,
                                             double (&e)[6]) {
  const double lam[6] = {lam2, -lam2, lam3, -lam3, lam5, -lam5};
  factors<FAM>(P, k, c, h, fc, lam, e);
}

template <int FAM, class PT>
__device__ __forceinline__ double one_factor(const PT& P, int k, double c, double h, double fc,
                                             double lam) {
  const double l[1] = {lam};
  double e[1];
  factors<FAM>(P, k, c, h, fc, l, e);
  return e[0];
}

// F = f(centre) from the axes' phi in order.  Its error is common to every
// node, so the inner sum is kept in units of 2^-58, roundings of phi included, as
// a 64-bit integer modulo 2^64 (for |S| < 512 and every |phi| < 512, where the
// rounded S tells the multiple of 64; in FP64 otherwise), and the product peak's
// product as a sum of two doubles.
template <int FAM>
struct Centre {
  double S, lo = 0.0;
  i64 v = 0;
  bool fixed = true;
  template <class PT>
  __device__ __forceinline__ void add(const PT& P, int k, double c, double fc) {
    using SF = Sep<FAM>;
    if constexpr (SF::kMul) {
      if (k == 0) {
        S = fc;
      } else {
        const double p = __dmul_rn(S, fc);
        lo = fma(lo, fc, fma(S, fc, -p));
        S = p;
      }
    } else {
      if (k == 0) {
        S = SF::kBase ? __dadd_rn(SF::base(P), fc) : fc;
        if (SF::kBase) take(SF::base(P));
      } else {
        S = __dadd_rn(S, fc);
      }
      take(fc);
      v += low_fixed<FAM>(P, k, c, fc);
    }
  }
  __device__ __forceinline__ void take(double x) {
    v += to_fixed(x, 58);
    fixed = fixed && small(x);
  }
  __device__ __forceinline__ static bool small(double x) {  // |x| < 512
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) < 0x40800000u;
  }
  __device__ __forceinline__ double value(int d) const {
    if constexpr (Sep<FAM>::kMul) {
      const double r = Sep<FAM>::g(d, S);
      return fma(-__dmul_rn(r, lo), r, r);
    } else {
      if (!fixed || !small(S)) return Sep<FAM>::g(d, S);
      const i64 x = FAM == GMQ_DISCONTINUOUS ? v : -v;
      if (sincos_near(S)) return exp_fixed(x);  // |S| < 16
      const int n = round_mul_int(S, 1.44269504f);
      return exp_wide(x, FAM == GMQ_DISCONTINUOUS ? n : -n);
    }
  }
  __device__ __forceinline__ void sincos(double& sn, double& cs) const {
    if (!fixed || !small(S)) {
      gm_sincos(S, &sn, &cs);
      return;
    }
    // less the whole turns (2 pi 2^58 = L + L1 2^-32) that a rounded S of 16 and
    // more tells
    const i64 L = 0x1921fb54442d1846ll;
    const int n = sincos_near(S) ? 0 : round_mul_int(S, 0.159154943f);
    sincos_fixed(v - n * L - (((i64)n * 0x9898cc51ll) >> 32), 58, &sn, &cs);
  }
};

// Workspace of one region (entries `ws` doubles apart): the lambda3 factors
// E3 [2d], for kReal their axes' exponents [d], and the class-5 chains A, B, C; with T > 1 lanes also phi at the
// centre [d], the factors of lambda2 and lambda5 [2d each] and F [2].  For
// kReal, chains over axes [0, a), [a, a + b), [a + b, d) of the factors of
// c +- lambda5 h.  For kRotation every factor is two entries (cosine, sine
// of the + sign; - is its conjugate) and every chain entry is two, A's
// chains headed by F.
// The rotation's chains have three parts from d = 8 on: 56 words a region
// instead of 80 put twelve warps on an SM, not eight.
__host__ __device__ constexpr int fac_c(int kind, int d) {
  return kind == kRotation && d == 8 ? 2 : sep_c(d);
}
__host__ __device__ constexpr int fac_b(int kind, int d) {
  return kind == kRotation && d == 8 ? 3 : sep_b(d);
}
__host__ __device__ constexpr int fac_a(int kind, int d) {
  return d - fac_b(kind, d) - fac_c(kind, d);
}

struct FacLayout {
  int e3, x3, A, B, C, phiC, e2, e5, F, words;
};

__host__ __device__ constexpr FacLayout fac_layout(int d, int kind, bool lanes) {
  FacLayout s{};
  const int m = kind == kRotation ? 2 : 1;
  s.e3 = 0;
  s.x3 = 2 * d;
  s.A = kind == kRotation ? 2 * d : 3 * d;
  const int b = fac_b(kind, d), c = fac_c(kind, d);
  s.B = s.A + m * (1 << fac_a(kind, d));
  s.C = s.B + (b ? m * (1 << b) : 0);
  int w = s.C + (c ? m * (1 << c) : 0);
  s.phiC = s.e2 = s.e5 = s.F = -1;
  if (lanes) {
    s.phiC = w;
    s.e2 = w + d;
    s.e5 = w + 3 * d;
    s.F = w + 5 * d;
    w += 5 * d + 2;
  }
  s.words = w;
  return s;
}

// The largest dimension whose rotation tables (twice as many words as the
// real ones) fit a block of 128 one-thread regions; above it the cosine
// keeps the separable form, whatever the lane mapping.
constexpr int kFacRotationMaxDim = 14;

__host__ __device__ constexpr bool fac_used(int kind, int d) {
  return kind == kReal || (kind == kRotation && d <= kFacRotationMaxDim);
}

// Words of one region's workspace: the factored and the separable form
// share it (a region uses one, or first one and then the other; the cosine
// never both).
__host__ __device__ constexpr int region64_words(int d, int kind, bool flag, bool lanes) {
  if (kind == kRotation && fac_used(kind, d)) return fac_layout(d, kind, lanes).words;
  const int s = sep_layout(d, flag, lanes).words;
  const int f = fac_used(kind, d) ? fac_layout(d, kind, lanes).words : 0;
  return s > f ? s : f;
}

// The largest workspace over dimensions 1 .. dmax (batched kernels).
__host__ __device__ constexpr int region64_words_max(int dmax, int kind, bool flag, bool lanes) {
  int m = 0;
  for (int d = 1; d <= dmax; ++d) {
    const int w = region64_words(d, kind, flag, lanes);
    if (w > m) m = w;
  }
  return m;
}

// Room for the factors: exponents of the factors' largest products and of F
// within +-2^9 each, so that no product of an integrand value's parts leaves
// the normal range.
constexpr int kFacExpRoom = 480;

__device__ __forceinline__ int exp_magnitude(double v) {
  const int e = ((__double2hiint(v) >> 20) & 0x7ff) - 1023;
  return e < 0 ? -e : e;
}

// A factor, or -0 where the discontinuous family's f is 0 (a flagged
// coordinate): every product with it is then 0, it bounds no table's exponent,
// and its sign tells it from a factor that underflowed.
template <int FAM, class PT>
__device__ __forceinline__ double flag_factor(const PT& P, int k, double c, double h, double lam,
                                              double e) {
  if constexpr (Sep<FAM>::kFlag) {
    if (Sep<FAM>::flag(P, k, fma(lam, h, c))) return -0.0;
  }
  return e;
}
__device__ __forceinline__ int factor_room(double e) {
  return __double2hiint(e) == (int)0x80000000u ? 0 : exp_magnitude(e);
}

// Class sums as sums of products of two 53-bit fixed-point numbers.  A number
// is v 2^(53 - E) rounded, in two signed limbs h 2^27 + l (|h| <= 2^26, |l| <=
// 2^26); 2^E bounds the table it comes from, so its error is at most 2^-54 of
// the table's largest entry, an FP64 rounding of that entry.  A product is
// h h' 2^54 + (h l' + l h') 2^27 + l l'; the first two terms are three
// multiply-adds to 64 bits (12 cycles of an SM quarter against 76 for an FP64
// instruction), the third, up to 2^-54 of the largest product, is added for all
// products of two tables at once (sum l times sum l': left out, 2^12 products
// with a few large ones are 1e-15 off).  Sums are exact integers: no order of
// the nodes and no lane mapping changes a bit.
struct Limbs {
  int h, l;
};

__device__ __forceinline__ Limbs limbs_split(i64 q) {
  Limbs r;
  r.l = ((int)q << 5) >> 5;
  r.h = (int)((q - r.l) >> 27);
  return r;
}
__device__ __forceinline__ double limbs_pack(Limbs v) { return __hiloint2double(v.h, v.l); }
__device__ __forceinline__ Limbs limbs_unpack(double w) {
  Limbs r;
  r.h = __double2hiint(w);
  r.l = __double2loint(w);
  return r;
}
// |v| <= 2^E; ties away from zero, for the rotation's entries of both signs
__device__ __forceinline__ double limbs_of(double v, int E) {
  return limbs_pack(limbs_split(to_fixed(v, 53 - E)));
}
// x 2^-k rounded to nearest, to even on ties (for k < 32), 0 <= k <= 62
__device__ __forceinline__ i64 shift_even(i64 x, int k) {
  const i64 r = x + (((i64)1 << k) >> 1);
  const i64 q = r >> k;
  const bool tie = k > 0 && ((unsigned)r & ((1u << min(k, 31)) - 1u)) == 0u;
  return tie ? q & ~(i64)1 : q;
}
// |v| < 2^E; ties to even: entries of one sign lose the one or two bits by which
// they are below the table's largest, and ties rounded up put 0.6 to 0.9 of 2^-53
// on the class sums
__device__ __forceinline__ double limbs_even(double v, int E) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff, k = E + 1022 - e;
  const i64 m = ((i64)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  const i64 q = k < 56 ? shift_even(m, k) : 0;
  return limbs_pack(limbs_split(hi < 0 ? -q : q));
}

constexpr int kLimbRun = 512;  // products that a LimbAcc takes before it may overflow

struct LimbAcc {
  i64 hh = 0, mid = 0;
  __device__ __forceinline__ void add(Limbs a, Limbs b) {
    hh += (i64)a.h * b.h;
    mid += (i64)a.h * b.l;
    mid += (i64)a.l * b.h;
  }
  // the same for a b that was just split from a product (mad_wide)
  __device__ __forceinline__ void add_split(Limbs a, Limbs b) {
    mad_wide(hh, a.h, b.h);
    mad_wide(mid, a.h, b.l);
    mad_wide(mid, a.l, b.h);
  }
  __device__ __forceinline__ void sub(Limbs a, Limbs b) {
    hh -= (i64)a.h * b.h;
    mid -= (i64)a.h * b.l;
    mid -= (i64)a.l * b.h;
  }
  // the sum as one number in units of 2^-53 of the products' bound, rounded (for
  // up to 64 products)
  __device__ __forceinline__ i64 number() const { return (hh << 1) + ((mid + (1 << 25)) >> 26); }
  // a b as a number of the same kind; what was rounded off, in units of 2^-37 of
  // its last place, is added to rest
  __device__ __forceinline__ static Limbs product(Limbs a, Limbs b, i64& rest) {
    LimbAcc r;
    r.add(a, b);
    const i64 up = (r.mid + (1 << 25)) >> 26;
    rest += (((r.mid - (up << 26)) << 27) + (i64)a.l * b.l) >> 16;
    return limbs_split((r.hh << 1) + up);
  }
};

// 128-bit total of LimbAccs, in units of 2^27 products' last places.
struct LimbSum {
  i64 hi = 0;
  u64 lo = 0;
  __device__ __forceinline__ void add(i64 h, u64 l) {
    lo += l;
    hi += h + (lo < l ? 1 : 0);
  }
  __device__ __forceinline__ void take(LimbAcc& a) {
    add(a.hh >> 37, (u64)a.hh << 27);
    add(a.mid >> 63, (u64)a.mid);
    a.hh = 0;
    a.mid = 0;
  }
  // x y 2^-k, 0 < k < 64
  __device__ __forceinline__ void add_product(i64 x, i64 y, int k) {
    const i64 h = __mul64hi(x, y);
    const u64 l = (u64)x * (u64)y;
    add(h >> k, (l >> k) | ((u64)h << (64 - k)));
  }
  // x 2^(48 - k), k >= 0
  __device__ __forceinline__ void add_scaled(i64 x, int k) {
    const int r = k - 48;
    add(x >> min(16 + k, 63), r < 0 ? (u64)x << -r : (u64)(x >> min(r, 63)));
  }
  // times 2^(E - 79): E the sum of the two tables' bounds
  __device__ __forceinline__ double value(int E) const {
    const double v = fma((double)hi, 0x1p64, (double)lo);
    return __dmul_rn(v, __hiloint2double((944 + max(E, -900)) << 20, 0));  // 2^(E - 79)
  }
};

template <int T>
__device__ __forceinline__ void lanes_add(LimbSum& x, unsigned mask) {
  if constexpr (T > 32) {
    __shared__ i64 sh[T];
    __shared__ u64 sl[T];
    const int l = threadIdx.x & (T - 1);
#pragma unroll
    for (int off = T / 2; off >= 32; off >>= 1) {
      __syncthreads();
      sh[l] = x.hi;
      sl[l] = x.lo;
      __syncthreads();
      x.add(sh[l ^ off], sl[l ^ off]);
    }
  }
  constexpr int W = T < 32 ? T : 32;
#pragma unroll
  for (int off = W / 2; off > 0; off >>= 1) {
    const i64 h = __shfl_xor_sync(mask, x.hi, off, W);
    const u64 l = __shfl_xor_sync(mask, x.lo, off, W);
    x.add(h, l);
  }
}

// Two 64-bit sums over the group, in every lane.
template <int T>
__device__ __forceinline__ void lanes_add(i64& x, i64& y, unsigned mask) {
  if constexpr (T > 32) {
    __shared__ i64 sx[T], sy[T];
    const int l = threadIdx.x & (T - 1);
#pragma unroll
    for (int off = T / 2; off >= 32; off >>= 1) {
      __syncthreads();
      sx[l] = x;
      sy[l] = y;
      __syncthreads();
      x += sx[l ^ off];
      y += sy[l ^ off];
    }
  }
  constexpr int W = T < 32 ? T : 32;
#pragma unroll
  for (int off = W / 2; off > 0; off >>= 1) {
    x += __shfl_xor_sync(mask, x, off, W);
    y += __shfl_xor_sync(mask, y, off, W);
  }
}

// What is left out of a class-5 sum, from sums over its tables: the products of
// low limbs, and above d = 8 what the products B C were rounded by times the A
// they are multiplied with (its high limbs: the rest is 2^-27 of that).
struct LimbRest {
  i64 la = 0, lb = 0, ha = 0, rb = 0;  // sums of A's l, B's l, A's h, B C's rests
  __device__ __forceinline__ void add_to(LimbSum& s) const {
    s.add_product(la, lb, 27);
    s.add_product(ha, rb, 37);
  }
};

// Exponent E with v < 2^E; a zero (a flagged factor), below every factor with
// room, gets one that leaves its fixed-point value 0.
__device__ __forceinline__ int exp_bound(double v) {
  return max(((__double2hiint(v) >> 20) & 0x7ff) - 1022, -900);
}

// The leaves that a lane of T owns when a tree has 2^lg leaf positions:
// [p0, p0 + cnt), bit-reversed as the butterfly of lanes_tree expects; with
// fewer leaves than lanes, lane l < 2^lg owns one.
template <int T>
__device__ __forceinline__ void lane_leaves(int lane, int lg, int& p0, int& cnt) {
  if constexpr (T == 1) {
    p0 = 0;
    cnt = 1 << lg;
  } else {
    constexpr int bits = ilog2c(T);
    if (lg >= bits) {
      cnt = 1 << (lg - bits);
      p0 = cnt * (int)(__brev((unsigned)lane) >> (32 - bits));
    } else {
      cnt = lane < (1 << lg) ? 1 : 0;
      p0 = lg ? (int)(__brev((unsigned)lane) >> (32 - lg)) : 0;
    }
  }
}

__device__ __forceinline__ int lg_ceil(int n) { return n <= 1 ? 0 : 32 - __clz(n - 1); }

// Class 5 of the real factors by one thread: pattern m = (m_A, hi), value A[m_A]
// B[hi] (above d = 8 A[m_A] (B[.] C[.])); CH entries of A stay in registers while
// hi runs, so a product costs one shared-memory read in CH.
template <int CH, class WF>
__device__ __forceinline__ void fac_class5(const WF& W, const FacLayout& Ly, int pa, int pb,
                                           LimbSum& sum) {
  const int nA = 1 << pa, nB = 1 << pb;
  int la = 0, lb = 0;  // at most 16 entries each
  LimbAcc acc;         // at most 256 products
  for (int lo = 0; lo < nA; lo += CH) {
    Limbs a[CH];
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      a[i] = limbs_unpack(W(Ly.A + lo + i));
      la += a[i].l;
    }
    lb = 0;  // the same for every stretch of A
    for (int hi = 0; hi < nB; ++hi) {
      const Limbs b = limbs_unpack(W(Ly.B + hi));
      lb += b.l;
#pragma unroll
      for (int i = 0; i < CH; ++i) acc.add(a[i], b);
    }
  }
  acc.mid += ((i64)la * lb) >> 27;
  sum.take(acc);
}
// above d = 8
template <int CH, class WF>
__device__ __forceinline__ void fac_class5c(const WF& W, const FacLayout& Ly, int pa, int pb,
                                            int pc, LimbSum& sum) {
  const int nA = 1 << pa, nhi = 1 << (pb + pc), bm = (1 << pb) - 1;
  LimbRest rest;
  for (int lo = 0; lo < nA; lo += CH) {
    Limbs a[CH];
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      a[i] = limbs_unpack(W(Ly.A + lo + i));
      rest.la += a[i].l;
      rest.ha += a[i].h;
    }
    LimbAcc acc;
    rest.lb = rest.rb = 0;
    for (int hi = 0; hi < nhi; ++hi) {
      const Limbs b = LimbAcc::product(limbs_unpack(W(Ly.B + (hi & bm))),
                                       limbs_unpack(W(Ly.C + (hi >> pb))), rest.rb);
      rest.lb += b.l;
#pragma unroll
      for (int i = 0; i < CH; ++i) acc.add_split(a[i], b);
      if (((hi + 1) & (kLimbRun / CH - 1)) == 0) sum.take(acc);
    }
    sum.take(acc);
  }
  rest.add_to(sum);
}

// Class sums and split axis of one region from per-axis factors (kReal);
// arguments as region_sums64.  False: the factors lack exponent room and
// nothing was written to `o` (every lane of the group returns the same).
template <int FAM, int T, class PT, class CH>
__device__ __forceinline__ bool region_sums64_real(const PT& P, int d, const unsigned short* pairs,
                                                   const CH& ch, double lam2, double lam3,
                                                   double lam5, double* w, int ws, double ratio,
                                                   RegionSums& o) {
  using SF = Sep<FAM>;
  const int lane = (T == 1) ? 0 : (int)(threadIdx.x & (unsigned)(T - 1));
  const unsigned mask = group_mask<T>();
  const FacLayout Ly = fac_layout(d, kReal, T > 1);
  const int pa = sep_a(d), pb = sep_b(d), pc = sep_c(d);
  auto W = [&](int e) -> double& { return w[(long long)e * ws]; };
  unsigned zc = 0u;  // discontinuous family: the axes whose centre is flagged
  double F, s2, s3, dbest = -1.0;  // class sums and differences relative to F
  int kbest = 0, room = 0;
  unsigned top5 = 0;  // bit k: axis k's larger lambda5 factor is the - one
  // first axis and length of the chain part that axis k belongs to
  auto part = [&](int k, int& e0, int& i) {
    e0 = k < pa ? Ly.A : (k < pa + pb ? Ly.B : Ly.C);
    i = k < pa ? k : (k < pa + pb ? k - pa : k - pa - pb);
  };
  // sums of an axis's node pairs and its fourth difference
  auto axis = [&](int k, double p2, double m2, double p3, double m3, double& q2, double& q3) {
    double f0 = 1.0;
    if constexpr (SF::kFlag) {
      if (zc & ~(1u << k)) p2 = m2 = p3 = m3 = 0.0;
      if (zc) f0 = 0.0;
    }
    q2 = __dadd_rn(p2, m2);
    q3 = __dadd_rn(p3, m3);
    const double two_f0 = f0 + f0;
    const double D = fabs(__dsub_rn(__dsub_rn(q2, two_f0),
                                    __dmul_rn(ratio, __dsub_rn(q3, two_f0))));
    // D >= 0: the order of the bit patterns
    if (__double_as_longlong(D) > __double_as_longlong(dbest)) {
      dbest = D;
      kbest = k;
    }
  };
  if constexpr (SF::kFlag) {
    for (int k = 0; k < d; ++k) {
      double c, h;
      ch(k, c, h);
      zc |= (unsigned)SF::flag(P, k, c) << k;
    }
  }
  if constexpr (T == 1) {
    PairTree t2, t3;
    Centre<FAM> top;
    for (int k = 0; k < d; ++k) {
      // (no return from here: lanes that left the loop at different axes would
      // run what follows one group after the other; the product peak's factors
      // hardly ever lack room, and the test costs it 6 %)
      if (!SF::kMul && room > kFacExpRoom) continue;
      double c, h;
      ch(k, c, h);
      const double fc = SF::phi(P, k, c);
      top.add(P, k, c, fc);
      double e[6];
      axis_factors<FAM>(P, k, c, h, fc, lam2, lam3, lam5, e);
      const double p2 = flag_factor<FAM>(P, k, c, h, lam2, e[0]);
      const double m2 = flag_factor<FAM>(P, k, c, h, -lam2, e[1]);
      const double p3 = flag_factor<FAM>(P, k, c, h, lam3, e[2]);
      const double m3 = flag_factor<FAM>(P, k, c, h, -lam3, e[3]);
      const double p5 = flag_factor<FAM>(P, k, c, h, lam5, e[4]);
      const double m5 = flag_factor<FAM>(P, k, c, h, -lam5, e[5]);
      room += max(max(factor_room(p2), factor_room(m2)),
                  max(max(factor_room(p3), factor_room(m3)),
                      max(factor_room(p5), factor_room(m5))));
      W(Ly.e3 + 2 * k) = p3;
      W(Ly.e3 + 2 * k + 1) = m3;
      top5 |= (unsigned)(__double_as_longlong(m5) > __double_as_longlong(p5)) << k;
      double q2, q3;
      axis(k, p2, m2, p3, m3, q2, q3);
      t2.push(q2);
      t3.push(q3);
      // the part's class-5 chains, by doubling
      int e0, i;
      part(k, e0, i);
      if (i == 0) {
        W(e0) = p5;
        W(e0 + 1) = m5;
      } else {
        const int n = 1 << i;
        for (int t = 0; t < n; ++t) {
          const double v = W(e0 + t);
          W(e0 + t + n) = __dmul_rn(v, m5);
          W(e0 + t) = __dmul_rn(v, p5);
        }
      }
    }
    F = top.value(d);
    bool pr;
    s2 = t2.flush(pr);
    s3 = t3.flush(pr);
    if (room > kFacExpRoom || exp_magnitude(F) > kFacExpRoom) return false;
  } else {
    // 1. lanes over the 6 d factors: row r of axis k: +-lambda2, +-lambda3,
    //    +-lambda5
    int big = 0;
    for (int t = lane; t < 6 * d; t += T) {
      const int k = t / 6, r = t - 6 * k;
      double c, h;
      ch(k, c, h);
      const double lam = r < 2 ? lam2 : (r < 4 ? lam3 : lam5);
      const double fc = SF::phi(P, k, c);
      const double ls = (r & 1) ? -lam : lam;
      const double e =
          flag_factor<FAM>(P, k, c, h, ls, one_factor<FAM>(P, k, c, h, fc, ls));
      W((r < 2 ? Ly.e2 : (r < 4 ? Ly.e3 : Ly.e5)) + 2 * k + (r & 1)) = e;
      if (r == 0) W(Ly.phiC + k) = fc;
    }
    group_sync<T>(mask);
    // 2. lanes over the tasks: F (and its room, by the lane that forms it)
    //    and every class-5 chain, left to right
    const int nA = 1 << pa, nB = pb ? 1 << pb : 0, nC = pc ? 1 << pc : 0;
    for (int t = lane; t < 1 + nA + nB + nC; t += T) {
      if (t == 0) {
        Centre<FAM> top;
        for (int k = 0; k < d; ++k) {
          double c, h;
          ch(k, c, h);
          top.add(P, k, c, W(Ly.phiC + k));
        }
        const double Fv = top.value(d);
        for (int k = 0; k < d; ++k) {
          int m = 0;
#pragma unroll
          for (int s = 0; s < 2; ++s)
            m = max(m, max(factor_room(W(Ly.e2 + 2 * k + s)),
                           max(factor_room(W(Ly.e3 + 2 * k + s)),
                               factor_room(W(Ly.e5 + 2 * k + s)))));
          big += m;
        }
        W(Ly.F) = Fv;
        W(Ly.F + 1) = (big > kFacExpRoom || exp_magnitude(Fv) > kFacExpRoom) ? 1.0 : 0.0;
      } else {
        int e = t - 1, e0 = Ly.A, j0 = 0, nb = pa;
        if (e >= nA) {
          e -= nA;
          e0 = Ly.B;
          j0 = pa;
          nb = pb;
          if (e >= nB) {
            e -= nB;
            e0 = Ly.C;
            j0 = pa + pb;
            nb = pc;
          }
        }
        double acc = W(Ly.e5 + 2 * j0 + (e & 1));
        for (int i = 1; i < nb; ++i)
          acc = __dmul_rn(acc, W(Ly.e5 + 2 * (j0 + i) + ((e >> i) & 1)));
        W(e0 + e) = acc;
      }
    }
    group_sync<T>(mask);
    F = W(Ly.F);
    if (__double2hiint(W(Ly.F + 1)) != 0) {
      group_sync<T>(mask);  // every lane has read the verdict before the workspace is used again
      return false;
    }
    // 3. lanes over the axes (leaf positions of the trees of classes 2, 3)
    PairTree t2, t3;
    int p0, cnt;
    lane_leaves<T>(lane, lg_ceil(d), p0, cnt);
    const int p1 = min(p0 + cnt, d);
    for (int k = p0; k < p1; ++k) {
      double q2, q3;
      axis(k, W(Ly.e2 + 2 * k), W(Ly.e2 + 2 * k + 1), W(Ly.e3 + 2 * k), W(Ly.e3 + 2 * k + 1), q2,
           q3);
      t2.push(q2);
      t3.push(q3);
    }
    lanes_argmax<T>(dbest, kbest, mask);
    bool pr2, pr3;
    const double x2 = t2.flush(pr2), x3 = t3.flush(pr3);
    s2 = lanes_tree<T>(x2, pr2, mask);
    s3 = lanes_tree<T>(x3, pr3, mask);
    for (int k = 0; k < d; ++k)
      top5 |= (unsigned)(__double_as_longlong(W(Ly.e5 + 2 * k + 1)) >
                         __double_as_longlong(W(Ly.e5 + 2 * k))) << k;
  }
  // the tables as limbs: the lambda3 factors, an exponent for each axis, and
  // the chains, whose largest entry is the product of the larger factors
  const int nA = 1 << pa, nB = pb ? 1 << pb : 0, nC = pc ? 1 << pc : 0;
  const int EA = exp_bound(W(Ly.A + (int)(top5 & (unsigned)(nA - 1))));
  const int EB = pb ? exp_bound(W(Ly.B + (int)((top5 >> pa) & (unsigned)(nB - 1)))) : 0;
  const int EC = pc ? exp_bound(W(Ly.C + (int)(top5 >> (pa + pb)))) : 0;
  if constexpr (T > 1) group_sync<T>(mask);  // every lane has read the doubles
  int M1 = -4096, M2 = -4096;                // the two largest exponents of E3's axes
  for (int k = lane; k < d; k += T) {
    const double p3 = W(Ly.e3 + 2 * k), m3 = W(Ly.e3 + 2 * k + 1);
    const int E = max(exp_bound(p3), exp_bound(m3));
    W(Ly.e3 + 2 * k) = limbs_even(p3, E);
    W(Ly.e3 + 2 * k + 1) = limbs_even(m3, E);
    W(Ly.x3 + k) = __hiloint2double(E, 0);
    M2 = max(M2, min(M1, E));
    M1 = max(M1, E);
  }
  for (int q = lane; q < nA + nB + nC; q += T)
    W(Ly.A + q) = limbs_even(W(Ly.A + q), q < nA ? EA : (q < nA + nB ? EB : EC));
  if constexpr (T > 1) group_sync<T>(mask);
  if constexpr (T > 1 || SF::kFlag) {
    // (a flagged centre leaves the pairs that move its axis)
    M1 = M2 = -4096;
    const unsigned move = zc & (zc - 1u);  // the flagged axes but the lowest
    const int first = zc ? __ffs((int)zc) - 1 : -1;
    for (int k = 0; k < d; ++k) {
      const int E = __double2hiint(W(Ly.x3 + k));
      if (k == first) {
        M2 = max(M2, M1);
        M1 = E;
      } else if (first < 0) {
        M2 = max(M2, min(M1, E));
        M1 = max(M1, E);
      } else if (move == 0u || ((move >> k) & 1u)) {
        if (k < first)
          M1 = max(M1, E);
        else
          M2 = max(M2, E);
      }
    }
  }
  // class 4: the four nodes of the pairs j < k, a pair's exact sum rounded to
  // 2^-54 of the largest product that two axes can have
  LimbSum s5;
  LimbAcc acc;
  i64 s4 = 0;
  const int np = d * (d - 1) / 2;
  for (int p = lane; p < np; p += T) {
    const unsigned pr = pairs[p];
    const int j = (int)(pr >> 8), k = (int)(pr & 255u);
    const Limbs j0 = limbs_unpack(W(Ly.e3 + 2 * j)), j1 = limbs_unpack(W(Ly.e3 + 2 * j + 1));
    const Limbs k0 = limbs_unpack(W(Ly.e3 + 2 * k)), k1 = limbs_unpack(W(Ly.e3 + 2 * k + 1));
    if constexpr (SF::kFlag) {
      if (zc & ~((1u << j) | (1u << k))) continue;
    }
    LimbAcc pair;
    pair.add(j0, k0);
    pair.add(j0, k1);
    pair.add(j1, k0);
    pair.add(j1, k1);
    pair.mid += ((i64)(j0.l + j1.l) * (k0.l + k1.l)) >> 27;
    const int sh = min(
        M1 + M2 - __double2hiint(W(Ly.x3 + j)) - __double2hiint(W(Ly.x3 + k)), 62);
    s4 += shift_even(pair.number(), sh);
  }
  // class 5
  const Limbs one{1 << 26, 0};
  if constexpr (T == 1) {
    if (pb == 0) {  // d = 1
      for (int q = 0; q < nA; ++q) acc.add(limbs_unpack(W(Ly.A + q)), one);
      s5.take(acc);
    } else if (pc) {
      fac_class5c<8>(W, Ly, pa, pb, pc, s5);
    } else if (nA >= 8) {
      fac_class5<8>(W, Ly, pa, pb, s5);
    } else if (nA >= 4) {
      fac_class5<4>(W, Ly, pa, pb, s5);
    } else {
      fac_class5<2>(W, Ly, pa, pb, s5);
    }
  } else {
    int run = 0;
    LimbRest rest;
    for (int q = lane; q < nA; q += T) {
      const Limbs a = limbs_unpack(W(Ly.A + q));
      rest.la += a.l;
      rest.ha += a.h;
    }
    for (int m = lane; m < (1 << d); m += T) {
      const int hi = m >> pa;
      Limbs b = pb ? limbs_unpack(W(Ly.B + (hi & (nB - 1)))) : one;
      i64 rb = 0;
      if (pc) b = LimbAcc::product(b, limbs_unpack(W(Ly.C + (hi >> pb))), rb);
      if ((m & (nA - 1)) == 0) {  // once for every hi
        rest.lb += b.l;
        rest.rb += rb;
      }
      acc.add(limbs_unpack(W(Ly.A + (m & (nA - 1)))), b);
      if (++run == kLimbRun) {
        s5.take(acc);
        run = 0;
      }
    }
    s5.take(acc);
    LimbSum t4;
    t4.add(s4 >> 63, (u64)s4);
    lanes_add<T>(t4, mask);
    s4 = (i64)t4.lo;
    lanes_add<T>(s5, mask);
    lanes_add<T>(rest.la, rest.lb, mask);
    if (pc) lanes_add<T>(rest.ha, rest.rb, mask);
    rest.add_to(s5);
  }
  double f0 = F;
  if constexpr (SF::kFlag) f0 = zc ? 0.0 : F;
  o.s1 = f0;
  o.s2 = __dmul_rn(F, s2);
  o.s3 = __dmul_rn(F, s3);
  const double scale4 = __hiloint2double((970 + max(M1 + M2, -900)) << 20, 0);  // 2^(M1 + M2 - 53)
  o.s4 = __dmul_rn(F, __dmul_rn((double)s4, scale4));
  o.s5 = __dmul_rn(F, s5.value(EA + EB + EC));
  o.f0 = f0;
  o.dbest = __dmul_rn(fabs(F), dbest);
  o.kbest = kbest;
  return true;
}

// cos and sin of lam a h, |lam| < 1, for N lam: the angle in units of 2^-58 (2^-54
// where |a h| is 16 and more), a h and its rounding error times lam; in FP64 where
// |a h| is 256 and more.  An angle is shared by half of the nodes: rounded
// relative to its own size it moved I7 of steep integrands by twice what nodes'
// own inner sums, rounded each for itself, do.
template <class PT, int N>
__device__ __forceinline__ void rotations(const PT& P, int k, double h, const double (&lam)[N],
                                          double (&cs)[N], double (&sn)[N]) {
  const double ah = __dmul_rn(P.a[k], h);
  if (below_256(ah)) {
    const int q = sincos_near(ah) ? 58 : 54;
    const i64 lin = to_fixed(ah, q + 1) + to_fixed(fma(P.a[k], h, -ah), q + 1);
#pragma unroll
    for (int i = 0; i < N; ++i)
      sincos_fixed(fixed_mul_signed(lin, lam_fixed(lam[i])), q, &sn[i], &cs[i]);
  } else {
#pragma unroll 1
    for (int i = 0; i < N; ++i) gm_sincos(__dmul_rn(lam[i], ah), &sn[i], &cs[i]);
  }
}

// The same for the cosine: f = Re(F prod (cos Delta_k +- i sin Delta_k)),
// F = cos S_0 + i sin S_0, Delta = a lambda h.
template <int FAM, int T, class PT, class CH>
__device__ __forceinline__ void region_sums64_rotation(const PT& P, int d,
                                                       const unsigned short* pairs, const CH& ch,
                                                       double lam2, double lam3, double lam5,
                                                       double* w, int ws, double ratio,
                                                       RegionSums& o) {
  using SF = Sep<FAM>;
  const int lane = (T == 1) ? 0 : (int)(threadIdx.x & (unsigned)(T - 1));
  const unsigned mask = group_mask<T>();
  const FacLayout Ly = fac_layout(d, kRotation, T > 1);
  const int pa = fac_a(kRotation, d), pb = fac_b(kRotation, d), pc = fac_c(kRotation, d);
  auto W = [&](int e) -> double& { return w[(long long)e * ws]; };
  double Fc, Fs, s2, s3, dbest = -1.0;
  int kbest = 0;
  // the + and - nodes of one generator and axis
  auto nodes = [&](double ec, double es, double& qp, double& qm) {
    const double p = __dmul_rn(Fc, ec);
    qp = fma(-Fs, es, p);
    qm = fma(Fs, es, p);
  };
  auto axis = [&](int k, double c2, double n2, double c3, double n3, double& q2, double& q3) {
    double p2, m2, p3, m3;
    nodes(c2, n2, p2, m2);
    nodes(c3, n3, p3, m3);
    const double two_f0 = __dmul_rn(2.0, Fc);
    q2 = __dadd_rn(p2, m2);
    q3 = __dadd_rn(p3, m3);
    const double D = fabs(__dsub_rn(__dsub_rn(q2, two_f0),
                                    __dmul_rn(ratio, __dsub_rn(q3, two_f0))));
    // D >= 0: the order of the bit patterns
    if (__double_as_longlong(D) > __double_as_longlong(dbest)) {
      dbest = D;
      kbest = k;
    }
  };
  // (x, y) (c +- i s)
  auto rotate = [](double x, double y, double c, double s, double& rx, double& ry) {
    rx = fma(-y, s, __dmul_rn(x, c));
    ry = fma(x, s, __dmul_rn(y, c));
  };
  if constexpr (T == 1) {
    Centre<FAM> top;
    for (int k = 0; k < d; ++k) {
      double c, h;
      ch(k, c, h);
      top.add(P, k, c, SF::phi(P, k, c));
    }
    top.sincos(Fs, Fc);
    PairTree t2, t3;
    for (int k = 0; k < d; ++k) {
      double c, h;
      ch(k, c, h);
      const double lam[3] = {lam2, lam3, lam5};
      double cs[3], sn[3];
      rotations(P, k, h, lam, cs, sn);
      const double c2 = cs[0], n2 = sn[0], c3 = cs[1], n3 = sn[1], c5 = cs[2], n5 = sn[2];
      W(Ly.e3 + 2 * k) = c3;
      W(Ly.e3 + 2 * k + 1) = n3;
      double q2, q3;
      axis(k, c2, n2, c3, n3, q2, q3);
      t2.push(q2);
      t3.push(q3);
      const int e0 = k < pa ? Ly.A : (k < pa + pb ? Ly.B : Ly.C);
      const int i = k < pa ? k : (k < pa + pb ? k - pa : k - pa - pb);
      if (i == 0 && k > 0) {  // B and C start from 1
        W(e0) = c5;
        W(e0 + 1) = n5;
        W(e0 + 2) = c5;
        W(e0 + 3) = -n5;
      } else {
        const int n = 1 << i;
        for (int t = 0; t < n; ++t) {
          const double x = k ? W(e0 + 2 * t) : Fc, y = k ? W(e0 + 2 * t + 1) : Fs;
          const double xc = __dmul_rn(x, c5), yc = __dmul_rn(y, c5);
          W(e0 + 2 * (t + n)) = fma(y, n5, xc);
          W(e0 + 2 * (t + n) + 1) = fma(-x, n5, yc);
          W(e0 + 2 * t) = fma(-y, n5, xc);
          W(e0 + 2 * t + 1) = fma(x, n5, yc);
        }
      }
    }
    bool pr;
    s2 = t2.flush(pr);
    s3 = t3.flush(pr);
  } else {
    // 1. lanes over the 3 d rotations, and phi at the centre
    for (int t = lane; t < 3 * d; t += T) {
      const int k = t / 3, r = t - 3 * k;
      double c, h;
      ch(k, c, h);
      const double lam[1] = {r == 0 ? lam2 : (r == 1 ? lam3 : lam5)};
      double cs[1], sn[1];
      rotations(P, k, h, lam, cs, sn);
      const int e = (r == 0 ? Ly.e2 : (r == 1 ? Ly.e3 : Ly.e5)) + 2 * k;
      W(e) = cs[0];
      W(e + 1) = sn[0];
      if (r == 0) W(Ly.phiC + k) = SF::phi(P, k, c);
    }
    group_sync<T>(mask);
    // 2. F, then the class-5 chains (A's headed by F)
    if (lane == 0) {
      Centre<FAM> top;
      for (int k = 0; k < d; ++k) {
        double c, h;
        ch(k, c, h);
        top.add(P, k, c, W(Ly.phiC + k));
      }
      double sn, cs;
      top.sincos(sn, cs);
      W(Ly.F) = cs;
      W(Ly.F + 1) = sn;
    }
    group_sync<T>(mask);
    Fc = W(Ly.F);
    Fs = W(Ly.F + 1);
    const int nA = 1 << pa, nB = pb ? 1 << pb : 0, nC = pc ? 1 << pc : 0;
    for (int t = lane; t < nA + nB + nC; t += T) {
      int e = t, e0 = Ly.A, j0 = 0, nb = pa;
      if (e >= nA) {
        e -= nA;
        e0 = Ly.B;
        j0 = pa;
        nb = pb;
        if (e >= nB) {
          e -= nB;
          e0 = Ly.C;
          j0 = pa + pb;
          nb = pc;
        }
      }
      double x = Fc, y = Fs;
      for (int i = 0; i < nb; ++i) {
        const double c5 = W(Ly.e5 + 2 * (j0 + i)), n5 = W(Ly.e5 + 2 * (j0 + i) + 1);
        const double sg = ((e >> i) & 1) ? -n5 : n5;
        if (i == 0 && j0 > 0) {
          x = c5;
          y = sg;
        } else {
          double rx, ry;
          rotate(x, y, c5, sg, rx, ry);
          x = rx;
          y = ry;
        }
      }
      W(e0 + 2 * e) = x;
      W(e0 + 2 * e + 1) = y;
    }
    group_sync<T>(mask);
    // 3. lanes over the axes
    PairTree t2, t3;
    int p0, cnt;
    lane_leaves<T>(lane, lg_ceil(d), p0, cnt);
    const int p1 = min(p0 + cnt, d);
    for (int k = p0; k < p1; ++k) {
      double q2, q3;
      axis(k, W(Ly.e2 + 2 * k), W(Ly.e2 + 2 * k + 1), W(Ly.e3 + 2 * k), W(Ly.e3 + 2 * k + 1), q2,
           q3);
      t2.push(q2);
      t3.push(q3);
    }
    lanes_argmax<T>(dbest, kbest, mask);
    bool pr2, pr3;
    const double x2 = t2.flush(pr2), x3 = t3.flush(pr3);
    s2 = lanes_tree<T>(x2, pr2, mask);
    s3 = lanes_tree<T>(x3, pr3, mask);
  }
  // the chains as limbs (every entry is at most 1)
  const int nA = 1 << pa, nB = pb ? 1 << pb : 0, nC = pc ? 1 << pc : 0;
  for (int e = lane; e < 2 * (nA + nB + nC); e += T) W(Ly.A + e) = limbs_of(W(Ly.A + e), 0);
  if constexpr (T > 1) group_sync<T>(mask);
  LimbSum s4, s5;
  LimbAcc acc;
  int run = 0;
  // class 5: Re(A B) (Re(A (B C)) above d = 8)
  auto bc_of = [&](int hi, Limbs& x, Limbs& y) {
    if (!pb) {
      x = Limbs{1 << 26, 0};
      y = Limbs{0, 0};
      return;
    }
    const int eb = Ly.B + 2 * (hi & (nB - 1));
    x = limbs_unpack(W(eb));
    y = limbs_unpack(W(eb + 1));
    if (pc) {
      const int ec = Ly.C + 2 * (hi >> pb);
      const Limbs u = limbs_unpack(W(ec)), v = limbs_unpack(W(ec + 1));
      LimbAcc r, i;
      r.add(x, u);
      r.sub(y, v);
      i.add(x, v);
      i.add(y, u);
      x = limbs_split(r.number());
      y = limbs_split(i.number());
    }
  };
  if constexpr (T == 1) {
    auto walk = [&](auto entries) {  // so many entries of A in registers
      constexpr int N = decltype(entries)::value;
      for (int lo = 0; lo < nA; lo += N) {
        Limbs ax[N], ay[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          ax[i] = limbs_unpack(W(Ly.A + 2 * (lo + i)));
          ay[i] = limbs_unpack(W(Ly.A + 2 * (lo + i) + 1));
        }
        for (int hi = 0; hi < (1 << (pb + pc)); ++hi) {
          Limbs bx, by;
          bc_of(hi, bx, by);
#pragma unroll
          for (int i = 0; i < N; ++i) {
            acc.add(ax[i], bx);
            acc.sub(ay[i], by);
          }
          if (((hi + 1) & (kLimbRun / (2 * N) - 1)) == 0) s5.take(acc);
        }
        s5.take(acc);
      }
    };
    if (nA >= 4)
      walk(std::integral_constant<int, 4>());
    else
      walk(std::integral_constant<int, 2>());
  } else {
    for (int m = lane; m < (1 << d); m += T) {
      Limbs bx, by;
      bc_of(m >> pa, bx, by);
      const int ea = Ly.A + 2 * (m & (nA - 1));
      acc.add(limbs_unpack(W(ea)), bx);
      acc.sub(limbs_unpack(W(ea + 1)), by);
      if ((run += 2) == kLimbRun) {
        s5.take(acc);
        run = 0;
      }
    }
    s5.take(acc);
  }
  // a pair needs F turned by its first axis, formed in FP64 once per axis and
  // sign and kept in the chains' place (4 d <= 2 (2^a + 2^b + 2^c) for every d)
  if constexpr (T > 1) group_sync<T>(mask);  // the chains and lambda3's doubles have been read
  const int J = Ly.A;
  for (int k = lane; k < d; k += T) {
    const double c3 = W(Ly.e3 + 2 * k), n3 = W(Ly.e3 + 2 * k + 1);
    double x, y;
    rotate(Fc, Fs, c3, n3, x, y);
    W(J + 4 * k) = limbs_of(x, 0);
    W(J + 4 * k + 1) = limbs_of(y, 0);
    rotate(Fc, Fs, c3, -n3, x, y);
    W(J + 4 * k + 2) = limbs_of(x, 0);
    W(J + 4 * k + 3) = limbs_of(y, 0);
    W(Ly.e3 + 2 * k) = limbs_of(c3, 0);
    W(Ly.e3 + 2 * k + 1) = limbs_of(n3, 0);
  }
  if constexpr (T > 1) group_sync<T>(mask);
  // class 4: the four nodes of the pairs j < k, real part of J (c +- i n)
  const int np = d * (d - 1) / 2;
  run = 0;
  for (int p = lane; p < np; p += T) {
    const unsigned pr = pairs[p];
    const int j = (int)(pr >> 8), k = (int)(pr & 255u);
    const Limbs ck = limbs_unpack(W(Ly.e3 + 2 * k)), nk = limbs_unpack(W(Ly.e3 + 2 * k + 1));
#pragma unroll
    for (int sj = 0; sj < 2; ++sj) {
      const Limbs x = limbs_unpack(W(J + 4 * j + 2 * sj));
      const Limbs y = limbs_unpack(W(J + 4 * j + 2 * sj + 1));
      acc.add(x, ck);
      acc.sub(y, nk);
      acc.add(x, ck);
      acc.add(y, nk);
    }
    if ((run += 8) == kLimbRun) {
      s4.take(acc);
      run = 0;
    }
  }
  s4.take(acc);
  if constexpr (T > 1) {
    lanes_add<T>(s4, mask);
    lanes_add<T>(s5, mask);
  }
  o.s1 = Fc;
  o.s2 = s2;
  o.s3 = s3;
  o.s4 = s4.value(0);
  o.s5 = s5.value(0);
  o.f0 = Fc;
  o.dbest = dbest;
  o.kbest = kbest;
}

// The class sums and the split axis of one region: from per-axis factors
// where the integrand has them, in fixed point for the corner peak, from the
// separable form otherwise (the polynomial; the cosine above d = 14; a region
// whose factors or inner sums lack exponent room).  Arguments as region_sums64; w points at the
// region's workspace of region64_words(d, ...) entries.
template <int FAM, int T, class PT, class CH>
__device__ __forceinline__ void region_sums(const PT& P, int d, const unsigned short* pairs,
                                            const CH& ch, double lam2, double lam3, double lam5,
                                            double* w, int ws, double ratio, RegionSums& o) {
  if constexpr (Fac<FAM>::kind == kReal) {
    if (region_sums64_real<FAM, T>(P, d, pairs, ch, lam2, lam3, lam5, w, ws, ratio, o)) return;
  } else if constexpr (Fac<FAM>::kind == kRotation) {
    if (fac_used(kRotation, d)) {
      region_sums64_rotation<FAM, T>(P, d, pairs, ch, lam2, lam3, lam5, w, ws, ratio, o);
      return;
    }
  }
  if constexpr (FAM == GMQ_CORNER_PEAK) {
    if (region_sums64_corner<T>(P, d, pairs, ch, lam2, lam3, lam5, w, ws, ratio, o)) return;
  }
  region_sums64<FAM, T>(P, d, pairs, ch, lam2, lam3, lam5, w, ws, ratio, o);
}

}  // namespace gmq
