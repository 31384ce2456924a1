// gm_factor64.cuh -- class sums of one region for the integrands that are
// products of one factor per axis (exponentials and the product peak) or the
// real part of such a product (the cosine): node values from per-axis
// factors.  Shared by the single-integral and the batched FP64 rule kernels.
//
// Bound: the FP64 pipe (one warp instruction in 64 cycles per SM quarter;
// integer and shared-memory instructions beside it are nearly free), so the
// design counts FP64 instructions.  With S = S_0 + Delta_j (+ Delta_k) an
// exponential node is f = F e_j (e_k): F = f(centre), e = exp(-Delta) one of
// six factors per axis (c +- lambda h for three generators), formed once per
// region, and every node's value is one product that the accumulating fused
// multiply-add forms on the way: 401 nodes at d = 8 cost 368 fused
// multiply-adds and 48 exponentials instead of 401 exponentials, 401 chain
// steps and 401 adds.  The product peak's factors are ratios of its
// per-axis denominators (a reciprocal each); the cosine's are rotations
// (cos Delta, sin Delta), two fused multiply-adds per node.  Measured at d = 8,
// 2^20 regions, one thread per region: C0 8.14 -> 2.23 ms (4080 -> 1163 FP64
// instructions a region), Gaussian 8.25 -> 2.34, product peak 4.71 -> 2.00,
// cosine 10.99 -> 3.31 ms, the FP64 pipe 88-91 % active.
//
// Accuracy: F is a common factor of every node, so its error scales the
// region's value and is not amplified by the rule's weights of both signs
// (sum |w| is 5.8 at d = 8); the factors carry an error near 2^-53 each.
// Factors may over- or underflow where f does not (a factor is relative to
// the centre): regions whose factors' exponents do not leave room are
// evaluated by region_sums64, decided from the region alone, so that every
// lane mapping takes the same path.
//
// Summation order (fixed, the same for T = 1, 4, 32, 128 lanes): classes 2
// and 3 one leaf per axis (the sum of its two nodes); class 4 one leaf per
// pair of axes (its four nodes left to right by fused multiply-add); class 5
// leaves of max(8, 2^d / 128) consecutive sign patterns, left to right by
// fused multiply-add.  Leaves are combined by the adjacent-pairwise tree.
// The lane mapping only places leaves: T lanes own consecutive leaves in bit
// reversed order, as in gm_region64.cuh.
#pragma once

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

// e(P, j, x, fc): the factor of x on axis j relative to the centre, whose
// phi is fc
template <>
struct Fac<GMQ_C0> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double e(const PT& P, int j, double x, double fc) {
    return gexp(fma(-P.a[j], fabs(__dsub_rn(x, P.u[j])), fc));
  }
};

template <>
struct Fac<GMQ_GAUSSIAN> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double e(const PT& P, int j, double x, double fc) {
    const double t = __dsub_rn(x, P.u[j]);
    return gexp(fma(-__dmul_rn(P.b[j], t), t, fc));
  }
};

template <>
struct Fac<GMQ_DISCONTINUOUS> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double e(const PT& P, int j, double x, double fc) {
    return gexp(fma(P.a[j], x, -fc));
  }
};

template <>
struct Fac<GMQ_PRODUCT_PEAK> {
  static constexpr int kind = kReal;
  template <class PT>
  __device__ __forceinline__ static double e(const PT& P, int j, double x, double fc) {
    return __dmul_rn(fc, gm_rcp(Sep<GMQ_PRODUCT_PEAK>::phi(P, j, x)));
  }
};

template <>
struct Fac<GMQ_OSCILLATORY> {
  static constexpr int kind = kRotation;
};

// Workspace of one region (entries `ws` doubles apart): the lambda3 factors
// E3 [2d] and the class-5 chains A, B, C; with T > 1 lanes also phi at the
// centre [d], the factors of lambda2 and lambda5 [2d each] and F [2].  For
// kReal, chains over axes [0, a), [a, a + b), [a + b, d) of the factors of
// c +- lambda5 h.  For kRotation every factor is two entries (cosine, sine
// of the + sign; - is its conjugate) and every chain entry is two, A's
// chains headed by F.
struct FacLayout {
  int e3, A, B, C, phiC, e2, e5, F, words;
};

__host__ __device__ constexpr FacLayout fac_layout(int d, int kind, bool lanes) {
  FacLayout s{};
  const int m = kind == kRotation ? 2 : 1;
  s.e3 = 0;
  s.A = 2 * d * m;
  s.B = s.A + m * (1 << sep_a(d));
  s.C = s.B + (sep_b(d) ? m * (1 << sep_b(d)) : 0);
  int w = s.C + (sep_c(d) ? m * (1 << sep_c(d)) : 0);
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
// share it (a region uses one, or first one and then the other).
__host__ __device__ constexpr int region64_words(int d, int kind, bool flag, bool lanes) {
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

// Sum of `n` leaves, leaf(p) the value of leaf p, over a tree of 2^lg >= n
// positions by the T lanes of a group.
template <int T, class Leaf>
__device__ __forceinline__ double leaf_sum(int n, int lg, int lane, unsigned mask, Leaf leaf) {
  PairTree t;
  int p0, cnt;
  lane_leaves<T>(lane, lg, p0, cnt);
  const int p1 = min(p0 + cnt, n);
  for (int p = p0; p < p1; ++p) t.push(leaf(p));
  bool present;
  const double x = t.flush(present);
  return lanes_tree<T>(x, present, mask);
}

// log2 of the leaf positions of class 5 (leaves of at least 8 patterns, at
// most 128 leaves) and of the pairs of axes (<= 120) and axes (<= 16)
__device__ __forceinline__ int fac_lg5(int d) { return d <= 3 ? 0 : min(7, d - 3); }
__device__ __forceinline__ int lg_ceil(int n) { return n <= 1 ? 0 : 32 - __clz(n - 1); }

// Class 5 of the real factors: pattern m = (m_A, hi), value A[m_A] *
// (B[hi] or B[.] C[.]); a leaf runs over whole stretches of m_A.
// zero(m): the discontinuous family's nodes that are 0.
template <bool kFlag, class WF, class Zero>
__device__ __forceinline__ double fac_leaf5(const WF& W, const FacLayout& Ly, int pa, int pb,
                                            int pc, int m0, int cs, const Zero& zero) {
  const int am = (1 << pa) - 1;
  const int run = min(cs, 1 << pa);
  double x = 0.0;
  for (int s = 0; s < cs; s += run) {
    const int m = m0 + s, hi = m >> pa, ea = Ly.A + (m & am);
    double bc = 1.0;
    if (pb) bc = W(Ly.B + (hi & ((1 << pb) - 1)));
    if (pc) bc = __dmul_rn(bc, W(Ly.C + (hi >> pb)));
#pragma unroll 4
    for (int q = 0; q < run; ++q) {
      double a = W(ea + q);
      if (kFlag && zero(m + q)) a = 0.0;
      x = (s | q) ? fma(a, bc, x) : __dmul_rn(a, bc);
    }
  }
  return x;
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
  using FF = Fac<FAM>;
  const int lane = (T == 1) ? 0 : (int)(threadIdx.x & (unsigned)(T - 1));
  const unsigned mask = group_mask<T>();
  const FacLayout Ly = fac_layout(d, kReal, T > 1);
  const int pa = sep_a(d), pb = sep_b(d), pc = sep_c(d);
  auto W = [&](int e) -> double& { return w[(long long)e * ws]; };
  auto op = [](double x, double y) -> double {
    if constexpr (SF::kMul)
      return __dmul_rn(x, y);
    else
      return __dadd_rn(x, y);
  };
  // flag masks of the discontinuous family (x_j > u_j): centre; c +- lambda3
  // h and c +- lambda5 h (+ in bits 0..15, - in bits 16..31)
  unsigned zc = 0u, z3 = 0u, z5 = 0u;
  double F, s2, s3, dbest = -1.0;  // class sums and differences relative to F
  int kbest = 0, room = 0;
  // first axis and length of the chain part that axis k belongs to
  auto part = [&](int k, int& e0, int& i) {
    e0 = k < pa ? Ly.A : (k < pa + pb ? Ly.B : Ly.C);
    i = k < pa ? k : (k < pa + pb ? k - pa : k - pa - pb);
  };
  // sums of an axis's node pairs and its fourth difference
  auto axis = [&](int k, double p2, double m2, double p3, double m3, bool fp2, bool fm2,
                  double& q2, double& q3) {
    double f0 = 1.0;
    if constexpr (SF::kFlag) {
      if (zc & ~(1u << k)) p2 = m2 = p3 = m3 = 0.0;
      if (zc) f0 = 0.0;
      if (fp2) p2 = 0.0;
      if (fm2) m2 = 0.0;
      if ((z3 >> k) & 1u) p3 = 0.0;
      if ((z3 >> (k + 16)) & 1u) m3 = 0.0;
    }
    q2 = __dadd_rn(p2, m2);
    q3 = __dadd_rn(p3, m3);
    const double two_f0 = f0 + f0;
    const double D = fabs(__dsub_rn(__dsub_rn(q2, two_f0),
                                    __dmul_rn(ratio, __dsub_rn(q3, two_f0))));
    if (D > dbest) {
      dbest = D;
      kbest = k;
    }
  };
  if constexpr (T == 1) {
    if constexpr (SF::kFlag) {
      for (int k = 0; k < d; ++k) {
        double c, h;
        ch(k, c, h);
        zc |= (unsigned)SF::flag(P, k, c) << k;
      }
    }
    PairTree t2, t3;
    double S = 0.0;
    for (int k = 0; k < d; ++k) {
      double c, h;
      ch(k, c, h);
      const double fc = SF::phi(P, k, c);
      S = k ? op(S, fc) : fc;
      const double x2p = fma(lam2, h, c), x2m = fma(-lam2, h, c);
      const double x3p = fma(lam3, h, c), x3m = fma(-lam3, h, c);
      const double x5p = fma(lam5, h, c), x5m = fma(-lam5, h, c);
      const double p2 = FF::e(P, k, x2p, fc), m2 = FF::e(P, k, x2m, fc);
      const double p3 = FF::e(P, k, x3p, fc), m3 = FF::e(P, k, x3m, fc);
      const double p5 = FF::e(P, k, x5p, fc), m5 = FF::e(P, k, x5m, fc);
      room += max(max(exp_magnitude(p2), exp_magnitude(m2)),
                  max(max(exp_magnitude(p3), exp_magnitude(m3)),
                      max(exp_magnitude(p5), exp_magnitude(m5))));
      W(Ly.e3 + 2 * k) = p3;
      W(Ly.e3 + 2 * k + 1) = m3;
      bool fp2 = false, fm2 = false;
      if constexpr (SF::kFlag) {
        fp2 = SF::flag(P, k, x2p);
        fm2 = SF::flag(P, k, x2m);
        z3 |= ((unsigned)SF::flag(P, k, x3p) << k) | ((unsigned)SF::flag(P, k, x3m) << (k + 16));
        z5 |= ((unsigned)SF::flag(P, k, x5p) << k) | ((unsigned)SF::flag(P, k, x5m) << (k + 16));
      }
      double q2, q3;
      axis(k, p2, m2, p3, m3, fp2, fm2, q2, q3);
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
    F = SF::g(d, S);
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
      const double x = fma((r & 1) ? -lam : lam, h, c);
      const double fc = SF::phi(P, k, c);
      const double e = FF::e(P, k, x, fc);
      W((r < 2 ? Ly.e2 : (r < 4 ? Ly.e3 : Ly.e5)) + 2 * k + (r & 1)) = e;
      if (r == 0) W(Ly.phiC + k) = fc;
    }
    if constexpr (SF::kFlag) {
      for (int k = 0; k < d; ++k) {
        double c, h;
        ch(k, c, h);
        zc |= (unsigned)SF::flag(P, k, c) << k;
        z3 |= ((unsigned)SF::flag(P, k, fma(lam3, h, c)) << k) |
              ((unsigned)SF::flag(P, k, fma(-lam3, h, c)) << (k + 16));
        z5 |= ((unsigned)SF::flag(P, k, fma(lam5, h, c)) << k) |
              ((unsigned)SF::flag(P, k, fma(-lam5, h, c)) << (k + 16));
      }
    }
    group_sync<T>(mask);
    // 2. lanes over the tasks: F (and its room, by the lane that forms it)
    //    and every class-5 chain, left to right
    const int nA = 1 << pa, nB = pb ? 1 << pb : 0, nC = pc ? 1 << pc : 0;
    for (int t = lane; t < 1 + nA + nB + nC; t += T) {
      if (t == 0) {
        double S = W(Ly.phiC);
        for (int k = 1; k < d; ++k) S = op(S, W(Ly.phiC + k));
        const double Fv = SF::g(d, S);
        for (int k = 0; k < d; ++k) {
          int m = 0;
#pragma unroll
          for (int s = 0; s < 2; ++s)
            m = max(m, max(exp_magnitude(W(Ly.e2 + 2 * k + s)),
                           max(exp_magnitude(W(Ly.e3 + 2 * k + s)),
                               exp_magnitude(W(Ly.e5 + 2 * k + s)))));
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
      bool fp2 = false, fm2 = false;
      if constexpr (SF::kFlag) {
        double c, h;
        ch(k, c, h);
        fp2 = SF::flag(P, k, fma(lam2, h, c));
        fm2 = SF::flag(P, k, fma(-lam2, h, c));
      }
      double q2, q3;
      axis(k, W(Ly.e2 + 2 * k), W(Ly.e2 + 2 * k + 1), W(Ly.e3 + 2 * k), W(Ly.e3 + 2 * k + 1), fp2,
           fm2, q2, q3);
      t2.push(q2);
      t3.push(q3);
    }
    // argmax over the lanes: larger D wins, the lower axis on ties (T = 128:
    // the d <= 16 leaves sit in warp 0, whose lane 0 alone uses the axis)
    constexpr int WL = T < 32 ? T : 32;
#pragma unroll
    for (int off = WL / 2; off > 0; off >>= 1) {
      const double od = __shfl_xor_sync(mask, dbest, off, WL);
      const int ok = __shfl_xor_sync(mask, kbest, off, WL);
      if (od > dbest || (od == dbest && ok < kbest)) {
        dbest = od;
        kbest = ok;
      }
    }
    bool pr2, pr3;
    const double x2 = t2.flush(pr2), x3 = t3.flush(pr3);
    s2 = lanes_tree<T>(x2, pr2, mask);
    s3 = lanes_tree<T>(x3, pr3, mask);
  }
  // class 4: one leaf per pair j < k, signs ++, +-, -+, --
  const int np = d * (d - 1) / 2;
  const double s4 = leaf_sum<T>(np, lg_ceil(np), lane, mask, [&](int p) -> double {
    const unsigned pr = pairs[p];
    const int j = (int)(pr >> 8), k = (int)(pr & 255u);
    double j0 = W(Ly.e3 + 2 * j), j1 = W(Ly.e3 + 2 * j + 1);
    double k0 = W(Ly.e3 + 2 * k), k1 = W(Ly.e3 + 2 * k + 1);
    if constexpr (SF::kFlag) {
      if (zc & ~((1u << j) | (1u << k))) j0 = j1 = 0.0;
      if ((z3 >> j) & 1u) j0 = 0.0;
      if ((z3 >> (j + 16)) & 1u) j1 = 0.0;
      if ((z3 >> k) & 1u) k0 = 0.0;
      if ((z3 >> (k + 16)) & 1u) k1 = 0.0;
    }
    return fma(j1, k1, fma(j1, k0, fma(j0, k1, __dmul_rn(j0, k0))));
  });
  // class 5
  const int lg5 = fac_lg5(d), cs = 1 << (d - lg5);
  const unsigned dmask = (1u << d) - 1u;
  const double s5 = leaf_sum<T>(1 << lg5, lg5, lane, mask, [&](int p) -> double {
    return fac_leaf5<SF::kFlag>(W, Ly, pa, pb, pc, p * cs, cs, [&](int m) -> bool {
      return ((((unsigned)~m & z5) | ((unsigned)m & (z5 >> 16))) & dmask) != 0u;
    });
  });
  double f0 = F;
  if constexpr (SF::kFlag) f0 = zc ? 0.0 : F;
  o.s1 = f0;
  o.s2 = __dmul_rn(F, s2);
  o.s3 = __dmul_rn(F, s3);
  o.s4 = __dmul_rn(F, s4);
  o.s5 = __dmul_rn(F, s5);
  o.f0 = f0;
  o.dbest = __dmul_rn(fabs(F), dbest);
  o.kbest = kbest;
  return true;
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
  const int pa = sep_a(d), pb = sep_b(d), pc = sep_c(d);
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
    if (D > dbest) {
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
    double S = SF::base(P);
    for (int k = 0; k < d; ++k) {
      double c, h;
      ch(k, c, h);
      S = __dadd_rn(S, SF::phi(P, k, c));
    }
    gm_sincos(S, &Fs, &Fc);
    PairTree t2, t3;
    for (int k = 0; k < d; ++k) {
      double c, h;
      ch(k, c, h);
      const double ah = __dmul_rn(P.a[k], h);
      double c2, n2, c3, n3, c5, n5;
      gm_sincos(__dmul_rn(lam2, ah), &n2, &c2);
      gm_sincos(__dmul_rn(lam3, ah), &n3, &c3);
      gm_sincos(__dmul_rn(lam5, ah), &n5, &c5);
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
      const double ah = __dmul_rn(P.a[k], h);
      double sn, cs;
      gm_sincos(__dmul_rn(r == 0 ? lam2 : (r == 1 ? lam3 : lam5), ah), &sn, &cs);
      const int e = (r == 0 ? Ly.e2 : (r == 1 ? Ly.e3 : Ly.e5)) + 2 * k;
      W(e) = cs;
      W(e + 1) = sn;
      if (r == 0) W(Ly.phiC + k) = SF::phi(P, k, c);
    }
    group_sync<T>(mask);
    // 2. F, then the class-5 chains (A's headed by F)
    if (lane == 0) {
      double S = SF::base(P);
      for (int k = 0; k < d; ++k) S = __dadd_rn(S, W(Ly.phiC + k));
      double sn, cs;
      gm_sincos(S, &sn, &cs);
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
    constexpr int WL = T < 32 ? T : 32;
#pragma unroll
    for (int off = WL / 2; off > 0; off >>= 1) {
      const double od = __shfl_xor_sync(mask, dbest, off, WL);
      const int ok = __shfl_xor_sync(mask, kbest, off, WL);
      if (od > dbest || (od == dbest && ok < kbest)) {
        dbest = od;
        kbest = ok;
      }
    }
    bool pr2, pr3;
    const double x2 = t2.flush(pr2), x3 = t3.flush(pr3);
    s2 = lanes_tree<T>(x2, pr2, mask);
    s3 = lanes_tree<T>(x3, pr3, mask);
  }
  // class 4: F turned by j (both signs), then the four nodes of the pair
  const int np = d * (d - 1) / 2;
  const double s4 = leaf_sum<T>(np, lg_ceil(np), lane, mask, [&](int p) -> double {
    const unsigned pr = pairs[p];
    const int j = (int)(pr >> 8), k = (int)(pr & 255u);
    const double cj = W(Ly.e3 + 2 * j), nj = W(Ly.e3 + 2 * j + 1);
    const double ck = W(Ly.e3 + 2 * k), nk = W(Ly.e3 + 2 * k + 1);
    double px, py, mx, my;
    rotate(Fc, Fs, cj, nj, px, py);
    rotate(Fc, Fs, cj, -nj, mx, my);
    double x = __dmul_rn(px, ck);
    x = fma(-py, nk, x);
    x = fma(px, ck, x);
    x = fma(py, nk, x);
    x = fma(mx, ck, x);
    x = fma(-my, nk, x);
    x = fma(mx, ck, x);
    return fma(my, nk, x);
  });
  // class 5: Re(A B) (Re(A (B C)) above d = 8)
  const int lg5 = fac_lg5(d), cs = 1 << (d - lg5);
  const int am = (1 << pa) - 1, run = min(cs, 1 << pa);
  const double s5 = leaf_sum<T>(1 << lg5, lg5, lane, mask, [&](int p) -> double {
    double x = 0.0;
    for (int s = 0; s < cs; s += run) {
      const int m = p * cs + s, hi = m >> pa, ea = Ly.A + 2 * (m & am);
      double bx = 1.0, by = 0.0;
      if (pb) {
        const int eb = Ly.B + 2 * (hi & ((1 << pb) - 1));
        bx = W(eb);
        by = W(eb + 1);
      }
      if (pc) {
        const int ec = Ly.C + 2 * (hi >> pb);
        double rx, ry;
        rotate(bx, by, W(ec), W(ec + 1), rx, ry);
        bx = rx;
        by = ry;
      }
#pragma unroll 4
      for (int q = 0; q < run; ++q) {
        const double ax = W(ea + 2 * q), ay = W(ea + 2 * q + 1);
        x = (s | q) ? fma(ax, bx, x) : __dmul_rn(ax, bx);
        x = fma(-ay, by, x);
      }
    }
    return x;
  });
  o.s1 = Fc;
  o.s2 = s2;
  o.s3 = s3;
  o.s4 = s4;
  o.s5 = s5;
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
