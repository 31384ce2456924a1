// gm_region32.cuh -- mixed-form evaluation of one region by one thread,
// shared by the single-integral mixed kernels (gm_rule.cuh) and the batched
// mixed kernel, so both compute a region with the same operations in the
// same order.
//
// Mixed form: node coordinates are FP32 (the caller's table, built by
// mixed_coord_rows), the integrand runs in FP32, and the class sums are
// FP32 with Knuth TwoSum compensation, converted to FP64 before the
// weights; the fourth differences and everything after the class sums are
// FP64 (region_finish64).
#pragma once

#include "gm_region64.cuh"
#include "gmq_common.cuh"
#include "gmq_families.cuh"

namespace gmq {

// The seven FP32 node-coordinate rows of one axis of a region (kXC, kXP2,
// kXM2, kXP3, kXM3, kXP5, kXM5 at out[row * stride]), formed in FP32 from
// the centre split into two FP32 parts, c = c_hi + c_lo, and the FP32
// half-width: x = c_hi + fma(+-lambda, h, c_lo).  The offset c_lo +
// lambda h is small and nearly exact, so x is c + lambda h rounded once to
// FP32 up to rare one-ulp differences -- the rounding the FP32 integrand
// sees in any case -- while the FP64 work per axis is three conversions and
// one subtraction (the FP64 pipe issues at 1/64 of the FP32 rate).
__device__ __forceinline__ void mixed_coord_rows(double c, double h, float l2, float l3,
                                                 float l5, float* out, int stride) {
  const float c_hi = __double2float_rn(c);
  const float c_lo = __double2float_rn(__dsub_rn(c, f2d_exact(c_hi)));
  const float hf = __double2float_rn(h);
  out[kXC * stride] = c_hi;
  out[kXP2 * stride] = __fadd_rn(c_hi, __fmaf_rn(l2, hf, c_lo));
  out[kXM2 * stride] = __fadd_rn(c_hi, __fmaf_rn(-l2, hf, c_lo));
  out[kXP3 * stride] = __fadd_rn(c_hi, __fmaf_rn(l3, hf, c_lo));
  out[kXM3 * stride] = __fadd_rn(c_hi, __fmaf_rn(-l3, hf, c_lo));
  out[kXP5 * stride] = __fadd_rn(c_hi, __fmaf_rn(l5, hf, c_lo));
  out[kXM5 * stride] = __fadd_rn(c_hi, __fmaf_rn(-l5, hf, c_lo));
}

// Generic dimension: every node in the order of its definition (centre;
// per axis +l2, -l2, +l3, -l3; pairs j < k with sign patterns ++, +-, -+,
// --; sign patterns m = 0 .. 2^d - 1).  P holds FP32 parameters;
// tab(row, j) is the FP32 node coordinate; pairs as in region_sums64.
template <int FAM, class PT, class Tab>
__device__ __forceinline__ void region_mixed_flat(const PT& P, int d, const unsigned short* pairs,
                                                  const Tab& tab, double ratio, RegionSums& o) {
  const int b4 = 1 + 4 * d;             // first pair node
  const int b5 = b4 + 2 * d * (d - 1);  // first sign-pattern node
  const int N = b5 + (1 << d);
  Acc<float> S1, S2, S3, S4, S5;
  double f0 = 0.0, two_f0 = 0.0, q0 = 0.0, q1 = 0.0, q2 = 0.0, dbest = -1.0;
  int kbest = 0;
  for (int i = 0; i < N; ++i) {
    int kind, k1 = -1, r1 = kXC, k2 = -1, r2 = kXC, w = 0;
    unsigned m = 0u;
    if (i == 0) {
      kind = 1;
    } else if (i < b4) {
      const int q = i - 1;
      k1 = q >> 2;
      w = q & 3;
      r1 = kXP2 + w;
      kind = (w < 2) ? 2 : 3;
    } else if (i < b5) {
      const int q = i - b4;
      const unsigned pr = pairs[q >> 2];
      k1 = (int)(pr >> 8);
      k2 = (int)(pr & 255u);
      r1 = (q & 2) ? kXM3 : kXP3;
      r2 = (q & 1) ? kXM3 : kXP3;
      kind = 4;
    } else {
      m = (unsigned)(i - b5);
      kind = 5;
    }
    const float v = Family<FAM>::template eval<float>(P, d, [&](int j) -> float {
      int row;
      if (kind == 5)
        row = ((m >> j) & 1u) ? kXM5 : kXP5;
      else
        row = (j == k1) ? r1 : ((j == k2) ? r2 : kXC);
      return tab(row, j);
    });
    if (kind == 5) {
      S5.add(v);
    } else if (kind == 4) {
      S4.add(v);
    } else if (kind == 1) {
      S1.add(v);
      f0 = f2d_exact(v);
      two_f0 = __dmul_rn(2.0, f0);
    } else {
      if (kind == 2)
        S2.add(v);
      else
        S3.add(v);
      const double vd = f2d_exact(v);
      if (w == 0) {
        q0 = vd;
      } else if (w == 1) {
        q1 = vd;
      } else if (w == 2) {
        q2 = vd;
      } else {
        const double t1 = __dsub_rn(__dadd_rn(q0, q1), two_f0);
        const double t2 = __dsub_rn(__dadd_rn(q2, vd), two_f0);
        const double Dk = fabs(__dsub_rn(t1, __dmul_rn(ratio, t2)));
        if (Dk > dbest) {
          dbest = Dk;
          kbest = k1;
        }
      }
    }
  }
  o.s1 = S1.value();
  o.s2 = S2.value();
  o.s3 = S3.value();
  o.s4 = S4.value();
  o.s5 = S5.value();
  o.f0 = f0;
  o.dbest = dbest;
  o.kbest = kbest;
}

// The FP32 integrands as chains: y(P, j, x) is what axis j's coordinate x enters
// the inner chain as, step appends it to the chain s of axes 0 .. j - 1, and out
// is the integrand from the whole chain; step2 and outs work on pairs of nodes
// (paired FP32 instructions).  Exactly the operations of Family<FAM>::eval in
// their order, so a node's value has its bits, and nodes that agree on axes 0 ..
// j share the chain so far.
template <int FAM>
struct Chain {
  static constexpr bool kPeak = FAM == GMQ_PRODUCT_PEAK, kGauss = FAM == GMQ_GAUSSIAN;
  static constexpr bool kC0 = FAM == GMQ_C0, kDisc = FAM == GMQ_DISCONTINUOUS;
  static constexpr bool kPoly = FAM == GMQ_POLY_SUMSQ11;
  template <class PT>
  __device__ __forceinline__ static float init(const PT& P) {
    if constexpr (FAM == GMQ_OSCILLATORY) return P.c0;
    return kPeak || FAM == GMQ_CORNER_PEAK ? 1.0f : 0.0f;
  }
  template <class PT>
  __device__ __forceinline__ static float y(const PT& P, int j, float x) {
    if constexpr (kPeak || kGauss || kC0) {
      const float t = x - P.u[j];
      if constexpr (kPeak) return fmaf(t, t, P.b[j]);
      return kC0 ? fabsf(t) : t * t;
    }
    return x;
  }
  // a: the axis' factor of y (not used by the product peak and the polynomial);
  // u: its threshold (the discontinuous family: -inf, whose exponential is 0,
  // from the first coordinate above it)
  // (a slope beyond FP32's range is kept finite there: infinity times a coordinate
  // would make a NaN of the -inf)
  template <class PT>
  __device__ __forceinline__ static float coef(const PT& P, int j) {
    if constexpr (kDisc) return fminf(fmaxf(P.a[j], -3.402823466e38f), 3.402823466e38f);
    return kGauss ? P.b[j] : P.a[j];
  }
  __device__ __forceinline__ static float step(float s, float a, float u, float v) {
    if constexpr (kPeak) return s * v;
    if constexpr (kPoly) return fmaf(v, v, s);
    if constexpr (kDisc) return v > u ? -__int_as_float(0x7f800000) : fmaf(a, v, s);
    return fmaf(a, v, s);
  }
  __device__ __forceinline__ static float2 step2(float2 s, float a, float u, float2 v) {
    if constexpr (kPeak) return __fmul2_rn(s, v);
    if constexpr (kPoly) return __ffma2_rn(v, v, s);
    const float2 r = __ffma2_rn(bc2(a), v, s);
    if constexpr (kDisc) {
      const float ninf = -__int_as_float(0x7f800000);
      return make_float2(v.x > u ? ninf : r.x, v.y > u ? ninf : r.y);
    }
    return r;
  }
  __device__ __forceinline__ static float out(int d, float s) {
    if constexpr (FAM == GMQ_OSCILLATORY) return gcos(s);
    if constexpr (kPeak) return grcp(s);
    if constexpr (FAM == GMQ_CORNER_PEAK) return grcp(ipow(s, d + 1));
    if constexpr (kGauss || kC0) return gexp(-s);
    if constexpr (kDisc) return gexp(s);
    const float s2 = s * s, s4 = s2 * s2, s8 = s4 * s4;
    return s8 * s2 * s;
  }
  // out of N pairs of nodes.  The reciprocal and the cosine have fast forms with
  // the same bits on a range that every integrand in use stays in; one test for
  // all pairs, not one for each, so that their instructions interleave.
  template <int D, int N>
  __device__ __forceinline__ static void outs(float2 (&s)[N]) {
    if constexpr (kPeak || FAM == GMQ_CORNER_PEAK) {
      if constexpr (FAM == GMQ_CORNER_PEAK) {
        // the binary powering of ipow
        constexpr int e = D + 1, low = e & -e;
        float2 r[N];
#pragma unroll
        for (int b = 1; b <= e; b <<= 1) {
#pragma unroll
          for (int n = 0; n < N; ++n) {
            if (b > 1) s[n] = __fmul2_rn(s[n], s[n]);
            if (b == low)
              r[n] = s[n];
            else if (e & b)
              r[n] = __fmul2_rn(r[n], s[n]);
          }
        }
#pragma unroll
        for (int n = 0; n < N; ++n) s[n] = r[n];
      }
      unsigned far = 0u;
      float2 q[N];
#pragma unroll
      for (int n = 0; n < N; ++n) {
        far |= rcpf_far(s[n].x) | rcpf_far(s[n].y);
        q[n] = rcpf2(s[n]);
      }
      if (far) {
#pragma unroll
        for (int n = 0; n < N; ++n) q[n] = make_float2(grcp(s[n].x), grcp(s[n].y));
      }
#pragma unroll
      for (int n = 0; n < N; ++n) s[n] = q[n];
    } else if constexpr (FAM == GMQ_OSCILLATORY) {
      bool near = true;
#pragma unroll
      for (int n = 0; n < N; ++n)
        near = near && fabsf(s[n].x) < 32768.0f && fabsf(s[n].y) < 32768.0f;
      if (near) {
#pragma unroll
        for (int n = 0; n < N; ++n) s[n] = gm_cosf2_near(s[n]);
      } else {
#pragma unroll
        for (int n = 0; n < N; ++n) s[n] = make_float2(gm_cosf(s[n].x), gm_cosf(s[n].y));
      }
    } else if constexpr (kPoly) {
#pragma unroll
      for (int n = 0; n < N; ++n) {
        const float2 s2 = __fmul2_rn(s[n], s[n]), s4 = __fmul2_rn(s2, s2), s8 = __fmul2_rn(s4, s4);
        const float2 p = __fmul2_rn(s8, s2);
        // scalar: the assembler fuses a paired product into the paired addition
        // that takes it (Acc2), rounding mode or not, and the node loses its rounding
        s[n] = make_float2(__fmul_rn(p.x, s[n].x), __fmul_rn(p.y, s[n].y));
      }
    } else {
#pragma unroll
      for (int n = 0; n < N; ++n) s[n] = make_float2(out(D, s[n].x), out(D, s[n].y));
    }
  }
};

// Two compensated FP32 sums side by side (Knuth's TwoSum, paired instructions).
struct Acc2 {
  float2 s = {0.0f, 0.0f}, c = {0.0f, 0.0f};
  __device__ __forceinline__ void add(float2 v) {
    auto neg = [](float2 x) { return make_float2(-x.x, -x.y); };
    const float2 t = __fadd2_rn(s, v);
    const float2 bp = __fadd2_rn(t, neg(s));
    const float2 ap = __fadd2_rn(t, neg(bp));
    c = __fadd2_rn(c, __fadd2_rn(__fadd2_rn(s, neg(ap)), __fadd2_rn(v, neg(bp))));
    s = t;
  }
  // both sums as one (the FP64 pipe adds once: at small D it is what bounds)
  __device__ __forceinline__ Acc<float> one() const {
    Acc<float> a;
    a.s = s.x;
    a.c = __fadd_rn(c.x, c.y);
    a.add(s.y);
    return a;
  }
  __device__ __forceinline__ double value() const { return one().value(); }
  __device__ __forceinline__ double value(const Acc2& b) const {
    Acc<float> x = one();
    const Acc<float> y = b.one();
    x.c = __fadd_rn(x.c, y.c);
    x.add(y.s);
    return x.value();
  }
};

// Dimension D known at compile time (3 <= D <= 16), one thread per region.
// Bound: FP32 issue.  Evaluated node by node a node's chain costs D steps (12 of
// 26 FP32 operations for the corner peak at D = 12), so nodes are walked as a
// tree over the axes in chain order, where those that agree on the first axes
// share the chain so far -- the same operations on the same operands, hence the
// same bits.  Sign patterns: the outer axes' prefixes are kept in registers and
// renewed from the axis that changes on, the last four axes are unrolled to 16
// patterns (30 steps), so a pattern costs two steps instead of D.  Classes 2
// to 4 share the prefix up to the first moved axis (and, for a pair, the
// stretch between the two); only the chain after the last moved axis is walked
// for each.  Nodes come in pairs on the paired FP32 instructions.  Class sums
// are compensated; their compensations round in the order of the nodes, so that
// the walk's class sums differ from the node-by-node kernel's by up to 1e-14 of
// the terms for smooth integrands and 5e-12 where terms cancel or differ in size
// (d = 12, Gaussian 7e-13, cosine 5e-12).
// tab(row, j): the thread's own column of node coordinates, overwritten with
// y of them.  2^20 regions, d = 12 / d = 8: corner peak 4.83 -> 3.54 / 0.477 ->
// 0.386 ms, product peak 4.79 -> 2.98 / 0.482 -> 0.387, Gaussian 4.08 -> 2.95 /
// 0.424 -> 0.347, C0 3.66 -> 2.97 / 0.391 -> 0.349, cosine 5.78 -> 4.65 / 0.618
// -> 0.478, polynomial 3.19 -> 2.32 / 0.417 -> 0.396; up to d = 5 the FP64 differences and weights bound both forms alike.
template <int FAM, int D, class PT, class Tab>
__device__ __forceinline__ void region_mixed_walk(const PT& Pf, const Tab& tab, double ratio,
                                                  RegionSums& o) {
  static_assert(D >= 3 && D <= 16, "the walk needs D >= 3");
  using CH = Chain<FAM>;
  float a[D], yc[D];
#pragma unroll
  for (int j = 0; j < D; ++j) {
    a[j] = CH::coef(Pf, j);
#pragma unroll
    for (int row = 0; row < kXRows; ++row) tab(row, j) = CH::y(Pf, j, tab(row, j));
    yc[j] = tab(kXC, j);
  }
  auto thr = [&](int j) -> float { return CH::kDisc ? Pf.u[j] : 0.0f; };
  // the centres of axes k .. D - 1 appended
  auto rest2 = [&](float2 s, int k) -> float2 {
#pragma unroll
    for (int i = 0; i < D; ++i)
      if (i >= k) s = CH::step2(s, a[i], thr(i), bc2(yc[i]));
    return s;
  };
  const float s0 = CH::init(Pf);
  double dbest = -1.0;
  int kbest = 0;
  // class 1
  float sc = s0;
#pragma unroll
  for (int j = 0; j < D; ++j) sc = CH::step(sc, a[j], thr(j), yc[j]);
  const double f0 = f2d_exact(CH::out(D, sc));
  const double two_f0 = __dmul_rn(2.0, f0);
  // classes 2 and 3: per axis k the pairs (+l2, -l2) and (+l3, -l3), and
  // the fourth difference of axis k
  Acc2 S2, S3, S4, S4b, S5, S5b;  // two chains of sums where nodes come in numbers
  float pre = s0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    float2 v[2] = {
        rest2(CH::step2(bc2(pre), a[k], thr(k), make_float2(tab(kXP2, k), tab(kXM2, k))), k + 1),
        rest2(CH::step2(bc2(pre), a[k], thr(k), make_float2(tab(kXP3, k), tab(kXM3, k))), k + 1)};
    CH::template outs<D>(v);
    const float2 v2 = v[0], v3 = v[1];
    S2.add(v2);
    S3.add(v3);
    const double t1 = __dsub_rn(__dadd_rn(f2d_exact(v2.x), f2d_exact(v2.y)), two_f0);
    const double t2 = __dsub_rn(__dadd_rn(f2d_exact(v3.x), f2d_exact(v3.y)), two_f0);
    const double Dk = fabs(__dsub_rn(t1, __dmul_rn(ratio, t2)));
    if (Dk > dbest) {
      dbest = Dk;
      kbest = k;
    }
    pre = CH::step(pre, a[k], thr(k), yc[k]);
  }
  // class 4: pairs j < k, the two signs on axis j side by side
  pre = s0;
  for (int j = 0; j < D - 1; ++j) {
    const float aj = CH::coef(Pf, j), uj = thr(j);
    float2 q = CH::step2(bc2(pre), aj, uj, make_float2(tab(kXP3, j), tab(kXM3, j)));
#pragma unroll
    for (int k = 1; k < D; ++k) {
      if (k > j) {
        float2 v[2] = {rest2(CH::step2(q, a[k], thr(k), bc2(tab(kXP3, k))), k + 1),
                       rest2(CH::step2(q, a[k], thr(k), bc2(tab(kXM3, k))), k + 1)};
        CH::template outs<D>(v);
        S4.add(v[0]);
        S4b.add(v[1]);
        q = CH::step2(q, a[k], thr(k), bc2(yc[k]));
      }
    }
    pre = CH::step(pre, aj, uj, tab(kXC, j));
  }
  // class 5: O outer axes, bit b of the counter being the sign of axis O - 1 - b;
  // I inner axes unrolled
  constexpr int I = D < 4 ? D : 4, O = D - I;
  float p5[I], m5[I], p[O + 1];
#pragma unroll
  for (int i = 0; i < I; ++i) {
    p5[i] = tab(kXP5, O + i);
    m5[i] = tab(kXM5, O + i);
  }
  p[0] = s0;
  for (unsigned t = 0; t < (1u << O); ++t) {
    const int from = t ? O - __ffs((int)t) : 0;  // the first axis whose sign changed
#pragma unroll
    for (int k = 0; k < O; ++k)
      if (k >= from)
        p[k + 1] = CH::step(p[k], a[k], thr(k), tab((t >> (O - 1 - k)) & 1u ? kXM5 : kXP5, k));
    float2 v[1 << (I - 1)];
    v[0] = CH::step2(bc2(p[O]), a[O], thr(O), make_float2(p5[0], m5[0]));
#pragma unroll
    for (int i = 1; i < I; ++i) {
#pragma unroll
      for (int n = (1 << (i - 1)) - 1; n >= 0; --n) {
        const float2 s = v[n];
        v[2 * n] = CH::step2(s, a[O + i], thr(O + i), bc2(p5[i]));
        v[2 * n + 1] = CH::step2(s, a[O + i], thr(O + i), bc2(m5[i]));
      }
    }
    CH::template outs<D>(v);
#pragma unroll
    for (int n = 0; n < (1 << (I - 1)); n += 2) {
      S5.add(v[n]);
      S5b.add(v[n + 1]);
    }
  }
  o.s1 = f0;
  o.s2 = S2.value();
  o.s3 = S3.value();
  o.s4 = S4.value(S4b);
  o.s5 = S5.value(S5b);
  o.f0 = f0;
  o.dbest = dbest;
  o.kbest = kbest;
}

}  // namespace gmq
