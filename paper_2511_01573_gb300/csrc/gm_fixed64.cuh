// gm_fixed64.cuh -- class sums of one region for the corner peak in 64-bit
// fixed point: the inner sum, its reciprocal and its power on the integer
// pipes.
//
// Bound: GB300 issues an FP64 instruction for a warp once in ~76 cycles per
// SM quarter (1.68 lanes per clock and SM, measured) but a 32 x 32 -> 64 bit
// multiply-add in 4 and an integer add in 1 to 2, so a 64-bit fixed-point
// product (two or three multiply-adds) is some five times cheaper than an
// FP64 one.  A corner-peak node costs 12 FP64 instructions in the separable
// form, ~900 cycles; here it costs about 85 instructions, one of them an FP32
// reciprocal.  d = 8, 2^20 regions, one thread per region: 9.41 -> 1.57 ms (4829
// -> 222 FP64 instructions a region; issue slots 60 % busy, twelve warps an SM).
//
// Scaling: with inv about 1 / (the smallest S of the nodes) (8 significant bits),
// s = S inv lies in (1, 4) and f = inv^(d+1) s^-(d+1).  S is linear in the
// coordinates, so every node's s is an integer sum of the centre's and of
// +-lambda a_k h_k inv in units of 2^-58: exact, whatever the order.  Values u =
// s^-(d+1) < 1 are in units of 2^-64 and class sums are exact 96-bit integers, so
// no lane mapping can change a bit.  Classes 1 to 4, whose nodes move one axis or
// two, and class 5 have an inv each, so that the largest u of the sums is near 1:
// u is rounded to 2^-64 and not to its own size, which with one inv for the whole
// box (S down to a corner that is no node) left f(centre) at d = 16 with 30 bits.
// Errors relative to the sums: 2^-59 per term of s and 2^-60 of 1 / s, both times
// d + 1; of a power 2^-64 per node, whose mean is added back (pow_bias).
// Regions where S is not positive, spans a factor of about 4 or more, or
// leaves no exponent room are evaluated by region_sums64.
#pragma once

#include "gm_region64.cuh"

namespace gmq {

// 2^64 / s for s = v / 2^58 in (1 + 2^-9, 4).  An FP32 reciprocal of the
// leading bits gives y0 (23 bits, relative error below 2^-20); e = 1 - s y0
// follows exactly from the low 64 bits of v Y0, and y0 (1 + e + e^2) leaves
// e^3 < 2^-60.
__device__ __forceinline__ u64 fixed_rcp(i64 v) {
  const float x = __fadd_rn(__uint_as_float((unsigned)(v >> 37) | 0x3f800000u), -1.0f);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  const unsigned y0 = __float_as_uint(__fmaf_rn(r, 0.25f, 1.0f)) & 0x7fffffu;
  const i64 e = -(i64)((u64)v * y0);  // 2^81 (1 - s y0), |e| < 2^61
  const int eh = (int)(e >> 32);
  const i64 c = ((e >> 17) + (i64)((u64)((i64)eh * eh) >> 34)) >> 4;  // 2^60 (e + e^2)
  const i64 t = (i64)((u64)c * y0);                                   // 2^83 y0 (e + e^2)
  return ((u64)y0 << 41) + (u64)(t >> 19);
}

// u[i]^e, e >= 1, by the binary powering of ipow; N values side by side, so
// that the loop's overhead and the products' latency are shared.
template <int N>
__device__ __forceinline__ void fixed_pow(u64 (&u)[N], int e) {
  while (!(e & 1)) {
#pragma unroll
    for (int i = 0; i < N; ++i) u[i] = fixed_sqr(u[i]);
    e >>= 1;
  }
  u64 r[N];
#pragma unroll
  for (int i = 0; i < N; ++i) r[i] = u[i];
  while (e >>= 1) {
#pragma unroll
    for (int i = 0; i < N; ++i) u[i] = fixed_sqr(u[i]);
    if (e & 1) {
#pragma unroll
      for (int i = 0; i < N; ++i) r[i] = fixed_mul(r[i], u[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) u[i] = r[i];
}

// What n powers u^e of fixed_pow lack in the mean, in units of 2^-64: the last
// product drops 5/4 of them (a square 5/6).
__device__ __forceinline__ u64 pow_bias(int n, int e) {
  return (u64)((e & (e - 1)) ? (5 * n + 2) >> 2 : (5 * n + 3) / 6);
}

// inv^e rounded to FP64 (2^-59 beside), inv positive and normal: the classes'
// factors, whose errors do not cancel between them.
__device__ __forceinline__ double pow_rounded(double inv, int e) {
  const int hi = __double2hiint(inv);
  const u64 u = ((u64)((hi & 0xfffff) | 0x100000) << 43) | ((u64)(unsigned)__double2loint(inv) << 11);
  const int x = ((hi >> 20) & 0x7ff) - 1022;  // inv = u 2^(x - 64)
  u64 r = u;
  int rx = x;
  auto times = [&](u64 v, int vx) {
    r = fixed_mul(r, v);
    rx += vx;
    if ((i64)r >= 0) {
      r <<= 1;
      --rx;
    }
  };
  for (int b = 30 - __clz(e); b >= 0; --b) {
    times(r, rx);
    if ((e >> b) & 1) times(u, x);
  }
  return __longlong_as_double((i64)(((u64)(rx + 1021) << 52) + (((r >> 10) + 1) >> 1)));
}

// Sum of 64-bit values in 96 bits.
struct FixedAcc {
  u64 lo = 0;
  unsigned hi = 0;
  __device__ __forceinline__ void add(u64 v) {
    lo += v;
    hi += lo < v ? 1u : 0u;
  }
  __device__ __forceinline__ void add(const FixedAcc& o) {
    add(o.lo);
    hi += o.hi;
  }
  // in units of 2^-64 of the values' scale
  __device__ __forceinline__ double value() const {
    return fma((double)lo, 0x1p-64, (double)hi);
  }
};

// The group's total in every lane.
template <int T>
__device__ __forceinline__ void lanes_add(FixedAcc& x, unsigned mask) {
  if constexpr (T > 32) {
    __shared__ u64 sl[T];
    __shared__ unsigned sh[T];
    const int l = threadIdx.x & (T - 1);
#pragma unroll
    for (int off = T / 2; off >= 32; off >>= 1) {
      __syncthreads();
      sl[l] = x.lo;
      sh[l] = x.hi;
      __syncthreads();
      FixedAcc o;
      o.lo = sl[l ^ off];
      o.hi = sh[l ^ off];
      x.add(o);
    }
  }
  constexpr int W = T < 32 ? T : 32;
#pragma unroll
  for (int off = W / 2; off > 0; off >>= 1) {
    FixedAcc o;
    o.lo = __shfl_xor_sync(mask, x.lo, off, W);
    o.hi = __shfl_xor_sync(mask, x.hi, off, W);
    x.add(o);
  }
}

// Class sums and split axis of one region of the corner peak; arguments as
// region_sums64 (the workspace fits the separable form's: [d] steps of
// lambda3, the class-5 chains, with T > 1 lanes [2d] steps of lambda2 and
// lambda5).  False: the region's S does not fit, and nothing was written to `o` (every lane of the group returns the same).
template <int T, class PT, class CH>
__device__ __forceinline__ bool region_sums64_corner(const PT& P, int d,
                                                     const unsigned short* pairs, const CH& ch,
                                                     double lam2, double lam3, double lam5,
                                                     double* w, int ws, double ratio,
                                                     RegionSums& o) {
  const int lane = (T == 1) ? 0 : (int)(threadIdx.x & (unsigned)(T - 1));
  const unsigned mask = group_mask<T>();
  const int pa = sep_a(d), pb = sep_b(d), pc = sep_c(d);
  const int eA = d, eB = eA + (1 << pa), eC = eB + (pb ? 1 << pb : 0);
  const int e2 = eC + (pc ? 1 << pc : 0), e5 = e2 + d;
  auto W = [&](int e) -> i64& { return reinterpret_cast<i64*>(w)[(long long)e * ws]; };
  // S at the centre as a sum of two doubles (f moves by d + 1 times the
  // relative error of S, all nodes alike, and the FP64 pipe has room) and, in
  // FP32, the reach of the nodes that move one axis or two and of those that move
  // all, by every lane
  double S = 1.0, Slo = 0.0;
  float all = 0.0f, m1 = 0.0f, m2 = 0.0f;  // sum of |a h| and the two largest
  for (int k = 0; k < d; ++k) {
    double c, h;
    ch(k, c, h);
    const double p = __dmul_rn(P.a[k], c);
    const double t = __dadd_rn(S, p);
    Slo = __dadd_rn(Slo, __dadd_rn(fma(P.a[k], c, -p), __dsub_rn(p, __dsub_rn(t, S))));
    S = t;
    const float ah = abs_f32(P.a[k]) * abs_f32(h);
    all += ah;
    m2 = fmaxf(m2, fminf(m1, ah));
    m1 = fmaxf(m1, ah);
  }
  const float Sf = __double2float_rn(S);
  // inv: the leading 8 bits of 1 / (S - reach), rounded up, so that s > 1; v: s of
  // the centre.  False: s does not fit.
  auto scale = [&](float reach, double& inv, i64& v) -> bool {
    const float smin = Sf - reach;
    const unsigned ex = __float_as_uint(smin) >> 23;  // sign and exponent
    if (ex - (127u - 40u) > 80u) return false;  // not in [2^-40, 2^41): negative, 0, NaN
    // (two units of the eighth bit above the truncated quotient put the
    // smallest s between 1 + 2^-8 and 1 + 2^-6, less 2^-20 for the reach)
    const float q =
        __uint_as_float((__float_as_uint(__fdiv_rn(1.0f, smin)) & 0xffff0000u) + 0x20000u);
    inv = f2d_exact(q);
    const double s0 = __dmul_rn(S, inv);
    v = to_fixed(s0, 58) + to_fixed(fma(Slo, inv, fma(S, inv, -s0)), 58);
    return (Sf + reach) * q < 3.98f;
  };
  double inv, inv5;
  i64 v0, v05;
  if (!scale((float)lam3 * (m1 + m2), inv, v0) || !scale((float)lam5 * all, inv5, v05)) return false;
  const int e = d + 1;
  // 2^64 s^-(d+1) of the nodes at s = v 2^-58
  auto nodes = [&](auto& v) {
#pragma unroll
    for (auto& x : v) x = fixed_rcp((i64)x);
    fixed_pow(v, e);
  };
  const double l2 = __dmul_rn(lam2, inv), l3 = __dmul_rn(lam3, inv), l5 = __dmul_rn(lam5, inv5);
  auto steps = [&](int k, i64& g2, i64& g3, i64& g5) {
    double c, h;
    ch(k, c, h);
    const double t = __dmul_rn(P.a[k], h);
    g2 = to_fixed(__dmul_rn(l2, t), 58);
    g3 = to_fixed(__dmul_rn(l3, t), 58);
    g5 = to_fixed(__dmul_rn(l5, t), 58);
  };
  u64 c0[1] = {(u64)v0};
  nodes(c0);
  const u64 u0 = c0[0];
  FixedAcc s2, s3, s4, s5;
  double dbest = -1.0;
  int kbest = 0;
  // the four nodes of axis k and its fourth difference (second differences in
  // units of 2^-62)
  auto axis = [&](int k, i64 g2, i64 g3) {
    u64 u[4] = {(u64)(v0 + g2), (u64)(v0 - g2), (u64)(v0 + g3), (u64)(v0 - g3)};
    nodes(u);
    s2.add(u[0]);
    s2.add(u[1]);
    s3.add(u[2]);
    s3.add(u[3]);
    const i64 d2 = (i64)(u[0] >> 2) + (i64)(u[1] >> 2) - (i64)(u0 >> 1);
    const i64 d3 = (i64)(u[2] >> 2) + (i64)(u[3] >> 2) - (i64)(u0 >> 1);
    const double D = fabs(__dsub_rn((double)d2, __dmul_rn(ratio, (double)d3)));
    if (D > dbest) {
      dbest = D;
      kbest = k;
    }
  };
  if constexpr (T == 1) {
    for (int k = 0; k < d; ++k) {
      i64 g2, g3, g5;
      steps(k, g2, g3, g5);
      W(k) = g3;
      axis(k, g2, g3);
      // the part's class-5 chains, by doubling (A's headed by the centre)
      const int e0 = k < pa ? eA : (k < pa + pb ? eB : eC);
      const int i = k < pa ? k : (k < pa + pb ? k - pa : k - pa - pb);
      if (i == 0) {
        const i64 head = k ? 0 : v05;
        W(e0) = head + g5;
        W(e0 + 1) = head - g5;
      } else {
        const int n = 1 << i;
        for (int t = 0; t < n; ++t) {
          const i64 v = W(e0 + t);
          W(e0 + t + n) = v - g5;
          W(e0 + t) = v + g5;
        }
      }
    }
  } else {
    for (int k = lane; k < d; k += T) {
      i64 g2, g3, g5;
      steps(k, g2, g3, g5);
      W(k) = g3;
      W(e2 + k) = g2;
      W(e5 + k) = g5;
      axis(k, g2, g3);
    }
    group_sync<T>(mask);
    const int nA = 1 << pa, nB = pb ? 1 << pb : 0, nC = pc ? 1 << pc : 0;
    for (int t = lane; t < nA + nB + nC; t += T) {
      int q0 = t, e0 = eA, j0 = 0, nb = pa;
      i64 v = v05;
      if (q0 >= nA) {
        q0 -= nA;
        e0 = eB;
        j0 = pa;
        nb = pb;
        v = 0;
        if (q0 >= nB) {
          q0 -= nB;
          e0 = eC;
          j0 = pa + pb;
          nb = pc;
        }
      }
      for (int i = 0; i < nb; ++i) {
        const i64 g5 = W(e5 + j0 + i);
        v += ((q0 >> i) & 1) ? -g5 : g5;
      }
      W(e0 + q0) = v;
    }
    group_sync<T>(mask);
    lanes_argmax<T>(dbest, kbest, mask);
  }
  // class 4
  const int np = d * (d - 1) / 2;
  for (int p = lane; p < np; p += T) {
    const unsigned pr = pairs[p];
    const i64 gj = W((int)(pr >> 8)), gk = W((int)(pr & 255u));
    u64 u[4] = {(u64)(v0 + gj + gk), (u64)(v0 + gj - gk), (u64)(v0 - gj + gk),
                (u64)(v0 - gj - gk)};
    nodes(u);
#pragma unroll
    for (int q = 0; q < 4; ++q) s4.add(u[q]);
  }
  // class 5: T = 1 walks stretches of A with the rest of the sum fixed
  if constexpr (T == 1) {
    const int nlo = 1 << pa, nhi = 1 << (d - pa), bm = (1 << pb) - 1;
    for (int hi = 0; hi < nhi; ++hi) {
      i64 bc = pb ? W(eB + (hi & bm)) : 0;
      if (pc) bc += W(eC + (hi >> pb));
      if (nlo >= 4) {
        for (int q = 0; q < nlo; q += 4) {
          u64 u[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) u[i] = (u64)(W(eA + q + i) + bc);
          nodes(u);
#pragma unroll
          for (int i = 0; i < 4; ++i) s5.add(u[i]);
        }
      } else {  // d <= 2: A has two entries
        u64 u[2] = {(u64)(W(eA) + bc), (u64)(W(eA + 1) + bc)};
        nodes(u);
        s5.add(u[0]);
        s5.add(u[1]);
      }
    }
  } else {
    const int am = (1 << pa) - 1, bm = (1 << pb) - 1;
    for (int m = lane; m < (1 << d); m += T) {
      i64 v = W(eA + (m & am));
      if (pb) v += W(eB + ((m >> pa) & bm));
      if (pc) v += W(eC + (m >> (pa + pb)));
      u64 u[1] = {(u64)v};
      nodes(u);
      s5.add(u[0]);
    }
    lanes_add<T>(s2, mask);
    lanes_add<T>(s3, mask);
    lanes_add<T>(s4, mask);
    lanes_add<T>(s5, mask);
  }
  s2.add(pow_bias(2 * d, e));
  s3.add(pow_bias(2 * d, e));
  s4.add(pow_bias(4 * np, e));
  s5.add(pow_bias(1 << d, e));
  const double F = pow_rounded(inv, e), F5 = pow_rounded(inv5, e);
  o.s1 = __dmul_rn(F, __dmul_rn((double)(u0 + 1), 0x1p-64));
  o.s2 = __dmul_rn(F, s2.value());
  o.s3 = __dmul_rn(F, s3.value());
  o.s4 = __dmul_rn(F, s4.value());
  o.s5 = __dmul_rn(F5, s5.value());
  o.f0 = o.s1;
  o.dbest = __dmul_rn(__dmul_rn(F, 0x1p-62), dbest);
  o.kbest = kbest;
  return true;
}

}  // namespace gmq
