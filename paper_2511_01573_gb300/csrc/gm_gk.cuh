// gm_gk.cuh -- the tensor-product Gauss-Kronrod (7, 15) rule (paper Sec. 3
// names a tensor-product Gauss-Kronrod rule as one of the rules the method
// can use, without its order or split axis -- the readings here are the
// classic G7/K15 pair and the directional error estimates).
//
// On a region c +- h the rule evaluates f at the 15^d nodes c + h o xi,
// xi in {K15 nodes}^d, and forms
//   I_K = prod h_k sum_i (prod_k wK[i_k]) f,   I_G likewise with the G7
//   weights (0 at the 8 Kronrod-only nodes),   eps = |I_K - I_G|,
//   E_k = prod h_k |sum_i (prod_{j != k} wK[i_j]) (wK[i_k] - wG[i_k]) f|,
// the error estimate in direction k; the split axis is argmax_k E_k (lowest
// index on ties), or the widest axis when every E_k is below 1e-11 of the
// magnitude of the terms (prod h_k sum |wK f|).  d <= GMQ_GK_MAX_DIM.
//
// Mapping: a 128-thread block per region for d >= 4 (3375 rows and more), a
// warp per region below.  The node grid is walked by rows -- a row fixes the
// digits of axes 1..d-1 and runs axis 0 over its 15 nodes -- lane l of the L
// lanes of a region taking rows l, l + L, ...  Butterflies, then a fixed
// order over the warps, combine the lanes' sums.
//
// Bound: the FP64 pipe with f evaluated at every node, ~25 instructions a node.
// Integrands that are products of one factor per axis (gm_factor64.cuh) hold
// wK e for the 15 nodes of every axis, relative to the centre's value; a row is
// the product of its digits' entries, and each node two products (its terms of
// I_K and of E_0), three integer multiply-adds each.  Row sums
// give the E_k of the other axes.  The nodes of I_G are the 7^d with odd
// digits; they are walked on their own, because a lane that skips the term
// saves nothing when another lane of its warp needs it.  f >= 0 for these
// integrands, so sum |wK f| is I_K's sum.  d = 4, C0, 2500 regions: 6.57 ->
// 0.27 ms (0.71 with FP64 products).  Other integrands, and regions whose
// factors lack exponent room, evaluate f at every node.
#pragma once

#include "gm_factor64.cuh"
#include "gmq_common.cuh"
#include "gmq_families.cuh"

namespace gmq {

// 1-D tables on [-1, 1], ascending nodes; wg = 0 at Kronrod-only nodes;
// r = 1 - wg / wk.
struct GkConst {
  double x[15], wk[15], wg[15], r[15];
};

// Computed once on the host (gmq_api.cu); each context keeps a device copy.
const GkConst& gk_const();

struct GkArgs {
  RuleArgs A;
  const GkConst* K;  // device copy of the tables
};

constexpr int kGkBlock = 128;

// Sums of one region: I_K, I_G, sum |wK f| and the directional terms,
// without the factor prod h_k.
struct GkSums {
  double K = 0.0, G = 0.0, A = 0.0;
  double E[GMQ_GK_MAX_DIM];
};

// Combine the sums of the region's 32 W lanes in a fixed order: every lane
// of the region's first warp returns the total (of A unless it is K's).  scratch:
// [W][9].  SOME: leave out the sums that a dimension lacks (with f at every node
// the adds cost nothing that the tests for them would not).
template <int W, bool SOME>
__device__ __forceinline__ void gk_combine(GkSums& s, int d, bool a_is_k, double* scratch) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    s.K += __shfl_xor_sync(0xffffffffu, s.K, off);
    s.G += __shfl_xor_sync(0xffffffffu, s.G, off);
    if (!SOME || !a_is_k) s.A += __shfl_xor_sync(0xffffffffu, s.A, off);
#pragma unroll
    for (int k = 0; k < GMQ_GK_MAX_DIM; ++k)
      if (!SOME || k < d) s.E[k] += __shfl_xor_sync(0xffffffffu, s.E[k], off);
  }
  if constexpr (W > 1) {
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      double* o = scratch + w * (3 + GMQ_GK_MAX_DIM);
      o[0] = s.K;
      o[1] = s.G;
      o[2] = s.A;
#pragma unroll
      for (int k = 0; k < GMQ_GK_MAX_DIM; ++k)
        if (!SOME || k < d) o[3 + k] = s.E[k];
    }
    __syncthreads();
    if (w == 0) {
      for (int v = 1; v < W; ++v) {
        const double* o = scratch + v * (3 + GMQ_GK_MAX_DIM);
        s.K += o[0];
        s.G += o[1];
        if (!SOME || !a_is_k) s.A += o[2];
#pragma unroll
        for (int k = 0; k < GMQ_GK_MAX_DIM; ++k)
          if (!SOME || k < d) s.E[k] += o[3 + k];
      }
    }
  }
}

// f at every node.  xt: node coordinates [d][15]; xs: this lane's current
// node, entries 32 W apart.
template <int FAM, int W>
__device__ __forceinline__ void gk_sums_nodes(const SmemParams<double>& P, const GkConst& K, int d,
                                              int lane, const double* xt, double* xs, GkSums& s) {
  constexpr int L = 32 * W;
  int rows = 1;
  for (int k = 1; k < d; ++k) rows *= 15;
  auto X = [&](int j) -> double { return xs[j * L]; };
  for (int row = lane; row < rows; row += L) {
    // digits of axes 1..d-1, their weight products and coordinates
    int q = row;
    double wr = 1.0, gr = 1.0;
    int dig[GMQ_GK_MAX_DIM];
#pragma unroll
    for (int k = 1; k < GMQ_GK_MAX_DIM; ++k) {
      if (k < d) {
        dig[k] = q % 15;
        q /= 15;
        wr = wr * K.wk[dig[k]];
        gr = gr * K.wg[dig[k]];
        xs[k * L] = xt[k * 15 + dig[k]];
      }
    }
    double rk = 0.0, rg = 0.0, ra = 0.0, e0 = 0.0;
    for (int j = 0; j < 15; ++j) {
      xs[0] = xt[j];
      const double v = Family<FAM>::template eval<double>(P, d, X);
      const double t = __dmul_rn(__dmul_rn(K.wk[j], wr), v);  // wK-product * f
      rk = __dadd_rn(rk, t);
      rg = fma(__dmul_rn(K.wg[j], gr), v, rg);
      ra = fma(__dmul_rn(K.wk[j], wr), fabs(v), ra);
      e0 = fma(K.r[j], t, e0);
    }
    s.K = __dadd_rn(s.K, rk);
    s.G = __dadd_rn(s.G, rg);
    s.A = __dadd_rn(s.A, ra);
    s.E[0] = __dadd_rn(s.E[0], e0);
#pragma unroll
    for (int k = 1; k < GMQ_GK_MAX_DIM; ++k)
      if (k < d) s.E[k] = fma(K.r[dig[k]], rk, s.E[k]);
  }
}

// An axis entry of a row's product: 64-bit mantissa (the 53 bits of a double at
// the top) and its biased exponent in the low eleven bits; 0 for 0.  Kept in
// integer registers throughout: as a double it can be a signalling NaN, which a
// select of doubles was seen to quieten.
__device__ __forceinline__ u64 gk_word(double v) {
  const u64 b = (u64)__double_as_longlong(v);
  if (b << 1 == 0) return 0;
  return ((b << 11) | 0x8000000000000000ull) + ((b >> 52) & 0x7ff);
}

// The same from per-axis factors, relative to F.  kt: wK e [d][15], axis 0's and
// rt's (r wK e of axis 0 [15]) as limbs (gm_factor64.cuh) below 2^E[0] and 2^(E[0]
// + 1), the other axes' as gk_word; gt: wG e [d][15].  Every row's product has its
// own exponent: rounded to one bound for all, 15^5 rows of which a few are large
// put I_K of d = 6 up to 3e-12 off.  A row's product, the node products and sums
// run on the integer pipes; a row leaves the FP64 pipe its sum's conversion and
// the E_k of the other axes.
template <int W>
__device__ __forceinline__ void gk_sums_factors(const GkConst& K, int d, int lane,
                                                const double* kt, const double* gt,
                                                const double* rt, const int* E, GkSums& s) {
  constexpr int L = 32 * W;
  int rows = 1, grows = 1, Er = 0;
  for (int k = 1; k < d; ++k) {
    rows *= 15;
    grows *= 7;
    Er += E[k];
  }
  int lk = 0, lr = 0;  // sums of the low limbs, whose products a row adds at once
#pragma unroll
  for (int j = 0; j < 15; ++j) {
    lk += limbs_unpack(kt[j]).l;
    lr += limbs_unpack(rt[j]).l;
  }
  LimbSum sk, se;
  for (int row = lane; row < rows; row += L) {
    int q = row, x = 0;
    u64 m = 0;
    int dig[GMQ_GK_MAX_DIM];
#pragma unroll
    for (int k = 1; k < GMQ_GK_MAX_DIM; ++k) {
      if (k < d) {
        dig[k] = q % 15;
        q /= 15;
        const u64 w = reinterpret_cast<const u64*>(kt)[k * 15 + dig[k]];
        const u64 v = w & ~0x7ffull;
        x += (int)(w & 0x7ff) - 1022;
        m = k == 1 ? v : fixed_mul(m, v);
      }
    }
    // m 2^(x - 64) as limbs times 2^x (at most d - 2 <= 4 leading zeros)
    Limbs kr{1 << 26, 0};
    if (d > 1) {
      const int lz = __clz((int)(m >> 32));
      m <<= lz;
      x -= lz;
      kr = limbs_split((i64)(m >> 11) + (i64)((m >> 10) & 1));
    }
    LimbAcc rk, re;
#pragma unroll
    for (int j = 0; j < 15; ++j) {
      rk.add_split(limbs_unpack(kt[j]), kr);
      re.add_split(limbs_unpack(rt[j]), kr);
    }
    rk.mid += ((i64)lk * kr.l) >> 27;
    re.mid += ((i64)lr * kr.l) >> 27;
    const i64 nk = rk.number();
    double v = (double)nk;
    if (nk != 0) v = __hiloint2double(__double2hiint(v) + (int)((unsigned)x << 20), __double2loint(v));
#pragma unroll
    for (int k = 1; k < GMQ_GK_MAX_DIM; ++k)
      if (k < d) s.E[k] = fma(K.r[dig[k]], v, s.E[k]);
    sk.add_scaled(nk, Er - x);
    se.add_scaled(re.number(), Er - x);
  }
  // numbers are in units of 2^(E0 + x - 53), sums in 2^(E0 + Er - 101)
  s.K = sk.value(E[0] + Er - 22);
  s.E[0] = se.value(E[0] + 1 + Er - 22);
  const double unit = __hiloint2double((970 + E[0]) << 20, 0);  // 2^(E0 - 53)
#pragma unroll
  for (int k = 1; k < GMQ_GK_MAX_DIM; ++k) s.E[k] = __dmul_rn(unit, s.E[k]);
  for (int row = lane; row < grows; row += L) {
    int q = row;
    double gr = 1.0;
#pragma unroll
    for (int k = 1; k < GMQ_GK_MAX_DIM; ++k) {
      if (k < d) {
        const double v = gt[k * 15 + 2 * (q % 7) + 1];
        q /= 7;
        gr = k == 1 ? v : __dmul_rn(gr, v);
      }
    }
    double rg = __dmul_rn(gt[1], gr);
#pragma unroll
    for (int j = 3; j < 15; j += 2) rg = fma(gt[j], gr, rg);
    s.G = __dadd_rn(s.G, rg);
  }
}

// W warps per region, kGkBlock / (32 W) regions per block.
template <int FAM, int W>
__global__ void __launch_bounds__(kGkBlock) k_rule_gk(const GkArgs G) {
  using SF = Sep<FAM>;
  constexpr int L = 32 * W, RB = kGkBlock / L;
  constexpr bool kFactors = Fac<FAM>::kind == kReal;
  constexpr int NT = GMQ_GK_MAX_DIM * 15;
  __shared__ GkConst K;
  __shared__ SmemParams<double> P;
  __shared__ double xt[RB][NT];                      // node coordinates per axis
  __shared__ double xs[RB][GMQ_GK_MAX_DIM * L];      // each lane's current node
  __shared__ double ft[RB][kFactors ? 2 * NT + 15 : 1];
  __shared__ int room[RB][GMQ_GK_MAX_DIM];
  __shared__ int bound[RB][GMQ_GK_MAX_DIM];  // high word of the axis' largest wK e, then its bound
  __shared__ double scratch[W * (3 + GMQ_GK_MAX_DIM)];
  const RuleArgs& A = G.A;
  const int d = A.P.d;
  const int tid = threadIdx.x, w = tid / L, lane = tid % L;
  for (int i = tid; i < 60; i += blockDim.x) (&K.x[0])[i] = (&G.K->x[0])[i];
  for (int j = tid; j < d; j += blockDim.x) {
    P.a[j] = A.P.a[j];
    P.u[j] = A.P.u[j];
    P.b[j] = A.P.b[j];
  }
  if (tid == 0) P.c0 = A.P.c0;
  if (lane < GMQ_GK_MAX_DIM) room[w][lane] = bound[w][lane] = 0;
  __syncthreads();
  const int64_t r = (int64_t)blockIdx.x * RB + w;
  const bool active = r < A.n;
  double* kt = ft[w];
  double* gt = kt + NT;
  double* rt = gt + NT;
  if (active)
    for (int q = lane; q < d * 15; q += L) {
      const int k = q / 15, j = q - 15 * k;
      const double c = A.c[(int64_t)k * A.ld + r];
      const double x = fma(K.x[j], A.h[(int64_t)k * A.ld + r], c);
      xt[w][q] = x;
      if constexpr (kFactors) {
        double e = one_factor<FAM>(P, k, c, A.h[(int64_t)k * A.ld + r], SF::phi(P, k, c), K.x[j]);
        atomicMax(&room[w][k], exp_magnitude(e));
        if constexpr (SF::kFlag) {
          if (SF::flag(P, k, x)) e = 0.0;
        }
        const double ke = __dmul_rn(K.wk[j], e);
        kt[q] = ke;
        atomicMax(&bound[w][k], __double2hiint(ke));
        gt[q] = __dmul_rn(K.wg[j], e);
        if (k == 0) rt[j] = __dmul_rn(K.r[j], ke);
      }
    }
  __syncthreads();
  if constexpr (kFactors) {
    if (active && lane < d) bound[w][lane] = exp_bound(__hiloint2double(bound[w][lane], 0));
    __syncthreads();
    if (active) {
      for (int q = lane; q < 15; q += L) kt[q] = limbs_even(kt[q], bound[w][0]);
      for (int q = 15 + lane; q < d * 15; q += L)
        reinterpret_cast<u64*>(kt)[q] = gk_word(kt[q]);
      for (int j = lane; j < 15; j += L) rt[j] = limbs_even(rt[j], bound[w][0] + 1);
    }
    __syncthreads();
  }
  if (!active) return;  // the whole warp (W = 1): its lanes share the region
  GkSums s;
#pragma unroll
  for (int k = 0; k < GMQ_GK_MAX_DIM; ++k) s.E[k] = 0.0;
  double F = 1.0;
  bool factors = false;
  if constexpr (kFactors) {
    Centre<FAM> top;
    int big = 0;
    for (int k = 0; k < d; ++k) {
      const double c = A.c[(int64_t)k * A.ld + r];
      top.add(P, k, c, SF::phi(P, k, c));
      big += room[w][k];
    }
    F = top.value(d);
    factors = big <= kFacExpRoom && exp_magnitude(F) <= kFacExpRoom;
    if (factors)
      gk_sums_factors<W>(K, d, lane, kt, gt, rt, bound[w], s);
    else
      F = 1.0;
  }
  if (!factors) gk_sums_nodes<FAM, W>(P, K, d, lane, xt[w], xs[w] + lane, s);
  gk_combine<W, kFactors>(s, d, factors, scratch);
  if (lane != 0) return;
  if (factors) s.A = s.K;
  s.K = __dmul_rn(F, s.K);
  s.G = __dmul_rn(F, s.G);
  s.A = __dmul_rn(F, s.A);
#pragma unroll
  for (int k = 0; k < GMQ_GK_MAX_DIM; ++k) s.E[k] = __dmul_rn(F, s.E[k]);
  double hprod = 1.0, vol = 1.0;
  for (int k = 0; k < d; ++k) {
    const double hk = A.h[(int64_t)k * A.ld + r];
    hprod = __dmul_rn(hprod, hk);
    vol = __dmul_rn(vol, __dmul_rn(2.0, hk));
  }
  const double ik = __dmul_rn(hprod, s.K), ig = __dmul_rn(hprod, s.G);
  const double scale = __dmul_rn(hprod, s.A);
  int best = 0;
  double eb = __dmul_rn(hprod, fabs(s.E[0]));
#pragma unroll
  for (int k = 1; k < GMQ_GK_MAX_DIM; ++k) {
    if (k < d) {
      const double ek = __dmul_rn(hprod, fabs(s.E[k]));
      if (ek > eb) {
        eb = ek;
        best = k;
      }
    }
  }
  int ax = best;
  if (!(eb > __dadd_rn(__dmul_rn(1e-11, scale), 1e-300))) {
    ax = 0;
    double hb = A.h[r];
    for (int k = 1; k < d; ++k) {
      const double hk = A.h[(int64_t)k * A.ld + r];
      if (hk > hb) {
        hb = hk;
        ax = k;
      }
    }
  }
  const double cs = A.c[(int64_t)ax * A.ld + r];
  const double hh = __dmul_rn(0.5, A.h[(int64_t)ax * A.ld + r]);
  const bool bad = (hh == 0.0) || (__dsub_rn(cs, hh) == cs) || (__dadd_rn(cs, hh) == cs);
  A.i7[r] = ik;
  A.err[r] = fabs(__dsub_rn(ik, ig));
  if (A.volfrac) A.volfrac[r] = __ddiv_rn(vol, A.R.vol_omega);
  A.axis[r] = (uint8_t)(ax | (bad ? 0x80 : 0));
}

template <int FAM, int W>
cudaError_t launch_rule_gk_warps(const GkArgs& G, cudaStream_t s) {
  constexpr int RB = kGkBlock / (32 * W);
  const int64_t blocks = (G.A.n + RB - 1) / RB;
  if (blocks == 0) return cudaSuccess;
  k_rule_gk<FAM, W><<<(unsigned)blocks, kGkBlock, 0, s>>>(G);
  return cudaGetLastError();
}

// A block per region from d = 4 on: 3375 rows are 27 turns of 128 lanes (225
// rows of d = 3 would leave the last of two turns 3/4 empty).
template <int FAM>
cudaError_t launch_rule_gk_family(const GkArgs& G, cudaStream_t s) {
  return G.A.P.d >= 4 ? launch_rule_gk_warps<FAM, 4>(G, s) : launch_rule_gk_warps<FAM, 1>(G, s);
}

#define GMQ_DEFINE_GK_FAMILY(FAMV) \
  template cudaError_t launch_rule_gk_family<FAMV>(const GkArgs& G, cudaStream_t s);

}  // namespace gmq
