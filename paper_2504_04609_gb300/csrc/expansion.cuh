// Kernel apply of the squared-distance grid cost by block expansions (FP32, log domain).
//
//   out_i = log2 sum_j 2^(in_j - (xt_i - xt_j)^2),   xt sorted
//
// needs no n^2 exponentials: a sum of Gaussians is smooth in x_i (the idea of the fast Gauss
// transform, Greengard & Strain, SIAM J. Sci. Stat. Comput. 12, 1991).  The bins are cut into nb
// blocks of b consecutive bins with centres c_J; with D = c_I - c_J, di = xt_i - c_I, dj = xt_j - c_J
//   in_j - (xt_i - xt_j)^2 = [in_j - dj^2 + 2 D dj] - D^2 - [2 D di + di^2] + 2 di dj.
// The two brackets are a factor per column and one per row, exact and in the log domain whatever D
// is (the classical expansion about the source centre loses all relative precision far from it,
// where a log-domain potential may still make the block the largest).  Only 2^(2 di dj) couples row
// and column, and with block half-widths h <= EX_HMAX its exponent is at most 0.75 in natural units,
// so the polynomial of degree 7 in di dj whose relative error is smallest (1.9e-8, below FP32's
// 6e-8) replaces it:
//   moments   M_IJ,m = sum_j 2^(in_j - A_J - dj^2 + 2 D dj) dj^m            (m = 0..7, per block pair)
//   rows      out_i  = log2 sum_J 2^(A_J - D^2 - 2 D di) sum_m c_m M_IJ,m di^m - di^2.
// Cost per row: about 2 nb (8 multiply-adds + 1 exponential) against n exponentials; nb grows with
// the grid's length in kernel widths, 0.68 (xt_max - xt_min), not with n: 9 blocks at eps = 1e-2 on
// [0, 1], 12 at 5e-3, 18 at 2e-3.
//
// Ranges: A_J is the block's largest in_j - dj^2 rounded up to an integer, D^2 is split into an
// integer and a fraction, and a row block's reference R_I is an integer, so differences of large
// potentials are exact and every rounding is relative to an exponent near 0.  The column factor
// spans 2 |D| h <= 72 around 1 (ex_plan refuses longer grids), so a term lost to underflow is 2^-50
// of its block's sum.  Block pairs whose every term is below 2^-42 of every sum of the row block are
// left out (n of them change a sum by less than its FP32 rounding for n < 2^17).
#pragma once

#include "exp_api.h"
#include "kernels.cuh"

namespace otlm {

constexpr int EX_M = 8;              // moments per block pair
constexpr int EX_NB = 32;            // most blocks (a 32-bit mask of column blocks per row block)
constexpr int EX_MIN_N = 128;        // below this a row of n exponentials costs no more
constexpr float EX_HMAX = 0.7355f;   // half-width with 2 ln2 h^2 = 0.75
constexpr float EX_TILT = 72.f;      // bound of 2 |D| h
constexpr float EX_SKIP = 42.f;      // log2 units below which a block pair is left out

// Shared-memory scratch (floats) of the apply by `warps` warps: centres, block maxima, row references,
// masks, then EX_M coefficients per block pair of a round (four row blocks per warp).
constexpr int EX_HEAD = 4 * EX_NB;
__host__ __device__ constexpr int ex_scratch_floats(int warps) {
  return EX_HEAD + EX_M * EX_NB * (4 * warps < EX_NB ? 4 * warps : EX_NB);
}
// Groups of (up to) four row blocks a round may take with `floats` of scratch.
__device__ __forceinline__ int ex_round_groups(int warps, int nb, int floats) {
  return min(warps, (floats - EX_HEAD) / (EX_M * 4 * nb));
}

__device__ __forceinline__ float ex_quantum(float x0, float x1) {
  const int e = (__float_as_int(fmaxf(fabsf(x0), fabsf(x1))) >> 23) & 255;
  return __int_as_float((max(e, 20) - 18) << 23);
}
__device__ __forceinline__ float ex_center(const float* xt, int J, int b, int n, float q) {
  const float x0 = xt[J * b], x1 = xt[min(n, (J + 1) * b) - 1];
  return rintf(0.5f * (x0 + x1) / q) * q;
}

// The fewest equal blocks that satisfy the bounds (one full warp; `sorted` uniform).
__device__ __forceinline__ ExPlan ex_plan_warp(const float* xt, int n, bool sorted) {
  const int lane = threadIdx.x & 31;
  ExPlan pl{0, 0, 1.f};
  if (!sorted || n < EX_MIN_N) return pl;
  const float x0 = xt[0], x1 = xt[n - 1], len = fabsf(x1 - x0);
  if (!(len <= 2.f * EX_HMAX * EX_NB)) return pl;
  const float q = ex_quantum(x0, x1);
  for (int nb = max(1, (int)(len / (2.f * EX_HMAX))); nb <= EX_NB; ++nb) {
    const int b = max(32, ((n + nb - 1) / nb + 7) / 8 * 8), cnt = (n + b - 1) / b;
    bool ok = true;
    if (lane < cnt) {
      const float c = ex_center(xt, lane, b, n, q);
      const float h = fmaxf(fabsf(xt[lane * b] - c), fabsf(xt[min(n, (lane + 1) * b) - 1] - c));
      ok = h <= EX_HMAX && 2.f * len * h <= EX_TILT;
    }
    if (__all_sync(0xffffffffu, ok)) {
      pl.b = b; pl.nb = cnt; pl.q = q;
      return pl;
    }
  }
  return pl;
}

// Block-wide: is xt[0..n) monotone?  (Every thread of the CTA; a NaN fails both tests.)
__device__ __forceinline__ bool ex_sorted(const float* xt, int n) {
  bool up = true, down = true;
  for (int j = threadIdx.x; j + 1 < n; j += blockDim.x) {
    const float a = xt[j], b = xt[j + 1];
    up &= b >= a;
    down &= b <= a;
  }
  const bool u = __syncthreads_and(up), d = __syncthreads_and(down);
  return u || d;
}

__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// powers (1, v), (v^2, v^3), (v^4, v^5), (v^6, v^7)
__device__ __forceinline__ void ex_powers(float v, uint64_t (&p)[4]) {
  const float v2 = v * v;
  const uint64_t s = f2_pack(v2, v2);
  p[0] = f2_pack(1.f, v);
  p[1] = f2_mul(p[0], s);
  p[2] = f2_mul(p[1], s);
  p[3] = f2_mul(p[2], s);
}
// One warp: moments of the column blocks J0 + (lane / L) for G consecutive row blocks, L lanes per
// column block; d2[g] = 2 D of the lane's column block, [j0, j1) its bins (empty: zeros).  Lanes take
// bins L apart; the powers of dj are shared by the G row blocks.  The 8 G totals over L lanes are
// formed by a transposing butterfly (31 shuffles for L = 32, 28 for L = 8, whose four column blocks
// share them); those of the first gs row blocks are stored at cf[(g nb + J) * 8 + m].
template <int G, int L>
__device__ __forceinline__ void ex_moments(const float* in_s, const float* xt, int j0, int j1, float cJ, float aJ,
                                           const float (&d2)[G], float* cf, int nb, int J, int gs) {
  using P = Prec<float>;
  const int lane = threadIdx.x & 31, l = lane % L;
  uint64_t acc[G][4];
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[g][k] = 0ull;
#pragma unroll 2
  for (int j = j0 + l; j < j1; j += L) {
    const float v = xt[j] - cJ;
    const float h = fmaf(-v, v, in_s[j] - aJ);
    uint64_t p[4];
    ex_powers(v, p);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float w = P::exp2(fmaf(d2[g], v, h));
      const uint64_t w2 = f2_pack(w, w);
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[g][k] = f2_fma(w2, p[k], acc[g][k]);
    }
  }
  float r[32];
#pragma unroll
  for (int g = 0; g < 4; ++g)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (g < G) f2_unpack(acc[g < G ? g : 0][k], r[8 * g + 2 * k], r[8 * g + 2 * k + 1]);
      else r[8 * g + 2 * k] = r[8 * g + 2 * k + 1] = 0.f;
    }
#pragma unroll
  for (int s = L / 2, c = 16; s > 0; s >>= 1, c >>= 1) {
    const bool up = lane & s;
#pragma unroll
    for (int q = 0; q < c; ++q) {
      const float keep = up ? r[q + c] : r[q], give = up ? r[q] : r[q + c];
      r[q] = keep + __shfl_xor_sync(0xffffffffu, give, s);
    }
  }
  if constexpr (L == 32) {  // lane g * 8 + m holds M_g,m
    if ((lane >> 3) < gs) cf[((lane >> 3) * nb + J) * EX_M + (lane & 7)] = r[0];
  } else {  // lane 2 g + m / 4 of the eight holds M_g,m .. M_g,m+3
    static_assert(L == 8, "eight or 32 lanes per column block");
    if ((l >> 1) < gs && J < nb)
      *reinterpret_cast<float4*>(cf + ((l >> 1) * nb + J) * EX_M + (l & 1) * 4) = make_float4(r[0], r[1], r[2], r[3]);
  }
}

// One warp: Q x 32 rows i0 + 32 q + lane (< i1) of a row block, summed over the column blocks of
// `mask`; cf = the row block's coefficients [nb][8].
template <int Q>
__device__ __forceinline__ void ex_rows(const float* xt, int i0, int i1, float cI, const float* cent, unsigned mask,
                                        const float* cf, float (&di2)[Q], float (&sum)[Q]) {
  using P = Prec<float>;
  const int lane = threadIdx.x & 31;
  float nd2[Q];
  uint64_t p[Q][4], acc[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int i = i0 + 32 * q + lane;
    const float d = i < i1 ? xt[i] - cI : 0.f;
    di2[q] = d * d;
    nd2[q] = -2.f * d;
    ex_powers(d, p[q]);
    acc[q] = 0ull;
  }
  for (unsigned m = mask; m; m &= m - 1) {
    const int J = __ffs(m) - 1;
    const float D = cI - cent[J];
    const float4 c0 = *reinterpret_cast<const float4*>(cf + EX_M * J);
    const float4 c1 = *reinterpret_cast<const float4*>(cf + EX_M * J + 4);
    const uint64_t k0 = f2_pack(c0.x, c0.y), k1 = f2_pack(c0.z, c0.w), k2 = f2_pack(c1.x, c1.y), k3 = f2_pack(c1.z, c1.w);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const float e = P::exp2(D * nd2[q]);
      const uint64_t poly = f2_fma(k3, p[q][3], f2_fma(k2, p[q][2], f2_fma(k1, p[q][1], f2_mul(k0, p[q][0]))));
      acc[q] = f2_fma(poly, f2_pack(e, e), acc[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float a, b;
    f2_unpack(acc[q], a, b);
    sum[q] = a + b;
  }
}

// The apply for row blocks [I0, I1) by the T warps of a CTA: in_s [n] in shared memory (written
// before the call; the first barrier is here), xt [n] (shared or global), scr = shared scratch, 16-byte
// aligned, of ex_scratch_floats(T) floats for gr = T or less for gr = ex_round_groups(T, ...).
// row(i, pre, base, sum, di2) is called once per row by one thread, with
// out_i = base + (log2(sum) - di2), base an integer and sum = 0 for an empty (or non-finite) input;
// pre = load(i) was called before the row's sums, so that what the row's epilogue reads arrives
// meanwhile.
template <int T, class Load, class Row>
__device__ __forceinline__ void ex_apply(const float* in_s, const float* xt, int n, const ExPlan& pl, int I0, int I1,
                                         float* scr, int gr, Load load, Row row) {
  using P = Prec<float>;
  // coefficients of the polynomial for 2^(2 t) = e^(2 ln2 t), |2 ln2 t| <= 0.75: (2 ln2)^m a_m with
  // a_m the degree-7 polynomial of smallest relative error for e^t on [-0.75, 0.75] (Remez exchange)
  constexpr double K = 2.0 * kLn2;
  constexpr double K2 = K * K, K4 = K2 * K2;
  float* cent = scr;
  float* amax = scr + EX_NB;
  float* ref = scr + 2 * EX_NB;
  unsigned* mask_s = reinterpret_cast<unsigned*>(scr + 3 * EX_NB);
  float* cf = scr + EX_HEAD;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = pl.nb, b = pl.b;
  if (tid < nb) cent[tid] = ex_center(xt, tid, b, n, pl.q);
  __syncthreads();
  // block maxima of in_j - dj^2, rounded up
  bool bad = false;
  for (int J = warp; J < nb; J += T) {
    const float c = cent[J];
    const int j1 = min(n, (J + 1) * b);
    float mx = -CUDART_INF_F;
#pragma unroll 4
    for (int j = J * b + lane; j < j1; j += 32) {
      const float d = xt[j] - c, v = in_s[j];
      bad |= !(v < CUDART_INF_F);
      mx = fmaxf(mx, fmaf(-d, d, v));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) amax[J] = ceilf(mx);
  }
  bad = __syncthreads_or(bad);
  // which column blocks matter to each row block (bounds over the block pair)
  const float aJ = lane < nb ? amax[lane] : -CUDART_INF_F, cJl = lane < nb ? cent[lane] : 0.f;
  for (int I = I0 + warp; I < I1; I += T) {
    const float dm = fabsf(cent[I] - cJl), lo = fmaxf(dm - EX_HMAX, 0.f), hi = dm + EX_HMAX;
    // every term of the pair <= top; some term of the pair >= low at every row of the block
    const float top = aJ + (lo >= EX_HMAX ? lo * (2.f * EX_HMAX - lo) : EX_HMAX * EX_HMAX);
    float low = aJ - 1.f - hi * (hi + 2.f * EX_HMAX);
    for (int o = 16; o > 0; o >>= 1) low = fmaxf(low, __shfl_xor_sync(0xffffffffu, low, o));
    const unsigned mk = __ballot_sync(0xffffffffu, !bad && lane < nb && aJ > -CUDART_INF_F && top >= low - EX_SKIP);
    if (lane == 0) mask_s[I] = mk;
  }
  __syncthreads();
  // row blocks go in groups of three or four (equal shares), a round takes up to gr <= T groups
  const int ng = (I1 - I0 + 3) / 4, cpb = (b + 127) / 128, per = ((b + 31) / 32 + cpb - 1) / cpb;
  const bool narrow = b < 256;  // 8 lanes per column block (four at a time) for short blocks
  const int nr = narrow ? (nb + 3) / 4 : nb;
  for (int g0 = 0; g0 < ng; g0 += gr) {
    const int gn = min(gr, ng - g0);
    const int Ia = I0 + (I1 - I0) * g0 / ng, Ib = I0 + (I1 - I0) * (g0 + gn) / ng;
    // moments: items of one group and one (or four) column blocks
    for (int t = warp; t < gn * nr; t += T) {
      const int gi = g0 + t / nr, I = I0 + (I1 - I0) * gi / ng, G = I0 + (I1 - I0) * (gi + 1) / ng - I;
      const int J = narrow ? (t % nr) * 4 + (lane >> 3) : t % nr;
      bool on = false;
      float d2[4];
      const float cJ = J < nb ? cent[J] : 0.f, a = J < nb ? amax[J] : 0.f;
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const bool in = g < G && J < nb;
        on |= in && ((mask_s[in ? I + g : I] >> J) & 1);
        d2[g] = in ? 2.f * (cent[I + g] - cJ) : 0.f;
      }
      if (!__any_sync(0xffffffffu, on)) continue;
      const int j0 = on ? J * b : 0, j1 = on ? min(n, j0 + b) : 0;
      float* c = cf + (I - Ia) * nb * EX_M;
      if (G == 4) {
        if (narrow) ex_moments<4, 8>(in_s, xt, j0, j1, cJ, a, d2, c, nb, J, 4);
        else ex_moments<4, 32>(in_s, xt, j0, j1, cJ, a, d2, c, nb, J, 4);
      } else {  // three (or, for fewer than three row blocks, the first ones of three)
        const float e2[3] = {d2[0], d2[1], d2[2]};
        if (narrow) ex_moments<3, 8>(in_s, xt, j0, j1, cJ, a, e2, c, nb, J, G);
        else ex_moments<3, 32>(in_s, xt, j0, j1, cJ, a, e2, c, nb, J, G);
      }
    }
    __syncthreads();
    // coefficients: moments times c_m and the pair's scale relative to the row block's reference
    for (int I = Ia + warp; I < Ib; I += T) {
      const unsigned mk = mask_s[I];
      float* c = cf + ((I - Ia) * nb + lane) * EX_M;
      const bool on = (mk >> lane) & 1;
      const float D = on ? cent[I] - cent[lane] : 0.f;
      const float dd = __fmul_rn(D, D), de = __fmaf_rn(D, D, -dd), di = rintf(dd);
      const float ai = on ? amax[lane] - di : -CUDART_INF_F, df = __fadd_rn(__fsub_rn(dd, di), de);
      const float m0 = on ? c[0] : 0.f;
      const int k = m0 > 0.f ? ((__float_as_int(m0) >> 23) & 255) - 127 : 0;
      float e = m0 > 0.f ? ai + (float)(k + 1) : -CUDART_INF_F;
      for (int o = 16; o > 0; o >>= 1) e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, o));
      const bool live = e > -CUDART_INF_F;
      if (on) {
        // the moments are first scaled by 2^-k, k the exponent of M_0, so that the remaining scale
        // underflows only where the pair is below 2^-126 of the block's largest at its centre
        const float dn = __int_as_float((127 - k) << 23);
        const float s = live ? P::exp2((ai + (float)k - e) - df) : 0.f;
        float4 u = *reinterpret_cast<float4*>(c), w = *reinterpret_cast<float4*>(c + 4);
        u.x = (u.x * dn) * (s * float(0.9999999849645456)); u.y = (u.y * dn) * (s * float(1.000000111089353 * K));
        u.z = (u.z * dn) * (s * float(0.5000009663519951 * K2)); u.w = (u.w * dn) * (s * float(0.1666651273327656 * K2 * K));
        w.x = (w.x * dn) * (s * float(0.04165746988152903 * K4)); w.y = (w.y * dn) * (s * float(0.008338260296134993 * K4 * K));
        w.z = (w.z * dn) * (s * float(0.0014161683551980183 * K4 * K2)); w.w = (w.w * dn) * (s * float(0.0001953347388479001 * K4 * K2 * K));
        *reinterpret_cast<float4*>(c) = u;
        *reinterpret_cast<float4*>(c + 4) = w;
      }
      if (lane == 0) ref[I] = live ? e : 0.f;
    }
    __syncthreads();
    // rows: items of up to 128 rows of one block
    for (int t = warp; t < (Ib - Ia) * cpb; t += T) {
      const int I = Ia + t / cpb, r0 = I * b + (t % cpb) * per * 32, i1 = min(n, (I + 1) * b);
      const float* c = cf + (I - Ia) * nb * EX_M;
      const unsigned mk = mask_s[I];
      const float base = ref[I];
      const int iend = min(i1, r0 + per * 32);
      auto go = [&](auto qc) {
        constexpr int Q = decltype(qc)::value;
        float di2[Q], sum[Q];
        decltype(load(0)) pre[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) pre[q] = load(min(r0 + 32 * q + lane, iend - 1));
        ex_rows<Q>(xt, r0, iend, cent[I], cent, mk, c, di2, sum);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const int i = r0 + 32 * q + lane;
          if (i < iend) row(i, pre[q], base, sum[q], di2[q]);
        }
      };
      const int groups = (iend - r0 + 31) / 32;
      if (groups >= 4) go(std::integral_constant<int, 4>{});
      else if (groups == 3) go(std::integral_constant<int, 3>{});
      else if (groups == 2) go(std::integral_constant<int, 2>{});
      else if (groups == 1) go(std::integral_constant<int, 1>{});
    }
    __syncthreads();  // the round's coefficients have been read
  }
}

}  // namespace otlm
