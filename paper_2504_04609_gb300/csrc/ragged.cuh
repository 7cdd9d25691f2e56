// Uneven batch in one persistent launch: every problem has its own grid x [n_p], dictionary
// D [n_p][k_p], eps_p and target y [n_p] (concatenated, with offsets).  One CTA solves one problem
// at a time, all of its iterations (Algorithm 1), with the problem's state in shared memory:
//   xt (scaled grid), G2, LA2, F2, LB2, S  (6 n_p floats) and W, xcol, reduction scratch.
// CTAs take problems from a device-side queue (an atomic counter over an order sorted by
// decreasing n_p^2, i.e. largest work first), so the 256x spread in work per problem balances
// across the SMs without any host round trip.
//
// The kernel apply inside a CTA: block expansions (expansion.cuh) wherever the problem's grid
// qualifies, which is decided per problem in the kernel from the grid itself.  Other grids (unsorted,
// or with fewer than 32 bins per 1.47 kernel widths) are summed term by term: thread t owns R consecutive rows (R even, a compile-time
// constant picked from n_p); with its own centre c_t (the middle of its rows) the exponent
// in_j - m_i - (xt_i - xt_j)^2 becomes FFMA(2 di, dj, h_j) - q_i with h_j = in_j - dj^2 formed
// once per column and q_i = m_i + di^2 once per row; rows are processed in packed pairs
// (fma/add.f32x2).  Shift: the previous sums (later iterations), the diagonal term (first
// iteration), or an exact max pass when any sum leaves [2^-60, 2^60].
//
// 800 problems, n 256..4096, k 8..128, eps 2e-3..5e-2, 20 iterations: 45.4 ms with every apply term by
// term and row-at-a-time dictionary passes (exponent unit and load latency), 6.8 ms with expansions
// and passes that keep 16 loads of D in flight per warp.  What is left is D: 0.6 MB per problem, read
// twice per iteration, mostly from DRAM.
#pragma once

#include "expansion.cuh"

namespace otlm {

struct RaggedArgs {
  int batch;
  const int* order;   // problem ids, largest work first
  int* next;          // queue position (zeroed before the launch)
  const int* n;
  const int* k;
  const float* eps;
  const long long* off_n;  // start of problem p in x, y, g, t
  const long long* off_D;  // start of problem p in D
  const long long* off_k;  // start of problem p in w
  const float* x;
  const float* D;
  const float* y;
  float* w;                // in: initial weights (> 0), out: result
  const float* g_in;       // initial target potentials (eps log u1) or null
  float* g_out;            // final potentials or null
  float* t_out;            // transported target marginal or null
  int* iters;
  float* err;
  int* status;
  int datafit, penalty, max_iter;
  float lam, alpha, tol;
  float beta;                     // squared-l2 weight of the elastic net
  int mm_steps;                   // MM steps per iteration (>= 1)
  int n_max, k_max;
  long long tot_n, tot_D, tot_k;  // packed sizes of x/y, D and w (sum n, sum n k, sum k)
  int smem_floats;                // dynamic shared memory of the launch, in floats
  // a small batch sharing one grid, dictionary and eps (n == null; one CTA per problem, no queue)
  int n_all, k_all;
  float eps_all, xs_all;          // xs_all = 1 / sqrt(eps ln2)
  float* dw;                      // [batch] weight change of the last update, or null
  int empty_t0;                   // t = 0 where the target sum is empty, whatever g is there
  // rows per thread by size bucket (n in (256 b, 256 (b + 1)]), as log2 R; raised to the fewest
  // that cover n with this CTA size (0: always the fewest)
  unsigned char rows_log2[16];
};

constexpr int RAGGED_BUCKETS = 16;
__host__ __device__ inline int ragged_bucket(int n) { return n <= 256 ? 0 : (n - 1) / 256 < 15 ? (n - 1) / 256 : 15; }

// Dynamic shared memory (floats) of a problem of n_max bins, k_max atoms: its state, then a part that the
// warps' sums of D^T r and the expansion's scratch take in turn. `full` is the scratch of one round; the
// least one serves in rounds of two groups and more (up to 16 blocks still one round of 8 warps), so that
// what the scratch adds does not cost a CTA its place on the SM (ragged_prepare).
template <int NT>
struct RaggedSmem {
  static constexpr int LEAST = EX_HEAD + EX_M * EX_NB * 8;
  static __host__ __device__ size_t state(int n_max, int k_max) { return (6 * (size_t)n_max + 3 * (size_t)k_max + 64 + 3) / 4 * 4; }
  static __host__ __device__ size_t floats(int n_max, int k_max, bool full) {
    const size_t sums = (NT / 32) * (size_t)k_max, scr = full ? ex_scratch_floats(NT / 32) : LEAST;
    return state(n_max, k_max) + (sums > scr ? sums : scr);
  }
};

// Sum pass of the in-CTA apply: acc2 = sum_j 2^(FFMA(2 di, dj, h_j) + nq) on packed row pairs.
template <int R>
__device__ __forceinline__ void ragged_sum(const float* xt, const float* in, int n, int i0, float xc,
                                           const uint64_t (&nq2)[R / 2], uint64_t (&acc2)[R / 2]) {
  using P = Prec<float>;
  constexpr int QP = R / 2;
  uint64_t tdi2[QP];
#pragma unroll
  for (int q = 0; q < QP; ++q) {
    const int a = min(i0 + 2 * q, n - 1), b = min(i0 + 2 * q + 1, n - 1);
    tdi2[q] = f2_pack(2.f * (xt[a] - xc), 2.f * (xt[b] - xc));
    acc2[q] = f2_pack(0.f, 0.f);
  }
#pragma unroll 2
  for (int j = 0; j < n; ++j) {
    const float dj = xt[j] - xc;
    const float h = fmaf(-dj, dj, in[j]);
    const uint64_t dj2 = f2_pack(dj, dj), h2 = f2_pack(h, h);
#pragma unroll
    for (int q = 0; q < QP; ++q) {
      const uint64_t u2 = f2_add(f2_fma(tdi2[q], dj2, h2), nq2[q]);
      float u0, u1;
      f2_unpack(u2, u0, u1);
      acc2[q] = f2_add(acc2[q], f2_pack(P::exp2(u0), P::exp2(u1)));
    }
  }
}

// One kernel apply inside the CTA: out_i = log2 sum_j 2^(in_j - (xt_i - xt_j)^2) for i < n.
// shift_prev: out holds the previous sums (shift = out_i); otherwise the diagonal in_i.
// ratio (optional): ratio_i = a_new_i / a_old_i (exact when the previous-sum shift held).
// Rows past n are computed on clamped rows and never stored.  Live through the column loop:
// three packed registers per row pair (shift, offset, accumulator).
template <int NT, int R>
__device__ void ragged_apply(const float* xt, const float* in, float* out, int n, bool shift_prev, float* ratio) {
  using P = Prec<float>;
  constexpr int QP = R / 2;
  const int i0 = threadIdx.x * R;
  const bool active = i0 < n;
  const float xc = active ? 0.5f * (xt[i0] + xt[min(i0 + R - 1, n - 1)]) : 0.f;
  const float* src = shift_prev ? out : in;
  bool bad = false;
  uint64_t nq2[QP], acc2[QP];
#pragma unroll
  for (int q = 0; q < QP; ++q) {
    float v[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = min(i0 + 2 * q + c, n - 1);
      const float m = active ? src[i] : 0.f;
      const float d = active ? xt[i] - xc : 0.f;
      bad |= active && !isfinite(m);
      v[c] = -(m + d * d);
    }
    nq2[q] = f2_pack(v[0], v[1]);
  }
  bool exact = __syncthreads_or(bad);
  if (!exact) {
    if (active) ragged_sum<R>(xt, in, n, i0, xc, nq2, acc2);
    bool b2 = false;
#pragma unroll
    for (int q = 0; q < QP; ++q) {
      float a0, a1;
      f2_unpack(acc2[q], a0, a1);
      b2 |= active && !(a0 >= 8.673617379884035e-19f && a0 <= 1.152921504606847e18f);
      b2 |= active && !(a1 >= 8.673617379884035e-19f && a1 <= 1.152921504606847e18f);
    }
    exact = __syncthreads_or(b2);
  }
  if (exact) {
    // exact shift: m_i = max_j (in_j - (xt_i - xt_j)^2), then the sum again
    float m[R];
#pragma unroll
    for (int r = 0; r < R; ++r) m[r] = -CUDART_INF_F;
    if (active)
      for (int j = 0; j < n; ++j) {
        const float dj = xt[j] - xc;
        const float h = fmaf(-dj, dj, in[j]);
#pragma unroll
        for (int r = 0; r < R; ++r) m[r] = fmaxf(m[r], fmaf(2.f * (xt[min(i0 + r, n - 1)] - xc), dj, h));
      }
#pragma unroll
    for (int q = 0; q < QP; ++q) {
      float v[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int r = 2 * q + c;
        const float d = active ? xt[min(i0 + r, n - 1)] - xc : 0.f;
        float mm = m[r] - d * d;
        if (!(mm > -CUDART_INF_F)) mm = 0.f;  // every term vanishes
        v[c] = -(mm + d * d);
      }
      nq2[q] = f2_pack(v[0], v[1]);
    }
    if (active) ragged_sum<R>(xt, in, n, i0, xc, nq2, acc2);
  }
  __syncthreads();  // every thread has read `out` and `in` before `out` is overwritten
  const bool prev_ratio = shift_prev && !exact;
#pragma unroll
  for (int q = 0; q < QP; ++q) {
    float nq[2], acc[2];
    f2_unpack(nq2[q], nq[0], nq[1]);
    f2_unpack(acc2[q], acc[0], acc[1]);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = i0 + 2 * q + c;
      if (!active || i >= n) continue;
      const float d = xt[i] - xc;
      const float v = acc[c] > 0.f ? (-nq[c] - d * d) + P::log2(acc[c]) : P::ninf();
      if (ratio) ratio[i] = prev_ratio ? acc[c] : (shift_prev ? P::exp2(v - out[i]) : 1.f);
      out[i] = v;
    }
  }
  __syncthreads();
}

__device__ __forceinline__ float block_sum_f(float v, float* red) { return block_sum<float>(v, red); }

// The same apply by block expansions (expansion.cuh), for grids that qualify.  Out of line: one copy
// serves the source and target applies of every rows-per-thread variant.
template <int NT>
__device__ __noinline__ void ragged_apply_ex(const float* xt, const float* in, float* out, int n, ExPlan pl, float* scr,
                                             int gr, float* ratio) {
  using P = Prec<float>;
  ex_apply<NT / 32>(in, xt, n, pl, 0, pl.nb, scr, gr, [](int) { return 0; }, [&](int i, int, float base, float sum, float di2) {
    if (ratio) ratio[i] = sum > 0.f ? sum * P::exp2((base - out[i]) - di2) : 0.f;
    out[i] = sum > 0.f ? base + (P::log2(sum) - di2) : P::ninf();
  });
  __syncthreads();
}

// The two dictionary passes of an iteration.  D [n][k] is read from L2 or HBM twice per iteration
// and is what an iteration waits for, so a warp keeps U rows x KQ loads of 32 columns in flight
// (U KQ = 16); lanes are columns, warps take rows.
//   ragged_dtr: red_k[warp][j] = sum over the warp's rows of D_ij r_i
//   ragged_dw : row_done(i, sum_j D_ij w_j), once per row by one lane; U rows are summed over the
//               lanes by one transposing butterfly
template <int NT, int KQ>
__device__ __forceinline__ void ragged_dtr(const float* D, const float* r, int n, int k, int k_max, float* red_k) {
  constexpr int NW = NT / 32, U = KQ >= 8 ? 2 : (KQ >= 4 ? 4 : 8);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float acc[KQ];
#pragma unroll
  for (int q = 0; q < KQ; ++q) acc[q] = 0.f;
  for (int i0 = warp * U; i0 < n; i0 += NW * U) {
    float d[U][KQ];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int q = 0; q < KQ; ++q) {
        const int j = lane + 32 * q;
        d[u][q] = (i0 + u < n && j < k) ? D[(size_t)(i0 + u) * k + j] : 0.f;
      }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float ri = i0 + u < n ? r[i0 + u] : 0.f;
#pragma unroll
      for (int q = 0; q < KQ; ++q) acc[q] = fmaf(d[u][q], ri, acc[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < KQ; ++q)
    if (lane + 32 * q < k) red_k[warp * k_max + lane + 32 * q] = acc[q];
}
template <int NT, int KQ, class F>
__device__ __forceinline__ void ragged_dw(const float* D, const float* W, int n, int k, F row_done) {
  constexpr int NW = NT / 32, U = KQ >= 8 ? 2 : (KQ >= 4 ? 4 : 8);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float w[KQ];
#pragma unroll
  for (int q = 0; q < KQ; ++q) w[q] = lane + 32 * q < k ? W[lane + 32 * q] : 0.f;
  for (int i0 = warp * U; i0 < n; i0 += NW * U) {
    float s[U];
    {
      float d[U][KQ];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int q = 0; q < KQ; ++q) {
          const int j = lane + 32 * q;
          d[u][q] = (i0 + u < n && j < k) ? D[(size_t)(i0 + u) * k + j] : 0.f;
        }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        s[u] = 0.f;
#pragma unroll
        for (int q = 0; q < KQ; ++q) s[u] = fmaf(d[u][q], w[q], s[u]);
      }
    }
    // transpose while the values outnumber one: lanes with bit o set keep the upper half
#pragma unroll
    for (int o = 16, c = U; o > 0; o >>= 1) {
      if (c > 1) {
        c >>= 1;
#pragma unroll
        for (int u = 0; u < c; ++u) {
          const bool up = lane & o;
          const float keep = up ? s[u + c] : s[u], give = up ? s[u] : s[u + c];
          s[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      } else {
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
      }
    }
    // lane l holds the total of row i0 + (the top log2 U bits of l)
    const int i = i0 + lane / (32 / U);
    if (lane % (32 / U) == 0 && i < n) row_done(i, s[0]);
  }
}

// D^T r by columns per lane, and S = D w with F2 = log2 S - LA2 (F2 not null) and the thread's share
// of the mass.  Out of line: shared by every rows-per-thread variant.
template <int NT>
__device__ __noinline__ void ragged_dtr_any(const float* D, const float* r, int n, int k, int k_max, float* red_k) {
  if (k <= 32) ragged_dtr<NT, 1>(D, r, n, k, k_max, red_k);
  else if (k <= 64) ragged_dtr<NT, 2>(D, r, n, k, k_max, red_k);
  else if (k <= 128) ragged_dtr<NT, 4>(D, r, n, k, k_max, red_k);
  else ragged_dtr<NT, 8>(D, r, n, k, k_max, red_k);
}
template <int NT>
__device__ __noinline__ float ragged_dw_any(const float* D, const float* W, const float* LA2, float* S, float* F2, int n,
                                            int k) {
  using P = Prec<float>;
  float mass = 0.f;
  auto row_done = [&](int i, float s) {
    if (s < P::tiny()) s = 0.f;
    S[i] = s;
    if (F2) F2[i] = s > 0.f ? P::log2(s) - LA2[i] : P::ninf();
    mass += s;
  };
  if (k <= 32) ragged_dw<NT, 1>(D, W, n, k, row_done);
  else if (k <= 64) ragged_dw<NT, 2>(D, W, n, k, row_done);
  else if (k <= 128) ragged_dw<NT, 4>(D, W, n, k, row_done);
  else ragged_dw<NT, 8>(D, W, n, k, row_done);
  return mass;
}

template <int NT, int R>
__device__ void ragged_solve_one(const RaggedArgs& A, int p, float* sm) {
  using P = Prec<float>;
  const bool shared = A.n == nullptr;
  const int n = shared ? A.n_all : A.n[p], k = shared ? A.k_all : A.k[p];
  const float eps = shared ? A.eps_all : A.eps[p];
  const float eps_ln2 = eps * float(kLn2);
  const long long on = shared ? (long long)p * n : A.off_n[p], oD = shared ? 0 : A.off_D[p],
                  ok = shared ? (long long)p * k : A.off_k[p];
  const float* x = A.x + (shared ? 0 : on);
  // a problem whose sizes or offsets fall outside the packed arrays is marked invalid and not
  // touched; the barrier also separates the previous problem's last reads from this one's writes
  const bool valid = n >= 2 && n <= A.n_max && k >= 1 && k <= A.k_max && (n + NT - 1) / NT <= R && on >= 0 &&
                     on + n <= A.tot_n && oD >= 0 && oD + (long long)n * k <= A.tot_D && ok >= 0 &&
                     ok + k <= A.tot_k &&
                     (long long)RaggedSmem<NT>::floats(A.n_max, A.k_max, false) <= A.smem_floats;
  if (!__syncthreads_and(valid)) {
    if (threadIdx.x == 0) {
      A.iters[p] = 0;
      A.err[p] = CUDART_NAN_F;
      A.status[p] = ST_INVALID;
    }
    return;
  }
  const float* D = A.D + oD;
  float* xt = sm;
  float* G2 = xt + A.n_max;
  float* LA2 = G2 + A.n_max;
  float* F2 = LA2 + A.n_max;
  float* LB2 = F2 + A.n_max;
  float* S = LB2 + A.n_max;
  float* W = S + A.n_max;
  float* xcol = W + A.k_max;
  float* Wp = xcol + A.k_max;     // weights before the last update
  float* red = Wp + A.k_max;      // 32 floats + scalars
  float* scr = sm + RaggedSmem<NT>::state(A.n_max, A.k_max);  // the expansion's scratch
  float* red_k = scr;             // [NT/32][k_max], between the applies
  __shared__ ExPlan plan_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = NT / 32;

  const float xs = shared ? A.xs_all : rsqrtf(eps_ln2);
  for (int i = tid; i < n; i += NT) {
    xt[i] = x[i] * xs;
    G2[i] = A.g_in ? A.g_in[on + i] / eps_ln2 : 0.f;
  }
  for (int j = tid; j < k; j += NT) W[j] = A.w[ok + j];
  __syncthreads();
  const bool sorted = ex_sorted(xt, n);
  if (warp == 0) {
    const ExPlan pl = ex_plan_warp(xt, n, sorted);
    if (lane == 0) plan_s = pl;
  }
  // column sums x_j (F2 holds ones until the first iteration)
  for (int i = tid; i < n; i += NT) F2[i] = 1.f;
  __syncthreads();
  const ExPlan plan = plan_s;
  const int gr = plan.nb ? ex_round_groups(NW, plan.nb, A.smem_floats - (int)(scr - sm)) : 1;
  ragged_dtr_any<NT>(D, F2, n, k, A.k_max, red_k);
  __syncthreads();
  for (int j = tid; j < k; j += NT) {
    float s = 0.f;
    for (int w8 = 0; w8 < NW; ++w8) s += red_k[w8 * A.k_max + j];
    xcol[j] = s;
  }
  __syncthreads();

  // S = D w, F2 = log2 S - LA2 (when asked for) and the mass
  auto source_step = [&](bool write_f2) -> float {
    const float mass = ragged_dw_any<NT>(D, W, LA2, S, write_f2 ? F2 : nullptr, n, k);
    __syncthreads();
    return block_sum_f(mass, red);
  };
  float mass = source_step(false);

  int it = 0;
  float e = 0.f;
  int st = ST_MAX_ITER;
  for (;; ++it) {
    // source apply; F2 doubles as the ratio buffer a_new / a_old
    if (plan.nb) ragged_apply_ex<NT>(xt, G2, LA2, n, plan, scr, gr, it > 0 ? F2 : nullptr);
    else ragged_apply<NT, R>(xt, G2, LA2, n, it > 0, F2);
    if (it > 0) {
      float part = 0.f;
      for (int i = tid; i < n; i += NT)
        if (S[i] > 0.f) part += S[i] * fabsf(F2[i] - 1.f);
      part = block_sum_f(part, red);
      e = part / mass;
      if (e != e) { st = ST_NONFINITE; break; }
      if (A.tol > 0.f && e <= A.tol) { st = ST_CONVERGED; break; }
    }
    if (it >= A.max_iter) { st = ST_MAX_ITER; break; }
    // MM step: nu_j = log w_j + (ln2 / x_j) sum_i D_ij (LA2_i - log2 S_i), then S = D w; mm_steps
    // times with the same LA2, the last one also writing F2
    for (int m = 0; m < A.mm_steps; ++m) {
      for (int i = tid; i < n; i += NT) F2[i] = S[i] > 0.f ? LA2[i] - P::log2(S[i]) : 0.f;  // the log ratios
      __syncthreads();
      ragged_dtr_any<NT>(D, F2, n, k, A.k_max, red_k);
      __syncthreads();
      for (int j = tid; j < k; j += NT) {
        float sum = 0.f;
        for (int w8 = 0; w8 < NW; ++w8) sum += red_k[w8 * A.k_max + j];
        const float xj = xcol[j];
        const float dl = sum * float(kLn2) / xj;
        if (m == 0) Wp[j] = W[j];
        const float nu = P::log(W[j]) + dl;
        const float shift = (A.penalty == PEN_L1 || A.penalty == PEN_ELASTIC) ? A.alpha / (eps * xj) : 0.f;
        float wn;
        if (A.penalty == PEN_L2SQ || A.penalty == PEN_ELASTIC) {
          const float c = (A.penalty == PEN_ELASTIC ? A.beta : A.alpha) / (eps * xj);
          wn = wright_omega<float>(P::log(c) + nu - shift) / c;
        } else {
          // w e^(dl - shift): no rounding of log w, whose size is that of the weights' whole range
          wn = fabsf(dl - shift) < 60.f ? W[j] * P::exp(dl - shift) : P::exp(nu - shift);
        }
        W[j] = wn;
      }
      __syncthreads();
      const float m_mass = source_step(m + 1 == A.mm_steps);
      if (m + 1 == A.mm_steps) mass = m_mass;
    }
    // target apply and the datafit step (Table 1) in log2 units
    if (plan.nb) ragged_apply_ex<NT>(xt, F2, LB2, n, plan, scr, gr, nullptr);
    else ragged_apply<NT, R>(xt, F2, LB2, n, it > 0, nullptr);
    const float kl_coef = A.lam / (eps + A.lam), tv_bound = A.lam / eps_ln2, loe = A.lam / eps;
    const float lloe = logf(A.lam / eps);
    for (int j = tid; j < n; j += NT) {
      const float v = LB2[j], yv = A.y[on + j];
      float gn;
      switch (A.datafit) {
        case DF_BALANCED: gn = P::log2(yv) - v; break;
        case DF_KL: gn = kl_coef * (P::log2(yv) - v); break;
        case DF_TV: gn = fminf(fmaxf(P::log2(yv) - v, -tv_bound), tv_bound); break;
        default: {  // L2 or Poisson (reading A7; -lam where y = 0), one Wright omega
          const bool pois = A.datafit == DF_POISSON;
          if (pois && !(yv > 0.f)) {
            gn = -tv_bound;
            break;
          }
          const float l2c = pois ? lloe * float(kLog2e) + P::log2(yv) : 0.f;
          const float z = pois ? (l2c - v) * float(kLn2) + loe : lloe + v * float(kLn2) + loe * yv;
          const float om = wright_omega<float>(z);
          gn = pois ? l2c - P::log2(om) - v : (loe * yv - om) * float(kLog2e);
        }
      }
      G2[j] = gn;
    }
    __syncthreads();
  }
  // outputs
  for (int j = tid; j < k; j += NT) A.w[ok + j] = W[j];
  for (int i = tid; i < n; i += NT) {
    if (A.g_out) A.g_out[on + i] = G2[i] * eps_ln2;
    if (A.t_out) A.t_out[on + i] = it > 0 && !(A.empty_t0 && !(LB2[i] > P::ninf())) ? P::exp2(G2[i] + LB2[i]) : 0.f;
  }
  if (A.dw) {  // ||w - w_before||_1 / ||w||_1 of the last update
    float num = 0.f, den = 0.f;
    for (int j = tid; j < k; j += NT) {
      num += fabsf(W[j] - Wp[j]);
      den += fabsf(W[j]);
    }
    num = block_sum_f(num, red);
    den = block_sum_f(den, red);
    if (tid == 0) A.dw[p] = it > 0 ? num / den : CUDART_NAN_F;
  }
  if (tid == 0) {
    if (A.iters) A.iters[p] = it;
    if (A.err) A.err[p] = e;
    if (A.status) A.status[p] = st;
  }
  __syncthreads();
}

// Persistent kernel: CTAs take problems from the queue until it is empty.  RMAX = rows per
// thread for the largest n the handle supports (n_max <= NT * RMAX).
template <int NT, int RMAX>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1) ragged_kernel(RaggedArgs A) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_idx;
  const bool shared = A.n == nullptr;  // one CTA per problem, no queue
  for (bool first = true;; first = false) {
    int p = blockIdx.x;
    if (shared) {
      if (!first) break;
    } else {
      if (threadIdx.x == 0) s_idx = atomicAdd(A.next, 1);
      __syncthreads();
      const int idx = s_idx;
      __syncthreads();
      if (idx >= A.batch) break;
      p = A.order[idx];
    }
    const int n = shared ? A.n_all : A.n[p];
    // rows per thread: the tuned choice for n's size bucket, at least the fewest that cover n
    // (more rows per thread amortise each column's shared-memory reads over more exponentials,
    // fewer keep more threads busy)
    const int need = (n + NT - 1) / NT;
    int rows = 1 << (A.rows_log2[ragged_bucket(n)] > 0 ? A.rows_log2[ragged_bucket(n)] : 1);
    while (rows < need) rows <<= 1;
    if (rows <= 2) ragged_solve_one<NT, 2>(A, p, sm);
    else if (RMAX >= 4 && rows <= 4) ragged_solve_one<NT, (RMAX >= 4 ? 4 : 2)>(A, p, sm);
    else if (RMAX >= 8 && rows <= 8) ragged_solve_one<NT, (RMAX >= 8 ? 8 : 2)>(A, p, sm);
    else if (RMAX >= 16 && rows <= 16) ragged_solve_one<NT, (RMAX >= 16 ? 16 : 2)>(A, p, sm);
    else if (RMAX >= 32 && rows <= 32) ragged_solve_one<NT, (RMAX >= 32 ? 32 : 2)>(A, p, sm);
    else if (threadIdx.x == 0 && !shared) {  // more rows per thread than this CTA size supports
      A.iters[p] = 0;
      A.err[p] = CUDART_NAN_F;
      A.status[p] = ST_INVALID;
    }
  }
}

}  // namespace otlm

namespace otlm {

// Variants the tuner chooses among: CTA size NT with rows per thread up to RMAX (n <= 4096).
constexpr int RAGGED_VARIANTS = 3;
inline int ragged_nt(int v) { return v == 0 ? 128 : (v == 1 ? 256 : 512); }
inline int ragged_rmax_log2(int v) { return v == 0 ? 5 : (v == 1 ? 4 : 3); }

// Dynamic shared memory of variant v for n <= n_max, k <= k_max; *fn: its kernel. The kernel's limit is one
// value for the process and is set to the largest size there is (RAGGED_N_MAX bins, 256 atoms): a limit
// that followed the call would be lowered by one host thread between another's setting and launch.
constexpr int RAGGED_N_MAX = 4096, RAGGED_K_MAX = 256;
template <int NT, int RMAX>
inline cudaError_t ragged_allow(int n_max, int k_max, bool full, size_t* smem, const void** fn) {
  static_assert(RAGGED_N_MAX <= NT * RMAX, "rows per thread cover the largest problem");
  *smem = RaggedSmem<NT>::floats(n_max, k_max, full) * 4;
  *fn = (const void*)ragged_kernel<NT, RMAX>;
  return cudaFuncSetAttribute(*fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(RaggedSmem<NT>::floats(RAGGED_N_MAX, RAGGED_K_MAX, true) * 4));
}
inline cudaError_t ragged_allow(int v, int n_max, int k_max, bool full, size_t* smem, const void** fn) {
  if (n_max > RAGGED_N_MAX || k_max > RAGGED_K_MAX) return cudaErrorInvalidValue;
  if (v == 0) return ragged_allow<128, 32>(n_max, k_max, full, smem, fn);
  if (v == 1) return ragged_allow<256, 16>(n_max, k_max, full, smem, fn);
  return ragged_allow<512, 8>(n_max, k_max, full, smem, fn);
}
// The full scratch unless the least one lets more CTAs share an SM.  456 unsorted problems of 3300 to 4096
// bins, k = 128, 6 iterations, 256 threads: one CTA per SM 24.0 ms, two 19.4; sorted ones 4.32 and 3.28.
inline cudaError_t ragged_prepare(int v, int n_max, int k_max, int* blocks_per_sm, size_t* smem) {
  *blocks_per_sm = 0;
  for (const bool full : {true, false}) {
    size_t bytes = 0;
    const void* fn = nullptr;
    int blocks = 0;
    cudaError_t e = ragged_allow(v, n_max, k_max, full, &bytes, &fn);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, ragged_nt(v), bytes);
    if (e != cudaSuccess) return e;
    if (blocks > *blocks_per_sm) {
      *blocks_per_sm = blocks;
      *smem = bytes;
    }
  }
  return cudaSuccess;
}

// A small batch sharing grid, dictionary and eps, whole solves in one launch (one CTA per problem).
// The smallest calls are latency: an iteration of three launches is 20 to 30 us whatever its size,
// while a CTA that keeps its problem in shared memory pays barriers only.
inline cudaError_t ragged_small(const RaggedArgs& a0, cudaStream_t s) {
  RaggedArgs a = a0;
  const int v = a.n_all <= 512 ? 1 : 2;
  size_t smem = 0;
  const void* fn = nullptr;
  const cudaError_t e = ragged_allow(v, a.n_all, a.k_all, true, &smem, &fn);
  if (e != cudaSuccess) return e;
  a.n_max = a.n_all; a.k_max = a.k_all;
  a.tot_n = (long long)a.batch * a.n_all; a.tot_D = (long long)a.n_all * a.k_all; a.tot_k = (long long)a.batch * a.k_all;
  a.smem_floats = (int)(smem / 4);
  if (v == 1) ragged_kernel<256, 16><<<a.batch, 256, smem, s>>>(a);
  else ragged_kernel<512, 8><<<a.batch, 512, smem, s>>>(a);
  return cudaGetLastError();
}

inline void ragged_launch(int v, dim3 grid, size_t smem, cudaStream_t s, const RaggedArgs& a) {
  if (v == 0) ragged_kernel<128, 32><<<grid, 128, smem, s>>>(a);
  else if (v == 1) ragged_kernel<256, 16><<<grid, 256, smem, s>>>(a);
  else ragged_kernel<512, 8><<<grid, 512, smem, s>>>(a);
}

}  // namespace otlm
