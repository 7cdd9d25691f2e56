// FP64 applies with a stored kernel matrix (grid costs, n <= F64_MAX_N).
//
// GB300 runs two FP64 multiply-adds per SM and clock, so a double exp2 (some twenty of them) per
// (problem, row, column) is what an FP64 log-sum-exp apply waits for, and a single problem's few
// tiles leave most SMs idle besides.  K_ij = 2^(-c_ij) is computed once per solve instead and the
// scalings are kept in the linear domain, u = 2^G2, where FP64's range (2^+-1022) holds them:
//   a_i = sum_j K_ij u1_j,   b_j = sum_i K_ij u2_i        (K is symmetric for a grid cost)
// one multiply-add per element, rows spread over all SMs.  The potentials' logarithms stay the
// state.  A sum is taken only where nothing that left the range can matter to it, and redone from the
// potentials around its largest term elsewhere:
//   - within [2^-900, 2^900]: what a scaling below 2^-1022 lost is at most n 2^-1074 in all;
//   - at least 2^-1000 times the problem's largest scaling: an entry K_ij below 2^-1022 is off by at
//     most 2^-1074, which a scaling of 2^1000 (transport beyond sqrt(1022 eps ln2)) makes visible; n times
//     that times the largest scaling is then below 2^-62 of the sum (n <= 4096).
//   one target, n = 200, k = 10, 500 iterations: 765 ms with log-sum-exp tiles of 4 problems x 128
//   rows (2 CTAs on 2 SMs), 14.2 ms now, three launches of 8 to 12 us per iteration whose serial FP64
//   logarithms are what is left; objective of 16 problems, n = 512: 3.2 ms -> 144 us.
#pragma once

#include "kernels.cuh"

namespace otlm {

constexpr int F64_MAX_N = 4096;  // K: 128 MiB

struct F64Buf {
  double* K = nullptr;   // [n][n]
  double *U1 = nullptr, *U2 = nullptr, *IA = nullptr, *LY = nullptr;  // [batch][n] u1, u2, 1 / a, log2 y
  explicit operator bool() const { return K != nullptr; }
};
inline size_t f64_bytes(int n_max, int batch_max) {
  return 8 * ((size_t)n_max * n_max + 4 * (size_t)batch_max * n_max);
}
inline F64Buf f64_carve(void* base, int n_max, int batch_max) {
  F64Buf b;
  if (!base) return b;
  b.K = static_cast<double*>(base);
  b.U1 = b.K + (size_t)n_max * n_max;
  b.U2 = b.U1 + (size_t)batch_max * n_max;
  b.IA = b.U2 + (size_t)batch_max * n_max;
  b.LY = b.IA + (size_t)batch_max * n_max;
  return b;
}

static __global__ void f64_build_kernel(const double* xt, int n, double* K, int abs_cost) {
  const size_t nn = (size_t)n * n;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
    const double d = xt[e / n] - xt[e % n];
    K[e] = ::exp2(abs_cost ? -::fabs(d) : -d * d);
  }
}

// u = 2^G2 of given potentials and, with y, log2 y of the targets (constant over the solve).
static __global__ void f64_scale_kernel(const double* G2, double* U, const double* y, double* LY, size_t count) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    U[e] = ::exp2(G2[e]);
    if (y) LY[e] = ::log2(y[e]);
  }
}

// One warp per row and PB problems: lanes over the columns, K read once for the PB problems; the CTA's
// warps hand their sums to one warp, whose lanes finish a row and problem each (an FP64 instruction
// costs a warp 64 clocks whether one lane or all are active).
//   source: 1 / a into IA, a into A.out, the MM log ratio r = log2(a / S) into R (if given), and the
//           violation's share s |a_new / a_old - 1| = s |a_new IA_old - 1|
//   target: b into A.out, the datafit step G2, and u1 = 2^G2 (u1 given)
//           (target sums are always stored as log2 b, which the datafit step needs)
// A sum outside the linear range is redone by its warp; the source side then stores its logarithm in
// A.out with IA = 0.  lin_out = 0 (objective): A.out takes log2 of the sum and nothing else is written.
struct F64Row {
  double v;    // the sum, or its log2 when `log` is set
  int log;
};
__device__ __forceinline__ double f64_log2a(const F64Buf& F, const double* a, size_t idx) {
  return F.IA[idx] > 0.0 ? ::log2(a[idx]) : a[idx];
}
// log2(a / s) of a linear a with ia = 1 / a and s > 0: one logarithm while s ia is a normal number.  Far
// from every atom s passes through 2^-1022 .. 2^-1074 and s ia is rounded to few bits or to 0.
__device__ __forceinline__ double f64_log_ratio(double a, double ia, double s) {
  const double q = s * ia;
  return q >= 0x1p-1022 && q <= 0x1p1023 ? -::log2(q) : ::log2(a) - ::log2(s);
}

template <int EPI, int PB, int NWARP>
__global__ void __launch_bounds__(32 * NWARP) f64_apply_kernel(ApplyArgs<double> A, F64Buf F, const double* aout, double* R,
                                                              const int* done, int abs_cost, int lin_out) {
  using P = Prec<double>;
  __shared__ F64Row row_s[NWARP][PB];
  __shared__ double part_s[NWARP][PB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * NWARP + warp, n = A.n;
  pdl_wait();
  const int na = *A.n_active, b0 = blockIdx.y * PB;
  if (b0 >= na) return;
  int p[PB];
#pragma unroll
  for (int q = 0; q < PB; ++q) {
    p[q] = b0 + q < na ? A.active[b0 + q] : -1;
    if (p[q] >= 0 && done && done[p[q]]) p[q] = -1;
  }
  const double* U = EPI == EPI_SOURCE ? F.U1 : F.U2;
  double acc[PB];
  int top[PB];  // largest upper half of the scalings (>= 0): their order, and the exponent
#pragma unroll
  for (int q = 0; q < PB; ++q) {
    acc[q] = 0.0;
    top[q] = 0;
  }
#pragma unroll 4
  for (int j = i < n ? lane : n; j < n; j += 32) {
    const double k = F.K[(size_t)i * n + j];
#pragma unroll
    for (int q = 0; q < PB; ++q)
      if (p[q] >= 0) {
        const double u = U[(size_t)p[q] * n + j];
        acc[q] = fma(k, u, acc[q]);
        top[q] = max(top[q], __double2hiint(u));
      }
  }
#pragma unroll
  for (int q = 0; q < PB; ++q) {
    for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    top[q] = __reduce_max_sync(0xffffffffu, top[q]);
    if (p[q] < 0 || i >= n) continue;
    const size_t o = (size_t)p[q] * n;
    F64Row rw{acc[q], 0};
    // the largest scaling is below 2^(exponent + 1); its bound of the sum, at least 2^-900
    const int low = max((top[q] >> 20) - 1023 + 1 - 1000, -900);
    if (!(acc[q] >= __hiloint2double((low + 1023) << 20, 0) && acc[q] <= 0x1p900)) {  // rare: from the potentials
      const double xi = A.xt[i];
      auto term = [&](int j) {
        const double d = xi - A.xt[j];
        double in;
        if (EPI == EPI_SOURCE) in = A.G2[o + j];
        else in = A.S[o + j] > 0.0 ? P::log2(A.S[o + j]) - (lin_out ? f64_log2a(F, aout, o + j) : aout[o + j]) : P::ninf();
        return in - (abs_cost ? ::fabs(d) : d * d);
      };
      double m = P::ninf(), s = 0.0;
      for (int j = lane; j < n; j += 32) m = fmax(m, term(j));
      for (int z = 16; z > 0; z >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, z));
      if (!(m > P::ninf())) m = 0.0;
      for (int j = lane; j < n; j += 32) s += P::exp2(term(j) - m);
      for (int z = 16; z > 0; z >>= 1) s += __shfl_xor_sync(0xffffffffu, s, z);
      rw.v = s > 0.0 ? m + P::log2(s) : P::ninf();
      rw.log = 1;
    }
    if (lane == 0) row_s[warp][q] = rw;
  }
  __syncthreads();
  if (threadIdx.x < NWARP * PB) {
    const int w = threadIdx.x / PB, q = threadIdx.x % PB, r = blockIdx.x * NWARP + w;
    int pq = b0 + q < na ? A.active[b0 + q] : -1;
    if (pq >= 0 && done && done[pq]) pq = -1;
    double part = 0.0;
    if (pq >= 0 && r < n) {
      const size_t idx = (size_t)pq * n + r;
      const F64Row rw = row_s[w][q];
      if (EPI == EPI_SOURCE) {
        const double s = A.S[idx];
        if (!lin_out) {
          A.out[idx] = rw.log ? rw.v : P::log2(rw.v);
        } else {
          const double ia_old = A.check ? F.IA[idx] : 0.0;
          if (A.check && s > 0.0) {
            if (!rw.log && ia_old > 0.0) {
              const double ratio = rw.v * ia_old;  // at most 2^1800: a jump beyond 2^64 is capped
              part = ratio > 0x1p64 ? fmin(s * ratio, 0x1p120) : s * fabs(ratio - 1.0);
            } else {
              const double dl = (rw.log ? rw.v : P::log2(rw.v)) - f64_log2a(F, A.out, idx);
              part = dl > 64.0 ? P::exp2(fmin(P::log2(s) + dl, 120.0)) : s * fabs(P::expm1(dl * kLn2));
            }
          }
          const double ia = rw.log ? 0.0 : 1.0 / rw.v;
          A.out[idx] = rw.v;
          F.IA[idx] = ia;
          R[idx] = s > 0.0 ? (rw.log ? rw.v - P::log2(s) : f64_log_ratio(rw.v, ia, s)) : 0.0;
        }
      } else {
        const double v = rw.log ? rw.v : P::log2(rw.v);
        A.out[idx] = v;
        const double yv = A.y[idx], ly = F.LY[idx];
        double gn;
        switch (A.datafit) {
          case DF_BALANCED: gn = ly - v; break;
          case DF_KL: gn = A.kl_coef * (ly - v); break;
          case DF_TV: gn = fmin(fmax(ly - v, -A.tv_bound), A.tv_bound); break;
          case DF_POISSON: gn = poisson_g2<double>(A.log_lam_over_eps, A.lam_over_eps, A.tv_bound, v, yv); break;
          default: {
            const double z = A.log_lam_over_eps + v * kLn2 + A.lam_over_eps * yv;
            gn = (A.lam_over_eps * yv - wright_omega_f64(z)) * kLog2e;
          }
        }
        A.G2[idx] = gn;
        if (lin_out) F.U1[idx] = P::exp2(gn);
      }
    }
    if (EPI == EPI_SOURCE) part_s[w][q] = part;
  }
  if (EPI == EPI_SOURCE && A.check) {  // the CTA's rows, one addition per problem
    __syncthreads();
    if (threadIdx.x < PB) {
      double t = 0.0;
      for (int w = 0; w < NWARP; ++w) t += part_s[w][threadIdx.x];
      const int pq = b0 + threadIdx.x < na ? A.active[b0 + threadIdx.x] : -1;
      if (pq >= 0 && t != 0.0) atomicAdd(A.err_acc + pq, t);
    }
  }
}

// In a struct of its own: with these members in MMArgs, mm_kernel<float> took 7 % longer (1 problem of 8192
// bins, 21 launches: 4.63 ms, 4.98 with them).
struct MMArgsF64 : MMArgs<double> {
  const double* R;   // the first step's log ratios
  const double* IA;  // 1 / a
  double* U2;        // out: S / a
};

// MM step and source step of a problem (one CTA): the stopping decision and the update's constants
// are formed beside phase A, the update takes two logarithms and one division per weight, and the
// mass and the weight change are reduced by different warps: each FP64 instruction on the critical
// path costs a warp 64 clocks. Same arithmetic as mm_kernel (Table 2), FP64 only.
template <int KQ>
__global__ void __launch_bounds__(256) f64_mm_kernel(MMArgsF64 A) {
  using P = Prec<double>;
  constexpr int KP = KQ * 32;
  __shared__ double red_s[8][KP], w_s[KP], w0_s[KP], c_s[KP], ic_s[KP], ix_s[KP], sum_s[8];
  __shared__ int stop;
  const int slot = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_wait();
  if (slot >= *A.n_active) return;
  const int p = A.active[slot], n = A.n, k = A.k;
  if (A.done[p]) return;
  const size_t o = (size_t)p * n;
  double* S = A.S + o;
  if (tid == 255) {  // convergence decision of the previous iteration
    int st = -1;
    if (A.it > 0) {
      const double e = A.err_acc[p] / A.mass[p];
      A.err[p] = e;
      st = stop_decision<double>(e, A.dw[p], A.tol, A.dw_tol, false, false, A.it, A.max_iter);
      A.err_acc[p] = 0.0;
    }
    stop = st;
  }
  for (int j = tid; j < k; j += 256) {
    const double xj = A.xcol[j], c = (A.penalty == PEN_ELASTIC ? A.beta : A.alpha) / (A.eps * xj);
    w0_s[j] = A.W[(size_t)p * k + j];
    c_s[j] = c;
    ic_s[j] = 1.0 / c;
    ix_s[j] = kLn2 / xj;
  }
  for (int m = 0; m < A.mm_steps; ++m) {
    double acc[KQ];
#pragma unroll
    for (int q = 0; q < KQ; ++q) acc[q] = 0.0;
    for (int base = warp * 32; base < n; base += 256) {
      const int i = base + lane;
      double r = 0.0;
      if (i < n) {
        if (m == 0) {
          r = A.R[o + i];
        } else {
          const double s = S[i], ia = A.IA[o + i];
          r = s > 0.0 ? (ia > 0.0 ? f64_log_ratio(A.LA2[o + i], ia, s) : A.LA2[o + i] - P::log2(s)) : 0.0;
        }
      }
      const int cnt = min(32, n - base);
#pragma unroll 4
      for (int t = 0; t < cnt; ++t) {
        const double rt = __shfl_sync(0xffffffffu, r, t);
        const double* Drow = A.D + (size_t)(base + t) * k;
#pragma unroll
        for (int q = 0; q < KQ; ++q) {
          const int j = lane + 32 * q;
          acc[q] = fma(j < k ? Drow[j] : 0.0, rt, acc[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < KQ; ++q) red_s[warp][lane + 32 * q] = acc[q];
    __syncthreads();
    if (m == 0 && stop >= 0) {
      if (tid == 0) {
        A.status[p] = stop;
        A.iters[p] = A.it;
        A.done[p] = 1;
      }
      return;
    }
    for (int j = tid; j < k; j += 256) {
      double sum = 0.0;
#pragma unroll
      for (int w8 = 0; w8 < 8; ++w8) sum += red_s[w8][j];
      const double wold = m == 0 ? w0_s[j] : w_s[j], dl = sum * ix_s[j];
      // l1 and elastic net: shifted by alpha / (eps x_j) = alpha ix / (eps ln2)
      const double shift = (A.penalty == PEN_L1 || A.penalty == PEN_ELASTIC) ? A.alpha * ix_s[j] / (A.eps * kLn2) : 0.0;
      double wn;
      if (A.penalty == PEN_L2SQ || A.penalty == PEN_ELASTIC) {
        const double om = wright_omega_f64(log_product(c_s[j], wold) + dl - shift);
        wn = ic_s[j] <= 0x1p1023 ? om * ic_s[j] : om / c_s[j];
      } else wn = fabs(dl - shift) < 600.0 ? wold * P::exp(dl - shift) : P::exp(P::log(wold) + dl - shift);
      w_s[j] = wn;
      if (m + 1 == A.mm_steps) A.W[(size_t)p * k + j] = wn;
    }
    __syncthreads();
    const bool last = m + 1 == A.mm_steps;
    double mass = 0.0;
    for (int i = tid; i < n; i += 256) {
      double s = 0.0;
#pragma unroll 4
      for (int j = 0; j < k; ++j) s = fma(A.Dt[(size_t)j * n + i], w_s[j], s);
      S[i] = s;
      mass += s;
      if (last) {  // u2 = s / a; IA = 0 marks a sum held as its logarithm in LA2
        const double ia = A.IA[o + i];
        A.U2[o + i] = s > 0.0 ? (ia > 0.0 ? s * ia : P::exp2(P::log2(s) - A.LA2[o + i])) : 0.0;
      }
    }
    if (last) {
      for (int z = 16; z > 0; z >>= 1) mass += __shfl_xor_sync(0xffffffffu, mass, z);
      if (lane == 0) sum_s[warp] = mass;
    }
    __syncthreads();
  }
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += sum_s[w];
    A.mass[p] = t;
  }
  if (warp == 1) {  // weight change of this iteration's update
    double num = 0.0, den = 0.0;
    for (int j = lane; j < k; j += 32) {
      num += fabs(w_s[j] - w0_s[j]);
      den += fabs(w_s[j]);
    }
    for (int z = 16; z > 0; z >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, z);
      den += __shfl_xor_sync(0xffffffffu, den, z);
    }
    if (lane == 0) A.dw[p] = num / den;
  }
}
static inline cudaError_t launch_f64_mm(const MMArgsF64& a, int batch, cudaStream_t s) {
  if (a.k <= 32) (void)launch_pdl(true, f64_mm_kernel<1>, dim3(batch), dim3(256), 0, s, a);
  else if (a.k <= 64) (void)launch_pdl(true, f64_mm_kernel<2>, dim3(batch), dim3(256), 0, s, a);
  else if (a.k <= 128) (void)launch_pdl(true, f64_mm_kernel<4>, dim3(batch), dim3(256), 0, s, a);
  else (void)launch_pdl(true, f64_mm_kernel<8>, dim3(batch), dim3(256), 0, s, a);
  return cudaGetLastError();
}

// R: the log ratios' buffer of a solve's source applies.  aout: the source sums (for the target side's
// exact path).  Eight warps per CTA once there are several warps per SM; a small problem spreads over
// more SMs with two.
template <int EPI>
static inline cudaError_t launch_f64_apply(const ApplyArgs<double>& a, const F64Buf& F, const double* aout, double* R,
                                           const int* done, int batch, int abs_cost, int lin_out, int sms,
                                           cudaStream_t s) {
  if (batch >= 4) {
    (void)launch_pdl(true, f64_apply_kernel<EPI, 4, 8>, dim3((a.n + 7) / 8, (batch + 3) / 4), dim3(256), 0, s, a, F, aout, R, done, abs_cost, lin_out);
  } else if ((long long)a.n * batch > 8LL * sms) {
    (void)launch_pdl(true, f64_apply_kernel<EPI, 1, 8>, dim3((a.n + 7) / 8, batch), dim3(256), 0, s, a, F, aout, R, done, abs_cost, lin_out);
  } else {
    (void)launch_pdl(true, f64_apply_kernel<EPI, 1, 2>, dim3((a.n + 1) / 2, batch), dim3(64), 0, s, a, F, aout, R, done, abs_cost, lin_out);
  }
  return cudaGetLastError();
}

}  // namespace otlm
