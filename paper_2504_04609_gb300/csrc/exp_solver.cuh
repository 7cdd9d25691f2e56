// Batched kernel applies by block expansions (expansion.cuh) for a batch sharing one squared-distance
// grid, with the iteration's row work fused in: one CTA reads a problem's row once, applies K and
// finishes the rows it computed.
//
//   source apply (EXA_SOURCE): in = G2;  out = LA2, the source-marginal violation and the stopping
//     decision of the previous iteration (stop_decision), and on tensor-core handles the MM log
//     ratios r = LA2 - log2 S as the TF32 hi/lo operand of D^T r
//   target apply (EXA_TARGET): in = F2 = log2 S - LA2 (formed on the fly);  out = LB2, the datafit
//     step G2 (Table 1) and, on tensor-core handles, the mass sum S
//
// The row is staged in shared memory (n <= EXA_MAX_N).  Small batches split a problem's row blocks
// over `parts` CTAs (grid.y), each forming the moments of its own row blocks from the whole row; the
// last CTA of a problem to finish adds the violation's partial sums in a fixed order and decides.
// A grid without a plan (ExPlan.nb = 0) never gets here: the host chooses other kernels, or the device
// counts no active problem for these.
#pragma once

#include "expansion.cuh"

namespace otlm {


inline size_t exa_smem_bytes(int n, int warps) {
  return 4 * ((size_t)(n + 3) / 4 * 4 + ex_scratch_floats(warps));
}

static __global__ void __launch_bounds__(1024) ex_plan_kernel(const float* xt, int n, ExPlan* plan, int batch,
                                                              int* with_plan, int* without) {
  const bool sorted = ex_sorted(xt, n);
  if (threadIdx.x < 32) {
    const ExPlan pl = ex_plan_warp(xt, n, sorted);
    if (threadIdx.x == 0) {
      *plan = pl;
      if (with_plan) *with_plan = pl.nb > 0 ? batch : 0;
      if (without) *without = pl.nb > 0 ? 0 : batch;
    }
  }
}

// Datafit step (Table 1) in log2 units; FAST: the Wright omega of the tensor-core path.
template <bool FAST>
__device__ __forceinline__ float exa_datafit(const ExArgs& A, float v, float yv) {
  using P = Prec<float>;
  switch (A.datafit) {
    case DF_BALANCED: return P::log2(yv) - v;
    case DF_KL: return A.kl_coef * (P::log2(yv) - v);
    case DF_TV: return fminf(fmaxf(P::log2(yv) - v, -A.tv_bound), A.tv_bound);
    default: {
      const bool pois = A.datafit == DF_POISSON;
      if (pois && !(yv > 0.f)) return -A.tv_bound;
      const float l2c = pois ? A.log_lam_over_eps * float(kLog2e) + P::log2(yv) : 0.f;
      const float z = pois ? (l2c - v) * float(kLn2) + A.lam_over_eps
                           : A.log_lam_over_eps + v * float(kLn2) + A.lam_over_eps * yv;
      const float om = FAST ? wright_omega_fast(z) : wright_omega<float>(z);
      return pois ? l2c - P::log2(om) - v : (A.lam_over_eps * yv - om) * float(kLog2e);
    }
  }
}

__device__ __forceinline__ float exa_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

template <int EPI, bool TC, int T>
__global__ void __launch_bounds__(32 * T, T == 4 ? 7 : 1) ex_apply_kernel(ExArgs A) {
  using P = Prec<float>;
  constexpr int NT = 32 * T;
  extern __shared__ __align__(16) float smem[];
  __shared__ float red[32];
  __shared__ int last_s;
  const int slot = blockIdx.x, prt = blockIdx.y, parts = gridDim.y;
  pdl_wait();
  if (slot >= *A.n_active) return;
  const int p = A.active[slot], n = A.n, tid = threadIdx.x;
  if (A.done[p]) return;
  const size_t o = (size_t)p * n;
  const float* yp = A.y + o;  // the problem's rows
  float *sp = A.S + o, *lap = A.LA2 + o, *lbp = A.LB2 + o, *gp = A.G2 + o;
  float* in_s = smem;
  float* scr = smem + (n + 3) / 4 * 4;
  const ExPlan pl = *A.plan;
  float mass = 0.f;
  if (EPI == EXA_SOURCE) {
#pragma unroll 8
    for (int j = tid; j < n; j += NT) in_s[j] = gp[j];
  } else {
#pragma unroll 8
    for (int j = tid; j < n; j += NT) {
      const float s = sp[j], la = lap[j];
      in_s[j] = s > 0.f ? P::log2(s) - la : P::ninf();
      mass += s;
    }
    if (TC) {
      mass = block_sum(mass, red);
      if (tid == 0 && prt == 0) A.mass[p] = mass;
    }
  }
  float part = 0.f;
  struct Pre { float a, b; };  // source: S, LA2 of the previous iteration; target: y
  auto load = [&](int i) {
    Pre q{0.f, 0.f};
    if (EPI == EXA_SOURCE) {
      if (A.check || TC) q.a = sp[i];
      if (A.check) q.b = lap[i];
    } else q.a = yp[i];
    return q;
  };
  auto row = [&](int i, Pre pre, float base, float sum, float di2) {
    const float v = sum > 0.f ? base + (P::log2(sum) - di2) : P::ninf();
    if (EPI == EXA_SOURCE) {
      const float s = pre.a;
      if (A.check && s > 0.f) {
        // s |a_new / a_old - 1|; the difference of the references is exact, so the ratio keeps FP32
        // relative precision; a jump beyond 2^64 is taken in log form, capped at 2^120
        const float dl = (base - pre.b) - di2;
        if (!(sum > 0.f)) part += s;
        else if (dl + P::log2(sum) > 64.f) part += P::exp2(fminf(P::log2(s) + (dl + P::log2(sum)), 120.f));
        else part += s * fabsf(sum * P::exp2(dl) - 1.f);
      }
      lap[i] = v;
      if (TC) {
        const float r = s > 0.f ? v - P::log2(s) : 0.f, hi = exa_tf32(r);
        const size_t ro = (size_t)slot * A.ld + i;
        A.Rhi[ro] = hi;
        A.Rlo[ro] = exa_tf32(r - hi);
      }
    } else {
      lbp[i] = v;
      gp[i] = exa_datafit<TC>(A, v, pre.a);
    }
  };
  if constexpr (T == 4) {  // one CTA per problem
    ex_apply<T>(in_s, A.xt, n, pl, 0, pl.nb, scr, T, load, row);
  } else {
    const int I0 = pl.nb * prt / parts, I1 = pl.nb * (prt + 1) / parts;
    if (I1 > I0) ex_apply<T>(in_s, A.xt, n, pl, I0, I1, scr, T, load, row);
  }
  if (EPI == EXA_TARGET || !A.check) return;

  // ---- violation of the previous iteration's plan and the stopping decision --------------------
  part = block_sum(part, red);
  if (parts > 1) {
    if (tid == 0) {
      A.part[o + prt] = part;
      __threadfence();
      last_s = atomicAdd(A.count + p, 1) == parts - 1;
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    if (tid == 0) {
      part = 0.f;
      for (int q = 0; q < parts; ++q) part += __ldcg(A.part + o + q);
      A.count[p] = 0;
    }
  }
  float dw = 0.f;
  if (TC) {  // weight change of the previous iteration's update
    float num = 0.f, den = 0.f;
    for (int j = tid; j < A.k; j += NT) {
      const float wv = A.W[(size_t)p * A.k + j];
      num += fabsf(wv - A.Wprev[(size_t)p * A.k + j]);
      den += fabsf(wv);
    }
    num = block_sum(num, red);
    den = block_sum(den, red);
    dw = num / den;
  }
  if (tid == 0) {
    const float e = part / A.mass[p];
    if (TC) A.dw[p] = dw;
    else dw = A.dw[p];
    A.err[p] = e;
    const int st = stop_decision<float>(e, dw, A.tol, A.dw_tol, false, false, A.it, A.max_iter);
    if (st >= 0) {
      A.status[p] = st;
      A.iters[p] = A.it;
      A.done[p] = 1;
    }
  }
}

// Log ratios r = LA2 - log2 S as the TF32 operand, for the MM steps after an iteration's first.
static __global__ void __launch_bounds__(256) ex_ratio_kernel(ExArgs A) {
  const int slot = blockIdx.x;
  if (slot >= *A.n_active) return;
  const size_t o = (size_t)A.active[slot] * A.n, ro = (size_t)slot * A.ld;
  for (int i = threadIdx.x; i < A.n; i += 256) {
    const float s = A.S[o + i];
    const float r = s > 0.f ? A.LA2[o + i] - Prec<float>::log2(s) : 0.f, hi = exa_tf32(r);
    A.Rhi[ro + i] = hi;
    A.Rlo[ro + i] = exa_tf32(r - hi);
  }
}

// CTAs per problem: enough for two per SM, at most one per possible row block (and one per bin: the
// partial violations live in the problem's own row).
inline int exa_parts(int batch, int n, int sms) {
  const int want = (2 * sms + batch - 1) / batch;
  return want < 1 ? 1 : (want > EX_NB ? (EX_NB < n ? EX_NB : n) : (want < n ? want : n));
}

template <int EPI, bool TC, int T>
static inline cudaError_t launch_ex_cfg(const ExArgs& a, int batch, int parts, int sms, cudaStream_t stream) {
  size_t smem = exa_smem_bytes(a.n, T);
  // CTAs that leave SMs idle get an SM each: more than half its shared memory (one target at n = 16384, 20
  // iterations: 2.33 ms where two may share an SM, 2.22 with one; four: 2.38, 2.21)
  if (parts > 1 && (long long)batch * parts <= sms && smem < 116 * 1024) smem = 116 * 1024;
  if (smem > 48 * 1024) {  // the largest size for every call: the limit is the process's, threads would lower it
    const cudaError_t e = cudaFuncSetAttribute(ex_apply_kernel<EPI, TC, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)exa_smem_bytes(EXA_MAX_N, T));
    if (e != cudaSuccess) return e;
  }
  // CTAs that leave SMs idle are launched late: early ones share SMs beside a running GEMM (one target at
  // n = 16384, 20 iterations: 2.43 ms early, 2.23 late)
  return launch_pdl(parts == 1 || a.early, ex_apply_kernel<EPI, TC, T>, dim3(batch, parts), dim3(32 * T), smem, stream, a);
}
// Four warps per problem where there are at least four problems per SM (1024 x 1024, in the
// first version: two, four, eight warps 35, 32, 74 us an apply), else eight and several CTAs per problem.
template <int EPI, bool TC>
static inline cudaError_t launch_ex_apply(const ExArgs& a, int batch, int sms, cudaStream_t stream) {
  if (batch >= 4 * sms && a.n <= 8192) return launch_ex_cfg<EPI, TC, 4>(a, batch, 1, sms, stream);
  return launch_ex_cfg<EPI, TC, 8>(a, batch, exa_parts(batch, a.n, sms), sms, stream);
}

// ---- MM step and source step of a batch sharing the dictionary (FP32) ---------------------------
// One CTA takes PB problems through an iteration's weight update: NU = D^T r with r = LA2 - log2 S,
// Table 2's update, S = D w, mm_steps times with the same LA2.  Against one CTA per problem, each
// entry of D that is read from L2 serves PB problems, and the multiply-adds run on packed pairs of
// problems.  Arithmetic is FP32 throughout, as in mm_kernel.
//   phase A: a chunk of 256 rows' log ratios is staged as [row][problem]; warps take rows, lanes
//            columns; the warps' sums are added in order
//   phase C: threads take rows (Dt is read coalesced along rows), the weights are broadcast
constexpr int MMB_NT = 256, MMB_NW = MMB_NT / 32, MMB_CHUNK = MMB_NT;

template <int PB, int KQ>
struct MmbSmem {
  static constexpr int KP = 32 * KQ;
  static constexpr int RS = MMB_CHUNK * PB;                     // staged ratios
  static constexpr int RED = MMB_NW * KP * (PB < 4 ? PB : 4);        // warps' sums of up to 4 problems
  static constexpr int U = RS > RED ? RS : RED;
  static constexpr size_t bytes = 4 * (size_t)(U + 3 * KP * PB);  // + weights [k][PB] (new), starting weights, NU
};

template <int PB, int KQ>
__global__ void __launch_bounds__(MMB_NT) mm_batch_kernel(MMBArgs A) {
  using P = Prec<float>;
  using SM = MmbSmem<PB, KQ>;
  constexpr int KP = SM::KP, H = PB > 1 ? PB / 2 : 1, G = PB < 4 ? PB : 4;
  extern __shared__ __align__(16) float smem[];
  float* rs = smem;               // [MMB_CHUNK][PB], then the warps' sums
  float* w_s = smem + SM::U;      // [KP][PB]
  float* w0_s = w_s + KP * PB;
  float* nu_s = w0_s + KP * PB;   // [PB][KP]
  __shared__ float red[32];
  __shared__ int p_s[PB];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = A.n, k = A.k;
  pdl_wait();
  const int na = *A.n_active, slot0 = blockIdx.x * PB;
  if (slot0 >= na) return;
  if (tid < PB) {
    const int p = slot0 + tid < na ? A.active[slot0 + tid] : -1;
    p_s[tid] = (p >= 0 && !A.done[p]) ? p : -1;
  }
  __syncthreads();
  bool any = false;
#pragma unroll
  for (int q = 0; q < PB; ++q) any |= p_s[q] >= 0;
  if (!any) return;
  for (int e = tid; e < k * PB; e += MMB_NT) {
    const int q = e / k, j = e - q * k, p = p_s[q];
    const float w = p >= 0 ? A.W[(size_t)p * k + j] : 1.f;
    w_s[j * PB + q] = w;
    w0_s[j * PB + q] = w;
  }
  for (int m = 0; m < A.mm_steps; ++m) {
    // ---- phase A ----
    uint64_t acc[H][KQ];
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
      for (int q = 0; q < KQ; ++q) acc[h][q] = 0ull;
    for (int c0 = 0; c0 < n; c0 += MMB_CHUNK) {
      __syncthreads();
      {
        const int i = c0 + tid;  // one row of the chunk per thread
        float s[PB], la[PB];
#pragma unroll
        for (int q = 0; q < PB; ++q) {
          const int p = p_s[q];
          const bool in = i < n && p >= 0;
          s[q] = in ? A.S[(size_t)p * n + i] : 0.f;
          la[q] = in ? A.LA2[(size_t)p * n + i] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < PB; ++q) rs[tid * PB + q] = s[q] > 0.f ? la[q] - P::log2(s[q]) : 0.f;
      }
      __syncthreads();
      const int cnt = min(MMB_CHUNK, n - c0);
      constexpr int U = KQ >= 8 ? 2 : (KQ >= 4 ? 4 : 8);
      float d[U][KQ];
      auto load = [&](int r0) {
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int q = 0; q < KQ; ++q) {
            const int j = lane + 32 * q;
            d[u][q] = (r0 + u < cnt && j < k) ? __ldg(A.D + (size_t)(c0 + r0 + u) * k + j) : 0.f;
          }
      };
      load(warp * U);
      for (int r0 = warp * U; r0 < cnt; r0 += MMB_NW * U) {
        float cur[U][KQ];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int q = 0; q < KQ; ++q) cur[u][q] = d[u][q];
        if (r0 + MMB_NW * U < cnt) load(r0 + MMB_NW * U);  // the next rows arrive while these are used
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float* rr = rs + (r0 + u) * PB;  // rows past cnt were staged as 0
          uint64_t r2[H];
          if constexpr (PB >= 4) {
#pragma unroll
            for (int h = 0; h < H; h += 2) {
              const float4 v = *reinterpret_cast<const float4*>(rr + 2 * h);
              r2[h] = f2_pack(v.x, v.y);
              r2[h + 1] = f2_pack(v.z, v.w);
            }
          } else r2[0] = f2_pack(rr[0], 0.f);
#pragma unroll
          for (int q = 0; q < KQ; ++q) {
            const uint64_t d2 = f2_pack(cur[u][q], cur[u][q]);
#pragma unroll
            for (int h = 0; h < H; ++h) acc[h][q] = f2_fma(d2, r2[h], acc[h][q]);
          }
        }
      }
    }
    // the warps' sums, up to four problems at a time
#pragma unroll
    for (int g = 0; g < PB; g += G) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < KQ; ++q)
#pragma unroll
        for (int h = 0; h < (G + 1) / 2; ++h) {
          float a, b;
          f2_unpack(acc[g / 2 + h][q], a, b);
          rs[(warp * G + 2 * h) * KP + lane + 32 * q] = a;
          if (G > 1) rs[(warp * G + 2 * h + 1) * KP + lane + 32 * q] = b;
        }
      __syncthreads();
      for (int e = tid; e < G * KP; e += MMB_NT) {
        float sum = 0.f;
#pragma unroll
        for (int w8 = 0; w8 < MMB_NW; ++w8) sum += rs[w8 * G * KP + e];
        nu_s[g * KP + e] = sum;
      }
    }
    __syncthreads();
    // ---- phase B: penalty update (Table 2), as mm_kernel ----
    for (int e = tid; e < k * PB; e += MMB_NT) {
      const int q = e / k, j = e - q * k, p = p_s[q];
      if (p < 0) continue;
      const float xj = A.xcol[j], wold = w_s[j * PB + q];
      const float nu = P::log(wold) + nu_s[q * KP + j] * float(kLn2) / xj;
      const float shift = (A.penalty == PEN_L1 || A.penalty == PEN_ELASTIC) ? A.alpha / (A.eps * xj) : 0.f;
      float wn;
      if (A.penalty == PEN_L2SQ || A.penalty == PEN_ELASTIC) {
        const float c = (A.penalty == PEN_ELASTIC ? A.beta : A.alpha) / (A.eps * xj);
        wn = wright_omega<float>(P::log(c) + nu - shift) / c;
      } else wn = P::exp(nu - shift);
      w_s[j * PB + q] = wn;
      if (m + 1 == A.mm_steps) A.W[(size_t)p * k + j] = wn;
    }
    __syncthreads();
    // ---- phase C: S = D w ----
    constexpr int IPT = 2, JB = 8;  // rows per thread, columns of D in flight
    float mass[PB];
#pragma unroll
    for (int q = 0; q < PB; ++q) mass[q] = 0.f;
    for (int c0 = 0; c0 < n; c0 += MMB_NT * IPT) {
      uint64_t s2[IPT][H];
#pragma unroll
      for (int t = 0; t < IPT; ++t)
#pragma unroll
        for (int h = 0; h < H; ++h) s2[t][h] = 0ull;
      for (int j0 = 0; j0 < k; j0 += JB) {
        float d[JB][IPT];
#pragma unroll
        for (int jj = 0; jj < JB; ++jj)
#pragma unroll
          for (int t = 0; t < IPT; ++t) {
            const int i = c0 + t * MMB_NT + tid;
            d[jj][t] = (i < n && j0 + jj < k) ? __ldg(A.Dt + (size_t)(j0 + jj) * n + i) : 0.f;
          }
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {
          const float* ww = w_s + min(j0 + jj, k - 1) * PB;  // (past k: times 0)
          uint64_t w2[H];
          if constexpr (PB >= 4) {
#pragma unroll
            for (int h = 0; h < H; h += 2) {
              const float4 v = *reinterpret_cast<const float4*>(ww + 2 * h);
              w2[h] = f2_pack(v.x, v.y);
              w2[h + 1] = f2_pack(v.z, v.w);
            }
          } else w2[0] = f2_pack(ww[0], 0.f);
#pragma unroll
          for (int t = 0; t < IPT; ++t) {
            const uint64_t d2 = f2_pack(d[jj][t], d[jj][t]);
#pragma unroll
            for (int h = 0; h < H; ++h) s2[t][h] = f2_fma(d2, w2[h], s2[t][h]);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < IPT; ++t) {
        const int i = c0 + t * MMB_NT + tid;
        if (i >= n) continue;
#pragma unroll
        for (int h = 0; h < H; ++h) {
          float v[2];
          f2_unpack(s2[t][h], v[0], v[1]);
#pragma unroll
          for (int c = 0; c < (PB > 1 ? 2 : 1); ++c) {
            const int q = 2 * h + c, p = p_s[q];
            // a subnormal mass counts as 0, as in source_marginal
            const float s = v[c] < P::tiny() ? 0.f : v[c];
            if (p >= 0) A.S[(size_t)p * n + i] = s;
            mass[q] += s;
          }
        }
      }
    }
    if (m + 1 == A.mm_steps) {
#pragma unroll
      for (int q = 0; q < PB; ++q) {
        const float ms = block_sum(mass[q], red);
        if (tid == 0 && p_s[q] >= 0) A.mass[p_s[q]] = ms;
      }
    }
  }
  // weight change of this iteration's update: ||w - w_start||_1 / ||w||_1, one warp per problem
  __syncthreads();
  for (int q = warp; q < PB; q += MMB_NT / 32) {
    float num = 0.f, den = 0.f;
    for (int j = lane; j < k; j += 32) {
      num += fabsf(w_s[j * PB + q] - w0_s[j * PB + q]);
      den += fabsf(w_s[j * PB + q]);
    }
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (lane == 0 && p_s[q] >= 0) A.dw[p_s[q]] = num / den;
  }
}

template <int PB, int KQ>
static inline cudaError_t launch_mmb_cfg(const MMBArgs& a, int batch, cudaStream_t s) {
  constexpr size_t smem = MmbSmem<PB, KQ>::bytes;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(mm_batch_kernel<PB, KQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(true, mm_batch_kernel<PB, KQ>, dim3((batch + PB - 1) / PB), dim3(MMB_NT), smem, s, a);
}
template <int PB>
static inline cudaError_t launch_mmb_pb(const MMBArgs& a, int batch, cudaStream_t s) {
  if (a.k <= 32) return launch_mmb_cfg<PB, 1>(a, batch, s);
  if (a.k <= 64) return launch_mmb_cfg<PB, 2>(a, batch, s);
  if (a.k <= 128) return launch_mmb_cfg<PB, 4>(a, batch, s);
  return launch_mmb_cfg<PB, 8>(a, batch, s);
}
// Problems per CTA: one up to a problem per SM; then four, which D's reads from L2 serve at once (1024
// problems, 50 iterations of the FP32 batch: 4.34 ms with eight and 128 CTAs, 4.11 with four and 256), and
// eight (half the reads of D) once four would leave more than four CTAs per SM.  Lines not measured
// between: 20 iterations at n = 1024, k = 64 take 1.03 ms for 200 problems, 1.48 for 305, 1.72 for 400, 1.92 for
// 800, 2.59 for 1600 and 5.28 for 4000.
static inline cudaError_t launch_mm_batch(const MMBArgs& a, int batch, int sms, cudaStream_t s) {
  if (batch <= sms) return launch_mmb_pb<1>(a, batch, s);
  if (batch <= 16 * sms) return launch_mmb_pb<4>(a, batch, s);
  return launch_mmb_pb<8>(a, batch, s);
}

}  // namespace otlm
