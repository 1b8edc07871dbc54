// Ground-state Lanczos kernels (float64): full reorthogonalisation and the
// vector updates of ed_ground_state.
//
// H(A = 0) is real, so every Lanczos vector is p(H) v_0 with a real polynomial
// p, and the inner product of any two of them is real: the imaginary part of
// a computed one is rounding.  The recursion is therefore the real symmetric
// one of H on pairs (Re, Im), and its projections take real coefficients: two
// float64 multiply-adds per element and vector where complex ones take four.
// These passes are bound by the FP64 pipe (two multiply-adds per cycle and
// SM), so that halves their time.
//
// One projection pass per step is enough where it does not cancel: w is first
// orthogonalised against v_k and v_{k-1} by the recursion itself, which is
// what takes the large components out, and the pass over all vectors then
// removes rounding-level ones.  A second pass follows if the first took more
// than half of |w|^2 away (the criterion of Daniel, Gragg, Kaufman and
// Stewart, Math. Comp. 30, 772 (1976)); the decision stays on the device.
// 12-site torus, (6,5), D = 731,808, 285 steps: the two complex passes of the
// earlier form took 1.07 s of a solve of 1.36 s; the solve now takes 0.29 s,
// 0.06 s of it the products H v.
#include "device.cuh"

namespace ed {

namespace {

constexpr int kThreads = 256;

template <int K, typename F>
__device__ __forceinline__ void sum_then(double (&v)[K], double* partials, unsigned* counter, F&& fin) {
  __shared__ double red[32 * K];
  __shared__ int flag;
  if (reduce_last_block<K>(v, blockIdx.x, 0, gridDim.x, partials, counter, red, &flag))
    if (threadIdx.x == 0) fin(v);
}

// S.alpha[k] = Re<v, w>
__global__ void __launch_bounds__(kThreads)
k_gs_dot(const double2* v, const double2* w, int64_t D, GsScalars* S, int k, double* partials,
         unsigned* counter) {
  double acc[1] = {0.0};
  for (int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x; t < D; t += (int64_t)gridDim.x * kThreads) {
    const double2 a = v[t], b = w[t];
    acc[0] += a.x * b.x;
    acc[0] += a.y * b.y;
  }
  sum_then<1>(acc, partials, counter, [&](double (&s)[1]) { S->alpha[k] = s[0]; });
}

// w -= alpha_k v + beta_{k-1} vp (vp null for k = 0); S.before = |w|^2
__global__ void __launch_bounds__(kThreads)
k_gs_sub(double2* w, const double2* v, const double2* vp, int64_t D, GsScalars* S, int k,
         double* partials, unsigned* counter) {
  const double al = S->alpha[k], be = vp ? S->beta[k - 1] : 0.0;
  double acc[1] = {0.0};
  for (int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x; t < D; t += (int64_t)gridDim.x * kThreads) {
    double2 o = w[t];
    const double2 a = v[t];
    o.x -= al * a.x;
    o.y -= al * a.y;
    if (vp) {
      const double2 b = vp[t];
      o.x -= be * b.x;
      o.y -= be * b.y;
    }
    w[t] = o;
    acc[0] += o.x * o.x;
    acc[0] += o.y * o.y;
  }
  sum_then<1>(acc, partials, counter, [&](double (&s)[1]) {
    S->before = s[0];
    S->again = 1;   // the first pass always runs
  });
}

// partial[block][i] = Re<V_i, w> over the block's chunk of kThreads * E
// elements, i < k.  w stays in registers; the vectors are taken kDots at a
// time and their lane sums folded together (a fold halves the values and the
// lanes at once: about one addition per vector and warp instead of five).
constexpr int kDots = 8;
template <int E>
__global__ void __launch_bounds__(kThreads)
k_gs_multidot(const double2* V, int64_t ldV, int k, const double2* w, int64_t D, double* partial,
              const GsScalars* S) {
  if (!S->again) return;
  __shared__ double red[kThreads / 32][kDots];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t0 = blockIdx.x * (int64_t)(kThreads * E) + threadIdx.x;
  double2 x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int64_t t = t0 + e * kThreads;
    x[e] = t < D ? w[t] : make_double2(0.0, 0.0);
  }
  for (int i0 = 0; i0 < k; i0 += kDots) {
    double s[kDots];
#pragma unroll
    for (int q = 0; q < kDots; ++q) {
      s[q] = 0.0;
      if (i0 + q >= k) continue;   // uniform over the grid
      const double2* Vi = V + (size_t)(i0 + q) * ldV;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int64_t t = t0 + e * kThreads;
        const double2 a = t < D ? __ldcs(Vi + t) : make_double2(0.0, 0.0);
        s[q] += a.x * x[e].x;
        s[q] += a.y * x[e].y;
      }
    }
    // fold: after the step with offset o, lane l holds the values q whose
    // bit agrees with bit o of l; kDots = 8 values fold into lane bits 4..2
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int o = 16 >> b;
      const bool up = lane & o;
#pragma unroll
      for (int q = 0; q < (kDots >> (b + 1)); ++q) {
        const double keep = up ? s[2 * q + 1] : s[2 * q], give = up ? s[2 * q] : s[2 * q + 1];
        s[q] = keep + __shfl_xor_sync(full, give, o);
      }
    }
    s[0] += __shfl_xor_sync(full, s[0], 2);
    s[0] += __shfl_xor_sync(full, s[0], 1);
    // the value of lane l: bit 0 of its index from lane bit 4, bit 1 from 3, bit 2 from 2
    if ((lane & 3) == 0) red[warp][((lane >> 4) & 1) | ((lane >> 2) & 2) | (lane & 4)] = s[0];
    __syncthreads();
    if (threadIdx.x < kDots && i0 + (int)threadIdx.x < k) {
      double r = 0.0;
#pragma unroll
      for (int q = 0; q < kThreads / 32; ++q) r += red[q][threadIdx.x];
      partial[(size_t)blockIdx.x * k + i0 + threadIdx.x] = r;
    }
    __syncthreads();
  }
}

// c[i] = sum over blocks of partial[block][i], one warp per i
__global__ void __launch_bounds__(kThreads)
k_gs_reduce(const double* partial, int nblk, int k, double* c, const GsScalars* S) {
  if (!S->again) return;
  const int i = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= k) return;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int b = lane;
  for (; b + 96 < nblk; b += 128)
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += partial[(size_t)(b + 32 * q) * k + i];
  for (; b < nblk; b += 32) s[0] += partial[(size_t)b * k + i];
  double r = (s[0] + s[1]) + (s[2] + s[3]);
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if (lane == 0) c[i] = r;
}

// w -= sum_i c_i V_i, |w|^2 fused; pass 0 decides on the second pass
__global__ void __launch_bounds__(kThreads)
k_gs_multiaxpy(const double2* V, int64_t ldV, int k, const double* c, double2* w, int64_t D,
               GsScalars* S, int pass, double* partials, unsigned* counter) {
  if (!S->again) return;   // uniform over the grid: set before this kernel
  extern __shared__ double cs[];
  for (int i = threadIdx.x; i < k; i += kThreads) cs[i] = c[i];
  __syncthreads();
  double acc[1] = {0.0};
  constexpr int E = 2;
  for (int64_t t0 = blockIdx.x * (int64_t)(kThreads * E) + threadIdx.x; t0 < D;
       t0 += (int64_t)gridDim.x * kThreads * E) {
    double2 o[E];
    bool ok[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      ok[e] = t0 + e * kThreads < D;
      o[e] = ok[e] ? w[t0 + e * kThreads] : make_double2(0.0, 0.0);
    }
    const double2* Vt = V + t0;
    int i = 0;
    constexpr int U = 8;
    for (; i + U <= k; i += U) {
      double2 a[U][E];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < E; ++e)
          a[u][e] = ok[e] ? __ldcs(Vt + (size_t)(i + u) * ldV + e * kThreads) : make_double2(0.0, 0.0);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < E; ++e) {
          o[e].x -= cs[i + u] * a[u][e].x;
          o[e].y -= cs[i + u] * a[u][e].y;
        }
    }
    for (; i < k; ++i)
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (ok[e]) {
          const double2 a = __ldcs(Vt + (size_t)i * ldV + e * kThreads);
          o[e].x -= cs[i] * a.x;
          o[e].y -= cs[i] * a.y;
        }
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (ok[e]) {
        w[t0 + e * kThreads] = o[e];
        acc[0] += o[e].x * o[e].x;
        acc[0] += o[e].y * o[e].y;
      }
  }
  sum_then<1>(acc, partials, counter, [&](double (&s)[1]) {
    S->norm2 = s[0];
    S->again = pass == 0 && s[0] < 0.5 * S->before ? 1 : 0;
  });
}

// beta_k = |w|, v_{k+1} = w / beta_k
__global__ void __launch_bounds__(kThreads)
k_gs_next(const double2* w, double2* vn, int64_t D, GsScalars* S, int k) {
  const double b = sqrt(S->norm2), s = 1.0 / b;
  if (blockIdx.x == 0 && threadIdx.x == 0) S->beta[k] = b;
  for (int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x; t < D; t += (int64_t)gridDim.x * kThreads) {
    const double2 o = w[t];
    vn[t] = make_double2(o.x * s, o.y * s);
  }
}

// (sv[0], si[0]) = the block's largest value and its first index
__device__ __forceinline__ void larger_of(double* sv, int64_t* si) {
  __syncthreads();
  for (int o = kThreads / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      const double b = sv[threadIdx.x + o];
      const int64_t i = si[threadIdx.x + o];
      if (b > sv[threadIdx.x] || (b == sv[threadIdx.x] && i < si[threadIdx.x])) {
        sv[threadIdx.x] = b;
        si[threadIdx.x] = i;
      }
    }
    __syncthreads();
  }
}

// Largest |y_t| and its first index, then y *= conj(y_max) / |y_max| with the
// largest element exactly real (the phase convention of the result).
__global__ void __launch_bounds__(kThreads)
k_gs_absmax(const double2* y, int64_t D, double* val, int64_t* idx) {
  double best = -1.0;
  int64_t at = 0;
  for (int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x; t < D; t += (int64_t)gridDim.x * kThreads) {
    const double a = hypot(y[t].x, y[t].y);
    if (a > best) { best = a; at = t; }
  }
  __shared__ double sv[kThreads];
  __shared__ int64_t si[kThreads];
  sv[threadIdx.x] = best;
  si[threadIdx.x] = at;
  larger_of(sv, si);
  if (threadIdx.x == 0) { val[blockIdx.x] = sv[0]; idx[blockIdx.x] = si[0]; }
}
__global__ void __launch_bounds__(kThreads)
k_gs_phase(const double2* y, double2* out, int64_t D, const double* val, const int64_t* idx, int nblk) {
  __shared__ double sv[kThreads];
  __shared__ int64_t si[kThreads];
  sv[threadIdx.x] = (int)threadIdx.x < nblk ? val[threadIdx.x] : -2.0;
  si[threadIdx.x] = (int)threadIdx.x < nblk ? idx[threadIdx.x] : 0;
  larger_of(sv, si);
  const double best = sv[0];
  const int64_t at = si[0];
  const double2 z = y[at];
  const double pr = z.x / best, pi = -z.y / best;
  for (int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x; t < D; t += (int64_t)gridDim.x * kThreads) {
    const double2 v = y[t];
    out[t] = t == at ? make_double2(best, 0.0)
                     : make_double2(v.x * pr - v.y * pi, v.x * pi + v.y * pr);
  }
}

int grid_of(int64_t n, int per) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(kGsMaxBlocks, (n + per - 1) / per));
}

// elements per block of k_gs_multidot: small chunks fill the chip at Ns = 12,
// large ones keep the partial sums small at Ns = 14 and 16
bool wide(int64_t D) { return D > (int64_t)kGsMaxBlocks * 4 * kThreads; }

int64_t dot_blocks(int64_t D) {
  const int64_t per = (wide(D) ? 16 : 4) * (int64_t)kThreads;
  return (D + per - 1) / per;
}

}  // namespace

cudaError_t launch_gs_step(const double2* V, int64_t D, int k, double2* w, GsScalars* S,
                           double* coef, double* partials, unsigned* counter, double2* vnext,
                           cudaStream_t s) {
  // The partial projections, dot_blocks(D) x (k + 1) doubles, go where v_{k+1}
  // will be: 2 D doubles, and k < D, k < kGsMaxVectors make them fit (one block
  // up to 1024 elements, at most D / 1024 + 1 blocks of 200 above).
  double* dots = reinterpret_cast<double*>(vnext);
  const int g = grid_of(D, 2 * kThreads);
  const double2* vk = V + (size_t)k * D;
  k_gs_dot<<<g, kThreads, 0, s>>>(vk, w, D, S, k, partials, counter);
  k_gs_sub<<<g, kThreads, 0, s>>>(w, vk, k > 0 ? vk - D : nullptr, D, S, k, partials, counter);
  const int nb = (int)dot_blocks(D), n = k + 1;
  if ((int64_t)nb * n > 2 * D) return cudaErrorInvalidValue;
  for (int pass = 0; pass < 2; ++pass) {
    if (wide(D)) k_gs_multidot<16><<<nb, kThreads, 0, s>>>(V, D, n, w, D, dots, S);
    else k_gs_multidot<4><<<nb, kThreads, 0, s>>>(V, D, n, w, D, dots, S);
    k_gs_reduce<<<(n + kThreads / 32 - 1) / (kThreads / 32), kThreads, 0, s>>>(dots, nb, n, coef, S);
    k_gs_multiaxpy<<<g, kThreads, n * sizeof(double), s>>>(V, D, n, coef, w, D, S, pass, partials,
                                                           counter);
  }
  k_gs_next<<<g, kThreads, 0, s>>>(w, vnext, D, S, k);
  return cudaGetLastError();
}

cudaError_t launch_gs_phase(const double2* y, double2* out, int64_t D, double* val, int64_t* idx,
                            cudaStream_t s) {
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(kGsPhaseBlocks, (D + 1023) / 1024));
  k_gs_absmax<<<nb, kThreads, 0, s>>>(y, D, val, idx);
  k_gs_phase<<<grid_of(D, 2 * kThreads), kThreads, 0, s>>>(y, out, D, val, idx, nb);
  return cudaGetLastError();
}

}  // namespace ed
