// Per-site double occupancies <n_i,up n_i,dn> = sum over u, d that both
// contain site i of |psi_ud|^2 (Eq. (13)), for ed_double_occupation and
// ed_double_occupation_static.
//
// Bound by the FP64 pipe (two operations per cycle and SM), so the additions
// count.  A thread owns one column d and walks rows u in ascending word
// order: whether site i is in u is then uniform over the block (a branch, not
// a masked addition, which takes the pipe's time also where it is masked off),
// and whether it is in d is applied once at the end.  |psi|^2 goes to one of
// 16 sums, that of the row's low four bits, and to the sum of the run of rows
// that share the higher bits; when those change, the run's sum goes to the
// sites of the next four bits and to the next longer run: about 3 additions
// per element where one per site takes up to Ns + 1.  The accumulators of a
// warp are folded together (a fold halves the values and the lanes at once),
// 16 additions instead of 80.  Ns = 14 ladder, (7,7), complex128: 509 -> 197
// us for the kernel, 104 -> 12 us for the final sums (one warp per site instead
// of one thread), and with the scratch kept in the context 632 -> 232 us for
// the call.
#pragma once

#include "device.cuh"

namespace ed {

constexpr int kDoccBlocks = 1024;   // most blocks: partial[kDoccVals][kDoccBlocks]
constexpr int kDoccThreads = 256;

// Threads per block, column blocks and rows per block for a sector.
struct DoccShape {
  int threads, cols, rows, blocks;
};
inline DoccShape docc_shape(int dim_up, int dim_dn) {
  DoccShape s;
  s.threads = dim_dn >= kDoccThreads ? kDoccThreads : (dim_dn + 31) / 32 * 32;
  s.cols = (dim_dn + s.threads - 1) / s.threads;
  const int chunks = kDoccBlocks / s.cols;   // >= 20 (rows have at most 12870 columns)
  // at least 16 rows a thread: folding its sums costs as much as about 9 rows
  // (us per call with at least 1 / 8 / 16: 495 x 495 90 / 57 / 60, 70 x 70 49 /
  // 50 / 46, 924 x 924 92 / 82 / 73)
  s.rows = std::max(16, (dim_up + chunks - 1) / chunks);
  s.blocks = s.cols * ((dim_up + s.rows - 1) / s.rows);
  return s;
}

// Runs f(i) for the set bits i < 4 of n, a branch per value of n (uniform).
template <typename F>
__device__ __forceinline__ void for_bits4(uint32_t n, F&& f) {
  switch (n & 15u) {
    case 1: f(0); break;
    case 2: f(1); break;
    case 3: f(0); f(1); break;
    case 4: f(2); break;
    case 5: f(0); f(2); break;
    case 6: f(1); f(2); break;
    case 7: f(0); f(1); f(2); break;
    case 8: f(3); break;
    case 9: f(0); f(3); break;
    case 10: f(1); f(3); break;
    case 11: f(0); f(1); f(3); break;
    case 12: f(2); f(3); break;
    case 13: f(0); f(2); f(3); break;
    case 14: f(1); f(2); f(3); break;
    case 15: f(0); f(1); f(2); f(3); break;
    default: break;
  }
}

template <typename C>
static __global__ void __launch_bounds__(kDoccThreads)
k_docc(const C* psi, SectorDev sd, int cols, int rows, double* partial) {
  static_assert(kMaxSites == 16, "four groups of four sites");
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int d = (int)(blockIdx.x % cols) * blockDim.x + threadIdx.x;
  const int u0 = (int)(blockIdx.x / cols) * rows, u1 = min(sd.dim_up, u0 + rows);
  const bool on = d < sd.dim_dn;
  double a[kMaxSites];   // sum over rows u that contain site i, of this column
#pragma unroll
  for (int i = 0; i < kMaxSites; ++i) a[i] = 0.0;
  double low[16];        // sum over rows with these low four bits
#pragma unroll
  for (int i = 0; i < 16; ++i) low[i] = 0.0;
  double run[3] = {0.0, 0.0, 0.0};   // |psi|^2 since bits >= 4, 8, 12 changed
  double all = 0.0;                  // |psi|^2
  const C* col = psi + (on ? d : 0);
  constexpr int U = 4;
  for (int u = u0; u < u1; u += U) {
    double q[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      q[k] = 0.0;
      if (on && u + k < u1) {
        const C p = __ldcs(col + (size_t)(u + k) * sd.dim_dn);
        const double x = (double)p.x, y = (double)p.y;
        q[k] = x * x;
        q[k] += y * y;
      }
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (u + k >= u1) continue;   // uniform over the block, as all below
      const uint32_t w = __ldg(sd.up_word + u + k);
      const uint32_t change = u + k + 1 < u1 ? w ^ __ldg(sd.up_word + u + k + 1) : 0xffffffffu;
      switch (w & 15u) {
        case 0: low[0] += q[k]; break;
        case 1: low[1] += q[k]; break;
        case 2: low[2] += q[k]; break;
        case 3: low[3] += q[k]; break;
        case 4: low[4] += q[k]; break;
        case 5: low[5] += q[k]; break;
        case 6: low[6] += q[k]; break;
        case 7: low[7] += q[k]; break;
        case 8: low[8] += q[k]; break;
        case 9: low[9] += q[k]; break;
        case 10: low[10] += q[k]; break;
        case 11: low[11] += q[k]; break;
        case 12: low[12] += q[k]; break;
        case 13: low[13] += q[k]; break;
        case 14: low[14] += q[k]; break;
        default: low[15] += q[k]; break;
      }
      run[0] += q[k];
      if (change >> 4) {
        for_bits4(w >> 4, [&](int i) { a[4 + i] += run[0]; });
        run[1] += run[0];
        run[0] = 0.0;
        if (change >> 8) {
          for_bits4(w >> 8, [&](int i) { a[8 + i] += run[1]; });
          run[2] += run[1];
          run[1] = 0.0;
          if (change >> 12) {
            for_bits4(w >> 12, [&](int i) { a[12 + i] += run[2]; });
            all += run[2];
            run[2] = 0.0;
          }
        }
      }
    }
  }
#pragma unroll
  for (int n = 1; n < 16; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if ((n >> i) & 1) a[i] += low[n];
  const uint32_t dw = on ? __ldg(sd.dn_word + d) : 0u;
#pragma unroll
  for (int i = 0; i < kMaxSites; ++i)
    if (!((dw >> i) & 1u)) a[i] = 0.0;
#pragma unroll
  for (int b = 0; b < 4; ++b) {   // fold the 16 sums into lane bits 4..1
    const int o = 16 >> b;
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < (kMaxSites >> (b + 1)); ++i) {
      const double keep = up ? a[2 * i + 1] : a[2 * i], give = up ? a[2 * i] : a[2 * i + 1];
      a[i] = keep + __shfl_xor_sync(full, give, o);
    }
  }
  a[0] += __shfl_xor_sync(full, a[0], 1);
  for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(full, all, o);
  __shared__ double red[kDoccThreads / 32][kDoccVals];
  if (lane == 0) red[warp][kMaxSites] = all;
  // the site of a lane: bit 0 of its index from lane bit 4, .. bit 3 from bit 1
  if ((lane & 1) == 0)
    red[warp][((lane >> 4) & 1) | ((lane >> 2) & 2) | (lane & 4) | ((lane << 2) & 8)] = a[0];
  __syncthreads();
  if (threadIdx.x < kDoccVals) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w][threadIdx.x];
    partial[(size_t)threadIdx.x * kDoccBlocks + blockIdx.x] = s;
  }
}

// out[i] = sum over blocks of partial[i][block], one warp per value
static __global__ void __launch_bounds__(32 * kDoccVals)
k_docc_sum(const double* partial, int blocks, double* out) {
  const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int b = lane;
  for (; b + 96 < blocks; b += 128)
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += partial[(size_t)i * kDoccBlocks + b + 32 * q];
  for (; b < blocks; b += 32) s[0] += partial[(size_t)i * kDoccBlocks + b];
  double r = (s[0] + s[1]) + (s[2] + s[3]);
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if (lane == 0) out[i] = r;
}

// scratch: the partial sums, then kDoccVals results
static_assert(kDoccScratchDoubles == (size_t)(kDoccBlocks + 1) * kDoccVals, "docc scratch");

// partial[0][block] = sum of (sites in both u and d) |psi_ud|^2 over the block's
// elements: the average where |psi|^2 is not finite, in which every element
// counts, also one that no site weighs (0 times infinity is not a number).
template <typename C>
static __global__ void __launch_bounds__(kDoccThreads)
k_docc_weighted(const C* psi, SectorDev sd, double* partial) {
  __shared__ double red[kDoccThreads / 32];
  const int64_t D = (int64_t)sd.dim_up * sd.dim_dn;
  double v[1] = {0.0};
  for (int64_t t = blockIdx.x * (int64_t)kDoccThreads + threadIdx.x; t < D;
       t += (int64_t)gridDim.x * kDoccThreads) {
    const int u = (int)(t / sd.dim_dn), d = (int)(t - (int64_t)u * sd.dim_dn);
    const C p = psi[t];
    const double q = (double)p.x * p.x + (double)p.y * p.y;
    v[0] += __popc(__ldg(sd.up_word + u) & __ldg(sd.dn_word + d)) * q;
  }
  block_reduce<1>(v, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = v[0];
}

static inline cudaError_t launch_docc(bool fp64, const void* psi, const SectorDev& sd, double* scratch,
                                      cudaStream_t s) {
  const DoccShape h = docc_shape(sd.dim_up, sd.dim_dn);
  if (fp64)
    k_docc<double2><<<h.blocks, h.threads, 0, s>>>(static_cast<const double2*>(psi), sd, h.cols,
                                                   h.rows, scratch);
  else
    k_docc<float2><<<h.blocks, h.threads, 0, s>>>(static_cast<const float2*>(psi), sd, h.cols,
                                                  h.rows, scratch);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_docc_sum<<<1, 32 * kDoccVals, 0, s>>>(scratch, h.blocks, scratch + (size_t)kDoccBlocks * kDoccVals);
  return cudaGetLastError();
}

static inline cudaError_t launch_docc_weighted(bool fp64, const void* psi, const SectorDev& sd,
                                               double* scratch, cudaStream_t s) {
  const int64_t D = (int64_t)sd.dim_up * sd.dim_dn;
  const int nb = (int)std::min<int64_t>(kDoccBlocks, (D + kDoccThreads - 1) / kDoccThreads);
  if (fp64)
    k_docc_weighted<<<nb, kDoccThreads, 0, s>>>(static_cast<const double2*>(psi), sd, scratch);
  else
    k_docc_weighted<<<nb, kDoccThreads, 0, s>>>(static_cast<const float2*>(psi), sd, scratch);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // (the other sums of k_docc_sum are not read)
  k_docc_sum<<<1, 32 * kDoccVals, 0, s>>>(scratch, nb, scratch + (size_t)kDoccBlocks * kDoccVals);
  return cudaGetLastError();
}

}  // namespace ed
