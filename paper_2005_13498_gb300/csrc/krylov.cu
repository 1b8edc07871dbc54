// Persistent Krylov kernel: whole midpoint (or CFET4) sub-steps of one vector
// in one cooperative launch, for sectors whose rows fit the shared memory of
// the chip.
//
// With one kernel per Lanczos pass a small sector pays a launch, a chain of
// dependent table loads, a tail and a cold start 2 m + 2 times per sub-step.
// Here every CTA (one per SM) owns the rows c, c + G, c + 2 G, .. (G CTAs) for
// the whole launch: they stay in shared memory as the tile the within-row
// gathers (T_dn) read, w never leaves the CTA, the connection lists and the
// ELL words stay in shared memory and L1, and per Lanczos step only two
// grid-wide sums are left (alpha_j, then beta_j together with the visibility
// of x_{j+1}, whose rows the T_up gathers of the other CTAs read through L2).
// Measured per call, separate kernels of the time -> this kernel, complex64:
// 10 steps of the 12-site torus (D = 853,776, m = 20) 8.40 -> 7.23 ms, 20 steps
// of the (2,6) sector of a 10-site chain (D = 9,450, m = 22) 8.16 -> 6.00 ms.
// What bounds it: for the small sectors the latency of the passes and of the
// sums (4.5 us each: 2.1 us from a CTA's store to the last CTA's successful
// poll across the two dies, the rest dependent float64 additions at about
// 50 ns); for the torus the shared-memory and L2 gathers (21 of 37 us per
// Lanczos step).
// It is used when two copies of a CTA's rows fit its shared memory: up to
// about 15 MB of state (D = 1.9 M).  complex64 only: a complex128 form gained 3
// to 18 % over the separate kernels.
//
// The coefficients of all sub-steps of a launch are in shared memory before its
// first pass.  Loaded sub-step by sub-step into one table, right before the
// pass that reads it, they came out wrong in some builds of the complex128 form
// (energies off by up to 1e-6, other values in every run; never without a
// field, never in a launch's first sub-step), though a block barrier stood
// between and no reason was found in the source.  With the tables of the whole
// launch that same form was right, and the same bit by bit, in 180 runs over
// three sectors.  The complex64 form had shown no such error; its results did
// not change.
//
// Grid-wide sums: each CTA publishes its float64 partial as two 64-bit words
// that carry the sum's epoch in their upper halves, and one warp of every CTA
// polls all CTAs' words and adds them in CTA order, so that no counter, no
// second round trip and no broadcast is needed and every CTA holds the same
// total.  All scalars of the recursion (and the small exponential) are then
// computed by every CTA alike.  Every poll is bounded: a wait that runs out
// records ED_ERR_TIMEOUT and ends the CTA.  The launch is cooperative, so the
// CTAs are resident together, and it starts only when all of them can be: beside
// kernels that kept 1, 40 or 150 SMs for 300 ms no wait of 20,000 polls ran out.
#include "device.cuh"

namespace ed {

namespace {

constexpr int kErrTimeout = 4;    // ED_ERR_TIMEOUT
constexpr int kErrNumeric = 7;    // ED_ERR_NUMERIC
constexpr int kUpBatch = 6;
constexpr int kPollLanes = (kKrylovMaxGrid + 31) / 32;

// two rows per 16-byte tile column, 20 warps at 96 registers (980 bytes of
// spill stores and 1628 of spill loads in the code of the paired form)
constexpr int NT = 640, NR = 2;
using TIO = TileIO<float2, NR>;

// Scalars of the Lanczos recursion in shared memory, 1-based as LanczosState.
struct Scalars {
  double alpha[kMaxKrylov + 2], beta[kMaxKrylov + 2], inv[kMaxKrylov + 2];
  double al[64], be[64], yre[64], yim[64];
  // y of the check before, or of one vector less in the step's exponential
  double yprev_re[64], yprev_im[64];
  double tot[2], part[2][4];
  double beta0, scale, as, conv_delta;
  double utab[kMaxSites + 1];   // U n
  int m_eff, stop, status, conv, err, step;
};

// The block barrier; every warp reconverges first (its lanes leave loops apart).
__device__ __forceinline__ void block_sync() {
  __syncwarp();
  __syncthreads();
}

// A published partial: the halves of a float64, each with the sum's epoch in
// the upper 32 bits of its word, so that no ordering between the two words
// is needed.  Slots of one sum lie side by side (16 bytes a CTA): a warp
// polls 32 CTAs with four lines.
__device__ __forceinline__ void ld_slot(const ulonglong2* p, uint64_t& w0, uint64_t& w1) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_slot(ulonglong2* p, double v, uint32_t epoch) {
  const uint64_t bits = (uint64_t)__double_as_longlong(v), e = (uint64_t)epoch << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(e | (bits >> 32)),
               "l"(e | (bits & 0xffffffffull))
               : "memory");
}

// v = sum over all CTAs of the threads' v (K values), left in S.tot of every
// CTA; `after` runs in thread 0 with the totals in place, before the other
// threads go on.  DATA: vectors written before the call are read by other
// CTAs after it.  False when a wait gave up (in all threads of the CTA).
template <int K, bool DATA, typename F>
__device__ __forceinline__ bool grid_sum(const double (&v)[K], double* redS, Scalars& S,
                                         const KrylovArgs& k, uint32_t& epoch, F&& after) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned full = 0xffffffffu;
  constexpr int QW = 4;   // warps (one per SM sub-partition) that add the threads' values
  double part[K];
#pragma unroll
  for (int kk = 0; kk < K; ++kk) {
    if (kk > 0) block_sync();
    redS[tid] = v[kk];
    block_sync();
    if (warp < QW) {
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < NT / (32 * QW); ++i) s += redS[tid + i * 32 * QW];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
      part[kk] = s;
    }
  }
  if (warp < QW && lane == 0)
#pragma unroll
    for (int kk = 0; kk < K; ++kk) S.part[kk][warp] = part[kk];
  block_sync();
  ++epoch;
  if (warp == 0) {
    const int G = gridDim.x;
    ulonglong2* base = k.slots + (size_t)(epoch & 1u) * 2 * kKrylovMaxGrid;
    if (lane == 0) {
      if constexpr (DATA) asm volatile("fence.acq_rel.gpu;" ::: "memory");
      const bool withheld = k.a.tma_withhold >= 0 && blockIdx.x == 0 &&
                            epoch == (uint32_t)k.a.tma_withhold + 1u;   // test hook
      if (!withheld)
#pragma unroll
        for (int kk = 0; kk < K; ++kk)
          st_slot(base + kk * kKrylovMaxGrid + blockIdx.x,
                  (S.part[kk][0] + S.part[kk][1]) + (S.part[kk][2] + S.part[kk][3]), epoch);
    }
    __syncwarp();
    uint64_t w[kPollLanes][K][2];
    bool all = false;
    for (uint32_t it = 0; it < k.a.wait_limit && !all; ++it) {
      all = true;
#pragma unroll
      for (int q = 0; q < kPollLanes; ++q)
        if (lane + 32 * q < G)
#pragma unroll
          for (int kk = 0; kk < K; ++kk)
            ld_slot(base + kk * kKrylovMaxGrid + lane + 32 * q, w[q][kk][0], w[q][kk][1]);
#pragma unroll
      for (int q = 0; q < kPollLanes; ++q)
        if (lane + 32 * q < G)
#pragma unroll
          for (int kk = 0; kk < K; ++kk)
            all = all && (uint32_t)(w[q][kk][0] >> 32) == epoch && (uint32_t)(w[q][kk][1] >> 32) == epoch;
    }
    const bool ok = __all_sync(full, all);
    if constexpr (DATA) asm volatile("fence.acq_rel.gpu;" ::: "memory");
    if (ok) {
#pragma unroll
      for (int kk = 0; kk < K; ++kk) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < kPollLanes; ++q)
          if (lane + 32 * q < G)
            s += __longlong_as_double((long long)((w[q][kk][0] << 32) |
                                                  (w[q][kk][1] & 0xffffffffull)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
        if (lane == 0) S.tot[kk] = s;
      }
      if (lane == 0) after();
    } else if (lane == 0) {
      S.err = 1;
    }
  }
  block_sync();
  return !S.err;
}

// L2 loads of the column pair (2p, 2p+1) of a row: the vectors are written by
// other SMs during the kernel, so nothing may come from L1.  SELF: the pair is
// one this thread wrote earlier in the kernel.  __ldcg tells the compiler
// nothing about the memory it reads, so it may be moved ahead of a store to the
// same address; these loads name the memory and stay behind it.
template <typename T4>
__device__ __forceinline__ T4 ldl2(const T4* p) {
  static_assert(sizeof(T4) == 16 || sizeof(T4) == 8, "16- or 8-byte loads");
  T4 v;
  if constexpr (sizeof(T4) == 16) {
    uint64_t a, b;
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    reinterpret_cast<uint64_t*>(&v)[0] = a;
    reinterpret_cast<uint64_t*>(&v)[1] = b;
  } else {
    uint64_t a;
    asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    *reinterpret_cast<uint64_t*>(&v) = a;
  }
  return v;
}
template <bool VEC, bool SELF>
__device__ __forceinline__ void ldcg_pair(const float2* row, int p, int dim, float2& v0, float2& v1) {
  if constexpr (VEC) {
    const float4* a = reinterpret_cast<const float4*>(row) + p;
    const float4 f = SELF ? ldl2(a) : __ldcg(a);
    v0.x = f.x; v0.y = f.y; v1.x = f.z; v1.y = f.w;
  } else {
    v0 = SELF ? ldl2(row + 2 * p) : __ldcg(row + 2 * p);
    v1 = make_float2(0.f, 0.f);
    if (2 * p + 1 < dim) v1 = SELF ? ldl2(row + 2 * p + 1) : __ldcg(row + 2 * p + 1);
  }
}

// The off-diagonal part of H x for one item, NR tile rows x 64 columns (two
// columns per lane): acc[r][h] of row r and column 2 p + h (pcl: the pair p,
// clamped to the row).  T_dn over the ELL slots of the tile (two slots per turn,
// words a turn ahead), then T_up row by row with the signed coefficients,
// kUpBatch source rows in flight.
template <bool VEC>
__device__ __forceinline__ void off_diagonal(
    const SectorDev& sd, const float2* tile, int t, int pcl, const float2* x,
    const uint2* const (&list)[NR], const int (&deg)[NR], const float2* coefQ,
    float2 (&acc)[NR][2]) {
  const int lane = threadIdx.x & 31;
  const int dim_dn = sd.dim_dn;
  const int q0 = __ldg(sd.dn_tslot_off + t), q1 = __ldg(sd.dn_tslot_off + t + 1);
  const uint32_t* ellp = TIO::ellp_for(sd.dn_ellp32, sd.dn_ellpr) + lane;
  const uint2* grp2 = reinterpret_cast<const uint2*>(sd.dn_slot_grp);
  float2 s0[NR], s1[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    s0[r] = s1[r] = make_float2(0.f, 0.f);
    acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
  }
  auto flush = [&](uint32_t g) {
    const float2 c = coefQ[2 * g];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      cmac(acc[r][0], c, s0[r]);
      cmac(acc[r][1], c, s1[r]);
      s0[r] = s1[r] = make_float2(0.f, 0.f);
    }
  };
  if (q0 < q1) {
    uint32_t na = __ldg(ellp + (size_t)q0 * 32), nb = __ldg(ellp + (size_t)(q0 + 1) * 32);
    uint2 ng = __ldg(grp2 + (q0 >> 1));
    uint32_t gcur = ng.x;
    for (int q = q0; q < q1; q += 2) {
      const uint32_t ea = na, eb = nb;
      const uint2 gg = ng;
      if (q + 2 < q1) {
        na = __ldg(ellp + (size_t)(q + 2) * 32);
        nb = __ldg(ellp + (size_t)(q + 3) * 32);
        ng = __ldg(grp2 + ((q + 2) >> 1));
      }
      uint32_t oa0, oa1, ob0, ob1;
      float ga0, ga1, gb0, gb1;
      TIO::unpack<float>(ea, oa0, oa1, ga0, ga1);
      TIO::unpack<float>(eb, ob0, ob1, gb0, gb1);
      float2 a0[NR], a1[NR], b0[NR], b1[NR];
      TIO::load_off(tile, oa0, a0);
      TIO::load_off(tile, oa1, a1);
      TIO::load_off(tile, ob0, b0);
      TIO::load_off(tile, ob1, b1);
      if (gg.x != gcur) { flush(gcur); gcur = gg.x; }   // uniform over the warp
#pragma unroll
      for (int r = 0; r < NR; ++r) { cax(s0[r], ga0, a0[r]); cax(s1[r], ga1, a1[r]); }
      if (gg.y != gcur) { flush(gcur); gcur = gg.y; }
#pragma unroll
      for (int r = 0; r < NR; ++r) { cax(s0[r], gb0, b0[r]); cax(s1[r], gb1, b1[r]); }
    }
    flush(gcur);
  }
  constexpr int NB = kUpBatch;
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    float2 sa[2], sb[2];
    sa[0] = sa[1] = sb[0] = sb[1] = make_float2(0.f, 0.f);
    for (int e = 0; e < deg[r]; e += NB) {
      float2 v[NB][2];
      uint32_t cs[NB];
#pragma unroll
      for (int i = 0; i < NB; ++i)
        if (e + i < deg[r]) {   // uniform over the warp
          const uint2 en = list[r][e + i];
          cs[i] = en.y;
          ldcg_pair<VEC, false>(x + en.x, pcl, dim_dn, v[i][0], v[i][1]);
        }
#pragma unroll
      for (int i = 0; i < NB; ++i)
        if (e + i < deg[r]) {
          const float2 c = coefQ[cs[i]];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            sa[h] = ffma2(make_float2(c.x, c.x), v[i][h], sa[h]);
            sb[h] = ffma2(make_float2(c.y, c.y), v[i][h], sb[h]);
          }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      acc[r][h].x += sa[h].x - sb[h].y;
      acc[r][h].y += sa[h].y + sb[h].x;
    }
  }
}

// The a-posteriori check of step j (as k_conv_check), by one warp.
__device__ __noinline__ void conv_check(Scalars& S, int j, double tau, double eps_tol) {
  const int lane = threadIdx.x & 31;
  for (int i = lane; i < 64; i += 32) {
    S.al[i] = i < j ? S.alpha[i + 1] : 0.0;
    S.be[i] = i < j - 1 ? S.beta[i + 1] : 0.0;
  }
  __syncwarp();
  tridiag_expm_e1(S.al, S.be, j, tau, S.yre, S.yim);
  double dn = 0.0, yn = 0.0;
  for (int i = lane; i < j; i += 32) {
    const double pr = i < j - 1 ? S.yprev_re[i] : 0.0, pi = i < j - 1 ? S.yprev_im[i] : 0.0;
    dn += (S.yre[i] - pr) * (S.yre[i] - pr) + (S.yim[i] - pi) * (S.yim[i] - pi);
    yn += S.yre[i] * S.yre[i] + S.yim[i] * S.yim[i];
  }
  for (int o = 16; o > 0; o >>= 1) {
    dn += __shfl_xor_sync(0xffffffffu, dn, o);
    yn += __shfl_xor_sync(0xffffffffu, yn, o);
  }
  __syncwarp();
  for (int i = lane; i < j; i += 32) {
    S.yprev_re[i] = S.yre[i];
    S.yprev_im[i] = S.yim[i];
  }
  if (lane == 0) {
    const double ny = sqrt(yn);
    const double delta = sqrt(dn) / ny;
    const double eps = delta < 1.0 ? fmin(1.0 + ny, delta / (1.0 - delta) * ny) : 1.0 + ny;
    // S.as holds the breakdown scale seen by step j until this pass' alpha
    if (eps < eps_tol || S.beta[j] < eps_tol * S.as) {
      S.conv_delta = delta;
      S.conv = j;
    }
  }
  __syncwarp();
}

// Dynamic shared memory: Scalars, Share, then the arrays of Share.  Every
// function takes its pointers from here, so that the compiler knows them to
// be shared memory (through a generic pointer the gathers of apply_pass ran
// 1.5 x slower).
extern __shared__ __align__(16) unsigned char smem_raw[];

// The CTA's share of the sector: held in registers through the whole kernel
// these would spill.
struct Share {
  SectorDev sd;
  VecDev vd;
  int off_w, off_q, off_l, off_d;   // byte offsets of the arrays below
  int n_groups, max_deg, nloc, ld, npairs, ntile, items, nwork;
};
constexpr int kOffShare = (sizeof(Scalars) + 15) & ~15;
constexpr int kOffX = (kOffShare + sizeof(Share) + 15) & ~15;
__device__ __forceinline__ Scalars& scalars() { return *reinterpret_cast<Scalars*>(smem_raw); }
__device__ __forceinline__ Share& share() { return *reinterpret_cast<Share*>(smem_raw + kOffShare); }
// rows of x_j and w: [tile rows][dim_dn + zero columns][NR]
__device__ __forceinline__ float2* tile_x() { return reinterpret_cast<float2*>(smem_raw + kOffX); }
__device__ __forceinline__ float2* tile_w() { return reinterpret_cast<float2*>(smem_raw + share().off_w); }
// Signed coefficients, 2 n_groups to a row (c_g and -c_g of every group): a row for each sub-step of the launch, then, with energies, one for
// its first time and one for the time after each sub-step.  All of them are
// written before the first grid-wide sum and only read after it, so that no
// pass depends on a hand-over within the launch.
__device__ __forceinline__ const float2* coef_q(int row) {
  return reinterpret_cast<const float2*>(smem_raw + share().off_q) + row * 2 * share().n_groups;
}
// T_up entries [rows][max_deg]: source offset, coefficient slot; their numbers
__device__ __forceinline__ uint2* up_list() { return reinterpret_cast<uint2*>(smem_raw + share().off_l); }
__device__ __forceinline__ int* up_deg() { return reinterpret_cast<int*>(smem_raw + share().off_d); }

// w = s_in H x - s_prev x_prev of the CTA's rows into tileW, H with the
// coefficients of the given row; returns the thread's Re<x, w>.  Inlined in the
// Lanczos loop and in the energies.
template <bool VEC>
__device__ __forceinline__ double apply_pass(const float2* x, const float2* xp, float s_in,
                                             float s_prev, int row) {
  const Scalars& S = scalars();
  const Share& h = share();
  // the loads below must not move up across the grid-wide sum before the
  // pass: they depend on pointers that are opaque from here on
  asm volatile("" : "+l"(x) : : "memory");
  asm volatile("" : "+l"(xp) : : "memory");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int G = gridDim.x, cta = blockIdx.x;
  const SectorDev& sd = h.sd;
  const int dim_dn = sd.dim_dn, npairs = h.npairs, ntile = h.ntile, nloc = h.nloc;
  const int pitch = h.ld * NR;
  const float2* const tileX = tile_x();
  float2* const tileW = tile_w();
  const uint2* const list = up_list();
  const int* const degS = up_deg();
  const float2* const coefQ = coef_q(row);
  double dot = 0.0;
  if (warp >= h.nwork) return dot;
  for (int it = warp; it < h.items; it += h.nwork) {
    const int b = it / ntile, t = it - b * ntile, p = 32 * t + lane;
    const float2* tile = tileX + b * pitch;
    const uint2* lst[NR];
    int deg[NR], urow[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int li = b * NR + r;
      const bool have = li < nloc;
      lst[r] = list + (have ? li : 0) * h.max_deg;
      deg[r] = have ? degS[li] : 0;
      urow[r] = cta + (have ? li : 0) * G;
    }
    float2 acc[NR][2];
    off_diagonal<VEC>(sd, tile, t, min(p, npairs - 1), x, lst, deg, coefQ, acc);
    if (p >= npairs) continue;
    const int d0 = 2 * p;
    const bool has1 = d0 + 1 < dim_dn;
    const uint32_t dw0 = __ldg(sd.dn_word + d0), dw1 = has1 ? __ldg(sd.dn_word + d0 + 1) : 0u;
    float2 xa[NR], xb[NR], oa[NR], ob[NR];
    TIO::load(tile, d0, xa);
    TIO::load(tile, d0 + 1, xb);
    float da = 0.f;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      oa[r] = ob[r] = make_float2(0.f, 0.f);
      if (b * NR + r >= nloc) continue;
      const uint32_t uw = __ldg(sd.up_word + urow[r]);
      float g0 = (float)S.utab[__popc(uw & dw0)], g1 = (float)S.utab[__popc(uw & dw1)];
      if (sd.up_eps) {
        const float eu = (float)__ldg(sd.up_eps + urow[r]);
        g0 += eu + (float)__ldg(sd.dn_eps + d0);
        g1 += eu + (has1 ? (float)__ldg(sd.dn_eps + d0 + 1) : 0.f);
      }
      float2 a0 = acc[r][0], a1 = acc[r][1];
      a0.x += g0 * xa[r].x;
      a0.y += g0 * xa[r].y;
      a1.x += g1 * xb[r].x;
      a1.y += g1 * xb[r].y;
      float2 o0, o1;
      if (xp) {
        float2 p0, p1;
        ldcg_pair<VEC, false>(xp + (size_t)urow[r] * dim_dn, p, dim_dn, p0, p1);
        o0.x = s_in * a0.x - s_prev * p0.x;
        o0.y = s_in * a0.y - s_prev * p0.y;
        o1.x = s_in * a1.x - s_prev * p1.x;
        o1.y = s_in * a1.y - s_prev * p1.y;
      } else {
        o0.x = s_in * a0.x; o0.y = s_in * a0.y;
        o1.x = s_in * a1.x; o1.y = s_in * a1.y;
      }
      oa[r] = o0;
      ob[r] = o1;
      da += xa[r].x * o0.x + xa[r].y * o0.y;
      if (has1) da += xb[r].x * o1.x + xb[r].y * o1.y;
    }
    TIO::store(tileW + b * pitch, d0, oa);
    if (has1) TIO::store(tileW + b * pitch, d0 + 1, ob);
    dot += (double)da;
  }
  return dot;
}

template <bool VEC>
__global__ void __launch_bounds__(NT, 1) k_krylov(KrylovArgs k) {
  constexpr int NW = NT / 32;
  Scalars& S = scalars();
  Share& h = share();
  __shared__ double redS[NT];
  __shared__ float2 cf[kMaxKrylov + 1];
  __shared__ float2 cf_lo;

  const BatchArgs& a = k.a;
  if (threadIdx.x == 0) {
    h.vd = a.vec[0];
    h.sd = a.sec[a.vec[0].sector];
  }
  block_sync();
  const SectorDev& sd = h.sd;
  const VecDev& vd = h.vd;
  LanczosState* st = a.st;
  const int dim_up = sd.dim_up, dim_dn = sd.dim_dn;
  const int npairs = (dim_dn + 1) >> 1, ntile = (dim_dn + 63) >> 6;
  const int G = gridDim.x, cta = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nloc = (dim_up - cta + G - 1) / G;   // rows cta, cta + G, ..
  const int nblk = (nloc + NR - 1) / NR;         // tile rows of NR rows
  const int ld = dim_dn + kZeroCols;
  const int RB = (k.rows + NR - 1) / NR;
  const int tile_bytes = RB * ld * 16;
  const int off_q = kOffX + 2 * tile_bytes;
  const int n_coef = 2 * a.n_groups;   // to a row
  const int off_l = off_q + krylov_coef_rows(k.n_steps, k.energy) * n_coef * (int)sizeof(float2);
  float2* const tileX = tile_x();
  float2* const tileW = reinterpret_cast<float2*>(smem_raw + kOffX + tile_bytes);
  float2* const coefQ = reinterpret_cast<float2*>(smem_raw + off_q);
  uint2* const list = reinterpret_cast<uint2*>(smem_raw + off_l);
  int* const degS = reinterpret_cast<int*>(list + (size_t)k.rows * k.max_deg);
  float2* x1 = static_cast<float2*>(vd.x1);
  float2* V = static_cast<float2*>(vd.V);
  const int m = st->m;
  const double eps_tol = st->eps_tol;
  const int items = nblk * ntile;
  // with the adaptive exit the last warp runs the checks beside the passes
  const int nwork = eps_tol > 0.0 ? NW - 1 : NW;

  // ---- once per launch: connection lists and rows of the CTA
  for (int li = 0; li < nloc; ++li) {
    const int u = cta + li * G;
    const int e0 = __ldg(sd.up_off + u), ne = __ldg(sd.up_off + u + 1) - e0;
    for (int i = tid; i < ne; i += NT) {
      const uint32_t en = __ldg(sd.up_ent + e0 + i);
      const uint32_t g = (en >> kEntGroupShift) & 0xFFu;
      list[(size_t)li * k.max_deg + i] =
          make_uint2((en & kEntRankMask) * (uint32_t)dim_dn, 2u * g + (en >> 31));
    }
    if (tid == 0) degS[li] = ne;
  }
  for (int i = tid; i < RB * ld; i += NT) {
    const int b = i / ld, d = i - b * ld;
    float2 v[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int li = b * NR + r;
      v[r] = li < nloc && d < dim_dn ? ldl2(x1 + (size_t)(cta + li * G) * dim_dn + d) : make_float2(0.f, 0.f);
    }
    TIO::store(tileX + (size_t)b * ld * NR, d, v);
    float2 z[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) z[r] = make_float2(0.f, 0.f);
    TIO::store(tileW + (size_t)b * ld * NR, d, z);
  }
  if (tid == 0) {
    h.off_w = kOffX + tile_bytes;
    h.off_q = off_q;
    h.n_groups = a.n_groups;
    h.off_l = off_l;
    h.off_d = off_l + k.rows * k.max_deg * (int)sizeof(uint2);
    h.max_deg = k.max_deg;
    h.nloc = nloc;
    h.ld = ld;
    h.npairs = npairs;
    h.ntile = ntile;
    h.items = items;
    h.nwork = nwork;
    S.err = 0;
    S.status = 0;
    S.step = st->step;
  }
  for (int i = tid; i <= kMaxSites; i += NT) S.utab[i] = a.U * (double)i;
  block_sync();
  uint32_t epoch = 0;
  const int step0 = S.step;

  for (int i = tid; i < krylov_coef_rows(k.n_steps, k.energy) * n_coef; i += NT) {
    const int row = i / n_coef, slot = i - row * n_coef;
    const bool obs = row >= k.n_steps;
    const float2 c = reinterpret_cast<const float2*>(
        obs ? a.coefs_obs : a.coefs)[(size_t)(step0 + row - (obs ? k.n_steps : 0)) * a.n_groups +
                                     (slot >> 1)];
    const float sg = (slot & 1) ? -1.f : 1.f;
    coefQ[i] = make_float2(sg * c.x, sg * c.y);
  }
  block_sync();
  // one pass over the items: f(tile row, column tile, column pair)
  auto for_items = [&](auto&& f) {
    for (int it = warp; it < items; it += nwork) {
      if (warp >= nwork) break;
      const int b = it / ntile, t = it - b * ntile;
      f(b, t, 32 * t + lane);
    }
  };
  // psi -> per-thread |psi|^2 and sum of double occupancies of tile values
  auto weigh = [&](int b, int p, const float2 (&va)[NR], const float2 (&vb)[NR], double& n2, double& dd) {
    const int d0 = 2 * p;
    const bool has1 = d0 + 1 < dim_dn;
    const uint32_t dw0 = __ldg(sd.dn_word + d0), dw1 = has1 ? __ldg(sd.dn_word + d0 + 1) : 0u;
    float nl = 0.f, wl = 0.f;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (b * NR + r >= nloc) continue;
      const uint32_t uw = __ldg(sd.up_word + cta + (b * NR + r) * G);
      const float qa = va[r].x * va[r].x + va[r].y * va[r].y;
      const float qb = has1 ? vb[r].x * vb[r].x + vb[r].y * vb[r].y : 0.f;
      nl += qa + qb;
      wl += (float)__popc(uw & dw0) * qa + (float)__popc(uw & dw1) * qb;
    }
    n2 += (double)nl;
    dd += (double)wl;
  };
  // outputs and scalars of a state with |psi|^2 = tot[0], in thread 0
  auto new_state = [&](int slot) {
    const double n2 = S.tot[0];
    const double b0 = sqrt(n2);
    S.beta0 = b0;
    S.inv[1] = b0 > 0.0 ? 1.0 / b0 : 0.0;
    S.scale = 1.0;
    S.m_eff = m;
    S.conv = 0;
    S.stop = b0 > 0.0 && isfinite(b0) ? 0 : 1;
    if (!isfinite(b0)) S.status = kErrNumeric;
    if (cta == 0) {
      if (vd.out_docc) vd.out_docc[slot] = S.tot[1] / a.Ns;
      if (vd.out_norm2) vd.out_norm2[slot] = n2;
    }
  };
  auto energy = [&](int slot) -> bool {
    const double v[1] = {apply_pass<VEC>(x1, nullptr, 1.f, 0.f, k.n_steps + slot - step0)};
    return grid_sum<1, false>(v, redS, S, k, epoch, [&]() {
      if (cta == 0 && vd.out_energy) vd.out_energy[slot] = S.tot[0] / a.Ns;
    });
  };
  // profile mode: time of the phase that ends here, by kernel kind (CTA 0)
  uint64_t last = 0;
  auto mark = [&](int kind) {
    if (k.prof && cta == 0 && tid == 0) {
      uint64_t now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (kind >= 0) {
        k.prof[2 * kind] += now - last;
        k.prof[2 * kind + 1] += 1;
      }
      last = now;
    }
  };
  auto finish = [&]() {
    if (tid == 0 && S.err) st->status = kErrTimeout;
    if (tid == 0 && cta == 0 && !S.err) {
      if (S.status) st->status = S.status;
      st->step = S.step;
      st->m_eff = S.m_eff;
    }
  };

  // ---- observables of the state at the launch's first time
  {
    double v[2] = {0.0, 0.0};
    for_items([&](int b, int t, int p) {
      if (p >= npairs) return;
      float2 xa[NR], xb[NR];
      TIO::load(tileX + (size_t)b * ld * NR, 2 * p, xa);
      TIO::load(tileX + (size_t)b * ld * NR, 2 * p + 1, xb);
      weigh(b, p, xa, xb, v[0], v[1]);
    });
    if (!grid_sum<2, true>(v, redS, S, k, epoch, [&]() { new_state(step0); })) { finish(); return; }
    if (k.energy && step0 == 0 && !energy(0)) { finish(); return; }
  }

  for (int s = 0; s < k.n_steps; ++s) {
    mark(-1);
    // ---- Lanczos recursion
    for (int j = 1; j <= m && !S.stop; ++j) {
      const float2* x = j == 1 ? x1 : V + (size_t)(j - 2) * vd.D;
      const float2* xp = j < 2 ? nullptr : j == 2 ? x1 : V + (size_t)(j - 3) * vd.D;
      const float s_in = (float)S.inv[j];
      const float s_prev = j >= 2 ? (float)(S.beta[j - 1] * S.inv[j - 1]) : 0.f;
      if (warp >= nwork && j >= 2) conv_check(S, j - 1, a.tau, eps_tol);
      const double v[1] = {apply_pass<VEC>(x, xp, s_in, s_prev, s)};
      if (!grid_sum<1, false>(v, redS, S, k, epoch, [&]() {
            const double re = S.tot[0];
            S.alpha[j] = re * S.inv[j];
            S.as = S.alpha[j] * S.inv[j];
            if (!isfinite(re)) {
              S.status = kErrNumeric;
              S.stop = 1;
              S.m_eff = j > 1 ? j - 1 : 1;
            } else if (S.conv > 0) {
              S.stop = 1;
              S.m_eff = S.conv;
            }
          })) { finish(); return; }
      mark(KK_APPLY);
      if (S.stop || j == m) break;
      // x_{j+1} = w - alpha_j s_j x_j, into the tile and V
      const float as = (float)S.as;
      float2* xn = V + (size_t)(j - 1) * vd.D;
      double nrm[1] = {0.0};
      for_items([&](int b, int t, int p) {
        if (p >= npairs) return;
        const int d0 = 2 * p;
        const bool has1 = d0 + 1 < dim_dn;
        float2* tx = tileX + (size_t)b * ld * NR;
        float2 xa[NR], xb[NR], wa[NR], wb[NR];
        TIO::load(tx, d0, xa);
        TIO::load(tx, d0 + 1, xb);
        TIO::load(tileW + (size_t)b * ld * NR, d0, wa);
        TIO::load(tileW + (size_t)b * ld * NR, d0 + 1, wb);
        float nl = 0.f;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          float2 o0, o1;
          o0.x = wa[r].x - as * xa[r].x;
          o0.y = wa[r].y - as * xa[r].y;
          o1.x = has1 ? wb[r].x - as * xb[r].x : 0.f;
          o1.y = has1 ? wb[r].y - as * xb[r].y : 0.f;
          xa[r] = o0;
          xb[r] = o1;
          if (b * NR + r < nloc) {
            store_pair<float2, VEC>(xn + (size_t)(cta + (b * NR + r) * G) * dim_dn, p, dim_dn, o0, o1);
            nl += o0.x * o0.x + o0.y * o0.y + o1.x * o1.x + o1.y * o1.y;
          }
        }
        TIO::store(tx, d0, xa);
        if (has1) TIO::store(tx, d0 + 1, xb);
        nrm[0] += (double)nl;
      });
      if (!grid_sum<1, true>(nrm, redS, S, k, epoch, [&]() {
            const double beta = sqrt(S.tot[0]);
            const double sc = fmax(S.scale, fabs(S.alpha[j]));
            S.beta[j] = beta;
            S.as = sc;   // read by the check of step j
            if (!isfinite(beta)) {
              S.status = kErrNumeric;
              S.stop = 1;
              S.m_eff = j;
            } else if (beta <= a.break_tol * sc) {
              S.stop = 1;
              S.m_eff = j;
            } else {
              S.inv[j + 1] = 1.0 / beta;
              S.scale = fmax(sc, beta);
            }
          })) { finish(); return; }
      mark(KK_UPDATE);
    }
    // ---- the small exponential (by every CTA alike)
    const int n = S.m_eff;
    const bool zero = !(S.beta0 > 0.0 && isfinite(S.beta0));
    if (S.conv > 0 && S.conv == n && !zero) {   // y^(n) and delta are the check's
      for (int i = tid; i < n; i += NT) { S.yre[i] = S.yprev_re[i]; S.yim[i] = S.yprev_im[i]; }
      block_sync();
    } else {
      for (int i = tid; i < 64; i += NT) {
        S.al[i] = i < n && !zero ? S.alpha[i + 1] : 0.0;
        S.be[i] = i < n - 1 && !zero ? S.beta[i + 1] : 0.0;
      }
      block_sync();
      if (warp == 0) tridiag_expm_e1(S.al, S.be, n, a.tau, S.yre, S.yim);
      else if (warp == 1 && n > 1)
        tridiag_expm_e1(S.al, S.be, n - 1, a.tau, S.yprev_re, S.yprev_im);
      block_sync();
      if (warp == 1) {
        double dn = 0.0, yn = 0.0;
        if (n > 1)
          for (int i = lane; i < n; i += 32) {
            const double pr = i < n - 1 ? S.yprev_re[i] : 0.0, pi = i < n - 1 ? S.yprev_im[i] : 0.0;
            dn += (S.yre[i] - pr) * (S.yre[i] - pr) + (S.yim[i] - pi) * (S.yim[i] - pi);
            yn += S.yre[i] * S.yre[i] + S.yim[i] * S.yim[i];
          }
        for (int o = 16; o > 0; o >>= 1) {
          dn += __shfl_xor_sync(0xffffffffu, dn, o);
          yn += __shfl_xor_sync(0xffffffffu, yn, o);
        }
        if (lane == 0) S.conv_delta = n > 1 ? sqrt(dn / yn) : 0.0;
      }
    }
    if (warp == 0)
      for (int i = lane; i < n; i += 32) {
        // (a norm that is not finite goes on into the state, as in k_expm)
        const double f = S.beta0 * S.inv[i + 1];
        const double re = f * S.yre[i], im = f * S.yim[i];
        cf[i].x = (float)re;
        cf[i].y = (float)im;
        if (i == 0) {
          cf_lo.x = (float)(re - (double)(float)re);
          cf_lo.y = (float)(im - (double)(float)im);
        }
      }
    block_sync();
    if (tid == 0 && cta == 0) {
      if (vd.out_delta) vd.out_delta[S.step] = S.conv_delta;
      if (vd.out_meff) vd.out_meff[S.step] = n;
    }
    mark(KK_EXPM);
    // ---- psi = sum_j c_j x_j (the order of k_combine), observables fused
    double v[2] = {0.0, 0.0};
    const int nv = zero ? 1 : n;
    for_items([&](int b, int t, int p) {
      if (p >= npairs) return;
      const int d0 = 2 * p;
      const bool has1 = d0 + 1 < dim_dn;
      float2 pa[NR], pb[NR];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        pa[r] = pb[r] = make_float2(0.f, 0.f);
        if (b * NR + r >= nloc) continue;
        const size_t off = (size_t)(cta + (b * NR + r) * G) * dim_dn;
        float2 x0, x1v;
        ldcg_pair<VEC, true>(x1 + off, p, dim_dn, x0, x1v);
        float2 o0 = make_float2(0.f, 0.f), o1 = make_float2(0.f, 0.f);
        cmac(o0, cf_lo, x0);
        cmac(o1, cf_lo, x1v);
        const float2* Vr = V + off;
#pragma unroll 8
        for (int jj = 1; jj < nv; ++jj) {
          float2 y0, y1;
          ldcg_pair<VEC, true>(Vr + (size_t)(jj - 1) * vd.D, p, dim_dn, y0, y1);
          cmac(o0, cf[jj], y0);
          cmac(o1, cf[jj], y1);
        }
        cmac(o0, cf[0], x0);
        cmac(o1, cf[0], x1v);
        store_pair<float2, VEC>(x1 + off, p, dim_dn, o0, o1);
        pa[r] = o0;
        pb[r] = o1;
      }
      TIO::store(tileX + (size_t)b * ld * NR, d0, pa);
      if (has1) TIO::store(tileX + (size_t)b * ld * NR, d0 + 1, pb);
      weigh(b, p, pa, pb, v[0], v[1]);
    });
    if (!grid_sum<2, true>(v, redS, S, k, epoch, [&]() {
          S.step = S.step + 1;
          new_state(S.step);
        })) { finish(); return; }
    mark(KK_COMBINE);
    if (k.energy) {
      if (!energy(S.step)) { finish(); return; }
      mark(KK_ENERGY);
    }
  }
  finish();
}

}  // namespace

size_t krylov_smem(int rows, int dim_dn, int max_deg, int n_groups, int coef_rows) {
  const size_t rb = (rows + NR - 1) / NR;
  return kOffX + 2 * rb * (size_t)(dim_dn + kZeroCols) * 16 +
         (size_t)coef_rows * 2 * n_groups * 8 + (size_t)rows * max_deg * 8 + (size_t)rows * 4;
}

int krylov_carveout(size_t smem) {
  constexpr int kKiB[] = {8, 16, 32, 64, 100, 132, 164, 196, 228};
  constexpr size_t own = NT * sizeof(double) + (kMaxKrylov + 2) * sizeof(float2) + 1024;
  for (int c : kKiB)
    if (smem + own <= (size_t)c * 1024) return c;
  return 228;
}

template <bool VEC>
static cudaError_t prepare_t(size_t smem, int* ctas) {
  *ctas = 0;
  const cudaError_t e = allow_smem(k_krylov<VEC>, smem);
  if (e == cudaErrorInvalidValue) return cudaSuccess;   // too large
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, k_krylov<VEC>, NT, smem);
}

cudaError_t krylov_prepare(bool vec, size_t smem, int* ctas_per_sm) {
  return vec ? prepare_t<true>(smem, ctas_per_sm) : prepare_t<false>(smem, ctas_per_sm);
}

cudaError_t launch_krylov(bool vec, const KrylovArgs& k, int grid, size_t smem,
                          cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(k.slots, 0, kKrylovSlotBytes, s);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<KrylovArgs*>(&k)};
  const void* f = vec ? (const void*)k_krylov<true> : (const void*)k_krylov<false>;
  return cudaLaunchCooperativeKernel(f, dim3(grid), dim3(NT), args, smem, s);
}

}  // namespace ed
