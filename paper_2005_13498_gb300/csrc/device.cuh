// Device helpers shared by the kernel translation units: complex arithmetic,
// block reductions, the shared-memory tile layout and the tridiagonal
// exponential.
#pragma once

#include "kernels.cuh"

namespace ed {

// ---------------------------------------------------------------- host side
// Lets `kernel` be launched with smem bytes of dynamic shared memory.  The
// limit belongs to the function, for every context and thread of the process,
// so it only ever takes one value, the most the device gives a block beside
// the kernel's static arrays: set to what one sector needs, it would refuse
// the launches another context was prepared for.
template <typename K>
inline cudaError_t allow_smem(K* kernel, size_t smem) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  const int64_t most = 227 * 1024 - (int64_t)fa.sharedSizeBytes;
  if ((int64_t)smem > most) return cudaErrorInvalidValue;
  if (fa.maxDynamicSharedSizeBytes >= most) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// ---------------------------------------------------------------- utilities
template <typename R> struct C2T;
template <> struct C2T<float> { using T = float2; };
template <> struct C2T<double> { using T = double2; };

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }

// Two independent round-to-nearest FP32 FMAs in one packed instruction
// (fma.rn.f32x2, sm_100 and later): (a.x b.x + c.x, a.y b.y + c.y), the same
// values as two scalar FMAs.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long ra, rb, rc, rd;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rc) : "f"(c.x), "f"(c.y));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(ra), "l"(rb), "l"(rc));
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
  return d;
}
// s += g v (complex s, v; real g)
template <typename C, typename R>
__device__ __forceinline__ void cax(C& s, R g, const C& v) {
  if constexpr (sizeof(R) == 4) {
    s = ffma2(make_float2(g, g), v, s);
  } else {
    s.x += g * v.x;
    s.y += g * v.y;
  }
}
// acc += c s (complex), each component a chain of two fused multiply-adds
// into acc: no product is rounded on its own (two FMAs per component, where
// acc + (a b - c d) takes a multiply, an FMA and an add)
template <typename C>
__device__ __forceinline__ void cmac(C& acc, const C c, const C s) {
  if constexpr (sizeof(C) == 8) {
    acc = ffma2(make_float2(c.x, c.x), s, acc);
    acc = ffma2(make_float2(-c.y, c.y), make_float2(s.y, s.x), acc);
  } else {
    acc.x = __fma_rn(-c.y, s.y, __fma_rn(c.x, s.x, acc.x));
    acc.y = __fma_rn(c.y, s.x, __fma_rn(c.x, s.y, acc.y));
  }
}
// the same for the two complex64 values of a 16-byte word
__device__ __forceinline__ void cmac4(float4& acc, const float2 c, const float4 s) {
  float2 a = make_float2(acc.x, acc.y), b = make_float2(acc.z, acc.w);
  cmac(a, c, make_float2(s.x, s.y));
  cmac(b, c, make_float2(s.z, s.w));
  acc = make_float4(a.x, a.y, b.x, b.y);
}

template <typename R> __device__ __forceinline__ typename C2T<R>::T
load_coef(const void* p, int idx) {
  return reinterpret_cast<const typename C2T<R>::T*>(p)[idx];
}

// Block reduction of K doubles; the result is valid in thread 0.
template <int K>
__device__ __forceinline__ void block_reduce(double (&v)[K], double* red) {
  const unsigned full = 0xffffffffu;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(full, v[k], o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[wid * K + k] = v[k];
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      v[k] = lane < nw ? red[lane * K + k] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(full, v[k], o);
    }
  }
}

// Write this block's partials; the last block of [b0, b1) sums all partials
// in block order.  Returns true in every thread of the last block; the totals
// are valid in thread 0.
template <int K>
__device__ __forceinline__ bool reduce_last_block(double (&v)[K], int blk, int b0,
                                                  int b1, double* partials,
                                                  unsigned* counter,
                                                  double* red, int* flag) {
  block_reduce<K>(v, red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) partials[(size_t)blk * K + k] = v[k];
    __threadfence();
    unsigned ticket = atomicAdd(counter, 1u);
    *flag = (ticket == (unsigned)(b1 - b0 - 1));
  }
  __syncthreads();
  if (!*flag) return false;
  __threadfence();
  double acc[K];
#pragma unroll
  for (int k = 0; k < K; ++k) acc[k] = 0.0;
  for (int b = b0 + threadIdx.x; b < b1; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] += __ldcg(&partials[(size_t)b * K + k]);
  block_reduce<K>(acc, red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = acc[k];
    *counter = 0u;
  }
  return true;
}

// Column pair (2p, 2p+1) of a row: one 16-byte access for aligned complex64
// rows (VEC), else two element accesses with the second column checked.
// STREAM: data read or written once in this pass (the previous Krylov vector,
// the output w): evict-first cache hints, so that the vector whose rows are
// gathered stays in L2.
template <typename C, bool VEC, bool STREAM = false>
__device__ __forceinline__ void load_pair(const C* row, int p, int dim, C& v0, C& v1) {
  if constexpr (VEC) {
    const float4* a = reinterpret_cast<const float4*>(row) + p;
    const float4 f = STREAM ? __ldcs(a) : *a;
    v0.x = f.x; v0.y = f.y; v1.x = f.z; v1.y = f.w;
  } else {
    const int d = 2 * p;
    v0 = STREAM ? __ldcs(row + d) : row[d];
    if (d + 1 < dim) v1 = STREAM ? __ldcs(row + d + 1) : row[d + 1]; else v1 = czero<C>();
  }
}
template <typename C, bool VEC, bool STREAM = false>
__device__ __forceinline__ void store_pair(C* row, int p, int dim, C v0, C v1) {
  if constexpr (VEC) {
    float4* a = reinterpret_cast<float4*>(row) + p;
    const float4 f = make_float4(v0.x, v0.y, v1.x, v1.y);
    if (STREAM) __stcs(a, f); else *a = f;
  } else {
    const int d = 2 * p;
    if (STREAM) __stcs(row + d, v0); else row[d] = v0;
    if (d + 1 < dim) { if (STREAM) __stcs(row + d + 1, v1); else row[d + 1] = v1; }
  }
}

template <typename R>
__device__ __forceinline__ R sign_of(uint32_t ent) {
  // +1 or -1 from bit 31
  if constexpr (sizeof(R) == 4) return __int_as_float((int)((ent & 0x80000000u) | 0x3f800000u));
  else return (ent & 0x80000000u) ? -1.0 : 1.0;
}

// Shared-memory tile of NR rows, stored column by column.  When the NR values
// of a column fill two 16-byte chunks (complex64 x 4 rows, complex128 x 2
// rows) the two chunks of column d are swapped for d mod 8 >= 4, so that the
// chunk a lane reads for a random column lands in any of the eight 16-byte
// bank groups (bank conflicts of random column gathers drop by about half).
template <typename C, int NR>
struct TileIO {
  static constexpr int kBytes = NR * (int)sizeof(C);
  __device__ static __forceinline__ void load(const C* tile, int d, C (&v)[NR]) {
    if constexpr (kBytes == 32) {
      const float4* t = reinterpret_cast<const float4*>(tile);
      const int sw = (d >> 2) & 1;
      const float4 a = t[2 * d + sw], b = t[2 * d + (sw ^ 1)];
      if constexpr (sizeof(C) == 8) {
        v[0].x = a.x; v[0].y = a.y; v[1].x = a.z; v[1].y = a.w;
        v[2].x = b.x; v[2].y = b.y; v[3].x = b.z; v[3].y = b.w;
      } else {
        v[0] = *reinterpret_cast<const C*>(&a);
        v[1] = *reinterpret_cast<const C*>(&b);
      }
    } else if constexpr (kBytes == 16) {
      const float4 a = reinterpret_cast<const float4*>(tile)[d];
      v[0] = *reinterpret_cast<const C*>(&a);
      if constexpr (NR == 2) v[1] = *(reinterpret_cast<const C*>(&a) + 1);
    } else {
#pragma unroll
      for (int r = 0; r < NR; ++r) v[r] = tile[(size_t)d * NR + r];
    }
  }
  // load by a table entry: the byte offset of the column (of its first
  // chunk, tile_offset, for 32-byte columns) from the ELL copy of this
  // column width (ell_for)
  __device__ static __forceinline__ void load_ent(const C* tile, uint32_t ent, C (&v)[NR]) {
    const uint32_t off = ent & 0x7FFFFFFFu;
    if constexpr (kBytes == 32) {
      const char* base = reinterpret_cast<const char*>(tile);
      const float4 a = *reinterpret_cast<const float4*>(base + off);
      const float4 b = *reinterpret_cast<const float4*>(base + (off ^ 16u));
      if constexpr (sizeof(C) == 8) {
        v[0].x = a.x; v[0].y = a.y; v[1].x = a.z; v[1].y = a.w;
        v[2].x = b.x; v[2].y = b.y; v[3].x = b.z; v[3].y = b.w;
      } else {
        v[0].x = __longlong_as_double(((long long)__float_as_int(a.y) << 32) | (unsigned)__float_as_int(a.x));
        v[0].y = __longlong_as_double(((long long)__float_as_int(a.w) << 32) | (unsigned)__float_as_int(a.z));
        v[1].x = __longlong_as_double(((long long)__float_as_int(b.y) << 32) | (unsigned)__float_as_int(b.x));
        v[1].y = __longlong_as_double(((long long)__float_as_int(b.w) << 32) | (unsigned)__float_as_int(b.z));
      }
    } else if constexpr (kBytes == 16) {
      const float4 a = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(tile) + off);
      if constexpr (sizeof(C) == 8) {
        v[0].x = a.x; v[0].y = a.y; v[1].x = a.z; v[1].y = a.w;
      } else {
        v[0].x = __longlong_as_double(((long long)__float_as_int(a.y) << 32) | (unsigned)__float_as_int(a.x));
        v[0].y = __longlong_as_double(((long long)__float_as_int(a.w) << 32) | (unsigned)__float_as_int(a.z));
      }
    } else if constexpr (kBytes == 8) {
      v[0] = *reinterpret_cast<const C*>(reinterpret_cast<const char*>(tile) + off);
    } else {
      load(tile, (int)(off >> 5), v);
    }
  }
  // load by a byte offset: of the column (of its first chunk for 32-byte
  // columns, whose second chunk is at offset ^ 16)
  __device__ static __forceinline__ void load_off(const C* tile, uint32_t off, C (&v)[NR]) {
    load_ent(tile, off, v);
  }
  // packed ELL word of one lane and slot: bits 0-14 the column unit of the
  // lane's first column's entry, bit 15 the sign of the second, bits 16-30
  // the unit of the second, bit 31 the sign of the first; a unit is 8 bytes
  // for 8-byte columns and 16 bytes otherwise (only 8-, 16- and 32-byte
  // columns occur in the configuration table)
  static_assert(kBytes == 8 || kBytes == 16 || kBytes == 32, "packed ELL column widths");
  static constexpr int kUnitShift = kBytes == 8 ? 3 : 4;
  template <typename R>
  __device__ static __forceinline__ void unpack(uint32_t e, uint32_t& off0, uint32_t& off1,
                                                R& g0, R& g1) {
    off0 = (e & 0x7FFFu) << kUnitShift;
    off1 = ((e >> 16) & 0x7FFFu) << kUnitShift;
    g0 = sign_of<R>(e);
    g1 = sign_of<R>(e << 16);
  }
  __device__ static __forceinline__ const uint32_t* ellp_for(const uint32_t* p32,
                                                             const uint32_t* prank) {
    if constexpr (kBytes == 32) return p32;
    else return prank;
  }
  // the ELL copy whose entries hold byte offsets for this column width
  __device__ static __forceinline__ const uint32_t* ell_for(const uint32_t* ell32,
                                                            const uint32_t* ell16,
                                                            const uint32_t* ell8) {
    if constexpr (kBytes == 16) return ell16;
    else if constexpr (kBytes == 8) return ell8;
    else return ell32;
  }
  __device__ static __forceinline__ void store(C* tile, int d, const C (&v)[NR]) {
    if constexpr (kBytes == 32) {
      float4* t = reinterpret_cast<float4*>(tile);
      const int sw = (d >> 2) & 1;
      float4 a, b;
      if constexpr (sizeof(C) == 8) {
        a = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        b = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
      } else {
        a = *reinterpret_cast<const float4*>(&v[0]);
        b = *reinterpret_cast<const float4*>(&v[1]);
      }
      t[2 * d + sw] = a;
      t[2 * d + (sw ^ 1)] = b;
    } else if constexpr (kBytes == 16) {
      float4 a;
      *reinterpret_cast<C*>(&a) = v[0];
      if constexpr (NR == 2) *(reinterpret_cast<C*>(&a) + 1) = v[1];
      reinterpret_cast<float4*>(tile)[d] = a;
    } else {
#pragma unroll
      for (int r = 0; r < NR; ++r) tile[(size_t)d * NR + r] = v[r];
    }
  }
};

// Comparisons of finite float64 values on the integer units (a float64
// comparison takes a slot of the FP64 pipe).
__device__ __forceinline__ bool is_zero(double a) {
  return (__double_as_longlong(a) << 1) == 0;
}
__device__ __forceinline__ bool same(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b) || (is_zero(a) && is_zero(b));
}

// The off-diagonal part of H x for one row of Psi and the 64 columns of ELL
// tile t, complex128: acc[h] of column 2 p + h of the lane's pair p (pcl: p
// clamped to the row).  get(e): entry e < ne of the row's T_up list (source
// row's element offset; group | sign << 31), sorted by group.
//
// FP64-pipe bound (a warp instruction occupies the SM's pipe for 16 cycles),
// so the operations count: T_dn slots and T_up entries of one bond group share
// one signed sum, a group whose coefficient equals the previous one's joins
// its sum (the two directions of a bond that carries no phase; every bond at
// A = 0), and a real coefficient costs half a complex product.  On the 2x7
// ladder that is 75 operations per element where sums and products per group
// and direction took 104: Lanczos pass 1.95 -> 1.55 ms (90 % of the pipe), the
// step 65.6 -> 52.2 ms with the update; 1.51 and 51.0 ms with the Lanczos scale
// in the caller's coefficients.  With the T_up additions and the
// products selected by short conditional blocks the compiler predicated them,
// and switched-off instructions take the pipe's time as well: 1.94 ms.
__device__ __forceinline__ void ldcg2(const double2* row, int p, int dim, double2& v0, double2& v1) {
  v0 = __ldcg(row + 2 * p);
  v1 = czero<double2>();
  if (2 * p + 1 < dim) v1 = __ldcg(row + 2 * p + 1);
}

template <typename Get>
__device__ __forceinline__ void off_diagonal_c128(const SectorDev& sd, const double2* tile, int t,
                                                  int pcl, const double2* x, int ne, Get&& get,
                                                  const double2* coefS, double2 (&acc)[2]) {
  using C = double2;
  using TIO = TileIO<C, 1>;
  const int lane = threadIdx.x & 31;
  const int dim_dn = sd.dim_dn;
  const uint32_t* ellp = TIO::ellp_for(sd.dn_ellp32, sd.dn_ellpr) + lane;
  int q = __ldg(sd.dn_tslot_off + t), e = 0;
  const int q1 = __ldg(sd.dn_tslot_off + t + 1);
  constexpr uint32_t kEnd = 0xFFFFu;
  uint32_t word = 0u, gq = kEnd;
  if (q < q1) { word = __ldg(ellp + (size_t)q * 32); gq = __ldg(sd.dn_slot_grp + q); }
  uint32_t ge = e < ne ? get(e).y & 0xFFu : kEnd;
  C s0 = czero<C>(), s1 = s0, cur = s0;
  acc[0] = acc[1] = s0;
  auto flush = [&]() {
    acc[0].x += cur.x * s0.x; acc[0].y += cur.x * s0.y;
    acc[1].x += cur.x * s1.x; acc[1].y += cur.x * s1.y;
    if (!is_zero(cur.y)) {   // uniform over the block
      acc[0].x -= cur.y * s0.y; acc[0].y += cur.y * s0.x;
      acc[1].x -= cur.y * s1.y; acc[1].y += cur.y * s1.x;
    }
  };
  bool any = false;
  for (;;) {
    const uint32_t g = min(gq, ge);   // uniform over the warp
    if (g == kEnd) break;
    const C c = coefS[g];
    if (!any) {
      cur = c;
      any = true;
    } else if (!(same(c.x, cur.x) && same(c.y, cur.y))) {
      flush();
      s0 = s1 = czero<C>();
      cur = c;
    }
    // the group's first T_up rows load while its T_dn slots are gathered
    constexpr int NB = 4;
    C v[NB][2];
    double sg[NB];
    int nb = 0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      if (nb == i && e + i < ne) {
        const uint2 m = get(e + i);
        if ((m.y & 0xFFu) == g) {
          ldcg2(x + m.x, pcl, dim_dn, v[i][0], v[i][1]);
          sg[i] = (m.y >> 31) ? -1.0 : 1.0;
          nb = i + 1;
        }
      }
    }
    while (gq == g) {
      const uint32_t w = word;
      ++q;
      if (q < q1) { word = __ldg(ellp + (size_t)q * 32); gq = __ldg(sd.dn_slot_grp + q); }
      else gq = kEnd;
      uint32_t o0, o1;
      double g0, g1;
      TIO::unpack<double>(w, o0, o1, g0, g1);
      C a0[1], a1[1];
      TIO::load_off(tile, o0, a0);
      TIO::load_off(tile, o1, a1);
      cax(s0, g0, a0[0]);
      cax(s1, g1, a1[0]);
    }
    // one branch per count: short conditional blocks become predicated
    // instructions, and those take the pipe's time also when switched off
    auto add = [&](int i) {
      cax(s0, sg[i], v[i][0]);
      cax(s1, sg[i], v[i][1]);
    };
    switch (nb) {
      case 1: add(0); break;
      case 2: add(0); add(1); break;
      case 3: add(0); add(1); add(2); break;
      case 4: add(0); add(1); add(2); add(3); break;
      default: break;
    }
    e += nb;
    while (e < ne && (get(e).y & 0xFFu) == g) {
      const uint2 m = get(e);
      C u0, u1;
      ldcg2(x + m.x, pcl, dim_dn, u0, u1);
      const double s = (m.y >> 31) ? -1.0 : 1.0;
      cax(s0, s, u0);
      cax(s1, s, u1);
      ++e;
    }
    ge = e < ne ? get(e).y & 0xFFu : kEnd;
  }
  if (any) flush();
}

// -------------------------------------------------------------------- expm
// 1/k for the Taylor coefficients (evaluated by the compiler)
struct InvK {
  double v[81];
};
constexpr InvK make_inv_k() {
  InvK t{};
  t.v[0] = 0.0;
  for (int k = 1; k <= 80; ++k) t.v[k] = 1.0 / (double)k;
  return t;
}
static __constant__ InvK kInvK = make_inv_k();

// exp(-i tau T) e_1 for the real symmetric tridiagonal T of size n <= 64,
// one warp.  T is shifted by the centre sigma of its Gershgorin interval,
// whose half-width h bounds |T - sigma| (2-norm), and the time step is split
// into nsub pieces with rho = |tau| h / nsub <= 3/2.  Each piece is a Taylor
// series with a term count K fixed up front: the k-th term of a piece has
// norm at most rho^k / k! (the state keeps unit norm), and the terms past K
// sum to less than rho^(K+1) / (K+1)! / (1 - rho / (K+2)) <= 1e-17, below
// rounding; K <= 24 for rho <= 3/2.  The rounding errors of a piece are at
// most e^rho units, no more than those of the 2 rho / 1 pieces of rho = 1/2
// it replaces (e^1.5 = 4.5 against 3 e^0.5 = 4.9).
//
// Bound by the latency of dependent float64 operations (about 50 ns each):
// (-i)^k (T - sigma)^k applied to a real vector alternates between a real and
// an imaginary one, so the first piece, which starts from e_1, is one real
// recurrence, and a later one two independent real ones.  Lane l owns rows l
// and l + 32 in registers, the neighbours' values come by shuffles.
template <int ROWS, int PARTS>
static __device__ __forceinline__ void taylor_piece(const double (&ash)[2], const double (&bl)[2],
                                                    const double (&bu)[2], int K,
                                                    double (&yr)[2], double (&yi)[2]) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double t[PARTS][ROWS];   // part 0: the terms of the real start, 1: of the imaginary one
#pragma unroll
  for (int h = 0; h < ROWS; ++h) {
    t[0][h] = yr[h];
    if constexpr (PARTS == 2) t[1][h] = yi[h];
  }
  for (int k = 1; k <= K; ++k) {
    const double f = kInvK.v[k];
    // (-i)^k: the sign and whether the term of a real start is imaginary
    const double sg = (k & 3) == 1 || (k & 3) == 2 ? -1.0 : 1.0;
#pragma unroll
    for (int q = 0; q < PARTS; ++q) {
      double nt[ROWS];
#pragma unroll
      for (int h = 0; h < ROWS; ++h) {
        double dn = __shfl_up_sync(full, t[q][h], 1), up = __shfl_down_sync(full, t[q][h], 1);
        if constexpr (ROWS == 2) {
          // rows 31 and 32 are neighbours across the two halves
          const double c0 = __shfl_sync(full, t[q][1], 0), c1 = __shfl_sync(full, t[q][0], 31);
          if (h == 0 && lane == 31) up = c0;
          if (h == 1 && lane == 0) dn = c1;
        }
        double v = ash[h] * t[q][h];
        v += bl[h] * dn;
        v += bu[h] * up;
        nt[h] = f * v;
      }
#pragma unroll
      for (int h = 0; h < ROWS; ++h) {
        t[q][h] = nt[h];
        // part 0 adds sg t to (k odd ? im : re); part 1, i times that, adds
        // sg t to (k odd ? -re : im)
        if (q == 0) {
          if (k & 1) yi[h] += sg * nt[h]; else yr[h] += sg * nt[h];
        } else {
          if (k & 1) yr[h] -= sg * nt[h]; else yi[h] += sg * nt[h];
        }
      }
    }
  }
}

static __device__ __noinline__ void tridiag_expm_e1(const double* al, const double* be, int n,
                                                    double tau, double* yre, double* yim) {
  const int lane = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  double lo = 1e300, hi = -1e300;
  for (int i = lane; i < n; i += 32) {
    const double r = (i > 0 ? fabs(be[i - 1]) : 0.0) + (i < n - 1 ? fabs(be[i]) : 0.0);
    lo = fmin(lo, al[i] - r);
    hi = fmax(hi, al[i] + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(full, lo, o));
    hi = fmax(hi, __shfl_xor_sync(full, hi, o));
  }
  const double sigma = 0.5 * (lo + hi), half = 0.5 * (hi - lo);
  int nsub = (int)ceil(fabs(tau) * half / 1.5);
  if (nsub < 1) nsub = 1;
  if (nsub > 4096) nsub = 4096;
  const double ts = tau / nsub;
  // the term count from the bound (uniform over the warp), in float32 with a
  // margin of 10 % for its rounding
  int K = 1;
  {
    const float rho = (float)(fabs(ts) * half);
    float b = rho;   // rho^k / k!, k = 1
    for (int k = 1; k <= 78; ++k) {
      const float nb = b * rho / (float)(k + 1);   // rho^(k+1) / (k+1)!
      K = k;
      if (nb <= 0.9e-17f * (1.0f - rho / (float)(k + 2))) break;
      b = nb;
    }
  }
  // per-lane rows: shifted diagonal and off-diagonals times the piece length
  double ash[2], bl[2], bu[2], yr[2], yi[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    ash[h] = i < n ? ts * (al[i] - sigma) : 0.0;
    bl[h] = (i < n && i > 0) ? ts * be[i - 1] : 0.0;
    bu[h] = (i < n - 1) ? ts * be[i] : 0.0;
    yr[h] = i == 0 ? 1.0 : 0.0;
    yi[h] = 0.0;
  }
  if (n <= 32) {
    taylor_piece<1, 1>(ash, bl, bu, K, yr, yi);
    for (int sub = 1; sub < nsub; ++sub) taylor_piece<1, 2>(ash, bl, bu, K, yr, yi);
  } else {
    taylor_piece<2, 1>(ash, bl, bu, K, yr, yi);
    for (int sub = 1; sub < nsub; ++sub) taylor_piece<2, 2>(ash, bl, bu, K, yr, yi);
  }
  // undo the shift: multiply by exp(-i tau sigma)
  double sn, cs;
  sincos(-tau * sigma, &sn, &cs);
  __syncwarp();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = lane + 32 * h;
    if (i < 64) {
      yre[i] = i < n ? yr[h] * cs - yi[h] * sn : 0.0;
      yim[i] = i < n ? yr[h] * sn + yi[h] * cs : 0.0;
    }
  }
  __syncwarp();
}

}  // namespace ed
