// Multigrid inner solvers of the block-triangular preconditioner (Section 4,
// Eq. hybridPrec; the paper's M_II^(h) uses smoothed aggregation on A_uu and
// an AMG on C~_pi).  Everything here runs on structured lattices:
//
//  * displacement hierarchy: level 0 = A_uu on the Q1 node lattice (27-point
//    3x3-block stencil); smoothed aggregation with 3x3x3 node aggregates,
//    tentative prolongator = indicator x I_3 on free dofs, one damped block-
//    Jacobi smoothing step of the prolongator, Galerkin coarse operators
//    (which stay 27-point block stencils);
//  * interface-pressure hierarchy: level 0 = C~_pi on faces (11-entry ELL
//    rows), faces -> cells by averaging (weight 1/2 per adjacent cell, 1 on
//    a boundary face, 0 on a drained face) giving a 25-point cell stencil,
//    then scalar smoothed aggregation (125-point coarse stencils);
//  * V(1,1) cycles with Chebyshev smoothing preconditioned by the (block)
//    diagonal, exact dense solve on the last level.
//
// Galerkin products are formed in two deterministic gather passes, Q = A P
// on the fine lattice and A_c = P^T Q per coarse point: no atomics, no
// sparse-matrix hashing.
#include "lattice.cuh"
#include "tune.h"
#include "u64.cuh"

#include <type_traits>

#include <algorithm>
#include <cmath>

namespace mhfp {

namespace {

// <hot:k_cheb_u0> (bench.py hashes this region to tell whether profiles/traffic.json still applies)
// Chebyshev step of the finest displacement level in FP64 (the rows, the forms
// and their times: u64.cuh): r = b - A xin, d = cd d + cr D^-1 r, xout = xin + d.
template <U64Form F>
__global__ void __launch_bounds__(u64_threads(F), F == U64_ROW ? 13 : 0)
    k_cheb_u0(Lat32 L, const double* __restrict__ val, const double* __restrict__ dinv, const double* __restrict__ b,
              const double* __restrict__ xin, double* __restrict__ xout, double* __restrict__ d,
              const double* __restrict__ cf, bool first, long long lb) {
  const double cd = cf[0], cr = cf[1];
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  const long long N = L.N;
  const unsigned n = blockIdx.x * u64_nodes(F) + threadIdx.x;
  const bool valid = n < (unsigned)N;
  if (F == U64_NODE) {
    if (!valid) return;
    double acc[3] = {0.0, 0.0, 0.0};
    u64_rows(L, n, val, xin, nullptr, 0.0, acc);
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[a] = b[3LL * n + a] - acc[a];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const long long r = 3LL * n + a;
      double z = 0.0;
#pragma unroll
      for (int t = 0; t < 3; ++t) z += dinv[(3 * a + t) * N + n] * acc[t];
      const double dn = first ? cr * z : cd * d[r] + cr * z;
      d[r] = dn;
      xout[r] = xin[r] + dn;
    }
  } else {
    __shared__ double rs[3][u64_nodes(F)];
    const int comp = threadIdx.y % 3, s = threadIdx.y / 3;
    const long long r = 3LL * n + comp;
    double v = 0.0;
    if (F == U64_SPLIT) v = u64_row_split(L, n, valid, comp, s, val, xin, nullptr, 0.0);
    else if (valid) v = u64_row(L, n, comp, val, xin, nullptr, 0.0);
    if (s == 0) rs[comp][threadIdx.x] = valid ? b[r] - v : 0.0;
    __syncthreads();
    if (!valid || s != 0) return;
    double z = 0.0;
#pragma unroll
    for (int t = 0; t < 3; ++t) z += dinv[(3 * comp + t) * N + n] * rs[t][threadIdx.x];
    const double dn = first ? cr * z : cd * d[r] + cr * z;
    d[r] = dn;
    xout[r] = xin[r] + dn;
  }
}
// </hot:k_cheb_u0>

// <hot:k_cheb_u0_sym> (hashed like the region above)
// The finest displacement level in FP32 with symmetric storage (A_uu is
// symmetric): per node the diagonal 3x3 block (slot 0) and the blocks
// A(n, n + e_o) of the 13 neighbours with stencil index o = 13 + u > 13
// (slots u = 1..13), i.e. the last 14 offsets of the full layout.  The
// lower blocks are read transposed from the neighbour that owns them:
// A(n, n - e_o) = A(n - e_o, n)^T, slot u of node n - e_o.  Each stored
// block is read by its owner and by one neighbour at most a lattice plane
// apart, so the second read hits L2 and HBM carries each value once.
// Node-blocked layout: nodes in blocks of 32; a block holds its 126 rows
// (slot u, entry e: row 9 u + e) of 32 values each, so the rows a warp
// streams are one contiguous 16 KB range (sym_base).
// UNR slots per loop iteration: 2 keeps two slots' loads in flight (the
// 5-blocks-per-SM variant has the registers for it), 1 one slot.
// lanes of p's warp that hold a node (blocks are whole warps of 32 nodes)
__device__ __forceinline__ unsigned sym_lanes(const Lat& L, long long p) {
  const long long left = L.N - (p & ~31LL);
  return left >= 32 ? 0xffffffffu : ((1u << left) - 1u);
}

// Slot 1 is the +x neighbour, so node p's lower block of that slot is the
// own block of node p - 1, the previous lane's: every lane loads its own
// slot-1 block and the lower one arrives by warp shuffle (lane 0 loads it).
// `mask` holds the lanes of the warp with a node (all lanes call this).
template <typename T, int UNR = 1>
__device__ __forceinline__ void sym_residual(const Lat& L, long long p, const T* __restrict__ up,
                                             const T* __restrict__ x, T r[3], unsigned mask) {
  int i, j, k;
  L.ijk(p, i, j, k);
  const T* own = up + sym_base(p);
  {
    const T x0 = x[3 * p], x1 = x[3 * p + 1], x2 = x[3 * p + 2];
#pragma unroll
    for (int a = 0; a < 3; ++a) r[a] -= own[(3 * a) * 32] * x0 + own[(3 * a + 1) * 32] * x1 + own[(3 * a + 2) * 32] * x2;
  }
  {
    T v[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) v[e] = own[(9 + e) * 32];
    if (i + 1 < L.Lx) {
      const long long q = p + 1;
      const T x0 = x[3 * q], x1 = x[3 * q + 1], x2 = x[3 * q + 2];
#pragma unroll
      for (int a = 0; a < 3; ++a) r[a] -= v[3 * a] * x0 + v[3 * a + 1] * x1 + v[3 * a + 2] * x2;
    }
    const bool first = (threadIdx.x & 31) == 0;
    const T* w = up + sym_base(first && i > 0 ? p - 1 : p) + 9 * 32;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T t0 = __shfl_up_sync(mask, v[a], 1), t1 = __shfl_up_sync(mask, v[3 + a], 1),
        t2 = __shfl_up_sync(mask, v[6 + a], 1);
      if (first) {
        t0 = w[a * 32];
        t1 = w[(3 + a) * 32];
        t2 = w[(6 + a) * 32];
      }
      if (i > 0) {
        const long long q = p - 1;
        r[a] -= t0 * x[3 * q] + t1 * x[3 * q + 1] + t2 * x[3 * q + 2];
      }
    }
  }
#pragma unroll UNR
  for (int u = 2; u <= 13; ++u) {
    int dx, dy, dz;
    St<ST_BOX1>::off(13 + u, dx, dy, dz);
    const long long s = dx + (long long)L.Lx * (dy + (long long)L.Ly * dz);
    if (L.in(i + dx, j + dy, k + dz)) {
      const long long q = p + s;
      const T* v = own + u * 9 * 32;
      const T x0 = x[3 * q], x1 = x[3 * q + 1], x2 = x[3 * q + 2];
#pragma unroll
      for (int a = 0; a < 3; ++a) r[a] -= v[(3 * a) * 32] * x0 + v[(3 * a + 1) * 32] * x1 + v[(3 * a + 2) * 32] * x2;
    }
    if (L.in(i - dx, j - dy, k - dz)) {
      const long long q = p - s;
      const T* v = up + sym_base(q) + u * 9 * 32;
      const T x0 = x[3 * q], x1 = x[3 * q + 1], x2 = x[3 * q + 2];
#pragma unroll
      for (int a = 0; a < 3; ++a) r[a] -= v[a * 32] * x0 + v[(3 + a) * 32] * x1 + v[(6 + a) * 32] * x2;
    }
  }
}

// MINB resident blocks per SM: 8 (32 registers) fills the SMs in one wave
// when the level has at most 152 x 2048 nodes; 6 (40 registers) keeps more
// loads in flight per thread on larger levels.  The set-up autotuner picks.
template <typename T, int MINB>
__global__ void __launch_bounds__(256, MINB) k_resid_u0_sym(Lat L, const T* __restrict__ up,
                                                            const T* __restrict__ x, const T* __restrict__ b,
                                                            T* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.N) return;
  T r[3] = {b[3 * p], b[3 * p + 1], b[3 * p + 2]};
  sym_residual<T, (MINB <= 5 ? 2 : 1)>(L, p, up, x, r, sym_lanes(L, p));
#pragma unroll
  for (int a = 0; a < 3; ++a) y[3 * p + a] = r[a];
}

template <typename T, int MINB>
__global__ void __launch_bounds__(256, MINB) k_cheb_u0_sym(Lat L, const T* __restrict__ up,
                                                           const T* __restrict__ dinv, const T* __restrict__ b,
                                                           const T* __restrict__ xin, T* __restrict__ xout,
                                                           T* __restrict__ d, const T* __restrict__ cf, bool first,
                                                           long long lb) {
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.N) return;
  T r[3] = {b[3 * p], b[3 * p + 1], b[3 * p + 2]};
  if (xin) sym_residual<T, (MINB <= 5 ? 2 : 1)>(L, p, up, xin, r, sym_lanes(L, p));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T z = dinv[(3 * a) * L.N + p] * r[0] + dinv[(3 * a + 1) * L.N + p] * r[1] + dinv[(3 * a + 2) * L.N + p] * r[2];
    const T dn = first ? cf[1] * z : cf[0] * d[3 * p + a] + cf[1] * z;
    d[3 * p + a] = dn;
    xout[3 * p + a] = (xin ? xin[3 * p + a] : T(0)) + dn;
  }
}

// </hot:k_cheb_u0_sym>

// <hot:k_cheb_u0_tma> (hashed like the regions above)
// The same FP32 symmetric-storage sweep and residual, fed by bulk copies.
// A persistent CTA takes node blocks of TMA_NB consecutive nodes.  Its
// producer warp streams, for each block, the 14 stored slots u: the 9 rows
// of the nodes' own blocks A(p, p + e_u) and, for u >= 1, the 9 rows of the
// neighbours' blocks A(p - e_u, p) (read transposed).  In the node-blocked
// layout a slot's 9 rows of one 32-node block are 1152 contiguous bytes, one
// cp.async.bulk copy: 8 for the own rows, 8 or 9 for the transposed ones
// (the node range p - s_u starts anywhere); TMA_S slots in flight; a "full"
// mbarrier per slot buffer counts the bytes, an "empty" one the consumer
// warps that are done with it.  The TMA_NW consumer warps
// (one node per lane) never wait for one another: each waits only for its
// data, and loads the next slot's neighbour x before it waits.  The
// products are summed in the order of sym_residual, so results are
// bit-identical to it.  Every mbarrier wait is bounded: after about 2^31
// clocks the warp records MHFP_WAIT_TIMEOUT in *err and stops; the
// producer waits (bounded) for every copy it issued before the CTA exits.
constexpr int TMA_NW = 8;                    // consumer warps
constexpr int TMA_NB = 32 * TMA_NW;          // nodes per node block
constexpr int TMA_S = 3;                     // slot buffers
constexpr int TMA_CH = 9 * 32;               // floats of one slot of one 32-node block
constexpr int TMA_STAGE = (2 * TMA_NW + 1) * TMA_CH;  // floats per stage: 8 own + 9 transposed chunks
constexpr int TMA_THREADS = 32 * (TMA_NW + 1);
constexpr size_t TMA_SMEM = (size_t)TMA_S * TMA_STAGE * sizeof(float) + 2 * TMA_S * sizeof(unsigned long long);
constexpr int MHFP_WAIT_TIMEOUT = 8;

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bulk_to_smem(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait for the phase with the given parity; false on timeout
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
  const long long t0 = clock64();
  while (!mbar_test(bar, parity))
    if (clock64() - t0 > (1LL << 31)) return false;
  return true;
}

struct TmaSweep {
  const float* up;   // symmetric half, node-blocked (+ 8 zeroed blocks)
  const float* dinv; // [9][N]
  const float *b, *xin;
  float *xout, *d;
  const float* cf;   // {cd, cr} (null: the residual)
  bool first;
  int* err;
};

// lattice shift of slot u (node p's stored neighbour is p + shift)
__device__ __forceinline__ int sym_shift(const Lat& L, int u) {
  int dx, dy, dz;
  St<ST_BOX1>::off(13 + u, dx, dy, dz);
  return u == 0 ? 0 : dx + L.Lx * (dy + L.Ly * dz);
}

// issue the copies of stage (node block wb, slot u) into buf: own chunks
// 0..7 (the zeroed padding covers the last node block), then the chunks
// holding nodes p0 - s_u .. p0 - s_u + 255, first chunk index clo =
// (p0 - s_u) >> 5; chunks before node 0 are not copied (never read)
__device__ __forceinline__ void tma_issue(const TmaSweep& a, const Lat& L, int wb, int u, float* buf,
                                          unsigned long long* bar) {
  const long long p0 = (long long)wb * TMA_NB;
  const long long c0 = p0 >> 5;
  const unsigned ch_bytes = TMA_CH * 4;
  long long clo = 0;
  int first = 0, last = -1;
  if (u > 0) {
    const long long q0 = p0 - sym_shift(L, u);
    clo = q0 >> 5;
    last = (int)(((q0 + TMA_NB - 1) >> 5) - clo);
    first = clo < 0 ? (int)(-clo) : 0;
  }
  const int ntr = last >= first ? last - first + 1 : 0;
  mbar_expect_tx(bar, (unsigned)(TMA_NW + ntr) * ch_bytes);
#pragma unroll 1
  for (int w = 0; w < TMA_NW; ++w) bulk_to_smem(buf + w * TMA_CH, a.up + ((c0 + w) * 126 + u * 9) * 32, ch_bytes, bar);
#pragma unroll 1
  for (int m = first; m <= last; ++m)
    bulk_to_smem(buf + (TMA_NW + m) * TMA_CH, a.up + ((clo + m) * 126 + u * 9) * 32, ch_bytes, bar);
}

// x of node pc's neighbours in slot u (+s and -s; 0 outside the lattice)
__device__ __forceinline__ void sym_x(const Lat& L, const float* __restrict__ x, long long pc, int i, int j, int k,
                                      int u, float xp[3], float xm[3]) {
  int dx, dy, dz;
  St<ST_BOX1>::off(13 + u, dx, dy, dz);
  const int su = sym_shift(L, u);
  const bool inp = u == 0 || L.in(i + dx, j + dy, k + dz), inm = u > 0 && L.in(i - dx, j - dy, k - dz);
  const long long qp = inp ? pc + su : pc, qm = inm ? pc - su : pc;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const float vp = x[3 * qp + e], vm = x[3 * qm + e];
    xp[e] = inp ? vp : 0.f;
    xm[e] = inm ? vm : 0.f;
  }
}

template <bool CHEB>
__global__ void __launch_bounds__(TMA_THREADS, 3) k_sym_tma(Lat L, TmaSweep a0, long long lb) {
  // lane blockIdx.z's vectors (the matrix rows are shared)
  TmaSweep a = a0;
  a.b = lane_ptr(a.b, lb);
  a.xin = lane_ptr(a.xin, lb);
  a.xout = lane_ptr(a.xout, lb);
  a.d = lane_ptr(a.d, lb);
  extern __shared__ __align__(128) unsigned char tma_smem[];
  float* stage = (float*)tma_smem;
  unsigned long long* full = (unsigned long long*)(tma_smem + (size_t)TMA_S * TMA_STAGE * sizeof(float));
  unsigned long long* empty = full + TMA_S;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nblocks = (int)((L.N + TMA_NB - 1) / TMA_NB);
  const int my = (nblocks - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;  // node blocks of this CTA
  const int units = my * 14;
  if (threadIdx.x == 0) {
    for (int s = 0; s < TMA_S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], TMA_NW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == TMA_NW) {
    // producer: lane 0 issues every unit once its buffer is free
    if (lane == 0) {
      bool ok = true;
      int g = 0;
      for (; g < units && ok; ++g) {
        const int buf = g % TMA_S;
        if (g >= TMA_S) ok = mbar_wait(&empty[buf], (unsigned)(g / TMA_S - 1) & 1u);
        if (!ok) break;
        tma_issue(a, L, (int)blockIdx.x + (g / 14) * (int)gridDim.x, g % 14, stage + (size_t)buf * TMA_STAGE,
                  &full[buf]);
      }
      // every issued copy lands before the CTA may exit
      for (int h = (g > TMA_S ? g - TMA_S : 0); h < g; ++h)
        if (!mbar_wait(&full[h % TMA_S], (unsigned)(h / TMA_S) & 1u)) ok = false;
      if (!ok) atomicOr(a.err, MHFP_WAIT_TIMEOUT);
    }
  } else {
    bool ok = true;
    int g = 0;
    const int t = warp * 32 + lane;
    for (int k = 0; k < my && ok; ++k) {
      const int wb = (int)blockIdx.x + k * (int)gridDim.x;
      const long long p0 = (long long)wb * TMA_NB;
      const long long p = p0 + t;
      const bool valid = p < L.N;
      const long long pc = valid ? p : L.N - 1;
      int i, j, kk;
      L.ijk(pc, i, j, kk);
      float r[3] = {a.b[3 * pc], a.b[3 * pc + 1], a.b[3 * pc + 2]};
      float xp[3], xm[3];
      sym_x(L, a.xin, pc, i, j, kk, 0, xp, xm);
      for (int u = 0; u < 14; ++u, ++g) {
        const int buf = g % TMA_S;
        // the next slot's x, in flight while this slot's rows are waited for
        float np[3], nm[3];
        sym_x(L, a.xin, pc, i, j, kk, u < 13 ? u + 1 : 13, np, nm);
        // the warp decides together (every lane's wait is bounded)
        if (!__all_sync(0xffffffffu, mbar_wait(&full[buf], (unsigned)(g / TMA_S) & 1u))) {
          ok = false;
          break;
        }
        const float* st = stage + (size_t)buf * TMA_STAGE;
        const float* own = st + warp * TMA_CH + lane;
        if (u == 0) {
#pragma unroll
          for (int e = 0; e < 3; ++e)
            r[e] -= own[(3 * e) * 32] * xp[0] + own[(3 * e + 1) * 32] * xp[1] + own[(3 * e + 2) * 32] * xp[2];
        } else {
          int dx, dy, dz;
          St<ST_BOX1>::off(13 + u, dx, dy, dz);
          if (L.in(i + dx, j + dy, kk + dz)) {
#pragma unroll
            for (int e = 0; e < 3; ++e)
              r[e] -= own[(3 * e) * 32] * xp[0] + own[(3 * e + 1) * 32] * xp[1] + own[(3 * e + 2) * 32] * xp[2];
          }
          if (L.in(i - dx, j - dy, kk - dz)) {
            const long long su = sym_shift(L, u);
            const long long q = p - su;  // >= 0 here
            const int m = (int)((q >> 5) - ((p0 - su) >> 5));
            const float* tr = st + (TMA_NW + m) * TMA_CH + (int)(q & 31);
#pragma unroll
            for (int e = 0; e < 3; ++e)
              r[e] -= tr[e * 32] * xm[0] + tr[(3 + e) * 32] * xm[1] + tr[(6 + e) * 32] * xm[2];
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[buf]);  // this warp is done with the buffer
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          xp[e] = np[e];
          xm[e] = nm[e];
        }
      }
      if (!ok) break;
      if (valid) {
        if (CHEB) {
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const float z = a.dinv[(3 * e) * L.N + p] * r[0] + a.dinv[(3 * e + 1) * L.N + p] * r[1] +
                            a.dinv[(3 * e + 2) * L.N + p] * r[2];
            const float dn = a.first ? a.cf[1] * z : a.cf[0] * a.d[3 * p + e] + a.cf[1] * z;
            a.d[3 * p + e] = dn;
            a.xout[3 * p + e] = a.xin[3 * p + e] + dn;
          }
        } else {
#pragma unroll
          for (int e = 0; e < 3; ++e) a.xout[3 * p + e] = r[e];
        }
      }
    }
    if (!ok && lane == 0) atomicOr(a.err, MHFP_WAIT_TIMEOUT);
  }
  __syncthreads();  // no warp leaves while copies into this CTA's shared memory may be in flight
}
// </hot:k_cheb_u0_tma>

// ---------------------------------------------------------------- transfers
// Prolongation x += P x_c and restriction b_c = P^T r between lattice levels.
// P couples coarse point (I, J, K) to the fine box of width w = 3 + 2R around
// it, fine (3I - R .. 3I + 2 + R) and so on.  The cycles read it coarse-point
// major, Pc[J][entry][WP]: entry e = BF x BC block entry, then the w^3 box
// points (x fastest) padded to WP = 128 (R = 1) or 352 (R = 2), out-of-lattice
// points zero (BF unknowns per fine point, BC per coarse point: 3 x 3 or
// 1 x 1 for M_II^(h), 3 x 6 and 6 x 6 with the rigid-body modes).  Against the
// set-up's [slot][entry][fine point] this leaves out the slots that are zero
// by structure (a fine point with index 1 mod 3 has one coarse neighbour per
// axis, not two: 4.6 of 8 slots at R = 1, 12.7 of 27 at R = 2, so 366 MB
// instead of 618 MB on the finest level at 128^3) and makes the restriction a
// stream: 64.7 us there (5.7 TB/s) against 131 us gathering from the set-up's
// layout, 48.5 against 75 us on the 2.1 M-point cell level; 11.8 against 27 us
// and 9.8 against 16 us at 64^3.
// stencil radius of the levels with BF unknowns per point: the displacement
// levels are 27-point lattices, the scalar ones 25- or 125-point
template <int BF>
constexpr int transfer_r() { return BF == 1 ? 2 : 1; }
template <int R>
struct Box {
  static constexpr int w = 3 + 2 * R, n = w * w * w, WP = R == 1 ? 128 : 352, ns = (2 + 2 * R) / 3 + 1;
};

// the set-up's P into the cycles' layout and precision: one thread per value
template <int BB, int R, typename T>
__global__ void __launch_bounds__(128) k_pack_P(Lat32 F, Lat32 C, const double* __restrict__ P, T* __restrict__ Pc) {
  using B = Box<R>;
  constexpr unsigned NB = (B::WP + 127) / 128;  // blocks of 128 per coarse point
  const unsigned J = blockIdx.x / NB, e = threadIdx.x + (blockIdx.x % NB) * 128;
  if (e >= (unsigned)B::WP) return;
  int I, Jj, K;
  C.ijk(J, I, Jj, K);
  const int ex = e % B::w, ey = (e / B::w) % B::w, ez = e / (B::w * B::w);
  const int a = 3 * I - R + ex, b = 3 * Jj - R + ey, c = 3 * K - R + ez;
  const bool in = e < (unsigned)B::n && (unsigned)a < (unsigned)F.Lx && (unsigned)b < (unsigned)F.Ly &&
                  (unsigned)c < (unsigned)F.Lz;
  const unsigned fp = in ? (unsigned)a + (unsigned)F.Lx * ((unsigned)b + (unsigned)F.Ly * (unsigned)c) : 0u;
  const int sl = in ? (I - p_lo(a, R)) + B::ns * ((Jj - p_lo(b, R)) + B::ns * (K - p_lo(c, R))) : 0;
#pragma unroll 1
  for (int t = 0; t < BB; ++t)
    Pc[((size_t)J * BB + t) * B::WP + e] = in ? (T)P[(size_t)(sl * BB + t) * (unsigned)F.N + fp] : T(0);
}

// Restriction, W warps per coarse point: the lanes split the box points, each
// lane issuing the loads of its points before the sums; a fixed-order xor
// reduction per warp, then over the W warps through shared memory.  With
// dinvc also the coarse level's first Chebyshev step from zero (d = cr D^-1 b,
// x = d, the same sums as its own kernel would form from bc).
template <int BF, int BC, int R, int W, typename T>
__global__ void __launch_bounds__(256) k_restrict_f(Lat32 F, Lat32 C, const T* __restrict__ Pc,
                                                    const T* __restrict__ r, T* __restrict__ bc,
                                                    const T* __restrict__ dinvc, const T* __restrict__ cfc, T* __restrict__ xc,
                                                    T* __restrict__ dc, long long lb) {
  r = lane_ptr(r, lb);
  bc = lane_ptr(bc, lb);
  xc = lane_ptr(xc, lb);
  dc = lane_ptr(dc, lb);
  using B = Box<R>;
  constexpr int PER = (B::n + 32 * W - 1) / (32 * W);  // box points per lane
  constexpr int KB = BF * BC > 9 ? 1 : (PER > 4 ? 4 : PER);  // of them in flight
  __shared__ T part[W > 1 ? 8 : 1][BC];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = wid % W;
  const unsigned J = blockIdx.x * (8 / W) + wid / W;
  const bool valid = J < (unsigned)C.N;
  T acc[BC];
#pragma unroll
  for (int q = 0; q < BC; ++q) acc[q] = T(0);
  if (valid) {
    int I, Jj, K;
    C.ijk(J, I, Jj, K);
    const T* pj = Pc + (unsigned)(J * (BF * BC)) * (size_t)B::WP;
#pragma unroll
    for (int k0 = 0; k0 < PER; k0 += KB) {
      T pv[KB][BF * BC], rv[KB][BF];
#pragma unroll
      for (int kk = 0; kk < KB; ++kk) {
        const int e = lane + 32 * (sub + W * (k0 + kk));
        const int ex = e % B::w, ey = (e / B::w) % B::w, ez = e / (B::w * B::w);
        const int a = 3 * I - R + ex, b = 3 * Jj - R + ey, c = 3 * K - R + ez;
        const bool ok = k0 + kk < PER && e < B::n && (unsigned)a < (unsigned)F.Lx && (unsigned)b < (unsigned)F.Ly &&
                        (unsigned)c < (unsigned)F.Lz;
        const unsigned fp = ok ? (unsigned)a + (unsigned)F.Lx * ((unsigned)b + (unsigned)F.Ly * (unsigned)c) : 0u;
        const int ec = ok ? e : 0;
#pragma unroll
        for (int t = 0; t < BF * BC; ++t) pv[kk][t] = pj[t * B::WP + ec];
#pragma unroll
        for (int t = 0; t < BF; ++t) {
          const T v = r[BF * fp + t];
          rv[kk][t] = ok ? v : T(0);
        }
      }
#pragma unroll
      for (int kk = 0; kk < KB; ++kk)
#pragma unroll
        for (int q = 0; q < BC; ++q)
#pragma unroll
          for (int t = 0; t < BF; ++t) acc[q] += pv[kk][t * BC + q] * rv[kk][t];
    }
  }
#pragma unroll
  for (int q = 0; q < BC; ++q)
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], m);
  if (W > 1) {
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < BC; ++q) part[wid][q] = acc[q];
    __syncthreads();
    if (sub != 0) return;
#pragma unroll
    for (int q = 0; q < BC; ++q)
#pragma unroll
      for (int u = 1; u < W; ++u) acc[q] += part[wid + u][q];
  }
  if (!valid || lane >= BC) return;
  // lane a takes component a
  T s = acc[0];
#pragma unroll
  for (int q = 1; q < BC; ++q) s = lane == q ? acc[q] : s;
  bc[BC * J + lane] = s;
  if (dinvc) {
    T z = T(0);
#pragma unroll
    for (int t = 0; t < BC; ++t) z += dinvc[(unsigned)(lane * BC + t) * (unsigned)C.N + J] * acc[t];
    dc[BC * J + lane] = cfc[1] * z;
    xc[BC * J + lane] = cfc[1] * z;
  }
}

// acc += the coarse points in the (sy, sz) slot pairs first, first + step, ...
// of fine point (a, b, c) (a pair without a coarse point is skipped: uniform along x)
template <int BF, int BC, int R, typename T>
__device__ __forceinline__ void prolong_sum(const Lat32& C, int a, int b, int c, const T* __restrict__ Pc,
                                            const T* __restrict__ xc, T acc[BF], int first, int step) {
  using B = Box<R>;
  const int lx = p_lo(a, R), ly = p_lo(b, R), lz = p_lo(c, R);
#pragma unroll 1
  for (int yz = first; yz < B::ns * B::ns; yz += step) {
    const int Jy = ly + yz % B::ns, Kz = lz + yz / B::ns;
    const int ey = b - 3 * Jy + R, ez = c - 3 * Kz + R;
    if ((unsigned)Jy >= (unsigned)C.Ly || (unsigned)Kz >= (unsigned)C.Lz || ey < 0 || ez < 0) continue;
    T pv[B::ns][BF * BC], xv[B::ns][BC];
#pragma unroll
    for (int sx = 0; sx < B::ns; ++sx) {
      const int Ix = lx + sx, ex = a - 3 * Ix + R;
      const bool in = (unsigned)Ix < (unsigned)C.Lx && ex >= 0;
      const unsigned J = in ? (unsigned)Ix + (unsigned)C.Lx * ((unsigned)Jy + (unsigned)C.Ly * (unsigned)Kz) : 0u;
      const unsigned e = in ? (unsigned)(ex + B::w * (ey + B::w * ez)) : 0u;
      const T* pj = Pc + (unsigned)(J * (BF * BC)) * (size_t)B::WP + e;
#pragma unroll
      for (int t = 0; t < BF * BC; ++t) pv[sx][t] = in ? pj[t * B::WP] : T(0);
#pragma unroll
      for (int t = 0; t < BC; ++t) xv[sx][t] = in ? xc[BC * J + t] : T(0);
    }
#pragma unroll
    for (int sx = 0; sx < B::ns; ++sx)
#pragma unroll
      for (int q = 0; q < BF; ++q)
#pragma unroll
        for (int t = 0; t < BC; ++t) acc[q] += pv[sx][q * BC + t] * xv[sx][t];
  }
}

// Large displacement levels read the set-up's fine-point major layout
// Pm[slot][entry][fine point], where every load of a warp is one line
// (coarse-point major it is a line per three lanes).  A warp takes one
// (sy, sz) slot pair for 32 fine points: one round of loads, the partial sums
// joined in order; pairs that are zero by structure are skipped, uniformly
// along x, so that 0.69 of P is read.  Microseconds, this form / a thread per
// fine point on the same layout / the same coarse-point major / all eight
// slots by a thread (before): 274,625 points 3 x 3 14.3 / 15.5 / 22.7 / 15.1,
// 2,146,689 points 86 / 91 / 126 / 108, 110,592 points 3 x 6 14.5 / 30.6 /
// 18.3 / 21.3, 68,921 points 3 x 3 FP64 13.9 / 20.5 / 17.7 / 14.7.
template <int BF, int BC, int R, typename T>
__global__ void __launch_bounds__(32 * Box<R>::ns * Box<R>::ns)
    k_prolong_f(Lat32 F, Lat32 C, const T* __restrict__ Pm, const T* __restrict__ xc, T* __restrict__ x,
                long long lb) {
  using B = Box<R>;
  constexpr int W = B::ns * B::ns;
  xc = lane_ptr(xc, lb);
  x = lane_ptr(x, lb);
  __shared__ T part[W][BF][32];
  // blocks take the fine points in descending order: the restriction went
  // through them in ascending order, so the last ones' x is still in L2
  const unsigned p = (gridDim.x - 1 - blockIdx.x) * 32 + threadIdx.x;
  const bool valid = p < (unsigned)F.N;
  const int yz = threadIdx.y;
  T acc[BF];
#pragma unroll
  for (int r = 0; r < BF; ++r) acc[r] = T(0);
  int a, b, c;
  F.ijk(valid ? p : 0u, a, b, c);
  const int lx = p_lo(a, R), Jy = p_lo(b, R) + yz % B::ns, Kz = p_lo(c, R) + yz / B::ns;
  if (valid && (unsigned)Jy < (unsigned)C.Ly && (unsigned)Kz < (unsigned)C.Lz && b - 3 * Jy + R >= 0 &&
      c - 3 * Kz + R >= 0) {
    T pv[B::ns][BF * BC], xv[B::ns][BC];
#pragma unroll
    for (int sx = 0; sx < B::ns; ++sx) {
      const bool in = (unsigned)(lx + sx) < (unsigned)C.Lx;
      const unsigned J = in ? (unsigned)(lx + sx) + (unsigned)C.Lx * ((unsigned)Jy + (unsigned)C.Ly * (unsigned)Kz) : 0u;
      const T* pj = Pm + (unsigned)((sx + B::ns * yz) * (BF * BC)) * (size_t)(unsigned)F.N + p;
#pragma unroll
      for (int t = 0; t < BF * BC; ++t) {
        const T v = pj[(size_t)t * (unsigned)F.N];
        pv[sx][t] = in ? v : T(0);
      }
#pragma unroll
      for (int t = 0; t < BC; ++t) {
        const T v = xc[BC * J + t];
        xv[sx][t] = in ? v : T(0);
      }
    }
#pragma unroll
    for (int sx = 0; sx < B::ns; ++sx)
#pragma unroll
      for (int q = 0; q < BF; ++q)
#pragma unroll
        for (int t = 0; t < BC; ++t) acc[q] += pv[sx][q * BC + t] * xv[sx][t];
  }
#pragma unroll
  for (int r = 0; r < BF; ++r) part[yz][r][threadIdx.x] = acc[r];
  __syncthreads();
  if (yz != 0 || !valid) return;
#pragma unroll
  for (int r = 0; r < BF; ++r) {
#pragma unroll
    for (int u = 1; u < W; ++u) acc[r] += part[u][r][threadIdx.x];
    x[BF * p + r] += acc[r];
  }
}

// Large scalar levels: a thread per fine point on the coarse-point major
// layout (262,144 points: 8.6 us, 10.1 with all 27 slots read before, 14.1
// split as above; 2,097,152 points: 54, 65 and 105)
template <int R, typename T>
__global__ void __launch_bounds__(256) k_prolong_s(Lat32 F, Lat32 C, const T* __restrict__ Pc,
                                                   const T* __restrict__ xc, T* __restrict__ x, long long lb) {
  xc = lane_ptr(xc, lb);
  x = lane_ptr(x, lb);
  const unsigned p = (gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
  if (p >= (unsigned)F.N) return;
  int a, b, c;
  F.ijk(p, a, b, c);
  T acc[1] = {T(0)};
  prolong_sum<1, 1, R, T>(C, a, b, c, Pc, xc, acc, 0, 1);
  x[p] += acc[0];
}

// small fine levels: a warp per (sy, sz) slot pair for 32 consecutive fine
// points, partial sums added in a fixed order through shared memory
template <int BF, int BC, int R, typename T>
__global__ void __launch_bounds__(32 * Box<R>::ns * Box<R>::ns)
    k_prolong_w(Lat32 F, Lat32 C, const T* __restrict__ Pc, const T* __restrict__ xc, T* __restrict__ x,
                long long lb) {
  constexpr int W = Box<R>::ns * Box<R>::ns;
  xc = lane_ptr(xc, lb);
  x = lane_ptr(x, lb);
  __shared__ T part[W][BF][32];
  const unsigned p = blockIdx.x * 32 + threadIdx.x;
  const bool valid = p < (unsigned)F.N;
  T acc[BF];
#pragma unroll
  for (int r = 0; r < BF; ++r) acc[r] = T(0);
  if (valid) {
    int a, b, c;
    F.ijk(p, a, b, c);
    prolong_sum<BF, BC, R, T>(C, a, b, c, Pc, xc, acc, threadIdx.y, W);
  }
#pragma unroll
  for (int r = 0; r < BF; ++r) part[threadIdx.y][r][threadIdx.x] = acc[r];
  __syncthreads();
  if (threadIdx.y != 0 || !valid) return;
#pragma unroll
  for (int r = 0; r < BF; ++r) {
    T sum = T(0);
#pragma unroll
    for (int u = 0; u < W; ++u) sum += part[u][r][threadIdx.x];
    x[BF * p + r] += sum;
  }
}

// face level (ELL, 11 slots) versions
// y = b - C x (y = C x when b is null) on the face level; the 11 columns of
// each row follow from the face topology (FaceTopo32::ell_cols), so only
// the values stream from memory
template <typename T>
__global__ void __launch_bounds__(256) k_spmv_ell(FaceTopo32 t, const T* __restrict__ val, const T* __restrict__ x,
                                                  const T* __restrict__ b, T* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  const unsigned f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= t.nF) return;
  unsigned col[11];
  t.ell_cols(f, col);
  T a = T(0);
#pragma unroll
  for (int q = 0; q < 11; ++q) a += val[q * t.nF + f] * x[col[q]];
  y[f] = b ? b[f] - a : a;
}

template <typename T>
__global__ void __launch_bounds__(256) k_cheb_ell(FaceTopo32 t, const T* __restrict__ val,
                                                  const T* __restrict__ dinv, const T* __restrict__ b,
                                                  const T* __restrict__ xin, T* __restrict__ xout, T* __restrict__ d,
                                                  const T* __restrict__ cf, bool first, long long lb) {
  const T cd = cf[0], cr = cf[1];
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  const unsigned f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= t.nF) return;
  T r = b[f];
  if (xin) {
    unsigned col[11];
    t.ell_cols(f, col);
#pragma unroll
    for (int q = 0; q < 11; ++q) r -= val[q * t.nF + f] * xin[col[q]];
  }
  const T dn = first ? cr * dinv[f] * r : cd * d[f] + cr * dinv[f] * r;
  d[f] = dn;
  xout[f] = (xin ? xin[f] : T(0)) + dn;
}

// faces -> cells Galerkin product of the interface-pressure hierarchy (set-up)
struct FaceTopo {
  int nx, ny, nz;
  long long nT, nF, nFx, nFy;
};

__device__ __forceinline__ long long ft_cell_face(const FaceTopo& d, int i, int j, int k, int lf) {
  switch (lf) {
    case 0: return i + (long long)(d.nx + 1) * (j + (long long)d.ny * k);
    case 1: return (i + 1) + (long long)(d.nx + 1) * (j + (long long)d.ny * k);
    case 2: return d.nFx + i + (long long)d.nx * (j + (long long)(d.ny + 1) * k);
    case 3: return d.nFx + i + (long long)d.nx * ((j + 1) + (long long)(d.ny + 1) * k);
    case 4: return d.nFx + d.nFy + i + (long long)d.nx * (j + (long long)d.ny * k);
    default: return d.nFx + d.nFy + i + (long long)d.nx * (j + (long long)d.ny * (k + 1));
  }
}

// face -> up to two cells as lattice coordinates (valid flags)
__device__ __forceinline__ int ft_face_cells(const FaceTopo& d, long long f, int c[2][3]) {
  int i, j, k, ax;
  if (f < d.nFx) {
    ax = 0; i = (int)(f % (d.nx + 1)); long long r = f / (d.nx + 1); j = (int)(r % d.ny); k = (int)(r / d.ny);
  } else if (f < d.nFx + d.nFy) {
    long long g = f - d.nFx;
    ax = 1; i = (int)(g % d.nx); long long r = g / d.nx; j = (int)(r % (d.ny + 1)); k = (int)(r / (d.ny + 1));
  } else {
    long long g = f - d.nFx - d.nFy;
    ax = 2; i = (int)(g % d.nx); long long r = g / d.nx; j = (int)(r % d.ny); k = (int)(r / d.ny);
  }
  const int lim[3] = {d.nx, d.ny, d.nz};
  int cnt = 0;
  int base[3] = {i, j, k};
  base[ax] -= 1;
  if (base[ax] >= 0) { c[cnt][0] = base[0]; c[cnt][1] = base[1]; c[cnt][2] = base[2]; ++cnt; }
  base[ax] += 1;
  if (base[ax] < lim[ax]) { c[cnt][0] = base[0]; c[cnt][1] = base[1]; c[cnt][2] = base[2]; ++cnt; }
  return cnt;
}

template <typename T>
__global__ void __launch_bounds__(256) k_restrict_faces(FaceTopo32 t, const T* __restrict__ pw,
                                                        const T* __restrict__ r, T* __restrict__ bc,
                                                        const T* __restrict__ dinvc, const T* __restrict__ cfc, T* __restrict__ xc,
                                                        T* __restrict__ dc, long long lb) {
  r = lane_ptr(r, lb);
  bc = lane_ptr(bc, lb);
  xc = lane_ptr(xc, lb);
  dc = lane_ptr(dc, lb);
  const unsigned Tc = blockIdx.x * blockDim.x + threadIdx.x;
  if (Tc >= t.nT) return;
  const unsigned q = t.d_nx.div(Tc);
  const int i = (int)(Tc - q * (unsigned)t.nx);
  const int k = (int)t.d_ny.div(q), j = (int)(q - (unsigned)k * (unsigned)t.ny);
  T s = T(0);
#pragma unroll
  for (int lf = 0; lf < 6; ++lf) {
    const unsigned f = t.face(i, j, k, lf);
    s += pw[f] * r[f];
  }
  bc[Tc] = s;
  if (dinvc) {  // the cell level's first Chebyshev step from zero, as k_restrict_f
    T z = T(0);
    z += dinvc[Tc] * s;
    dc[Tc] = cfc[1] * z;
    xc[Tc] = cfc[1] * z;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_prolong_faces(FaceTopo32 t, const T* __restrict__ pw,
                                                       const T* __restrict__ xc, T* __restrict__ x, long long lb) {
  xc = lane_ptr(xc, lb);
  x = lane_ptr(x, lb);
  // descending block order, as k_prolong_f
  const unsigned f = (gridDim.x - 1 - blockIdx.x) * blockDim.x + threadIdx.x;
  if (f >= t.nF) return;
  int c[2][3], lf[2];
  bool ok[2];
  t.cells(f, c, ok, lf);
  T s = T(0);
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (ok[q]) s += xc[t.cell(c[q][0], c[q][1], c[q][2])];
  x[f] += pw[f] * s;
}

// dense coarsest solve y = Ainv b, one block of 256 threads per row (each
// thread a strided slice of the row, then a fixed-order block sum); the
// inverse and the sums stay FP64 whatever the precision of the cycle's vectors
template <typename T>
__global__ void __launch_bounds__(256) k_dense_mv(int n, const double* __restrict__ Ainv, const T* __restrict__ b,
                                                  T* __restrict__ y, long long lb) {
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  // y = Ainv b (the coarsest level's dense FP64 inverse): a block of 8 warps
  // takes 2 rows, each row's columns split in quarters, one warp per
  // quarter, so that about 40 warps per SM keep the inverse streaming; the
  // four partial sums of a row are added in a fixed order
  __shared__ double part[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * 2 + (warp >> 2);
  const int chunk = (n + 3) / 4;
  const int c0 = (warp & 3) * chunk, c1 = min(n, c0 + chunk);
  double s = 0.0;
  if (row < n) {
    const double* a = Ainv + (long long)row * n;
#pragma unroll 4
    for (int c = c0 + lane; c < c1; c += 32) s += a[c] * widen(b[c]);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) part[warp] = s;
  __syncthreads();
  if (threadIdx.x < 2) {
    const int r = blockIdx.x * 2 + threadIdx.x;
    if (r < n) y[r] = (T)(((part[4 * threadIdx.x] + part[4 * threadIdx.x + 1]) + part[4 * threadIdx.x + 2]) +
                          part[4 * threadIdx.x + 3]);
  }
}

__global__ void k_cast_f32(long long n, const double* __restrict__ x, float* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (float)x[i];
}

// rows 0..125 of the FP64 offset-major values ([row][n]) into the
// node-blocked FP32 layout of the symmetric sweep
__global__ void k_cast_f32_sym(long long n, const double* __restrict__ x, float* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 126 * n) return;
  const long long row = i / n, q = i % n;
  y[sym_base(q) + 32 * row] = (float)x[i];
}

// ------------------------------------------------------------------ setup
template <int BS, int KIND>
__global__ void k_dinv(Lat L, const double* __restrict__ val, double* __restrict__ dinv) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= L.N) return;
  const double* v = val + (long long)St<KIND>::C * BS * BS * L.N + p;
  if (BS == 1) {
    dinv[p] = 1.0 / v[0];
  } else if (BS != 3) {
    // the SPD point block of the rigid-body-mode levels (6 x 6): Gauss-
    // Jordan elimination without pivoting (positive pivots of an SPD block)
    double m[BS][2 * BS];
    for (int r = 0; r < BS; ++r)
      for (int c = 0; c < BS; ++c) {
        m[r][c] = v[(long long)(r * BS + c) * L.N];
        m[r][BS + c] = (r == c) ? 1.0 : 0.0;
      }
    for (int c = 0; c < BS; ++c) {
      const double ip = 1.0 / m[c][c];
      for (int k = 0; k < 2 * BS; ++k) m[c][k] *= ip;
      for (int r = 0; r < BS; ++r) {
        if (r == c) continue;
        const double f = m[r][c];
        for (int k = 0; k < 2 * BS; ++k) m[r][k] -= f * m[c][k];
      }
    }
    for (int r = 0; r < BS; ++r)
      for (int c = 0; c < BS; ++c) dinv[(long long)(r * BS + c) * L.N + p] = m[r][BS + c];
  } else {
    double a[9];
    for (int q = 0; q < 9; ++q) a[q] = v[(long long)q * L.N];
    const double c00 = a[4] * a[8] - a[5] * a[7], c01 = a[5] * a[6] - a[3] * a[8], c02 = a[3] * a[7] - a[4] * a[6];
    const double det = a[0] * c00 + a[1] * c01 + a[2] * c02;
    const double id = 1.0 / det;
    double inv[9];
    inv[0] = c00 * id; inv[1] = (a[2] * a[7] - a[1] * a[8]) * id; inv[2] = (a[1] * a[5] - a[2] * a[4]) * id;
    inv[3] = c01 * id; inv[4] = (a[0] * a[8] - a[2] * a[6]) * id; inv[5] = (a[2] * a[3] - a[0] * a[5]) * id;
    inv[6] = c02 * id; inv[7] = (a[1] * a[6] - a[0] * a[7]) * id; inv[8] = (a[0] * a[4] - a[1] * a[3]) * id;
    for (int q = 0; q < 9; ++q) dinv[(long long)q * L.N + p] = inv[q];
  }
}

__global__ void k_dinv_ell(long long n, const double* __restrict__ val, double* __restrict__ dinv) {
  const long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (f < n) dinv[f] = 1.0 / val[f];
}

// One power-iteration step after r = A v: w = (D^-1 r) / *rho_v and, by the
// last block, *rho_w = ||w||, with *rho_v the norm of v: the iterates are
// never scaled by a pass of their own and the host reads only the last norm.
// Without dinv only *rho_w = ||r|| (the start vector's norm).
constexpr int POWER_BLOCKS = 304;
template <int BS>
__global__ void __launch_bounds__(256) k_power_step(long long N, const double* __restrict__ dinv,
                                                    const double* __restrict__ r, double* __restrict__ w,
                                                    const double* __restrict__ rho_v, double* __restrict__ rho_w,
                                                    double* __restrict__ partials, unsigned* __restrict__ counter) {
  __shared__ double sh[8];
  const double inv = dinv ? 1.0 / *rho_v : 0.0;
  double acc = 0.0;
  for (long long p = (long long)blockIdx.x * 256 + threadIdx.x; p < N; p += (long long)gridDim.x * 256) {
    double x[BS];
#pragma unroll
    for (int t = 0; t < BS; ++t) x[t] = r[BS * p + t];
    if (!dinv) {
#pragma unroll
      for (int t = 0; t < BS; ++t) acc = fma(x[t], x[t], acc);
      continue;
    }
#pragma unroll
    for (int a = 0; a < BS; ++a) {
      double s = 0.0;
#pragma unroll
      for (int t = 0; t < BS; ++t) s += dinv[(long long)(a * BS + t) * N + p] * x[t];
      s *= inv;
      w[BS * p + a] = s;
      acc = fma(s, s, acc);
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += sh[k];
    partials[blockIdx.x] = s;
  }
  if (!last_block(counter, gridDim.x) || threadIdx.x >= 32) return;
  const double n2 = warp_sum_of(partials, (int)gridDim.x);
  if (threadIdx.x == 0) *rho_w = sqrt(n2);
}

__global__ void k_power_start(long long n, double* __restrict__ v) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = 1.0 + (double)((7919LL * i) % 97) / 97.0;
}

// Smoothed prolongator: P[a, J] = [a in J] diag(active_a) - omega D_a^-1 sum_{b in J, b ~ a} A_ab diag(active_b)
template <int BS, int KIND>
__global__ void k_build_P(Lat F, Lat Cc, const double* __restrict__ val, const double* __restrict__ dinv,
                          const unsigned char* __restrict__ active, double omega, double* __restrict__ P) {
  const int R = St<KIND>::R;
  const int ns = p_slots(R);
  const int nslot = ns * ns * ns;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= F.N * nslot) return;
  const int s = (int)(tid / F.N);
  const long long p = tid - (long long)s * F.N;
  int a, b, c;
  F.ijk(p, a, b, c);
  const int sx = s % ns, sy = (s / ns) % ns, sz = s / (ns * ns);
  const int I = p_lo(a, R) + sx, J = p_lo(b, R) + sy, K = p_lo(c, R) + sz;
  double out[BS * BS];
  for (int q = 0; q < BS * BS; ++q) out[q] = 0.0;
  if (Cc.in(I, J, K)) {
    double ap[BS * BS];
    for (int q = 0; q < BS * BS; ++q) ap[q] = 0.0;
    for (int o = 0; o < St<KIND>::N; ++o) {
      int dx, dy, dz;
      St<KIND>::off(o, dx, dy, dz);
      const int na = a + dx, nb = b + dy, nc = c + dz;
      if (!F.in(na, nb, nc)) continue;
      if (na / 3 != I || nb / 3 != J || nc / 3 != K) continue;
      const long long q = F.id(na, nb, nc);
      const double* v = val + (long long)o * BS * BS * F.N + p;
      for (int r = 0; r < BS; ++r)
        for (int t = 0; t < BS; ++t) ap[r * BS + t] += v[(long long)(r * BS + t) * F.N] * (active[BS * q + t] ? 1.0 : 0.0);
    }
    for (int r = 0; r < BS; ++r)
      for (int t = 0; t < BS; ++t) {
        double z = 0.0;
        for (int u = 0; u < BS; ++u) z += dinv[(long long)(r * BS + u) * F.N + p] * ap[u * BS + t];
        out[r * BS + t] = -omega * z;
      }
    if (a / 3 == I && b / 3 == J && c / 3 == K)
      for (int r = 0; r < BS; ++r) out[r * BS + r] += active[BS * p + r] ? 1.0 : 0.0;
  }
  for (int q = 0; q < BS * BS; ++q) P[((long long)s * BS * BS + q) * F.N + p] = out[q];
}

__global__ void k_active_fine(long long nU, const unsigned char* __restrict__ fix, unsigned char* __restrict__ act) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < nU) act[r] = ((fix[r / 3] >> (r % 3)) & 1) ? 0 : 1;
}

template <int BS>
__global__ void k_active_coarse(Lat F, Lat Cc, const unsigned char* __restrict__ af, unsigned char* __restrict__ ac) {
  const long long J = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (J >= Cc.N) return;
  int I, Jj, K;
  Cc.ijk(J, I, Jj, K);
  unsigned char m[BS];
  for (int q = 0; q < BS; ++q) m[q] = 0;
  for (int c = 3 * K; c < 3 * K + 3 && c < F.Lz; ++c)
    for (int b = 3 * Jj; b < 3 * Jj + 3 && b < F.Ly; ++b)
      for (int a = 3 * I; a < 3 * I + 3 && a < F.Lx; ++a) {
        const long long p = F.id(a, b, c);
        for (int q = 0; q < BS; ++q) m[q] |= af[BS * p + q];
      }
  for (int q = 0; q < BS; ++q) ac[BS * J + q] = m[q] ? 1 : 0;
}

// Q[a, J] = sum_o A[a, a+o] P[a+o, J]   (fine point a, coarse J in its Q range;
// A blocks BF x BF, P and Q blocks BF x BC)
template <int BF, int BC, int KIND>
__global__ void k_build_Q(Lat F, Lat Cc, const double* __restrict__ val, const double* __restrict__ P,
                          double* __restrict__ Q) {
  const int R = St<KIND>::R;
  const int ns = p_slots(R), nq = q_slots(R);
  const int nqs = nq * nq * nq;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= F.N * nqs) return;
  const int s = (int)(tid / F.N);
  const long long p = tid - (long long)s * F.N;
  int a, b, c;
  F.ijk(p, a, b, c);
  const int I = q_lo(a, R) + s % nq, J = q_lo(b, R) + (s / nq) % nq, K = q_lo(c, R) + s / (nq * nq);
  double out[BF * BC];
  for (int q = 0; q < BF * BC; ++q) out[q] = 0.0;
  if (Cc.in(I, J, K)) {
    for (int o = 0; o < St<KIND>::N; ++o) {
      int dx, dy, dz;
      St<KIND>::off(o, dx, dy, dz);
      const int na = a + dx, nb = b + dy, nc = c + dz;
      if (!F.in(na, nb, nc)) continue;
      const int px = I - p_lo(na, R), py = J - p_lo(nb, R), pz = K - p_lo(nc, R);
      if (px < 0 || px >= ns || py < 0 || py >= ns || pz < 0 || pz >= ns) continue;
      const long long q = F.id(na, nb, nc);
      const int ps = px + ns * (py + ns * pz);
      const double* v = val + (long long)o * BF * BF * F.N + p;
      const double* pv = P + (long long)ps * BF * BC * F.N + q;
      for (int r = 0; r < BF; ++r)
        for (int t = 0; t < BC; ++t) {
          double z = 0.0;
          for (int u = 0; u < BF; ++u) z += v[(long long)(r * BF + u) * F.N] * pv[(long long)(u * BC + t) * F.N];
          out[r * BC + t] += z;
        }
    }
  }
  for (int q = 0; q < BF * BC; ++q) Q[((long long)s * BF * BC + q) * F.N + p] = out[q];
}

// The same for the scalar lattices.  Bound by the issue of the index work: most
// (offset, slot) pairs have no product, and a thread per slot tests all 25 or
// 125 offsets for each of 64 slots.  Here a thread has the row of slots along x
// in registers, so an offset's tests on y and z, its coefficient and its
// addresses are used for the whole row.  96^3, the 25-point level: 3.39 -> 1.50 ms.
template <int KIND>
__global__ void __launch_bounds__(256) k_build_Q1(Lat F, Lat Cc, const double* __restrict__ val,
                                                  const double* __restrict__ P, double* __restrict__ Q) {
  constexpr int R = St<KIND>::R, NS = (2 + 2 * R) / 3 + 1, NQ = (2 + 4 * R) / 3 + 1;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= F.N * (NQ * NQ)) return;
  const int s = (int)(tid / F.N);
  const long long p = tid - (long long)s * F.N;
  int a, b, c;
  F.ijk(p, a, b, c);
  const int I = q_lo(a, R), J = q_lo(b, R) + s % NQ, K = q_lo(c, R) + s / NQ;
  double acc[NQ];
#pragma unroll
  for (int j = 0; j < NQ; ++j) acc[j] = 0.0;
  if ((unsigned)J < (unsigned)Cc.Ly && (unsigned)K < (unsigned)Cc.Lz) {
    for (int o = 0; o < St<KIND>::N; ++o) {
      int dx, dy, dz;
      St<KIND>::off(o, dx, dy, dz);
      const int py = J - p_lo(b + dy, R), pz = K - p_lo(c + dz, R);
      if ((unsigned)py >= (unsigned)NS || (unsigned)pz >= (unsigned)NS) continue;
      if (!F.in(a + dx, b + dy, c + dz)) continue;
      const int lx = p_lo(a + dx, R) - I;  // the neighbour's first slot in the row
      const double v = val[(long long)o * F.N + p];
      const double* pv = P + (long long)(NS * (py + NS * pz)) * F.N + F.id(a + dx, b + dy, c + dz);
#pragma unroll
      for (int j = 0; j < NQ; ++j)
        if ((unsigned)(j - lx) < (unsigned)NS) acc[j] = fma(v, pv[(long long)(j - lx) * F.N], acc[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < NQ; ++j)
    Q[((long long)NQ * s + j) * F.N + p] = (unsigned)(I + j) < (unsigned)Cc.Lx ? acc[j] : 0.0;
}

// The same for 3 x 3 blocks on the 27-point lattice, bound by the FP64 pipe
// (125 block products, 3,375 FMA per fine point: 5.1 ms at 96^3).  In
// k_build_Q a warp's lanes have all three residues of the fine x index, so
// nine (offset, slot) pairs per axis are issued for five that are not zero.
// Here a warp takes 32 fine points of one residue RHO (a = 3 m + RHO), whose
// products are known at compile time: x slots of the neighbours 3 n: {n - 1, n},
// 3 n + 1: {n}, 3 n + 2: {n, n + 1}.  A block has the nine warps (residue,
// Jy slot) of a line's 96 points, so that the three residues share lines in
// L1; a lane keeps up to three x slots of 3 x 3 sums.  Slots that are zero by
// structure are not written (k_rap does not read them).  96^3, finest level:
// 17.3 ms before, 6.5 ms (the FP64 pipe active 0.97 of the time).
template <int RHO>
__device__ __forceinline__ void q3_line(const Lat32& F, unsigned p, int a, int dy, int dz, int py, int pz,
                                        const double* __restrict__ val, const double* __restrict__ P,
                                        double (&acc)[3][9]) {
  const size_t N = (unsigned)F.N;
  const int o0 = 3 * (dy + 1) + 9 * (dz + 1);
#pragma unroll
  for (int dx = -1; dx <= 1; ++dx) {
    const bool in = (unsigned)(a + dx) < (unsigned)F.Lx;
    double A[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) A[e] = val[(size_t)((o0 + dx + 1) * 9 + e) * N + p];
    // the neighbour (the point itself where there is none: its block is zero)
    const unsigned q = p + (unsigned)((in ? dx : 0) + F.Lx * dy + F.LxLy * dz);
    constexpr int QLO = RHO == 2 ? 0 : -1;  // q_lo(a) - m
    const int sig = (RHO + dx + 3) % 3, nm = (RHO + dx + 3) / 3 - 1;  // a + dx = 3 (m + nm) + sig
#pragma unroll
    for (int sx = 0; sx < 2; ++sx) {
      if (sig == 1 && sx == 1) continue;
      const int jx = nm + sx - (sig == 0 ? 1 : 0) - QLO;  // Q slot of coarse m + nm + sx (- 1)
      const double* pv = P + (size_t)((sx + 2 * (py + 2 * pz)) * 9) * N + q;
      double b[9];
#pragma unroll
      for (int e = 0; e < 9; ++e) b[e] = pv[(size_t)e * N];
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
          for (int u = 0; u < 3; ++u) acc[jx][3 * r + t] = fma(A[3 * r + u], b[3 * u + t], acc[jx][3 * r + t]);
    }
  }
}

template <int RHO>
__device__ __forceinline__ void q3_point(const Lat32& F, const Lat32& C, int a, int b, int c, int sy,
                                         const double* __restrict__ val, const double* __restrict__ P,
                                         double* __restrict__ Q) {
  const size_t N = (unsigned)F.N;
  const int Jy = q_lo(b, 1) + sy;
  if ((unsigned)Jy >= (unsigned)C.Ly || b - 3 * Jy + 2 < 0) return;
  const unsigned p = (unsigned)(a + F.Lx * b) + (unsigned)F.LxLy * (unsigned)c;
#pragma unroll 1
  for (int sz = 0; sz < 3; ++sz) {
    const int Jz = q_lo(c, 1) + sz;
    if ((unsigned)Jz >= (unsigned)C.Lz || c - 3 * Jz + 2 < 0) continue;
    double acc[3][9];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int e = 0; e < 9; ++e) acc[j][e] = 0.0;
#pragma unroll 1
    for (int dz = -1; dz <= 1; ++dz) {
      const int nc = c + dz, pz = Jz - p_lo(nc, 1);
      if ((unsigned)nc >= (unsigned)F.Lz || (unsigned)(nc - 3 * Jz + 1) >= 5u) continue;
#pragma unroll 1
      for (int dy = -1; dy <= 1; ++dy) {
        const int nb = b + dy, py = Jy - p_lo(nb, 1);
        if ((unsigned)nb >= (unsigned)F.Ly || (unsigned)(nb - 3 * Jy + 1) >= 5u) continue;
        q3_line<RHO>(F, p, a, dy, dz, py, pz, val, P, acc);
      }
    }
#pragma unroll
    for (int j = 0; j < (RHO == 1 ? 3 : 2); ++j)
#pragma unroll
      for (int e = 0; e < 9; ++e) Q[(size_t)((j + 3 * (sy + 3 * sz)) * 9 + e) * N + p] = acc[j][e];
  }
}

__global__ void __launch_bounds__(288, 2) k_build_Q3(Lat32 F, Lat32 C, const double* __restrict__ val,
                                                     const double* __restrict__ P, double* __restrict__ Q) {
  const unsigned nx = (unsigned)(F.Lx + 95) / 96;
  const unsigned line = blockIdx.x / nx, c = line / (unsigned)F.Ly, b = line - c * (unsigned)F.Ly;
  const int m = (int)(blockIdx.x - line * nx) * 32 + (int)(threadIdx.x & 31), w = threadIdx.x >> 5;
  const int a = 3 * m + w % 3;
  if (a >= F.Lx) return;
  if (w % 3 == 0) q3_point<0>(F, C, a, (int)b, (int)c, w / 3, val, P, Q);
  else if (w % 3 == 1) q3_point<1>(F, C, a, (int)b, (int)c, w / 3, val, P, Q);
  else q3_point<2>(F, C, a, (int)b, (int)c, w / 3, val, P, Q);
}

// A_c[J, J+oc] = sum_{a in box(J)} P[a, J]^T Q[a, J+oc]   (BC x BC blocks).
// A_c is symmetric: the centre and the offsets after it are formed, the rest
// are their transposes (half the products; the stored operator is exactly
// symmetric).  Bound by the FP64 pipe on large levels (96^3: the finest
// displacement level 1.65 ms, the pipe active 0.88 of the time, the 25-point
// level 1.0 ms, 0.83); all levels, every offset formed -> this: 5.5 -> 2.1 ms
// (displacement) and 2.6 -> 1.1 ms (interface pressure).
template <int BF, int BC, int CKIND>
__global__ void k_rap(Lat F, Lat Cc, int R, const double* __restrict__ P, const double* __restrict__ Q,
                      const unsigned char* __restrict__ ac, double* __restrict__ Ac) {
  constexpr int NO = St<CKIND>::N, MID = St<CKIND>::C;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= Cc.N * (NO - MID)) return;
  const int oc = MID + (int)(tid / Cc.N);
  const long long J = tid - (long long)(oc - MID) * Cc.N;
  int I, Jj, K;
  Cc.ijk(J, I, Jj, K);
  int ox, oy, oz;
  St<CKIND>::off(oc, ox, oy, oz);
  const int I2 = I + ox, J2 = Jj + oy, K2 = K + oz;
  double out[BC * BC];
  for (int q = 0; q < BC * BC; ++q) out[q] = 0.0;
  const bool in = Cc.in(I2, J2, K2);
  if (in) {
    const int ns = p_slots(R), nq = q_slots(R);
    // the fine points in both P's range of J and Q's range of J + oc
    auto lo = [&](int j, int j2) { return max(max(3 * j - R, 3 * j2 - 2 * R), 0); };
    auto hi = [&](int j, int j2, int n) { return min(min(3 * j + 2 + R, 3 * j2 + 2 + 2 * R), n - 1); };
    for (int c = lo(K, K2); c <= hi(K, K2, F.Lz); ++c) {
      const int pz = K - p_lo(c, R), qz = K2 - q_lo(c, R);
      for (int b = lo(Jj, J2); b <= hi(Jj, J2, F.Ly); ++b) {
        const int py = Jj - p_lo(b, R), qy = J2 - q_lo(b, R);
        for (int a = lo(I, I2); a <= hi(I, I2, F.Lx); ++a) {
          const int px = I - p_lo(a, R), qx = I2 - q_lo(a, R);
          const long long p = F.id(a, b, c);
          const double* pv = P + (long long)(px + ns * (py + ns * pz)) * BF * BC * F.N + p;
          const double* qv = Q + (long long)(qx + nq * (qy + nq * qz)) * BF * BC * F.N + p;
          for (int r = 0; r < BC; ++r)
            for (int t = 0; t < BC; ++t) {
              double z = 0.0;
              for (int u = 0; u < BF; ++u) z += pv[(long long)(u * BC + r) * F.N] * qv[(long long)(u * BC + t) * F.N];
              out[r * BC + t] += z;
            }
        }
      }
    }
  }
  if (oc == MID) {
    for (int r = 0; r < BC; ++r)
      if (!ac[BC * J + r]) out[r * BC + r] = 1.0;
    for (int r = 0; r < BC; ++r)  // the block itself symmetric: its upper triangle
      for (int t = 0; t < r; ++t) out[r * BC + t] = out[t * BC + r];
  }
  for (int q = 0; q < BC * BC; ++q) Ac[((long long)oc * BC * BC + q) * Cc.N + J] = out[q];
  if (oc == MID) return;
  const int om = NO - 1 - oc;  // the opposite offset
  if (in) {
    const long long q2 = Cc.id(I2, J2, K2);
    for (int r = 0; r < BC; ++r)
      for (int t = 0; t < BC; ++t) Ac[((long long)om * BC * BC + t * BC + r) * Cc.N + q2] = out[r * BC + t];
  }
  if (!Cc.in(I - ox, Jj - oy, K - oz))
    for (int q = 0; q < BC * BC; ++q) Ac[((long long)om * BC * BC + q) * Cc.N + J] = 0.0;
}

// ------------------------------------------- rigid-body-mode near-kernel
// M_III^(h) (Section 5: smoothed aggregation with the six rigid-body modes
// as the near-kernel of A_uu).  Per aggregate (3x3x3 box of lattice points)
// one warp factorises the near-kernel restricted to the aggregate's dofs,
// N_K = Q_K R_K, by classical Gram-Schmidt applied twice in mode order
// (translations x, y, z, rotations about x, y, z); a mode left with at
// most 1e-10 of its norm is dropped (zero column of Q_K, zero row of R_K,
// the coarse dof inactive).  The lanes hold the rows (lane l: rows l,
// l + 32, ...), dot products are fixed-order xor butterflies.  Q_K is
// stored per fine point, Pt[(a BC + j)][p] = Q_K(row of dof a of point p, j);
// R_K as the coarse point's near-kernel, Nc[(a 6 + j)][K] = R_K(a, j).
constexpr int RBM_K = 6;
constexpr double RBM_DROP = 1e-10;

__device__ __forceinline__ double warp_sum_xor(double v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

// near-kernel rows of the aggregate's dofs: the fine level (BF = 3) takes
// the rigid-body modes of the node coordinates (about the centroid cen,
// rows of prescribed dofs zero); a coarse level (BF = 6) takes the previous
// level's R blocks
template <int BF>
__device__ __forceinline__ void rbm_rows(const Lat& F, int I, int J, int K, int row, const double* __restrict__ coords,
                                         const unsigned char* __restrict__ active, const double* __restrict__ Nprev,
                                         double cx, double cy, double cz, double n[RBM_K], long long& p, int& a,
                                         bool& ok) {
  // row = local point (box order, i fastest) * BF + dof
  const int lp = row / BF;
  a = row - lp * BF;
  const int ex = lp % 3, ey = (lp / 3) % 3, ez = lp / 9;
  const int i = 3 * I + ex, j = 3 * J + ey, k = 3 * K + ez;
  ok = lp < 27 && F.in(i, j, k);
  p = ok ? F.id(i, j, k) : 0;
  for (int m = 0; m < RBM_K; ++m) n[m] = 0.0;
  if (!ok || !active[BF * p + a]) return;
  if (BF == 3) {
    const double x = coords[3 * p] - cx, y = coords[3 * p + 1] - cy, z = coords[3 * p + 2] - cz;
    n[a] = 1.0;
    // rotation about x: (0, -z, y); about y: (z, 0, -x); about z: (-y, x, 0)
    if (a == 0) { n[4] = z; n[5] = -y; }
    if (a == 1) { n[3] = -z; n[5] = x; }
    if (a == 2) { n[3] = y; n[4] = -x; }
  } else {
    for (int m = 0; m < RBM_K; ++m) n[m] = Nprev[(long long)(a * RBM_K + m) * F.N + p];
  }
}

template <int BF, int RPL>
__global__ void __launch_bounds__(128) k_rbm_tentative(Lat F, Lat Cc, const double* __restrict__ coords,
                                                        const unsigned char* __restrict__ active,
                                                        const double* __restrict__ Nprev, double cx, double cy,
                                                        double cz, double* __restrict__ Pt, double* __restrict__ Nc,
                                                        unsigned char* __restrict__ ac) {
  const long long Kc = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (Kc >= Cc.N) return;  // whole warps leave together
  int I, J, K;
  Cc.ijk(Kc, I, J, K);
  double v[RPL][RBM_K], q[RPL][RBM_K];
  long long pp[RPL];
  int aa[RPL];
  bool ok[RPL];
#pragma unroll
  for (int t = 0; t < RPL; ++t) {
    rbm_rows<BF>(F, I, J, K, lane + 32 * t, coords, active, Nprev, cx, cy, cz, v[t], pp[t], aa[t], ok[t]);
#pragma unroll
    for (int m = 0; m < RBM_K; ++m) q[t][m] = 0.0;
  }
  double R[RBM_K][RBM_K];
#pragma unroll
  for (int a = 0; a < RBM_K; ++a)
#pragma unroll
    for (int b = 0; b < RBM_K; ++b) R[a][b] = 0.0;
  bool kept[RBM_K];
#pragma unroll
  for (int j = 0; j < RBM_K; ++j) {
    double w[RPL];
    double s0 = 0.0;
#pragma unroll
    for (int t = 0; t < RPL; ++t) {
      w[t] = v[t][j];
      s0 += w[t] * w[t];
    }
    const double n0 = sqrt(warp_sum_xor(s0));
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
      double h[RBM_K];
#pragma unroll
      for (int i = 0; i < RBM_K; ++i) {
        if (i >= j) break;
        double d = 0.0;
#pragma unroll
        for (int t = 0; t < RPL; ++t) d += q[t][i] * w[t];
        h[i] = warp_sum_xor(d);
      }
#pragma unroll
      for (int i = 0; i < RBM_K; ++i) {
        if (i >= j) break;
        R[i][j] += h[i];
#pragma unroll
        for (int t = 0; t < RPL; ++t) w[t] -= h[i] * q[t][i];
      }
    }
    double s1 = 0.0;
#pragma unroll
    for (int t = 0; t < RPL; ++t) s1 += w[t] * w[t];
    const double nv = sqrt(warp_sum_xor(s1));
    kept[j] = n0 > 0.0 && nv > RBM_DROP * n0;
    const double inv = kept[j] ? 1.0 / nv : 0.0;
#pragma unroll
    for (int t = 0; t < RPL; ++t) q[t][j] = kept[j] ? w[t] * inv : 0.0;
    R[j][j] = kept[j] ? nv : 0.0;
  }
#pragma unroll
  for (int t = 0; t < RPL; ++t)
    if (ok[t])
#pragma unroll
      for (int j = 0; j < RBM_K; ++j) Pt[(long long)(aa[t] * RBM_K + j) * F.N + pp[t]] = q[t][j];
  if (lane == 0) {
#pragma unroll
    for (int a = 0; a < RBM_K; ++a) {
#pragma unroll
      for (int b = 0; b < RBM_K; ++b) Nc[(long long)(a * RBM_K + b) * Cc.N + Kc] = R[a][b];
      ac[RBM_K * Kc + a] = kept[a] ? 1 : 0;
    }
  }
}

// Smoothed prolongator from the per-point tentative blocks:
// P[a, J] = Pt[a] [agg(a) = J] - omega D_a^-1 sum_{b ~ a, agg(b) = J} A_ab Pt[b]
template <int BF, int BC, int KIND>
__global__ void k_build_P_t(Lat F, Lat Cc, const double* __restrict__ val, const double* __restrict__ dinv,
                            const double* __restrict__ Pt, double omega, double* __restrict__ P) {
  const int R = St<KIND>::R;
  const int ns = p_slots(R);
  const int nslot = ns * ns * ns;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= F.N * nslot) return;
  const int s = (int)(tid / F.N);
  const long long p = tid - (long long)s * F.N;
  int a, b, c;
  F.ijk(p, a, b, c);
  const int sx = s % ns, sy = (s / ns) % ns, sz = s / (ns * ns);
  const int I = p_lo(a, R) + sx, J = p_lo(b, R) + sy, K = p_lo(c, R) + sz;
  double out[BF * BC];
  for (int q = 0; q < BF * BC; ++q) out[q] = 0.0;
  if (Cc.in(I, J, K)) {
    double ap[BF * BC];
    for (int q = 0; q < BF * BC; ++q) ap[q] = 0.0;
    for (int o = 0; o < St<KIND>::N; ++o) {
      int dx, dy, dz;
      St<KIND>::off(o, dx, dy, dz);
      const int na = a + dx, nb = b + dy, nc = c + dz;
      if (!F.in(na, nb, nc)) continue;
      if (na / 3 != I || nb / 3 != J || nc / 3 != K) continue;
      const long long q = F.id(na, nb, nc);
      const double* v = val + (long long)o * BF * BF * F.N + p;
      for (int r = 0; r < BF; ++r)
        for (int t = 0; t < BC; ++t) {
          double z = 0.0;
          for (int u = 0; u < BF; ++u) z += v[(long long)(r * BF + u) * F.N] * Pt[(long long)(u * BC + t) * F.N + q];
          ap[r * BC + t] += z;
        }
    }
    for (int r = 0; r < BF; ++r)
      for (int t = 0; t < BC; ++t) {
        double z = 0.0;
        for (int u = 0; u < BF; ++u) z += dinv[(long long)(r * BF + u) * F.N + p] * ap[u * BC + t];
        out[r * BC + t] = -omega * z;
      }
    if (a / 3 == I && b / 3 == J && c / 3 == K)
      for (int q = 0; q < BF * BC; ++q) out[q] += Pt[(long long)q * F.N + p];
  }
  for (int q = 0; q < BF * BC; ++q) P[((long long)s * BF * BC + q) * F.N + p] = out[q];
}

// Galerkin faces -> cells: A_1[T, T'] = sum_{f in T, g} pw_f C_fg pw_g [T' adjacent to g]
__global__ void k_rap_faces(FaceTopo d, const int* __restrict__ col, const double* __restrict__ C,
                            const double* __restrict__ pw, double* __restrict__ A1, unsigned char* __restrict__ act) {
  const long long Tc = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (Tc >= d.nT) return;
  const int i = (int)(Tc % d.nx), j = (int)((Tc / d.nx) % d.ny), k = (int)(Tc / ((long long)d.nx * d.ny));
  double acc[25];
  for (int q = 0; q < 25; ++q) acc[q] = 0.0;
  bool any = false;
  for (int lf = 0; lf < 6; ++lf) {
    const long long f = ft_cell_face(d, i, j, k, lf);
    const double wf = pw[f];
    if (wf == 0.0) continue;
    any = true;
    for (int q = 0; q < 11; ++q) {
      const long long g = col[q * d.nF + f];
      const double v = C[q * d.nF + f];
      const double wg = pw[g];
      if (v == 0.0 || wg == 0.0) continue;
      int cc[2][3];
      const int cnt = ft_face_cells(d, g, cc);
      for (int e = 0; e < cnt; ++e) {
        const int o = St<ST_DIAMOND2>::idx(cc[e][0] - i, cc[e][1] - j, cc[e][2] - k);
        if (o >= 0) acc[o] += wf * v * wg;
      }
    }
  }
  act[Tc] = any ? 1 : 0;
  if (!any) acc[12] = 1.0;
  for (int q = 0; q < 25; ++q) A1[(long long)q * d.nT + Tc] = acc[q];
}

// ------------------------------------------------------------------ host helpers
// the face level's topology for the sweeps and transfers (32-bit: nF < 2^31)
FaceTopo32 face_topo(const Ctx& c) {
  if (c.nF >= (1LL << 31) / 11) throw Error{MHFP_ERR_ARG, "too many faces for 32-bit face indexing"};
  return FaceTopo32::make(c.nx, c.ny, c.nz, c.nT, c.nF, c.nFx, c.nFy);
}

// y = b - A x (y = A x when b is null) on a lattice level with schedule sched
template <typename T>
void launch_spmv(Ctx& c, const StructOp& A, int bs, const T* val, const T* rows, const T* x, const T* b, T* y,
                 int sched) {
  sweep_spmv<T>(c.stream, A, bs, val, rows, x, b, y, sched);
}

void level_spmv(Ctx& c, Level& L, const double* x, const double* b, double* y) {
  if (L.faces) {
    k_spmv_ell<double><<<lgrid(grid_for(L.n, 256)), 256, 0, c.stream>>>(face_topo(c), L.ell ? L.ell : c.Cpi, x, b, y,
                                                                         lbytes());
  } else if (L.bs == 3 && !L.rowd) {
    launch_u64(c.stream, lat32_of(L.A), (const double*)L.A.val, (const double*)nullptr, 0.0, x,
               (const double*)nullptr, b, y);
  } else {
    launch_spmv<double>(c, L.A, L.bs, L.A.val, L.rowd, x, b, y, default_schedule(L.A, L.rowd != nullptr, false));
  }
  MHFP_LAUNCH_CHECK();
}

void alloc_work(Ctx& c, Level& L) {
  L.x = dalloc_n<double>(c, L.n);
  L.b = dalloc_n<double>(c, L.n);
  L.r = dalloc_n<double>(c, L.n);
  L.d = dalloc_n<double>(c, L.n);
  L.y = dalloc_n<double>(c, L.n);
}

// rho(D^-1 A) by power iteration from the fixed start vector: two launches
// per iteration and one read at the end (five launches and a read before)
double spectral_radius(Ctx& c, Level& L) {
  const long long n = L.n;
  double* v = L.x;
  double* w = L.y;
  ensure_workspace(c);
  // the partial sums, the block counter and the norms of the last two
  // iterates (scal[4], scal[5], in turn) are the Krylov workspace's
  unsigned* counter = (unsigned*)(c.dflag + 1);
  auto step = [&](const double* dinv, const double* r, double* out, int it) {
    dispatch_bs(L.bs, [&](auto BS) {
      k_power_step<BS.value><<<std::min<unsigned>(grid_for(L.npts, 256), POWER_BLOCKS), 256, 0, c.stream>>>(
          L.npts, dinv, r, out, c.scal + 4 + (it + 1) % 2, c.scal + 4 + it % 2, c.partials, counter);
    });
    MHFP_LAUNCH_CHECK();
  };
  k_power_start<<<grid_for(n, 256), 256, 0, c.stream>>>(n, v);
  MHFP_LAUNCH_CHECK();
  step(nullptr, v, nullptr, 0);
  for (int it = 0; it < c.opt.power_iters; ++it) {
    level_spmv(c, L, v, nullptr, L.r);
    step(L.dinv, L.r, w, it + 1);
    std::swap(v, w);
  }
  double h = 0.0;
  MHFP_CUDA(cudaMemcpyAsync(&h, c.scal + 4 + c.opt.power_iters % 2, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  MHFP_CUDA(cudaStreamSynchronize(c.stream));
  return h;
}

// Dense inverse of the coarsest level by block Gauss-Jordan elimination in
// place on the GPU (FP64, row-major).  The coarse operators are Galerkin
// products of SPD operators (Dirichlet rows carry a unit diagonal): elimination
// needs no pivoting, and with E the eliminated indices M[j][i] is M[i][j] if
// both or neither are in E and -M[i][j] otherwise, so only the upper triangle
// is kept until the end.  A pivot that is not positive and finite sets *err and
// the host reports a singular level.  GJ_B columns (k0 .. k0 + nb - 1) take
// three kernels: D = the diagonal block's inverse, the panels, and the rank-GJ_B
// update of the other tiles; n^3 / 2 FMA in all.  An SM has two FP64 FMA a
// clock, so even one block's product is long: D takes its reciprocal once per
// column, and tiles of 32 x 32 spread the update over the chip at the default
// sizes (n up to 375).  Column by column on [A | I] it took 1.5 n^3 FMA, two
// launches per column and a pass over the matrix for each: the two levels of a
// 64^3 set-up with coarse_max 512 (1,536 and 512 unknowns) 24.8 -> 5.9 ms of
// kernels, that set-up 52 -> 17.4 ms with the launches saved.
constexpr int GJ_B = 32;                      // columns per step, and the update's tile
constexpr int GJ_TRI = GJ_B * (GJ_B + 1) / 2;  // entries of D's upper triangle

__global__ void __launch_bounds__(GJ_TRI + 16) k_gj_diag(int n, int k0, const double* __restrict__ M,
                                                         double* __restrict__ D, int* __restrict__ err) {
  __shared__ double S[GJ_B][GJ_B + 1], row[GJ_B], inv;
  const int nb = min(GJ_B, n - k0), t = threadIdx.x;
  const bool on = t < GJ_TRI;
  int r = 0, q = t;  // entry t of the triangle: row r, column q >= r
  if (on)
    for (; q >= GJ_B; ++r) q += r + 1 - GJ_B;  // row r + 1 starts at its diagonal
  else
    q = 0;
  if (on) S[r][q] = q < nb ? M[(size_t)(k0 + r) * n + k0 + q] : (r == q ? 1.0 : 0.0);
  __syncthreads();
  for (int c = 0; c < nb; ++c) {
    if (t < GJ_B) {
      // row c times the reciprocal pivot; the eliminated columns' sign flips
      const double p = S[c][c], ip = 1.0 / p;
      if (t == 0) {
        if (!(p > 0.0 && p < 1e300)) *err = 1;
        inv = ip;
      }
      row[t] = (t < c ? -S[t][c] : S[c][t]) * ip;
    }
    __syncthreads();
    double v = 0.0;
    if (on) {
      const double fr = r <= c ? S[r][c] : S[c][r];
      v = r == c ? (q == c ? inv : row[q]) : (q == c ? -fr * inv : fma(-fr, row[q], S[r][q]));
    }
    __syncthreads();
    if (on) S[r][q] = v;
    __syncthreads();
  }
  if (on) D[r * GJ_B + q] = D[q * GJ_B + r] = S[r][q];
}

// V[u][j] = M[k0 + u][j] up to the sign, from the upper triangle, and
// R[u][j] = (D M_k)[u][j] (D itself in the block's own columns).  A block takes
// 32 columns and eight rows of R; those of blockIdx.y = 0 write V.
__global__ void __launch_bounds__(256) k_gj_panel(int n, int k0, const double* __restrict__ M,
                                                  const double* __restrict__ D, double* __restrict__ R,
                                                  double* __restrict__ V) {
  __shared__ double sD[8][GJ_B], sV[GJ_B][GJ_B + 1];
  const int nb = min(GJ_B, n - k0), j0 = blockIdx.x * GJ_B, u0 = blockIdx.y * 8;
  const int q = threadIdx.x & 31, w = threadIdx.x >> 5, j = j0 + q;
  // k0 is a multiple of 32: a block's columns lie left of the pivot block, in
  // it, or to its right
  const bool left = j0 < k0, own = j0 == k0;
  sD[w][q] = D[(u0 + w) * GJ_B + q];
  for (int x = w; x < GJ_B; x += 8) {
    if (left) sV[q][x] = q < nb ? M[(size_t)(j0 + x) * n + k0 + q] : 0.0;
    else sV[x][q] = x < nb && j < n && !own ? M[(size_t)(k0 + x) * n + j] : 0.0;
  }
  __syncthreads();
  if (j >= n) return;
  if (blockIdx.y == 0)
    for (int x = w; x < GJ_B; x += 8) V[(size_t)x * n + j] = sV[x][q];
  double s = 0.0;
  if (own) {
    s = sD[w][q];
  } else {
#pragma unroll 8
    for (int x = 0; x < GJ_B; ++x) s = fma(sD[w][x], sV[x][q], s);
    if (left) s = -s;
  }
  R[(size_t)(u0 + w) * n + j] = u0 + w < nb ? s : 0.0;
}

// upper tiles: rows outside the block M = (0 in the block's columns, M
// elsewhere) - V^T R, rows of the block M = R
__global__ void __launch_bounds__(256) k_gj_update(int n, int k0, double* __restrict__ M, const double* __restrict__ R,
                                                   const double* __restrict__ V) {
  __shared__ double sV[GJ_B][GJ_B], sR[GJ_B][GJ_B];
  const int i0 = blockIdx.y * GJ_B, j0 = blockIdx.x * GJ_B;
  if (i0 > j0) return;
  const int q = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int u = w; u < GJ_B; u += 8) {
    sV[u][q] = i0 + q < n ? V[(size_t)u * n + i0 + q] : 0.0;
    sR[u][q] = j0 + q < n ? R[(size_t)u * n + j0 + q] : 0.0;
  }
  __syncthreads();
  double acc[4] = {0.0, 0.0, 0.0, 0.0};  // rows i0 + w + 8 a, column j0 + q
  if (i0 != k0) {
#pragma unroll 8
    for (int u = 0; u < GJ_B; ++u) {
      const double rv = sR[u][q];
#pragma unroll
      for (int a = 0; a < 4; ++a) acc[a] = fma(sV[u][w + 8 * a], rv, acc[a]);
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = i0 + w + 8 * a, j = j0 + q;
    if (i >= n || j >= n) continue;
    double* m = M + (size_t)i * n + j;
    *m = i0 == k0 ? sR[w + 8 * a][q] : (j0 == k0 ? 0.0 : *m) - acc[a];
  }
}

// the lower triangle from the upper
__global__ void __launch_bounds__(256) k_gj_mirror(int n, double* __restrict__ M) {
  __shared__ double t[GJ_B][GJ_B + 1];
  const int i0 = blockIdx.y * GJ_B, j0 = blockIdx.x * GJ_B;
  if (i0 > j0) return;
  const int q = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int x = w; x < GJ_B; x += 8)
    if (i0 + x < n && j0 + q < n) t[x][q] = M[(size_t)(i0 + x) * n + j0 + q];
  __syncthreads();
  for (int x = w; x < GJ_B; x += 8) {
    const int j = j0 + x, i = i0 + q;  // entry (j, i) below the diagonal
    if (j < n && i < j) M[(size_t)j * n + i] = t[q][x];
  }
}

// Galerkin scratch of the set-up: one buffer for every level of a handle's
// hierarchies (the first level of the first one needs the most), given back
// when the scope that builds them ends, also by an exception
void release_setup_scratch(Ctx& c) {
  if (!c.setup_Q) return;
  void* q = c.setup_Q;
  c.setup_Q = nullptr;
  c.setup_Q_elems = 0;
  MHFP_CUDA(cudaStreamSynchronize(c.stream));  // its last kernel may still run
  dfree(c, q);
}
struct SetupScratch {
  Ctx& c;
  ~SetupScratch() {
    try {
      release_setup_scratch(c);
    } catch (...) {  // stays with the handle; the next check reports the device's error
    }
  }
};
double* setup_scratch(Ctx& c, size_t elems) {
  if (c.setup_Q_elems < elems) {
    release_setup_scratch(c);
    c.setup_Q = (double*)dalloc_own(c, elems * sizeof(double));
    c.setup_Q_elems = elems;
  }
  return c.setup_Q;
}
// the coarsest level's matrix (zeroed before): a row's stencil offsets have
// distinct columns, so the stores are plain
__global__ void k_gj_lattice(Lat L, int kind, int no, int bs, const double* __restrict__ val, double* __restrict__ M) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= L.N * no) return;
  const int o = (int)(t / L.N);
  const long long p = t - (long long)o * L.N;
  int i, j, k, dx, dy, dz;
  L.ijk(p, i, j, k);
  stencil_offset(kind, o, dx, dy, dz);
  if (!L.in(i + dx, j + dy, k + dz)) return;
  const long long q = L.id(i + dx, j + dy, k + dz), w = bs * L.N;
  for (int r = 0; r < bs; ++r)
    for (int s = 0; s < bs; ++s) M[(bs * p + r) * w + bs * q + s] = val[((long long)o * bs * bs + r * bs + s) * L.N + p];
}
// face rows (absent cells' slots name the row's own face with value 0)
__global__ void k_gj_faces(int n, const int* __restrict__ col, const double* __restrict__ val, double* __restrict__ M) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= n) return;
  for (int q = 0; q < 11; ++q) M[(long long)f * n + col[(long long)q * n + f]] += val[(long long)q * n + f];
}

// The dense inverse of the coarsest level, formed in L.dense_inv.  On a
// rebuild (permeability update) the panels are the handle's persistent ones
// (allocated once); otherwise they are the set-up's scratch.
void make_dense_coarse(Ctx& c, Level& L) {
  const int n = (int)L.n;
  const bool rebuild = L.dense_inv != nullptr;
  if (!rebuild) L.dense_inv = dalloc_n<double>(c, (size_t)n * n);
  const size_t elems = 2 * (size_t)GJ_B * n + GJ_B * GJ_B + 1;
  if (rebuild && c.gj_n < n) {
    c.gj_M = dalloc_n<double>(c, elems);
    c.gj_n = n;
  }
  double* R = rebuild ? c.gj_M : setup_scratch(c, elems);
  double* V = R + (size_t)GJ_B * n;
  double* D = V + (size_t)GJ_B * n;
  int* err = (int*)(D + GJ_B * GJ_B);
  double* M = L.dense_inv;
  MHFP_CUDA(cudaMemsetAsync(err, 0, sizeof(int), c.stream));
  MHFP_CUDA(cudaMemsetAsync(M, 0, (size_t)n * n * sizeof(double), c.stream));
  if (L.faces)
    k_gj_faces<<<grid_for(n, 128), 128, 0, c.stream>>>(n, c.ell_col, c.Cpi, M);
  else
    k_gj_lattice<<<grid_for(L.A.N * L.A.noff(), 128), 128, 0, c.stream>>>(lat_of(L.A), L.A.kind, L.A.noff(), L.A.bs,
                                                                          L.A.val, M);
  MHFP_LAUNCH_CHECK();
  const unsigned tiles = grid_for(n, GJ_B);
  for (int k0 = 0; k0 < n; k0 += GJ_B) {
    k_gj_diag<<<1, GJ_TRI + 16, 0, c.stream>>>(n, k0, M, D, err);
    MHFP_LAUNCH_CHECK();
    k_gj_panel<<<dim3(tiles, GJ_B / 8), 256, 0, c.stream>>>(n, k0, M, D, R, V);
    MHFP_LAUNCH_CHECK();
    k_gj_update<<<dim3(tiles, tiles), 256, 0, c.stream>>>(n, k0, M, R, V);
    MHFP_LAUNCH_CHECK();
  }
  k_gj_mirror<<<dim3(tiles, tiles), 256, 0, c.stream>>>(n, M);
  MHFP_LAUNCH_CHECK();
  int h_err = 0;
  MHFP_CUDA(cudaMemcpyAsync(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
  MHFP_CUDA(cudaStreamSynchronize(c.stream));
  if (h_err) throw Error{MHFP_ERR_ARG, "singular or indefinite coarsest multigrid level"};
}

// the Chebyshev recurrence's coefficients on [lmax / ratio, lmax]: step 0 is d
// = (1 / theta) D^-1 r, step s > 0 is d = cd d + cr D^-1 r.  They travel as a
// kernel argument: no copy from host memory that the stream would have to be
// waited for, in every level of a set-up and of a permeability update.
constexpr int CHEB_STEPS = 8;
struct ChebCoefficients {
  double v[2 * CHEB_STEPS];
};
__global__ void k_cheb_coefficients(ChebCoefficients h, double* __restrict__ cf, float* __restrict__ cff) {
  const int i = threadIdx.x;
  cf[i] = h.v[i];
  cff[i] = narrow(h.v[i]);
}

void write_cheb_coefficients(Ctx& c, Level& L) {
  const double lmin = L.lmax / c.opt.cheb_ratio;
  const double theta = 0.5 * (L.lmax + lmin), delta = 0.5 * (L.lmax - lmin), sigma = theta / delta;
  ChebCoefficients h;
  double rho = 1.0 / sigma;
  h.v[0] = 0.0;
  h.v[1] = 1.0 / theta;
  for (int s = 1; s < CHEB_STEPS; ++s) {
    const double rn = 1.0 / (2.0 * sigma - rho);
    h.v[2 * s] = rn * rho;
    h.v[2 * s + 1] = 2.0 * rn / delta;
    rho = rn;
  }
  if (!L.cf) L.cf = dalloc_n<double>(c, 2 * CHEB_STEPS);
  if (!L.cff) L.cff = dalloc_n<float>(c, 2 * CHEB_STEPS);
  k_cheb_coefficients<<<1, 2 * CHEB_STEPS, 0, c.stream>>>(h, L.cf, L.cff);
  MHFP_LAUNCH_CHECK();
}

void finish_level(Ctx& c, Level& L) {
  if (!L.dinv) L.dinv = dalloc_n<double>(c, (size_t)L.bs * L.bs * L.npts);
  if (L.faces) {
    k_dinv_ell<<<grid_for(L.n, 256), 256, 0, c.stream>>>(L.n, L.ell ? L.ell : c.Cpi, L.dinv);
  } else {
    const Lat lat = lat_of(L.A);
    dispatch_bs(L.bs, [&](auto BS) {
      dispatch_kind_bs<BS.value>(L.A.kind, [&](auto K) {
        k_dinv<BS.value, K.value><<<grid_for(lat.N, 256), 256, 0, c.stream>>>(lat, L.A.val, L.dinv);
      });
    });
  }
  MHFP_LAUNCH_CHECK();
  if (!L.faces && row_level(L.A)) {
    if (!L.rowd) L.rowd = dalloc_n<double>(c, sweep_row_elems<double>(L.A, L.bs));
    sweep_pack_rows<double>(c.stream, L.A, L.bs, L.A.val, L.rowd);
    MHFP_LAUNCH_CHECK();
  }
  L.lmax = 1.1 * spectral_radius(c, L);
  write_cheb_coefficients(c, L);
}

// the transfer kernels index the prolongator [slot][entry][fine point] in
// 32-bit unsigned arithmetic: refuse levels where that would wrap
void check_transfer_index(long long rows, long long n) {
  if (rows * n >= (1LL << 32)) throw Error{MHFP_ERR_ARG, "level too large for 32-bit transfer indexing"};
}

// one smoothed-aggregation coarsening step of a lattice level.  With
// `into` (a permeability update), the next level already exists and its
// values, its activity mask and L's prolongator are recomputed in place,
// with the handle's persistent Galerkin scratch.
Level coarsen(Ctx& c, Level& L, Level* into = nullptr) {
  const StructOp& A = L.A;
  const int R = stencil_radius(A.kind);
  L.R = R;
  L.cbs = L.bs;
  Level Cl;
  if (into) Cl = *into;
  Cl.bs = L.bs;
  Cl.A.Lx = (A.Lx + 2) / 3; Cl.A.Ly = (A.Ly + 2) / 3; Cl.A.Lz = (A.Lz + 2) / 3;
  Cl.A.N = (long long)Cl.A.Lx * Cl.A.Ly * Cl.A.Lz;
  Cl.A.bs = L.bs;
  Cl.A.kind = (R == 1) ? ST_BOX1 : ST_BOX2;
  Cl.npts = Cl.A.N;
  Cl.n = Cl.A.N * L.bs;
  Cl.R = stencil_radius(Cl.A.kind);
  const Lat F = lat_of(A), Cc = lat_of(Cl.A);
  const int ns = p_slots(R), nq = q_slots(R);
  const int bs2 = L.bs * L.bs;
  check_transfer_index((long long)ns * ns * ns * bs2, F.N);
  if (!L.P) L.P = dalloc_n<double>(c, (size_t)ns * ns * ns * bs2 * F.N);
  if (!Cl.active) Cl.active = dalloc_n<unsigned char>(c, Cl.n);
  if (!Cl.A.val) Cl.A.val = dalloc_n<double>(c, (size_t)Cl.A.noff() * bs2 * Cc.N);
  const size_t q_elems = (size_t)nq * nq * nq * bs2 * F.N;
  double* Q = nullptr;
  if (into) {
    if (c.upd_Q_elems < q_elems) {
      c.upd_Q = dalloc_n<double>(c, q_elems);
      c.upd_Q_elems = q_elems;
    }
    Q = c.upd_Q;
  } else {
    Q = setup_scratch(c, q_elems);
  }
  const double omega = 4.0 / (3.0 * L.lmax);
  {
    dispatch_bs13(L.bs, [&](auto BS) {
      dispatch_kind_bs<BS.value>(A.kind, [&](auto K) {
        k_build_P<BS.value, K.value><<<grid_for(F.N * ns * ns * ns, 256), 256, 0, c.stream>>>(F, Cc, A.val, L.dinv,
                                                                                             L.active, omega, L.P);
        MHFP_LAUNCH_CHECK();
        k_active_coarse<BS.value><<<grid_for(Cc.N, 256), 256, 0, c.stream>>>(F, Cc, L.active, Cl.active);
        MHFP_LAUNCH_CHECK();
        if constexpr (BS.value == 3) {
          const Lat32 F32 = lat32_of(A), C32 = lat32_of(Cl.A);
          k_build_Q3<<<(unsigned)((F32.Lx + 95) / 96) * (unsigned)(A.Ly * A.Lz), 288, 0, c.stream>>>(F32, C32, A.val,
                                                                                                  L.P, Q);
        } else {
          // rows of slots once they give every SM a block: 8,000 points of 25
          // offsets 28 us against 37; 343 points of 125 offsets 60 against 41
          if (F.N * nq * nq >= 152LL * 256)
            k_build_Q1<K.value><<<grid_for(F.N * nq * nq, 256), 256, 0, c.stream>>>(F, Cc, A.val, L.P, Q);
          else
            k_build_Q<1, 1, K.value><<<grid_for(F.N * nq * nq * nq, 256), 256, 0, c.stream>>>(F, Cc, A.val, L.P, Q);
        }
        MHFP_LAUNCH_CHECK();
      });
      // coarse levels of the 27-point displacement lattice stay 27-point; the
      // scalar levels become 125-point
      if constexpr (BS.value == 3)
        k_rap<BS.value, BS.value, ST_BOX1><<<grid_for(Cc.N * 14, 128), 128, 0, c.stream>>>(F, Cc, R, L.P, Q,
                                                                                           Cl.active, Cl.A.val);
      else
        k_rap<BS.value, BS.value, ST_BOX2><<<grid_for(Cc.N * 63, 128), 128, 0, c.stream>>>(F, Cc, R, L.P, Q,
                                                                                             Cl.active, Cl.A.val);
      MHFP_LAUNCH_CHECK();
    });
  }
  return Cl;
}

void build_u_level0(Ctx& c) {
  c.hu.clear();
  Level L0;
  L0.bs = 3;
  L0.A = c.Auu;
  L0.npts = c.nN;
  L0.n = c.nU;
  L0.R = 1;
  L0.active = dalloc_n<unsigned char>(c, c.nU);
  k_active_fine<<<grid_for(c.nU, 256), 256, 0, c.stream>>>(c.nU, c.node_fix, L0.active);
  MHFP_LAUNCH_CHECK();
  c.hu.push_back(L0);
}

void build_u(Ctx& c) {
  build_u_level0(c);
  while (c.hu.back().npts > c.opt.coarse_max && c.hu.size() < 8) {
    Level& L = c.hu.back();
    alloc_work(c, L);
    finish_level(c, L);
    Level Cl = coarsen(c, L);
    c.hu.push_back(Cl);
  }
  Level& last = c.hu.back();
  alloc_work(c, last);
  make_dense_coarse(c, last);
}

// The displacement hierarchy of M_III^(h): the same aggregates, with the six
// rigid-body modes as the near-kernel.  Level 0 is A_uu (3 dofs per node);
// every coarse point carries 6 dofs (a mode its aggregate cannot represent
// leaves an inactive dof with a unit diagonal).  P = (I - omega D^-1 A) P_t
// with P_t the Gram-Schmidt factors of the aggregates, Galerkin coarse
// operators in the same two gather passes as M_II^(h).
void build_u_rbm(Ctx& c) {
  build_u_level0(c);
  // centroid of the nodes (the rotations' axis point), summed in node order
  double cen[3] = {0, 0, 0};
  {
    std::vector<double> xyz(3 * c.nN);
    MHFP_CUDA(cudaMemcpyAsync(xyz.data(), c.coords, xyz.size() * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
    MHFP_CUDA(cudaStreamSynchronize(c.stream));
    for (long long p = 0; p < c.nN; ++p)
      for (int a = 0; a < 3; ++a) cen[a] += xyz[3 * p + a];
    for (int a = 0; a < 3; ++a) cen[a] /= (double)c.nN;
  }
  const double* Nprev = nullptr;
  while (c.hu.back().npts > c.opt.coarse_max && c.hu.size() < 8) {
    Level& L = c.hu.back();
    alloc_work(c, L);
    finish_level(c, L);
    const int BFv = L.bs;
    const StructOp& A = L.A;
    L.R = 1;
    L.cbs = RBM_K;
    Level Cl;
    Cl.bs = RBM_K;
    Cl.A.Lx = (A.Lx + 2) / 3; Cl.A.Ly = (A.Ly + 2) / 3; Cl.A.Lz = (A.Lz + 2) / 3;
    Cl.A.N = (long long)Cl.A.Lx * Cl.A.Ly * Cl.A.Lz;
    Cl.A.bs = RBM_K;
    Cl.A.kind = ST_BOX1;
    Cl.npts = Cl.A.N;
    Cl.n = Cl.A.N * RBM_K;
    Cl.R = 1;
    const Lat F = lat_of(A), Cc = lat_of(Cl.A);
    const int ns = p_slots(1), nq = q_slots(1);
    const int pb = BFv * RBM_K;
    double* Pt = dalloc_n<double>(c, (size_t)pb * F.N);
    double* Nc = dalloc_n<double>(c, (size_t)RBM_K * RBM_K * Cc.N);
    Cl.active = dalloc_n<unsigned char>(c, Cl.n);
    check_transfer_index((long long)ns * ns * ns * pb, F.N);
    L.P = dalloc_n<double>(c, (size_t)ns * ns * ns * pb * F.N);
    Cl.A.val = dalloc_n<double>(c, (size_t)27 * RBM_K * RBM_K * Cc.N);
    MHFP_CUDA(cudaMemsetAsync(Pt, 0, (size_t)pb * F.N * sizeof(double), c.stream));
    const double omega = 4.0 / (3.0 * L.lmax);
    double* Q = setup_scratch(c, (size_t)nq * nq * nq * pb * F.N);
    {
      const unsigned warps = grid_for(Cc.N * 32, 128);
      auto galerkin = [&](auto BF) {
        constexpr int bf = decltype(BF)::value;
        k_build_P_t<bf, RBM_K, ST_BOX1><<<grid_for(F.N * ns * ns * ns, 256), 256, 0, c.stream>>>(F, Cc, A.val, L.dinv,
                                                                                                 Pt, omega, L.P);
        MHFP_LAUNCH_CHECK();
        k_build_Q<bf, RBM_K, ST_BOX1><<<grid_for(F.N * nq * nq * nq, 256), 256, 0, c.stream>>>(F, Cc, A.val, L.P, Q);
        MHFP_LAUNCH_CHECK();
        k_rap<bf, RBM_K, ST_BOX1><<<grid_for(Cc.N * 14, 128), 128, 0, c.stream>>>(F, Cc, 1, L.P, Q, Cl.active,
                                                                                   Cl.A.val);
        MHFP_LAUNCH_CHECK();
      };
      if (BFv == 3) {
        k_rbm_tentative<3, 3><<<warps, 128, 0, c.stream>>>(F, Cc, c.coords, L.active, nullptr, cen[0], cen[1], cen[2],
                                                           Pt, Nc, Cl.active);
        MHFP_LAUNCH_CHECK();
        galerkin(std::integral_constant<int, 3>{});
      } else {
        k_rbm_tentative<RBM_K, 6><<<warps, 128, 0, c.stream>>>(F, Cc, c.coords, L.active, Nprev, cen[0], cen[1],
                                                               cen[2], Pt, Nc, Cl.active);
        MHFP_LAUNCH_CHECK();
        galerkin(std::integral_constant<int, RBM_K>{});
      }
    }
    Nprev = Nc;
    c.hu.push_back(Cl);
  }
  Level& last = c.hu.back();
  alloc_work(c, last);
  make_dense_coarse(c, last);
}

void build_pi(Ctx& c) {
  c.hpi.clear();
  Level L0;
  L0.faces = true;
  L0.bs = 1;
  L0.npts = c.nF;
  L0.n = c.nF;
  c.hpi.push_back(L0);
  if (c.nF <= c.opt.coarse_max) {
    alloc_work(c, c.hpi.back());
    make_dense_coarse(c, c.hpi.back());
    return;
  }
  {
    Level& F = c.hpi.back();
    alloc_work(c, F);
    finish_level(c, F);
    Level L1;
    L1.bs = 1;
    L1.A.Lx = c.nx; L1.A.Ly = c.ny; L1.A.Lz = c.nz;
    L1.A.N = c.nT; L1.A.bs = 1; L1.A.kind = ST_DIAMOND2;
    L1.npts = c.nT; L1.n = c.nT; L1.R = 2;
    L1.A.val = dalloc_n<double>(c, (size_t)25 * c.nT);
    L1.active = dalloc_n<unsigned char>(c, c.nT);
    k_rap_faces<<<grid_for(c.nT, 128), 128, 0, c.stream>>>(FaceTopo{c.nx, c.ny, c.nz, c.nT, c.nF, c.nFx, c.nFy},
                                                           c.ell_col, c.Cpi, c.pw, L1.A.val, L1.active);
    MHFP_LAUNCH_CHECK();
    c.hpi.push_back(L1);
  }
  while (c.hpi.back().npts > c.opt.coarse_max && c.hpi.size() < 8) {
    Level& L = c.hpi.back();
    alloc_work(c, L);
    finish_level(c, L);
    Level Cl = coarsen(c, L);
    c.hpi.push_back(Cl);
  }
  Level& last = c.hpi.back();
  alloc_work(c, last);
  make_dense_coarse(c, last);
}

// coarse points below which the restriction takes four warps each (at one
// warp, on the set-up's layout, 1,040 points of a 3 x 3 FP64 level took 11.1 us
// instead of 7.5, 4,096 points of a 6 x 6 level 16.2 instead of 4.4)
constexpr long long RESTRICT_WIDE = 6000;
// fine points from which the prolongation takes its wide forms (k_prolong_f, k_prolong_s)
constexpr long long PROLONG_WIDE = 65536;

// (re)write a level's prolongator in the cycles' layout and precision
template <typename T>
void pack_P(Ctx& c, const Level& L, const Level& C, T* Pc) {
  const Lat32 F = lat32_of(L.A), Cc = lat32_of(C.A);
  dispatch_pair(L.bs, C.bs, [&](auto BF, auto BC) {
    constexpr int R = transfer_r<BF.value>();
    k_pack_P<BF.value * BC.value, R, T>
        <<<(unsigned)(C.A.N * ((Box<R>::WP + 127) / 128)), 128, 0, c.stream>>>(F, Cc, L.P, Pc);
  });
  MHFP_LAUNCH_CHECK();
}
size_t setup_P_size(const Level& L) {
  const size_t ns = (size_t)p_slots(L.R);
  return ns * ns * ns * L.bs * L.cbs * L.npts;
}
size_t packed_P_size(const Level& L, const Level& C) {
  return (size_t)C.A.N * L.bs * C.bs * (L.bs == 1 ? Box<2>::WP : Box<1>::WP);
}

// the FP64 cycles' prolongators (allocated on the first call)
void make_fp64_transfers(Ctx& c, std::vector<Level>& H) {
  for (size_t l = 0; l + 1 < H.size(); ++l) {
    if (!H[l].P) continue;
    if (!H[l].Pd) H[l].Pd = dalloc_n<double>(c, packed_P_size(H[l], H[l + 1]));
    pack_P<double>(c, H[l], H[l + 1], H[l].Pd);
  }
}

// ------------------------------------------------------------------ V-cycle
// Pointers of one level in the precision T of the cycle: the FP64 arrays
// built by the set-up, or their FP32 copies for the mixed-precision cycle.
template <typename T>
struct LV {
  const T *val, *rows, *dinv, *P, *Pm, *ell, *pw, *cf;  // P: coarse-point major, Pm: fine-point major
  T *r, *d, *y;
};
LV<double> view(Ctx& c, Level& L, double) {
  return {L.A.val, L.rowd, L.dinv, L.Pd, L.P, L.ell ? L.ell : c.Cpi, c.pw, L.cf, L.r, L.d, L.y};
}
LV<float> view(Ctx& c, Level& L, float) { return {L.valf, L.rowf, L.dinvf, L.Pf, L.Pmf, c.Cpif, c.pwf, L.cff, L.rf, L.df, L.yf}; }
double* bvec(Level& L, double) { return L.b; }
float* bvec(Level& L, float) { return L.bf; }
double* xvec(Level& L, double) { return L.x; }
float* xvec(Level& L, float) { return L.xf; }

template <typename T>
void level_spmv_t(Ctx& c, Level& L, const T* x, const T* b, T* y) {
  const LV<T> v = view(c, L, T());
  if (L.faces) {
    k_spmv_ell<T><<<lgrid(grid_for(L.n, 256)), 256, 0, c.stream>>>(face_topo(c), v.ell, x, b, y, lbytes());
  } else {
    launch_spmv<T>(c, L.A, L.bs, v.val, v.rows, x, b, y, L.tpp ? L.tpp : default_schedule(L.A, v.rows != nullptr, sizeof(T) == 4));
  }
  MHFP_LAUNCH_CHECK();
}

// one Chebyshev sweep on a lattice level with schedule sched (the first
// sweep from zero has no stencil work and always runs one point per thread)
template <typename T>
void launch_cheb(Ctx& c, Level& L, const LV<T>& v, const T* b, const T* xin, T* out, int step, int sched) {
  if (!xin) {
    sweep_cheb_zero<T>(c.stream, L.A.N, L.bs, v.dinv, b, out, v.d, v.cf);
    return;
  }
  sweep_cheb<T>(c.stream, L.A, L.bs, v.val, v.rows, v.dinv, b, xin, out, v.d, v.cf + 2 * step, step == 0, sched);
}

// The symmetric FP32 sweep and residual of the finest displacement level
// with L.tpp resident blocks per SM (6 or 8; 0: 8 when one wave of 8 blocks
// of 256 per SM covers the level, else 6).
// schedule of the finest FP32 displacement level: 6 or 8 resident blocks of
// 256 threads per SM (0: 8 when one wave of 8 blocks per SM covers the
// level, else 6)
int sym_minb(const Level& L) {
  if (L.tpp >= 4 && L.tpp <= 8) return L.tpp;
  return L.A.N <= 152LL * 8 * 256 ? 8 : 6;
}

// the bulk-copy-fed variant (schedule 4): persistent CTAs, 4 per SM
void launch_sym_tma(Ctx& c, const Level& L, bool cheb, const float* b, const float* xin, float* xout, float* d,
                    const float* cf, bool first) {
  const Lat lat = lat_of(L.A);
  if (lat.N >= (1LL << 31) - TMA_NB) throw Error{MHFP_ERR_ARG, "level too large for the bulk-copy sweep"};
  const long long nblocks = (lat.N + TMA_NB - 1) / TMA_NB;
  const unsigned grid = (unsigned)std::min<long long>(nblocks, 3LL * c.n_sm);
  static bool attr = false;  // the dynamic shared memory above 48 KB, once per process
  if (!attr) {
    MHFP_CUDA(cudaFuncSetAttribute(k_sym_tma<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TMA_SMEM));
    MHFP_CUDA(cudaFuncSetAttribute(k_sym_tma<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TMA_SMEM));
    attr = true;
  }
  TmaSweep a{L.symf, L.dinvf, b, xin, xout, d, cf, first, c.d_flag};
  if (cheb) k_sym_tma<true><<<lgrid(grid), TMA_THREADS, TMA_SMEM, c.stream>>>(lat, a, lbytes());
  else k_sym_tma<false><<<lgrid(grid), TMA_THREADS, TMA_SMEM, c.stream>>>(lat, a, lbytes());
}
void launch_cheb_sym(Ctx& c, const Level& L, const float* b, const float* xin, float* xout, float* d, const float* cf,
                     bool first) {
  const Lat lat = lat_of(L.A);
  if (!xin) {  // the first step from zero has no stencil work
    sweep_cheb_zero<float>(c.stream, lat.N, 3, L.dinvf, b, xout, d, cf);
    MHFP_LAUNCH_CHECK();
    return;
  }
  const int mb = sym_minb(L);
  if (mb == 4)
    launch_sym_tma(c, L, true, b, xin, xout, d, cf, first);
  else if (mb == 5)
    k_cheb_u0_sym<float, 5><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, L.dinvf, b, xin,
                                                                                xout, d, cf, first, lbytes());
  else if (mb == 7)
    k_cheb_u0_sym<float, 7><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, L.dinvf, b, xin,
                                                                                xout, d, cf, first, lbytes());
  else if (mb == 8)
    k_cheb_u0_sym<float, 8><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, L.dinvf, b, xin,
                                                                                xout, d, cf, first, lbytes());
  else
    k_cheb_u0_sym<float, 6><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, L.dinvf, b, xin,
                                                                                xout, d, cf, first, lbytes());
  MHFP_LAUNCH_CHECK();
}
void launch_resid_sym(Ctx& c, const Level& L, const float* x, const float* b, float* y) {
  const Lat lat = lat_of(L.A);
  const int mb = sym_minb(L);
  if (mb == 4)
    launch_sym_tma(c, L, false, b, x, y, nullptr, nullptr, true);
  else if (mb == 5)
    k_resid_u0_sym<float, 5><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, x, b, y,
                                                                                 lbytes());
  else if (mb == 7)
    k_resid_u0_sym<float, 7><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, x, b, y,
                                                                                 lbytes());
  else if (mb == 8)
    k_resid_u0_sym<float, 8><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, x, b, y,
                                                                                 lbytes());
  else
    k_resid_u0_sym<float, 6><<<lgrid(grid_for(lat.N, 256)), 256, 0, c.stream>>>(lat, L.symf, x, b, y,
                                                                                 lbytes());
  MHFP_LAUNCH_CHECK();
}

// Device time of one call of `body` (which enqueues kernels on c.stream):
// `reps` calls captured once into a CUDA graph on a private stream, the
// graph uploaded and replayed up to four times under events, the fastest
// replay kept (best_replay_us).  Timing graph replays leaves out host launch
// overhead, as in the solve, which runs as graphs.
template <class F>
float graph_time_us(Ctx& c, int reps, float best_us, F&& body) {
  cudaStream_t user = c.stream, st = nullptr;
  MHFP_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
  MHFP_CUDA(cudaStreamSynchronize(user));
  const long long l0 = g_launches;
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ge = nullptr;
  c.stream = st;
  cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    try {
      for (int r = 0; r < reps; ++r) body();
    } catch (...) {
      cudaStreamEndCapture(st, &g);
      if (g) cudaGraphDestroy(g);
      c.stream = user;
      cudaStreamDestroy(st);
      throw;
    }
    e = cudaStreamEndCapture(st, &g);
  }
  c.stream = user;
  g_launches = l0;
  if (e == cudaSuccess) e = cudaGraphInstantiate(&ge, g, 0);
  if (g) cudaGraphDestroy(g);
  if (e == cudaSuccess) e = cudaGraphUpload(ge, st);  // not in the first replay's time
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  const float best = best_replay_us(best_us * reps, [&] {
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventRecord(e0, st);
    if (e == cudaSuccess) e = cudaGraphLaunch(ge, st);
    if (e == cudaSuccess) e = cudaEventRecord(e1, st);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    return 1e3f * ms;
  });
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (ge) cudaGraphExecDestroy(ge);
  cudaStreamDestroy(st);
  MHFP_CUDA(e);
  return best / reps;
}

// sweeps per timed replay: about 40 us of them at 3 TB/s, 2 to 5 (ten
// sweeps, replayed four times whatever the candidate, took 32 of the 122 ms of
// a 96^3 set-up and 14 of 34 ms at 45 x 52 x 39)
int tune_reps(double bytes) { return (int)std::min(5.0, std::max(2.0, 40.0 / (bytes / 3e6))); }

// Set-up autotuner for the finest displacement level in FP32: time the four
// occupancy variants of the symmetric sweep and the bulk-copy-fed one and keep
// the fastest in L.tpp.
void autotune_fine_sym(Ctx& c, Level& L) {
  MHFP_CUDA(cudaMemsetAsync(L.bf, 0, L.n * sizeof(float), c.stream));
  MHFP_CUDA(cudaMemsetAsync(L.xf, 0, L.n * sizeof(float), c.stream));
  MHFP_CUDA(cudaMemsetAsync(L.df, 0, L.n * sizeof(float), c.stream));
  float best = 1e30f;
  int best_minb = 0;
  for (int minb : {8, 7, 6, 5, 4}) {
    L.tpp = minb;
    const float us = graph_time_us(c, tune_reps(4.0 * 126 * L.A.N), best, [&] { launch_cheb_sym(c, L, L.bf, L.xf, L.yf, L.df, L.cff + 2, false); });
    if (us < best) {
      best = us;
      best_minb = minb;
    }
  }
  L.tpp = best_minb;
  L.sweep_us = best;
}

// Set-up autotuner: time the launch schedules of a coarse level's Chebyshev
// sweep (one point per thread; offsets split over 4, 8 or 16 warps: same
// arithmetic up to the order of the partial sums) and keep the fastest for
// this level's sweeps and residuals.
template <typename T>
void autotune_level(Ctx& c, Level& L) {
  const LV<T> v = view(c, L, T());
  T* b = bvec(L, T());
  T* x = xvec(L, T());
  MHFP_CUDA(cudaMemsetAsync(b, 0, L.n * sizeof(T), c.stream));
  MHFP_CUDA(cudaMemsetAsync(x, 0, L.n * sizeof(T), c.stream));
  MHFP_CUDA(cudaMemsetAsync(v.d, 0, L.n * sizeof(T), c.stream));
  float best = 1e30f;
  int best_tpp = default_schedule(L.A, v.rows != nullptr, sizeof(T) == 4);
  // likely winners first: a candidate that has lost is dropped early
  const std::vector<int> cand = v.rows ? std::vector<int>{32, 64, 8, 4, 16} : std::vector<int>{1, 4, 8, 16};
  for (int tpp : cand) {
    const float us = graph_time_us(c, tune_reps((double)sizeof(T) * L.A.noff() * L.bs * L.bs * L.A.N), best, [&] {
      launch_cheb<T>(c, L, v, b, x, v.y, 1, tpp);
      MHFP_LAUNCH_CHECK();
    });
    if (us < best) {
      best = us;
      best_tpp = tpp;
    }
  }
  L.tpp = best_tpp;
  L.sweep_us = best;
}

// Chebyshev smoothing of level l from x0 (null: from zero) into dst.  Each
// step reads neighbours of its input, so it cannot update in place: the
// steps write dst and alt in turn, chosen so that the last one writes dst
// (the first step's output differs from x0 when alt is the buffer that x0
// is not, or x0 is null).
// output buffer of step s of a smoothing into dst that alternates with alt
template <typename T>
T* step_out(int deg, int s, T* dst, T* alt) {
  return ((deg - 1 - s) % 2 == 0) ? dst : alt;
}

// With first_done the first step (from zero, x0 null) was already taken by
// the restriction that produced b (its output in that step's buffer, its
// direction in the level's d): the smoothing goes on from the second step.
template <typename T>
void smooth(Ctx& c, std::vector<Level>& H, int l, const T* b, const T* x0, T* dst, T* alt, bool time_it,
            bool first_done = false) {
  Level& L = H[l];
  const LV<T> v = view(c, L, T());
  const int deg = c.opt.cheb_degree;
  const T* xin = first_done ? step_out(deg, 0, dst, alt) : x0;
  for (int s = first_done ? 1 : 0; s < deg; ++s) {
    T* out = step_out(deg, s, dst, alt);
    if (time_it && xin) timing_begin(c, 0);
    if (L.faces) {
      k_cheb_ell<T><<<lgrid(grid_for(L.n, 256)), 256, 0, c.stream>>>(face_topo(c), v.ell, v.dinv, b, xin, out, v.d,
                                                                     v.cf + 2 * s, s == 0, lbytes());
    } else if (time_it) {
      if constexpr (std::is_same<T, float>::value) {
        launch_cheb_sym(c, L, b, xin, out, v.d, v.cf + 2 * s, s == 0);
      } else {
        const Lat32 lat = lat32_of(L.A);
        if (!xin)  // the first step from zero has no stencil work
          sweep_cheb_zero<T>(c.stream, lat.N, 3, v.dinv, b, out, v.d, v.cf);
        else
          dispatch_u64(lat.N, U64_SPLIT_NODES, U64_ROW_STEP, [&](auto F) {
            constexpr U64Form f = decltype(F)::value;
            k_cheb_u0<f><<<u64_grid<f>(lat.N), u64_block<f>(), 0, c.stream>>>(
                lat, v.val, v.dinv, b, xin, out, v.d, v.cf + 2 * s, s == 0, lbytes());
          });
      }
    } else {
      launch_cheb<T>(c, L, v, b, xin, out, s, L.tpp ? L.tpp : default_schedule(L.A, v.rows != nullptr, sizeof(T) == 4));
    }
    MHFP_LAUNCH_CHECK();
    // algorithmic bytes of a Chebyshev sweep: the matrix values (27 blocks
    // per node in FP64, the 14 stored blocks of the symmetric FP32 copy) and
    // the 3x3 inverse diagonal per node, b, x_in, x_out and d read/written
    const double blocks = std::is_same<T, float>::value ? 14.0 : 27.0;
    if (time_it && xin) timing_end(c, 0, (blocks * 9 + 9) * sizeof(T) * L.npts + 5.0 * sizeof(T) * L.n);
    xin = out;
  }
}

template <typename T>
void vcycle_level(Ctx& c, std::vector<Level>& H, int l, const T* b, T* x, bool pre_done = false) {
  Level& L = H[l];
  const LV<T> v = view(c, L, T());
  if (L.dense_inv) {
    const int n = (int)L.n;
    k_dense_mv<T><<<lgrid((n + 1) / 2), 256, 0, c.stream>>>(n, L.dense_inv, b, x, lbytes());
    MHFP_LAUNCH_CHECK();
    return;
  }
  const bool fine_u = (&H == &c.hu) && l == 0;
  // the pre-smoothed and corrected iterate lives in s_buf, chosen so that the
  // post-smoothing's last step writes x: the level's other work vector when
  // the degree is odd, x itself when it is even (no copy back)
  T* s_buf = (c.opt.cheb_degree % 2 == 1) ? v.y : x;
  smooth<T>(c, H, l, b, nullptr, s_buf, s_buf == x ? v.y : x, fine_u, pre_done);
  if (fine_u) {
    if constexpr (std::is_same<T, float>::value) {
      launch_resid_sym(c, L, s_buf, b, v.r);
    } else {
      launch_u64(c.stream, lat32_of(L.A), v.val, (const double*)nullptr, 0.0, (const double*)s_buf,
                 (const double*)nullptr, b, v.r);
      MHFP_LAUNCH_CHECK();
    }
  } else {
    level_spmv_t<T>(c, L, s_buf, b, v.r);
  }
  Level& C = H[l + 1];
  T* cb = bvec(C, T());
  T* cx = xvec(C, T());
  // the restriction also takes the coarse level's first Chebyshev step from
  // zero (d = cr D^-1 b into that step's buffer), unless it is the dense one
  const bool fuse = !C.dense_inv;
  const LV<T> cv = view(c, C, T());
  const int deg = c.opt.cheb_degree;
  T* cs_buf = (deg % 2 == 1) ? cv.y : cx;
  const T* fdinv = fuse ? cv.dinv : nullptr;
  const T* fcr = fuse ? cv.cf : nullptr;
  T* fx = fuse ? step_out(deg, 0, cs_buf, cs_buf == cx ? cv.y : cx) : nullptr;
  T* fd = fuse ? cv.d : nullptr;
  if (L.faces) {
    k_restrict_faces<T><<<lgrid(grid_for(c.nT, 256)), 256, 0, c.stream>>>(face_topo(c), v.pw, v.r, cb, fdinv, fcr,
                                                                          fx, fd, lbytes());
  } else {
    const Lat32 F = lat32_of(L.A), Cc = lat32_of(C.A);
    dispatch_pair(L.bs, C.bs, [&](auto BF, auto BC) {
      constexpr int R = transfer_r<BF.value>();
      // four warps per coarse point where one each would leave SMs idle, and
      // for the blocks of the rigid-body modes (one box point per lane)
      auto launch = [&](auto W) {
        k_restrict_f<BF.value, BC.value, R, W.value, T><<<lgrid(grid_for(C.A.N, 8 / W.value)), 256, 0, c.stream>>>(
            F, Cc, v.P, v.r, cb, fdinv, fcr, fx, fd, lbytes());
      };
      if constexpr (BF.value * BC.value > 9) {
        launch(std::integral_constant<int, 4>{});
      } else {
        if (C.A.N < RESTRICT_WIDE) launch(std::integral_constant<int, 4>{});
        else launch(std::integral_constant<int, 1>{});
      }
    });
  }
  MHFP_LAUNCH_CHECK();
  vcycle_level<T>(c, H, l + 1, cb, cx, fuse);
  if (L.faces) {
    k_prolong_faces<T><<<lgrid(grid_for(c.nF, 256)), 256, 0, c.stream>>>(face_topo(c), v.pw, cx, s_buf, lbytes());
  } else {
    const Lat32 F = lat32_of(L.A), Cc = lat32_of(C.A);
    dispatch_pair(L.bs, C.bs, [&](auto BF, auto BC) {
      constexpr int R = transfer_r<BF.value>();
      if (L.A.N < PROLONG_WIDE)
        k_prolong_w<BF.value, BC.value, R, T>
            <<<lgrid(grid_for(L.A.N, 32)), dim3(32, Box<R>::ns * Box<R>::ns), 0, c.stream>>>(F, Cc, v.P, cx, s_buf,
                                                                                             lbytes());
      else if constexpr (BF.value == 1)
        k_prolong_s<R, T><<<lgrid(grid_for(L.A.N, 256)), 256, 0, c.stream>>>(F, Cc, v.P, cx, s_buf, lbytes());
      else
        k_prolong_f<BF.value, BC.value, R, T>
            <<<lgrid(grid_for(L.A.N, 32)), dim3(32, Box<R>::ns * Box<R>::ns), 0, c.stream>>>(F, Cc, v.Pm, cx, s_buf,
                                                                                             lbytes());
    });
  }
  MHFP_LAUNCH_CHECK();
  smooth<T>(c, H, l, b, s_buf, x, v.y, fine_u);
}

float* cast_copy(Ctx& c, const double* src, size_t n) {
  float* d = dalloc_n<float>(c, n);
  k_cast_f32<<<grid_for((long long)n, 256), 256, 0, c.stream>>>((long long)n, src, d);
  MHFP_LAUNCH_CHECK();
  return d;
}

// FP32 copies of a hierarchy built in FP64 (the last level keeps its FP64
// dense inverse).  With fine_sym, level 0 (the finest displacement level,
// 27-point 3x3-block stencil) keeps only its symmetric half: the diagonal
// block and the 13 offsets after it, the last 14 x 9 x N values of the
// offset-major FP64 array.
void make_fp32(Ctx& c, std::vector<Level>& H, bool fine_sym) {
  for (size_t l = 0; l < H.size(); ++l) {
    Level& L = H[l];
    const size_t bs2 = (size_t)L.bs * L.bs;
    if (fine_sym && l == 0 && !L.dense_inv) {
      const long long N = L.A.N;
      // node-blocked: ceil(N / 32) blocks of 126 x 32 values, plus 8 zeroed
      // blocks that the bulk-copy sweep's last node block reads past the end
      const size_t sym_elems = (size_t)((N + 31) / 32 + TMA_NW) * 126 * 32;
      L.symf = dalloc_n<float>(c, sym_elems);
      MHFP_CUDA(cudaMemsetAsync(L.symf, 0, sym_elems * sizeof(float), c.stream));
      k_cast_f32_sym<<<grid_for(126 * N, 256), 256, 0, c.stream>>>(N, L.A.val + 13 * 9 * N, L.symf);
      MHFP_LAUNCH_CHECK();
    } else if (!L.faces) {
      L.valf = cast_copy(c, L.A.val, (size_t)L.A.noff() * bs2 * L.A.N);
      if (L.rowd) {
        L.rowf = dalloc_n<float>(c, sweep_row_elems<float>(L.A, L.bs));
        sweep_pack_rows<float>(c.stream, L.A, L.bs, L.valf, L.rowf);
        MHFP_LAUNCH_CHECK();
      }
    }
    if (L.dinv) L.dinvf = cast_copy(c, L.dinv, bs2 * L.npts);
    if (L.P) {
      L.Pf = dalloc_n<float>(c, packed_P_size(L, H[l + 1]));
      pack_P<float>(c, L, H[l + 1], L.Pf);
      if (L.bs > 1 && L.A.N >= PROLONG_WIDE) L.Pmf = cast_copy(c, L.P, setup_P_size(L));
    }
    L.xf = dalloc_n<float>(c, L.n);
    L.bf = dalloc_n<float>(c, L.n);
    L.rf = dalloc_n<float>(c, L.n);
    L.df = dalloc_n<float>(c, L.n);
    L.yf = dalloc_n<float>(c, L.n);
  }
}

}  // namespace

void build_hierarchies(Ctx& c) {
  {
    const SetupScratch scratch{c};
    if (c.opt.near_kernel == 1) build_u_rbm(c);
    else build_u(c);
    build_pi(c);
  }
  if (c.opt.precision == 1) {
    make_fp32(c, c.hu, true);
    make_fp32(c, c.hpi, false);
    c.Cpif = cast_copy(c, c.Cpi, (size_t)11 * c.nF);
    c.pwf = cast_copy(c, c.pw, c.nF);
  } else {
    make_fp64_transfers(c, c.hu);
    make_fp64_transfers(c, c.hpi);
  }
  if (c.opt.autotune) {
    // the finest displacement level runs k_cheb_u0 (FP64) or the symmetric
    // FP32 sweep, whose five variants are timed; tune the others
    // (schedules fixed by the options are not tuned)
    if (c.opt.precision == 1 && !c.hu[0].dense_inv && !c.opt.fine_blocks) autotune_fine_sym(c, c.hu[0]);
    for (auto* H : {&c.hu, &c.hpi})
      for (size_t l = 0; l < H->size(); ++l) {
        Level& L = (*H)[l];
        if (L.faces || L.dense_inv || (H == &c.hu && l == 0) || c.opt.schedule) continue;
        if (c.opt.precision == 1) autotune_level<float>(c, L);
        else autotune_level<double>(c, L);
      }
  }
  // schedules forced by the options
  if (c.opt.fine_blocks && c.opt.precision == 1 && !c.hu[0].dense_inv) c.hu[0].tpp = c.opt.fine_blocks;
  if (c.opt.schedule)
    for (auto* H : {&c.hu, &c.hpi})
      for (size_t l = 0; l < H->size(); ++l) {
        Level& L = (*H)[l];
        if (!L.faces && !L.dense_inv && !(H == &c.hu && l == 0)) L.tpp = c.opt.schedule;
      }
}

// The interface-pressure hierarchy after a permeability update: C~_pi has
// new values on the same pattern, so every level keeps its size, buffers
// and launch schedule; the diagonal inverses, lmax, prolongators, Galerkin
// products, dense coarsest inverse and FP32 copies are recomputed in place.
void rebuild_pi_hierarchy(Ctx& c) {
  auto& H = c.hpi;
  if (H.size() == 1) {
    make_dense_coarse(c, H[0]);
  } else {
    finish_level(c, H[0]);
    Level& L1 = H[1];
    k_rap_faces<<<grid_for(c.nT, 128), 128, 0, c.stream>>>(FaceTopo{c.nx, c.ny, c.nz, c.nT, c.nF, c.nFx, c.nFy},
                                                           c.ell_col, c.Cpi, c.pw, L1.A.val, L1.active);
    MHFP_LAUNCH_CHECK();
    for (size_t l = 1; l + 1 < H.size(); ++l) {
      finish_level(c, H[l]);
      H[l + 1] = coarsen(c, H[l], &H[l + 1]);
    }
    make_dense_coarse(c, H.back());
  }
  if (c.opt.precision == 1) {
    auto recast = [&](float* dst, const double* src, size_t n) {
      k_cast_f32<<<grid_for((long long)n, 256), 256, 0, c.stream>>>((long long)n, src, dst);
      MHFP_LAUNCH_CHECK();
    };
    for (size_t l = 0; l < H.size(); ++l) {
      Level& L = H[l];
      const size_t bs2 = (size_t)L.bs * L.bs;
      if (!L.faces && L.valf) recast(L.valf, L.A.val, (size_t)L.A.noff() * bs2 * L.A.N);
      if (L.rowf) {
        sweep_pack_rows<float>(c.stream, L.A, L.bs, L.valf, L.rowf);
        MHFP_LAUNCH_CHECK();
      }
      if (L.dinv && L.dinvf) recast(L.dinvf, L.dinv, bs2 * L.npts);
      if (L.P && L.Pf) pack_P<float>(c, L, H[l + 1], L.Pf);
    }
    recast(c.Cpif, c.Cpi, (size_t)11 * c.nF);
    recast(c.pwf, c.pw, c.nF);
  } else {
    make_fp64_transfers(c, H);
  }
}

namespace {
void build_mixed_levels(Ctx& c) {
  const SetupScratch scratch{c};
  if (c.opt.near_kernel == 1) build_u_rbm(c);
  else build_u(c);
  c.hq.clear();
  Level Q;
  Q.faces = true;
  Q.bs = 1;
  Q.npts = c.nF;
  Q.n = c.nF;
  Q.ell = c.Aqq;
  c.hq.push_back(Q);
  alloc_work(c, c.hq.back());
  finish_level(c, c.hq.back());
  c.hcp.clear();
  Level L0;
  L0.bs = 1;
  L0.A.Lx = c.nx; L0.A.Ly = c.ny; L0.A.Lz = c.nz;
  L0.A.N = c.nT; L0.A.bs = 1; L0.A.kind = ST_DIAMOND2;
  L0.A.val = c.Cp;
  L0.npts = c.nT;
  L0.n = c.nT;
  L0.R = 2;
  L0.active = dalloc_n<unsigned char>(c, c.nT);
  MHFP_CUDA(cudaMemsetAsync(L0.active, 1, c.nT, c.stream));
  c.hcp.push_back(L0);
  while (c.hcp.back().npts > c.opt.coarse_max && c.hcp.size() < 8) {
    Level& L = c.hcp.back();
    alloc_work(c, L);
    finish_level(c, L);
    Level Cl = coarsen(c, L);
    c.hcp.push_back(Cl);
  }
  Level& last = c.hcp.back();
  alloc_work(c, last);
  make_dense_coarse(c, last);
}
}  // namespace

// The mixed formulation's inner solvers (opt.formulation = 1): the
// displacement hierarchy as for the hybrid form, A_qq as a single face level
// (its Chebyshev smoother stands for the paper's incomplete Cholesky), and
// the smoothed-aggregation hierarchy of C~_p started on the cell lattice.
void build_mixed_hierarchies(Ctx& c) {
  build_mixed_levels(c);
  make_fp64_transfers(c, c.hu);
  make_fp64_transfers(c, c.hcp);
  if (c.opt.autotune)
    for (auto* H : {&c.hu, &c.hcp})
      for (size_t l = 0; l < H->size(); ++l) {
        Level& L = (*H)[l];
        if (L.faces || L.dense_inv || (H == &c.hu && l == 0) || c.opt.schedule) continue;
        autotune_level<double>(c, L);
      }
  if (c.opt.schedule)
    for (auto* H : {&c.hu, &c.hcp})
      for (size_t l = 0; l < H->size(); ++l) {
        Level& L = (*H)[l];
        if (!L.faces && !L.dense_inv && !(H == &c.hu && l == 0)) L.tpp = c.opt.schedule;
      }
}

// x = the Chebyshev smoother of level 0 of H applied to b from x = 0 (the
// mixed formulation's A_qq solve)
void chebyshev_from_zero(Ctx& c, std::vector<Level>& H, const double* b, double* x) {
  smooth<double>(c, H, 0, b, nullptr, x, view(c, H[0], double()).y, false);
}

int level_schedule(Ctx& c, std::vector<Level>& H, int l) {
  const Level& L = H[l];
  if (&H == &c.hu && l == 0) return L.symf ? sym_minb(L) : 0;  // FP64: the full-storage k_cheb_u0
  const bool fp32 = c.opt.precision == 1;
  return L.tpp ? L.tpp : default_schedule(L.A, (fp32 ? (void*)L.rowf : (void*)L.rowd) != nullptr, fp32);
}

// timed as class 4 (displacement) or 5 (interface pressure)
void vcycle(Ctx& c, std::vector<Level>& H, const double* b, double* x, bool pre_done) {
  const int cls = (&H == &c.hu) ? 4 : 5;
  timing_begin(c, cls);
  vcycle_level<double>(c, H, 0, b, x, pre_done);
  timing_end(c, cls, 0.0);
}
void vcycle(Ctx& c, std::vector<Level>& H, const float* b, float* x, bool pre_done) {
  const int cls = (&H == &c.hu) ? 4 : 5;
  timing_begin(c, cls);
  vcycle_level<float>(c, H, 0, b, x, pre_done);
  timing_end(c, cls, 0.0);
}

namespace {
template <typename T>
FirstStep<T> first_step_t(Ctx& c, Level& L, T* x) {
  if (L.dense_inv) return {};
  const LV<T> v = view(c, L, T());
  T* s_buf = (c.opt.cheb_degree % 2 == 1) ? v.y : x;
  return {v.dinv, v.cf + 1, step_out(c.opt.cheb_degree, 0, s_buf, s_buf == x ? v.y : x), v.d};
}
}  // namespace
FirstStep<double> first_step(Ctx& c, std::vector<Level>& H, double* x) { return first_step_t<double>(c, H[0], x); }
FirstStep<float> first_step(Ctx& c, std::vector<Level>& H, float* x) { return first_step_t<float>(c, H[0], x); }

void level_apply(Ctx& c, std::vector<Level>& H, int l, const double* x, double* y) {
  level_spmv_t<double>(c, H[l], x, nullptr, y);
}

namespace {
__global__ void k_narrow(long long n, const double* __restrict__ x, float* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (float)x[i];
}
__global__ void k_widen(long long n, const float* __restrict__ x, double* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (double)x[i];
}
}  // namespace

// One V-cycle in the precision of the solve: FP64 directly, or, with
// precision 1, the FP32 cycle on b rounded to FP32 (the FP32 work vectors of
// the whole system, c.tf and c.zf, hold b and x).
void vcycle_api(Ctx& c, std::vector<Level>& H, const double* b, double* x) {
  if (c.opt.precision != 1) {
    vcycle(c, H, b, x);
    return;
  }
  const long long n = H[0].n;
  k_narrow<<<grid_for(n, 256), 256, 0, c.stream>>>(n, b, c.tf);
  MHFP_LAUNCH_CHECK();
  vcycle(c, H, (const float*)c.tf, c.zf);
  k_widen<<<grid_for(n, 256), 256, 0, c.stream>>>(n, c.zf, x);
  MHFP_LAUNCH_CHECK();
}

}  // namespace mhfp
