// Sweeps and residuals of the coarse lattice levels (displacement levels
// below the finest one, the interface-pressure cell levels), compiled once
// per value type (MHFP_SWEEP_T = float or double) so the many launch-schedule
// instantiations build in parallel.
#include "lattice.cuh"

#ifndef MHFP_SWEEP_T
#error "compile with -DMHFP_SWEEP_T=float or -DMHFP_SWEEP_T=double"
#endif

namespace mhfp {
namespace {

// ------------------------------------------------------- coarse-level sweeps
// Sweeps and residuals of the coarse lattice levels and of the interface-
// pressure cell levels.  Their data is a few to a few tens of MB, so the cost
// is latency and issue, not bytes: index arithmetic is 32-bit (the lattice
// point is split with multiply-high division by invariant integers,
// Granlund & Montgomery 1994, no 64-bit division), stencil offsets are
// compile-time constants, bounds are three small per-axis masks, and every
// offset of a chunk issues its loads before any is used (an out-of-lattice
// neighbour reads the point itself and is then replaced by 0).

// r -= sum over the offsets o with o % step == first of A(p, p + e_o) x(p + e_o)
template <int BS, int KIND, int CHUNK, typename T>
__device__ __forceinline__ void coarse_residual(const Lat32& L, unsigned p, const T* __restrict__ val,
                                                const T* __restrict__ x, T r[BS], int first, int step) {
  constexpr int R = Sf<KIND>::R, NO = Sf<KIND>::N;
  int i, j, k;
  L.ijk(p, i, j, k);
  bool mx[2 * R + 1], my[2 * R + 1], mz[2 * R + 1];
#pragma unroll
  for (int t = -R; t <= R; ++t) {
    mx[t + R] = (unsigned)(i + t) < (unsigned)L.Lx;
    my[t + R] = (unsigned)(j + t) < (unsigned)L.Ly;
    mz[t + R] = (unsigned)(k + t) < (unsigned)L.Lz;
  }
  const unsigned N = (unsigned)L.N;
#pragma unroll
  for (int o0 = 0; o0 < NO; o0 += CHUNK) {
    T vv[CHUNK][BS * BS], xx[CHUNK][BS];
#pragma unroll
    for (int c = 0; c < CHUNK; ++c) {
      const int o = o0 + c;
      if (o < NO && o % step == first) {
        const int dx = Sf<KIND>::x(o), dy = Sf<KIND>::y(o), dz = Sf<KIND>::z(o);
        const bool in = mx[dx + R] && my[dy + R] && mz[dz + R];
        const unsigned q = in ? p + (unsigned)(dx + L.Lx * dy + L.LxLy * dz) : p;
        const T* row = val + (size_t)o * BS * BS * N;
#pragma unroll
        for (int e = 0; e < BS * BS; ++e) vv[c][e] = row[e * N + p];
#pragma unroll
        for (int s = 0; s < BS; ++s) {
          const T xs = x[BS * q + s];
          xx[c][s] = in ? xs : T(0);  // a select, not a multiply (no FP64 pipe work)
        }
      }
    }
#pragma unroll
    for (int c = 0; c < CHUNK; ++c)
      if (o0 + c < NO && (o0 + c) % step == first)
#pragma unroll
        for (int a = 0; a < BS; ++a)
#pragma unroll
          for (int s = 0; s < BS; ++s) r[a] -= vv[c][a * BS + s] * xx[c][s];
  }
}

// one point per thread: loads of CHUNK offsets in flight at once
template <int BS, typename T>
constexpr int f_chunk() { return BS == 6 ? 1 : (sizeof(T) == 4 ? (BS == 1 ? 25 : 3) : (BS == 1 ? 8 : 1)); }

// y = b - A x, or y = A x when b is null
template <int BS, int KIND, typename T>
__global__ void __launch_bounds__(256) k_spmv_f(Lat32 L, const T* __restrict__ val, const T* __restrict__ x,
                                                const T* __restrict__ b, T* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= (unsigned)L.N) return;
  T r[BS];
#pragma unroll
  for (int a = 0; a < BS; ++a) r[a] = T(0);
  coarse_residual<BS, KIND, f_chunk<BS, T>(), T>(L, p, val, x, r, 0, 1);
#pragma unroll
  for (int a = 0; a < BS; ++a) y[BS * p + a] = b ? b[BS * p + a] + r[a] : -r[a];
}

// Chebyshev step: r = b - A xin, d = cd d + cr D^-1 r, xout = xin + d with cf = {cd, cr} in device
// memory; FIRST (cd = 0): d is only written
template <typename T, int BS>
__device__ __forceinline__ void cheb_update(unsigned p, unsigned N, const T r[BS], const T* __restrict__ dinv,
                                            const T* __restrict__ xin, T* __restrict__ xout, T* __restrict__ d,
                                            const T* __restrict__ cf, bool first) {
  const T cd = cf[0], cr = cf[1];
#pragma unroll
  for (int a = 0; a < BS; ++a) {
    T z = T(0);
#pragma unroll
    for (int s = 0; s < BS; ++s) z += dinv[(a * BS + s) * N + p] * r[s];
    const T dn = first ? cr * z : cd * d[BS * p + a] + cr * z;
    d[BS * p + a] = dn;
    xout[BS * p + a] = (xin ? xin[BS * p + a] : T(0)) + dn;
  }
}

template <int BS, int KIND, typename T>
__global__ void __launch_bounds__(256) k_cheb_f(Lat32 L, const T* __restrict__ val, const T* __restrict__ dinv,
                                                const T* __restrict__ b, const T* __restrict__ xin,
                                                T* __restrict__ xout, T* __restrict__ d, const T* __restrict__ cf, bool first,
                                                long long lb) {
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= (unsigned)L.N) return;
  T r[BS];
#pragma unroll
  for (int a = 0; a < BS; ++a) r[a] = b[BS * p + a];
  coarse_residual<BS, KIND, f_chunk<BS, T>(), T>(L, p, val, xin, r, 0, 1);
  cheb_update<T, BS>(p, (unsigned)L.N, r, dinv, xin, xout, d, cf, first);
}

// the first Chebyshev step from x = 0: d = cr D^-1 b, xout = d (no stencil)
template <int BS, typename T>
__global__ void __launch_bounds__(256) k_cheb_zero(long long npts, const T* __restrict__ dinv,
                                                   const T* __restrict__ b, T* __restrict__ xout, T* __restrict__ d,
                                                   const T* __restrict__ cf, long long lb) {
  b = lane_ptr(b, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  const T cr = cf[1];
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npts) return;
  T r[BS];
#pragma unroll
  for (int a = 0; a < BS; ++a) r[a] = b[BS * p + a];
#pragma unroll
  for (int a = 0; a < BS; ++a) {
    T z = T(0);
#pragma unroll
    for (int s = 0; s < BS; ++s) z += dinv[(a * BS + s) * npts + p] * r[s];
    d[BS * p + a] = cr * z;
    xout[BS * p + a] = cr * z;
  }
}

// Warp-split offsets: blockDim = (32, W); warp y takes the offsets o with
// o % W == y for 32 consecutive points, so every load instruction reads one
// stored row for 32 consecutive points; the W partial sums meet in shared
// memory and are added in a fixed order.
template <int BS, typename T>
constexpr int w_chunk() { return BS == 6 ? 1 : (sizeof(T) == 4 ? (BS == 1 ? 8 : 2) : (BS == 1 ? 4 : 1)); }

template <int BS, int KIND, int W, typename T>
__device__ __forceinline__ bool wsplit_residual(const Lat32& L, const T* __restrict__ val, const T* __restrict__ x,
                                                T (&part)[W][BS][32], unsigned& p, T r[BS]) {
  p = blockIdx.x * 32 + threadIdx.x;
  const bool valid = p < (unsigned)L.N;
  T acc[BS];
#pragma unroll
  for (int a = 0; a < BS; ++a) acc[a] = T(0);
  if (valid && x) coarse_residual<BS, KIND, w_chunk<BS, T>(), T>(L, p, val, x, acc, threadIdx.y, W);
#pragma unroll
  for (int a = 0; a < BS; ++a) part[threadIdx.y][a][threadIdx.x] = acc[a];
  __syncthreads();
  if (threadIdx.y != 0 || !valid) return false;
#pragma unroll
  for (int a = 0; a < BS; ++a) {
    T s = T(0);
#pragma unroll
    for (int u = 0; u < W; ++u) s += part[u][a][threadIdx.x];
    r[a] = s;  // = -(A x)_a
  }
  return true;
}

template <int BS, int KIND, int W, typename T>
__global__ void __launch_bounds__(32 * W) k_spmv_w(Lat32 L, const T* __restrict__ val, const T* __restrict__ x,
                                                   const T* __restrict__ b, T* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  __shared__ T part[W][BS][32];
  unsigned p;
  T r[BS];
  if (!wsplit_residual<BS, KIND, W, T>(L, val, x, part, p, r)) return;
#pragma unroll
  for (int a = 0; a < BS; ++a) y[BS * p + a] = b ? b[BS * p + a] + r[a] : -r[a];
}

template <int BS, int KIND, int W, typename T>
__global__ void __launch_bounds__(32 * W) k_cheb_w(Lat32 L, const T* __restrict__ val, const T* __restrict__ dinv,
                                                   const T* __restrict__ b, const T* __restrict__ xin,
                                                   T* __restrict__ xout, T* __restrict__ d, const T* __restrict__ cf, bool first,
                                                long long lb) {
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  __shared__ T part[W][BS][32];
  unsigned p;
  T r[BS];
  if (!wsplit_residual<BS, KIND, W, T>(L, val, xin, part, p, r)) return;
#pragma unroll
  for (int a = 0; a < BS; ++a) r[a] += b[BS * p + a];
  cheb_update<T, BS>(p, (unsigned)L.N, r, dinv, xin, xout, d, cf, first);
}

// Row-major levels: LPP lanes per point on values Ar[point][row a][PP], the
// NO x BS (offset, component) pairs of a row padded to PP = a multiple of 32
// (zeros).  On levels of up to some ten thousand points the split kernels
// above are bound by the latency of their serial chunks; here every load of a
// row is issued at once and consecutive lanes read consecutive values, and the
// sums meet in a fixed-order xor reduction (sizes and times: default_schedule).
template <int BS, int KIND>
constexpr int row_pairs() { return Sf<KIND>::N * BS; }
template <int BS, int KIND>
constexpr int row_pad() { return (row_pairs<BS, KIND>() + 31) / 32 * 32; }

template <int BS, int KIND>
__device__ __forceinline__ void pair_of(int e, int& dx, int& dy, int& dz, int& s) {
  static_assert(KIND != ST_DIAMOND2, "row-major levels are 27- or 125-point boxes");
  constexpr int w = KIND == ST_BOX1 ? 3 : 5, R = w / 2;
  const int o = e / BS;
  s = e - o * BS;
  dx = o % w - R;
  dy = (o / w) % w - R;
  dz = o / (w * w) - R;
}

// r = A x at point p (the same in each of the point's LPP lanes)
template <int BS, int KIND, int LPP, typename T>
__device__ __forceinline__ void row_product(const Lat32& L, unsigned p, const T* __restrict__ Ar,
                                            const T* __restrict__ x, T r[BS]) {
  constexpr int PP = row_pad<BS, KIND>(), NP = row_pairs<BS, KIND>(), PER = PP / LPP;
  constexpr int CH = PER <= 8 ? PER : (PER % 8 == 0 ? 8 : 6);  // pairs in flight per lane
  static_assert(PP % LPP == 0 && PER % CH == 0, "chunks cover the padded row exactly");
  const int l = threadIdx.x % LPP;
  int i, j, k;
  L.ijk(p, i, j, k);
#pragma unroll
  for (int a = 0; a < BS; ++a) r[a] = T(0);
  const T* row = Ar + (size_t)p * (BS * PP) + l;
#pragma unroll
  for (int c0 = 0; c0 < PER; c0 += CH) {
    T av[CH][BS], xv[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int e = l + LPP * (c0 + c);
      int dx, dy, dz, s;
      pair_of<BS, KIND>(e, dx, dy, dz, s);
      const bool in = e < NP && (unsigned)(i + dx) < (unsigned)L.Lx && (unsigned)(j + dy) < (unsigned)L.Ly &&
                      (unsigned)(k + dz) < (unsigned)L.Lz;
      const unsigned q = in ? p + (unsigned)(dx + L.Lx * dy + L.LxLy * dz) : p;
      const T v = x[BS * q + (in ? s : 0)];
      xv[c] = in ? v : T(0);
#pragma unroll
      for (int a = 0; a < BS; ++a) av[c][a] = row[a * PP + LPP * (c0 + c)];
    }
#pragma unroll
    for (int c = 0; c < CH; ++c)
#pragma unroll
      for (int a = 0; a < BS; ++a) r[a] += av[c][a] * xv[c];
  }
#pragma unroll
  for (int a = 0; a < BS; ++a)
#pragma unroll
    for (int m = LPP / 2; m > 0; m >>= 1) r[a] += __shfl_xor_sync(0xffffffffu, r[a], m);
}

template <int BS, typename T>
__device__ __forceinline__ T pick(const T v[BS], int a) {
  T s = v[0];
#pragma unroll
  for (int q = 1; q < BS; ++q) s = a == q ? v[q] : s;
  return s;
}

template <int BS, int KIND, int LPP, typename T>
__global__ void __launch_bounds__(128) k_spmv_r(Lat32 L, const T* __restrict__ Ar, const T* __restrict__ x,
                                                const T* __restrict__ b, T* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  const unsigned p0 = (blockIdx.x * 128 + threadIdx.x) / LPP;
  const unsigned p = p0 < (unsigned)L.N ? p0 : (unsigned)L.N - 1;  // the whole warp takes part in the reduction
  const int a = threadIdx.x % LPP;
  T r[BS];
  row_product<BS, KIND, LPP, T>(L, p, Ar, x, r);
  if (p0 >= (unsigned)L.N || a >= BS) return;
  const T v = pick<BS, T>(r, a);
  y[BS * p + a] = b ? b[BS * p + a] - v : v;
}

template <int BS, int KIND, int LPP, typename T>
__global__ void __launch_bounds__(128) k_cheb_r(Lat32 L, const T* __restrict__ Ar, const T* __restrict__ dinv,
                                                const T* __restrict__ b, const T* __restrict__ xin,
                                                T* __restrict__ xout, T* __restrict__ d, const T* __restrict__ cf, bool first,
                                                long long lb) {
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  const unsigned p0 = (blockIdx.x * 128 + threadIdx.x) / LPP;
  const unsigned p = p0 < (unsigned)L.N ? p0 : (unsigned)L.N - 1;
  const int a = threadIdx.x % LPP;
  // lane a's row of D^-1 and its vector entries, in flight with the stencil's
  T di[BS], bv[BS], dv = T(0), xv = T(0);
  const int ac = a < BS ? a : 0;
#pragma unroll
  for (int t = 0; t < BS; ++t) {
    di[t] = dinv[(ac * BS + t) * (unsigned)L.N + p];
    bv[t] = b[BS * p + t];
  }
  if (!first) dv = d[BS * p + ac];
  const T cd = cf[0], cr = cf[1];
  xv = xin[BS * p + ac];
  T r[BS];
  row_product<BS, KIND, LPP, T>(L, p, Ar, xin, r);
  if (p0 >= (unsigned)L.N || a >= BS) return;
  T z = T(0);
#pragma unroll
  for (int t = 0; t < BS; ++t) z += di[t] * (bv[t] - r[t]);
  const T dn = first ? cr * z : cd * dv + cr * z;
  d[BS * p + a] = dn;
  xout[BS * p + a] = xv + dn;
}

// offset-major values into the row-major layout: a thread per value
template <int BS, int KIND, typename T>
__global__ void __launch_bounds__(256) k_pack_rows(long long N, const T* __restrict__ val, T* __restrict__ Ar) {
  constexpr int PP = row_pad<BS, KIND>(), NP = row_pairs<BS, KIND>();
  const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
  if (t >= N * BS * PP) return;
  const int e = (int)(t % PP), a = (int)((t / PP) % BS);
  const long long p = t / (BS * PP);
  const int o = e / BS, s = e - o * BS;
  Ar[t] = e < NP ? val[(long long)(o * BS * BS + a * BS + s) * N + p] : T(0);
}

}  // namespace

// the row-major kernels' block sizes and kinds
template <class F>
void dispatch_rows(int bs, int kind, int lpp, F&& f) {
  auto with = [&](auto BS, auto K) {
    if (lpp == 8) f(BS, K, std::integral_constant<int, 8>{});
    else f(BS, K, std::integral_constant<int, 32>{});
  };
  if (bs == 3) with(std::integral_constant<int, 3>{}, std::integral_constant<int, ST_BOX1>{});
  else if (bs == 6) with(std::integral_constant<int, 6>{}, std::integral_constant<int, ST_BOX1>{});
  else with(std::integral_constant<int, 1>{}, std::integral_constant<int, ST_BOX2>{});
}

template <typename T>
void sweep_spmv(cudaStream_t stream, const StructOp& A, int bs, const T* val, const T* rows, const T* x, const T* b,
                T* y, int sched) {
  const Lat32 L = lat32_of(A);
  if (const int lpp = rows ? row_lanes(sched) : 0) {
    dispatch_rows(bs, A.kind, lpp, [&](auto BS, auto K, auto LPP) {
      k_spmv_r<BS.value, K.value, LPP.value, T><<<lgrid(grid_for(A.N * LPP.value, 128)), 128, 0, stream>>>(
          L, rows, x, b, y, lbytes());
    });
    return;
  }
  dispatch_bs(bs, [&](auto BS) {
    dispatch_kind_bs<BS.value>(A.kind, [&](auto K) {
      dispatch_sched(sched, [&](auto S) {
        if constexpr (S.value == 1)
          k_spmv_f<BS.value, K.value, T><<<lgrid(grid_for(A.N, 256)), 256, 0, stream>>>(L, val, x, b, y, lbytes());
        else
          k_spmv_w<BS.value, K.value, S.value, T><<<lgrid(grid_for(A.N, 32)), dim3(32, S.value), 0, stream>>>(
              L, val, x, b, y, lbytes());
      });
    });
  });
}

template <typename T>
void sweep_cheb(cudaStream_t stream, const StructOp& A, int bs, const T* val, const T* rows, const T* dinv, const T* b,
                const T* xin, T* out, T* d, const T* cf, bool first, int sched) {
  const Lat32 lat = lat32_of(A);
  if (const int lpp = rows ? row_lanes(sched) : 0) {
    dispatch_rows(bs, A.kind, lpp, [&](auto BS, auto K, auto LPP) {
      k_cheb_r<BS.value, K.value, LPP.value, T><<<lgrid(grid_for(A.N * LPP.value, 128)), 128, 0, stream>>>(
          lat, rows, dinv, b, xin, out, d, cf, first, lbytes());
    });
    return;
  }
  dispatch_bs(bs, [&](auto BS) {
    dispatch_kind_bs<BS.value>(A.kind, [&](auto K) {
      dispatch_sched(sched, [&](auto S) {
        if constexpr (S.value == 1)
          k_cheb_f<BS.value, K.value, T><<<lgrid(grid_for(A.N, 256)), 256, 0, stream>>>(
              lat, val, dinv, b, xin, out, d, cf, first, lbytes());
        else
          k_cheb_w<BS.value, K.value, S.value, T><<<lgrid(grid_for(A.N, 32)), dim3(32, S.value), 0, stream>>>(
              lat, val, dinv, b, xin, out, d, cf, first, lbytes());
      });
    });
  });
}

template <typename T>
size_t sweep_row_elems(const StructOp& A, int bs) {
  size_t n = 0;
  dispatch_rows(bs, A.kind, 32, [&](auto BS, auto K, auto) { n = (size_t)A.N * BS.value * row_pad<BS.value, K.value>(); });
  return n;
}

template <typename T>
void sweep_pack_rows(cudaStream_t stream, const StructOp& A, int bs, const T* val, T* rows) {
  dispatch_rows(bs, A.kind, 32, [&](auto BS, auto K, auto) {
    k_pack_rows<BS.value, K.value, T><<<grid_for((long long)sweep_row_elems<T>(A, bs), 256), 256, 0, stream>>>(A.N, val, rows);
  });
}

template <typename T>
void sweep_cheb_zero(cudaStream_t stream, long long npts, int bs, const T* dinv, const T* b, T* out, T* d,
                     const T* cf) {
  dispatch_bs(bs, [&](auto BS) {
    k_cheb_zero<BS.value, T><<<lgrid(grid_for(npts, 256)), 256, 0, stream>>>(npts, dinv, b, out, d, cf, lbytes());
  });
}

template void sweep_spmv<MHFP_SWEEP_T>(cudaStream_t, const StructOp&, int, const MHFP_SWEEP_T*, const MHFP_SWEEP_T*,
                                       const MHFP_SWEEP_T*, const MHFP_SWEEP_T*, MHFP_SWEEP_T*, int);
template void sweep_cheb<MHFP_SWEEP_T>(cudaStream_t, const StructOp&, int, const MHFP_SWEEP_T*, const MHFP_SWEEP_T*,
                                       const MHFP_SWEEP_T*, const MHFP_SWEEP_T*, const MHFP_SWEEP_T*, MHFP_SWEEP_T*,
                                       MHFP_SWEEP_T*, const MHFP_SWEEP_T*, bool, int);
template size_t sweep_row_elems<MHFP_SWEEP_T>(const StructOp&, int);
template void sweep_pack_rows<MHFP_SWEEP_T>(cudaStream_t, const StructOp&, int, const MHFP_SWEEP_T*, MHFP_SWEEP_T*);
template void sweep_cheb_zero<MHFP_SWEEP_T>(cudaStream_t, long long, int, const MHFP_SWEEP_T*, const MHFP_SWEEP_T*,
                                            MHFP_SWEEP_T*, MHFP_SWEEP_T*, const MHFP_SWEEP_T*);

}  // namespace mhfp
