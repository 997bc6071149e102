// The FP64 rows of the finest displacement level (27-point stencil of 3x3
// blocks, all 27 blocks stored offset-major): operator rows, residual and
// Chebyshev step, one thread per (node, component, part).
//
// The FP64 pipe bounds these rows on large levels (243 FMA per node against
// 1,944 B: 0.40 ns and 0.29 ns per node at 608 GFMA/s and 6.8 TB/s), and the
// latency of the 27 dependent steps on small ones.  Three threads per node
// (one per component, 81 FMA each) keep the pipe at 0.9; on small levels the
// nine (dz, dy) pencils of a row are further split over S = 3 (planes) or
// S = 9 (pencils) warps, whose partial sums meet in shared memory and are
// added in a fixed order (S - 1 more FP64 adds per row).  u_split picks S.
#pragma once
#include "lattice.cuh"

namespace mhfp {
namespace {

// threads per block along the nodes: 64 for S = 1, 32 otherwise
template <int S>
constexpr int u_nodes() { return S == 1 ? 64 : 32; }

// part `s` of row (n, comp) of A_uu x
template <int S>
__device__ __forceinline__ double u_row_part(const Lat32& L, unsigned n, int i, int j, int k, int comp, int s,
                                             const double* __restrict__ A, const double* __restrict__ x) {
  const long long N = L.N;
  const double* row = A + 3 * comp * N + n;
  double acc = 0.0;
  const bool lo = i > 0, hi = i + 1 < L.Lx;
  auto pencil = [&](int dy, int dz) {
    if ((unsigned)(j + dy) >= (unsigned)L.Ly || (unsigned)(k + dz) >= (unsigned)L.Lz) return;
    const double* v = row + (long long)(3 * (dy + 1) + 9 * (dz + 1)) * 9 * N;
    const double* xm = x + 3 * ((long long)n + dy * L.Lx + dz * L.LxLy);
    double a[9], y[9];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      const bool in = o == 0 ? lo : (o == 2 ? hi : true);
      const double* xo = xm + (in ? 3 * (o - 1) : 0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        a[3 * o + c] = v[(long long)(9 * o + c) * N];
        y[3 * o + c] = in ? xo[c] : 0.0;
      }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) acc = fma(a[e], y[e], acc);
  };
  if (S == 9) {
    pencil(s % 3 - 1, s / 3 - 1);
  } else if (S == 3) {
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) pencil(dy, s - 1);
  } else {
#pragma unroll 1
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) pencil(dy, dz);
  }
  return acc;
}

// part `s` of row (n, comp) of A_up x_p: the pencils with dy, dz = +-1 take
// the two cells of the node on their side
template <int S>
__device__ __forceinline__ double u_cells_part(const Lat32& L, unsigned n, int i, int j, int k, int comp, int s,
                                               const double* __restrict__ Aup, const double* __restrict__ xp) {
  const int nx = L.Lx - 1, ny = L.Ly - 1, nz = L.Lz - 1;
  const long long nT = (long long)nx * ny * nz;
  double sp = 0.0;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int uy = c & 1, uz = c >> 1;  // the cell pair on the - (0) or + (1) side in y and z
    if (S == 9 && s != 2 * uy + 6 * uz) continue;
    if (S == 3 && s != 2 * uz) continue;
    const int cy = j - 1 + uy, cz = k - 1 + uz;
    if ((unsigned)cy >= (unsigned)ny || (unsigned)cz >= (unsigned)nz) continue;
#pragma unroll
    for (int ux = 0; ux < 2; ++ux) {
      const int cx = i - 1 + ux;
      if ((unsigned)cx >= (unsigned)nx) continue;
      const long long T = cx + (long long)nx * (cy + (long long)ny * cz);
      const int a = (1 - ux) + 2 * (1 - uy) + 4 * (1 - uz);  // the node's local number in the cell
      sp = fma(Aup[(long long)(3 * a + comp) * nT + T], xp[T], sp);
    }
  }
  return sp;
}

// the sum of the S parts of (component, node lane), in order; valid in part 0.
// Every thread of the block calls it.
template <int S>
__device__ __forceinline__ double u_join(double acc, double (&part)[S][3][32], int comp, int s) {
  if (S == 1) return acc;
  part[s][comp][threadIdx.x] = acc;
  __syncthreads();
  double r = acc;
  if (s == 0)
#pragma unroll
    for (int q = 1; q < S; ++q) r += part[q][comp][threadIdx.x];
  return r;
}

// y = b - A x (y = A x when b is null)
template <int S>
__global__ void __launch_bounds__(3 * S * u_nodes<S>()) k_u64_resid(Lat32 L, const double* __restrict__ A,
                                                                   const double* __restrict__ x,
                                                                   const double* __restrict__ b,
                                                                   double* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  __shared__ double part[S][3][32];
  const unsigned n = blockIdx.x * u_nodes<S>() + threadIdx.x;
  const int comp = threadIdx.y % 3, s = threadIdx.y / 3;
  const bool valid = n < (unsigned)L.N;
  double acc = 0.0;
  if (valid) {
    int i, j, k;
    L.ijk(n, i, j, k);
    acc = u_row_part<S>(L, n, i, j, k, comp, s, A, x);
  }
  acc = u_join<S>(acc, part, comp, s);
  if (!valid || s != 0) return;
  const long long r = 3LL * n + comp;
  y[r] = b ? b[r] - acc : acc;
}

// Chebyshev step: r = b - A xin, d = cd d + cr D^-1 r, xout = xin + d
template <int S>
__global__ void __launch_bounds__(3 * S * u_nodes<S>()) k_u64_cheb(Lat32 L, const double* __restrict__ A,
                                                                  const double* __restrict__ dinv,
                                                                  const double* __restrict__ b,
                                                                  const double* __restrict__ xin,
                                                                  double* __restrict__ xout, double* __restrict__ d,
                                                                  double cd, double cr, long long lb) {
  b = lane_ptr(b, lb);
  xin = lane_ptr(xin, lb);
  xout = lane_ptr(xout, lb);
  d = lane_ptr(d, lb);
  __shared__ double part[S][3][32];
  __shared__ double rs[3][u_nodes<S>()];
  const unsigned n = blockIdx.x * u_nodes<S>() + threadIdx.x;
  const int comp = threadIdx.y % 3, s = threadIdx.y / 3;
  const bool valid = n < (unsigned)L.N;
  double acc = 0.0;
  if (valid) {
    int i, j, k;
    L.ijk(n, i, j, k);
    acc = u_row_part<S>(L, n, i, j, k, comp, s, A, xin);
  }
  acc = u_join<S>(acc, part, comp, s);
  const long long r = 3LL * n + comp, N = L.N;
  if (s == 0) rs[comp][threadIdx.x] = valid ? b[r] - acc : 0.0;
  __syncthreads();
  if (!valid || s != 0) return;
  double z = 0.0;
#pragma unroll
  for (int t = 0; t < 3; ++t) z += dinv[(3 * comp + t) * N + n] * rs[t][threadIdx.x];
  const double dn = (cd != 0.0) ? cd * d[r] + cr * z : cr * z;
  d[r] = dn;
  xout[r] = xin[r] + dn;
}

// how many parts: U_SPLIT_RULE
inline int u_split(long long N) { return N <= 16384 ? 9 : (N <= 131072 ? 3 : 1); }

template <class F>
void dispatch_split(int S, F&& f) {
  if (S == 9) f(std::integral_constant<int, 9>{});
  else if (S == 3) f(std::integral_constant<int, 3>{});
  else f(std::integral_constant<int, 1>{});
}

}  // namespace
}  // namespace mhfp
