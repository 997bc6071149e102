// The FP64 rows of the finest displacement level (27-point stencil of 3x3
// blocks, all 27 blocks stored offset-major, out-of-lattice blocks zero): the
// operator's u rows, the residual and the Chebyshev step.
//
// Large levels are bound by the FP64 pipe (243 FMA per node at 608 GFMA/s:
// 0.40 ns; 1,944 B at 6.8 TB/s: 0.29 ns), small ones by the latency of the
// stencil's serial chain.  Two forms:
//  * SPLIT = 0: a thread per node and its three rows; x is read once for nine
//    products, a pencil (three blocks) of loads ahead of its products.
//  * SPLIT = 1: nine threads per node, one per (component, stencil plane) and
//    27 products each; the planes' partial sums meet in shared memory and are
//    added in plane order.
// Measured, microseconds, SPLIT = 1 / SPLIT = 0 / the loop they replace (a
// thread per node over 27 offsets; for the operator a thread per row):
//     nodes      residual            Chebyshev step      operator rows
//       729     4.2 / 13.1 / 24      5.1 / 20.8 / 23.0   4.7 / 14.7 / 11.8
//     9,261     6.2 / 13.3 / 25      6.9 / 21.4 / 23.5   7.0 / 14.9 / 12.2
//    68,921    35.9 / 36.1 / 60     40.1 / 55.2 / 56.0  39.9 / 41.4 / 41.7
//   148,877    72.0 / 72.8 / -      79.9 / 75.4 / 75.1  80.4 / 82.3 / 79.8
//   274,625     129 / 122  / 196     142 / 146  / 143    144 / 138  / 138
// 2,146,689     966 / 886  / 1580   1079 / 971  / 961   1083 / 1014 / 1007
// so levels up to U64_SPLIT_NODES take SPLIT = 1 (the FP64 pipe's time at
// 2,146,689 nodes: 858, 890 and 943).
#pragma once
#include "lattice.cuh"

namespace mhfp {
namespace {

constexpr long long U64_SPLIT_NODES = 120000;
constexpr int U64_NODES = 32;      // nodes per block, SPLIT = 1 (288 threads)
constexpr int U64_NODES_1 = 128;   // nodes and threads per block, SPLIT = 0

// out = so ? so[r] * (bsub ? bsub[r] - y : y) : (bsub ? bsub[r] - y : y)
__device__ __forceinline__ double finish(double y, long long r, const double* so, const double* bsub) {
  double v = bsub ? bsub[r] - y : y;
  return so ? so[r] * v : v;
}

// rows [C0, C0 + NC) of node n: acc += the stencil's pencil (., dy, dz); an
// absent neighbour counts as x = 0 (a select: its stored block is zero, but
// the x read in its place may not be finite)
template <int NC>
__device__ __forceinline__ void u64_pencil(const Lat32& L, unsigned n, int i, int j, int k, int dy, int dz, int c0,
                                           const double* __restrict__ A, const double* __restrict__ x,
                                           double (&acc)[NC]) {
  if ((unsigned)(j + dy) >= (unsigned)L.Ly || (unsigned)(k + dz) >= (unsigned)L.Lz) return;
  const long long N = L.N;
  const double* v = A + ((long long)(3 * (dy + 1) + 9 * (dz + 1)) * 9 + 3 * c0) * N + n;
  const double* xm = x + 3 * ((long long)n + dy * L.Lx + (long long)dz * L.LxLy);
  double a[3][3 * NC], y[9];
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    const bool in = o == 0 ? i > 0 : (o == 2 ? i + 1 < L.Lx : true);
    const double* xo = xm + (in ? 3 * (o - 1) : 0);
#pragma unroll
    for (int e = 0; e < 3 * NC; ++e) a[o][e] = v[(long long)(9 * o + e) * N];
#pragma unroll
    for (int c = 0; c < 3; ++c) y[3 * o + c] = in ? xo[c] : 0.0;
  }
#pragma unroll
  for (int o = 0; o < 3; ++o)
#pragma unroll
    for (int r = 0; r < NC; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[r] = fma(a[o][3 * r + c], y[3 * o + c], acc[r]);
}

// rows of node n: acc += cup A_up x_p over the cells on the z side uz (0: -, 1: +)
template <int NC>
__device__ __forceinline__ void u64_cells(const Lat32& L, int i, int j, int k, int uz, int c0,
                                          const double* __restrict__ Aup, const double* __restrict__ xp, double cup,
                                          double (&acc)[NC]) {
  const int nx = L.Lx - 1, ny = L.Ly - 1, nz = L.Lz - 1;
  const long long nT = (long long)nx * ny * nz;
  const int cz = k - 1 + uz;
  if ((unsigned)cz >= (unsigned)nz) return;
  double av[4][NC], p[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int ux = c & 1, uy = c >> 1, cx = i - 1 + ux, cy = j - 1 + uy;
    const bool in = (unsigned)cx < (unsigned)nx && (unsigned)cy < (unsigned)ny;
    const long long T = in ? cx + (long long)nx * (cy + (long long)ny * cz) : 0;
    const int a = (1 - ux) + 2 * (1 - uy) + 4 * (1 - uz);  // the node's local number in the cell
    p[c] = in ? xp[T] : 0.0;
#pragma unroll
    for (int r = 0; r < NC; ++r) av[c][r] = Aup[(long long)(3 * a + c0 + r) * nT + T];
  }
#pragma unroll
  for (int r = 0; r < NC; ++r) {
    double sp = av[0][r] * p[0];
#pragma unroll
    for (int c = 1; c < 4; ++c) sp = fma(av[c][r], p[c], sp);
    acc[r] = fma(cup, sp, acc[r]);
  }
}

// all three rows of node n of A_uu x (+ cup A_up x_p when Aup is given), the
// stencil planes z0 .. z1
__device__ __forceinline__ void u64_rows(const Lat32& L, unsigned n, const double* __restrict__ A,
                                         const double* __restrict__ x, const double* __restrict__ Aup, double cup,
                                         double (&acc)[3], int z0 = -1, int z1 = 1) {
  int i, j, k;
  L.ijk(n, i, j, k);
#pragma unroll 1
  for (int dz = z0; dz <= z1; ++dz)
#pragma unroll 1
    for (int dy = -1; dy <= 1; ++dy) u64_pencil<3>(L, n, i, j, k, dy, dz, 0, A, x, acc);
  if (Aup) {
    const double* xp = x + 3LL * L.N;
#pragma unroll 1
    for (int uz = 0; uz < 2; ++uz)
      if (uz ? z1 == 1 : z0 == -1) u64_cells<3>(L, i, j, k, uz, 0, Aup, xp, cup, acc);
  }
}

// SPLIT = 1: row (node, component) of the same; the planes' parts joined in
// plane 0, where the sum is returned.  Every thread of the block calls it.
__device__ __forceinline__ double u64_row_split(const Lat32& L, unsigned n, bool valid, int comp, int s,
                                                const double* __restrict__ A, const double* __restrict__ x,
                                                const double* __restrict__ Aup, double cup) {
  __shared__ double part[2][3][U64_NODES];
  double acc[1] = {0.0};
  if (valid) {
    int i, j, k;
    L.ijk(n, i, j, k);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) u64_pencil<1>(L, n, i, j, k, dy, s - 1, comp, A, x, acc);
    if (Aup && s != 1) u64_cells<1>(L, i, j, k, s >> 1, comp, Aup, x + 3LL * L.N, cup, acc);
  }
  if (s > 0) part[s - 1][comp][threadIdx.x] = acc[0];
  __syncthreads();
  return s == 0 ? (acc[0] + part[0][comp][threadIdx.x]) + part[1][comp][threadIdx.x] : 0.0;
}

// y = b - A x (y = A x when b is null); with Aup the operator's u rows, y =
// finish(A_uu x_u + cup A_up x_p) with so and b
template <int SPLIT>
__global__ void __launch_bounds__(SPLIT ? 9 * U64_NODES : U64_NODES_1)
    k_u64(Lat32 L, const double* __restrict__ A, const double* __restrict__ Aup, double cup,
          const double* __restrict__ x, const double* __restrict__ so, const double* __restrict__ b,
          double* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  if (SPLIT) {
    const unsigned n = blockIdx.x * U64_NODES + threadIdx.x;
    const int comp = threadIdx.y % 3, s = threadIdx.y / 3;
    const bool valid = n < (unsigned)L.N;
    const double v = u64_row_split(L, n, valid, comp, s, A, x, Aup, cup);
    const long long r = 3LL * n + comp;
    if (valid && s == 0) y[r] = finish(v, r, so, b);
  } else {
    const unsigned n = blockIdx.x * U64_NODES_1 + threadIdx.x;
    if (n >= (unsigned)L.N) return;
    double acc[3] = {0.0, 0.0, 0.0};
    u64_rows(L, n, A, x, Aup, cup, acc);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[3LL * n + c] = finish(acc[c], 3LL * n + c, so, b);
  }
}

template <class... Args>
void launch_u64(cudaStream_t stream, const Lat32& L, Args... args) {
  if (L.N <= U64_SPLIT_NODES)
    k_u64<1><<<lgrid(grid_for(L.N, U64_NODES)), dim3(U64_NODES, 9), 0, stream>>>(L, args..., lbytes());
  else
    k_u64<0><<<lgrid(grid_for(L.N, U64_NODES_1)), U64_NODES_1, 0, stream>>>(L, args..., lbytes());
}

}  // namespace
}  // namespace mhfp
