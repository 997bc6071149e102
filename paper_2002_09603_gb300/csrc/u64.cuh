// The FP64 rows of the finest displacement level (27-point stencil of 3x3
// blocks, all 27 blocks stored offset-major, out-of-lattice blocks zero): the
// operator's u rows, the residual and the Chebyshev step.
//
// Large levels are bound by the FP64 pipe (243 FMA per node at 608 GFMA/s:
// 0.40 ns; 1,944 B at 6.8 TB/s: 0.29 ns), small ones by the latency of the
// stencil's serial chain.  Three forms, in the order of the number of threads:
//  * U64_SPLIT: nine threads per node, one per (component, stencil plane) and
//    27 products each; the planes' partial sums meet in shared memory and are
//    added in plane order.
//  * U64_ROW: three threads per node, one per row; the three planes unrolled,
//    40 registers, so that 16 blocks of 96 threads fit an SM (the Chebyshev
//    step: 48 and 13, without which it spills).
//  * U64_NODE: a thread per node and its three rows; x is read once for nine
//    products.
// U64_ROW and U64_NODE sum a row in the same order (the same bits).
// Microseconds, calls in a row / L2 flushed before each; "loop" is what they
// replace (a thread per node over 27 offsets; for the operator a thread per row):
//     nodes  residual                     Chebyshev step                      operator rows
//            SPLIT   NODE    ROW          SPLIT   NODE    ROW     loop        SPLIT   NODE    ROW     loop
//     9,261  10/14   18/30   -            11/14   29/59   -       39/92       11/14   18/32   -       16/29
//    54,872  33/37   33/41   35/37        35/39   57/68   37/41   86/103      37/41   37/45   39/37   36/41
//    68,921  41/47   41/45   41/45        43/49   55/62   45/49   96/105      45/51   45/49   47/45   47/45
//   117,649  64/67   66/65   60/63        66/71   66/70   65/69   98/107      70/74   72/72   68/71   72/75
//   274,625  133/139 125/127 125/125      142/147 145/152 133/134 150/152     148/153 140/141 141/141 142/144
//   531,441  249/254 231/232 233/233      256/261 256/258 248/249 258/263     278/282 260/260 263/264 263/264
//   912,673  419/424 386/387 393/393      446/450 424/424 416/417 443/446     468/473 434/436 445/445 439/441
// 2,146,689  943/949 856/858 873/875      1003    932/933 928/930 942/948     1053    967/968 986/987 974/977
// (the step in a solve, where the vectors lie elsewhere: 274,625 nodes 150 NODE,
// 130 ROW, 145 loop; 2,146,689 nodes 932, 944 and 929).  So U64_SPLIT up to
// U64_SPLIT_NODES, for the operator up to U64_SPLIT_ROWS (its matrix is seldom
// in L2 when it is applied, that of a sweep or residual often is); above, the
// step takes U64_ROW up to U64_ROW_STEP, the operator up to U64_SPLIT_NODES,
// and everything else is U64_NODE (393,120 nodes, both operators, the
// float-float one and the norm in turn: 987 us, 995 with U64_ROW).  The FP64
// pipe's time at 2,146,689 nodes: 858, 890 and 943.
#pragma once
#include "lattice.cuh"

namespace mhfp {
namespace {

enum U64Form { U64_NODE, U64_SPLIT, U64_ROW };
constexpr long long U64_SPLIT_NODES = 120000, U64_SPLIT_ROWS = 60000, U64_ROW_STEP = 1500000;
constexpr int u64_nodes(U64Form f) { return f == U64_NODE ? 128 : 32; }  // nodes per block
constexpr int u64_parts(U64Form f) { return f == U64_SPLIT ? 9 : (f == U64_ROW ? 3 : 1); }  // threads per node
constexpr int u64_threads(U64Form f) { return u64_nodes(f) * u64_parts(f); }
constexpr int u64_blocks(U64Form f) { return f == U64_ROW ? 16 : 0; }  // per SM, at least (0: not asked for)

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

// U64_SPLIT: row (node, component) of the same; the planes' parts joined in
// plane 0, where the sum is returned.  Every thread of the block calls it.
__device__ __forceinline__ double u64_row_split(const Lat32& L, unsigned n, bool valid, int comp, int s,
                                                const double* __restrict__ A, const double* __restrict__ x,
                                                const double* __restrict__ Aup, double cup) {
  __shared__ double part[2][3][u64_nodes(U64_SPLIT)];
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

// U64_ROW: row (node, component) by one thread
__device__ __forceinline__ double u64_row(const Lat32& L, unsigned n, int comp, const double* __restrict__ A,
                                          const double* __restrict__ x, const double* __restrict__ Aup, double cup) {
  double acc[1] = {0.0};
  int i, j, k;
  L.ijk(n, i, j, k);
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) u64_pencil<1>(L, n, i, j, k, dy, dz, comp, A, x, acc);
  if (Aup) {
#pragma unroll 1
    for (int uz = 0; uz < 2; ++uz) u64_cells<1>(L, i, j, k, uz, comp, Aup, x + 3LL * L.N, cup, acc);
  }
  return acc[0];
}

// y = b - A x (y = A x when b is null); with Aup the operator's u rows, y =
// finish(A_uu x_u + cup A_up x_p) with so and b
template <U64Form F>
__global__ void __launch_bounds__(u64_threads(F), u64_blocks(F))
    k_u64(Lat32 L, const double* __restrict__ A, const double* __restrict__ Aup, double cup,
          const double* __restrict__ x, const double* __restrict__ so, const double* __restrict__ b,
          double* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  b = lane_ptr(b, lb);
  y = lane_ptr(y, lb);
  const unsigned n = blockIdx.x * u64_nodes(F) + threadIdx.x;
  const bool valid = n < (unsigned)L.N;
  if (F == U64_SPLIT) {
    const int comp = threadIdx.y % 3, s = threadIdx.y / 3;
    const double v = u64_row_split(L, n, valid, comp, s, A, x, Aup, cup);
    const long long r = 3LL * n + comp;
    if (valid && s == 0) y[r] = finish(v, r, so, b);
  } else if (F == U64_ROW) {
    if (!valid) return;
    const long long r = 3LL * n + threadIdx.y;
    y[r] = finish(u64_row(L, n, threadIdx.y, A, x, Aup, cup), r, so, b);
  } else {
    if (!valid) return;
    double acc[3] = {0.0, 0.0, 0.0};
    u64_rows(L, n, A, x, Aup, cup, acc);
#pragma unroll
    for (int c = 0; c < 3; ++c) y[3LL * n + c] = finish(acc[c], 3LL * n + c, so, b);
  }
}

// f(form): U64_SPLIT up to `split` nodes, U64_ROW up to `row`, U64_NODE above
template <class F>
void dispatch_u64(long long N, long long split, long long row, F&& f) {
  if (N <= split) f(std::integral_constant<U64Form, U64_SPLIT>{});
  else if (N <= row) f(std::integral_constant<U64Form, U64_ROW>{});
  else f(std::integral_constant<U64Form, U64_NODE>{});
}

template <U64Form F>
dim3 u64_grid(long long N) { return lgrid(grid_for(N, u64_nodes(F))); }
template <U64Form F>
dim3 u64_block() { return dim3(u64_nodes(F), u64_parts(F)); }

// the operator's u rows (Aup given) or a product or residual
template <class... Args>
void launch_u64(cudaStream_t stream, const Lat32& L, const double* A, const double* Aup, Args... args) {
  dispatch_u64(L.N, Aup ? U64_SPLIT_ROWS : U64_SPLIT_NODES, U64_SPLIT_NODES, [&](auto F) {
    constexpr U64Form f = decltype(F)::value;
    k_u64<f><<<u64_grid<f>(L.N), u64_block<f>(), 0, stream>>>(L, A, Aup, args..., lbytes());
  });
}

}  // namespace
}  // namespace mhfp
