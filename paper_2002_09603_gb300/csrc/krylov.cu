// Right-preconditioned flexible GMRES(m) (Section 5: GMRES, right
// preconditioning, zero initial guess, stop on the 2-norm of the residual
// relative to the initial one).  Classical Gram-Schmidt applied twice with
// deterministic two-stage reductions; Givens rotations and the triangular
// solve run in one thread on the device; the host reads one 8-byte residual
// estimate per iteration.
#include "common.cuh"

#include <algorithm>
#include <chrono>
#include <cmath>

namespace mhfp {

namespace {

constexpr int RED_BLOCKS = 608;   // 4 x 152 SMs
constexpr int RED_THREADS = 256;

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
  __syncthreads();
  return s;  // valid in thread 0
}

// Gram-Schmidt kernels.  On GB300 the FP64 pipe (about 2 FMA per clock per
// SM) bounds these passes, so they are written for occupancy: few registers
// per thread, many rows in flight, independent FMA chains.
constexpr int GS_BLOCKS = 1216;   // 8 x 152 SMs
constexpr int GS_COLS = 8;        // columns per block in the dot kernel (w is read once per 8 columns)
constexpr int GS_DOT_BLOCKS = 608;  // 4 x 152 SMs at most (gs_dot_blocks): the fewer the
                                    // blocks, the fewer FP64 adds in their reductions

// Sum of a[0..7] over the warp by a transposed butterfly: each exchange
// halves the number of live columns per lane, so the eight sums cost 7 + 2
// FP64 adds and shuffles per lane instead of 40.  Lane 4q + r (r = 0..3)
// returns the warp's sum for column q.
__device__ __forceinline__ double warp_sum8(const double (&a)[GS_COLS]) {
  const unsigned lane = threadIdx.x & 31u;
  const bool h16 = lane & 16u, h8 = lane & 8u, h4 = lane & 4u;
  double k[4], m[2];
#pragma unroll
  for (int q = 0; q < 4; ++q)  // columns 4 h16 + q
    k[q] = (h16 ? a[4 + q] : a[q]) + __shfl_xor_sync(0xffffffffu, h16 ? a[q] : a[4 + q], 16);
#pragma unroll
  for (int q = 0; q < 2; ++q)  // columns 4 h16 + 2 h8 + q
    m[q] = (h8 ? k[2 + q] : k[q]) + __shfl_xor_sync(0xffffffffu, h8 ? k[q] : k[2 + q], 8);
  double t = (h4 ? m[1] : m[0]) + __shfl_xor_sync(0xffffffffu, h4 ? m[0] : m[1], 4);  // column lane >> 2
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  return t;
}

// acc[q] += V[:, c0 + q] . w over this thread's rows for q < NC (the
// valid columns of the block's group, so no predicated-off FMA is issued),
// and nw += w . w when NORM
template <int NC, bool NORM>
__device__ __forceinline__ void gs_rows(long long n, const double* __restrict__ V, int c0,
                                        const double* __restrict__ w, double (&acc)[GS_COLS], double& nw) {
  const long long stride = (long long)gridDim.x * blockDim.x;
#pragma unroll 1
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride) {
    const double wr = w[r];
#pragma unroll
    for (int q = 0; q < NC; ++q) acc[q] = fma(V[(long long)(c0 + q) * n + r], wr, acc[q]);
    if (NORM) nw = fma(wr, wr, nw);
  }
}

// hout[c] = V[:, c] . w for the columns c <= j, eight per block row
// (blockIdx.y), and *nrm2 = w . w when given.  Nothing happens when *skip.
__global__ void __launch_bounds__(RED_THREADS, 4) k_gs_dots(long long n, const double* __restrict__ V, int j,
                                                             const double* __restrict__ w,
                                                             double* __restrict__ partials, double* __restrict__ hout,
                                                             double* __restrict__ nrm2,
                                                             const int* __restrict__ skip,
                                                             unsigned* __restrict__ counters, long long lb) {
  static_assert(GS_COLS == 8, "warp_sum8 reduces eight columns");
  V = lane_ptr(V, lb);
  w = lane_ptr(w, lb);
  partials = lane_ptr(partials, lb);
  hout = lane_ptr(hout, lb);
  nrm2 = lane_ptr(nrm2, lb);
  skip = lane_ptr(skip, lb);
  counters = lane_ptr(counters, lb);
  const int ncols = j + 1, c0 = blockIdx.y * GS_COLS;
  if (c0 >= ncols || (skip && *skip)) return;
  __shared__ double sh[RED_THREADS / 32][GS_COLS];
  __shared__ double shn[RED_THREADS / 32];
  const bool do_norm = nrm2 != nullptr && blockIdx.y == 0;
  double acc[GS_COLS] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, nw = 0.0;
  const int nc = ncols - c0 < GS_COLS ? ncols - c0 : GS_COLS;
  // block-uniform branch on the number of valid columns in this group
  switch (nc + (do_norm ? 16 : 0)) {
    case 1: gs_rows<1, false>(n, V, c0, w, acc, nw); break;
    case 2: gs_rows<2, false>(n, V, c0, w, acc, nw); break;
    case 3: gs_rows<3, false>(n, V, c0, w, acc, nw); break;
    case 4: gs_rows<4, false>(n, V, c0, w, acc, nw); break;
    case 5: gs_rows<5, false>(n, V, c0, w, acc, nw); break;
    case 6: gs_rows<6, false>(n, V, c0, w, acc, nw); break;
    case 7: gs_rows<7, false>(n, V, c0, w, acc, nw); break;
    case 8: gs_rows<8, false>(n, V, c0, w, acc, nw); break;
    case 17: gs_rows<1, true>(n, V, c0, w, acc, nw); break;
    case 18: gs_rows<2, true>(n, V, c0, w, acc, nw); break;
    case 19: gs_rows<3, true>(n, V, c0, w, acc, nw); break;
    case 20: gs_rows<4, true>(n, V, c0, w, acc, nw); break;
    case 21: gs_rows<5, true>(n, V, c0, w, acc, nw); break;
    case 22: gs_rows<6, true>(n, V, c0, w, acc, nw); break;
    case 23: gs_rows<7, true>(n, V, c0, w, acc, nw); break;
    case 24: gs_rows<8, true>(n, V, c0, w, acc, nw); break;
    default: break;
  }
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const double t = warp_sum8(acc);
  if ((lane & 3u) == 0) sh[wid][lane >> 2] = t;
  if (do_norm) {
    for (int o = 16; o > 0; o >>= 1) nw += __shfl_xor_sync(0xffffffffu, nw, o);
    if (lane == 0) shn[wid] = nw;
  }
  __syncthreads();
  const int nb = gridDim.x;
  if ((int)threadIdx.x < nc) {
    double s = 0.0;
    for (int k = 0; k < RED_THREADS / 32; ++k) s += sh[k][threadIdx.x];
    partials[(long long)(c0 + threadIdx.x) * nb + blockIdx.x] = s;
  }
  if (do_norm && threadIdx.x == 32) {
    double s = 0.0;
    for (int k = 0; k < RED_THREADS / 32; ++k) s += shn[k];
    partials[(long long)ncols * nb + blockIdx.x] = s;
  }
  if (!last_block(counters + blockIdx.y, nb)) return;
  for (int q = wid; q < nc + (do_norm ? 1 : 0); q += RED_THREADS / 32) {
    const int c = q < nc ? c0 + q : ncols;  // the norm's partials are row ncols
    const double s = warp_sum_of(partials + (long long)c * nb, nb);
    if (lane == 0) {
      if (q < nc) hout[c] = s;
      else *nrm2 = s;
    }
  }
}

__global__ void k_reduce_partials(int nb, const double* __restrict__ partials, double* __restrict__ out, int accumulate,
                                  long long lb) {
  partials = lane_ptr(partials, lb);
  out = lane_ptr(out, lb);
  __shared__ double sh[RED_THREADS / 32];
  double v = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) v += partials[(long long)blockIdx.x * nb + b];
  const double s = block_sum(v, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = accumulate ? out[blockIdx.x] + s : s;
}

// What the last block of k_gemv_sub does with ||w||^2: the DGKS test after a
// first pass, or the Hessenberg column and its Givens rotation after the last.
//
// DGKS test (Daniel, Gragg, Kaufman & Stewart, 1976): after one classical
// Gram-Schmidt projection, reorthogonalise only if the norm fell below
// 1/sqrt(2) of its value before the projection (nrm0 = ||w||^2 before).
// flag = 1 means "skip the second projection": then h2 is zero and the norm
// after the first pass is the final one.
struct GsTail {
  int givens;               // 0: DGKS test, 1: Givens
  const double* nrm0;       // DGKS: ||w||^2 before
  int* flag;                // DGKS: decision
  double* h2;               // second pass's coefficients (null: none)
  double* nrm2;             // the final ||w||^2
  const double* h1;         // Givens: first pass's coefficients
  double *H, *cs, *sn, *g, *scal;
  int m;
  __device__ __forceinline__ GsTail lane(long long lb) const {
    return {givens, lane_ptr(nrm0, lb), lane_ptr(flag, lb), lane_ptr(h2, lb), lane_ptr(nrm2, lb), lane_ptr(h1, lb),
            lane_ptr(H, lb), lane_ptr(cs, lb), lane_ptr(sn, lb), lane_ptr(g, lb), lane_ptr(scal, lb), m};
  }
};

// One Arnoldi step's Hessenberg column, by one warp: h = h1 + h2 (j+1
// entries; h2 null after a single Gram-Schmidt pass), the new subdiagonal
// ||w|| = sqrt(nrm2); apply the previous rotations, make the new one, update
// g.  scal[0] = |g_{j+1}|, scal[1] = 1/||w|| (0 on breakdown).
// The previous rotations are a linear recurrence, a_{i+1} = -s_i a_i + c_i
// h_{i+1} with a_0 = h_0, of which column entry i is c_i a_i + s_i h_{i+1}: one
// thread walking it took 0.27 us per rotation (the latency of its FP64
// chain), so the warp composes the maps a -> M a + K by a scan, 32 at a time.
// |M| <= 1 throughout.
__device__ __forceinline__ void givens_step(int j, const GsTail& t, double nrm2) {
  const int lane = threadIdx.x & 31;
  double* out = t.H + (long long)j * (t.m + 1);
  auto entry = [&](int i) { return t.h2 ? t.h1[i] + t.h2[i] : t.h1[i]; };
  const double gj = t.g[j];
  double a = entry(0);  // a_base, the same in every lane
  for (int base = 0; base < j; base += 32) {
    const int i = base + lane;
    const bool on = i < j;
    const double c = on ? t.cs[i] : 1.0, s = on ? t.sn[i] : 0.0, h = on ? entry(i + 1) : 0.0;
    double M = on ? -s : 1.0, K = on ? c * h : 0.0;  // lanes past the column: the identity
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double Mu = __shfl_up_sync(0xffffffffu, M, d), Ku = __shfl_up_sync(0xffffffffu, K, d);
      if (lane >= d) {
        K = fma(M, Ku, K);
        M *= Mu;
      }
    }
    const double next = fma(M, a, K);  // a_{i+1}
    double ai = __shfl_up_sync(0xffffffffu, next, 1);
    if (lane == 0) ai = a;
    if (on) out[i] = c * ai + s * h;
    a = __shfl_sync(0xffffffffu, next, 31);
  }
  // lane 0: the rotation's length, lane 1: ||w||; both with their reciprocal
  const double len = sqrt(lane == 0 ? fma(a, a, nrm2) : nrm2);
  const double inv = len > 0.0 ? 1.0 / len : 0.0;
  const double hn = __shfl_sync(0xffffffffu, len, 1), ihn = __shfl_sync(0xffffffffu, inv, 1);
  if (lane != 0) return;
  const double c = len > 0.0 ? a * inv : 1.0, s = len > 0.0 ? hn * inv : 0.0;
  t.cs[j] = c;
  t.sn[j] = s;
  out[j] = len;
  out[j + 1] = 0.0;
  t.g[j + 1] = -s * gj;
  t.g[j] = c * gj;
  t.scal[0] = fabs(s * gj);
  t.scal[1] = ihn;
}

// rows r, r + stride (NR = 2) or r alone (NR = 1): v -= V h, four columns'
// loads in flight per row
template <int NR>
__device__ __forceinline__ void sub_rows(long long n, const double* __restrict__ V, int ncols, const double* nh,
                                         long long r, long long stride, double (&v)[NR]) {
#pragma unroll 1
  for (int c = 0; c < ncols; c += 4) {
    double x[4][NR];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c + u < ncols)
#pragma unroll
        for (int q = 0; q < NR; ++q) x[u][q] = V[(long long)(c + u) * n + r + q * stride];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c + u < ncols)
#pragma unroll
        for (int q = 0; q < NR; ++q) v[q] = fma(x[u][q], nh[c + u], v[q]);
  }
}

// w -= V h over the columns c <= j, one FMA chain per row (ncols + 1 FP64
// operations per row, the norm included; at 15 M rows the FP64 pipe bounds
// it), then the tail on the norm of the updated w.  When *skip only the tail
// runs, on the norm that is already there.
__global__ void __launch_bounds__(RED_THREADS, 4) k_gemv_sub(long long n, const double* __restrict__ V, int j,
                                                              const double* __restrict__ h, double* __restrict__ w,
                                                              double* __restrict__ partials,
                                                              const int* __restrict__ skip,
                                                              unsigned* __restrict__ counter, GsTail t, long long lb) {
  V = lane_ptr(V, lb);
  h = lane_ptr(h, lb);
  w = lane_ptr(w, lb);
  partials = lane_ptr(partials, lb);
  skip = lane_ptr(skip, lb);
  counter = lane_ptr(counter, lb);
  const int ncols = j + 1;
  if (skip && *skip) {
    if (blockIdx.x == 0 && threadIdx.x < 32) {
      t = t.lane(lb);
      givens_step(j, t, *t.nrm2);
    }
    return;
  }
  __shared__ double sh[RED_THREADS / 32];
  __shared__ double nh[64];
  for (int c = threadIdx.x; c < ncols; c += blockDim.x) nh[c] = -h[c];
  __syncthreads();
  double acc = 0.0;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += 2 * stride) {
    if (r + stride < n) {
      double v[2] = {w[r], w[r + stride]};
      sub_rows<2>(n, V, ncols, nh, r, stride, v);
      w[r] = v[0];
      w[r + stride] = v[1];
      acc = fma(v[0], v[0], acc);
      acc = fma(v[1], v[1], acc);
    } else {
      double v[1] = {w[r]};
      sub_rows<1>(n, V, ncols, nh, r, stride, v);
      w[r] = v[0];
      acc = fma(v[0], v[0], acc);
    }
  }
  const double p = block_sum(acc, sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = p;
  if (!last_block(counter, gridDim.x) || threadIdx.x >= 32) return;
  t = t.lane(lb);
  const double nrm = warp_sum_of(partials, gridDim.x);
  if (t.givens) {
    if (threadIdx.x == 0) *t.nrm2 = nrm;
    givens_step(j, t, nrm);
  } else {
    const bool enough = nrm > 0.5 * t.nrm0[0];
    if (threadIdx.x == 0) {
      *t.flag = enough ? 1 : 0;
      if (enough) *t.nrm2 = nrm;
    }
    if (enough)
      for (int c = threadIdx.x; c < ncols; c += 32) t.h2[c] = 0.0;
  }
}

__global__ void __launch_bounds__(RED_THREADS) k_norm_partials(long long n, const double* __restrict__ x,
                                                                double* __restrict__ partials, long long lb) {
  x = lane_ptr(x, lb);
  partials = lane_ptr(partials, lb);
  __shared__ double sh[RED_THREADS / 32];
  double acc = 0.0;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x)
    acc += x[r] * x[r];
  const double t = block_sum(acc, sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

// x_r + sum_c Z[r, c] y_c for c < k, four columns' loads in flight.  With an
// FP32 Z every product is exact in FP64 (the same sums as with the widened
// columns); widen() keeps the conversions off the FP64 pipe.
template <typename ZT>
__device__ __forceinline__ double gemv_row(long long r, long long ld, const ZT* __restrict__ Z, int k,
                                           const double* __restrict__ y, double s) {
#pragma unroll 1
  for (int c = 0; c < k; c += 4) {
    ZT z[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c + u < k) z[u] = Z[(long long)(c + u) * ld + r];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c + u < k) s += widen(z[u]) * y[c + u];
  }
  return s;
}

// x += Z y
template <typename ZT>
__global__ void k_gemv_add(long long n, long long ld, const ZT* __restrict__ Z, int ncols,
                           const double* __restrict__ y, double* __restrict__ x) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) x[r] = gemv_row(r, ld, Z, ncols, y, x[r]);
}

// The next basis vector and the preconditioner's input from it: v = x s and
// t = v mul (FP64, or rounded to FP32 in the mixed form), in one pass.  s is
// s_dev[0], or s_host when s_dev is null; mul is the shared unscaling D_s^-1.
template <typename T>
__global__ void k_next_basis(long long n, const double* __restrict__ x, const double* __restrict__ s_dev,
                             double s_host, const double* __restrict__ mul, double* __restrict__ v,
                             T* __restrict__ t, long long lb) {
  x = lane_ptr(x, lb);
  s_dev = lane_ptr(s_dev, lb);
  v = lane_ptr(v, lb);
  t = lane_ptr(t, lb);
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  const double vr = x[r] * (s_dev ? s_dev[0] : s_host);
  v[r] = vr;
  const double tr = vr * mul[r];
  if constexpr (sizeof(T) == 4) t[r] = narrow(tr);
  else t[r] = tr;
}

// s is a shared elementwise scaling (not a work vector)
__global__ void k_ewise(long long n, const double* __restrict__ x, const double* __restrict__ s, int divide,
                        double* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  y = lane_ptr(y, lb);
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) y[r] = divide ? x[r] / s[r] : x[r] * s[r];
}

// back substitution R y = g (k x k upper triangle of the rotated H) by one
// warp, k <= 64: each lane keeps two entries of the right-hand side, column i
// is loaded while y_i's predecessor is applied (20-55 us in one thread for
// k = 15-50 before)
__device__ __forceinline__ void back_substitute(int k, int m, const double* __restrict__ H,
                                                const double* __restrict__ g, double* __restrict__ y) {
  const int lane = threadIdx.x & 31, l2 = lane + 32;
  double r0 = lane < k ? g[lane] : 0.0, r1 = l2 < k ? g[l2] : 0.0;
  const double d0 = lane < k ? H[(long long)lane * (m + 1) + lane] : 1.0;
  const double d1 = l2 < k ? H[(long long)l2 * (m + 1) + l2] : 1.0;
  const double* col = H + (long long)(k - 1) * (m + 1);
  double c0 = lane < k - 1 ? col[lane] : 0.0, c1 = l2 < k - 1 ? col[l2] : 0.0;
  for (int i = k - 1; i >= 0; --i) {
    double n0 = 0.0, n1 = 0.0;
    if (i > 0) {
      col = H + (long long)(i - 1) * (m + 1);
      n0 = lane < i - 1 ? col[lane] : 0.0;
      n1 = l2 < i - 1 ? col[l2] : 0.0;
    }
    const double rhs = __shfl_sync(0xffffffffu, i < 32 ? r0 : r1, i & 31);
    const double d = __shfl_sync(0xffffffffu, i < 32 ? d0 : d1, i & 31);
    const double yi = d != 0.0 ? rhs / d : 0.0;
    if (lane == 0) y[i] = yi;
    if (lane < i) r0 = fma(-c0, yi, r0);
    if (l2 < i) r1 = fma(-c1, yi, r1);
    c0 = n0;
    c1 = n1;
  }
}

__global__ void k_lsq(int k, int m, const double* __restrict__ H, const double* __restrict__ g, double* __restrict__ y) {
  back_substitute(k, m, H, g, y);
}

__global__ void k_set_g(int m, double beta, double* __restrict__ g) {
  const int i = threadIdx.x + blockIdx.x * blockDim.x;
  if (i <= m) g[i] = (i == 0) ? beta : 0.0;
}


// Blocks of the Gram-Schmidt kernels: no more than the rows fill, and fewer
// on shorter vectors, where the blocks' own reductions and the arrivals at the
// counter cost more than the rows (microseconds, 13 columns, 152 / 304 / 608
// blocks: 175,000 rows 10.3 / 12.6 / 16.2 for the dots and 16.4 / 15.9 / 17.6 for
// the update; 640,000 rows 22.4 / 22.8 / 26.6 and 31.0 / 27.1 / 28.6; 1,884,739
// rows 57.7 / 55.9 / 56.9 and 117 / 73.8 / 60.4, 912 blocks 75.2).
inline unsigned gs_dot_blocks(long long n) {
  return std::min<unsigned>(grid_for(n, RED_THREADS), n < 400000 ? 152u : (n < 4000000 ? 304u : GS_DOT_BLOCKS));
}
inline unsigned gs_sub_blocks(long long n) {
  return std::min<unsigned>(grid_for(n, RED_THREADS), n < 700000 ? 304u : (n < 4000000 ? 608u : GS_BLOCKS));
}

// hout[0..j] = V^T w; with nrm2 non-null also ||w||^2 into nrm2[0];
// with skip non-null nothing happens when *skip != 0
void gs_dots(Ctx& c, int j, double* hout, double* nrm2, const int* skip) {
  const dim3 grid = lgrid(gs_dot_blocks(c.n), j / GS_COLS + 1);
  k_gs_dots<<<grid, RED_THREADS, 0, c.stream>>>(c.n, c.V, j, c.w, c.partials, hout, nrm2, skip,
                                                (unsigned*)(c.dflag + 2), lbytes());
  MHFP_LAUNCH_CHECK();
}

// w -= V h, then the tail t (see GsTail)
void gs_sub(Ctx& c, int j, const double* h, const int* skip, const GsTail& t) {
  k_gemv_sub<<<lgrid(gs_sub_blocks(c.n)), RED_THREADS, 0, c.stream>>>(
      c.n, c.V, j, h, c.w, c.partials + (size_t)c.opt.restart * GS_BLOCKS, skip, (unsigned*)(c.dflag + 1), t,
      lbytes());
  MHFP_LAUNCH_CHECK();
}

// norm^2 into dst (device)
void norm2_dev(Ctx& c, const double* x, long long n, double* dst) {
  k_norm_partials<<<lgrid(RED_BLOCKS), RED_THREADS, 0, c.stream>>>(n, x, c.partials, lbytes());
  MHFP_LAUNCH_CHECK();
  k_reduce_partials<<<lgrid(1), RED_THREADS, 0, c.stream>>>(RED_BLOCKS, c.partials, dst, 0, lbytes());
  MHFP_LAUNCH_CHECK();
}

}  // namespace

void ensure_workspace(Ctx& c) {
  const int m = c.opt.restart;
  if (c.m_alloc == m) return;
  if (c.m_alloc != 0) throw Error{MHFP_ERR_STATE, "restart length cannot change after the first solve"};
  c.V = dalloc_n<double>(c, (size_t)(m + 1) * c.n);
  c.w = dalloc_n<double>(c, c.n);
  c.t = dalloc_n<double>(c, c.n);
  c.tmp = dalloc_n<double>(c, c.n);
  c.h = dalloc_n<double>(c, 2 * (size_t)(m + 1));
  c.H = dalloc_n<double>(c, (size_t)(m + 1) * m);
  c.cs = dalloc_n<double>(c, m);
  c.sn = dalloc_n<double>(c, m);
  c.g = dalloc_n<double>(c, m + 1);
  c.yv = dalloc_n<double>(c, m);
  c.npart = GS_BLOCKS;
  c.partials = dalloc_n<double>(c, (size_t)(m + 2) * GS_BLOCKS);
  c.scal = dalloc_n<double>(c, 8);
  c.dflag = dalloc_n<int>(c, 16);  // DGKS flag, then the Gram-Schmidt kernels' block counters
  MHFP_CUDA(cudaMemsetAsync(c.dflag, 0, 16 * sizeof(int), c.stream));
  if (!c.host_scal) MHFP_CUDA(cudaMallocHost(&c.host_scal, 8 * sizeof(double)));
  c.m_alloc = m;
}

// the preconditioned basis Z in the form the set-up asks for (FP32 in the
// mixed-precision solve, FP64 otherwise), allocated on first use
void ensure_zbasis(Ctx& c) {
  ensure_workspace(c);
  const size_t nz = (size_t)c.opt.restart * c.n;
  if (ff_krylov(c)) {
    if (!c.Zf) {
      c.ldz = (c.n + 3) & ~3LL;
      c.Zf = dalloc_n<float>(c, (size_t)c.opt.restart * c.ldz);
    }
  } else if (!c.Z) {
    c.Z = dalloc_n<double>(c, nz);
  }
}

void vec_scale(Ctx& c, const double* x, const double* s, bool divide, double* y, long long n) {
  k_ewise<<<lgrid(grid_for(n, 256)), 256, 0, c.stream>>>(n, x, s, divide ? 1 : 0, y, lbytes());
  MHFP_LAUNCH_CHECK();
}

__global__ void k_to_f32(long long n, const double* __restrict__ x, float* __restrict__ y, long long lb) {
  x = lane_ptr(x, lb);
  y = lane_ptr(y, lb);
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) y[r] = narrow(x[r]);
}

__global__ void k_to_f64(long long n, const float* __restrict__ x, double* __restrict__ y) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) y[r] = widen(x[r]);
}

// Back substitution with M (Eq. hybridPrec): pi, then p, then u; or, for the
// adjoint, forward substitution with M^T: u, then p, then pi.  The V-cycles
// are symmetric operators (Galerkin levels, R = P^T, the same Chebyshev
// polynomial before and after), so M^T reuses them unchanged.
template <typename T>
void precond_blocks(Ctx& c, const T* t, T* z, T* work_u, T* work_pi, bool transpose) {
  const T* tu = t;
  const T* tp = t + c.nU;
  const T* tpi = tp + c.nT;
  T* zu = z;
  T* zp = z + c.nU;
  T* zpi = zp + c.nT;
  if (!transpose) {
    vcycle(c, c.hpi, tpi, zpi);
    precond_p_step(c, tp, zpi, zp);
    const FirstStep<T> fs = first_step(c, c.hu, zu);
    precond_u_rhs(c, tu, zp, work_u, fs);
    vcycle(c, c.hu, (const T*)work_u, zu, fs.dinv != nullptr);
  } else {
    vcycle(c, c.hu, tu, zu);
    precondT_p_step(c, tp, zu, zp);
    precondT_pi_rhs(c, tpi, zp, work_pi);
    vcycle(c, c.hpi, (const T*)work_pi, zpi);
  }
}

// z = M^-1 v (or M^-T) with the FP32 V-cycles and Schur steps: v FP64, or,
// when null, already rounded in the handle's FP32 vector c.tf; the FP32
// result in zf_out (default: the handle's FP32 work vector) and, when z is
// given, widened into z
void apply_precond_mixed(Ctx& c, const double* v, double* z, bool transpose, float* zf_out = nullptr) {
  const long long n = c.n;
  float* zo = zf_out ? zf_out : c.zf;
  timing_begin(c, 3);
  if (v) {
    k_to_f32<<<lgrid(grid_for(n, 256)), 256, 0, c.stream>>>(n, v, c.tf, lbytes());
    MHFP_LAUNCH_CHECK();
  }
  // level-0 right-hand-side buffers are free at the finest levels
  precond_blocks<float>(c, c.tf, zo, c.hu[0].bf, c.hpi[0].bf, transpose);
  if (z) {
    k_to_f64<<<grid_for(n, 256), 256, 0, c.stream>>>(n, zo, z);
    MHFP_LAUNCH_CHECK();
  }
  timing_end(c, 3, 0.0);
}

// M_II^(m) of Eq. (prec) for the mixed formulation [u | p | q], by forward
// substitution: z_u = V_u(v_u), z_q = Chebyshev(A_qq) v_q, then
// z_p = V_Cp(v_p - A_pu z_u - dt A_pq z_q)
void apply_precond_btp(Ctx& c, const double* v, double* z) {
  const double* vu = v;
  const double* vp = v + c.nU;
  const double* vq = vp + c.nT;
  double* zu = z;
  double* zp = z + c.nU;
  double* zq = zp + c.nT;
  timing_begin(c, 3);
  vcycle(c, c.hu, vu, zu);
  chebyshev_from_zero(c, c.hq, vq, zq);
  double* tp = c.hcp[0].b;  // level 0's right-hand-side buffer is free here
  btp_p_rhs(c, vp, zu, zq, tp);
  vcycle(c, c.hcp, (const double*)tp, zp);
  timing_end(c, 3, 0.0);
}

void apply_precond(Ctx& c, const double* v, double* z, bool transpose) {
  if (c.opt.formulation == 1) {
    if (transpose) throw Error{MHFP_ERR_STATE, "the mixed formulation has no transposed preconditioner"};
    apply_precond_btp(c, v, z);
    return;
  }
  if (c.opt.precision == 1) {
    apply_precond_mixed(c, v, z, transpose);
    return;
  }
  timing_begin(c, 3);
  precond_blocks<double>(c, v, z, c.hu[0].b, c.hpi[0].b, transpose);
  timing_end(c, 3, 0.0);
}

// basis vector `col` from x: V[:, col] = x s and the preconditioner's input
// D_s^-1 V[:, col] in c.tf (FP32 form) or c.t
void enqueue_next_basis(Ctx& c, int col, const double* x, const double* s_dev, double s_host = 0.0) {
  const long long n = c.n;
  double* v = c.V + (long long)col * n;
  const dim3 grid = lgrid(grid_for(n, 256));
  if (c.opt.precision == 1)
    k_next_basis<float><<<grid, 256, 0, c.stream>>>(n, x, s_dev, s_host, c.ds_inv, v, c.tf, lbytes());
  else
    k_next_basis<double><<<grid, 256, 0, c.stream>>>(n, x, s_dev, s_host, c.ds_inv, v, c.t, lbytes());
  MHFP_LAUNCH_CHECK();
}

// Enqueue Arnoldi step j (V[:, j] and the preconditioner's input are there,
// enqueue_next_basis): z_j = M^-1 v_j, w = D_s A z_j, Gram-Schmidt with the
// Givens update, v_{j+1}, and the copy of |g_{j+1}| to pinned host memory.
void enqueue_arnoldi_step(Ctx& c, int j, bool transpose, bool host_copy = true) {
  const int m = c.opt.restart;
  const long long n = c.n;
  if (ff_krylov(c)) {
    // z_j stays in FP32 (it is the FP32 preconditioner's output): the
    // float-float operator reads it, and x += Z y widens it
    float* zfj = c.Zf + (long long)j * c.ldz;
    apply_precond_mixed(c, nullptr, nullptr, transpose, zfj);
    apply_operator_arnoldi(c, nullptr, zfj, c.w, c.ds, transpose);  // w = D_s A z_j
  } else {
    double* zj = c.Z + (long long)j * n;
    if (c.opt.precision == 1) apply_precond_mixed(c, nullptr, zj, transpose);
    else apply_precond(c, c.t, zj, transpose);
    apply_operator_arnoldi(c, zj, c.zf, c.w, c.ds, transpose);  // w = D_s A z_j
  }
  timing_begin(c, 2);
  // classical Gram-Schmidt with the DGKS reorthogonalisation test:
  // h1 = V^T w and ||w||^2; w -= V h1 and ||w||^2; then, only if the
  // norm dropped by more than 1/sqrt(2), h2 = V^T w and w -= V h2
  // (reorth = 0: the first pass alone, the second is not even queued)
  const bool reorth = c.opt.reorth != 0;
  double* h2 = c.h + (m + 1);
  GsTail tail{};
  tail.nrm0 = c.scal + 4;
  tail.flag = c.dflag;
  tail.h2 = reorth ? h2 : nullptr;
  tail.nrm2 = c.scal + 2;
  tail.h1 = c.h;
  tail.H = c.H;
  tail.cs = c.cs;
  tail.sn = c.sn;
  tail.g = c.g;
  tail.scal = c.scal;
  tail.m = m;
  tail.givens = reorth ? 0 : 1;
  gs_dots(c, j, c.h, reorth ? c.scal + 4 : nullptr, nullptr);
  gs_sub(c, j, c.h, nullptr, tail);
  if (reorth) {
    tail.givens = 1;
    gs_dots(c, j, h2, nullptr, c.dflag);
    gs_sub(c, j, h2, c.dflag, tail);
  }
  timing_end(c, 2, 8.0 * n * (2.0 * (j + 1) + 4.0));
  if (j + 1 < m) enqueue_next_basis(c, j + 1, c.w, c.scal + 1);  // the last step's successor is never used
  if (host_copy) MHFP_CUDA(cudaMemcpyAsync(c.host_scal, c.scal, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
}

namespace {

// Queue Arnoldi step j (no synchronisation).  With graphs enabled the step
// is captured once per (j, transpose) on a private stream and replayed into
// the handle's stream afterwards: one launch instead of about 50.
IterGraph* launch_arnoldi_step(Ctx& c, int j, bool transpose) {
  if (!c.opt.graphs) {
    enqueue_arnoldi_step(c, j, transpose);
    return nullptr;
  }
  auto& G = c.graphs[transpose ? 1 : 0];
  if ((int)G.size() < c.opt.restart) G.resize(c.opt.restart);
  IterGraph& ig = G[j];
  if (!ig.exec) {
    if (!c.cap_stream) MHFP_CUDA(cudaStreamCreateWithFlags(&c.cap_stream, cudaStreamNonBlocking));
    cudaStream_t user = c.stream;
    const long long l0 = g_launches;
    c.stream = c.cap_stream;
    c.timing.capturing = true;
    c.timing.capture_list = &ig.timed;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(c.cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      try {
        enqueue_arnoldi_step(c, j, transpose);
      } catch (...) {
        cudaStreamEndCapture(c.cap_stream, &graph);
        if (graph) cudaGraphDestroy(graph);
        c.stream = user;
        c.timing.capturing = false;
        throw;
      }
      e = cudaStreamEndCapture(c.cap_stream, &graph);
    }
    c.stream = user;
    c.timing.capturing = false;
    c.timing.capture_list = nullptr;
    MHFP_CUDA(e);
    ig.nkernels = g_launches - l0;
    g_launches = l0;  // nothing ran during the capture
    e = cudaGraphInstantiate(&ig.exec, graph, 0);
    cudaGraphDestroy(graph);
    MHFP_CUDA(e);
  }
  MHFP_CUDA(cudaGraphLaunch(ig.exec, c.stream));
  g_launches += ig.nkernels;
  return &ig;
}

// queue D_s (b - A x) and its squared norm into host_scal[0]
void enqueue_residual(Ctx& c, const FgState& f) {
  apply_operator(c, f.x, c.tmp, c.ds, f.b, f.transpose);
  norm2_dev(c, c.tmp, c.n, c.scal + 4);
  MHFP_CUDA(cudaMemcpyAsync(c.host_scal, c.scal + 4, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
}

void finish(Ctx& c, FgState& f, double true_rel) {
  f.converged = f.converged || true_rel <= 1.05 * f.tol;
  f.stats.iterations = f.total;
  f.stats.restarts = f.cycles;
  f.stats.converged = f.converged ? 1 : 0;
  f.stats.rel_residual = f.est;
  f.stats.true_rel_residual = true_rel;
  f.stats.solve_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - f.t0).count();
  f.phase = FgState::DONE;
  if (!f.converged) throw Error{MHFP_ERR_NOT_CONVERGED, "FGMRES reached maxit before the tolerance"};
}

}  // namespace

// Start a solve: x = 0 and ||D_s b|| queued; the caller synchronises the
// handle's stream and calls fgmres_advance until the state is DONE.
void fgmres_begin(Ctx& c, FgState& f, const double* b, double* x, double tol, bool transpose) {
  f = FgState{};
  f.b = b;
  f.x = x;
  f.tol = tol;
  f.transpose = transpose;
  f.t0 = std::chrono::steady_clock::now();
  ensure_zbasis(c);
  MHFP_CUDA(cudaMemsetAsync(x, 0, c.n * sizeof(double), c.stream));
  vec_scale(c, b, c.ds, false, c.tmp, c.n);
  norm2_dev(c, c.tmp, c.n, c.scal + 4);
  MHFP_CUDA(cudaMemcpyAsync(c.host_scal, c.scal + 4, sizeof(double), cudaMemcpyDeviceToHost, c.stream));
  f.phase = FgState::NEED_BNORM;
}

// One state transition, after the handle's stream has drained: read the
// scalar the last queued work produced and queue the next piece of work.
// Right-preconditioned FGMRES(m), zero initial guess (Section 5), on the
// equilibrated system; a cycle restarts from the true residual, and the
// solve ends when that true residual meets 1.05 tol (or maxit is reached).
void fgmres_advance(Ctx& c, FgState& f) {
  const int m = c.opt.restart;
  const long long n = c.n;
  switch (f.phase) {
    case FgState::NEED_BNORM: {
      f.bnorm = std::sqrt(c.host_scal[0]);
      if (!std::isfinite(f.bnorm)) throw Error{MHFP_ERR_NONFINITE, "non-finite right-hand side"};
      if (f.bnorm == 0.0) {
        f.converged = true;
        f.est = 0.0;
        finish(c, f, 0.0);
        return;
      }
      enqueue_residual(c, f);
      f.phase = FgState::NEED_BETA;
      return;
    }
    case FgState::NEED_BETA: {
      const double beta = std::sqrt(c.host_scal[0]);
      if (!std::isfinite(beta)) throw Error{MHFP_ERR_NONFINITE, "non-finite residual"};
      if (beta <= 1.05 * f.tol * f.bnorm) {
        f.converged = true;
        f.est = beta / f.bnorm;
        finish(c, f, beta / f.bnorm);
        return;
      }
      if (f.total >= c.opt.maxit) {
        finish(c, f, beta / f.bnorm);
        return;
      }
      enqueue_next_basis(c, 0, c.tmp, nullptr, 1.0 / beta);
      k_set_g<<<1, 64, 0, c.stream>>>(m, beta, c.g);
      MHFP_LAUNCH_CHECK();
      f.j = 0;
      f.graph = launch_arnoldi_step(c, 0, f.transpose);
      f.phase = FgState::NEED_RESID;
      return;
    }
    case FgState::NEED_RESID: {
      if (f.graph && c.timing.enabled)
        for (auto& t : f.graph->timed) {
          float ms = 0.f;
          MHFP_CUDA(cudaEventElapsedTime(&ms, t.start, t.stop));
          c.timing.total_ms[t.cls] += ms;
          c.timing.launches[t.cls] += 1;
          c.timing.bytes[t.cls] += t.bytes;
        }
      const double resid = c.host_scal[0];
      ++f.total;
      const int k = f.j + 1;
      f.est = resid / f.bnorm;
      if (!std::isfinite(resid)) throw Error{MHFP_ERR_NONFINITE, "non-finite Arnoldi residual"};
      if (resid <= f.tol * f.bnorm || f.total >= c.opt.maxit || k == m) {
        k_lsq<<<1, 32, 0, c.stream>>>(k, m, c.H, c.g, c.yv);
        MHFP_LAUNCH_CHECK();
        if (ff_krylov(c))
          k_gemv_add<float><<<grid_for(n, 256), 256, 0, c.stream>>>(n, c.ldz, c.Zf, k, c.yv, f.x);
        else
          k_gemv_add<double><<<grid_for(n, 256), 256, 0, c.stream>>>(n, n, c.Z, k, c.yv, f.x);
        MHFP_LAUNCH_CHECK();
        ++f.cycles;
        enqueue_residual(c, f);
        f.phase = FgState::NEED_BETA;
        return;
      }
      f.j = k;
      f.graph = launch_arnoldi_step(c, f.j, f.transpose);
      return;
    }
    default:
      return;
  }
}

// ---------------------------------------------------------------------------
// Device-driven solve: the whole FGMRES(m) -- restart cycles in a WHILE
// conditional node, Arnoldi step j in IF node j -- is one CUDA graph,
// launched once per solve.  The decisions the host loop makes (stop, restart,
// next step) are taken by single-thread kernels that read the residual
// estimates on the device and set the conditional handles.  Every loop is
// bounded: a cycle runs at most m steps and the WHILE ends once maxit steps
// have run.

// Several lanes (right-hand sides of one handle in lockstep): the control
// kernels run in one thread and walk the lanes, lane l's control block,
// scalars and Hessenberg data lb bytes after lane l - 1's.  A lane whose
// solve has ended (fin) is skipped; the set goes on while any lane has not
// ended, and a cycle's next step opens while any lane is live in it.  With
// one lane every decision is the single solve's.
template <class T>
__device__ __forceinline__ T* lane_at(T* p, int l, long long lb) {
  return (T*)((char*)p + (long long)l * lb);
}

__global__ void k_ctl_init(DevCtl* __restrict__ ctl, const double* __restrict__ nrm2, cudaGraphConditionalHandle hw,
                           int K, long long lb) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  bool any = false;
  for (int l = 0; l < K; ++l) {
    DevCtl* c = lane_at(ctl, l, lb);
    const double bn = sqrt(lane_at(nrm2, l, lb)[0]);
    c->bnorm = bn;
    c->tolb = c->tol * bn;
    c->est = 1.0;
    c->true_rel = 0.0;
    c->total = 0;
    c->cycles = 0;
    c->k = 0;
    c->converged = 0;
    c->status = 0;
    c->pad3 = 0;  // cycle starts, a second bound on the WHILE loop
    c->fin = 0;
    c->live = 0;
    if (!isfinite(bn)) {
      c->status = (int)MHFP_ERR_NONFINITE;
      c->fin = 1;
    } else if (bn == 0.0) {
      c->converged = 1;
      c->est = 0.0;
      c->fin = 1;
    } else {
      any = true;
    }
  }
  ctl->decides = 0;
  ctl->steps = 0;
  cudaGraphSetConditional(hw, any ? 1 : 0);
}

// start of a cycle: beta = ||D_s (b - A x)|| per lane; a lane stops, or
// takes part in the cycle; step 0 opens while any lane takes part
__global__ void k_cycle_decide(DevCtl* __restrict__ ctl, const double* __restrict__ nrm2, double* __restrict__ scal,
                               double* __restrict__ g, cudaGraphConditionalHandle hw,
                               const cudaGraphConditionalHandle* __restrict__ hif, int K, long long lb) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int m = ctl->m;
  ctl->decides += 1;
  bool any = false;
  for (int l = 0; l < K; ++l) {
    DevCtl* c = lane_at(ctl, l, lb);
    double* sc = lane_at(scal, l, lb);
    c->k = 0;
    c->live = 0;
    if (c->fin) {
      sc[6] = 0.0;
      continue;
    }
    const double beta = sqrt(lane_at(nrm2, l, lb)[0]);
    c->pad3 += 1;
    // every cycle either runs at least one step (total grows by one) or
    // stops; the count of cycle starts bounds the loop even if a step did
    // not run, so the WHILE node always terminates
    bool stop = c->pad3 > c->maxit + 1;
    if (stop) {
      c->true_rel = beta / c->bnorm;
    } else if (!isfinite(beta)) {
      c->status = (int)MHFP_ERR_NONFINITE;
      stop = true;
    } else if (beta <= 1.05 * c->tolb) {
      c->converged = 1;
      c->est = beta / c->bnorm;
      c->true_rel = beta / c->bnorm;
      stop = true;
    } else if (c->total >= c->maxit) {
      c->true_rel = beta / c->bnorm;
      stop = true;
    }
    if (stop) {
      c->fin = 1;
      sc[6] = 0.0;
      continue;
    }
    c->live = 1;
    any = true;
    double* gl = lane_at(g, l, lb);
    sc[6] = 1.0 / beta;
    gl[0] = beta;
    for (int i = 1; i <= m; ++i) gl[i] = 0.0;
  }
  if (!any) {
    cudaGraphSetConditional(hw, 0);
    for (int j = 0; j < m; ++j) cudaGraphSetConditional(hif[j], 0);
    return;
  }
  cudaGraphSetConditional(hif[0], 1);
  for (int j = 1; j < m; ++j) cudaGraphSetConditional(hif[j], 0);
}

// after Arnoldi step j: count it for every live lane, and open step j+1
// unless no lane is live any more (converged in the Arnoldi estimate, maxit
// or a non-finite residual); a lane that leaves keeps k, its step count of
// this cycle, for the update x += Z y
__global__ void k_step_done(DevCtl* __restrict__ ctl, const double* __restrict__ scal, int j,
                            cudaGraphConditionalHandle hnext, int has_next, cudaGraphConditionalHandle hw, int K,
                            long long lb) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  ctl->steps += 1;
  bool any_next = false, all_fin = true;
  for (int l = 0; l < K; ++l) {
    DevCtl* c = lane_at(ctl, l, lb);
    if (c->live) {
      const double resid = lane_at(scal, l, lb)[0];
      c->total += 1;
      c->k = j + 1;
      c->est = resid / c->bnorm;
      bool next = has_next && resid > c->tolb && c->total < c->maxit;
      if (!isfinite(resid)) {
        c->status = (int)MHFP_ERR_NONFINITE;
        c->fin = 1;
        next = false;
      }
      if (!next) c->live = 0;
      any_next = any_next || next;
    }
    all_fin = all_fin && c->fin;
  }
  if (all_fin) cudaGraphSetConditional(hw, 0);
  if (has_next) cudaGraphSetConditional(hnext, any_next ? 1 : 0);
}

__global__ void k_lsq_dev(const DevCtl* __restrict__ ctl, const double* __restrict__ H, const double* __restrict__ g,
                          double* __restrict__ y, long long lb) {
  ctl = lane_ptr(ctl, lb);
  back_substitute(ctl->k, ctl->m, lane_ptr(H, lb), lane_ptr(g, lb), lane_ptr(y, lb));
}

template <typename ZT>
__global__ void k_gemv_add_dev(long long n, long long ld, const ZT* __restrict__ Z, const DevCtl* __restrict__ ctl,
                               const double* __restrict__ y, double* __restrict__ x, long long lb) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  x = lane_ptr(x, lb);
  x[r] = gemv_row(r, ld, lane_ptr(Z, lb), lane_ptr(ctl, lb)->k, lane_ptr(y, lb), x[r]);
}

__global__ void k_cycle_end(DevCtl* __restrict__ ctl, long long lb) {
  ctl = lane_ptr(ctl, lb);
  if (threadIdx.x == 0 && blockIdx.x == 0 && ctl->k > 0) ctl->cycles += 1;
}

namespace {

template <typename... P, typename... A>
cudaGraphNode_t add_kernel(cudaGraph_t g, cudaGraphNode_t dep, void (*f)(P...), dim3 grid, dim3 block, A... args) {
  void* params[] = {(void*)&args...};
  cudaKernelNodeParams kp{};
  kp.func = (void*)f;
  kp.gridDim = grid;
  kp.blockDim = block;
  kp.sharedMemBytes = 0;
  kp.kernelParams = params;
  kp.extra = nullptr;
  cudaGraphNode_t node;
  MHFP_CUDA(cudaGraphAddKernelNode(&node, g, dep ? &dep : nullptr, dep ? 1 : 0, &kp));
  ++g_launches;  // counted like a launch; removed again after the build
  return node;
}

template <class F>
cudaGraph_t capture_piece(Ctx& c, F&& enqueue) {
  if (!c.cap_stream) MHFP_CUDA(cudaStreamCreateWithFlags(&c.cap_stream, cudaStreamNonBlocking));
  cudaStream_t user = c.stream;
  c.stream = c.cap_stream;
  c.suppress_events = true;
  cudaGraph_t graph = nullptr;
  MHFP_CUDA(cudaStreamBeginCapture(c.cap_stream, cudaStreamCaptureModeThreadLocal));
  try {
    enqueue();
  } catch (...) {
    cudaStreamEndCapture(c.cap_stream, &graph);
    if (graph) cudaGraphDestroy(graph);
    c.stream = user;
    c.suppress_events = false;
    throw;
  }
  cudaError_t e = cudaStreamEndCapture(c.cap_stream, &graph);
  c.stream = user;
  c.suppress_events = false;
  MHFP_CUDA(e);
  return graph;
}

cudaGraphNode_t add_child(cudaGraph_t parent, cudaGraphNode_t dep, cudaGraph_t child) {
  cudaGraphNode_t node;
  cudaError_t e = cudaGraphAddChildGraphNode(&node, parent, dep ? &dep : nullptr, dep ? 1 : 0, child);
  cudaGraphDestroy(child);
  MHFP_CUDA(e);
  return node;
}

cudaGraphNode_t add_conditional(cudaGraph_t parent, cudaGraphNode_t dep, cudaGraphConditionalHandle h,
                                cudaGraphConditionalNodeType type, cudaGraph_t* body) {
  cudaGraphNodeParams np{};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = h;
  np.conditional.type = type;
  np.conditional.size = 1;
  cudaGraphNode_t node;
  MHFP_CUDA(cudaGraphAddNode(&node, parent, dep ? &dep : nullptr, nullptr, dep ? 1 : 0, &np));
  *body = np.conditional.phGraph_out[0];
  return node;
}

__global__ void k_ctl_reset(DevCtl* __restrict__ ctl, double tol, int maxit, int m, long long lb) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  ctl = lane_ptr(ctl, lb);
  DevCtl h{};
  h.tol = tol;
  h.maxit = maxit;
  h.m = m;
  *ctl = h;
}

// Add one whole device-driven solve of handle c to graph G after `dep`:
// [b -> bcur, control block reset] x = 0, ||D_s b||, the control block's
// start, the WHILE node of the restart cycles (Arnoldi steps in IF nodes),
// [xcur -> x] and the control block -> host_slot.  The bracketed parts are
// added when rhs / x are given (batched graphs); the single-solve graph
// leaves them to the host.  d_hif: device array of `restart` IF handles for
// this solve.  With K lanes (c a lane workspace, lane l's work vectors lb
// bytes after lane l - 1's) the solve takes K right-hand sides rhs[0..K)
// in lockstep into x[0..K), control blocks to host_slot[0..K).  Returns the
// last node; the kernel counts go to *cnt.
struct SolveCounts {
  long long start = 0, cycle = 0, step = 0;
};

cudaGraphNode_t add_solve(Ctx& c, cudaGraph_t G, cudaGraphNode_t dep, bool transpose,
                          cudaGraphConditionalHandle* d_hif, const double* const* rhs, double* const* x, double tol,
                          DevCtl* const* host_slot, SolveCounts* cnt, int K = 1, long long lb = 0) {
  const int m = c.opt.restart;
  const long long n = c.n;
  const long long l0 = g_launches;
  LaneScope lanes(K, lb);
  // the WHILE node sits in G, the IF nodes in the WHILE body: each handle is
  // created on the graph that contains its node
  cudaGraphConditionalHandle hw;
  MHFP_CUDA(cudaGraphConditionalHandleCreate(&hw, G, 1, cudaGraphCondAssignDefault));
  DevCtl* ctl = c.ctl;
  cudaGraphNode_t last = dep;
  if (rhs) {
    for (int l = 0; l < K; ++l) {
      cudaGraphNode_t cp;
      MHFP_CUDA(cudaGraphAddMemcpyNode1D(&cp, G, last ? &last : nullptr, last ? 1 : 0,
                                         (char*)c.bcur + (long long)l * lb, rhs[l], n * sizeof(double),
                                         cudaMemcpyDeviceToDevice));
      last = cp;
    }
    last = add_kernel(G, last, k_ctl_reset, lgrid(1), dim3(32), ctl, tol, c.opt.maxit, m, lb);
  }
  // x = 0, ||D_s b|| and the control block
  last = add_child(G, last, capture_piece(c, [&] {
    MHFP_CUDA(lane_memset(c.xcur, 0, n * sizeof(double), c.stream));
    vec_scale(c, c.bcur, c.ds, false, c.tmp, n);
    norm2_dev(c, c.tmp, n, c.scal + 4);
  }));
  last = add_kernel(G, last, k_ctl_init, dim3(1), dim3(32), ctl, (const double*)(c.scal + 4), hw, K, lb);
  const long long nk_start = g_launches - l0;
  cudaGraph_t W;
  cudaGraphNode_t wnode = add_conditional(G, last, hw, cudaGraphCondTypeWhile, &W);
  std::vector<cudaGraphConditionalHandle> hif(m);
  for (int j = 0; j < m; ++j) MHFP_CUDA(cudaGraphConditionalHandleCreate(&hif[j], W, 0, 0));
  MHFP_CUDA(cudaMemcpy(d_hif, hif.data(), m * sizeof(cudaGraphConditionalHandle), cudaMemcpyHostToDevice));
  // while body: the cycle
  const long long l1 = g_launches;
  cudaGraphNode_t b = add_child(W, nullptr, capture_piece(c, [&] {
    apply_operator(c, c.xcur, c.tmp, c.ds, c.bcur, transpose);
    norm2_dev(c, c.tmp, n, c.scal + 4);
  }));
  b = add_kernel(W, b, k_cycle_decide, dim3(1), dim3(32), ctl, (const double*)(c.scal + 4), c.scal, c.g, hw,
                 (const cudaGraphConditionalHandle*)d_hif, K, lb);
  b = add_child(W, b, capture_piece(c, [&] {
    enqueue_next_basis(c, 0, c.tmp, c.scal + 6);
  }));
  const long long nk_cycle = g_launches - l1;
  long long nk_step = 0;
  for (int j = 0; j < m; ++j) {
    cudaGraph_t body;
    b = add_conditional(W, b, hif[j], cudaGraphCondTypeIf, &body);
    const long long l2 = g_launches;
    cudaGraphNode_t s = add_child(body, nullptr, capture_piece(c, [&] { enqueue_arnoldi_step(c, j, transpose, false); }));
    add_kernel(body, s, k_step_done, dim3(1), dim3(32), ctl, (const double*)c.scal, j,
               j + 1 < m ? hif[j + 1] : hif[j], j + 1 < m ? 1 : 0, hw, K, lb);
    nk_step = g_launches - l2;
  }
  const long long l3 = g_launches;
  b = add_child(W, b, capture_piece(c, [&] {
    k_lsq_dev<<<lgrid(1), 32, 0, c.stream>>>(ctl, c.H, c.g, c.yv, lbytes());
    MHFP_LAUNCH_CHECK();
    if (ff_krylov(c))
      k_gemv_add_dev<float><<<lgrid(grid_for(n, 256)), 256, 0, c.stream>>>(n, c.ldz, c.Zf, ctl, c.yv, c.xcur,
                                                                           lbytes());
    else
      k_gemv_add_dev<double><<<lgrid(grid_for(n, 256)), 256, 0, c.stream>>>(n, n, c.Z, ctl, c.yv, c.xcur,
                                                                            lbytes());
    MHFP_LAUNCH_CHECK();
    k_cycle_end<<<lgrid(1), 32, 0, c.stream>>>(ctl, lbytes());
    MHFP_LAUNCH_CHECK();
  }));
  const long long nk_end = g_launches - l3;
  last = wnode;
  if (x) {
    for (int l = 0; l < K; ++l) {
      cudaGraphNode_t cp;
      MHFP_CUDA(cudaGraphAddMemcpyNode1D(&cp, G, &last, 1, x[l], (const char*)c.xcur + (long long)l * lb,
                                         n * sizeof(double), cudaMemcpyDeviceToDevice));
      last = cp;
    }
  }
  // after the loop: the control blocks back to pinned host memory
  for (int l = 0; l < K; ++l) {
    cudaGraphNode_t fin;
    MHFP_CUDA(cudaGraphAddMemcpyNode1D(&fin, G, &last, 1, host_slot[l], (const char*)ctl + (long long)l * lb,
                                       sizeof(DevCtl), cudaMemcpyDeviceToHost));
    last = fin;
  }
  cnt->start = nk_start;
  cnt->cycle = nk_cycle + nk_end;
  cnt->step = nk_step;
  return last;
}

// the handle's device-side solve state (control block, current b and x)
void ensure_solve_state(Ctx& c) {
  ensure_zbasis(c);
  if (!c.ctl) {
    c.ctl = dalloc_n<DevCtl>(c, 1);
    MHFP_CUDA(cudaMallocHost(&c.host_ctl, sizeof(DevCtl)));
    c.bcur = dalloc_n<double>(c, c.n);
    c.xcur = dalloc_n<double>(c, c.n);
  }
}

void build_solve_graph(Ctx& c, bool transpose) {
  ensure_solve_state(c);
  const int ti = transpose ? 1 : 0;
  if (!c.d_hif[ti]) c.d_hif[ti] = dalloc_n<cudaGraphConditionalHandle>(c, c.opt.restart);
  const long long l0 = g_launches;
  cudaGraph_t G;
  MHFP_CUDA(cudaGraphCreate(&G, 0));
  SolveCounts cnt;
  DevCtl* slot = c.host_ctl;
  try {
    add_solve(c, G, nullptr, transpose, c.d_hif[ti], nullptr, nullptr, 0.0, &slot, &cnt);
  } catch (...) {
    g_launches = l0;
    cudaGraphDestroy(G);
    throw;
  }
  g_launches = l0;  // nothing ran during the build
  cudaGraphExec_t exec;
  cudaError_t e = cudaGraphInstantiate(&exec, G, 0);
  cudaGraphDestroy(G);
  MHFP_CUDA(e);
  c.solve_exec[ti] = exec;
  // launches of one solve = start + per cycle (cycle + end) + per step
  c.solve_nkernels[ti] = cnt.start;
  c.solve_cycle_kernels[ti] = cnt.cycle;
  c.solve_step_kernels[ti] = cnt.step;
}

// A lockstep workspace for K right-hand sides of handle `base`: a copy of
// the handle that shares every matrix, hierarchy and launch schedule, with
// its own work vectors (Krylov basis, Hessenberg data, control block, the
// levels' vectors) carved from one arena: lane 0's at the start, lane l's
// l * lane_bytes further.
Ctx* make_lane_ctx(Ctx& base, int K) {
  if (base.opt.formulation != 0)
    throw Error{MHFP_ERR_STATE, "right-hand sides in lockstep are solved for the hybrid system only"};
  ensure_solve_state(base);
  Ctx* lc = new Ctx(base);
  lc->allocs.clear();
  lc->arena = nullptr;
  lc->arena_left = 0;
  lc->timing = Timing{};
  lc->suppress_events = false;
  lc->cap_stream = nullptr;
  lc->graphs[0].clear();
  lc->graphs[1].clear();
  lc->solve_exec[0] = lc->solve_exec[1] = nullptr;
  lc->d_hif[0] = lc->d_hif[1] = nullptr;
  lc->host_scal = nullptr;
  lc->host_ctl = nullptr;
  // the lane layout: every work vector at a 256-byte aligned offset
  struct Slot {
    void** p;
    size_t bytes;
  };
  std::vector<Slot> slots;
  const int m = base.opt.restart;
  const size_t n = (size_t)base.n;
  auto add = [&](auto*& p, size_t bytes) { slots.push_back({(void**)&p, bytes}); };
  add(lc->V, (size_t)(m + 1) * n * sizeof(double));
  add(lc->w, n * sizeof(double));
  add(lc->t, n * sizeof(double));
  add(lc->tmp, n * sizeof(double));
  add(lc->h, 2 * (size_t)(m + 1) * sizeof(double));
  add(lc->H, (size_t)(m + 1) * m * sizeof(double));
  add(lc->cs, (size_t)m * sizeof(double));
  add(lc->sn, (size_t)m * sizeof(double));
  add(lc->g, (size_t)(m + 1) * sizeof(double));
  add(lc->yv, (size_t)m * sizeof(double));
  add(lc->partials, (size_t)(m + 2) * GS_BLOCKS * sizeof(double));
  add(lc->scal, 8 * sizeof(double));
  add(lc->dflag, 16 * sizeof(int));
  if (base.Zf) add(lc->Zf, (size_t)m * (size_t)base.ldz * sizeof(float));  // mixed precision: FP32 Z
  if (base.Z) add(lc->Z, (size_t)m * n * sizeof(double));                  // FP64 throughout
  if (base.tf) add(lc->tf, n * sizeof(float));
  if (base.zf) add(lc->zf, n * sizeof(float));
  add(lc->ctl, sizeof(DevCtl));
  add(lc->bcur, n * sizeof(double));
  add(lc->xcur, n * sizeof(double));
  for (auto* H : {&lc->hu, &lc->hpi})
    for (Level& L : *H) {
      const size_t ld = (size_t)L.n * sizeof(double), lf = (size_t)L.n * sizeof(float);
      for (double** v : {&L.x, &L.b, &L.r, &L.d, &L.y})
        if (*v) add(*v, ld);
      for (float** v : {&L.xf, &L.bf, &L.rf, &L.df, &L.yf})
        if (*v) add(*v, lf);
    }
  size_t lane = 0;
  std::vector<size_t> off(slots.size());
  for (size_t i = 0; i < slots.size(); ++i) {
    off[i] = lane;
    lane += (slots[i].bytes + 255) & ~(size_t)255;
  }
  try {
    char* arena = (char*)dalloc(*lc, lane * (size_t)K);
    MHFP_CUDA(cudaMemsetAsync(arena, 0, lane * (size_t)K, base.stream));
    for (size_t i = 0; i < slots.size(); ++i) *slots[i].p = arena + off[i];
    lc->lane_bytes = (long long)lane;
    lc->lanes = K;
  } catch (...) {
    dfree_all(*lc);
    delete lc;
    throw;
  }
  return lc;
}

void destroy_lane_ctx(Ctx* lc) {
  if (!lc) return;
  if (lc->cap_stream) cudaStreamDestroy(lc->cap_stream);
  dfree_all(*lc);
  delete lc;
}

}  // namespace

// One CUDA graph for many solves: every handle's entries run in list order
// in a branch of their own (they share its Krylov workspace); branches of
// different handles are independent, so one launch runs them all.  With
// max_lanes > 1 a handle's entries are taken in sets of up to max_lanes
// right-hand sides, each set one lockstep solve in a workspace of its own.
void build_batch_graph(BatchGraph& B, const std::vector<Ctx*>& cs, const std::vector<const double*>& rhs,
                       const std::vector<double*>& x, double tol, int max_lanes) {
  const long long l0 = g_launches;
  MHFP_CUDA(cudaGraphCreate(&B.graph, 0));
  const int count = (int)cs.size();
  B.counts.assign(count, {0, 0, 0});
  B.lanes.assign(count, 1);
  B.lead.assign(count, 0);
  MHFP_CUDA(cudaMallocHost(&B.host_ctl, (size_t)std::max(count, 1) * sizeof(DevCtl)));
  std::vector<std::pair<Ctx*, cudaGraphNode_t>> tail;  // last node of each handle's branch
  std::vector<bool> taken(count, false);
  try {
    for (int i = 0; i < count; ++i) {
      if (taken[i]) continue;
      Ctx& c = *cs[i];
      // this entry and the next entries of the same handle, up to max_lanes
      std::vector<int> set{i};
      for (int k = i + 1; k < count && (int)set.size() < max_lanes; ++k)
        if (cs[k] == &c && !taken[k]) set.push_back(k);
      for (int e : set) taken[e] = true;
      const int K = (int)set.size();
      ensure_solve_state(c);
      Ctx* run = &c;
      if (K > 1) {
        // one lockstep workspace per (handle, lane count), reused by the
        // handle's later sets, which run after this one in its branch
        Ctx* found = nullptr;
        for (Ctx* lc : B.lane_ctx)
          if (lc->lane_of == &c && lc->lanes == K) found = lc;
        if (!found) {
          found = make_lane_ctx(c, K);
          found->lane_of = &c;
          B.lane_ctx.push_back(found);
        }
        run = found;
      }
      cudaGraphConditionalHandle* d_hif = nullptr;
      MHFP_CUDA(cudaMalloc(&d_hif, (size_t)c.opt.restart * sizeof(cudaGraphConditionalHandle)));
      B.d_hif.push_back(d_hif);
      cudaGraphNode_t dep = nullptr;
      size_t slot = tail.size();
      for (size_t t = 0; t < tail.size(); ++t)
        if (tail[t].first == &c) slot = t;
      if (slot < tail.size()) dep = tail[slot].second;
      std::vector<const double*> r;
      std::vector<double*> xs;
      std::vector<DevCtl*> hs;
      for (int e : set) {
        r.push_back(rhs[e]);
        xs.push_back(x[e]);
        hs.push_back(&B.host_ctl[e]);
        B.lanes[e] = K;
        B.lead[e] = i;
      }
      SolveCounts cnt;
      const cudaGraphNode_t last = add_solve(*run, B.graph, dep, false, d_hif, r.data(), xs.data(), tol, hs.data(),
                                             &cnt, K, K > 1 ? run->lane_bytes : 0);
      B.counts[i] = {cnt.start + 1, cnt.cycle, cnt.step};  // + the control-block reset
      if (slot < tail.size()) tail[slot].second = last;
      else tail.push_back({&c, last});
    }
    g_launches = l0;
    MHFP_CUDA(cudaGraphInstantiate(&B.exec, B.graph, 0));
  } catch (...) {
    g_launches = l0;
    throw;
  }
}

void run_batch_graph(BatchGraph& B, cudaStream_t stream) {
  MHFP_CUDA(cudaGraphLaunch(B.exec, stream));
  MHFP_CUDA(cudaStreamSynchronize(stream));
  for (size_t i = 0; i < B.counts.size(); ++i) {
    if ((int)i != B.lead[i]) continue;  // a set's launches are counted once, at its first entry
    const DevCtl& h = B.host_ctl[i];
    if (B.lanes[i] == 1)
      g_launches += B.counts[i][0] + (long long)(h.cycles + 1) * B.counts[i][1] + (long long)h.total * B.counts[i][2];
    else  // lane 0 counts the set's cycle starts and steps
      g_launches += B.counts[i][0] + (long long)h.decides * B.counts[i][1] + (long long)h.steps * B.counts[i][2];
  }
}

void destroy_batch_graph(BatchGraph& B) {
  if (B.exec) cudaGraphExecDestroy(B.exec);
  if (B.graph) cudaGraphDestroy(B.graph);
  for (auto* p : B.d_hif) cudaFree(p);
  if (B.host_ctl) cudaFreeHost(B.host_ctl);
  for (Ctx* lc : B.lane_ctx) destroy_lane_ctx(lc);
  B = BatchGraph{};
}

void invalidate_graphs(Ctx& c) {
  MHFP_CUDA(cudaStreamSynchronize(c.stream));
  ++c.graph_gen;
  for (int t = 0; t < 2; ++t) {
    for (auto& g : c.graphs[t]) {
      if (g.exec) cudaGraphExecDestroy(g.exec);
      for (auto& p : g.timed) {
        cudaEventDestroy(p.start);
        cudaEventDestroy(p.stop);
      }
    }
    c.graphs[t].clear();
    if (c.solve_exec[t]) cudaGraphExecDestroy(c.solve_exec[t]);
    c.solve_exec[t] = nullptr;
  }
}

void solve_device_graph_launch(Ctx& c, const double* b, double tol, bool transpose) {
  const int t = transpose ? 1 : 0;
  if (!c.solve_exec[t]) build_solve_graph(c, transpose);
  c.solve_t0 = std::chrono::steady_clock::now();
  MHFP_CUDA(cudaMemcpyAsync(c.bcur, b, c.n * sizeof(double), cudaMemcpyDeviceToDevice, c.stream));
  DevCtl h{};
  h.tol = tol;
  h.maxit = c.opt.maxit;
  h.m = c.opt.restart;
  *c.host_ctl = h;
  MHFP_CUDA(cudaMemcpyAsync(c.ctl, c.host_ctl, sizeof(DevCtl), cudaMemcpyHostToDevice, c.stream));
  MHFP_CUDA(cudaGraphLaunch(c.solve_exec[t], c.stream));
  c.solve_pending = t;
}

void solve_device_graph_finish(Ctx& c, double* x, mhfp_stats* st) {
  const int t = c.solve_pending;
  MHFP_CUDA(cudaMemcpyAsync(x, c.xcur, c.n * sizeof(double), cudaMemcpyDeviceToDevice, c.stream));
  MHFP_CUDA(cudaStreamSynchronize(c.stream));
  const DevCtl& h = *c.host_ctl;
  g_launches += c.solve_nkernels[t] + (long long)(h.cycles + 1) * c.solve_cycle_kernels[t] +
                (long long)h.total * c.solve_step_kernels[t];
  mhfp_stats s{};
  s.iterations = h.total;
  s.restarts = h.cycles;
  s.converged = h.converged;
  s.rel_residual = h.est;
  s.true_rel_residual = h.true_rel;
  s.solve_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - c.solve_t0).count();
  if (st) *st = s;
  if (h.status == (int)MHFP_ERR_NONFINITE) throw Error{MHFP_ERR_NONFINITE, "non-finite value in the solve"};
  if (!h.converged) throw Error{MHFP_ERR_NOT_CONVERGED, "FGMRES reached maxit before the tolerance"};
}

// The bulk-copy sweep records a wait that ran out of time in bit 8 of the
// handle's device flag instead of hanging; read it after a solve.
void check_wait_flag(Ctx& c) {
  if (c.hu.empty() || c.hu[0].tpp != 4 || c.opt.precision != 1) return;
  int h = 0;
  MHFP_CUDA(cudaMemcpyAsync(&h, c.d_flag, sizeof(int), cudaMemcpyDeviceToHost, c.stream));
  MHFP_CUDA(cudaStreamSynchronize(c.stream));
  if (h & 8) {
    MHFP_CUDA(cudaMemsetAsync(c.d_flag, 0, sizeof(int), c.stream));
    throw Error{MHFP_ERR_CUDA, "a bulk copy of the finest displacement sweep did not arrive in time"};
  }
}

// Set-up autotuner of the Chebyshev degree (cheb_degree = 0 in the
// options): solve the step's load right-hand side (previous state zero) to
// 1e-8 with degrees 1, 2 and 3, each after one warm-up solve, and keep the
// fastest.  The captured graphs hold the degree's sweeps, so they are
// dropped between candidates and after the choice.
void autotune_cheb_degree(Ctx& c) {
  double* b = dalloc_n<double>(c, c.n);
  double* x = dalloc_n<double>(c, c.n);
  build_rhs(c, nullptr, 1.0, b);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  MHFP_CUDA(cudaEventCreate(&e0));
  MHFP_CUDA(cudaEventCreate(&e1));
  int best = 2;
  float best_ms = 1e30f;
  try {
    for (int deg = 1; deg <= 3; ++deg) {
      c.opt.cheb_degree = deg;
      invalidate_graphs(c);
      mhfp_stats st{};
      float ms = 1e30f;
      bool ok = true;
      for (int rep = 0; rep < 2 && ok; ++rep) {
        MHFP_CUDA(cudaEventRecord(e0, c.stream));
        try {
          fgmres_solve(c, b, x, 1e-8, &st);
        } catch (const Error& e) {
          if (e.status != MHFP_ERR_NOT_CONVERGED) throw;
          ok = false;
        }
        MHFP_CUDA(cudaEventRecord(e1, c.stream));
        MHFP_CUDA(cudaEventSynchronize(e1));
        MHFP_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      }
      if (ok && ms < best_ms) {
        best_ms = ms;
        best = deg;
      }
    }
  } catch (...) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    throw;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  c.opt.cheb_degree = best;
  invalidate_graphs(c);
}

void fgmres_solve(Ctx& c, const double* b, double* x, double tol, mhfp_stats* st, bool transpose) {
  if (c.opt.graphs == 2 && !c.timing.enabled) {
    solve_device_graph_launch(c, b, tol, transpose);
    try {
      solve_device_graph_finish(c, x, st);
    } catch (...) {
      check_wait_flag(c);
      throw;
    }
    check_wait_flag(c);
    return;
  }
  FgState f;
  fgmres_begin(c, f, b, x, tol, transpose);
  try {
    while (f.phase != FgState::DONE) {
      MHFP_CUDA(cudaStreamSynchronize(c.stream));
      fgmres_advance(c, f);
    }
  } catch (const Error& e) {
    if (st) *st = f.stats;
    check_wait_flag(c);
    throw;
  }
  if (st) *st = f.stats;
  check_wait_flag(c);
}

}  // namespace mhfp
