// Structured-lattice helpers shared by the multigrid translation units:
// stencil offset tables, lattice index views (64-bit and 32-bit with
// invariant-divisor decoding) and the compile-time dispatch of block sizes,
// stencil kinds and launch schedules.
#pragma once
#include "common.cuh"

#include <type_traits>

namespace mhfp {
namespace {

static __constant__ signed char c_dia[25][3] = {
    {0, 0, -2}, {0, -1, -1}, {-1, 0, -1}, {0, 0, -1}, {1, 0, -1}, {0, 1, -1}, {0, -2, 0}, {-1, -1, 0}, {0, -1, 0},
    {1, -1, 0}, {-2, 0, 0},  {-1, 0, 0},  {0, 0, 0},  {1, 0, 0},  {2, 0, 0},  {-1, 1, 0}, {0, 1, 0},  {1, 1, 0},
    {0, 2, 0},  {0, -1, 1},  {-1, 0, 1},  {0, 0, 1},  {1, 0, 1},  {0, 1, 1},  {0, 0, 2}};
static __constant__ signed char c_dia_idx[125] = {
    -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 0,  -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1,
    -1, -1, -1, -1, -1, -1, -1, 1,  -1, -1, -1, 2,  3,  4,  -1, -1, -1, 5,  -1, -1, -1, -1, -1, -1, -1,
    -1, -1, 6,  -1, -1, -1, 7,  8,  9,  -1, 10, 11, 12, 13, 14, -1, 15, 16, 17, -1, -1, -1, 18, -1, -1,
    -1, -1, -1, -1, -1, -1, -1, 19, -1, -1, -1, 20, 21, 22, -1, -1, -1, 23, -1, -1, -1, -1, -1, -1, -1,
    -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 24, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1};

template <int KIND>
struct St;
template <>
struct St<ST_BOX1> {
  static constexpr int N = 27, R = 1, C = 13;
  __device__ static void off(int o, int& x, int& y, int& z) { x = o % 3 - 1; y = (o / 3) % 3 - 1; z = o / 9 - 1; }
  __device__ static int idx(int x, int y, int z) {
    if (x < -1 || x > 1 || y < -1 || y > 1 || z < -1 || z > 1) return -1;
    return (x + 1) + 3 * ((y + 1) + 3 * (z + 1));
  }
};
template <>
struct St<ST_DIAMOND2> {
  static constexpr int N = 25, R = 2, C = 12;
  __device__ static void off(int o, int& x, int& y, int& z) { x = c_dia[o][0]; y = c_dia[o][1]; z = c_dia[o][2]; }
  __device__ static int idx(int x, int y, int z) {
    if (x < -2 || x > 2 || y < -2 || y > 2 || z < -2 || z > 2) return -1;
    return c_dia_idx[(x + 2) + 5 * ((y + 2) + 5 * (z + 2))];
  }
};
template <>
struct St<ST_BOX2> {
  static constexpr int N = 125, R = 2, C = 62;
  __device__ static void off(int o, int& x, int& y, int& z) { x = o % 5 - 2; y = (o / 5) % 5 - 2; z = o / 25 - 2; }
  __device__ static int idx(int x, int y, int z) {
    if (x < -2 || x > 2 || y < -2 || y > 2 || z < -2 || z > 2) return -1;
    return (x + 2) + 5 * ((y + 2) + 5 * (z + 2));
  }
};

struct Lat {
  int Lx, Ly, Lz;
  long long N;
  __device__ void ijk(long long p, int& i, int& j, int& k) const {
    i = (int)(p % Lx);
    const long long r = p / Lx;
    j = (int)(r % Ly);
    k = (int)(r / Ly);
  }
  __device__ bool in(int i, int j, int k) const { return i >= 0 && i < Lx && j >= 0 && j < Ly && k >= 0 && k < Lz; }
  __device__ long long id(int i, int j, int k) const { return i + (long long)Lx * (j + (long long)Ly * k); }
};

Lat lat_of(const StructOp& A) { return Lat{A.Lx, A.Ly, A.Lz, A.N}; }

// ------------------------------------------------------- lattice helpers
// 32-bit lattice indexing for the coarse levels (see the coarse-level sweeps
// below).
struct Lat32 {
  int Lx, Ly, Lz, N, LxLy;
  Div32 dx, dy;
  __device__ __forceinline__ void ijk(unsigned p, int& i, int& j, int& k) const {
    const unsigned r = dx.div(p);
    i = (int)(p - r * (unsigned)Lx);
    k = (int)dy.div(r);
    j = (int)(r - (unsigned)k * (unsigned)Ly);
  }
};

// box index (x+2) + 5 (y+2) + 25 (z+2) of the o-th offset with |d|_1 <= 2,
// in box order (the order of stencil_offset for ST_DIAMOND2)
__host__ __device__ constexpr int dia_box(int o) { return o == 0 ? 12 : o == 1 ? 32 : o == 2 ? 36 : o == 3 ? 37 : o == 4 ? 38 : o == 5 ? 42 : o == 6 ? 52 : o == 7 ? 56 : o == 8 ? 57 : o == 9 ? 58 : o == 10 ? 60 : o == 11 ? 61 : o == 12 ? 62 : o == 13 ? 63 : o == 14 ? 64 : o == 15 ? 66 : o == 16 ? 67 : o == 17 ? 68 : o == 18 ? 72 : o == 19 ? 82 : o == 20 ? 86 : o == 21 ? 87 : o == 22 ? 88 : o == 23 ? 92 : 112; }
constexpr bool dia_table_matches_box_order() {
  int n = 0;
  for (int b = 0; b < 125; ++b) {
    const int x = b % 5 - 2, y = (b / 5) % 5 - 2, z = b / 25 - 2;
    if ((x < 0 ? -x : x) + (y < 0 ? -y : y) + (z < 0 ? -z : z) > 2) continue;
    if (dia_box(n++) != b) return false;
  }
  return n == 25;
}
static_assert(dia_table_matches_box_order(), "diamond offset table out of box order");

// compile-time offsets of each stencil kind
template <int KIND>
struct Sf;
template <>
struct Sf<ST_BOX1> {
  static constexpr int N = 27, R = 1;
  __device__ static constexpr int x(int o) { return o % 3 - 1; }
  __device__ static constexpr int y(int o) { return (o / 3) % 3 - 1; }
  __device__ static constexpr int z(int o) { return o / 9 - 1; }
};
template <>
struct Sf<ST_BOX2> {
  static constexpr int N = 125, R = 2;
  __device__ static constexpr int x(int o) { return o % 5 - 2; }
  __device__ static constexpr int y(int o) { return (o / 5) % 5 - 2; }
  __device__ static constexpr int z(int o) { return o / 25 - 2; }
};
template <>
struct Sf<ST_DIAMOND2> {
  static constexpr int N = 25, R = 2;
  __device__ static constexpr int x(int o) { return dia_box(o) % 5 - 2; }
  __device__ static constexpr int y(int o) { return (dia_box(o) / 5) % 5 - 2; }
  __device__ static constexpr int z(int o) { return dia_box(o) / 25 - 2; }
};

// block sizes of lattice levels: 1 (interface pressure), 3 (displacement),
// 6 (coarse displacement levels with the rigid-body modes; 27-point only)
template <class F>
void dispatch_bs(int bs, F&& f) {
  if (bs == 3) f(std::integral_constant<int, 3>{});
  else if (bs == 6) f(std::integral_constant<int, 6>{});
  else f(std::integral_constant<int, 1>{});
}

// the block sizes of M_II^(h)'s smoothed aggregation (coarsen)
template <class F>
void dispatch_bs13(int bs, F&& f) {
  if (bs == 3) f(std::integral_constant<int, 3>{});
  else f(std::integral_constant<int, 1>{});
}

// stencil kinds a block size occurs with: the displacement levels (3 or 6
// dofs per point) are 27-point lattices, the scalar interface-pressure levels
// 25-point (cells) or 125-point (coarser); other pairs are not instantiated
template <int BS, class F>
void dispatch_kind_bs(int kind, F&& f) {
  if constexpr (BS != 1) {
    if (kind != ST_BOX1) throw Error{MHFP_ERR_ARG, "vector lattice levels are 27-point only"};
    f(std::integral_constant<int, ST_BOX1>{});
  } else {
    if (kind == ST_DIAMOND2) f(std::integral_constant<int, ST_DIAMOND2>{});
    else if (kind == ST_BOX2) f(std::integral_constant<int, ST_BOX2>{});
    else throw Error{MHFP_ERR_ARG, "scalar lattice levels are 25- or 125-point"};
  }
}

// (fine, coarse) block pairs of the transfers
template <class F>
void dispatch_pair(int bf, int bc, F&& f) {
  if (bf == 3 && bc == 3) f(std::integral_constant<int, 3>{}, std::integral_constant<int, 3>{});
  else if (bf == 3 && bc == 6) f(std::integral_constant<int, 3>{}, std::integral_constant<int, 6>{});
  else if (bf == 6 && bc == 6) f(std::integral_constant<int, 6>{}, std::integral_constant<int, 6>{});
  else f(std::integral_constant<int, 1>{}, std::integral_constant<int, 1>{});
}

// 32-bit lattice view for the coarse-level kernels (their indices e N + p
// and bs q + s stay below 2^31)
inline Lat32 lat32_of(const StructOp& A) {
  if ((long long)A.bs * A.bs * A.N >= (1LL << 31))
    throw Error{MHFP_ERR_ARG, "lattice level too large for 32-bit indexing"};
  Lat32 L;
  L.Lx = A.Lx;
  L.Ly = A.Ly;
  L.Lz = A.Lz;
  L.N = (int)A.N;
  L.LxLy = A.Lx * A.Ly;
  L.dx = Div32::make((unsigned)A.Lx);
  L.dy = Div32::make((unsigned)A.Ly);
  return L;
}

// Launch schedule of a level's sweeps and residuals: 1 = one point per
// thread, W = 4, 8, 16 = warp-split offsets over W warps, 32 and 64 = a warp,
// or eight lanes, per point on row-major values, which box levels have up to
// the size where a split schedule is as fast (row_level).  The set-up
// autotuner times all that apply.  Without it: row-major levels take a warp
// per point up to 2,048 points, and in FP32 with 3 or 6 unknowns per point at
// any size; above, scalar and 6 x 6 levels take eight lanes and 3 x 3 levels
// eight warps; other scalar levels of 64K points and up one point per thread
// and the rest eight warps.  Microseconds of a Chebyshev step, eight warps / best
// split / warp per point / eight lanes:
//   125-point FP32:  1,000 5.4 / 5.0 / 1.9 / 2.4;    10,648 5.9 / 5.8 / 4.5 / 3.5;    32,768 10.9 / 6.3 / 10.6 / 7.0
//   125-point FP64:  1,000 11.6 / 11.6 / 2.7 / 3.7;  10,648 21.0 / 15.4 / 10.8 / 5.9; 32,768 46.9 / 19.0 / 29.2 / 13.2
//   3 x 3 FP32:      1,000 3.6 / 3.1 / 2.0 / 3.6;    2,744 3.7 / 3.2 / 2.6 / 3.8;     4,096 3.8 / 3.2 / 3.0 / 3.9
//   3 x 3 FP64:      1,000 6.0 / 6.0 / 4.1 / 5.4;    2,744 6.3 / 6.3 / 7.5 / 6.4;     4,096 6.4 / 6.4 / 10.1 / 6.6
//   6 x 6 FP32:      2,744 8.7 / 8.2 / 3.8 / 8.3;    8,000 10.1 / 9.3 / 6.8 / 9.0;    16,384 17.6 / 15.6 / 12.5 / 13.2
//   6 x 6 FP64:      1,728 15.4 / 15.4 / 10.1 / 10.3; 4,096 15.9 / 15.9 / 21.7 / 13.5; 16,384 89 / 62 / 79 / 48
inline bool row_level(const StructOp& A) {
  if (A.kind == ST_DIAMOND2) return false;
  return A.N <= (A.bs == 1 ? 32768 : (A.bs == 3 ? 4096 : 16384));
}
inline int row_lanes(int sched) { return sched == 32 ? 32 : (sched == 64 ? 8 : 0); }
inline int default_schedule(const StructOp& A, bool rows, bool fp32) {
  if (rows) return A.N <= 2048 || (fp32 && A.bs > 1) ? 32 : (A.bs == 3 ? 8 : 64);
  return (A.bs == 1 && A.N >= 65536) ? 1 : 8;
}

template <class F>
void dispatch_sched(int sched, F&& f) {
  if (sched == 1) f(std::integral_constant<int, 1>{});
  else if (sched == 4) f(std::integral_constant<int, 4>{});
  else if (sched == 16) f(std::integral_constant<int, 16>{});
  else f(std::integral_constant<int, 8>{});
}

}  // namespace

// Coarse-level sweeps and residuals (sweep.cu, one object per value type):
// y = b - A x (y = A x when b is null) on a lattice level with launch
// schedule sched; one Chebyshev step from xin (see the kernels); the first
// Chebyshev step from x = 0 (no stencil work).  They queue one kernel on
// `stream` and do not check or count it: the caller does.
template <typename T>
void sweep_spmv(cudaStream_t stream, const StructOp& A, int bs, const T* val, const T* rows, const T* x, const T* b,
                T* y, int sched);
template <typename T>
void sweep_cheb(cudaStream_t stream, const StructOp& A, int bs, const T* val, const T* rows, const T* dinv, const T* b,
                const T* xin, T* out, T* d, const T* cf, bool first, int sched);
// row-major copy of a level's values (schedules 32 and 64; null: none)
template <typename T>
size_t sweep_row_elems(const StructOp& A, int bs);
template <typename T>
void sweep_pack_rows(cudaStream_t stream, const StructOp& A, int bs, const T* val, T* rows);
template <typename T>
void sweep_cheb_zero(cudaStream_t stream, long long npts, int bs, const T* dinv, const T* b, T* out, T* d, const T* cf);

}  // namespace mhfp
