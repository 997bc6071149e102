// The coarse-level sweeps and residuals of the library (sweep_spmv, sweep_cheb)
// under every launch schedule, against sums in FP64 on the host: lattices of
// one point, of sides with every remainder, and the largest that each of the
// row-major layouts takes; 1, 3 and 6 unknowns per point, one lane and three.
// Every result is compared with the rounding bound of its own sum.  Links
// against libmhfp.so; prints "ok" and returns 0, or the first mismatch and 1.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_2002_09603_gb300/csrc/lattice.cuh"

using namespace mhfp;

namespace {

unsigned long long state = 88172645463325252ull;
double rnd() {  // uniform in (-1, 1), exact in FP32
  state ^= state << 13;
  state ^= state >> 7;
  state ^= state << 17;
  return ((double)(state >> 41) - 4194304.0) / 4194304.0;
}

template <typename T>
struct Dev {
  T* p = nullptr;
  explicit Dev(const std::vector<T>& h) {
    if (cudaMalloc(&p, h.size() * sizeof(T)) != cudaSuccess) std::exit(2);
    cudaMemcpy(p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
  }
  ~Dev() { cudaFree(p); }
  std::vector<T> host(size_t n) const {
    std::vector<T> h(n);
    if (cudaMemcpy(h.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost) != cudaSuccess) std::exit(3);
    return h;
  }
};

template <typename T>
int check(int bs, int kind, int Lx, int Ly, int Lz, int lanes) {
  StructOp A;
  A.Lx = Lx;
  A.Ly = Ly;
  A.Lz = Lz;
  A.N = (long long)Lx * Ly * Lz;
  A.bs = bs;
  A.kind = kind;
  const int R = kind == ST_BOX1 ? 1 : 2, w = 2 * R + 1, no = w * w * w;
  const size_t N = (size_t)A.N, n = N * bs;
  const double u = sizeof(T) == 4 ? std::ldexp(1.0, -24) : std::ldexp(1.0, -53);  // unit roundoff
  auto neighbour = [&](long long p, int o, long long& q) {
    const int i = (int)(p % Lx) + o % w - R, j = (int)(p / Lx % Ly) + o / w % w - R, k = (int)(p / Lx / Ly) + o / (w * w) - R;
    q = i + (long long)Lx * (j + (long long)Ly * k);
    return i >= 0 && i < Lx && j >= 0 && j < Ly && k >= 0 && k < Lz;
  };
  std::vector<T> val((size_t)no * bs * bs * N), dinv((size_t)bs * bs * N);
  for (int o = 0; o < no; ++o)
    for (long long p = 0; p < A.N; ++p) {
      long long q;
      const bool in = neighbour(p, o, q);
      for (int e = 0; e < bs * bs; ++e) val[((size_t)o * bs * bs + e) * N + p] = in ? (T)rnd() : T(0);
    }
  for (T& v : dinv) v = (T)rnd();
  // lane l's vectors: x, b, d, out at the same offsets of its slice
  const size_t slice = (4 * n * sizeof(T) + 255) / 256 * 256 / sizeof(T);
  std::vector<T> vec(slice * lanes, T(0));
  for (int l = 0; l < lanes; ++l)
    for (size_t t = 0; t < 3 * n; ++t) vec[l * slice + t] = (T)rnd();
  const std::vector<T> cf = {T(0.375), T(0.8125)};
  const Dev<T> dval(val), ddinv(dinv), dcf(cf), drows(std::vector<T>(sweep_row_elems<T>(A, bs), T(7)));
  sweep_pack_rows<T>(nullptr, A, bs, dval.p, drows.p);
  // A x and sum |a| |x| per row
  std::vector<double> Ax(n * lanes, 0.0), mag(n * lanes, 0.0);
  for (int o = 0; o < no; ++o)
    for (long long p = 0; p < A.N; ++p) {
      long long q;
      if (!neighbour(p, o, q)) continue;
      for (int r = 0; r < bs; ++r)
        for (int s = 0; s < bs; ++s) {
          const double a = val[((size_t)o * bs * bs + r * bs + s) * N + p];
          for (int l = 0; l < lanes; ++l) {
            const double t = a * (double)vec[l * slice + bs * q + s];
            Ax[l * n + bs * p + r] += t;
            mag[l * n + bs * p + r] += std::fabs(t);
          }
        }
    }
  const double terms = no * bs + 2.0;
  auto bad = [&](const char* what, int sched, int l, size_t t, double got, double want, double tol) {
    if (std::fabs(got - want) <= tol) return false;
    std::printf("%s: bs %d kind %d lattice %d %d %d schedule %d lane %d entry %zu: %.17g, expected %.17g +- %.3g (FP%d)\n",
                what, bs, kind, Lx, Ly, Lz, sched, l, t, got, want, tol, (int)(8 * sizeof(T)));
    return true;
  };
  const LaneScope scope(lanes, (long long)(slice * sizeof(T)));
  for (int sched : {1, 4, 8, 16, 32, 64})
    for (int mode = 0; mode < 4; ++mode) {  // A x, b - A x, a first Chebyshev step, a later one
      const Dev<T> dv(vec);
      T *x = dv.p, *b = x + n, *d = b + n, *out = d + n;
      if (mode < 2) sweep_spmv<T>(nullptr, A, bs, dval.p, drows.p, x, mode ? b : nullptr, out, sched);
      else sweep_cheb<T>(nullptr, A, bs, dval.p, drows.p, ddinv.p, b, x, out, d, dcf.p, mode == 2, sched);
      const cudaError_t e = cudaDeviceSynchronize();
      if (e != cudaSuccess) {
        std::printf("schedule %d: %s\n", sched, cudaGetErrorString(e));
        return 1;
      }
      const std::vector<T> got = dv.host(vec.size());
      for (int l = 0; l < lanes; ++l) {
        const T* v = vec.data() + l * slice;
        const T* g = got.data() + l * slice;
        for (size_t p = 0; p < N; ++p)
          for (int r = 0; r < bs; ++r) {
            const size_t t = bs * p + r;
            if (mode < 2) {
              const double bt = mode ? (double)v[n + t] : 0.0, want = mode ? bt - Ax[l * n + t] : Ax[l * n + t];
              if (bad("residual", sched, l, t, g[3 * n + t], want, terms * u * (std::fabs(bt) + mag[l * n + t]))) return 1;
              continue;
            }
            // z = D^-1 (b - A x): the residual's bound through |D^-1|, and its own sum's
            double z = 0.0, ez = 0.0;
            for (int s = 0; s < bs; ++s) {
              const double di = dinv[((size_t)r * bs + s) * N + p], bt = v[n + bs * p + s];
              const double m = std::fabs(bt) + mag[l * n + bs * p + s];
              z += di * (bt - Ax[l * n + bs * p + s]);
              ez += std::fabs(di) * (terms + bs + 2.0) * u * m;
            }
            const double cd = mode == 2 ? 0.0 : (double)cf[0], cr = cf[1], dt = v[2 * n + t], xt = v[t];
            const double dn = cd * dt + cr * z, ed = cr * ez + 4.0 * u * (std::fabs(cd * dt) + std::fabs(cr * z));
            if (bad("d", sched, l, t, g[2 * n + t], dn, ed)) return 1;
            if (bad("x", sched, l, t, g[3 * n + t], xt + dn, ed + 2.0 * u * (std::fabs(xt) + std::fabs(dn)))) return 1;
          }
      }
    }
  return 0;
}

template <typename T>
int all() {
  const int small[][3] = {{1, 1, 1}, {2, 1, 1}, {1, 3, 2}, {5, 4, 3}, {7, 2, 9}, {33, 1, 4}, {13, 11, 15}};
  for (const auto& s : small)
    for (int bs : {1, 3, 6})
      if (check<T>(bs, bs == 1 ? ST_BOX2 : ST_BOX1, s[0], s[1], s[2], 1)) return 1;
  for (int bs : {1, 3, 6})
    if (check<T>(bs, bs == 1 ? ST_BOX2 : ST_BOX1, 7, 5, 6, 3)) return 1;
  return check<T>(1, ST_BOX2, 32, 32, 32, 1) || check<T>(3, ST_BOX1, 16, 16, 16, 1) || check<T>(6, ST_BOX1, 32, 32, 16, 1);
}

}  // namespace

int main() {
  if (all<float>() || all<double>()) return 1;
  std::printf("ok\n");
  return 0;
}
