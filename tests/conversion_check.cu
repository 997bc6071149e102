// The integer-pipe conversions between FP32 and FP64 (widen, narrow) against the
// device's own, bit for bit (NaN: NaN): widen over all 2^32 FP32 values; narrow
// over all 2^32 upper words of an FP64 value - every sign, exponent and 20 bits
// of the significand, so zeros, subnormals of either type, values past FP32's
// range, infinities and NaN - with lower words that complete the FP32
// significand in each of its 8 ways and leave a tail of nothing, one unit, just
// under, exactly and just over half, and all ones.  Prints "ok" and returns 0,
// or the first mismatch of each and returns 1.
#include <cstdio>

#include "../paper_2002_09603_gb300/csrc/common.cuh"

using mhfp::narrow;
using mhfp::widen;

namespace {

struct Report {
  unsigned long long bad, arg, got, want;
};

__device__ void note(Report* r, unsigned long long arg, unsigned long long got, unsigned long long want) {
  if (atomicAdd(&r->bad, 1ull) == 0) {
    r->arg = arg;
    r->got = got;
    r->want = want;
  }
}

__global__ void check_widen(Report* r) {
  const unsigned step = gridDim.x * blockDim.x;  // divides 2^32
  unsigned b = blockIdx.x * blockDim.x + threadIdx.x;
  for (unsigned k = 0; k < 0xffffffffu / step + 1u; ++k, b += step) {
    const float f = __uint_as_float(b);
    const double got = widen(f), want = (double)f;
    if (isnan(want) ? !isnan(got) : __double_as_longlong(got) != __double_as_longlong(want))
      note(r, b, __double_as_longlong(got), __double_as_longlong(want));
  }
}

__global__ void check_narrow(Report* r, unsigned lo) {
  const unsigned step = gridDim.x * blockDim.x;
  unsigned hi = blockIdx.x * blockDim.x + threadIdx.x;
  for (unsigned k = 0; k < 0xffffffffu / step + 1u; ++k, hi += step) {
    const double d = __hiloint2double((int)hi, (int)lo);
    const float got = narrow(d), want = __double2float_rn(d);
    if (isnan(want) ? !isnan(got) : __float_as_uint(got) != __float_as_uint(want))
      note(r, ((unsigned long long)hi << 32) | lo, __float_as_uint(got), __float_as_uint(want));
  }
}

}  // namespace

int main() {
  Report* d = nullptr;
  Report h[2];
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 2;
  check_widen<<<4096, 256>>>(d);
  for (unsigned top = 0; top < 8; ++top)
    for (unsigned tail : {0u, 1u, 0x0fffffffu, 0x10000000u, 0x10000001u, 0x1fffffffu})
      check_narrow<<<4096, 256>>>(d + 1, (top << 29) | tail);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) {
    std::printf("%s\n", cudaGetErrorString(cudaGetLastError()));
    return 2;
  }
  cudaFree(d);
  for (int i = 0; i < 2; ++i)
    if (h[i].bad)
      std::printf("%s: %llu mismatches, the first at %llx: %llx, expected %llx\n", i ? "narrow" : "widen", h[i].bad,
                  h[i].arg, h[i].got, h[i].want);
  if (h[0].bad || h[1].bad) return 1;
  std::printf("ok\n");
  return 0;
}
