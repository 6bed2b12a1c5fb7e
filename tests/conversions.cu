// f2d_int and d2f_int (csrc/ds_arith.cuh) against the conversion instructions,
// bit for bit: every float, and around every float x the doubles at x, just
// below, at and just above the tie to the next one, and below that next one
// (subnormals, the overflow edge, infinities and NaNs among them).  Built and run
// by tests/test_gpu_conversions.py.
#include <cstdio>

#include "ds_arith.cuh"

__global__ void check(unsigned long long* bad) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long v = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; v < (1ull << 32); v += step) {
    const float x = __uint_as_float((unsigned)v);
    const long long d = __double_as_longlong((double)x);
    if (__double_as_longlong(grom::f2d_int(x)) != d) atomicAdd(bad, 1ull);
    const long long add[5] = {0, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff};
    for (int q = 0; q < 5; ++q) {
      const double y = __longlong_as_double(d + add[q]);
      if (__float_as_uint(grom::d2f_int(y)) != __float_as_uint(__double2float_rn(y))) atomicAdd(bad + 1, 1ull);
    }
  }
}

int main() {
  unsigned long long *d, h[2] = {1, 1};
  cudaMalloc(&d, sizeof(h));
  cudaMemset(d, 0, sizeof(h));
  check<<<152 * 8, 256>>>(d);
  const cudaError_t e = cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost);
  std::printf("%s: %llu and %llu differ\n", cudaGetErrorString(e), h[0], h[1]);
  cudaFree(d);
  return e != cudaSuccess || h[0] || h[1];
}
