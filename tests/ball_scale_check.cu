// The flushing reciprocal square root of the ball projections against rsqrtf,
// over every non-negative float (NaN included): prints the number of inputs on
// which ball_scale (pd_math.cuh), and tgv_ball (pd_tgv_math.cuh) at the
// smallest radius its flushing form is used with and at two ordinary ones,
// give other bits than rsqrtf's form.
#include <cstdio>

#include "pd_math.cuh"
#include "pd_tgv_math.cuh"

__global__ void check(unsigned long long* bad) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long n = 0, m = 0;
  for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 31); i += step) {
    const float x = __uint_as_float((unsigned)i);
    const float a = fs::ball_scale(x), b = fminf(1.f, rsqrtf(x));
    if (__float_as_uint(a) != __float_as_uint(b)) ++n;
    for (float r : {1e-18f, 1.2f, 17.f}) {
      const float c = fs::tgv_ball<true>(x, r), d = fs::tgv_ball<false>(x, r);
      if (__float_as_uint(c) != __float_as_uint(d)) ++m;
    }
  }
  if (n) atomicAdd(bad, n);
  if (m) atomicAdd(bad + 1, m);
}

int main() {
  unsigned long long* d = nullptr;
  unsigned long long h[2] = {1, 1};
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 1;
  check<<<152 * 8, 256>>>(d);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  std::printf("%llu %llu\n", h[0], h[1]);
  cudaFree(d);
  return 0;
}
