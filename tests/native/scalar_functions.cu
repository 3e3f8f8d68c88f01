// Device run of the float64 reciprocal, reciprocal root and float32 rounding of rve_kern.cuh.  Reads float64
// numbers from argv[1]; writes per number recip_nr, rsqrt_nr (0 where it declines), round_to<float>
// as float64, and whether rsqrt_nr took it, to argv[2].
#include <stdio.h>
#include <stdlib.h>

#include "rve_kern.cuh"

__global__ void k_scalar(const double *x, long long n, double *out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  bool ok;
  out[4 * i] = recip_nr(x[i]);
  out[4 * i + 1] = rsqrt_nr(x[i], ok);
  out[4 * i + 2] = (double)round_to<float>(x[i]);
  out[4 * i + 3] = ok ? 1.0 : 0.0;
}

int main(int argc, char **argv) {
  if (argc != 3) return 2;
  FILE *f = fopen(argv[1], "rb");
  if (!f) return 2;
  fseek(f, 0, SEEK_END);
  const long long n = ftell(f) / 8;
  rewind(f);
  double *h = (double *)malloc(n * 40), *d = nullptr;
  if (!h || fread(h, 8, n, f) != (size_t)n) return 2;
  fclose(f);
  if (cudaMalloc(&d, n * 40) != cudaSuccess) return 3;
  if (cudaMemcpy(d, h, n * 8, cudaMemcpyHostToDevice) != cudaSuccess) return 3;
  k_scalar<<<(unsigned)((n + 255) / 256), 256>>>(d, n, d + n);
  if (cudaGetLastError() != cudaSuccess) return 3;
  if (cudaMemcpy(h, d + n, n * 32, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  f = fopen(argv[2], "wb");
  if (!f || fwrite(h, 8, 4 * n, f) != (size_t)(4 * n)) return 2;
  return fclose(f) ? 2 : 0;
}
