// Test program: the roots and seeds of p3t_internal.cuh and cutoff_math.cuh.
//   roots_check rsqrtf              -> mismatches with rsqrtf over every normal float
//   roots_check seed                -> largest |1 - x y^2| over every leading mantissa
//   roots_check eval <in> <out>     -> in: doubles x; out, for each x: the seed's y
//     and e, y (1 + e/2 + 3/8 e^2), y^3 (1 + 3/2 e + 15/8 e^2), inv_sqrt, inv_root4,
//     cbrt_pos, and CUDA's rsqrt(x), rsqrt(sqrt(x)), cbrt(x)
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../paper_2007_15432_gb300/csrc/cutoff_math.cuh"

__global__ void k_rsqrtf(unsigned long long *bad) {
  for (uint32_t b = 0x00800000u + blockIdx.x * blockDim.x + threadIdx.x; b < 0x7f800000u;
       b += gridDim.x * blockDim.x) {
    const float x = __uint_as_float(b);
    if (__float_as_uint(rsqrt_normal(x)) != __float_as_uint(rsqrtf(x))) atomicAdd(bad, 1ull);
  }
}

// every leading 20-bit mantissa, the rest zeros, ones or 0x5a5a5a5a, at even and odd
// exponents over the seed's range
__global__ void k_seed(unsigned long long *worst) {
  const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;  // < 2^20
  const uint32_t low[3] = {0u, 0xffffffffu, 0x5a5a5a5au};
  const uint32_t ex[8] = {512u, 513u, 800u, 1023u, 1024u, 1301u, 1534u, 1535u};
  double w = 0.0;
  for (int i = 0; i < 8; ++i)
    for (int j = 0; j < 3; ++j) {
      const double x = __hiloint2double((int)(ex[i] << 20 | m), (int)low[j]);
      w = fmax(w, fabs(rsqrt_seed(x).e));
    }
  atomicMax(worst, (unsigned long long)__double_as_longlong(w));
}

__global__ void k_eval(int n, const double *x, double *o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const RsqrtSeed s = rsqrt_seed(x[i]);
  const double y3 = s.y2 * s.y;
  double *r = o + 10 * (int64_t)i;
  r[0] = s.y;
  r[1] = s.e;
  r[2] = __fma_rn(s.y * s.e, __fma_rn(0.375, s.e, 0.5), s.y);
  r[3] = __fma_rn(y3 * s.e, __fma_rn(1.875, s.e, 1.5), y3);
  r[4] = inv_sqrt(x[i]);
  r[5] = inv_root4(x[i]);
  r[6] = cbrt_pos(x[i]);
  r[7] = rsqrt(x[i]);
  r[8] = rsqrt(sqrt(x[i]));
  r[9] = cbrt(x[i]);
}

int main(int argc, char **argv) {
  unsigned long long *d, h = 0;
  if (argc == 2) {
    if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 2;
    if (!strcmp(argv[1], "rsqrtf")) k_rsqrtf<<<1216, 256>>>(d);
    else k_seed<<<4096, 256>>>(d);
    if (cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    double w;
    memcpy(&w, &h, 8);
    if (!strcmp(argv[1], "rsqrtf")) printf("%llu\n", h);
    else printf("%.17g\n", w);
    return 0;
  }
  if (argc != 4) return 1;
  std::vector<double> x;
  FILE *f = fopen(argv[2], "rb");
  if (!f) return 1;
  double v;
  while (fread(&v, 8, 1, f) == 1) x.push_back(v);
  fclose(f);
  const int n = (int)x.size();
  std::vector<double> o(10 * (size_t)n);
  double *dx, *dout;
  if (cudaMalloc(&dx, 8 * (size_t)n) != cudaSuccess ||
      cudaMalloc(&dout, 80 * (size_t)n) != cudaSuccess)
    return 2;
  if (cudaMemcpy(dx, x.data(), 8 * (size_t)n, cudaMemcpyHostToDevice) != cudaSuccess) return 2;
  k_eval<<<(n + 127) / 128, 128>>>(n, dx, dout);
  if (cudaMemcpy(o.data(), dout, 80 * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  f = fopen(argv[3], "wb");
  if (!f || fwrite(o.data(), 80, n, f) != (size_t)n) return 1;
  fclose(f);
  return 0;
}
