// Rounding errors, in ulps, of the short FP64 reciprocal, reciprocal root and
// root (qrcp_, qrsqrt_, qroot_) and of the plain ones (rcp_, rrsqrt_, rsqrt_)
// on the same inputs: prints one JSON object; tests/test_gpu_rounding.py
// builds and runs it.  The errors come from exact residuals: 1 - x q (one
// fma), 1 - x q^2 with q^2 as a sum of two doubles, x - q^2 (one fma).
// Inputs: random mantissas (whose mean error is reported), mantissas close to
// 1 and to 2, where a step from the seed leaves its binade, and all 2^20
// mantissas that the hardware's seed distinguishes, at either end of the
// inputs that share it, for even and odd exponents.
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>

#include "physics.cuh"

using namespace mhd;

__device__ unsigned long long mix64(unsigned long long z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__device__ double from_bits(unsigned long long e, unsigned long long m) {
  return __longlong_as_double((long long)((e << 52) | (m & 0xfffffffffffffull)));
}

__device__ double ulps(int f, double x, double q) {
  double off;   // true value minus q, to 1e-10 of itself
  if (f == 0) {
    off = fma(-x, q, 1.0) * q;
  } else if (f == 1) {
    const double s = q * q, low = fma(q, q, -s);
    off = 0.5 * (fma(-x, s, 1.0) - x * low) * q;
  } else {
    off = fma(-q, q, x) / (2.0 * q);
  }
  const double ulp = from_bits((__double_as_longlong(q) >> 52 & 0x7ff), 0) * 2.220446049250313e-16;
  const double r = fabs(off) / ulp;
  return r == r ? r : 1e30;
}
__device__ double value(int f, bool plain, double x) {
  if (f == 0) return plain ? rcp_(x) : qrcp_(x);
  if (f == 1) return plain ? rrsqrt_(x) : qrsqrt_(x);
  return plain ? rsqrt_(x) : qroot_(x);
}

// kinds: 0 random mantissas, 1 mantissas near 1 and 2, 2 every seed
__global__ void check(int f, bool plain, int kind, unsigned long long n, double* out) {
  double most = 0.0, sum = 0.0;
  for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < n;
       t += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long z = mix64(t), w = mix64(z);
    double x;
    if (kind == 0) {
      x = from_bits(723 + (z >> 52) % 601, w);
    } else if (kind == 1) {
      const unsigned long long off = w >> (12 + 19 + z % 33);   // 2^-19 down to one ulp
      x = from_bits(1013 + (z >> 52) % 20, z & 1024 ? off : 0xfffffffffffffull - off);
    } else {
      const unsigned long long low = t & 2 ? (w & 0xffffffffull) : t & 1 ? 0xffffffffull : 0ull;
      x = from_bits(1023 + (t >> 2 & 1), (t >> 3 & 0xfffffull) << 32 | low);
    }
    const double r = ulps(f, x, value(f, plain, x));
    most = fmax(most, r);
    sum += r;
  }
  atomicMax((unsigned long long*)out, (unsigned long long)__double_as_longlong(most));
  atomicAdd(out + 1, sum);
}

int main() {
  double* d;
  if (cudaMalloc(&d, 2 * sizeof(double)) != cudaSuccess) return 1;
  const char* names[3] = {"rcp", "rsqrt", "root"};
  printf("{");
  for (int f = 0; f < 3; ++f)
    for (int plain = 0; plain < 2; ++plain) {
      double most = 0.0, mean = 0.0;
      for (int kind = 0; kind < 3; ++kind) {
        const unsigned long long n = kind == 2 ? 1ull << 23 : 1ull << 26;
        double h[2];
        if (cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
        check<<<152 * 8, 256>>>(f, plain, kind, n, d);
        if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
        most = h[0] > most ? h[0] : most;
        if (kind == 0) mean = h[1] / (double)n;
      }
      printf("%s\"%s%s\": [%.6f, %.6f]", f + plain ? ", " : "", plain ? "plain_" : "", names[f], most, mean);
    }
  printf("}\n");
  return 0;
}
