// The solvers of the FP64 kernels (hlld_flux_lean, hll_flux_lean) against the plain ones on random faces of every region, on the host
// (argument "host") or the device: prints one JSON object with the largest
// difference over its bound; tests/test_lean_flux.py builds and runs it.
// The bound of a face is 64 eps kappa in units of the flux scale, kappa = 1 +
// the larger of max(|rho (S-u)(S-S_M)|, bn^2) / |den| of its two sides: the
// star states divide by den, whose own rounding error that ratio amplifies;
// both solvers take tens of roundings.  A side that both solvers count as
// degenerate (|den| well inside the threshold) divides by nothing.  Also the
// reciprocals and roots those solvers use, against IEEE: within 2^-50 (a few
// roundings) over exponents 2^-300..2^300, and the IEEE value of zeros,
// subnormals, infinities, NaN and (roots) negative numbers; and the FP64
// characteristic half slope against the plain one, within 256 eps of the
// differences it limits, where the plain one does not cancel.
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>

#include "physics.cuh"

using namespace mhd;

__host__ __device__ inline unsigned long long mix64(unsigned long long z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
struct Rng {
  unsigned long long s;
  __host__ __device__ double u(double a, double b) {
    s = mix64(s);
    return a + (b - a) * (double)(s >> 11) * (1.0 / 9007199254740992.0);
  }
};

// kinds: 0 large jumps, 1 small jumps, 2 supersonic either way, 3 equal
// states, no normal or no transverse field, 4 at rest along a strong field
// with sheared tangential velocity (degenerate star states)
__host__ __device__ double face_excess(int kind, unsigned long long q, bool hll) {
  Rng g{mix64(q * 8 + kind)};
  const double jump = kind == 1 ? 1e-3 : kind == 2 ? 3.0 : 1.0;
  double base[7];
  for (int i = 0; i < 7; ++i) base[i] = i == 0 ? exp(g.u(-2, 2)) : i == 4 ? exp(g.u(-3, 2)) : g.u(-1, 1);
  double w[2][7], bn = g.u(-2, 2);
  for (int s = 0; s < 2; ++s)
    for (int i = 0; i < 7; ++i)
      w[s][i] = (i == 0 || i == 4 ? base[i] * exp(0.5 * jump * g.u(-1, 1)) : base[i] + jump * g.u(-1, 1));
  if (kind == 2) for (int s = 0; s < 2; ++s) w[s][1] += (q & 1 ? 4.0 : -4.0);
  if (kind == 3) {
    if (q % 3 == 0) bn = 0;
    if (q % 3 == 1) for (int s = 0; s < 2; ++s) w[s][5] = w[s][6] = 0;
    if (q % 5 == 0) for (int i = 0; i < 7; ++i) w[1][i] = w[0][i];
    if (q % 7 == 0) w[0][1] = w[1][1] = 0;
  }
  if (kind == 4)
    for (int s = 0; s < 2; ++s) {
      w[s][0] = 1;
      w[s][4] = 0.1;
      w[s][1] = w[s][5] = w[s][6] = 0;
      bn = (q & 1 ? 1.0 : -1.5);
    }
  double f[7], h[7], c1, c2;
  const double gam = (5.0 / 3.0), ig = 1.0 / (gam - 1.0);
  if (hll) {
    hll_flux_g<double>(w[0], w[1], bn, gam, ig, f, &c1);
    hll_flux_lean(w[0], w[1], bn, gam, ig, h, &c2);
  } else {
    hlld_flux_g<double>(w[0], w[1], bn, gam, ig, f, &c1);
    hlld_flux_lean(w[0], w[1], bn, gam, ig, h, &c2);
  }
  // conditioning of the star states, in FP64
  double kappa = 1.0;
  const double b2 = (double)bn * bn, cm = c1;
  if (!hll) {
    const double sl = fmin((double)w[0][1], (double)w[1][1]) - cm, sr = fmax((double)w[0][1], (double)w[1][1]) + cm;
    const double ml = w[0][0] * (sl - w[0][1]), mr = w[1][0] * (sr - w[1][1]);
    double pt[2];
    for (int s = 0; s < 2; ++s) pt[s] = w[s][4] + 0.5 * (b2 + (double)w[s][5] * w[s][5] + (double)w[s][6] * w[s][6]);
    const double sm = (mr * w[1][1] - ml * w[0][1] - pt[1] + pt[0]) / (mr - ml);
    for (int s = 0; s < 2; ++s) {
      const double num = (s == 0 ? ml : mr) * ((s == 0 ? sl : sr) - sm), den = num - b2;
      const double r = fabs(den) / fmax(fabs(num), b2);
      if (r > 0.5 * Eps<double>::degen) kappa = fmax(kappa, 1.0 + 1.0 / r);
    }
  }
  double speed = cm, rho = 0.5 * ((double)w[0][0] + w[1][0]);
  for (int s = 0; s < 2; ++s) for (int i = 1; i < 4; ++i) speed += fabs((double)w[s][i]);
  const double b = sqrt(rho) * speed, rc = rho * speed;
  const double scale[7] = {rc, rc * speed, rc * speed, rc * speed, rc * speed * speed, b * speed, b * speed};
  const double eps = 2.220446049250313e-16;
  // the plain fast speed takes the root of a difference that may cancel: an
  // error of up to sqrt(eps), which moves the flux of a jump by as much
  const double dc = fabs((double)c1 - (double)c2) / cm;
  double worst = dc <= sqrt(eps) ? 0.0 : 1e30;
  for (int i = 0; i < 7; ++i) {
    const double d = fabs((double)f[i] - (double)h[i]) / scale[i];
    worst = d <= worst ? worst : (d == d ? d : 1e30);
  }
  return worst / (64.0 * eps * kappa + dc);
}

__host__ __device__ inline double relative(double got, double ref) {
  if (got != got || ref != ref) return got != got && ref != ref ? 0.0 : 1.0;
  if (got == ref) return 0.0;
  return ref == 0.0 || ref - ref != 0.0 ? 1.0 : fabs(got - ref) / fabs(ref);
}
__host__ __device__ double math_excess(int kind, unsigned long long q, bool) {
  const double special[10] = {0.0, -0.0, 4.9e-324, -4.9e-324, 1.0 / 0.0, -1.0 / 0.0, 0.0 / 0.0, 2.2e-308, -1.0, -2.5};
  const unsigned long long z = mix64(q), e = 723 + (z >> 52) % 601;
  union { unsigned long long u; double d; } bits;
  bits.u = (e << 52) | (mix64(z) & 0xfffffffffffffull);
  const double x = q < 10 ? special[q] : kind == 0 && (z & 1) ? -bits.d : bits.d;
  const double got = kind == 0 ? qrcp_(x) : kind == 1 ? qrsqrt_(x) : qroot_(x);
  const double ref = kind == 0 ? 1.0 / x : kind == 1 ? 1.0 / sqrt(x) : sqrt(x);
  return relative(got, ref) / (q < 10 ? 1e-300 : 8.881784197001252e-16);   // 2^-50
}
__host__ __device__ double slope_excess(int kind, unsigned long long q, bool) {
  Rng g{mix64(q * 8 + kind + 77)};
  const double jump = kind == 0 ? 0.5 : 1e-2;
  double base[7], w[3][7], a[7], b[7], bn = g.u(-2, 2);
  for (int i = 0; i < 7; ++i) base[i] = i == 0 ? exp(g.u(-2, 2)) : i == 4 ? exp(g.u(-3, 2)) : g.u(-1, 1);
  if (kind == 2) bn = 0.0;
  if (kind == 3) base[5] = base[6] = 0.0;
  for (int s = 0; s < 3; ++s)
    for (int i = 0; i < 7; ++i)
      w[s][i] = i == 0 || i == 4 ? base[i] * exp(0.5 * jump * g.u(-1, 1)) : base[i] + jump * g.u(-1, 1);
  if (kind == 3) w[1][5] = w[1][6] = 0.0;
  char_half_slope<double>(w[0], w[1], w[2], bn, 5.0 / 3.0, a);
  char_half_slope(w[0], w[1], w[2], bn, 5.0 / 3.0, b);
  // the plain one takes the root of a difference of a^2, b^2 and their
  // discriminant's root: its rounding error relative to what is left is
  // amplified by a^2 over a^2 b_t^2 / (a^2 + b^2)
  const double ir = 1.0 / w[1][0], a2 = 5.0 / 3.0 * w[1][4] * ir;
  const double bt2 = (w[1][5] * w[1][5] + w[1][6] * w[1][6]) * ir, s = a2 + bn * bn * ir + bt2;
  const double kappa = kind == 3 ? 1.0 : 1.0 + s * s / (a2 * bt2 < 1e-3 * s * s ? 0.0 : a2 * bt2);
  double worst = 0.0, norm = 0.0;
  for (int i = 0; i < 7; ++i) {
    const double m = fabs(w[1][i] - w[0][i]) + fabs(w[2][i] - w[1][i]);
    norm += m * m;
  }
  for (int i = 0; i < 7; ++i) worst = fmax(worst, fabs(a[i] - b[i]));
  return worst / (sqrt(norm) * (256.0 * 2.220446049250313e-16) * kappa);
}

enum { FLUX, MATH, SLOPE };
__host__ __device__ inline double excess(int what, int kind, unsigned long long q, bool hll) {
  return what == FLUX ? face_excess(kind, q, hll) : what == MATH ? math_excess(kind, q, hll) : slope_excess(kind, q, hll);
}
__global__ void check(int what, int kind, bool hll, unsigned long long n, unsigned long long* word) {
  double m = 0.0;
  for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < n;
       q += (unsigned long long)gridDim.x * blockDim.x)
    m = fmax(m, excess(what, kind, q, hll));
  atomicMax(word, (unsigned long long)__double_as_longlong(m));
}

double worst(bool host, int what, int kind, bool hll) {
  double m = 0.0;
  if (host) {
    for (unsigned long long q = 0; q < 200000; ++q) {
      const double e = excess(what, kind, q, hll);
      m = e > m ? e : m;
    }
    return m;
  }
  unsigned long long* d;
  if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 1e30;
  check<<<512, 128>>>(what, kind, hll, 1ull << 22, d);
  if (cudaMemcpy(&m, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1e30;
  return m;
}

int main(int argc, char** argv) {
  const bool host = argc > 1 && !strcmp(argv[1], "host");
  printf("{");
  for (int hll = 0; hll < 2; ++hll)
    for (int kind = 0; kind < 5; ++kind)
      printf("%s\"%s%d\": %.3g", hll + kind ? ", " : "", hll ? "hll" : "hlld", kind, worst(host, FLUX, kind, hll));
  const char* names[3] = {"rcp", "rsqrt", "root"};
  for (int kind = 0; kind < 3; ++kind) printf(", \"%s\": %.3g", names[kind], worst(host, MATH, kind, false));
  for (int kind = 0; kind < 4; ++kind) printf(", \"slope%d\": %.3g", kind, worst(host, SLOPE, kind, false));
  printf("}\n");
  return 0;
}
