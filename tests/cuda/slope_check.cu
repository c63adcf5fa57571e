// The FP64 characteristic half slope (char_half_slope) where the transverse
// field is small, against the same projection in long double with roots
// that do not cancel, on the host or the device (argument "host" or "device"
// says where the slope under test runs): prints one JSON object with the
// largest difference over its bound by kind; tests/test_char_slope.py builds and
// runs it.  A difference that is not a number counts as 1e30.
// Kinds: |B_t| of 1e-2 ... 1e-10 of the sound speed (in velocity units) with a^2 above
// b^2 (even kinds) and below it (odd ones); the last two kinds have transverse fields
// of order one.
// Bound of a component: the wave amplitudes are sums of at most 20 products,
// each of at most 10 rounded factors, of a difference and coefficients 1, rho, a,
// sqrt(rho) or their quotients, so 256 eps of the largest such product of the
// differences; the slopes are Lipschitz in them.  beta = B_t / |B_t| and alpha
// are smooth in the state away from B_t = 0 and have no amplified errors:
// c_f^2 - a^2 and a^2 - c_s^2 come from a product, not from a difference.  The
// one amplified term is a^2 - b^2 itself, which cancels where the speeds meet:
// 1 + s / |a^2 - b^2|.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>

#include "physics.cuh"

using namespace mhd;

static unsigned long long mix64(unsigned long long z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
struct Rng {
  unsigned long long s;
  double u(double a, double b) {
    s = mix64(s);
    return a + (b - a) * (double)(s >> 11) * (1.0 / 9007199254740992.0);
  }
};
struct Item {
  double w[3][7], bn, slope[7];
};
static const double kGamma = 5.0 / 3.0;
enum { KINDS = 12, N = 20000 };

static void make(int kind, unsigned long long q, Item& t) {
  Rng g{mix64(q * 16 + kind)};
  double base[7];
  for (int i = 0; i < 7; ++i) base[i] = i == 0 ? exp(g.u(-2, 2)) : i == 4 ? exp(g.u(-2, 2)) : g.u(-1, 1);
  const double a = sqrt(kGamma * base[4] / base[0]), sr = sqrt(base[0]);
  t.bn = (q & 1 ? 1.0 : -1.0) * a * sr * (kind % 2 == 0 ? g.u(0.1, 0.8) : g.u(1.25, 3.0));
  const double small = kind >= 10 ? g.u(0.1, 1.0) : pow(10.0, -2.0 * (kind / 2 + 1)), angle = g.u(0, 6.28);
  base[5] = a * sr * small * cos(angle);
  base[6] = a * sr * small * sin(angle);
  for (int s = 0; s < 3; ++s)
    for (int i = 0; i < 7; ++i)
      t.w[s][i] = s == 1 ? base[i] : i == 0 || i == 4 ? base[i] * exp(0.3 * g.u(-1, 1)) : base[i] + 0.3 * g.u(-1, 1);
}

typedef long double L;
static L mc(L m, L p) {
  if ((m < 0) != (p < 0) || m == 0 || p == 0) return 0;
  const L r = fminl(fminl(fabsl(m), fabsl(p)), fabsl(m + p) / 4);
  return p < 0 ? -r : r;
}
// Projection on the eigenvectors of the primitive system (Roe & Balsara 1996).
static void reference(const Item& t, L* slope, L* scale) {
  const double* w = t.w[1];
  const L rho = w[0], sr = sqrtl(rho), a2 = (L)kGamma * w[4] / rho, a = sqrtl(a2), bn = t.bn / sr;
  const L bt = hypotl(w[5], w[6]) / sr, y = w[5] / (bt * sr), z = w[6] / (bt * sr), sg = t.bn >= 0 ? 1 : -1;
  const L bsq = bn * bn + bt * bt, d = a2 - bsq, disc = sqrtl(d * d + 4 * a2 * bt * bt);
  const L cf2 = (a2 + bsq + disc) / 2, cf = sqrtl(cf2), cs = a * fabsl(bn) / cf;
  const L big = (fabsl(d) + disc) / 2, other = a2 * bt * bt / big;
  const L af = sqrtl((d >= 0 ? big : other) / disc), as = sqrtl((d >= 0 ? other : big) / disc);
  const L fc = af * cf, sc = as * cs;
  L c[2][7];
  for (int s = 0; s < 2; ++s) {
    L v[7];
    for (int i = 0; i < 7; ++i) v[i] = (L)t.w[s + 1][i] - t.w[s][i];
    const L along = y * v[2] + z * v[3], across = z * v[2] - y * v[3], b = (y * v[5] + z * v[6]) / sr;
    const L xf = (fc * v[1] - sg * sc * along) / (2 * a2), yf = af * v[4] / (2 * a2 * rho) + as * b / (2 * a);
    const L xs = (sc * v[1] + sg * fc * along) / (2 * a2), ys = as * v[4] / (2 * a2 * rho) - af * b / (2 * a);
    const L xa = sg * across / 2, ya = (y * v[6] - z * v[5]) / (2 * sr);
    const L all[7] = {yf - xf, ya - xa, ys - xs, v[0] - v[4] / a2, ys + xs, ya + xa, yf + xf};
    for (int i = 0; i < 7; ++i) c[s][i] = all[i];
  }
  L k[7];
  for (int i = 0; i < 7; ++i) k[i] = mc(c[0][i], c[1][i]);
  const L F = k[6] + k[0], f = k[6] - k[0], S = k[4] + k[2], s = k[4] - k[2], A = k[5] + k[1], e = k[5] - k[1];
  slope[0] = rho * (af * F + as * S) + k[3];
  slope[1] = fc * f + sc * s;
  slope[2] = sg * (y * (fc * s - sc * f) + z * e);
  slope[3] = sg * (z * (fc * s - sc * f) - y * e);
  slope[4] = rho * a2 * (af * F + as * S);
  slope[5] = y * a * sr * (as * F - af * S) - z * sr * A;
  slope[6] = z * a * sr * (as * F - af * S) + y * sr * A;
  // the differences in units of speed, and back in each component's
  L speed = 0;
  const L c0 = a + fabsl(bn) + bt;
  for (int q = 0; q < 2; ++q)
    for (int i = 0; i < 7; ++i) {
      const L v = fabsl((L)t.w[q + 1][i] - t.w[q][i]);
      speed += i == 0 ? v * c0 / rho : i == 4 ? v / (rho * a) : i < 4 ? v : v / sr;
    }
  const L amplified = speed * (c0 / a) * (1 + (a2 + bsq) / fabsl(d));
  for (int i = 0; i < 7; ++i)
    scale[i] = amplified * (i == 0 ? rho / a : i == 4 ? rho * c0 : i < 4 ? 1 : sr);
}

__global__ void run(Item* t, int n, double gamma) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) char_half_slope(t[i].w[0], t[i].w[1], t[i].w[2], t[i].bn, gamma, t[i].slope);
}

int main(int argc, char** argv) {
  const bool host = argc > 1 && !strcmp(argv[1], "host");
  Item* t = new Item[N];
  printf("{");
  for (int kind = 0; kind < KINDS; ++kind) {
    for (int q = 0; q < N; ++q) make(kind, q, t[q]);
    if (host) {
      for (int q = 0; q < N; ++q) char_half_slope(t[q].w[0], t[q].w[1], t[q].w[2], t[q].bn, kGamma, t[q].slope);
    } else {
      Item* d;
      if (cudaMalloc(&d, N * sizeof(Item)) != cudaSuccess) return 1;
      cudaMemcpy(d, t, N * sizeof(Item), cudaMemcpyHostToDevice);
      run<<<(N + 127) / 128, 128>>>(d, N, kGamma);
      if (cudaMemcpy(t, d, N * sizeof(Item), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
      cudaFree(d);
    }
    double worst = 0.0;
    for (int q = 0; q < N; ++q) {
      L ref[7], scale[7];
      reference(t[q], ref, scale);
      for (int i = 0; i < 7; ++i) {
        const double r = (double)(fabsl((L)t[q].slope[i] - ref[i]) / (scale[i] * 256 * 2.220446049250313e-16L));
        if (!(r <= worst)) worst = r == r ? r : 1e30;
      }
    }
    printf("%s\"kind%d\": %.3g", kind ? ", " : "", kind, worst);
  }
  printf("}\n");
  return 0;
}
