// Check of the FP64 solver's arithmetic helpers on the device: reciprocal, root, halving,
// h^(-7/3), the cut to FP32 and the detector's FP32 pre-test, against CUDA's own operations on
// random arguments over their whole ranges and on listed edges.  tests/test_gpu_fp64_helpers.py
// builds it with the library's flags and runs it; exit status 0 = every bound holds.
//
// Bounds, in u = 2^-53.  rcp64: the step leaves e^3 of the approximation's 1.0e-6 and one
// rounding, 1.01 u.  sqrt64: the two steps leave 3/2 d^3 of 1.9e-6 and one rounding, 1.1 u
// (the residual that is checked is of the square, so twice that).  h_m73: r^7 keeps 2/3 u of
// the rounding of r^3 that the correction does not see and two roundings, the correction one,
// 3.7 u; 1 / (h h cbrt(h)) as CUDA rounds it 5 u.  half64 and cut32 are exact.
#include <cmath>
#include <cstdio>
#include <limits>

#include "dg2_device.cuh"

using namespace dg2;

constexpr double kU = 1.1102230246251565e-16;

// SplitMix64
__device__ unsigned long long mix(unsigned long long x) {
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
// a positive double with a random mantissa and an exponent in [lo, hi)
__device__ double draw(unsigned long long k, int lo, int hi) {
  const unsigned long long r = mix(k), e = 1023 + lo + mix(r) % (hi - lo);
  return __longlong_as_double((long long)(e << 52 | r >> 12));
}
__device__ double uniform(unsigned long long k) { return (double)(mix(k) >> 11) * kU; }

enum { RCP, ROOT, POW, HALF, CUT, CALM, CALM_SEEN, NEAR_SEEN, NSLOT };
__device__ double worst[NSLOT];  // non-negative: order as their bits
__device__ void note(int slot, double v) {
  if (!(v >= 0.0)) v = INFINITY;  // NaN fails
  atomicMax((unsigned long long*)&worst[slot], (unsigned long long)__double_as_longlong(v));
}
__device__ bool same(double a, double b) {
  return isnan(a) ? isnan(b) : __double_as_longlong(a) == __double_as_longlong(b);
}

__device__ void check_rcp(double x) {
  const double r = rcp64(x);
  note(RCP, fabs(fma(-x, r, 1.0)) / kU / 1.01);
  note(RCP, fabs(r * x - 1.0) / (4.0 * kU));
  note(RCP, fabs(r - 1.0 / x) / fabs(1.0 / x) / kU / 2.01);
}
__device__ void check_root(double x) {
  const double s = sqrt64(x), q = sqrt(x);
  if (x >= 0x1p-960) note(ROOT, fabs(fma(-s, s, x)) / x / kU / 2.2);
  note(ROOT, fabs(s - q) / q / kU / (x >= 1e-300 ? 2.1 : 3.0));
}
__device__ void check_pow(double h) {
  const double a = h_m73(h), b = 1.0 / (h * h * cbrt(h));
  if (h > 1e-30 && h < 1e30) note(POW, fabs(a - b) / b / kU / 8.7);
  else note(POW, same(a, b) ? 0.0 : INFINITY);
}
__device__ void check_half(double x) { note(HALF, same(half64(x), 0.5 * x) ? 0.0 : 2.0); }
__device__ void check_cut(double x) {
  const float c = cut32(x), a = (float)fabs(x);
  const float want = fabs(x) < 0x1p-126 ? 0.f : !(fabs(x) < 0x1p128) ? INFINITY : __double2float_rz(x);
  note(CUT, (c == want && (a == a || c == INFINITY)) ? 0.0 : 2.0);
}
// The pre-test against the test: a shock that the FP64 test sees is never called calm.
__device__ void check_calm(unsigned long long k) {
  const double tol = 1e-5, th = exp2(-6.0 + 12.0 * uniform(k)), size = exp2(-30.0 + 40.0 * uniform(k + 1));
  double v[6];
  for (int i = 0; i < 6; ++i)  // averages and slopes of three cells
    v[i] = size * ((i & 1) ? 0.1 : 1.0) * (1.0 + (k & 1 ? 1e-6 : 1.0) * (uniform(k + 2 + i) - 0.5));
  if (k & 2) {  // the east jump set within 1e-7 of the threshold
    const double mag = fabs(v[2]) + fabs(v[3]) * 0.57735026918962576;
    const double jump = th * (mag < tol ? tol : mag) * (1.0 + 1e-7 * (uniform(k + 9) - 0.5));
    v[4] = v[5] + (v[2] + v[3]) + jump;
  }
  float f[6], s = 0.f;
  for (int i = 0; i < 6; ++i) { f[i] = cut32(v[i]); s += fabsf(f[i]); }
  const bool quiet = calm(cut32(th), cut32(tol), f[0], f[1], f[2], f[3], f[4], f[5], s);
  const double jE = fabs((v[4] - v[5]) - (v[2] + v[3])), jW = fabs((v[2] - v[3]) - (v[0] + v[1]));
  double mag = fabs(v[2]) + fabs(v[3] * 0.57735026918962576);
  if (mag < tol) mag = tol;
  const bool shock = fmax(jE, jW) > th * mag;
  note(CALM, quiet && shock ? 2.0 : 0.0);
  if (quiet) note(CALM_SEEN, 1.0);
  if (shock) note(NEAR_SEEN, 1.0);
}

__global__ void random_arguments(int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const unsigned long long k = 64ull * t;
  const double x = draw(k, -1021, 1021);
  check_rcp(x);
  check_rcp(-x);
  check_root(draw(k + 2, -1022, 1023));
  check_pow(draw(k + 4, -110, 110));
  const double any = __longlong_as_double((long long)mix(k + 6));  // any bit pattern
  check_half(any);
  check_half(draw(k + 8, -1022, -1018));
  check_cut(any);
  check_cut(draw(k + 10, -130, -120));
  check_cut(-draw(k + 12, 120, 132));
  check_calm(64ull * t + (t & 3));
}

__global__ void edges() {
  const double inf = INFINITY, nan = NAN, tiny = 0x1p-1022, sub = 0x1p-1074;
  const double one[] = {1.0, 2.0, 0.5, 1.0 - kU, 1.0 + 2.0 * kU, 0x1p-1021, 0x1p1021, 1e-300, 1e300};
  for (double x : one) { check_rcp(x); check_root(x); }
  check_root(tiny);
  check_root(1.7976931348623157e308);
  const double zero[] = {0.0, sub, 0.5 * tiny, tiny - sub};
  for (double x : zero) note(ROOT, sqrt64(x) == 0.0 ? 0.0 : INFINITY);
  // as sqrt: no root of a negative number, and a NaN of either sign stays one
  const double bad[] = {-1.0, -tiny, -1e300, -inf, nan, -nan, __longlong_as_double(~0ll)};
  for (double x : bad) note(ROOT, isnan(sqrt64(x)) ? 0.0 : INFINITY);
  const double h[] = {1e-30, 1e30, nextafter(1e-30, 1.0), nextafter(1e30, 0.0), 1e-31, 1e31, 1e-5, 1.0, 8.0, 1e-300};
  for (double x : h) check_pow(x);
  const double e[] = {0.0, sub, 3.0 * sub, tiny, tiny - sub, tiny + sub, 2.0 * tiny, 2.0 * tiny - sub,
                      2.0 * tiny + 2.0 * sub, 4.0 * tiny, 1.7976931348623157e308, inf, nan};
  for (double x : e) { check_half(x); check_half(-x); check_cut(x); check_cut(-x); }
  const double c[] = {0x1p-126, nextafter(0x1p-126, 0.0), nextafter(0x1p-126, 1.0), 0x1p128,
                      nextafter(0x1p128, 0.0), 0x1.fffffep127, 1.0, 1.0 + kU};
  for (double x : c) { check_cut(x); check_cut(-x); }
}

int main() {
  const int n = 1 << 24;
  random_arguments<<<n / 256, 256>>>(n);
  edges<<<1, 1>>>();
  double w[NSLOT];
  cudaError_t e = cudaMemcpyFromSymbol(w, worst, sizeof w);
  if (e != cudaSuccess) {
    printf("%s\n", cudaGetErrorString(e));
    return 2;
  }
  const char* names[] = {"rcp64", "sqrt64", "h_m73", "half64", "cut32", "calm"};
  bool ok = w[CALM_SEEN] > 0.0 && w[NEAR_SEEN] > 0.0;
  for (int k = 0; k <= CALM; ++k) {
    printf("%s: %.4f of its bound\n", names[k], w[k]);
    ok = ok && w[k] <= 1.0;
  }
  return ok ? 0 : 1;
}
