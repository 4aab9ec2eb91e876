// Conversions between FP64 and float-float (ff.cuh) on values given by this program: ff_split keeps 47
// bits, the smallest and largest exponents behave as stated, and nothing that is not finite, or is too
// large for FP32, comes out finite; ff_join returns the value scaled by a power of two, 46 bits behind
// the leading one, infinite above the double range and NaN for a high part that is not finite.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "../paper_2407_06409_gb300/csrc/ff.cuh"

__global__ void split(const double* v, float2* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ff a = ff_split(v[i]);
  o[i] = make_float2(a.hi, a.lo);
}
__global__ void join(const float2* v, const int* shift, double* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) o[i] = ff_join(ff_quick_two_sum(v[i].x, v[i].y), shift[i]);   // joins take normalised pairs
}

static double bits(unsigned long long b) {
  double d;
  memcpy(&d, &b, 8);
  return d;
}

int main() {
  std::vector<double> v;
  srand(3);
  for (int i = 0; i < 20000; ++i) {   // every exponent from 2^-140 to 2^140, both signs
    const double m = 1.0 + (rand() + rand() / 2147483648.0) / 2147483648.0;
    v.push_back((i & 1 ? -m : m) * std::ldexp(1.0, i % 281 - 140));
  }
  for (double x : {0.0, -0.0, 5e-324, std::nextafter(1.0, 2.0), std::nextafter(2.0, 1.0), std::ldexp(1.0, 128),
                   std::nextafter(std::ldexp(1.0, 128), 0.0), 1e300, -1e300, std::ldexp(1.0, -126)})
    v.push_back(x);
  const size_t finite = v.size();
  for (unsigned long long b : {0x7ff0000000000000ULL, 0xfff0000000000000ULL, 0x7ff8000000000000ULL, 0xfff8000000000000ULL,
                               0x7ff0000000000001ULL, 0x7fffffffffffffffULL, 0xffffffffffffffffULL, 0x7fffffffffffffe0ULL})
    v.push_back(bits(b));
  const int n = (int)v.size();
  double *dv, *dj;
  float2* ds;
  int* dk;
  std::vector<int> k(n);
  for (int i = 0; i < n; ++i) k[i] = i % 601 - 300;
  std::vector<float2> s(n);
  std::vector<double> j(n);
  cudaMalloc(&dv, 8 * n);
  cudaMalloc(&dj, 8 * n);
  cudaMalloc(&ds, 8 * n);
  cudaMalloc(&dk, 4 * n);
  cudaMemcpy(dv, v.data(), 8 * n, cudaMemcpyHostToDevice);
  cudaMemcpy(dk, k.data(), 4 * n, cudaMemcpyHostToDevice);
  split<<<(n + 127) / 128, 128>>>(dv, ds, n);
  join<<<(n + 127) / 128, 128>>>(ds, dk, dj, n);
  cudaMemcpy(s.data(), ds, 8 * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(j.data(), dj, 8 * n, cudaMemcpyDeviceToHost);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  int bad = 0;
  auto fail = [&](int i, const char* what) {
    if (++bad <= 10) printf("%s: v %a -> %a + %a, 2^%d: %a\n", what, v[i], s[i].x, s[i].y, k[i], j[i]);
  };
  const double top = std::nextafter(std::ldexp(1.0, 128), 0.0);   // rounds up to 2^128
  for (int i = 0; i < n; ++i) {
    const double a = std::fabs(v[i]), hi = s[i].x, lo = s[i].y;
    if (i >= (int)finite || a >= top) {
      if (std::isfinite(s[i].x)) fail(i, "finite");
      if (!std::isnan(j[i])) fail(i, "joined to a number");
      continue;
    }
    // half a unit of the 47th bit; below 2^-80 the low part is gone, below 2^-126 all
    const double unit = a > 0 ? std::ldexp(1.0, std::ilogb(a)) : 0.0;
    const double tol = a < std::ldexp(1.0, -126) ? a : (a < std::ldexp(1.0, -79) ? unit * std::ldexp(1.0, -23) : unit * std::ldexp(1.0, -47));
    if (!(std::fabs(hi + lo - v[i]) <= tol)) fail(i, "split");
    const double x = std::ldexp(hi + lo, k[i]);
    if (!(std::fabs(j[i] - x) <= std::fabs(x) * std::ldexp(1.0, -46))) fail(i, "join");
  }
  // joins past the double range
  const float2 big[2] = {make_float2(1.5f, 0.f), make_float2(-3e38f, 0.f)};
  const int up[2] = {1024, 900};
  cudaMemcpy(ds, big, sizeof(big), cudaMemcpyHostToDevice);
  cudaMemcpy(dk, up, sizeof(up), cudaMemcpyHostToDevice);
  join<<<1, 32>>>(ds, dk, dj, 2);
  cudaMemcpy(j.data(), dj, 16, cudaMemcpyDeviceToHost);
  if (!(std::isinf(j[0]) && j[0] > 0) || !(std::isinf(j[1]) && j[1] < 0)) {
    printf("overflow: %a %a\n", j[0], j[1]);
    ++bad;
  }
  printf("%d values, %d wrong\n", n, bad);
  return bad ? 1 : 0;
}
