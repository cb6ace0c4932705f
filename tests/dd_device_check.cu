// Device check of the double-float -> double conversion (mf_dd.cuh): the device's conversion
// instructions against the host's integer form, which tests/dd_conversion_check.cu checks, on the same
// pairs -- normalised ones across the float range, powers of two with lo on either side, and zero,
// non-normalised and subnormal parts, inf and nan.  Prints "ok <count>" and exits 0, or the first difference.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "mf_dd.cuh"

__global__ void convert(const mf::dd* in, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = mf::dd_to_double(in[i]);
}

int main() {
  std::vector<mf::dd> v;
  std::mt19937_64 g(12345);
  std::uniform_real_distribution<double> u(1.0, 2.0);
  std::uniform_int_distribution<int> ex(-126, 127);
  for (int i = 0; i < 1000000; ++i) {
    const double x = std::ldexp(u(g), ex(g)) * ((i & 1) ? -1.0 : 1.0);
    const float h = (float)x;
    v.push_back(mf::dd(h, std::isinf(h) ? 0.0f : (float)(x - (double)h)));
  }
  for (int e = -126; e <= 127; ++e)
    for (int s = 24; s <= 60; ++s)
      for (int sg = 0; sg < 4; ++sg)
        v.push_back(mf::dd(std::ldexp((sg & 1) ? -1.0f : 1.0f, e), std::ldexp((sg & 2) ? -1.0f : 1.0f, e - s)));
  const float edge[] = {0.0f, -0.0f, 1.0f, -3.0f, 0.75f, 0x1p-126f, 0x1.fffffcp-127f, 0x1p-149f, -0x1p-140f, 0x1.fffffep127f,
                        INFINITY, -INFINITY, NAN};
  for (float h : edge)
    for (float l : edge) v.push_back(mf::dd(h, l));
  const int n = (int)v.size();
  mf::dd* in;
  double* out;
  std::vector<double> r(n);
  if (cudaMalloc(&in, n * sizeof(mf::dd)) != cudaSuccess || cudaMalloc(&out, n * sizeof(double)) != cudaSuccess) return 2;
  cudaMemcpy(in, v.data(), n * sizeof(mf::dd), cudaMemcpyHostToDevice);
  convert<<<(n + 255) / 256, 256>>>(in, out, n);
  if (cudaMemcpy(r.data(), out, n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  for (int i = 0; i < n; ++i) {
    const double want = mf::dd_to_double(v[i]);
    if (!(r[i] == want || (std::isnan(r[i]) && std::isnan(want)))) {
      std::printf("FAIL h=%a l=%a device %a host %a\n", v[i].hi, v[i].lo, r[i], want);
      return 1;
    }
  }
  std::printf("ok %d\n", n);
  return 0;
}
