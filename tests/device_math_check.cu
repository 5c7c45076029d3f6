// Evaluates the error-weight quotients and the step-factor root of
// csrc/qt_device.cuh on the device (test infrastructure, built and run by
// tests/test_gpu_error_weights.py).
//
// argv[1]: a file of int64 n, double x[n], w[n], r[n]; argv[2]: the output,
// double ratio(x, w)[n], float ratio((float)x, (float)w)[n] as doubles,
// inv_root10(r, seed as the step control forms it)[n].
#include "../paper_1110_0573_gb300/csrc/qt_device.cuh"

#include <cstdio>
#include <vector>

__global__ void eval(const double *in, double *out, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = in[i], w = in[n + i], r = in[2 * n + i];
  out[i] = qt::ratio(x, w);
  out[n + i] = (double)qt::ratio((float)x, (float)w);
  out[2 * n + i] = qt::inv_root10(r, qt::ex2_approx(-0.1f * qt::lg2_approx((float)r)));
}

int main(int argc, char **argv) {
  if (argc != 3) return 2;
  long long n = 0;
  FILE *f = fopen(argv[1], "rb");
  if (!f || fread(&n, 8, 1, f) != 1 || n < 1 || n > (1ll << 24)) return 3;
  std::vector<double> h(3 * n);
  if (fread(h.data(), 8, 3 * n, f) != (size_t)(3 * n)) return 4;
  fclose(f);
  double *in = nullptr, *out = nullptr;
  if (cudaMalloc(&in, 24 * n) != cudaSuccess || cudaMalloc(&out, 24 * n) != cudaSuccess) return 5;
  if (cudaMemcpy(in, h.data(), 24 * n, cudaMemcpyHostToDevice) != cudaSuccess) return 6;
  eval<<<(unsigned)((n + 255) / 256), 256>>>(in, out, n);
  if (cudaMemcpy(h.data(), out, 24 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 7;
  f = fopen(argv[2], "wb");
  if (!f || fwrite(h.data(), 8, 3 * n, f) != (size_t)(3 * n)) return 8;
  return fclose(f) ? 9 : 0;
}
