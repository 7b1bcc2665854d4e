// The sliced inverse with and without the lane that runs ahead: the same bits, each within its workspace.
// Arguments: m slices.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "emu.cuh"

using namespace omm;

int main(int argc, char** argv) {
  const int m = std::atoi(argv[1]), slices = std::atoi(argv[2]);
  const size_t mm = (size_t)m * m;
  const long canary = 1 << 20;
  std::mt19937_64 gen(m);
  std::normal_distribution<double> normal;
  std::vector<double> A(mm), P[2];
  for (int i = 0; i < m; ++i)
    for (int j = 0; j <= i; ++j) A[(size_t)i * m + j] = A[(size_t)j * m + i] = (i == j ? 3.0 : 0.0) + 0.5 * normal(gen) / std::sqrt((double)m);
  try {
    const cudaStream_t st = nullptr;
    for (int k = 0; k < 2; ++k) {
      const size_t bytes = spd_inverse_sliced_workspace_bytes(m, slices, k == 0);
      double *a, *p;
      char* work;
      int* flags;
      mem::alloc(&a, mm, st);
      mem::alloc(&p, mm, st);
      mem::alloc(&work, bytes + canary, st);
      mem::alloc(&flags, 2, st);
      OMM_CUDA_TRY(cudaMemset(work, 0xA5, bytes + canary));
      OMM_CUDA_TRY(cudaMemset(flags, 0, 2 * sizeof(int)));
      OMM_CUDA_TRY(cudaMemcpy(a, A.data(), mm * 8, cudaMemcpyHostToDevice));
      spd_inverse_sliced(st, m, a, p, work, flags, flags + 1, slices, k == 0);
      P[k].resize(mm);
      std::vector<unsigned char> tail(canary);
      int f[2];
      OMM_CUDA_TRY(cudaMemcpy(P[k].data(), p, mm * 8, cudaMemcpyDeviceToHost));
      OMM_CUDA_TRY(cudaMemcpy(tail.data(), work + bytes, canary, cudaMemcpyDeviceToHost));
      OMM_CUDA_TRY(cudaMemcpy(f, flags, sizeof(f), cudaMemcpyDeviceToHost));
      for (unsigned char c : tail)
        if (c != 0xA5) {
          std::printf("written past the workspace\n");
          return 1;
        }
      if (f[0] || f[1]) {
        std::printf("flags %d %d\n", f[0], f[1]);
        return 1;
      }
      for (void* q : {(void*)a, (void*)p, (void*)work, (void*)flags}) mem::release(q, st);
    }
  } catch (const CudaError& e) {
    std::printf("%s: %s\n", e.what, cudaGetErrorString(e.err));
    return 1;
  }
  if (std::memcmp(P[0].data(), P[1].data(), mm * 8) != 0) {
    std::printf("other bits without the lane that runs ahead\n");
    return 1;
  }
  double worst = 0.0;  // a few columns of A P = 1
  for (int j = 0; j < m; j += m / 7 + 1)
    for (int i = 0; i < m; ++i) {
      double sum = i == j ? -1.0 : 0.0;
      for (int k = 0; k < m; ++k) sum += A[(size_t)i * m + k] * P[0][(size_t)k * m + j];
      if (!(std::fabs(sum) <= worst)) worst = std::fabs(sum);
    }
  // 2^-16 of each product in the split form, less with slices and float32 leaves; 2^-44 with ten slices
  const double bound = 16.0 * std::sqrt((double)m) * std::ldexp(1.0, slices == 10 ? -44 : -16);
  std::printf("largest error %.1e, bound %.1e\n", worst, bound);
  return !(worst <= bound);
}
