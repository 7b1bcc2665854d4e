// One sliced product with an upper-triangular B and its block lists, its slabs filled with NaN beforehand:
// C (M x N) = A B^T against float64 sums on the host, of sampled rows and of every column. Arguments: M N.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "emu.cuh"

using namespace omm;

int main(int argc, char** argv) {
  const int M = std::atoi(argv[1]), N = std::atoi(argv[2]), K = N, S = 10;
  std::mt19937_64 gen(3);
  std::normal_distribution<double> normal;
  std::vector<double> A((size_t)M * K), B((size_t)N * K, 0.0), C((size_t)M * N);
  for (double& x : A) x = normal(gen);
  for (int i = 0; i < N; ++i)
    for (int j = i; j < K; ++j) B[(size_t)i * K + j] = normal(gen);
  try {
    const cudaStream_t st = nullptr;
    const long ld = (K + 7) / 8 * 8, slab_n = tc::sliced_workspace_doubles();
    double *a, *b, *c, *slab;
    __nv_bfloat16 *sa, *sb;
    int* err;
    mem::alloc(&a, A.size(), st);
    mem::alloc(&b, B.size(), st);
    mem::alloc(&c, C.size(), st);
    mem::alloc(&slab, slab_n, st);
    mem::alloc(&sa, (size_t)S * M * ld, st);
    mem::alloc(&sb, (size_t)S * N * ld, st);
    mem::alloc(&err, 1, st);
    OMM_CUDA_TRY(cudaMemcpy(a, A.data(), A.size() * 8, cudaMemcpyHostToDevice));
    OMM_CUDA_TRY(cudaMemcpy(b, B.data(), B.size() * 8, cudaMemcpyHostToDevice));
    OMM_CUDA_TRY(cudaMemset(slab, 0xFF, slab_n * 8));
    OMM_CUDA_TRY(cudaMemset(err, 0, sizeof(int)));
    tc::BlockLists lists;
    const int width = 256;
    tc::block_lists(st, b, N, K, K, 1, &width, &lists);
    emu::slice_rows(st, a, M, K, K, S, sa, ld, nullptr);
    emu::slice_rows(st, b, N, K, K, S, sb, ld, nullptr);
    emu::gemm(st, tc::make_operand(sa, M, K, ld, S, true), tc::make_operand(sb, N, K, ld, S, false), K, S,
              tc::Epilogue{c, N, N, 0, 1.0, 0.0, M, N, nullptr, err}, slab, &lists);
    int e = 0;
    OMM_CUDA_TRY(cudaMemcpy(&e, err, sizeof(int), cudaMemcpyDeviceToHost));
    OMM_CUDA_TRY(cudaMemcpy(C.data(), c, C.size() * 8, cudaMemcpyDeviceToHost));
    if (e != 0) {
      std::printf("a bounded wait expired (%d)\n", e);
      return 1;
    }
  } catch (const CudaError& e) {
    std::printf("%s: %s\n", e.what, cudaGetErrorString(e.err));
    return 1;
  }
  double worst = 0.0;
  for (int i = 0; i < M; i += 37)
    for (int j = 0; j < N; ++j) {
      double sum = 0.0;
      for (int k = j; k < K; ++k) sum += A[(size_t)i * K + k] * B[(size_t)j * K + k];
      const double d = std::fabs(C[(size_t)i * N + j] - sum);
      if (!(d <= worst)) worst = d;  // (a NaN stays)
    }
  // 2^-50 of each row's largest element (below 6.5 here), twice over the K products, with a factor 2
  const double bound = 2.0 * 2.0 * std::ldexp(1.0, -50) * 6.5 * 6.5 * K;
  std::printf("largest error %.2e, bound %.2e\n", worst, bound);
  return !(worst <= bound);
}
