// Float64 GEMM on the FP64 pipes (DFMA). GB300 keeps only a small float64
// rate (two FMA lanes per SM and clock), so a product is bound by how evenly
// its FMAs spread over the SMs, not by memory. Large products take 64x64
// tiles with a 4x4 register block per thread; smaller ones take 32x32 or
// 16x16 tiles, with the contraction split over the CTAs of a cluster where
// the tiles alone leave SMs idle (choose_split below).
// It serves the float64 OMM path, the float64 refinement and certificate of
// the mixed path, and the Cholesky inverse of the preconditioner.
#include "omm_internal.cuh"
#include "pdl.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

namespace omm {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;

__global__ void __launch_bounds__(NT)
dgemm_kernel(int transA, int transB, int M, int N, int K, double alpha,
             const double* __restrict__ A, long lda, long sA,
             const double* __restrict__ B, long ldb, long sB,
             double beta, double* C, long ldc, long sC, int tri, const int* skip) {
  dev::pdl_begin();
  if (skip != nullptr && (skip[0] | skip[1])) return;
  const int row0 = blockIdx.y * BM;
  const int col0 = blockIdx.x * BN;
  if ((tri & kTriLower) && col0 > row0 + BM - 1) return;
  A += (long)blockIdx.z * sA;
  B += (long)blockIdx.z * sB;
  C += (long)blockIdx.z * sC;

  __shared__ double As[BK][BM];
  __shared__ double Bs[BK][BN];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  double acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;

  int kbeg = 0, kend = K;
  if (tri & kTriKStart) kbeg = (max(row0, col0) / BK) * BK;
  if (tri & kTriKFromCol) kbeg = max(kbeg, (col0 / BK) * BK);
  if (tri & kTriKToRow) kend = min(K, row0 + BM);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int t = 0; t < (BM * BK) / NT; ++t) {
      const int idx = tid + t * NT;
      int i, k;
      double v = 0.0;
      if (!transA) {
        i = idx / BK; k = idx % BK;
        const int gi = row0 + i, gk = k0 + k;
        if (gi < M && gk < K) v = A[(long)gi * lda + gk];
      } else {
        k = idx / BM; i = idx % BM;
        const int gi = row0 + i, gk = k0 + k;
        if (gi < M && gk < K) v = A[(long)gk * lda + gi];
      }
      As[k][i] = v;
    }
#pragma unroll
    for (int t = 0; t < (BN * BK) / NT; ++t) {
      const int idx = tid + t * NT;
      int j, k;
      double v = 0.0;
      if (!transB) {
        k = idx / BN; j = idx % BN;
        const int gj = col0 + j, gk = k0 + k;
        if (gj < N && gk < K) v = B[(long)gk * ldb + gj];
      } else {
        j = idx / BK; k = idx % BK;
        const int gj = col0 + j, gk = k0 + k;
        if (gj < N && gk < K) v = B[(long)gj * ldb + gk];
      }
      Bs[k][j] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      double a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[k][ty + 16 * r];
#pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = Bs[k][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int gi = row0 + ty + 16 * r;
    if (gi >= M) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int gj = col0 + tx + 16 * c;
      if (gj >= N) continue;
      double* p = C + (long)gi * ldc + gj;
      const double v = alpha * acc[r][c];
      *p = (beta == 0.0) ? v : fma(beta, *p, v);
    }
  }
}

// ---- small products: T x T tiles (T = 16 or 32), the contraction split over the CTAs of a cluster
// The products of a small problem (n x m x m with n = 36, m = 207, say) have few 64 x 64 tiles, and
// every SM without one idles while the others work through 64 x 64 x K FMAs at two per clock: the
// products of an m = 207, n = 36 solve took 176 us each on 4 to 16 SMs, 12 now. (By this alone the energy
// and gradients of that system went from 65.6 to 11.1 ms, a solve of m = 416, n = 64 from 76.1 to 11.4; they
// take 7 to 8 with what followed.) Here a tile is 16 x 16 or 32 x 32 and CTA q of a
// cluster of KS sums the q-th part of the contraction; the partial tiles meet in shared memory over
// the cluster (fixed order, so results stay reproducible) and every CTA stores its share of the rows.
// The float64 pipe takes a warp's FMA every 16 clocks, so one output per thread and two
// shared-memory loads per FMA do not slow it.
constexpr int SK = 32;  // contracted columns per stage

template <int T>
__global__ void __launch_bounds__(NT)
dgemm_small_kernel(int transA, int transB, int M, int N, int K, double alpha, const double* __restrict__ A, long lda,
                   long sA, const double* __restrict__ B, long ldb, long sB, double beta, double* C, long ldc,
                   long sC, int tri, const int* skip, int ks) {
  dev::pdl_begin();
  if (skip != nullptr && (skip[0] | skip[1])) return;
  constexpr int R = T / 16;                // outputs per thread and dimension
  constexpr int LD = T * SK / NT;          // elements of each operand a thread stages
  const int part = blockIdx.x % ks;        // = the rank in the cluster (ks CTAs along x)
  const int row0 = blockIdx.y * T, col0 = (blockIdx.x / ks) * T;
  if ((tri & kTriLower) && col0 > row0 + T - 1) return;  // the whole cluster: one tile
  A += (long)blockIdx.z * sA;
  B += (long)blockIdx.z * sB;
  C += (long)blockIdx.z * sC;
  __shared__ double As[SK][T + 1];
  __shared__ double Bs[SK][T + 1];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  int kbeg = 0, kend = K;
  if (tri & kTriKStart) kbeg = (max(row0, col0) / SK) * SK;
  if (tri & kTriKFromCol) kbeg = max(kbeg, (col0 / SK) * SK);
  if (tri & kTriKToRow) kend = min(K, row0 + T);
  if (ks > 1) {  // this CTA's run of stages
    const int stages = (max(kend - kbeg, 0) + SK - 1) / SK;
    const int s0 = stages * part / ks, s1 = stages * (part + 1) / ks;
    kend = min(kend, kbeg + s1 * SK);
    kbeg += s0 * SK;
  }
  double ra[LD], rb[LD];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int t = 0; t < LD; ++t) {
      const int idx = tid + t * NT;
      const int ia = transA ? idx % T : idx / SK, ka = transA ? idx / T : idx % SK;
      const int jb = transB ? idx / SK : idx % T, kb = transB ? idx % SK : idx / T;
      const int gi = row0 + ia, gka = k0 + ka, gj = col0 + jb, gkb = k0 + kb;
      ra[t] = (gi < M && gka < kend) ? (transA ? A[(long)gka * lda + gi] : A[(long)gi * lda + gka]) : 0.0;
      rb[t] = (gj < N && gkb < kend) ? (transB ? B[(long)gj * ldb + gkb] : B[(long)gkb * ldb + gj]) : 0.0;
    }
  };
  double acc[R][R];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < R; ++c) acc[r][c] = 0.0;
  if (kbeg < kend) fetch(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += SK) {
#pragma unroll
    for (int t = 0; t < LD; ++t) {
      const int idx = tid + t * NT;
      const int ia = transA ? idx % T : idx / SK, ka = transA ? idx / T : idx % SK;
      const int jb = transB ? idx / SK : idx % T, kb = transB ? idx % SK : idx / T;
      As[ka][ia] = ra[t];
      Bs[kb][jb] = rb[t];
    }
    __syncthreads();
    if (k0 + SK < kend) fetch(k0 + SK);  // the next stage's loads run beside this stage's FMAs
    const int kn = min(SK, kend - k0);
#pragma unroll 8
    for (int k = 0; k < kn; ++k) {
      double a[R], b[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = As[k][ty + 16 * r];
#pragma unroll
      for (int c = 0; c < R; ++c) b[c] = Bs[k][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < R; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
    }
    __syncthreads();
  }
  auto store = [&](int i, int j, double v) {
    const int gi = row0 + i, gj = col0 + j;
    if (gi >= M || gj >= N) return;
    double* p = C + (long)gi * ldc + gj;
    v *= alpha;
    *p = (beta == 0.0) ? v : fma(beta, *p, v);
  };
  if (ks == 1) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < R; ++c) store(ty + 16 * r, tx + 16 * c, acc[r][c]);
    return;
  }
  // partial tiles in shared memory (the A stages' room holds T x T: SK = 32 >= T), then each CTA adds
  // T / ks rows of all of them in the order of the contraction
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  double* mine = &As[0][0];
  static_assert(SK >= T, "a partial tile fits the A stage");
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < R; ++c) mine[(ty + 16 * r) * T + tx + 16 * c] = acc[r][c];
  cluster.sync();
  const int per = T * T / ks;
  for (int e = tid; e < per; e += NT) {
    const int at = part * per + e;
    double v = 0.0;
    for (int q = 0; q < ks; ++q) v += cluster.map_shared_rank(mine, q)[at];
    store(at / T, at % T, v);
  }
  cluster.sync();  // no CTA leaves while another may still read its tile
}

int sms() {
  static const int n = [] {
    int dev = 0, c = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) c = 152;
    return c;
  }();
  return n;
}

struct Split {
  int tile, ks;
};

constexpr long kMaxGridY = 65535;

// The tile and the split with the shortest estimated time. An SM works off its CTAs' FMAs at two
// per clock (their loads overlap each other's FMAs); a CTA alone needs about 700 clocks per stage
// for its loads; meeting over a cluster costs about 2500 clocks and storing a partial tile.
Split choose_split(long M, long N, long K, long batch) {
  Split best{64, 1};
  double best_t = 0.0;
  const double nsm = sms();
  for (int tile : {64, 32, 16}) {
    if (tile < 64 && (M + tile - 1) / tile > kMaxGridY) continue;  // tile rows are grid rows
    const double tiles = (double)((M + tile - 1) / tile) * (double)((N + tile - 1) / tile) * (double)batch;
    for (int ks = 1; ks <= (tile == 64 ? 1 : 8); ks *= 2) {
      if (ks > 1 && K < (long)SK * ks) break;
      const double stages = (double)((K + SK - 1) / SK + ks - 1) / ks;
      const double per_sm = std::ceil(tiles * ks / nsm);
      const double fma = per_sm * tile * tile * stages * SK / 2.0;
      const double t = std::max(fma, 700.0 * stages) + (ks > 1 ? 2500.0 + per_sm * tile * tile / 2.0 : 0.0);
      if (best_t == 0.0 || t < best_t) {
        best = Split{tile, ks};
        best_t = t;
      }
    }
  }
  return best;
}

}  // namespace

void dgemm(cudaStream_t st, int transA, int transB, int M, int N, int K, double alpha,
           const double* A, long lda, long strideA, const double* B, long ldb, long strideB,
           double beta, double* C, long ldc, long strideC, int batch, int tri, const int* skip) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  const Split sp = choose_split(M, N, std::max(K, 1), batch);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(((N + sp.tile - 1) / sp.tile) * sp.ks), (unsigned)((M + sp.tile - 1) / sp.tile),
                     (unsigned)batch);
  cfg.blockDim = dim3(NT);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;  // see pdl.cuh
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)sp.ks;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  if (sp.tile == 64) {
    cfg.numAttrs = 1;
    OMM_CUDA_TRY(cudaLaunchKernelEx(&cfg, dgemm_kernel, transA, transB, M, N, K, alpha, A, lda, strideA, B, ldb, strideB,
                                    beta, C, ldc, strideC, tri, skip));
  } else {
    cfg.numAttrs = 2;
    auto kernel = sp.tile == 32 ? dgemm_small_kernel<32> : dgemm_small_kernel<16>;
    OMM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, transA, transB, M, N, K, alpha, A, lda, strideA, B, ldb, strideB, beta,
                                    C, ldc, strideC, tri, skip, sp.ks));
  }
  OMM_LAUNCH_CHECK();
}

}  // namespace omm
