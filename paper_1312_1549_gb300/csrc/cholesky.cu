// Float64 inverse of a symmetric positive definite matrix, for the kinetic
// preconditioner P = (S + T/tau)^-1 (Sec. 2.4, Eq. 17), computed once per
// geometry. Three stages, all on the device:
//   1. blocked right-looking Cholesky A = L L^T (64-column panels; the
//      diagonal block is factored and inverted by one CTA in shared memory,
//      the panel and the trailing update are float64 GEMMs),
//   2. Y = L^-1 by recursive halving: inv([L11 0; L21 L22]) =
//      [Y11 0; -Y22 L21 Y11  Y22], whose base cases are the inverted diagonal
//      blocks of stage 1,
//   3. P = Y^T Y (lower tiles only, K loop from the diagonal), then mirrored.
// A failed pivot (<= 0 or NaN) is recorded in info_dev and replaced by 1 so
// that the remaining stages stay finite; the caller reports the failure.
//
// spd_inverse_sliced computes the same P with float64-class products on the
// BF16 tensor cores (the fixed-point slicing of emu.cu), recursively on
// halves so that every product has a long contraction:
//   chol_inv([A11 A21^T; A21 A22]):  L11, Y11 = chol_inv(A11);
//     L21 = A21 Y11^T;  A22 -= L21 L21^T;  L22, Y22 = chol_inv(A22);
//     Y21 = -Y22 (L21 Y11)                         (Y = L^-1)
//   lauum(Y) = Y^T Y:  P22 = lauum(Y22);  P21 = Y22^T Y21;
//     P11 = lauum(Y11) + Y21^T Y21
// with leaves factored and inverted by one CTA (a second kernel or the same one writes the leaf's block of Y^T Y):
// 64 x 64 in float64 for float64-class results, 128 x 128 in float32 for the preconditioner. The
// P updates of a node run on a second stream as soon as its Y is final, beside the factorisation
// of the blocks that follow. W = L21 Y11 does not need the right half, so it runs on a third stream
// beside that half's factorisation: the chain of a node is three products instead of the four that
// -(Y22 L21) Y11 makes, and neither transposes nor copies. The chain is what bounds the inverse (51 nodes one
// after another at m = 3328): by this alone the float64-class inverse went from 17.9 to 15.7 ms (13.5 with what
// followed), a Cholesky-flavour solve of m = 2944 from 46.4 to 44.3 (43.3). W and Y21 take one slice more than the other products: sliced by columns W loses more than
// Y22 L21 by rows, and the error of P would be up to 30 % larger than in that order; with the extra slice it is
// 5 to 25 % smaller (against a refined inverse, m = 160 to 3328), for 3 % of the time.
#include "emu.cuh"
#include "leaf_f64.cuh"
#include "omm_internal.cuh"
#include "pdl.cuh"
#include "side_streams.cuh"
#include "split_device.cuh"
#include "tc_gemm.cuh"

#include <algorithm>

namespace omm {
namespace {

using dev::kLeaf64Threads;
using dev::NB;  // edge of a float64 leaf

__global__ void __launch_bounds__(kLeaf64Threads)
leaf_f64_kernel(double* A, long lda, int b, double* Linv, long ldi, int* info, int col_offset) {
  dev::pdl_begin();
  dev::leaf_f64_body(A, lda, b, Linv, ldi, info, col_offset);
}

// The Gram block Y^T Y (both triangles) of a leaf's inverse Y (b x b, zero above the diagonal) into Pblk: another
// 44 thousand FMAs, beside the factorisation instead of at the end of each leaf of its chain (20 of a leaf's 100 us;
// by this alone the float64-class inverse of m = 3328, 52 leaves, went from 14.5 to 13.6 ms).
__global__ void __launch_bounds__(kLeaf64Threads)
gram_f64_kernel(int b, const double* Y, long ldy, double* Pblk, long ldp) {
  dev::pdl_begin();
  __shared__ double X[NB][NB + 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kWarps = kLeaf64Threads / 32;
  for (int idx = tid; idx < NB * NB; idx += kLeaf64Threads) {
    const int i = idx / NB, j = idx % NB;
    X[i][j] = i < b && j < b ? Y[(long)i * ldy + j] : 0.0;
  }
  __syncthreads();
  // (X^T X)_ij = sum_{k >= i} X_ki X_kj for j <= i, mirrored: 8 x 8 blocks (I, J <= I), two rows per lane
  const int nb8 = (b + 7) / 8;
  for (int q = warp, I = 0, base = 0; I < nb8; ) {
    if (q >= base + I + 1) { base += I + 1; ++I; continue; }
    const int J = q - base;
    const int i = 8 * I + (lane >> 3), j = 8 * J + (lane & 7);
    double a0 = 0.0, a1 = 0.0;
    for (int k = 8 * I; k < b; ++k) {  // (X is zero above its diagonal)
      const double xj = X[k][j];
      a0 = fma(X[k][i], xj, a0);
      a1 = fma(X[k][i + 4], xj, a1);
    }
    if (i < b && j <= i) {
      Pblk[(long)i * ldp + j] = a0;
      Pblk[(long)j * ldp + i] = a0;
    }
    if (i + 4 < b && j <= i + 4) {
      Pblk[(long)(i + 4) * ldp + j] = a1;
      Pblk[(long)j * ldp + i + 4] = a1;
    }
    q += kWarps;
  }
}

// ---- float32 leaves of edge up to 128 for the preconditioner-grade inverse
constexpr int NL = 128;
constexpr int kLeafThreads = 512;
constexpr int kLeafSmem = (2 * NL * (NL + 1) + NL) * (int)sizeof(float);

// float64 <-> float32 on the integer pipe, so that the leaf's conversions stay off the narrow float64 units
__device__ __forceinline__ float to_f32(double x) { return dev::f32_rne_bits(x); }
__device__ __forceinline__ double to_f64(float v) { return dev::f64_of_f32(v); }

// One CTA: Cholesky factor of the b x b diagonal block at A (b <= 128, read only: the caller
// does not need L itself), its inverse X = L^-1 into Linv (NL x NL, row-major, zero above the
// diagonal) or, with Xhi, as the bf16 pair (Xhi, Xlo) of its b x b elements, and, with Pblk,
// the block X^T X (both triangles) -- all in float32, for the preconditioner, which needs far less
// than float64 accuracy. The layout is leaf_f64_kernel's: panels of eight columns factored in warp
// 0's registers, rank-8 updates on 8 x 8 blocks, the inverse by joining blocks of edge 8 to 64 with
// the contraction cut at the triangles. Bound by shared-memory loads and the panels' dependent chain.
// (With 16-column panels, dense joins and a third shared-memory matrix a leaf took 101 us, now 84.)
__global__ void __launch_bounds__(kLeafThreads)
leaf_f32_kernel(const double* A, long lda, int b, double* Linv, __nv_bfloat16* Xhi, __nv_bfloat16* Xlo, long ldx,
                int* info, int col_offset, double* Pblk, long ldp) {
  dev::pdl_begin();
  extern __shared__ float smf[];
  float (*L)[NL + 1] = reinterpret_cast<float (*)[NL + 1]>(smf);
  float (*X)[NL + 1] = reinterpret_cast<float (*)[NL + 1]>(smf + NL * (NL + 1));
  float* rdiag = smf + 2 * NL * (NL + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kWarps = kLeafThreads / 32;
  static_assert(kWarps == NL / 8, "a warp per diagonal block");
  for (int i = warp; i < NL; i += kWarps)
    for (int j = lane; j < NL; j += 32) {
      L[i][j] = (i < b && j <= i) ? to_f32(A[(long)i * lda + j]) : 0.f;
      X[i][j] = 0.f;
    }
  __syncthreads();
  for (int p0 = 0; p0 < b; p0 += 8) {
    const int pw = min(8, b - p0);
    if (warp == 0) {  // lane l holds rows p0 + l + 32 t
      float r[4][8];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int i = p0 + lane + 32 * t;
#pragma unroll
        for (int c = 0; c < 8; ++c) r[t][c] = (i < b && c < pw && p0 + c <= i) ? L[i][p0 + c] : 0.f;
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c < pw) {
          float d = __shfl_sync(0xffffffffu, r[0][c], c);  // the pivot, row p0 + c
          if (!(d > 0.f)) {
            if (lane == 0) atomicCAS(info, 0, col_offset + p0 + c + 1);
            d = 1.f;
          }
          float rs = rsqrtf(d);
          if (rs > 0.f) rs = fmaf(0.5f * rs, fmaf(-(d * rs), rs, 1.f), rs);  // (0 only for an infinite pivot)
          const float sq = sqrtf(d);
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int i = p0 + lane + 32 * t;
            if (i > p0 + c) r[t][c] *= rs;
            else if (i == p0 + c) r[t][c] = sq;
          }
          if (lane == 0) rdiag[p0 + c] = rs;
#pragma unroll
          for (int l = 0; l < 8; ++l) {
            if (l > c) {
              const float lc = __shfl_sync(0xffffffffu, r[0][c], l);  // L[p0 + l][p0 + c]
              if (lane >= l) r[0][l] = fmaf(-r[0][c], lc, r[0][l]);
#pragma unroll
              for (int t = 1; t < 4; ++t) r[t][l] = fmaf(-r[t][c], lc, r[t][l]);
            }
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int i = p0 + lane + 32 * t;
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (i < b && c < pw && p0 + c <= i) L[i][p0 + c] = r[t][c];
      }
    }
    __syncthreads();
    // trailing lower triangle in 8 x 8 blocks (I, J <= I), a warp per block, two rows per lane
    const int q0 = p0 + 8, nb8 = (b - q0 + 7) / 8;
    for (int q = warp, I = 0, base = 0; I < nb8;) {
      if (q >= base + I + 1) {
        base += I + 1;
        ++I;
        continue;
      }
      const int i = q0 + 8 * I + (lane >> 3), j = q0 + 8 * (q - base) + (lane & 7);
      float a0 = L[i][j], a1 = L[i + 4][j];  // (rows and columns past b hold zeros)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float lj = L[j][p0 + k];
        a0 = fmaf(-L[i][p0 + k], lj, a0);
        a1 = fmaf(-L[i + 4][p0 + k], lj, a1);
      }
      if (j <= i) L[i][j] = a0;
      if (j <= i + 4) L[i + 4][j] = a1;
      q += kWarps;
    }
    __syncthreads();
  }
  // inverses of the 8 x 8 diagonal blocks: warp w's lane c solves column c of block w
  if (8 * warp < b && lane < 8 && 8 * warp + lane < b) {
    const int o = 8 * warp, c = lane, e = min(8, b - o);
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = 0.f;
      if (i == c) x[i] = rdiag[o + i];
      if (i > c && i < e) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k >= c && k < i) acc = fmaf(L[o + i][o + k], x[k], acc);
        x[i] = -acc * rdiag[o + i];
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i >= c && i < e) X[o + i][o + c] = x[i];
  }
  __syncthreads();
  // Join blocks of edge s (see leaf_f64_kernel): T = L21 X11, kept transposed in the upper triangle of L,
  // then X21 = -X22 T; every warp has one unit of four rows (columns) of one pair
  for (int s = 8; s < b; s *= 2) {
    const int wpp = s / 4;  // warps per pair
    const int o = 2 * s * (warp / wpp), f = 4 * (warp % wpp) + (lane >> 3);
    if (o < b) {
      const int i = f;
      for (int g = 0; g < s; g += 8) {
        const int j = g + (lane & 7);
        float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 4
        for (int k = g; k < s; k += 2) {
          acc0 = fmaf(L[o + s + i][o + k], X[o + k][o + j], acc0);
          acc1 = fmaf(L[o + s + i][o + k + 1], X[o + k + 1][o + j], acc1);
        }
        L[o + j][o + s + i] = acc0 + acc1;
      }
    }
    __syncthreads();
    if (o < b) {
      const int j = f;
      for (int g = 0; g < s; g += 8) {
        const int i = g + (lane & 7);
        float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 4
        for (int k = 0; k < g + 8; k += 2) {
          acc0 = fmaf(X[o + s + i][o + s + k], L[o + j][o + s + k], acc0);
          acc1 = fmaf(X[o + s + i][o + s + k + 1], L[o + j][o + s + k + 1], acc1);
        }
        if (o + s + i < b) X[o + s + i][o + j] = -(acc0 + acc1);
      }
    }
    __syncthreads();
  }
  for (int idx = tid; idx < NL * NL; idx += kLeafThreads) {
    const int i = idx / NL, j = idx % NL;
    if (Xhi == nullptr) Linv[idx] = to_f64(X[i][j]);
    else if (i < b && j < b) dev::split_store_f32(X[i][j], Xhi, Xlo, (long)i * ldx + j);
  }
  if (Pblk != nullptr) {
    // (X^T X)_ij = sum_{k >= i} X_ki X_kj for j <= i, mirrored: 8 x 8 blocks (I, J <= I), two rows per lane
    const int nb8 = (b + 7) / 8;
    for (int q = warp, I = 0, base = 0; I < nb8;) {
      if (q >= base + I + 1) {
        base += I + 1;
        ++I;
        continue;
      }
      const int i = 8 * I + (lane >> 3), j = 8 * (q - base) + (lane & 7);
      float a0 = 0.f, a1 = 0.f;
#pragma unroll 4
      for (int k = 8 * I; k < b; ++k) {  // (X is zero above its diagonal)
        const float xj = X[k][j];
        a0 = fmaf(X[k][i], xj, a0);
        a1 = fmaf(X[k][i + 4], xj, a1);
      }
      if (i < b && j <= i) {
        const double v = to_f64(a0);
        Pblk[(long)i * ldp + j] = v;
        Pblk[(long)j * ldp + i] = v;
      }
      if (i + 4 < b && j <= i + 4) {
        const double v = to_f64(a1);
        Pblk[(long)(i + 4) * ldp + j] = v;
        Pblk[(long)j * ldp + i + 4] = v;
      }
      q += kWarps;
    }
  }
}

__global__ void zero_upper_kernel(int m, double* A) {
  const long count = (long)m * m;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < count;
       idx += (long)gridDim.x * blockDim.x) {
    const long i = idx / m, j = idx % m;
    if (j > i) A[idx] = 0.0;
  }
}

__global__ void copy_block_kernel(int rows, int cols, const double* src, long lds, double* dst, long ldd) {
  dev::pdl_begin();
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < rows * cols; idx += gridDim.x * blockDim.x) {
    const int i = idx / cols, j = idx % cols;
    dst[(long)i * ldd + j] = src[(long)i * lds + j];
  }
}
void copy_block(cudaStream_t st, int rows, int cols, const double* src, long lds, double* dst, long ldd) {
  const int blocks = std::max(1, std::min((rows * cols + 255) / 256, 608));
  launch_pdl(st, dim3(blocks), dim3(256), 0, copy_block_kernel, rows, cols, src, lds, dst, ldd);
  OMM_LAUNCH_CHECK();
}

struct Work {
  double* Dinv;  // nblk x NB x NB diagonal-block inverses
  double* tmp;   // up to m*m/4 (+ panel) scratch
};

// Y[r0:r1, r0:r1] (lower, in place) <- its inverse
void trtri_rec(cudaStream_t st, int m, double* Y, const Work& w, int r0, int r1) {
  const int nb_blocks = (r1 - r0 + NB - 1) / NB;
  if (nb_blocks <= 1) {
    const int b = r1 - r0;
    copy_block(st, b, b, w.Dinv + (long)(r0 / NB) * NB * NB, NB, Y + (long)r0 * m + r0, m);
    return;
  }
  const int mid = r0 + (nb_blocks / 2) * NB;
  trtri_rec(st, m, Y, w, r0, mid);
  trtri_rec(st, m, Y, w, mid, r1);
  const int n1 = mid - r0, n2 = r1 - mid;
  double* L21 = Y + (long)mid * m + r0;
  const double* Y11 = Y + (long)r0 * m + r0;
  const double* Y22 = Y + (long)mid * m + mid;
  // W = L21 * Y11  (n2 x n1); Y11 is lower triangular
  dgemm(st, 0, 0, n2, n1, n1, 1.0, L21, m, 0, Y11, m, 0, 0.0, w.tmp, n1, 0, 1, kTriKFromCol);
  // Y21 = -Y22 * W; Y22 is lower triangular
  dgemm(st, 0, 0, n2, n1, n2, -1.0, Y22, m, 0, w.tmp, n1, 0, 0.0, L21, m, 0, 1, kTriKToRow);
}

}  // namespace

size_t spd_inverse_workspace(int m) {
  const long nblk = (m + NB - 1) / NB;
  const long half = (m + 1) / 2 + NB;
  return (size_t)(nblk * NB * NB) + (size_t)(half * half) + (size_t)m * NB;
}

namespace {
// stage 1: A = L L^T in place (lower triangle; the upper one is zeroed)
void factor_blocked(cudaStream_t st, int m, double* A, const Work& w, int* info_dev) {
  const int nblk = (m + NB - 1) / NB;
  OMM_CUDA_TRY(cudaMemsetAsync(info_dev, 0, sizeof(int), st));
  for (int kb = 0; kb < nblk; ++kb) {
    const int k = kb * NB;
    const int b = (m - k < NB) ? (m - k) : NB;
    double* Akk = A + (long)k * m + k;
    launch_pdl(st, dim3(1), dim3(kLeaf64Threads), 0, leaf_f64_kernel, Akk, m, b, w.Dinv + (long)kb * NB * NB, NB, info_dev,
               k);
    OMM_LAUNCH_CHECK();
    const int r = m - k - b;
    if (r > 0) {
      double* A21 = A + (long)(k + b) * m + k;
      // L21 = A21 * Linv^T (to scratch, then back)
      dgemm(st, 0, 1, r, b, b, 1.0, A21, m, 0, w.Dinv + (long)kb * NB * NB, NB, 0, 0.0, w.tmp, b, 0);
      copy_block(st, r, b, w.tmp, b, A21, m);
      // A22 -= L21 L21^T (lower tiles)
      double* A22 = A + (long)(k + b) * m + (k + b);
      dgemm(st, 0, 1, r, r, b, -1.0, A21, m, 0, A21, m, 0, 1.0, A22, m, 0, 1, kTriLower);
    }
  }
  zero_upper_kernel<<<1024, 256, 0, st>>>(m, A);
  OMM_LAUNCH_CHECK();
}
}  // namespace

void spd_inverse(cudaStream_t st, int m, double* A, double* P, double* work, int* info_dev) {
  const int nblk = (m + NB - 1) / NB;
  Work w{work, work + (long)nblk * NB * NB};
  // 1. Cholesky
  factor_blocked(st, m, A, w, info_dev);
  // 2. Y = L^-1 in place
  trtri_rec(st, m, A, w, 0, m);
  // 3. P = Y^T Y (lower), mirrored
  dgemm(st, 1, 0, m, m, m, 1.0, A, m, 0, A, m, 0, 0.0, P, m, 0, 1, kTriLower | kTriKStart);
  launch_symmetrize_lower(st, m, P);
}

void spd_factor_inverse(cudaStream_t st, int m, double* A, double* Y, double* work, int* info_dev) {
  const int nblk = (m + NB - 1) / NB;
  Work w{work, work + (long)nblk * NB * NB};
  factor_blocked(st, m, A, w, info_dev);
  OMM_CUDA_TRY(cudaMemcpyAsync(Y, A, sizeof(double) * m * (size_t)m, cudaMemcpyDeviceToDevice, st));
  trtri_rec(st, m, Y, w, 0, m);
}

// ------------------------------------------------------------------ float64-class (sliced) variant
namespace {

constexpr int kInvSlices = 10;  // the most slices of a lane's products; W and Y21 take one more

long round_up(long x, long unit) { return (x + unit - 1) / unit * unit; }
long round8(long x) { return round_up(x, 8); }

// scratch of one stream's products
struct Lane {
  cudaStream_t st = nullptr;
  int slices = kInvSlices;   // fixed-point slices of every product on this lane
  double* tr0 = nullptr;     // float64 transposes
  double* tr1 = nullptr;
  __nv_bfloat16* sl0 = nullptr;  // slices of two operands
  __nv_bfloat16* sl1 = nullptr;
  double* slab = nullptr;     // float64 sums of the sliced products
};

struct SlicedWork : Streams {
  int m = 0;
  int nb = NB;               // leaf edge: 64 (float64 leaves) or 128 (float32 leaves)
  double* A = nullptr;       // the matrix, factor L in its lower triangle; blocks above the diagonal take W^T
  double* Y = nullptr;       // L^-1 (lower triangle, zero above)
  double* P = nullptr;
  double* leaf = nullptr;    // nb x nb inverse of a diagonal block
  int* info = nullptr;
  int* err = nullptr;
  // factorisation and inverse on `main`; the P = Y^T Y updates on `side`; the products W on `ahead`
  Lane main, side, ahead;
};

// C (M x N, ldc) = alpha A B^T + beta C with A (M x K, lda) and B (N x K, ldb) row-major;
// the slices of A go to sl0, those of B to sl1 (or B = A: one slicing, both maps); `more` slices than the lane's
void sliced_nt(Lane& L, int* err, int M, int N, int K, double alpha, const double* A, long lda, const double* B,
               long ldb, double beta, double* C, long ldc, int more = 0) {
  const long ld = round8(K);
  const int s = L.slices + more;
  emu::slice_rows(L.st, A, M, K, lda, s, L.sl0, ld, nullptr);
  const tc::Operand oa = tc::make_operand(L.sl0, M, K, ld, s, true);
  tc::Operand ob;
  if (B == A && ldb == lda && N == M) {
    ob = tc::make_operand(L.sl0, N, K, ld, s, false);
  } else {
    emu::slice_rows(L.st, B, N, K, ldb, s, L.sl1, ld, nullptr);
    ob = tc::make_operand(L.sl1, N, K, ld, s, false);
  }
  emu::gemm(L.st, oa, ob, K, s, tc::Epilogue{C, ldc, N, 0, alpha, beta, M, N, nullptr, err}, L.slab);
}

// leaf: factor A[r0:r0+b, r0:r0+b] in place, write its inverse into Y and Y_leaf^T Y_leaf into P
void leaf(SlicedWork& w, int r0, int b) {
  const long m = w.m;
  double* y = w.Y + r0 * m + r0;
  double* pb = w.P ? w.P + r0 * m + r0 : nullptr;
  if (w.nb == NL) {  // a preconditioner: 128-wide float32 leaves (see leaf_f32_kernel)
    launch_pdl(w.main.st, dim3(1), dim3(kLeafThreads), kLeafSmem, leaf_f32_kernel, w.A + r0 * m + r0, m, b, w.leaf,
               nullptr, nullptr, 0, w.info, r0, pb, m);
    OMM_LAUNCH_CHECK();
    copy_block(w.main.st, b, b, w.leaf, w.nb, y, m);
    return;
  }
  launch_pdl(w.main.st, dim3(1), dim3(kLeaf64Threads), 0, leaf_f64_kernel, w.A + r0 * m + r0, m, b, y, m, w.info, r0);
  OMM_LAUNCH_CHECK();
  if (pb == nullptr) return;
  w.wait(w.side.st, w.main.st);
  launch_pdl(w.side.st, dim3(1), dim3(kLeaf64Threads), 0, gram_f64_kernel, b, y, m, pb, m);
  OMM_LAUNCH_CHECK();
}

int half_of(int b, int nb) { return ((b / nb + 1) / 2) * nb; }  // a multiple of nb, about b / 2

// P21 = Y22^T Y21 and P11 += Y21^T Y21 of one node (its Y is final), on the side lane
void p_update(SlicedWork& w, int r0, int b1, int b2) {
  const long m = w.m;
  const int r1 = r0 + b1;
  Lane& L = w.side;
  const double* Y21 = w.Y + (long)r1 * m + r0;
  const double* Y22 = w.Y + (long)r1 * m + r1;
  // Y21^T (b1 x b2) serves both products
  emu::transpose(L.st, Y21, b2, b1, m, L.tr0, b2);
  // P21 = Y22^T Y21: A operand Y22^T (b2 x b2), B operand Y21^T
  emu::transpose(L.st, Y22, b2, b2, m, L.tr1, b2);
  sliced_nt(L, w.err, b2, b1, b2, 1.0, L.tr1, b2, L.tr0, b2, 0.0, w.P + (long)r1 * m + r0, m);
  // P11 = Y11^T Y11 (the updates of the left subtree, already queued on this lane) + Y21^T Y21
  sliced_nt(L, w.err, b1, b1, b2, 1.0, L.tr0, b2, L.tr0, b2, 1.0, w.P + (long)r0 * m + r0, m);
}

// Y and L of the block [r0, r0 + b) on the main lane; once a node's Y is final its contribution
// to P = Y^T Y is queued on the side lane, in post-order, so it runs beside the factorisation
// of the blocks that follow
void chol_inv(SlicedWork& w, int r0, int b) {
  if (b <= w.nb) {
    leaf(w, r0, b);
    return;
  }
  const long m = w.m;
  Lane& L = w.main;
  const int b1 = half_of(b, w.nb), b2 = b - b1, r1 = r0 + b1;
  chol_inv(w, r0, b1);
  double* A21 = w.A + (long)r1 * m + r0;
  double* A22 = w.A + (long)r1 * m + r1;
  double* A12 = w.A + (long)r0 * m + r1;
  const double* Y11 = w.Y + (long)r0 * m + r0;
  const double* Y22 = w.Y + (long)r1 * m + r1;
  double* Y21 = w.Y + (long)r1 * m + r0;
  // L21 = A21 Y11^T, over A21 (the product reads slices)
  sliced_nt(L, w.err, b2, b1, b1, 1.0, A21, m, Y11, m, 0.0, A21, m);
  if (w.ahead.st != L.st) w.wait(w.ahead.st, L.st);
  // W^T = Y11^T L21^T, over A12, which nothing reads (Y11^T: b1 x b1)
  emu::transpose(w.ahead.st, Y11, b1, b1, m, w.ahead.tr0, b1);
  sliced_nt(w.ahead, w.err, b1, b2, b1, 1.0, w.ahead.tr0, b1, A21, m, 0.0, A12, m, 1);
  const cudaEvent_t done = w.ahead.st != L.st ? w.record(w.ahead.st) : nullptr;
  // A22 -= L21 L21^T
  sliced_nt(L, w.err, b2, b2, b1, -1.0, A21, m, A21, m, 1.0, A22, m);
  chol_inv(w, r1, b2);
  // Y21 = -Y22 W
  if (done != nullptr) OMM_CUDA_TRY(cudaStreamWaitEvent(L.st, done, 0));
  sliced_nt(L, w.err, b2, b1, b2, -1.0, Y22, m, A12, m, 0.0, Y21, m, 1);
  if (w.P == nullptr) return;  // the factor and its inverse only
  // this node's Y is final: its P updates may start
  w.wait(w.side.st, L.st);
  p_update(w, r0, b1, b2);
}

// ------------------------------------------------------------------ preconditioner grade (3-term bf16 split)
// The same recursion with every operand kept as a bf16 pair in an m x m matrix of its own: A (the part still
// to be factored), L and Y = L^-1. The products read blocks of these matrices where they stand -- transposed
// factors as MN-major operands -- and their epilogues write the split of the result beside or instead of
// the float64 one, so a node of the recursion is four products on the main stream and two beside it,
// with no operand to split, transpose or copy (that was fourteen launches on the main stream, on a
// chain that runs node after node). Only A and P exist in float64: the leaves and the updates of A read A,
// P is the result.
struct SplitInverse : Streams {
  int m = 0;
  long ld = 0;
  // rows between the hi and the lo half of a pair: a product that contracts over rows of both operands (Y^T Y)
  // runs on to the end of a 64-row block, where zero rows have to follow row m
  long half = 0;
  double* A = nullptr;
  double* P = nullptr;
  __nv_bfloat16 *As = nullptr, *Ls = nullptr, *Ys = nullptr;  // [hi; lo], 2 half x ld each
  int* info = nullptr;
  int* err = nullptr;
  cudaStream_t st = nullptr, side = nullptr;

  enum Role { kA, kB };
  // block (r0, c0) as an operand: rows x cols with cols contracted, or (mn) rows contracted
  tc::Operand view(const __nv_bfloat16* x, int r0, int c0, int rows, int cols, Role role, bool mn) const {
    return tc::make_operand_view(x + r0 * ld + c0, half, cols, ld, 2, role == kA, 0, rows, mn, 2L * half - r0);
  }
  // the split of an M x N product into block (r0, c0) of x, alpha times it
  tc::Epilogue into(__nv_bfloat16* x, int r0, int c0, int M, int N, double alpha) const {
    tc::Epilogue ep{nullptr, 0, N, 0, alpha, 0.0, M, N, nullptr, err};
    ep.c_f32 = 1;
    ep.bf_hi = x + r0 * ld + c0;
    ep.bf_ld = ld;
    ep.bf_lo = half * ld;
    return ep;
  }

  void node(int r0, int b) {
    if (b <= NL) {
      __nv_bfloat16* y = Ys + r0 * ld + r0;
      const long at = (long)r0 * m + r0;
      launch_pdl(st, dim3(1), dim3(kLeafThreads), kLeafSmem, leaf_f32_kernel, A + at, m, b, nullptr, y, y + half * ld, ld, info,
                 r0, P + at, m);
      OMM_LAUNCH_CHECK();
      return;
    }
    const int b1 = half_of(b, NL), b2 = b - b1, r1 = r0 + b1;
    node(r0, b1);
    // L21 = A21 Y11^T
    emu::gemm_split(st, view(As, r1, r0, b2, b1, kA, false), view(Ys, r0, r0, b1, b1, kB, false), b1,
                    into(Ls, r1, r0, b2, b1, 1.0));
    // A22 -= L21 L21^T
    tc::Epilogue ea = into(As, r1, r1, b2, b2, -1.0);
    ea.C = A + (long)r1 * m + r1;
    ea.ldc = m;
    ea.c_f32 = 0;
    ea.beta = 1.0;
    emu::gemm_split(st, view(Ls, r1, r0, b2, b1, kA, false), view(Ls, r1, r0, b2, b1, kB, false), b1, ea);
    node(r1, b2);
    // Z = Y22 L21, in the place of A21
    emu::gemm_split(st, view(Ys, r1, r1, b2, b2, kA, false), view(Ls, r1, r0, b2, b1, kB, true), b2,
                    into(As, r1, r0, b2, b1, 1.0));
    // Y21 = -Z Y11
    emu::gemm_split(st, view(As, r1, r0, b2, b1, kA, false), view(Ys, r0, r0, b1, b1, kB, true), b1,
                    into(Ys, r1, r0, b2, b1, -1.0));
    // this node's Y is final: its part of P = Y^T Y, beside the factorisation of the blocks that follow
    wait(side, st);
    const tc::Operand y21 = view(Ys, r1, r0, b2, b1, kB, true);
    // P21 = Y22^T Y21; P11 += Y21^T Y21
    emu::gemm_split(side, view(Ys, r1, r1, b2, b2, kA, true), y21, b2,
                    tc::Epilogue{P + (long)r1 * m + r0, m, b1, 0, 1.0, 0.0, b2, b1, nullptr, err});
    emu::gemm_split(side, view(Ys, r1, r0, b2, b1, kA, true), y21, b2,
                    tc::Epilogue{P + (long)r0 * m + r0, m, b1, 0, 1.0, 1.0, b1, b1, nullptr, err});
  }
};

void prepare_leaf() {
  static const cudaError_t e =  // thread-safe, once
      cudaFuncSetAttribute(leaf_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLeafSmem);
  OMM_CUDA_TRY(e);
}

// Scratch of the split form from `base`, or its size alone.
size_t carve(SplitInverse& w, int m, void* base) {
  w.m = m;
  w.ld = round8(m);
  w.half = round_up(m, 64);
  const size_t pair = 2 * (size_t)w.half * w.ld;
  w.Ys = reinterpret_cast<__nv_bfloat16*>(round_up((long)reinterpret_cast<uintptr_t>(base), 256));
  w.Ls = w.Ys + pair;
  w.As = w.Ls + pair;
  return 3 * pair * sizeof(__nv_bfloat16) + 256;
}

// Scratch of the sliced form from `base`, or its size alone. `Y`: L^-1 is not the caller's; `side`: P is wanted;
// `ahead`: a lane of its own for the products W, which otherwise take the main lane's room and stream.
size_t carve(SlicedWork& w, int m, int slices, bool Y, bool side, bool ahead, void* base) {
  const long h = (m + 1) / 2 + NL;  // the largest off-diagonal block edge (either leaf size)
  uintptr_t p = reinterpret_cast<uintptr_t>(base);
  auto take = [&](size_t bytes) {
    void* at = reinterpret_cast<void*>(p = (p + 255) & ~uintptr_t(255));
    p += bytes;
    return at;
  };
  auto f64 = [&](size_t count) { return static_cast<double*>(take(count * sizeof(double))); };
  auto lane = [&](Lane& L, int most) {
    L.slices = slices;
    L.slab = f64(tc::sliced_workspace_doubles());
    for (__nv_bfloat16** sl : {&L.sl0, &L.sl1})
      *sl = static_cast<__nv_bfloat16*>(take((size_t)most * h * round8(h) * sizeof(__nv_bfloat16)));
  };
  w.m = m;
  if (Y) w.Y = f64((size_t)m * m);
  w.leaf = f64(NL * NL);
  lane(w.main, slices + 1);  // W and Y21 take one slice more
  if (side) {
    lane(w.side, slices);
    w.side.tr0 = f64((size_t)h * h);
    w.side.tr1 = f64((size_t)h * h);
  }
  if (ahead) lane(w.ahead, slices + 1);
  else w.ahead = w.main;
  w.ahead.tr0 = f64((size_t)h * h);
  return p - reinterpret_cast<uintptr_t>(base) + 256;
}

int slices_of(int slices) { return std::min(std::max(slices, 2), kInvSlices); }

// P = A^-1 in the 3-term split form
void split_impl(cudaStream_t st, int m, double* A, double* P, void* work, int* info_dev, int* err_dev) {
  SplitInverse w;
  carve(w, m, work);
  w.A = A;
  w.P = P;
  w.info = info_dev;
  w.err = err_dev;
  w.st = st;
  prepare_leaf();
  OMM_CUDA_TRY(cudaMemsetAsync(info_dev, 0, sizeof(int), st));
  // zeros above the diagonal of Y and past row m; and every element that a contraction over rows of Y or L may
  // touch past the end of a block has to be a number (it meets zeros of the other operand)
  OMM_CUDA_TRY(cudaMemsetAsync(w.Ys, 0, (w.As - w.Ys) * sizeof(__nv_bfloat16), st));
  OMM_CUDA_TRY(cudaMemsetAsync(P, 0, sizeof(double) * m * (size_t)m, st));
  tc::split(st, A, m, m, m, w.As, w.As + w.half * w.ld, w.ld, nullptr);
  w.side = w.fork(st);
  w.node(0, m);
  w.join(st);
  launch_symmetrize_lower(st, m, P);
}

// P = A^-1 (P != nullptr) and/or L, Y = L^-1 (Y_out != nullptr: A keeps L, zero above the diagonal)
void sliced_impl(cudaStream_t st, int m, double* A, double* P, double* Y_out, void* work, int* info_dev,
                 int* err_dev, int slices, bool ahead) {
  SlicedWork w;
  // preconditioner grade: 128-wide float32 leaves; float64-class: 64-wide float64 leaves
  w.nb = slices < kInvSlices ? NL : NB;
  carve(w, m, slices_of(slices), Y_out == nullptr, P != nullptr, ahead, work);
  if (Y_out) w.Y = Y_out;
  w.A = A;
  w.P = P;
  w.info = info_dev;
  w.err = err_dev;
  w.main.st = st;
  if (w.nb == NL) prepare_leaf();
  OMM_CUDA_TRY(cudaMemsetAsync(info_dev, 0, sizeof(int), st));
  OMM_CUDA_TRY(cudaMemsetAsync(w.Y, 0, sizeof(double) * m * (size_t)m, st));
  if (P) {
    OMM_CUDA_TRY(cudaMemsetAsync(P, 0, sizeof(double) * m * (size_t)m, st));
    w.side.st = w.fork(st);
  }
  w.ahead.st = ahead ? w.fork(st) : st;
  chol_inv(w, 0, m);
  w.join(st);
  if (P) launch_symmetrize_lower(st, m, P);
  if (Y_out) {
    zero_upper_kernel<<<1024, 256, 0, st>>>(m, A);
    OMM_LAUNCH_CHECK();
  }
}

}  // namespace

size_t spd_inverse_sliced_workspace_bytes(int m, int slices, bool ahead) {
  if (slices == 1) {
    SplitInverse w;
    return carve(w, m, nullptr);
  }
  SlicedWork w;
  return carve(w, m, slices_of(slices), true, true, ahead, nullptr);
}

size_t spd_factor_inverse_sliced_workspace_bytes(int m) {
  SlicedWork w;
  return carve(w, m, kInvSlices, false, false, true, nullptr);
}

void spd_inverse_sliced(cudaStream_t st, int m, double* A, double* P, void* work, int* info_dev, int* err_dev,
                        int slices, bool ahead) {
  if (slices == 1) split_impl(st, m, A, P, work, info_dev, err_dev);
  else sliced_impl(st, m, A, P, nullptr, work, info_dev, err_dev, slices, ahead);
}

void spd_factor_inverse_sliced(cudaStream_t st, int m, double* A, double* Y, void* work, int* info_dev,
                               int* err_dev) {
  sliced_impl(st, m, A, nullptr, Y, work, info_dev, err_dev, kInvSlices, true);
}

}  // namespace omm
