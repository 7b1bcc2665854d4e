// Float64-class contractions on the BF16 tensor cores by error-free
// fixed-point slicing (the Ozaki scheme: K. Ozaki, T. Ogita, S. Oishi,
// S. M. Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication and its applications", Numerical
// Algorithms 59 (2012)), used by the mixed path to refresh its state.
//
// Slicing: every row r of an operand gets a power of two sigma_r > 2 max|x|
// over the row, and x = sigma_r * sum_i a_i 2^-5(i+1) + O(sigma_r 2^-5s) with
// integers |a_i| <= 16 (bf16 holds a_i * 2^k exactly). For a pair of slices
// (i, j) every product a b <= 256 units of 2^(e_r + f_c - 5(i+j+2)), so all
// products of one level d = i + j share one unit per output element and a
// level of (d+1) pairs summed over K stays an integer below (d+1) K 256
// units: exact in the FP32 accumulator while that is <= 2^24. The pairs are
// therefore summed in chunks that keep this bound in units of the chunk's
// smallest level (level_chunks: 11 chunks for the Si512 contraction K = 6656,
// 5 for K = 64), so every chunk is exact, and the float64 epilogue adds the
// chunks. (Levels lumped beyond that bound are not exact: the tensor cores'
// FP32 adder truncates, and those errors grow linearly with K -- measured
// 1e-10 of |A||B| at K = 1000 with all levels in one accumulator.) With s = 10
// slices the result carries about 50 bits of each row-scaled operand.
#include "emu.cuh"
#include "pdl.cuh"
#include "tc_gemm.cuh"

#include <algorithm>
#include <new>

namespace omm {
namespace {

constexpr int kSliceBits = 5;

__device__ __forceinline__ bool stopped(const Scalars* sc) { return sc != nullptr && (sc->done | sc->halt); }

// TPR threads per row, four neighbouring columns per thread and step. The row scale sigma = 2^esig
// comes from the largest magnitude (compared as integer bit patterns). Each element becomes the
// integer N = rint(x 2^(5s - esig)) (|N| < 2^(5s-1)), whose balanced base-32 digits
// a_{s-1}, ..., a_0 in [-16, 16] give x = sigma sum_i a_i 2^-5(i+1) + r, |r| <= sigma 2^-(5s+1).
// Slice i holds a_i 2^(esig - 5(i+1)), exact in bf16 (at most 5 significant bits).
// Bound by memory (8 bytes in, 2s out per element) once nothing runs on the float64 pipe (two
// lanes per SM and clock) and the stores are wide: N is the significand shifted and rounded to
// nearest even as an integer; with 16 added to every lower digit, the balanced digits are plain
// 5-bit fields of N; a digit becomes its slice value by one float32 FMA on 2^23 + digit. Rows of up
// to 4 CH TPR columns stay in registers between the maximum and the digits; longer ones are read
// twice. (With one warp per row, a 2-byte store per slice and float64 conversions the 51 million
// elements of a 1024 x 6656 x 6656 product took 1.3 ms, 1.1 TB/s; 0.42 ms, 3.4 TB/s now.)
template <int TPR, int CH>
__global__ void __launch_bounds__(TPR < 256 ? 256 : TPR)
slice_rows_kernel(const double* __restrict__ src, long rows, long cols, long ld_src, int s,
                  __nv_bfloat16* __restrict__ dst, long ld_dst, long slice_stride, const Scalars* sc) {
  dev::pdl_begin();
  constexpr int THREADS = TPR < 256 ? 256 : TPR, RPB = THREADS / TPR, WPR = TPR / 32;
  if (stopped(sc)) return;
  const int sub = threadIdx.x / TPR, t = threadIdx.x % TPR;
  const long row = (long)blockIdx.x * RPB + sub;
  const bool active = row < rows;
  const double* x = src + (active ? row : 0) * ld_src;
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  auto load4 = [&](long c, unsigned long long (&u)[4]) {
    if (vec && c + 3 < cols) {
      const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(x + c), b = *reinterpret_cast<const ulonglong2*>(x + c + 2);
      u[0] = a.x; u[1] = a.y; u[2] = b.x; u[3] = b.y;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) u[k] = c + k < cols ? (unsigned long long)__double_as_longlong(x[c + k]) : 0ull;
    }
  };
  constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFull;
  unsigned long long v[CH][4];
  unsigned long long mx = 0;  // |x| as bits: ordered like the magnitudes (finite values)
  if (active) {
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      const long c = 4L * (t + h * TPR);
      if (c < cols) {
        load4(c, v[h]);
#pragma unroll
        for (int k = 0; k < 4; ++k) mx = max(mx, v[h][k] & kAbs);
      }
    }
    for (long c = 4L * (t + CH * TPR); c < cols; c += 4L * TPR) {
      unsigned long long u[4];
      load4(c, u);
#pragma unroll
      for (int k = 0; k < 4; ++k) mx = max(mx, u[k] & kAbs);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (WPR > 1) {
    __shared__ unsigned long long sh[THREADS / 32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WPR; ++w) mx = max(mx, sh[sub * WPR + w]);
  }
  if (!active) return;
  int e = 0;  // max|x| < 2^e (frexp convention; 0 for an all-zero row)
  const int ebits = (int)(mx >> 52);
  if (ebits > 0) e = ebits - 1022;
  else if (mx != 0) frexp(__longlong_as_double((long long)mx), &e);  // subnormal maximum
  const int esig = e + 1;  // sigma = 2^esig > 2 max|x|
  __nv_bfloat16* out = dst + row * ld_dst;
  const bool plain = esig <= 100 && esig - kSliceBits * s >= -125;  // every slice unit times 2^24 is a normal float32
  // 16 for every digit below the top one, in its place
  const unsigned long long bias = s > 1 ? 16ull * (((1ull << (kSliceBits * (s - 1))) - 1) / 31) : 0ull;
  auto emit = [&](long c, const unsigned long long (&u)[4]) {
    long long N[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned long long mag = u[k] & kAbs;
      const int eb = (int)(mag >> 52);
      const unsigned long long M = (mag & 0x000FFFFFFFFFFFFFull) | (eb ? 1ull << 52 : 0ull);
      const int shift = esig + 1075 - kSliceBits * s - (eb ? eb : 1);  // x 2^(5s - esig) = M 2^-shift
      unsigned long long q = 0;
      if (shift <= 0) q = M << -shift;  // (rows whose maximum is subnormal)
      else if (shift < 64) q = (M + ((1ull << (shift - 1)) - 1) + ((M >> shift) & 1ull)) >> shift;
      N[k] = (long long)((u[k] >> 63) ? 0ull - q : q) + (long long)bias;
    }
    for (int i = 0; i < s; ++i) {
      const int at = kSliceBits * (s - 1 - i);
      unsigned short h[4];
      if (plain) {
        const float unit = __uint_as_float((unsigned)(esig - kSliceBits * (i + 1) + 127) << 23);
        const int off = i > 0 ? 16 : 0;
        const float base = -(12582912.f + (float)off) * unit;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int field = i > 0 ? (int)((unsigned long long)N[k] >> at) & 31 : (int)(N[k] >> at);
          const float f = fmaf(__uint_as_float(0x4B400000u + (unsigned)field), unit, base);  // exact
          h[k] = (unsigned short)(__float_as_uint(f) >> 16);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int a = i > 0 ? ((int)((unsigned long long)N[k] >> at) & 31) - 16 : (int)(N[k] >> at);
          h[k] = __bfloat16_as_ushort(__float2bfloat16_rn(ldexpf((float)a, esig - kSliceBits * (i + 1))));
        }
      }
      __nv_bfloat16* o = out + i * slice_stride + c;
      // (ld_dst is a multiple of 8; columns past cols up to the next multiple of 4 are zeros)
      *reinterpret_cast<uint2*>(o) = make_uint2(h[0] | ((unsigned)h[1] << 16), h[2] | ((unsigned)h[3] << 16));
    }
  };
#pragma unroll
  for (int h = 0; h < CH; ++h) {
    const long c = 4L * (t + h * TPR);
    if (c < cols) emit(c, v[h]);
  }
  for (long c = 4L * (t + CH * TPR); c < cols; c += 4L * TPR) {
    unsigned long long u[4];
    load4(c, u);
    emit(c, u);
  }
}

// dst (cols x rows) = src^T, 32 x 32 shared-memory tiles
__global__ void transpose_kernel(const double* __restrict__ src, long rows, long cols, long ld_src,
                                 double* __restrict__ dst, long ld_dst) {
  dev::pdl_begin();
  __shared__ double tile[32][33];
  const long tiles_c = (cols + 31) / 32;
  const long r0 = (blockIdx.x / tiles_c) * 32, c0 = (blockIdx.x % tiles_c) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int k = ty; k < 32; k += 8) {
    const long r = r0 + k, c = c0 + tx;
    tile[k][tx] = (r < rows && c < cols) ? src[r * ld_src + c] : 0.0;
  }
  __syncthreads();
  for (int k = ty; k < 32; k += 8) {
    const long c = c0 + k, r = r0 + tx;
    if (c < cols && r < rows) dst[c * ld_dst + r] = tile[tx][k];
  }
}

long round8(long x) { return (x + 7) / 8 * 8; }

template <typename T>
void alloc(T** p, size_t count, cudaStream_t st) {
  mem::alloc(p, count, st);
}

}  // namespace

namespace emu {

void slice_rows(cudaStream_t st, const double* src, long rows, long cols, long ld_src, int s,
                __nv_bfloat16* dst, long ld_dst, const Scalars* sc) {
  if (rows <= 0) return;
  auto go = [&](auto kernel, int threads, int rows_per_block) {
    launch_pdl(st, dim3((unsigned)((rows + rows_per_block - 1) / rows_per_block)), dim3(threads), 0, kernel, src, rows,
               cols, ld_src, s, dst, ld_dst, rows * ld_dst, sc);
    OMM_LAUNCH_CHECK();
  };
  // a row's threads: as few as hold it in registers (4 CH TPR columns), so that short rows fill whole warps
  if (cols <= 128) go(slice_rows_kernel<32, 1>, 256, 8);
  else if (cols <= 512) go(slice_rows_kernel<32, 4>, 256, 8);
  else if (cols <= 2048) go(slice_rows_kernel<128, 4>, 256, 2);
  else go(slice_rows_kernel<256, 8>, 256, 1);
}

void transpose(cudaStream_t st, const double* src, long rows, long cols, long ld_src, double* dst, long ld_dst) {
  const long blocks = ((rows + 31) / 32) * ((cols + 31) / 32);
  launch_pdl(st, dim3((unsigned)blocks), dim3(256), 0, transpose_kernel, src, rows, cols, ld_src, dst, ld_dst);
  OMM_LAUNCH_CHECK();
}

tc::PairList level_chunks(int K, int s) {
  // A chunk's FP32 sum is exact while its magnitudes, in units of its smallest level, stay within
  // 2^24: a product of the level d adds 256 K units of its own level, 32 times as many for every
  // level below it that the chunk holds. The pairs are taken level by level, smallest first, into as
  // few chunks as that allows (5 for K = 64, 11 for K = 6656); the float64 epilogue adds the chunks.
  const long budget = std::max(1L, (1L << 24) / (256L * (K > 0 ? K : 1)));
  tc::PairList pl{};
  long used = 0;
  int bottom = -1;  // the smallest level of the open chunk
  auto close = [&]() {
    if (bottom < 0) return;
    if (pl.nchunk == tc::kMaxChunks) throw CudaError{cudaErrorInvalidValue, "emu: too many chunks"};
    pl.chunk_end[pl.nchunk++] = (unsigned char)pl.n;
    bottom = -1;
    used = 0;
  };
  for (int d = s - 1; d >= 0; --d) {
    for (int i = 0; i <= d; ++i) {
      long cost = bottom < 0 ? 1 : (bottom - d > 6 ? budget + 1 : 1L << (kSliceBits * (bottom - d)));
      if (bottom >= 0 && used + cost > budget) {
        close();
        cost = 1;
      }
      if (bottom < 0) bottom = d;
      if (pl.n == tc::kMaxPairs) throw CudaError{cudaErrorInvalidValue, "emu: too many slice pairs"};
      pl.a[pl.n] = (unsigned char)i;
      pl.b[pl.n] = (unsigned char)(d - i);
      ++pl.n;
      used += cost;
    }
  }
  close();
  return pl;
}

namespace {
thread_local Profiler* t_prof = nullptr;
}

void set_profiler(Profiler* p) { t_prof = p; }

void gemm(cudaStream_t st, const tc::Operand& A, const tc::Operand& B, int K, int s, const tc::Epilogue& ep,
          double* slab, const tc::BlockLists* sparse) {
  const tc::PairList pl = level_chunks(K, s);
  if (t_prof) t_prof->begin(st);
  tc::gemm_sliced(st, A, B, K, pl, ep, slab, sparse);
  // issued tensor flops (only the visited K blocks of a block-sparse product)
  if (t_prof) t_prof->end(st, 2.0 * ep.M * (double)ep.N * K * pl.n * tc::block_density(sparse));
}

void gemm_split(cudaStream_t st, const tc::Operand& A, const tc::Operand& B, int K, const tc::Epilogue& ep) {
  if (t_prof) t_prof->begin(st);
  tc::gemm_split(st, A, B, K, ep);
  if (t_prof) t_prof->end(st, 2.0 * ep.M * (double)ep.N * K * 3.0);
}

}  // namespace emu

struct EmuState {
  int m = 0, n = 0, s = 0;
  long ldm = 0, ld2n = 0;
  __nv_bfloat16* HSs = nullptr;  // s slices of [H~; S]     2m x m
  __nv_bfloat16* Cs = nullptr;   // s slices of C           n x m
  __nv_bfloat16* Ys = nullptr;   // s slices of [HC; SC]    2n x m
  __nv_bfloat16* Ws = nullptr;   // s slices of [S_W | H_W] n x 2n
  __nv_bfloat16* YTs = nullptr;  // s slices of [HC | SC]^T m x 2n
  double* T64 = nullptr;         // [HC; SC]^T in float64  m x 2n (also C^T and C^T S_W for D)
  __nv_bfloat16* CTs = nullptr;  // kDensitySlices slices of C^T          m x n
  __nv_bfloat16* XTs = nullptr;  // kDensitySlices slices of C^T S_W      m x n
  __nv_bfloat16* SWs = nullptr;  // kDensitySlices slices of S_W          n x n
  long ldn = 0;
  tc::Operand opHS, opC, opY, opW, opYT, opCT, opXT, opSW, opCTb;  // opCTb: C^T as a B operand
  int* err = nullptr;
  const tc::BlockLists* hs_blocks = nullptr;  // block sparsity of [H~; S] (256-row blocks), the mixed state's
};

namespace {
// D needs |dD| <= 1e-7 at O(1) entries: 8 slices (40 bits) leave a wide margin
constexpr int kDensitySlices = 8;

// float64 sums of the sliced products of one call: 80 MB, which only the streams that have such products
// running need, not every context (64 contexts of one batch held 5 GB between them)
struct Slab : mem::Lease<double> {
  explicit Slab(cudaStream_t st) : Lease((size_t)tc::sliced_workspace_doubles(), st) {}
};
}

EmuState* emu_create(cudaStream_t st, int m, int n, int slices, const double* HS, const tc::BlockLists* hs_blocks) {
  EmuState* es = new EmuState();
  try {
    es->m = m;
    es->n = n;
    es->s = slices;
    es->ldm = round8(m);
    es->ld2n = round8(2L * n);
    const long s = slices, ldm = es->ldm, ld2n = es->ld2n;
    alloc(&es->HSs, (size_t)s * 2 * m * ldm, st);
    alloc(&es->Cs, (size_t)s * n * ldm, st);
    alloc(&es->Ys, (size_t)s * 2 * n * ldm, st);
    alloc(&es->Ws, (size_t)s * n * ld2n, st);
    alloc(&es->YTs, (size_t)s * m * ld2n, st);
    alloc(&es->T64, (size_t)m * 2 * n, st);
    es->ldn = round8(n);
    alloc(&es->CTs, (size_t)kDensitySlices * m * es->ldn, st);
    alloc(&es->XTs, (size_t)kDensitySlices * m * es->ldn, st);
    alloc(&es->SWs, (size_t)kDensitySlices * n * es->ldn, st);
    alloc(&es->err, 1, st);
    OMM_CUDA_TRY(cudaMemsetAsync(es->err, 0, sizeof(int), st));
    emu::slice_rows(st, HS, 2L * m, m, m, slices, es->HSs, ldm, nullptr);
    es->hs_blocks = hs_blocks;
    es->opHS = tc::make_operand(es->HSs, 2L * m, m, ldm, slices, false);
    es->opC = tc::make_operand(es->Cs, n, m, ldm, slices, true);
    es->opY = tc::make_operand(es->Ys, 2L * n, m, ldm, slices, false);
    es->opW = tc::make_operand(es->Ws, n, 2L * n, ld2n, slices, true);
    es->opYT = tc::make_operand(es->YTs, m, 2L * n, ld2n, slices, false);
    es->opCT = tc::make_operand(es->CTs, m, n, es->ldn, kDensitySlices, true);
    es->opXT = tc::make_operand(es->XTs, m, n, es->ldn, kDensitySlices, true);
    es->opSW = tc::make_operand(es->SWs, n, n, es->ldn, kDensitySlices, false);
    es->opCTb = tc::make_operand(es->CTs, m, n, es->ldn, kDensitySlices, false);
  } catch (...) {
    emu_destroy(es, st);
    throw;
  }
  return es;
}

void emu_update_H(EmuState* es, cudaStream_t st, const double* HS) {
  emu::slice_rows(st, HS, 2L * es->m, es->m, es->m, es->s, es->HSs, es->ldm, nullptr);
}

void emu_destroy(EmuState* es, cudaStream_t st) {
  if (!es) return;
  void* bufs[] = {es->HSs, es->Cs, es->Ys, es->Ws, es->YTs, es->T64, es->CTs, es->XTs, es->SWs, es->err};
  for (void* b : bufs) mem::release(b, st);
  delete es;
}

int emu_error(EmuState* es, cudaStream_t st) {
  int e = 0;
  OMM_CUDA_TRY(cudaMemcpyAsync(&e, es->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  OMM_CUDA_TRY(cudaStreamSynchronize(st));
  return e;
}

// HC, SC, S_W, H_W, E~, G and max|G| from C with float64-class tensor-core products.
void emu_recompute_state(EmuState* es, cudaStream_t st, Scalars* sc, const double* C, double* Y4,
                         double* SWHW, double* G, double* part, double* part2) {
  const int m = es->m, n = es->n, s = es->s;
  const long nm = (long)n * m;
  const Slab slab(st);
  emu::slice_rows(st, C, n, m, m, s, es->Cs, es->ldm, nullptr);
  // [HC; SC] (n x m layout) = C [H~; S]^T
  emu::gemm(st, es->opC, es->opHS, m, s, tc::Epilogue{Y4, m, m, nm, 1.0, 0.0, n, 2 * m, nullptr, es->err},
            slab, es->hs_blocks);
  emu::slice_rows(st, Y4, 2L * n, m, m, s, es->Ys, es->ldm, nullptr);
  // [S_W | H_W] = C [SC; HC]^T
  emu::gemm(st, es->opC, es->opY, m, s,
            tc::Epilogue{SWHW + n, 2L * n, n, -(long)n, 1.0, 0.0, n, 2 * n, nullptr, es->err}, slab);
  launch_functional(st, n, SWHW, part2);
  launch_finish_functional(st, sc, part2, traces_blocks(n));
  // G = 8 HC - 4 [S_W | H_W] [HC; SC]
  emu::slice_rows(st, SWHW, n, 2L * n, 2L * n, s, es->Ws, es->ld2n, nullptr);
  emu::transpose(st, Y4, 2L * n, m, m, es->T64, 2L * n);
  emu::slice_rows(st, es->T64, m, 2L * n, 2L * n, s, es->YTs, es->ld2n, nullptr);
  launch_scale_copy(st, nm, Y4, 8.0, G, nullptr);
  emu::gemm(st, es->opW, es->opYT, 2 * n, s, tc::Epilogue{G, m, m, 0, -4.0, 1.0, n, m, nullptr, es->err},
            slab);
  launch_gmax(st, nm, G, part);
  launch_finish_gmax(st, sc, part);
}

}  // namespace omm

namespace omm {

namespace {
// out = a x + b y (float64, count elements)
__global__ void combine_kernel(long count, double a, const double* __restrict__ x, double b,
                               const double* __restrict__ y, double* out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count; i += (long)gridDim.x * blockDim.x)
    out[i] = fma(a, x[i], b * y[i]);
}
}  // namespace

// D = 2 C^T (2I - S_W) C (n x m layout of C), float64-class: X = C^T S_W from the sliced C^T and
// S_W, W = 4 C^T - 2 X in float64, then one sliced product D = W (C^T)^T. The B operand C^T is
// the same slice stack as the A operand, mapped with B-sized TMA boxes.
void emu_density(EmuState* es, cudaStream_t st, const double* C, const double* SWHW, double* D) {
  const int m = es->m, n = es->n, s = kDensitySlices;
  const long mn = (long)m * n;
  const Slab slab(st);
  double* CT = es->T64;       // m x n
  double* XT = es->T64 + mn;  // m x n
  emu::transpose(st, C, n, m, m, CT, n);
  emu::slice_rows(st, CT, m, n, n, s, es->CTs, es->ldn, nullptr);
  emu::slice_rows(st, SWHW, n, n, 2L * n, s, es->SWs, es->ldn, nullptr);   // S_W is symmetric
  emu::gemm(st, es->opCT, es->opSW, n, s, tc::Epilogue{XT, n, n, 0, 1.0, 0.0, m, n, nullptr, es->err}, slab);
  combine_kernel<<<(unsigned)std::min<long>((mn + 255) / 256, 4096), 256, 0, st>>>(mn, 4.0, CT, -2.0, XT, XT);
  OMM_LAUNCH_CHECK();
  emu::slice_rows(st, XT, m, n, n, s, es->XTs, es->ldn, nullptr);
  emu::gemm(st, es->opXT, es->opCTb, n, s, tc::Epilogue{D, m, m, 0, 1.0, 0.0, m, m, nullptr, es->err}, slab);
}

namespace {
// W (n x n) = -2 H_W - eta (4I - 2 S_W) from SWHW = [S_W | H_W] (n x 2n)
__global__ void edm_weights_kernel(int n, const double* __restrict__ SWHW, double eta, double* W) {
  const long count = (long)n * n;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < count; idx += (long)gridDim.x * blockDim.x) {
    const long i = idx / n, j = idx - i * n;
    const double* row = SWHW + i * 2L * n;
    W[idx] = -2.0 * row[n + j] - eta * ((i == j ? 4.0 : 0.0) - 2.0 * row[j]);
  }
}
}  // namespace

// out = -(2 C^T H~_W C + eta D) (dE/dS at the minimum), float64-class. With D = C^T (4I - 2 S_W) C both
// terms share the outer coefficients: V = C^T W with W = -2 H~_W - eta (4I - 2 S_W), then one sliced
// product out = V (C^T)^T (forming D first took a second m x m x n product: 5.4 ms at m = 6656, n = 1024).
void emu_minus_edm(EmuState* es, cudaStream_t st, const double* C, const double* SWHW, double eta, double* out) {
  const int m = es->m, n = es->n, s = kDensitySlices;
  const long mn = (long)m * n;
  const Slab slab(st);
  double* CT = es->T64;       // m x n
  double* VT = es->T64 + mn;  // m x n; first the n x n weights
  emu::transpose(st, C, n, m, m, CT, n);
  emu::slice_rows(st, CT, m, n, n, s, es->CTs, es->ldn, nullptr);
  const long nn = (long)n * n;
  edm_weights_kernel<<<(unsigned)std::min<long>((nn + 255) / 256, 4096), 256, 0, st>>>(n, SWHW, eta, VT);
  OMM_LAUNCH_CHECK();
  emu::slice_rows(st, VT, n, n, n, s, es->SWs, es->ldn, nullptr);  // symmetric like H~_W and S_W
  emu::gemm(st, es->opCT, es->opSW, n, s, tc::Epilogue{VT, n, n, 0, 1.0, 0.0, m, n, nullptr, es->err}, slab);
  emu::slice_rows(st, VT, m, n, n, s, es->XTs, es->ldn, nullptr);
  emu::gemm(st, es->opXT, es->opCTb, n, s, tc::Epilogue{out, m, m, 0, 1.0, 0.0, m, m, nullptr, es->err}, slab);
}

}  // namespace omm
