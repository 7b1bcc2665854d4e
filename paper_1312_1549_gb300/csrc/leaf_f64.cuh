// The float64 leaf of the Cholesky inverses, one thread block (leaf_f64_kernel in cholesky.cu). Needs nothing
// but the built-in device functions, so that it also runs under a thread-block emulator on the host.
#pragma once

namespace omm {
namespace dev {

// Factor the b x b diagonal block at A (ld lda) in place (lower) and write
// its inverse to Linv (ld ldi, zero above the diagonal), in float64 on one CTA.
// The factor and the inverse take 44 thousand FMAs each, 11 us
// each at the two per clock of one SM, so the work is laid out for that pipe:
// no FMA on zeros beyond 8-wide blocks, all eight warps busy, short dependent
// chains. Right-looking in panels of eight columns: a panel is factored with
// its rows in the registers of up to three warps (pivots and column entries by
// shuffles, one rsqrt per pivot on the chain), then all warps apply its rank-8
// update on 8 x 8 blocks.
// The inverse joins inverted diagonal blocks of edge 8, 16 and 32:
// X21 = -X22 (L21 X11), the contraction cut at the triangles.
// (One column at a time with three barriers each, one thread per column of the
// inverse and two divisions per pivot it took 150-215 us per block, 67 to 83 now; by this alone the float64-class
// inverse at m = 3328, 52 blocks one after another, went from 30.1 to 25.9 ms.)
constexpr int NB = 64;
constexpr int kLeaf64Threads = 256;

__device__ __forceinline__ void leaf_f64_body(double* A, long lda, int b, double* Linv, long ldi, int* info,
                                              int col_offset) {
  __shared__ double L[NB][NB + 1];
  __shared__ double X[NB][NB + 1];
  __shared__ double rdiag[NB], pivot[NB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kWarps = kLeaf64Threads / 32;
  for (int idx = tid; idx < NB * NB; idx += kLeaf64Threads) {
    const int i = idx / NB, j = idx % NB;
    L[i][j] = (i < b && j <= i) ? A[(long)i * lda + j] : 0.0;
    X[i][j] = 0.0;
  }
  __syncthreads();
  for (int p0 = 0; p0 < b; p0 += 8) {
    const int pw = min(8, b - p0);
    // lanes 0-7 of the first three warps hold the panel's diagonal rows (each warp factors its own copy,
    // so that no warp waits for another's pivots), lanes 8-31 the rows below, 24 to a warp
    const int i = lane < 8 ? p0 + lane : p0 + 8 + 24 * warp + lane - 8;
    double r[8];
    if (warp < 3 && (warp == 0 || p0 + 8 + 24 * warp < b)) {
#pragma unroll
      for (int c = 0; c < 8; ++c) r[c] = (i < b && c < pw && p0 + c <= i) ? L[i][p0 + c] : 0.0;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c < pw) {
          double d = __shfl_sync(0xffffffffu, r[c], c);  // the pivot, row p0 + c
          if (!(d > 0.0)) {
            if (warp == 0 && lane == 0) atomicCAS(info, 0, col_offset + p0 + c + 1);
            d = 1.0;
          }
          // 1 / sqrt(d) to the last place: one Newton step on rsqrt's value
          double rs = rsqrt(d);
          if (rs > 0.0) rs = fma(0.5 * rs, fma(-(d * rs), rs, 1.0), rs);  // (0 only for an infinite pivot)
          if (warp == 0 && lane == 0) {
            rdiag[p0 + c] = rs;
            pivot[p0 + c] = d;
          }
          r[c] *= rs;
#pragma unroll
          for (int l = 0; l < 8; ++l)
            if (l > c) r[l] = fma(-r[c], __shfl_sync(0xffffffffu, r[c], l), r[l]);  // L[p0 + l][p0 + c]
        }
      }
      // (entries above the diagonal, and the diagonal itself, are left to what follows)
      if (lane >= 8) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (i < b && c < pw) L[i][p0 + c] = r[c];
      }
    }
    __syncthreads();
    // the diagonal rows go back once every warp has read them (the update below touches later rows only)
    if (warp == 0 && lane < 8) {
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (i < b && c < pw && p0 + c < i) L[i][p0 + c] = r[c];
    }
    // trailing lower triangle in 8 x 8 blocks (I, J <= I), a warp per block, two rows per lane
    const int q0 = p0 + 8, nb8 = (b - q0 + 7) / 8;
    for (int q = warp, I = 0, base = 0; I < nb8; ) {
      if (q >= base + I + 1) { base += I + 1; ++I; continue; }
      const int J = q - base;
      const int i = q0 + 8 * I + (lane >> 3), j = q0 + 8 * J + (lane & 7);
      double a0 = L[i][j], a1 = L[i + 4][j];  // (rows and columns past b hold zeros)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const double lj = L[j][p0 + k];
        a0 = fma(-L[i][p0 + k], lj, a0);
        a1 = fma(-L[i + 4][p0 + k], lj, a1);
      }
      if (j <= i) L[i][j] = a0;
      if (j <= i + 4) L[i + 4][j] = a1;
      q += kWarps;
    }
    __syncthreads();
  }
  if (tid < b) {  // the factor's diagonal, sqrt(d), off the panels' chain
    const double d = pivot[tid], t = d * rdiag[tid];
    L[tid][tid] = rdiag[tid] > 0.0 ? fma(0.5 * rdiag[tid], fma(-t, t, d), t) : d;
  }
  // inverses of the 8 x 8 diagonal blocks: warp w's lane c solves column c of block w
  if (8 * warp < b && lane < 8 && 8 * warp + lane < b) {
    const int o = 8 * warp, c = lane, e = min(8, b - o);
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = 0.0;
      if (i == c) x[i] = rdiag[o + i];
      if (i > c && i < e) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k >= c && k < i) acc = fma(L[o + i][o + k], x[k], acc);
        x[i] = -acc * rdiag[o + i];
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i >= c && i < e) X[o + i][o + c] = x[i];
  }
  __syncthreads();
  // Join blocks of edge s: T = L21 X11 (kept transposed in the unused upper triangle of L: T[i][j] of
  // the pair at o in L[o + j][o + s + i]), X21 = -X22 T. For T a warp takes four rows and walks the
  // column groups of eight, contracting from the group's first column; for X21 four columns and the row
  // groups, contracting to the group's last row. (Rows past b are zero in L and X.)
  for (int s = 8; s < b; s *= 2) {
    const int wpp = s / 4;  // warps per pair
    const int pairs = (b + 2 * s - 1) / (2 * s);
    for (int u = warp; u < pairs * wpp; u += kWarps) {
      const int o = 2 * s * (u / wpp), i = 4 * (u % wpp) + (lane >> 3);
      for (int g = 0; g < s; g += 8) {
        const int j = g + (lane & 7);
        double acc0 = 0.0, acc1 = 0.0;
        for (int k = g; k < s; k += 2) {
          acc0 = fma(L[o + s + i][o + k], X[o + k][o + j], acc0);
          acc1 = fma(L[o + s + i][o + k + 1], X[o + k + 1][o + j], acc1);
        }
        L[o + j][o + s + i] = acc0 + acc1;
      }
    }
    __syncthreads();
    for (int u = warp; u < pairs * wpp; u += kWarps) {
      const int o = 2 * s * (u / wpp), j = 4 * (u % wpp) + (lane >> 3);
      for (int g = 0; g < s; g += 8) {
        const int i = g + (lane & 7);
        double acc0 = 0.0, acc1 = 0.0;
        for (int k = 0; k < g + 8; k += 2) {
          acc0 = fma(X[o + s + i][o + s + k], L[o + j][o + s + k], acc0);
          acc1 = fma(X[o + s + i][o + s + k + 1], L[o + j][o + s + k + 1], acc1);
        }
        if (o + s + i < b) X[o + s + i][o + j] = -(acc0 + acc1);
      }
    }
    __syncthreads();
  }
  for (int idx = tid; idx < NB * NB; idx += kLeaf64Threads) {
    const int i = idx / NB, j = idx % NB;
    if (i < b && j < b) {
      A[(long)i * lda + j] = (j <= i) ? L[i][j] : 0.0;
      Linv[(long)i * ldi + j] = X[i][j];
    }
  }
}

}  // namespace dev
}  // namespace omm
