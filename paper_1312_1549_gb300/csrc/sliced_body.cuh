// The sliced (float64-class) product: a pair list of slice products cut into chunks, every chunk an
// exact integer sum in the FP32 accumulator, the chunks added in float64. How its work is shared is in
// sliced_plan.cuh. Included by tc_gemm.cu.
//
// Sums: each CTA adds the pieces of a tile in a private 128 x TBN float64 slab laid out column by
// column, so that the 32 lanes of a warp (32 rows) touch 256 contiguous bytes, and a batch of columns
// is loaded before any is stored. (Adding every chunk to C itself, element by element in row order,
// serialised 256 dependent load-add-store round trips per thread and chunk, about 100 us.) The
// segment that holds a tile's first stage writes alpha x sum + beta C to C at its end; a worker whose
// share starts inside a tile leaves that segment's sum in its slab for slab_reduce_kernel.
#pragma once

// alpha v + beta C for 16 columns of one row (all loads of C before its stores)
__device__ __forceinline__ void store_row16(const Epilogue& ep, int row, int col0, const double (&v)[16]) {
  if (row >= ep.M || col0 >= ep.N) return;
  const int nvalid = min(16, ep.N - col0);
  const long blk0 = col0 / ep.split_cols, cb0 = col0 - blk0 * ep.split_cols;
  if (nvalid == 16 && cb0 + 16 <= ep.split_cols) {
    double* base = ep.C + blk0 * ep.split_stride + (long)row * ep.ldc + cb0;
    double c[16];
    if (ep.beta != 0.0) {
#pragma unroll
      for (int k = 0; k < 16; ++k) c[k] = base[k];
    }
    double o[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const double a = ep.alpha == 1.0 ? v[k] : ep.alpha * v[k];
      o[k] = ep.beta == 0.0 ? a : (ep.beta == 1.0 ? fma(ep.alpha, v[k], c[k]) : fma(ep.beta, c[k], a));
    }
    if ((reinterpret_cast<uintptr_t>(base) & 15) == 0) {
#pragma unroll
      for (int k = 0; k < 16; k += 2) *reinterpret_cast<double2*>(base + k) = make_double2(o[k], o[k + 1]);
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) base[k] = o[k];
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    if (k < nvalid) {
      const int col = col0 + k;
      const long blk = col / ep.split_cols;
      double* p = ep.C + blk * ep.split_stride + (long)row * ep.ldc + (col - blk * ep.split_cols);
      *p = combine(ep, v[k], p);
    }
  }
}

template <int TBN, bool PAIR>
__device__ __forceinline__ void sliced_body(const GroupDesc& g, const PairList& pl, const SlicedWork& w, int* err) {
  constexpr int TBH = PAIR ? TBN / 2 : TBN;  // B rows staged by each CTA
  constexpr int BH_BYTES = TBH * BK * 2;
  constexpr int SB = A_BYTES + BH_BYTES;     // one CTA's stage
  constexpr int NS = ring_stages(SB);
  constexpr uint32_t ACC_STRIDE = TBN;
  constexpr uint32_t COLS = 2 * TBN;         // two accumulators
  static_assert(NS >= 2 && NS * SB <= RING_BYTES && 2 * NS + 5 <= 28, "stage ring");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NS * SB);
  // bars as in pair_body: [0..NS) full, [NS..2NS) empty, [2NS..) accumulator full, [2NS+2..) accumulator
  // empty, [2NS+4] drain; with PAIR the full and accumulator-empty barriers of the even CTA serve both
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * NS + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rr = PAIR ? (int)cluster_ctarank() : 0;
  const bool leader = rr == 0;
  const int worker = PAIR ? (int)(blockIdx.x / 2) : (int)blockIdx.x;
  constexpr int BMT = PAIR ? 2 * BM : BM;
  auto chunk_end = [&](int c) { return pl.nchunk <= 0 ? pl.n : (int)pl.chunk_end[c]; };

  if (threadIdx.x == 0) {
    for (int q = 0; q < NS; ++q) {
      mbar_init(smem_u32(&bars[q]), 1);
      mbar_init(smem_u32(&bars[NS + q]), 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(smem_u32(&bars[2 * NS + q]), 1);                 // the MMA thread's commit
      mbar_init(smem_u32(&bars[2 * NS + 2 + q]), PAIR ? 8 : 4);  // one arrival per epilogue warp
    }
    mbar_init(smem_u32(&bars[2 * NS + 4]), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncwarp();
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if constexpr (PAIR) cluster_sync_all();
  else __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  dev::pdl_begin();

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer (with PAIR both CTAs)
    const CUtensorMap* mA = reinterpret_cast<const CUtensorMap*>(&g.a);
    const CUtensorMap* mB = reinterpret_cast<const CUtensorMap*>(&g.b);
    prefetch_tmap(mA);
    prefetch_tmap(mB);
    uint32_t it = 0;
    Walk walk(g, w, pl.n, worker);
    Segment s;
    while (!*abort_flag && walk.next(g, w, pl.n, s)) {
      const int ya = g.offA + s.mb * BMT + rr * BM, yb = g.offB + s.nb * TBN + rr * TBH;
      int p = s.s0 / s.kbs.count, k = s.s0 - p * s.kbs.count;
      for (int t = s.s0; t < s.s1; ++t, ++it) {
        const int q = it % NS;
        const uint32_t r = it / NS;
        if (!mbar_wait(smem_u32(&bars[NS + q]), (r & 1) ^ 1)) {
          *abort_flag = 1;
          atomicCAS(err, 0, 1);
          break;
        }
        const uint32_t sa = smem_u32(smem + q * SB);
        const int x = s.kbs.at(k) * BK, ra = (int)pl.a[p] * g.rowsA + ya, rb = (int)pl.b[p] * g.rowsB + yb;
        if constexpr (PAIR) {
          const uint32_t full = mapa_shared(smem_u32(&bars[q]), 0);
          if (leader) mbar_expect_tx(smem_u32(&bars[q]), 2 * SB);  // the bytes landing in both CTAs
          tma_load_2d_pair(sa, mA, full, x, ra);
          tma_load_2d_pair(sa + A_BYTES, mB, full, x, rb);
        } else {
          const uint32_t full = smem_u32(&bars[q]);
          mbar_expect_tx(full, SB);
          tma_load_2d(sa, mA, full, x, ra);
          tma_load_2d(sa + A_BYTES, mB, full, x, rb);
        }
        if (++k == s.kbs.count) {
          k = 0;
          ++p;
        }
      }
    }
    if (*abort_flag) {  // let the copies already issued land before the CTA releases its memory
      if (leader) {
        for (uint32_t j = it > (uint32_t)NS ? it - NS : 0u; j < it; ++j)
          mbar_wait(smem_u32(&bars[j % NS]), (j / NS) & 1);
      } else {  // these complete at the even CTA's barrier: give them time
        const uint64_t t0 = globaltimer();
        while (globaltimer() - t0 < PAIR_ABORT_SETTLE_NS) {
        }
      }
    }
  } else if (warp == 1 && lane == 0 && leader) {
    // ---------------- MMA issuer
    constexpr uint32_t idesc = idesc_bf16(BMT, TBN);
    uint32_t it = 0, lt = 0;
    Walk walk(g, w, pl.n, worker);
    Segment s;
    while (!*abort_flag && walk.next(g, w, pl.n, s)) {
      int c = 0;
      while (chunk_end(c) * s.kbs.count <= s.s0) ++c;
      for (int t = s.s0; t < s.s1 && !*abort_flag; ++c) {  // a piece: this segment's part of chunk c
        const int e = min(s.s1, chunk_end(c) * s.kbs.count);
        const uint32_t buf = lt & 1, use = lt >> 1;
        if (!mbar_wait(smem_u32(&bars[2 * NS + 2 + buf]), (use & 1) ^ 1)) {
          *abort_flag = 1;
          atomicCAS(err, 0, 4);
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem + buf * ACC_STRIDE;
        for (const int t0 = t; t < e; ++t, ++it) {
          const int q = it % NS;
          const uint32_t r = it / NS;
          if (!mbar_wait(smem_u32(&bars[q]), r & 1)) {
            *abort_flag = 1;
            atomicCAS(err, 0, 2);
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = smem_u32(smem + q * SB), sb = sa + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint32_t acc = (t > t0 || k > 0) ? 1u : 0u;
            if constexpr (PAIR) umma_bf16_pair(d, smem_desc(sa + k * 32), smem_desc(sb + k * 32), idesc, acc);
            else umma_bf16(d, smem_desc(sa + k * 32), smem_desc(sb + k * 32), idesc, acc);
          }
          if constexpr (PAIR) umma_commit_pair(smem_u32(&bars[NS + q]), 3);
          else umma_commit(smem_u32(&bars[NS + q]));
        }
        if constexpr (PAIR) umma_commit_pair(smem_u32(&bars[2 * NS + buf]), 3);
        else umma_commit(smem_u32(&bars[2 * NS + buf]));
        ++lt;
      }
    }
    if (*abort_flag) {  // every MMA issued so far is complete before the tensor memory is freed
      if constexpr (PAIR) umma_commit_pair_local(smem_u32(&bars[2 * NS + 4]));
      else umma_commit(smem_u32(&bars[2 * NS + 4]));
      mbar_wait(smem_u32(&bars[2 * NS + 4]), 0);
    }
  } else if (warp >= 2) {
    // ---------------- epilogue (with PAIR both CTAs: 128 rows each)
    const int lane_base = (warp & 3) * 32;
    const uint32_t acc_empty0 = PAIR ? mapa_shared(smem_u32(&bars[2 * NS + 2]), 0) : smem_u32(&bars[2 * NS + 2]);
    const uint32_t acc_empty1 = PAIR ? mapa_shared(smem_u32(&bars[2 * NS + 3]), 0) : smem_u32(&bars[2 * NS + 3]);
    const Epilogue ep = g.ep;
    double* slabs = w.slab + (long)blockIdx.x * 2 * BM * TBN + lane_base + lane;
    uint32_t lt = 0;
    bool failed = false;
    Walk walk(g, w, pl.n, worker);
    Segment s;
    while (!failed && walk.next(g, w, pl.n, s)) {
      const bool head = s.s0 == 0;  // this segment writes C; else its sum stays in slab 0
      double* slab = slabs + (head ? BM * TBN : 0);
      const int row0 = s.mb * BMT + rr * BM + lane_base, row = row0 + lane, n0 = s.nb * TBN;
      int c = 0;
      while (chunk_end(c) * s.kbs.count <= s.s0) ++c;
      for (int t = s.s0; t < s.s1; ++c) {
        const int e = min(s.s1, chunk_end(c) * s.kbs.count);
        const bool first = t == s.s0, last = e == s.s1;
        t = e;
        const uint32_t buf = lt & 1, use = lt >> 1;
        if (*abort_flag || !mbar_wait(smem_u32(&bars[2 * NS + buf]), use & 1)) {
          atomicCAS(err, 0, 3);
          failed = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // (a warp whose rows, and columns that, lie past the edge have nothing to add)
        const int ncol = row0 < ep.M ? min(TBN, ep.N - n0) : 0;
#pragma unroll 1
        for (int j = 0; 32 * j < ncol; ++j) {
          float v[32];
          tmem_ld32(tmem + buf * ACC_STRIDE + ((uint32_t)lane_base << 16) + (uint32_t)(j * 32), v);
          double* sl = slab + (long)(32 * j) * BM;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            double x[16];
            if (first) {  // (a real branch: a predicated float64 add costs as much as a needed one)
#pragma unroll
              for (int k = 0; k < 16; ++k) x[k] = widen(v[16 * h + k]);
            } else {
#pragma unroll
              for (int k = 0; k < 16; ++k) x[k] = sl[(16 * h + k) * BM];
#pragma unroll
              for (int k = 0; k < 16; ++k) x[k] += widen(v[16 * h + k]);
            }
            if (last && head) {
              store_row16(ep, row, n0 + 32 * j + 16 * h, x);
            } else {
#pragma unroll
              for (int k = 0; k < 16; ++k) sl[(16 * h + k) * BM] = x[k];
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          if constexpr (PAIR) mbar_arrive_cluster(buf ? acc_empty1 : acc_empty0);
          else mbar_arrive(buf ? acc_empty1 : acc_empty0);
        }
        ++lt;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if constexpr (PAIR) cluster_sync_all();
  else __syncthreads();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
  }
}

template <int TBN>
__global__ void __launch_bounds__(NTHREADS, 1)
sliced_kernel(const __grid_constant__ GroupDesc g, const __grid_constant__ PairList pl,
              const __grid_constant__ SlicedWork w, int* err) {
  sliced_body<TBN, false>(g, pl, w, err);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1)
sliced_pair_kernel(const __grid_constant__ GroupDesc g, const __grid_constant__ PairList pl,
                   const __grid_constant__ SlicedWork w, int* err) {
  sliced_body<256, true>(g, pl, w, err);
}

// C += alpha x (the slabs of the workers whose share starts inside the tile, in order). One CTA per
// 8 x 32 block of a left-over tile (a small product's few tiles have up to a hundred slabs each, and every
// slab costs a block of 32 x 32 some thousand clocks of float64 adds); bmt rows per tile, bmt / 128 CTAs per
// worker (rows 128 q .. of a tile belong to its q-th CTA). A tile that no share starts in is left alone.
__global__ void __launch_bounds__(256)
slab_reduce_kernel(const __grid_constant__ GroupDesc g, int npairs, const __grid_constant__ SlicedWork w, int bmt) {
  dev::pdl_begin();
  const int subs_n = g.bn / 32, subs = (bmt / 8) * subs_n;
  const int tile = w.full * w.nw + blockIdx.x / subs, sub = blockIdx.x % subs;
  const int mb = tile % w.tiles_m, nb = tile / w.tiles_m;
  const int r0 = (sub / subs_n) * 8, c0 = (sub % subs_n) * 32;
  const int row0 = mb * bmt + r0, col0 = nb * g.bn + c0;
  if (row0 >= g.ep.M || col0 >= g.ep.N) return;
  const Slabs slabs = slabs_of(g, w, npairs, tile);
  const int first = slabs.first, last = slabs.last;
  if (first >= last) return;
  const int ctas = bmt / BM;
  const int rr = threadIdx.x & 7, cc = threadIdx.x >> 3;  // eight rows (64 bytes) of a column
  const double* slab = w.slab + ((long)first * ctas + r0 / BM) * 2 * BM * g.bn + (r0 % BM) + rr + (long)(c0 + cc) * BM;
  const long step = (long)ctas * 2 * BM * g.bn;
  double v = 0.0;
  int q = first;
  for (; q + 8 <= last; q += 8, slab += 8 * step) {  // eight loads in flight
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = slab[k * step];
#pragma unroll
    for (int k = 0; k < 8; ++k) v += x[k];
  }
  for (; q < last; ++q, slab += step) v += *slab;
  __shared__ double t[32][9];
  t[cc][rr] = v;
  __syncthreads();
  const int col = col0 + (threadIdx.x & 31), row = row0 + (threadIdx.x >> 5);
  if (col >= g.ep.N || row >= g.ep.M) return;
  const long blk = col / g.ep.split_cols;
  double* p = g.ep.C + blk * g.ep.split_stride + (long)row * g.ep.ldc + (col - blk * g.ep.split_cols);
  *p = fma(g.ep.alpha, t[threadIdx.x & 31][threadIdx.x >> 5], *p);
}
