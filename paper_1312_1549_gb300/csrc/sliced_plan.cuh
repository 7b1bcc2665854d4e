// How a sliced product's work is shared among the SMs: the plan (host), the walk of one worker through
// its share, and the slabs of a tile (device and host, so that a test can follow them without a GPU).
//
// Work: a stage is one 64-wide K block of one slice pair of one output tile; a tile has npairs x
// (its K blocks) of them. A worker (a CTA, or with PAIR the two CTAs of a cluster) takes `full` whole
// tiles, tile index worker + k nw, and the stages of the tiles that are left over form one line that
// is shared evenly among nr workers, cutting tiles and even chunks where a share begins and ends: a part
// of an exact integer sum is exact too, so nothing is lost. (Whole tiles only left SMs idle: 104 tiles of
// 256 x 256 on 76 pairs take two rounds for 1.37 rounds of work, 36 tiles of 128 x 256 use 36 of 152
// SMs.) Workers on whole tiles, and on the same fraction of a tile, walk the slice pairs in step and
// share the slices through L2; shares at arbitrary places of the line do not (the slices of a
// 1024 x 6656 x 6656 product are 1 GB), which costs more than it balances once they outgrow L2 (that
// product with its slicing and its scratch: 5.3 ms in whole tiles, 5.5 with one even line, 3.9 with this, 3.0
// since the scratch comes from a pool; a 1495 x 260 state's products 0.9-1.4 ms each before, 0.14 now).
#pragma once

#include <algorithm>

#include "tc_gemm.cuh"

namespace omm {
namespace tc {

// K is consumed in stages of BK = 64 contracted columns (one 128-byte swizzle atom of bf16 per
// row). Stages of 32 columns (64-byte swizzle) were measured slower: twice the barrier and commit
// round trips per contracted column, for no gain in the bytes kept in flight.
constexpr int BM = 128, BN = 256, BK = 64;

// The K blocks of one output tile: all of them, or the listed ones where B is block-sparse.
struct KBlocks {
  const int* list;  // null: 0 .. count-1
  int count;
  __host__ __device__ __forceinline__ int at(int i) const { return list ? list[i] : i; }
};

struct SlicedWork {
  double* slab;  // 2 x 128 x TBN per CTA: [0] a share's first, headless segment, [1] scratch
  int nw;        // workers
  int full;      // whole tiles of each
  int nr;        // workers that share the left-over tiles' stages (0: none left)
  int tiles_m;   // tiles along M (the fast index)
  int tiles;     // all tiles
};

// the line of the stages of the left-over tiles, positions counted from the first stage of tile 0
struct Line {
  long base, len;
  __host__ __device__ __forceinline__ long begin(const SlicedWork& w, int worker) const { return base + len * worker / w.nr; }
};
__host__ __device__ __forceinline__ Line line_of(const GroupDesc& g, const SlicedWork& w, int npairs) {
  const int t0 = w.full * w.nw;
  Line l;
  if (g.kb_off != nullptr) {
    const int nb = t0 / w.tiles_m, mb = t0 - nb * w.tiles_m;
    const long unit = (long)npairs * w.tiles_m;
    l.base = t0 < w.tiles ? unit * g.kb_off[nb] + (long)npairs * mb * (g.kb_off[nb + 1] - g.kb_off[nb]) : 0;
    l.len = unit * g.kb_off[w.tiles / w.tiles_m] - l.base;
  } else {
    const long per = (long)npairs * ((g.K + BK - 1) / BK);
    l.base = per * t0;
    l.len = per * (w.tiles - t0);
  }
  return l;
}

// one tile's run of stages [s0, s1) inside a worker's work
struct Segment {
  int mb, nb;
  KBlocks kbs;
  int s0, s1;
};

// walks the segments of one worker; every role of its CTAs walks the same ones
struct Walk {
  int worker, k;
  long pos, end;
  __host__ __device__ __forceinline__ Walk(const GroupDesc& g, const SlicedWork& w, int npairs, int worker_) : worker(worker_), k(0) {
    pos = end = 0;
    if (worker < w.nr) {
      const Line l = line_of(g, w, npairs);
      pos = l.begin(w, worker);
      end = l.begin(w, worker + 1);
    }
  }
  __host__ __device__ __forceinline__ void kblocks(const GroupDesc& g, int nb, KBlocks& kbs) const {
    if (g.kb_off != nullptr) {
      const int o0 = g.kb_off[nb];
      kbs.list = g.kb_idx + o0;
      kbs.count = g.kb_off[nb + 1] - o0;
    } else {
      kbs.list = nullptr;
      kbs.count = (g.K + BK - 1) / BK;
    }
  }
  __host__ __device__ __forceinline__ bool next(const GroupDesc& g, const SlicedWork& w, int npairs, Segment& s) {
    if (k < w.full) {
      const int tile = worker + k * w.nw;
      ++k;
      s.mb = tile % w.tiles_m;
      s.nb = tile / w.tiles_m;
      kblocks(g, s.nb, s.kbs);
      s.s0 = 0;
      s.s1 = npairs * s.kbs.count;
      return true;
    }
    if (pos >= end) return false;
    if (g.kb_off != nullptr) {  // the column block whose tiles hold this position
      const long unit = (long)npairs * w.tiles_m;
      int lo = 0, hi = w.tiles / w.tiles_m - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (unit * g.kb_off[mid] <= pos) lo = mid; else hi = mid - 1;
      }
      kblocks(g, lo, s.kbs);
      const int per = npairs * s.kbs.count;
      const long rem = pos - unit * g.kb_off[lo];
      s.nb = lo;
      s.mb = (int)(rem / per);
      s.s0 = (int)(rem - (long)s.mb * per);
    } else {
      kblocks(g, 0, s.kbs);
      const int per = npairs * s.kbs.count;
      const long tile = pos / per;
      s.s0 = (int)(pos - tile * per);
      s.mb = (int)(tile % w.tiles_m);
      s.nb = (int)(tile / w.tiles_m);
    }
    const long stop = s.s0 + (end - pos), all = (long)npairs * s.kbs.count;
    s.s1 = (int)(stop < all ? stop : all);
    pos += s.s1 - s.s0;
    return true;
  }
};

// the workers [first, last) whose shares begin strictly inside a left-over tile: each holds a part of the
// tile's sum in its slab (none: first >= last)
struct Slabs {
  int first, last;
};
__host__ __device__ __forceinline__ Slabs slabs_of(const GroupDesc& g, const SlicedWork& w, int npairs, int tile) {
  const int nb = tile / w.tiles_m, mb = tile % w.tiles_m;
  long base, per;
  if (g.kb_off != nullptr) {
    const int o0 = g.kb_off[nb];
    per = (long)npairs * (g.kb_off[nb + 1] - o0);
    base = (long)npairs * w.tiles_m * o0 + mb * per;
  } else {
    per = (long)npairs * ((g.K + BK - 1) / BK);
    base = tile * per;
  }
  const Line line = line_of(g, w, npairs);
  int first = (int)((base - line.base) * w.nr / line.len);
  while (first < w.nr && line.begin(w, first) <= base) ++first;
  if (first >= w.nr || line.begin(w, first) >= base + per) return Slabs{0, 0};
  int last = (int)((base + per - line.base) * w.nr / line.len) + 1;  // one past the last such worker
  while (last > first && (last > w.nr || line.begin(w, last - 1) >= base + per)) --last;
  return Slabs{first, last};
}

struct SlicedPlan {
  SlicedWork work;  // the slab is the caller's
  int bn;           // tile width
  bool pair;        // 256-row tiles on pairs of SMs
  bool whole;       // every share ends with a tile
};
// pairs: clusters of two CTAs that the device holds at once; sms: its SMs
inline SlicedPlan plan_sliced(int M, int N, int K, const PairList& pl, const BlockLists* sparse, int pairs, int sms) {
  if (sparse != nullptr && (long)sparse->off_host.size() != (N + 255) / 256 + 1)
    throw CudaError{cudaErrorInvalidValue, "tc::plan_sliced: block lists do not match the tiles"};
  const long nkb = (K + BK - 1) / BK;
  const int nchunk = pl.nchunk > 0 ? pl.nchunk : 1;
  // Tile shape and number of workers with the shortest estimated time, in SM clocks. A stage takes as
  // long as its copies: about 55 bytes per clock land in an SM's shared memory, 32 KB for a pair's 256 x
  // 256 or one SM's 128 x 128 tile, 48 KB for 128 x 256. Adding a piece to a running sum costs a float64
  // add per element, about one per clock and SM, beside the stages that follow; the last piece's add and
  // about 5000 clocks of start-up are exposed, and where shares do not end with tiles the slab pass too.
  struct Shape { int bn; bool pair; double cycles; };
  const Shape shapes[3] = {{256, true, 600.0}, {256, false, 900.0}, {128, false, 600.0}};
  // shares at arbitrary places only while the slices stay in L2 (above)
  int slices = 0;
  for (int p = 0; p < pl.n; ++p) slices = std::max(slices, std::max((int)pl.a[p], (int)pl.b[p]) + 1);
  const bool resident = 2.0 * slices * ((double)M + N) * K <= 100e6;
  SlicedPlan best{};
  double best_t = 0.0;
  for (const Shape& sh : shapes) {
    if (sparse != nullptr && sh.bn != 256) continue;  // block lists are made for 256 rows
    const int bmt = sh.pair ? 2 * BM : BM, workers = sh.pair ? pairs : sms;
    const int tm = (M + bmt - 1) / bmt, tn = (N + sh.bn - 1) / sh.bn, tiles = tm * tn;
    const double per_tile = sparse ? (double)pl.n * sparse->nnz / tn : (double)pl.n * nkb;
    const int full = tiles / workers, left = tiles - full * workers;
    // The left-over tiles are the last ones, which a triangular B leaves with far fewer stages than the average
    // tile. A share has 8 stages or more where there are as many, and at least one (a tile has one or more): a
    // worker without any would leave a slab that slab_reduce_kernel adds unwritten.
    long line = (long)left * pl.n * nkb;
    if (sparse != nullptr) {
      const std::vector<int>& off = sparse->off_host;
      const int t0 = full * workers, nb = t0 / tm, mb = t0 - nb * tm;
      line = left ? pl.n * ((long)tm * (off[tn] - off[nb]) - (long)mb * (off[nb + 1] - off[nb])) : 0;
    }
    const int most = (int)std::min<long>(workers, std::max<long>(left, line / 8));
    const double add = (double)std::min(M, BM) * std::min(N, sh.bn);  // elements of one CTA's piece
    for (int k = 0; k < 2; ++k) {
      // left-over tiles in equal parts (one or more workers each), or evenly over all workers
      const int nr = left == 0 ? 0 : (k == 0 ? left * (most / left) : most);
      if (k == 1 && (left == 0 || !resident)) continue;
      const bool whole = nr == 0 || (sparse == nullptr && nr == left);
      const double stages = full * per_tile + (nr ? (double)line / nr : 0.0);
      const double t = std::max(stages * sh.cycles, nchunk * stages / per_tile * add) + add + 5000.0 +
                       (whole ? 0.0 : 9000.0 + add / 8.0);
      if (best_t == 0.0 || t < best_t) {
        best.work = SlicedWork{nullptr, full > 0 ? workers : nr, full, nr, tm, tiles};
        best.bn = sh.bn;
        best.pair = sh.pair;
        best.whole = whole;
        best_t = t;
      }
    }
  }
  return best;
}

}  // namespace tc
}  // namespace omm
