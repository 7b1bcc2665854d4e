// The plans of sliced products, followed on the host: every stage of every tile belongs to exactly one worker,
// every share of the left-over tiles' line has a length, and the slabs that a tile adds are those of the
// workers that hold a part of it.
#include <cstdio>
#include <numeric>
#include <random>
#include <vector>

#include "sliced_plan.cuh"

using namespace omm::tc;

static PairList pair_list(int slices) {
  PairList pl{};
  for (int d = slices - 1; d >= 0; --d)
    for (int i = 0; i <= d; ++i) {
      pl.a[pl.n] = (unsigned char)i;
      pl.b[pl.n++] = (unsigned char)(d - i);
    }
  pl.nchunk = 1;
  pl.chunk_end[0] = (unsigned char)pl.n;
  return pl;
}

// K blocks of each 256-wide column block
enum Pattern { kDense, kUpper, kLower, kShortTail, kRandom };
static std::vector<int> counts(Pattern p, int N, int nkb, std::mt19937& gen) {
  std::vector<int> c((N + 255) / 256);
  for (size_t b = 0; b < c.size(); ++b) {
    const int first = std::min<int>(nkb - 1, 4 * (int)b), end = std::min(nkb, 4 * ((int)b + 1));
    c[b] = p == kUpper ? nkb - first : p == kLower ? end : p == kShortTail ? (b + 2 < c.size() ? nkb : 1)
           : std::uniform_int_distribution<int>(1, nkb)(gen);
  }
  return c;
}

static int check(int M, int N, int K, Pattern p, int pairs, int slices, std::mt19937& gen) {
  const PairList pl = pair_list(slices);
  const int nkb = (K + BK - 1) / BK;
  BlockLists bl;
  std::vector<int> off(1, 0), idx(nkb);
  std::iota(idx.begin(), idx.end(), 0);
  GroupDesc g{};
  g.K = K;
  if (p != kDense) {
    for (int c : counts(p, N, nkb, gen)) off.push_back(off.back() + c);
    bl.nblocks = (int)off.size() - 1;
    bl.nnz = off.back();
    bl.dense = (long)bl.nblocks * nkb;
    bl.off_host = off;
    idx.resize(off.back() + nkb);
    g.kb_off = off.data();
    g.kb_idx = idx.data();
  }
  const SlicedPlan plan = plan_sliced(M, N, K, pl, p == kDense ? nullptr : &bl, pairs, 2 * pairs);
  const SlicedWork& w = plan.work;
  const int bmt = plan.pair ? 256 : 128, tm = (M + bmt - 1) / bmt, tn = (N + plan.bn - 1) / plan.bn;
  const char* bad = nullptr;
  if (w.tiles_m != tm || w.tiles != tm * tn || w.nw < 1 || w.nw > (plan.pair ? pairs : 2 * pairs) || w.nr > w.nw)
    bad = "sizes of the plan";
  std::vector<std::vector<int>> seen(w.tiles), parts(w.tiles);
  for (int t = 0; t < w.tiles; ++t)
    seen[t].assign((size_t)pl.n * (g.kb_off ? off[t / tm + 1] - off[t / tm] : nkb), 0);
  for (int worker = 0; worker < w.nw && !bad; ++worker) {
    if (worker < w.nr) {
      const Line l = line_of(g, w, pl.n);
      if (l.begin(w, worker) >= l.begin(w, worker + 1)) bad = "a share of length zero";
    }
    Walk walk(g, w, pl.n, worker);
    Segment s;
    int headless = 0;
    while (!bad && walk.next(g, w, pl.n, s)) {
      const int t = s.nb * tm + s.mb;
      if (t >= w.tiles || s.s0 >= s.s1 || s.s1 > (int)seen[t].size()) bad = "a segment outside its tile";
      for (int q = s.s0; !bad && q < s.s1; ++q) ++seen[t][q];
      if (!bad && s.s0 > 0) {
        parts[t].push_back(worker);
        if (++headless > 1) bad = "two parts in one slab";
      }
    }
  }
  for (int t = 0; t < w.tiles && !bad; ++t) {
    for (int c : seen[t])
      if (c != 1) bad = "a stage taken by none or by two";
    if (plan.whole ? !parts[t].empty() : t < w.full * w.nw && !parts[t].empty()) bad = "a part that nothing adds";
    if (!plan.whole && t >= w.full * w.nw && !bad) {
      const Slabs s = slabs_of(g, w, pl.n, t);
      std::vector<int> added;
      for (int q = s.first; q < s.last; ++q) added.push_back(q);
      if (added != parts[t]) bad = "slabs added that hold no part of the tile";
    }
  }
  if (bad)
    std::printf("M %d N %d K %d pattern %d pairs %d slices %d: %s\n", M, N, K, (int)p, pairs, slices, bad);
  return bad != nullptr;
}

int main() {
  std::mt19937 gen(11);
  int bad = 0;
  auto size = [&](double lo, double hi) {
    return (int)std::exp(std::uniform_real_distribution<double>(std::log(lo), std::log(hi))(gen));
  };
  for (int pairs : {74, 75, 76}) {
    // one left-over tile on pairs of SMs, its column block the last and short one
    for (int tn = 2; tn <= 40; ++tn)
      for (int tm = 1; tm <= 40; ++tm)
        if (tm * tn % pairs <= 2)
          for (Pattern p : {kUpper, kShortTail, kDense})
            bad += check(256 * tm - 128, 256 * tn - 192, 256 * tn - 192, p, pairs, 10, gen);
    for (int k = 0; k < 1500; ++k) {
      const int N = size(1, 9000), K = k % 2 ? N : size(1, 9000);
      bad += check(size(1, 9000), N, K, (Pattern)(k % 5), pairs, 1 + k % 11, gen);
    }
  }
  return bad != 0;
}
