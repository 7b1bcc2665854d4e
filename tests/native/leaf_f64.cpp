// The float64 leaf under every kind of warp order: the factor and the inverse have to be those of the block,
// bit for bit the same whatever the order.
#include "simt_cpu.h"

#include "leaf_f64.cuh"

#include <random>

int main() {
  using namespace omm::dev;
  std::mt19937 gen(5);
  std::normal_distribution<double> normal;
  std::vector<std::vector<int>> orders(2);
  constexpr int kWarps = kLeaf64Threads / 32;
  for (int w = 0; w < kWarps; ++w) {
    orders[0].push_back(w);
    orders[1].push_back(kWarps - 1 - w);
  }
  for (int k = 0; k < 3; ++k) {
    orders.push_back(orders[0]);
    std::shuffle(orders.back().begin(), orders.back().end(), gen);
  }
  int bad = 0;
  for (int b : {1, 5, 8, 9, 24, 31, 32, 33, 40, 57, 63, 64}) {
    std::vector<double> B(b * b), A(b * b), first;
    for (double& x : B) x = normal(gen) / std::sqrt(b);
    for (int i = 0; i < b; ++i)
      for (int j = 0; j < b; ++j) {
        A[i * b + j] = i == j ? 0.5 : 0.0;
        for (int k = 0; k < b; ++k) A[i * b + j] += B[i * b + k] * B[j * b + k];
      }
    for (size_t o = 0; o < orders.size(); ++o) {
      std::vector<double> L = A, X(b * b, -7.0);
      int info = 0;
      simt::run(kLeaf64Threads, orders[o], [&] { leaf_f64_body(L.data(), b, b, X.data(), b, &info, 0); });
      double eL = 0.0, eX = 0.0;
      for (int i = 0; i < b; ++i)
        for (int j = 0; j < b; ++j) {
          double ll = 0.0, lx = 0.0;
          for (int k = 0; k < b; ++k) {
            ll += L[i * b + k] * L[j * b + k];
            lx += L[i * b + k] * X[k * b + j];
          }
          eL = std::max(eL, std::fabs(ll - A[i * b + j]));
          eX = std::max(eX, std::fabs(lx - (i == j ? 1.0 : 0.0)));
        }
      std::vector<double> all = L;
      all.insert(all.end(), X.begin(), X.end());
      if (first.empty()) first = all;
      // Cholesky and triangular inverse: at most b u |L| |L^T| and b u |L| |L^-1|, |A| <= 5, |A^-1| <= 2
      if (info != 0 || !(eL <= b * 5.0 * 2.3e-16) || !(eX <= b * 8.0 * 2.3e-16) || all != first) {
        std::printf("b = %d, order %zu: info %d, |L L^T - A| %.1e, |L X - 1| %.1e, %s\n", b, o, info, eL, eX,
                    all == first ? "same bits" : "other bits than the first order");
        ++bad;
      }
    }
  }
  return bad != 0;
}
