// light_first and tree_order (csrc/tree_order.h) on random forests, caterpillars, stars and
// complete trees of up to 255 links: prints per shape the links, the stack depth in the order
// the library stores, and 1 if the order is a permutation in depth-first preorder whose
// children come by subtree size, smallest first.
#include <cstdio>
#include <random>

#include "../paper_2109_07719_gb300/csrc/tree_order.h"

using namespace abasim;
static std::mt19937 rng(7);

static void check(const std::vector<int>& par) {
  const int n = (int)par.size();
  const std::vector<int> light = light_first(par.data(), n);
  std::vector<int> at(n, -1), p2(n), size(n, 1);
  for (int l = 0; l < n; ++l) at[light[l]] = l;
  bool ok = true;
  for (int l = 0; l < n; ++l) ok &= at[l] >= 0;
  for (int l = 0; l < n; ++l) {
    p2[l] = par[light[l]] >= 0 ? at[par[light[l]]] : -1;
    ok &= p2[l] < l;
  }
  const TreeOrder to = tree_order(p2.data(), n);
  for (int l = 0; l < n; ++l) ok &= to.perm[l] == l;  // already in depth-first preorder
  for (int l = n - 1; l >= 0; --l)
    if (p2[l] >= 0) size[p2[l]] += size[l];
  std::vector<int> last(n, 0);
  for (int l = 0; l < n; ++l)
    if (p2[l] >= 0) {
      ok &= size[l] >= last[p2[l]];
      last[p2[l]] = size[l];
    }
  std::printf("%d %d %d\n", n, to.depth, ok ? 1 : 0);
}

int main() {
  for (int n : {1, 2, 3, 7, 15, 63, 127, 255}) {
    std::vector<int> chain, star, comb, binary, ternary;
    for (int i = 0; i < n; ++i) {
      chain.push_back(i - 1);
      star.push_back(i ? 0 : -1);
      comb.push_back(i == 0 ? -1 : i % 2 ? (i < 3 ? 0 : i - 2) : i - 1);
      binary.push_back(i ? (i - 1) / 2 : -1);
      ternary.push_back(i ? (i - 1) / 3 : -1);
    }
    for (auto* s : {&chain, &star, &comb, &binary, &ternary}) check(*s);
    for (int t = 0; t < 20; ++t) {
      std::vector<int> forest;
      for (int i = 0; i < n; ++i) forest.push_back((int)(rng() % (i + 1)) - 1);
      check(forest);
    }
  }
}
