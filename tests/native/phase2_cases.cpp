// phase2_program on random product tries: walked the way the forward kernels walk it, every group
// ends on its own product and no slot is read before it is written.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>

#include "tami_internal.h"

using namespace tami;

int main(int argc, char** argv) {
  std::mt19937 rng(argc > 1 ? std::atoi(argv[1]) : 1);
  auto draw = [&](int n) { return (int)(rng() % (unsigned)n); };
  for (int t = 0; t < 2000; ++t) {
    const int n_cden = 1 + draw(t % 7 ? 5 : kMaxCplxDens), g2_const = draw(2), want = 1 + draw(20);
    std::vector<int> pnode, g2node(g2_const, -1);
    std::vector<std::vector<int>> path(n_cden);          // the factors of every value
    for (int c = 0; c < n_cden; ++c) path[c] = {c};
    std::map<std::pair<int, int>, int> child;
    std::map<int, int> used;
    for (int g = 0; g < want; ++g) {
      int v = draw(n_cden);
      for (int len = draw(5); len > 0 && (int)path.size() < n_cden + kMaxProdNodes; --len) {
        const int c = draw(n_cden);
        auto it = child.find({v, c});
        if (it == child.end()) {
          it = child.insert({{v, c}, (int)path.size()}).first;
          pnode.push_back(v);
          pnode.push_back(c);
          auto f = path[v];
          f.push_back(c);
          path.push_back(f);
        }
        v = it->second;
      }
      if (used.insert({v, g}).second) g2node.push_back(v);   // one group per product
    }
    const int n_g2 = (int)g2node.size(), n_pnode = (int)pnode.size() / 2;
    int n_live = -1;
    const std::vector<int> prog = phase2_program(n_cden, g2_const, n_g2, g2node.data(), pnode.data(), n_pnode, &n_live);
    if (n_live < 0 || n_live > n_pnode) { std::printf("FAIL %d: %d slots for %d products\n", t, n_live, n_pnode); return 1; }
    std::vector<std::vector<int>> val(n_cden + n_live), none;
    for (int c = 0; c < n_cden; ++c) val[c] = {c};
    std::vector<int> run;
    size_t p = 0;
    for (int g = g2_const; g < n_g2; ++g) {
      const int e = prog.at(p++), src = e & 0xffff;
      if (src != kP2Last) run = val.at(src);
      for (int k = e >> 16; k > 0; --k) {
        const int x = prog.at(p++), slot = x >> 8, c = x & 255;
        if (run.empty() || c >= n_cden || (slot && slot < n_cden)) { std::printf("FAIL %d: operand\n", t); return 1; }
        run.push_back(c);
        if (slot) val.at(slot) = run;
      }
      if (run != path[g2node[g]]) { std::printf("FAIL %d: group %d\n", t, g); return 1; }
    }
    if (p != prog.size()) { std::printf("FAIL %d: words left\n", t); return 1; }
  }
  std::printf("ok\n");
  return 0;
}
