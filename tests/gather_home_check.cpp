// Host check of a gridding plan whose visibility sort uses larger tiles than
// its gridding (csrc/gather_plan.cpp, home_T), no GPU needed: the sort and the
// degridding units are those of a plan with T = home_T, and every tile's list,
// taken back to the caller's indices, that of a plan with T alone, with the
// same keys, chunks and owner work.
//
// usage: gather_home_check L J T home_T M seed   (prints "ok" or the failure)
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <utility>
#include <vector>

#include "gather_plan.h"

using namespace purify;

#define CHECK(cond)                      \
  do {                                   \
    if (!(cond)) {                       \
      std::printf("FAIL %s\n", #cond);   \
      return 1;                          \
    }                                    \
  } while (0)

int main(int argc, char** argv) {
  if (argc != 7) return 2;
  const int L = std::atoi(argv[1]), J = std::atoi(argv[2]), T = std::atoi(argv[3]), HT = std::atoi(argv[4]);
  const int64_t M = std::atoll(argv[5]);
  std::mt19937_64 rng(std::strtoull(argv[6], nullptr, 10));
  std::uniform_int_distribution<int> cell(0, L - 1);
  std::vector<int> k0(2 * M);
  for (int64_t i = 0; i < M; ++i) {  // a third on one dense cell (several chunks), the rest uniform
    k0[2 * i] = i % 3 == 0 ? L - 2 : cell(rng);
    k0[2 * i + 1] = i % 3 == 0 ? 1 : cell(rng);
  }
  auto params = [&](int t, int home) {
    GatherPlanParams p{};
    p.M = M;
    p.L = L;
    p.J = J;
    p.T = t;
    p.home_T = home;
    p.entry_bytes = 8 + 4 * (2 * (J + 2) + 1);
    p.fixed_bytes = 16384 + ((t / 2) * (t / 2) + 1) * 4;
    p.smem_budget = 56 * 1024;
    p.tab_stride = ((t / 2) * (t / 2) + 1 + 7) / 8 * 8;
    p.max_partials = 32768;
    return p;
  };
  GatherPlan both, fine, home;
  CHECK(build_gather_plan(k0.data(), params(T, HT), both) == 0);
  CHECK(build_gather_plan(k0.data(), params(T, 0), fine) == 0);
  CHECK(build_gather_plan(k0.data(), params(HT, 0), home) == 0);
  CHECK(both.perm == home.perm && both.home == home.home);
  CHECK(both.dchunks.size() == home.dchunks.size());
  for (size_t q = 0; q < both.dchunks.size(); ++q)
    CHECK(both.dchunks[q].x == home.dchunks[q].x && both.dchunks[q].y == home.dchunks[q].y &&
          both.dchunks[q].z == home.dchunks[q].z);
  CHECK(both.list_off == fine.list_off && both.lkey == fine.lkey && both.tab == fine.tab);
  CHECK(both.items == fine.items && both.nchunk == fine.nchunk && both.chunk_max == fine.chunk_max);
  for (int t = 0; t < both.ntiles; ++t) {
    std::vector<std::pair<int, int>> a, b;
    for (int e = both.list_off[t]; e < both.list_off[t + 1]; ++e) {
      a.emplace_back(both.lkey[e], both.perm[both.list[e]]);
      b.emplace_back(fine.lkey[e], fine.perm[fine.list[e]]);
    }
    std::sort(a.begin(), a.end());
    std::sort(b.begin(), b.end());
    CHECK(a == b);
  }
  std::printf("ok\n");
  return 0;
}
