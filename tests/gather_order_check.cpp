// Host check of the gridding plan's degridding order and of plans whose one
// tile is the whole grid (csrc/gather_plan.cpp), no GPU needed: the order holds
// every home tile's visibilities once, each in the run of the tile its first
// cell lies in, and summing the stored gather items' 2 x 2 contributions gives
// the scatter of every visibility's J x J footprint, wrapped at the grid's
// edges (§5: G sparse and fixed by the frequencies).
//
// usage: gather_order_check L J T home_T M seed   (prints "ok" or the failure)
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "gather_plan.h"

using namespace purify;

#define CHECK(cond)                    \
  do {                                 \
    if (!(cond)) {                     \
      std::printf("FAIL %s\n", #cond); \
      return 1;                        \
    }                                  \
  } while (0)

int main(int argc, char** argv) {
  if (argc != 7) return 2;
  const int L = std::atoi(argv[1]), J = std::atoi(argv[2]), T = std::atoi(argv[3]), HT = std::atoi(argv[4]);
  const int64_t M = std::atoll(argv[5]);
  std::mt19937_64 rng(std::strtoull(argv[6], nullptr, 10));
  std::uniform_int_distribution<int> cell(0, L - 1), val(-8, 8);
  std::vector<int> k0(2 * M);
  for (int64_t i = 0; i < M; ++i) {  // half uniform, half at the wrap-around edges
    k0[2 * i] = i % 2 ? cell(rng) : (L - J + cell(rng) % (2 * J)) % L;
    k0[2 * i + 1] = i % 2 ? cell(rng) : (L - J + cell(rng) % (2 * J)) % L;
  }
  const int NO = (T / 2) * (T / 2), W = T + J - 1, NT = kGridThreads;
  GatherPlanParams prm{};
  prm.M = M;
  prm.L = L;
  prm.J = J;
  prm.T = T;
  prm.home_T = HT;
  prm.entry_bytes = 8 + 4 * (2 * (J + 2) + 1);
  prm.fixed_bytes = 16384 + (NO + 1) * 4;
  prm.smem_budget = 56 * 1024;
  prm.tab_stride = (NO + 1 + 7) / 8 * 8;
  prm.max_partials = 32768;
  GatherPlan p;
  CHECK(build_gather_plan(k0.data(), prm, p) == 0);
  const int HD = L / HT, TD = L / T;

  // the degridding's order: a permutation of every home run
  CHECK((int64_t)p.dorder.size() == M && (int)p.home.size() == HD * HD + 1);
  for (int h = 0; h < HD * HD; ++h) {
    std::vector<int> run(p.dorder.begin() + p.home[h], p.dorder.begin() + p.home[h + 1]);
    std::sort(run.begin(), run.end());
    for (size_t q = 0; q < run.size(); ++q) {
      CHECK(run[q] == p.home[h] + (int)q);
      const int i = p.perm[run[q]];
      CHECK((k0[2 * i] / HT) * HD + k0[2 * i + 1] / HT == h);
    }
  }

  // the walk's meaning, in exact integers
  std::vector<long> wr(M * J), wc(M * J), v(M), scat((size_t)L * L, 0), gath((size_t)L * L, 0);
  for (auto* a : {&wr, &wc, &v})
    for (auto& x : *a) x = val(rng);
  for (int64_t i = 0; i < M; ++i)
    for (int a = 0; a < J; ++a)
      for (int b = 0; b < J; ++b)
        scat[(size_t)((k0[2 * i] + a) % L) * L + (k0[2 * i + 1] + b) % L] += wr[i * J + a] * wc[i * J + b] * v[i];
  for (size_t q = 0; q < p.chunks.size(); ++q) {
    const PlanI4 ch = p.chunks[q];
    const int Wt = p.tab[q * prm.tab_stride + NO], R0 = ch.x / TD * T, C0 = ch.x % TD * T;
    for (int j = 0; j < NT; ++j) {
      const int t0 = (int)(((int64_t)j * Wt + NT - 1) / NT), t1 = (int)(((int64_t)(j + 1) * Wt + NT - 1) / NT);
      for (int s = 0; s < t1 - t0; ++s) {
        const uint32_t it = p.items[(size_t)(p.item_row[q] + s) * NT + j];
        const int e = (int)(it & ((1u << kItemEntryBits) - 1)), ar = (int)((it >> 12) & 15u);
        const int bc = (int)((it >> 16) & 15u), o = (int)(it >> 20);
        CHECK(e < ch.z - ch.y && o < NO);
        CHECK(p.lkey[ch.y + e] >= 0 && p.lkey[ch.y + e] < W * W);
        const int i = p.perm[p.list[ch.y + e]];
        for (int a = 0; a < 2; ++a)
          for (int b = 0; b < 2; ++b) {
            const int ta = ar + a - 1, tb = bc + b - 1;  // unpadded taps
            if (ta < 0 || ta >= J || tb < 0 || tb >= J) continue;
            gath[(size_t)(R0 + 2 * (o / (T / 2)) + a) * L + C0 + 2 * (o % (T / 2)) + b] +=
                wr[i * J + ta] * wc[i * J + tb] * v[i];
          }
      }
    }
  }
  CHECK(gath == scat);
  std::printf("ok\n");
  return 0;
}
