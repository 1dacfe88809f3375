// Host check of the number of CTAs that share a bare box (cg_team_rule), on 152 SMs.
// Prints "ok" and exits 0, or prints the mismatches and exits 1.
#include <cstdio>
#include <vector>

#include "../../paper_2208_06097_gb300/csrc/sea_internal.cuh"

static int bad = 0;
static std::vector<int> boxes(std::initializer_list<std::pair<int, int>> sets) {  // (edge, count)
  std::vector<int> e;
  for (auto s : sets)
    for (int k = 0; k < 3 * s.second; ++k) e.push_back(s.first);
  return e;
}
static void expect(const char* what, const std::vector<int>& ext, int team) {
  const int got = sea::cg_team_rule((int)ext.size() / 3, ext.data(), 152);
  if (got != team) {
    printf("%s: %d instead of %d\n", what, got, team);
    ++bad;
  }
}

int main() {
  // by the number of boxes, two places an SM
  expect("1 of 16", boxes({{16, 1}}), 8);
  expect("38 of 16", boxes({{16, 38}}), 8);
  expect("39 of 16", boxes({{16, 39}}), 4);
  expect("76 of 16", boxes({{16, 76}}), 4);
  expect("152 of 16", boxes({{16, 152}}), 2);
  expect("153 of 16", boxes({{16, 153}}), 1);
  // 25^3 points do not fit one CTA's shared memory: teams of four and more solve
  // them, smaller ones leave them to one CTA of an SM each
  expect("38 of 25", boxes({{25, 38}}), 8);
  expect("76 of 25", boxes({{25, 76}}), 4);
  expect("152 of 25", boxes({{25, 152}}), 1);
  expect("77 of 25", boxes({{25, 77}}), 1);
  // 40^3 points fit no team
  expect("1 of 40", boxes({{40, 1}}), 8);
  expect("19 of 40", boxes({{40, 19}}), 8);
  expect("38 of 40", boxes({{40, 38}}), 4);
  expect("64 of 40", boxes({{40, 64}}), 2);
  expect("100 of 40", boxes({{40, 100}}), 1);
  expect("one of 40 among 37 of 16", boxes({{16, 37}, {40, 1}}), 8);
  expect("20 of 40, 15 of 18", boxes({{40, 20}, {18, 15}}), 4);
  printf(bad ? "" : "ok\n");
  return bad != 0;
}
