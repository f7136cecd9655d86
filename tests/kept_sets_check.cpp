// Host-only check of dfacto::KeptSets (csrc/kept_sets.h): what is kept goes back
// to the context it came from only, in bounded numbers, and to one taker each.
// Prints one line per check; exits non-zero if one failed.
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

#include "kept_sets.h"

static int fails = 0;
#define CHECK(cond)                                  \
  do {                                               \
    const bool ok = (cond);                          \
    std::printf("%s: %s\n", ok ? "ok" : "FAIL", #cond); \
    fails += !ok;                                    \
  } while (0)

int main() {
  using Kept = dfacto::KeptSets<int>;
  Kept k;
  int v = 0;
  CHECK(!k.take(1, &v));
  CHECK(k.give(1, 11) && k.give(2, 21) && k.give(1, 12));
  // another context of the same device, or the one after a reset, gets none of them
  CHECK(!k.take(3, &v));
  CHECK(k.take(2, &v) && v == 21);
  CHECK(!k.take(2, &v));
  int a = 0, b = 0;
  CHECK(k.take(1, &a) && k.take(1, &b) && a + b == 23 && a != b);
  CHECK(!k.take(1, &v));
  // bounds: per context, and in all
  size_t kept = 0;
  for (int i = 0; i < 100; ++i) kept += k.give(5, i);
  CHECK(kept == Kept::kPerContext);
  for (uint64_t c = 10; c < 1000; ++c) kept += k.give(c, 0);
  CHECK(kept == Kept::kInAll);
  // eight threads take and give: every set is held by one of them at a time
  Kept t;
  std::vector<std::atomic<int>> held(8);
  for (int i = 0; i < 8; ++i) t.give(7, i);
  std::atomic<int> clashes{0};
  std::vector<std::thread> th;
  for (int i = 0; i < 8; ++i)
    th.emplace_back([&] {
      for (int j = 0; j < 20000; ++j) {
        int s;
        if (!t.take(7, &s)) continue;
        if (held[s].fetch_add(1) != 0) ++clashes;
        held[s].fetch_sub(1);
        if (!t.give(7, s)) ++clashes;
      }
    });
  for (auto& x : th) x.join();
  CHECK(clashes == 0);
  std::printf(fails ? "FAILED %d\n" : "ALL OK\n", fails);
  return fails ? 1 : 0;
}
