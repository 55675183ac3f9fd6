// Goes through the schedules of attention launches (rf_attn_sched.cuh) on the host, for CTA counts
// from 1 to the most that a workspace is laid out for, and checks what the kernel relies on: every
// (item, KV tile) taken exactly once, a CTA's first unit not empty, partial slots inside the
// workspace and used once, the slots of an item listed in the order of its KV ranges, and both
// merge counters of every split item inside the counter area.
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>

#include "rf_attn_sched.cuh"

using namespace rf;

static const char* check(int A, int N, int H, int nkv, int G, int slots, int* kind) {
  const Sched s = make_sched(A, (N + 7) / 8 * 8, H, nkv, G, slots);
  const int T = s.pairs * H;
  *kind = s.even_q ? 2 : s.C > 1 ? 1 : 0;
  struct Range {
    int j0, j1, part, item;
  };
  std::vector<std::vector<Range>> items(T);
  std::vector<char> used(static_cast<size_t>(G) * std::max(slots, 1), 0);
  for (int w = 0; w < s.units; ++w) {
    const Unit u = get_unit(s, nkv, G, w);
    if (u.j0 >= u.j1) {
      if (u.pr != s.pairs) return "an empty share has a query tile";
      if (w < G) return "a CTA's first unit is empty";
      continue;
    }
    const int i = u.h * s.pairs + u.pr;
    if (u.pr < 0 || u.pr >= s.pairs || i < 0 || i >= T) return "an item out of range";
    if (u.j0 < 0 || u.j1 > nkv) return "KV tiles out of range";
    if (u.part < 0 ? u.j1 - u.j0 != nkv : u.part >= G * slots) return "a partial slot out of range";
    if (u.part >= 0 && used[u.part]++) return "a partial slot used twice";
    if (u.part >= 0 && (u.item < 0 || 2 * u.item + 1 >= kMaxGrid))
      return "a merge counter past the counter area";
    if (u.part >= 0 && s.even_q && u.j1 - u.j0 < kMinPiece) return "a piece too short";
    items[i].push_back({u.j0, u.j1, u.part, u.item});
  }
  for (auto& r : items) {
    std::sort(r.begin(), r.end(), [](const Range& a, const Range& b) { return a.j0 < b.j0; });
    int at = 0;
    for (const Range& x : r) {
      if (x.j0 != at) return "KV tiles missed or taken twice";
      at = x.j1;
    }
    if (at != nkv) return "KV tiles missed";
    if (r[0].part < 0) continue;
    for (const Range& x : r) {
      Unit u{};
      u.item = x.item;
      const Pieces p = item_pieces(s, nkv, G, u);
      if (p.n != static_cast<int>(r.size()) || p.n > kMaxSplit || (s.even_q && p.n > 5))
        return "wrong number of pieces";
      for (int c = 0; c < p.n; ++c)
        if (r[c].part != (c == 0 ? p.first : p.rest + c * p.stride))
          return "pieces out of the order of their KV ranges";
    }
  }
  return nullptr;
}

int main() {
  std::mt19937 rng(1);
  auto pick = [&](int lo, int hi) { return lo + static_cast<int>(rng() % (hi - lo + 1)); };
  const int grids[] = {152, 152, 152, 1, 2, 8, 132, 148, 160, 512, 513, 600, 1023, 1024};
  int n = 0, kinds[3] = {};
  while (n < 14000) {
    const int G = grids[n % 14], F = pick(1, 33), A = pick(0, F), H = pick(1, 48);
    const int N = n % 3 ? pick(1, 1600) : pick(1, 100);
    const long long pairs = (static_cast<long long>(A) * N / 128 + 2) / 2;
    if (pairs * H > 4000) continue;
    // the sequence may have other frames than the schedule's rows: any KV length
    const int nkv = n % 2 ? (F * N + 127) / 128 : pick(1, 400);
    int kind = 0;
    if (const char* what = check(A, N, H, nkv, G, n % 5 ? 2 : n % 2, &kind)) {
      std::printf("A=%d N=%d H=%d nkv=%d G=%d: %s\n", A, N, H, nkv, G, what);
      return 1;
    }
    ++n;
    ++kinds[kind];
  }
  if (std::min({kinds[0], kinds[1], kinds[2]}) < 500) {
    std::printf("too few of a kind: %d whole, %d in ranges, %d dealt evenly\n", kinds[0], kinds[1],
                kinds[2]);
    return 1;
  }
  std::printf("ok %d %d %d\n", kinds[0], kinds[1], kinds[2]);
  return 0;
}
