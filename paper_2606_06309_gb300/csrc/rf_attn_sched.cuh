// rf_attn_sched.cuh -- the schedule of an attention launch: which query tiles and KV tiles each CTA
// takes, and where the partial results of split items lie.  Integer arithmetic only, the same on
// the device and on the host, where a test goes through it.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define RF_HD __host__ __device__ __forceinline__
#else
#define RF_HD inline
#endif

namespace rf {

constexpr int BM = 128;       // query rows per tile
constexpr int BN = 128;       // keys per KV tile
constexpr int kMaxSplit = 16;          // KV ranges per split item
// KV tiles per piece where the tail is dealt out evenly, at least: a merge costs about as much as
// the KV steps of that many tiles.  Equal ranges may be as short as one tile.  At least four tiles
// there too are faster on short sequences (4 x 64 tokens x 2 heads x 64 8.1 us instead of 10.8,
// 8 x 200 x 2 x 128 23.5 instead of 29.2), but further from the exact result: the largest
// probability of every range is exactly 1 in bf16, so fewer ranges round more of the
// probabilities (error of 48 drawn shapes 1.04 times as large, 1.09 at most).
constexpr int kMinPiece = 4;
constexpr int kMaxGrid = 1024;  // the workspace has this many counters, and slots for as many CTAs

// The schedule every role derives identically from the active count on the device.
struct Sched {
  int R, tiles, pairs;  // active rows (padded per frame), query tiles and tile pairs per head
  int T_full;           // items processed whole
  int C;                // KV ranges per item of the split tail (1: no split)
  uint32_t even_q, even_r;  // tail dealt out evenly: its KV tiles / CTAs, the remainder (0: not)
  int units;            // T_full + tail items * C, or + 2 per CTA (some empty) when dealt evenly
};

// One unit of work: a tile pair of one head over KV tiles [j0, j1).
struct Unit {
  int h, pr, j0, j1;
  int part;  // split: partial slot, else -1
  int item;  // split: tail item index
};

// How the last, partly idle round of items is shared out (unmasked launches with a workspace),
// chosen by the KV tiles that the busiest CTA then processes:
//   whole        nkv
//   C ranges     nkv / C + kSplitCost, C = CTAs / items: every item in equal ranges, one per CTA
//   dealt evenly tail * nkv / CTAs + kEvenCost: every CTA takes the same share of the tail's KV
//                tiles, which may end in one item and begin the next (two partial slots per CTA)
// The costs are the boundary of a further unit and the merge, in KV tiles (dealt evenly, the
// partials of all items are written and read: 34 MB each way for 100 items on 152 CTAs, 10 us).
// Dealing evenly is considered where C ranges leave CTAs idle: more than a quarter as many items as
// CTAs (below, the items' ranges fill the chip and an item would be in more than five pieces).
// Measured (us per launch, whole or in C ranges -> dealt evenly): 13 x 1560 tokens x 1 head x 128
// (80 items) 186 -> 122; 9 of the 13 frames active (55 items) 107 -> 93; 7 x 1003 x 5 x 128, 5
// active (100 items of 55 tiles) 70.3 -> 66.9.
constexpr int kSplitCost = 3, kEvenCost = 10;
constexpr uint32_t kMinEvenShare = 12;  // KV tiles per CTA
// KV tile, counted over the whole tail, where CTA k's share begins; no piece is shorter than
// kMinPiece.
RF_HD uint32_t even_bound(const Sched& s, int nkv, int k, int G) {
  // (fits 32 bits: the tail has fewer items than CTAs, and make_sched checks CTAs * nkv)
  const uint32_t v = k * s.even_q + k * s.even_r / static_cast<uint32_t>(G);
  const uint32_t rem = v % static_cast<uint32_t>(nkv);
  if (rem < kMinPiece) return v - rem;
  return nkv - rem < kMinPiece ? v + (nkv - rem) : v;
}

// A active frames of Np rows (padded), H heads, nkv KV tiles, G CTAs; `slots` partial slots per CTA
// in the workspace, 0: the launch does not split.
RF_HD Sched make_sched(int A, int Np, int H, int nkv, int G, int slots) {
  Sched s;
  s.R = A * Np;
  s.tiles = (s.R + BM - 1) / BM;
  s.pairs = (s.tiles + 1) / 2;
  const int T = s.pairs * H;
  s.T_full = T;
  s.C = 1;
  s.even_q = s.even_r = 0;
  if (T > 0 && slots > 0) {
    const int rounds = (T + G - 1) / G;
    const int tail = T - (rounds - 1) * G;
    int c = G / tail;
    if (c > kMaxSplit) c = kMaxSplit;
    if (c > nkv) c = nkv;
    const int busiest = c >= 2 ? (nkv + c - 1) / c + kSplitCost : nkv;
    // (two merge counters per tail item: in C ranges there are at most G of them)
    if (slots == 2 && 4 * tail > G && 2 * tail <= kMaxGrid &&
        static_cast<uint32_t>(nkv) <= 0xFFFFFFFFu / G) {
      const uint32_t all = static_cast<uint32_t>(tail) * nkv, q = all / G;
      if (q >= kMinEvenShare && static_cast<int>(q) + 1 + kEvenCost < busiest) {
        s.T_full = (rounds - 1) * G;
        s.even_q = q;
        s.even_r = all % G;
        s.units = s.T_full + 2 * G;
        return s;
      }
    }
    if (c >= 2) {
      s.T_full = (rounds - 1) * G;
      s.C = c;
    }
  }
  s.units = s.T_full + (T - s.T_full) * s.C;
  return s;
}

RF_HD Unit get_unit(const Sched& s, int nkv, int G, int w) {
  Unit u;
  int item;
  u.part = -1;
  u.item = -1;
  if (w < s.T_full) {
    item = w;
    u.j0 = 0;
    u.j1 = nkv;
  } else if (s.even_q != 0) {
    // the CTA's share of the tail: what is left of the item it begins in, then the start of the
    // next one (perhaps nothing: j1 = 0).  A share is shorter than an item.
    int k = w - s.T_full;
    const bool second = k >= G;
    if (second) k -= G;
    const uint32_t lo = even_bound(s, nkv, k, G), hi = even_bound(s, nkv, k + 1, G);
    const uint32_t first = lo / static_cast<uint32_t>(nkv);
    const uint32_t begin = first * nkv, end = begin + nkv;
    if (!second) {
      u.item = static_cast<int>(first);
      u.j0 = static_cast<int>(lo - begin);
      u.j1 = static_cast<int>((hi < end ? hi : end) - begin);
    } else {
      u.item = static_cast<int>(first) + 1;
      u.j0 = 0;
      u.j1 = hi > end ? static_cast<int>(hi - end) : 0;
    }
    item = s.T_full + u.item;
    if (u.j1 - u.j0 < nkv) u.part = 2 * k + second;
  } else {
    const int k = w - s.T_full;
    const int ti = k / s.C, c = k - ti * s.C;
    item = s.T_full + ti;
    // 32-bit arithmetic on purpose (c <= 16, nkv < 2^24): a 64-bit divide here slowed the
    // single MMA-issuing thread by ~10% even on launches that never split
    u.j0 = (c * nkv) / s.C;
    u.j1 = ((c + 1) * nkv) / s.C;
    u.part = k;
    u.item = ti;
  }
  u.h = item / s.pairs;
  u.pr = item - u.h * s.pairs;
  if (u.j0 >= u.j1) u.pr = s.pairs;  // an empty share: neither query tile exists
  return u;
}

// The partial slots of a split item, in the order of their KV ranges: slot `first`, then
// `rest + c * stride` for c = 1 .. n - 1.
struct Pieces {
  int n, first, rest, stride;
};
RF_HD Pieces item_pieces(const Sched& s, int nkv, int G, const Unit& u) {
  if (s.even_q == 0) return Pieces{s.C, u.item * s.C, u.item * s.C, 1};
  // the CTAs whose shares meet the item: from the last that begins at or before it ...
  const uint32_t begin = static_cast<uint32_t>(u.item) * nkv, end = begin + nkv;
  int k0 = static_cast<int>(static_cast<float>(begin) /
                            (static_cast<float>(s.even_q) +
                             static_cast<float>(s.even_r) / static_cast<float>(G)));
  if (k0 > G - 1) k0 = G - 1;
  while (k0 > 0 && even_bound(s, nkv, k0, G) > begin) --k0;
  while (even_bound(s, nkv, k0 + 1, G) <= begin) ++k0;
  // ... to the first that ends at or after its end
  int k1 = k0;
  while (even_bound(s, nkv, k1 + 1, G) < end) ++k1;
  const bool second = even_bound(s, nkv, k0, G) < begin;  // its share began in the item before
  return Pieces{k1 - k0 + 1, 2 * k0 + second, 2 * k0, 2};
}

}  // namespace rf
