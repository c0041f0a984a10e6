// Launch plans: how the work of a call is cut over a device of `sms` SMs.  Host
// arithmetic without CUDA, from sizes alone, so that it can be checked on its
// own; times in the comments were measured on a GB300 (152 SMs).
#pragma once

#include <algorithm>
#include <cstdint>

namespace rolekv {

// Score ----------------------------------------------------------------------

// Key tiles of a cell, the unit in which a SnapKV chunk's row statistics are
// joined and, in small batches, split over CTAs.  The statistics of a row are
// joined cell by cell in both cases, so the scores do not depend on the split.
constexpr int kCellTiles = 4;

constexpr int kMeetingTiles = 7;   // cost of an item's start and meeting, in key tiles
constexpr int kJoinTiles = 3;      // and of joining a cut chunk's cells

// CTAs a chunk is cut into: the number of parts whose rounds of items cost
// least, in key tiles: a part's own, seven for its start and meeting, three
// more for the join of a cut chunk's cells.  8 units of 64 tiles: one CTA each
// 84 us, sixteen 19 us; 160 units: two rounds of whole chunks 172 us, five of
// quarters 143 us; 256 units: two rounds 176 us, seven of quarters 203 us; 76
// units of 9 tiles: whole 29 us, halves 31 us.  (Packed batches, whose chunks
// differ in length, are cut only while one round holds them.)
inline int score_parts(bool varlen, int64_t units, int n_chunks, int chunk_tiles, int sms) {
  const int cells = (chunk_tiles + kCellTiles - 1) / kCellTiles;
  const int64_t chunks = units * n_chunks;
  int parts = 1;
  if (chunks > 4 * static_cast<int64_t>(sms)) return parts;
  int64_t best = INT64_MAX;
  for (int x = 1; x <= cells && x * n_chunks <= sms; ++x) {
    const int64_t grid = sms / (n_chunks * x) * (n_chunks * x);
    const int64_t rounds = (chunks * x + grid - 1) / grid;
    if (x > 1 && rounds > 1 && (varlen || x > 8)) break;
    const int64_t tiles = std::min((cells + x - 1) / x * kCellTiles, chunk_tiles);
    const int64_t cost = rounds * (tiles + kMeetingTiles + (x > 1 ? kJoinTiles : 0));
    if (cost < best) {
      best = x == 1 ? cost - cost / 32 : cost;     // (whole chunks unless 3% dearer)
      parts = x;
    }
  }
  return parts;
}

// Decode ---------------------------------------------------------------------

constexpr int kDecodeRowsPerSplit = 1024;
constexpr int kDecodeSplitCost = 320;       // rows a CTA could stream while one starts and ends

// Rows of a split: a unit's splits are equal in length, a multiple of the
// kernel's 64-row stage, so that they finish together.  fine: as long as makes
// the fewest rows pass one after another through an SM's CTAs (whole waves of
// CTAs, and their starts); otherwise about kDecodeRowsPerSplit rows, which
// they never pass (a warp's sums would get longer, their error larger).  8
// units x 819 rows: 16.2 us in one split each, 6.7 us in seven; 32 x 3277 rows
// 17.5 and 12.5 us; 8 x 131072 163 and 100 us.  Of start costs 40 to 320 rows
// the last is best where the splits differ (256 x 820 rows 25.4 us, 26.4 at 80).
// heads: layers x KV heads, of sequences with m_max rows (varlen: at most
// m_max, `total` together).
inline int64_t decode_split_rows(bool varlen, int64_t heads, int64_t b, int64_t m_max, int64_t total, int d,
                                 int G, bool fine, int sms) {
  const int64_t ns = m_max > 0 ? (m_max + kDecodeRowsPerSplit - 1) / kDecodeRowsPerSplit : 1;
  int64_t r = (m_max + ns - 1) / ns;
  r = r > 0 ? (r + 63) / 64 * 64 : 64;
  if (!fine) return r;
  // CTAs resident at once: limited by their two stages of shared memory, or
  // with eight heads' sums at d = 64 by their registers (counted as six, 152
  // units of 3277 rows took 38.4 us against 33.2).  Packed splits leave their
  // slots one by one, and six suits them (23.7 us for 32 of 5 to 13 thousand
  // rows, 25.6 counted as five).
  const int64_t slots = static_cast<int64_t>(sms) * (d == 128 ? 3 : G > 4 && !varlen ? 5 : 6);
  int64_t best = INT64_MAX;
  for (int64_t x = 128; x <= kDecodeRowsPerSplit; x += 64) {
    int64_t cost;
    if (varlen) {
      // splits of many lengths (half a split more per sequence on average):
      // the rows and starts of a slot, and half a split until the last ends
      const int64_t ctas = heads * (x >= m_max ? b : total / x + (b + 1) / 2);
      cost = (heads * total + ctas * kDecodeSplitCost) / slots + (x + kDecodeSplitCost) / 2;
      // (one split each needs no merge: 512 rows of 1 to 300, 13.2 us against 14.2)
      if (x >= m_max) cost -= cost / 16;
    } else {
      const int64_t ctas = heads * b * ((m_max + x - 1) / x);
      cost = (ctas + slots - 1) / slots * (x + kDecodeSplitCost);
    }
    if (cost <= best) {
      best = cost;
      r = x;
    }
    if (x >= m_max) break;
  }
  return r;
}

// Quest ----------------------------------------------------------------------

constexpr int kQuestCtasPerSm = 3;
constexpr int kQuestWarps = 8;           // warps of a CTA, each taking whole pages
constexpr int kQuestLoads = 8 * 32;      // 16-byte loads a warp has in flight

struct QuestSplit {
  int64_t ctas, pages;                   // CTAs of the longest unit, pages of each
};

// CTAs per unit: the cut that takes least time by this account, in ns.  A CTA
// starts with the window mean (4 us and 1 us for 64 rows); then each of its
// warps takes every eighth page, 0.8 us and another 0.8 for each batch of
// loads of a page; the CTAs resident at once share 7 TB/s.  Dense units go in
// whole waves; packed ones, of many lengths, follow each other without gaps,
// and half a CTA passes until the last one ends.  64 units of 2048 16-token
// pages: 8 CTAs a unit are 1.12 waves (116 us), 7 just under one (84 us, 81 at
// the copy rate).  With keys alone counted (500 of them for a start), 300
// units of 1500 one-token pages took one CTA each, 245 us against 187 with
// three; 256 units of 32 64-token pages three, 31 us against 26 with one;
// 256 units of eight 512-token pages three, 72 us against 48; one packed unit
// of 65536 one-token pages at most 64, 127 us against 36 with 384.
// heads: layers x KV heads, of b sequences of n_max tokens (varlen: at most
// n_max, T together); rows: of the window, over the group's heads.
inline QuestSplit quest_split(bool varlen, int64_t heads, int64_t b, int64_t n_max, int64_t T, int64_t page,
                              int64_t rows, int d, int sms) {
  const int64_t slots = static_cast<int64_t>(sms) * kQuestCtasPerSm;
  const int64_t units = heads * b;
  const int64_t pages = (n_max + page - 1) / page;
  const int64_t start = 4000 + rows * 16;
  const int64_t page_ns = 800 * (1 + (page * (d / 8) + kQuestLoads - 1) / kQuestLoads);
  const auto stream_ns = [&](int64_t keys) { return keys * 2 * d / 7000; };   // at 7 TB/s
  // (the streams and the warps' turns hold each other up a little)
  const auto longer = [](int64_t x, int64_t y) { return std::max(x, y) + std::min(x, y) / 8; };
  const auto cost = [&](int64_t per) {
    const int64_t warp = (per + kQuestWarps - 1) / kQuestWarps * page_ns;
    if (varlen && b > 1) {
      const int64_t all = stream_ns(heads * T);
      const int64_t n = std::max(units, heads * (T / std::min(per * page, n_max) + (b + 1) / 2));
      if (n <= slots) return start + longer(all, warp);
      return std::max(all + start, n * (start + warp) / slots) + (start + warp) / 2;
    }
    const int64_t cut = (pages + per - 1) / per, n = units * cut, last = n % slots;
    return n / slots * (start + longer(stream_ns(slots * n_max / cut), warp)) +
           (last > 0 ? start + longer(stream_ns(last * n_max / cut), warp) : 0);
  };
  int64_t best = INT64_MAX, per = pages;
  const auto consider = [&](int64_t p) {
    p = p < 1 ? 1 : (p < pages ? p : pages);
    const int64_t c = cost(p);
    if (c < best) {
      best = c;
      per = p;
    }
  };
  // The CTAs of 1, 2, ... waves, and as many pages more as its warps take in
  // the same number of turns.
  const int64_t all_pages = varlen && b > 1 ? heads * ((T + page - 1) / page) : units * pages;
  const int64_t first = (units + slots - 1) / slots;
  for (int64_t w = first; w < first + 12; ++w) {
    int64_t p;
    if (varlen && b > 1) {
      const int64_t ctas = w * slots - heads * ((b + 1) / 2);   // less the sequences' short last ones
      p = ctas > 0 ? (all_pages + ctas - 1) / ctas : pages;
    } else {
      p = (pages + w * slots / units - 1) / (w * slots / units);
    }
    // (CTAs with an SM each to themselves are not joined for that)
    if (all_pages > p * sms) consider((p + kQuestWarps - 1) / kQuestWarps * kQuestWarps);
    consider(p);
    if (p <= 1) break;
  }
  consider(pages);
  return {(pages + per - 1) / per, per};
}

// Selection ------------------------------------------------------------------

// Longest row whose keys one CTA holds in shared memory.
constexpr int kSmemMaxN = 40960;

// How a unit's row is held.
enum { kOne = 0, kCluster = 1, kStream = 2 };

struct SelectRoute {
  int mode, ranks, threads;   // ranks: CTAs per unit (the cluster size)
  int groups;                 // groups (of four slots) a rank's memory holds
  bool wide;                  // the long rows' digits and list
};

#ifdef __CUDACC__
__host__ __device__
#endif
inline int plan_groups(int groups, int ranks) {
  return ((groups + ranks - 1) / ranks + 31) & ~31;
}

// Threads and memory of a unit on `ranks` CTAs.  Threads: enough for a short
// latency while the SMs hold all units, no more than leave room for several
// units on an SM otherwise (1024 x 8192 tokens: 60.7 us at 256 threads, 66.7
// at 512; 8 x 8192: 18.9 and 15.9; 304 CTAs of 512 threads fit: 320 x 2628
// 17.4 and 21.9, 560 x 6844 42 and 55).  One CTA of a row beyond 16384 tokens
// has 1024 from the first token on while each has an SM (16385 tokens, 38
// units 21.4 us, 23.9 at 512; 300 units 41.9 and 33.3).
inline SelectRoute select_shape(int n_max, int64_t units, int sms, int mode, int ranks) {
  SelectRoute r{mode, ranks, 0, plan_groups((n_max + 3 + 3) / 4, ranks), false};   // up to three leading slots
  const int slots = r.groups * 4;                  // of one rank
  r.wide = mode == kStream || slots > 16384 + 128 || (mode == kOne && n_max > 16384 && units <= sms);
  r.threads = r.wide ? 1024
              : slots > 8192 + 128 || (slots > 2048 + 128 && units <= 2 * static_cast<int64_t>(sms)) ? 512
                                                                                                     : 256;
  return r;
}

// Route of a call, by the row length and the number of units.  A unit on one
// CTA is bound by its serial phases (set-up, quotas, digit searches: 8 us for
// the shortest row) and by its passes over shared memory (about 6 us per 8192
// tokens at 1024 threads); a cluster divides the passes but pays some 1 us per
// exchange, eight of them: 18.4 us at 8192 tokens against 15.9 us for one CTA
// of 512 threads.  Clusters run in waves of as many as the device holds:
// held(route, alone) of them, alone with an SM for each CTA (a GPC's last SMs
// hold none: 36 of four CTAs, 15 of eight; 74 of four at 512 threads, two CTAs
// on an SM; 0 on a device too small for one).  Times, role quotas, pool 7,
// B = 0.1, of one CTA or streaming and of the cluster:
//   36 and 38 units x 20000   22.0 and 22.0; cluster of 4 22.1 and 24.0 us
//   38 units x 28000, 32768   26.1 and 28.3; 27.2 and 28.6 (GLOBAL 29.4 and
//                             33.2; 26.1 and 27.2)
//   74 and 76 x 40961, 65536  44.3 and 57.7; 34.8 and 54.8, 40.1 and 62.2
//   36, 72, 76 x 100000       81.8; 34.6, 66.9, 97.4 (one to three waves)
//   14, 16 x 150000           114.7; of 8 38.1 and 70.5, of 4 41.2 and 41.0
//   14, 26, 38 x 262144       189; of 8 45.0, 86.7, 128
// so: up to kSmemMaxN tokens clusters with an SM for each CTA, above 28672
// also those that share; beyond, of four CTAs one wave of 512 threads or two
// of 1024; above 131136 tokens of eight while they fit one wave, or three
// where four ranks hold no more.  (Three waves of four at 131072 tokens suit
// GLOBAL, 115 us against 125, and cost the other policies as much.)
template <class Held>
inline SelectRoute select_route(int n_max, int64_t units, int sms, Held held) {
  const auto waves = [&](const SelectRoute& r, bool alone, int64_t most) {
    return held(r, alone) * most >= units;
  };
  if (n_max <= kSmemMaxN) {
    if (n_max > 16384 && units <= sms / 4) {
      const SelectRoute r = select_shape(n_max, units, sms, kCluster, 4);
      if (waves(r, n_max <= 28672, 1)) return r;
    }
    return select_shape(n_max, units, sms, kOne, 1);
  }
  const SelectRoute four = select_shape(n_max, units, sms, kCluster, 4);
  const SelectRoute eight = select_shape(n_max, units, sms, kCluster, 8);
  const bool fits4 = n_max <= 4 * kSmemMaxN;
  if (n_max > 4 * 32768 + 64 && waves(eight, true, fits4 ? 1 : 3)) return eight;
  if (fits4 && waves(four, false, four.wide ? 2 : 1)) return four;
  return select_shape(n_max, units, sms, kStream, 1);
}

}  // namespace rolekv
