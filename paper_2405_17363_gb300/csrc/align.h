// Host-side alignment of an SpMV schedule's row ends (used once per pattern
// and lane count when a handle first needs it).
//
// sched::build (schedule.h) fixes the order of every row's entries, which
// fixes the row sum's bits; which lane runs a row, and in which slots, is
// free.  In its own layout some lane ends a row in almost every slot, so the
// product must store and reset its running sum conditionally after every
// multiply-add, and that select sits on the FP64 chain.  Here the rows are
// packed again, into the same number of slots per lane, so that all lanes
// end their rows in a few common slots (8 to 11 of 36 at 80 rows on 16 lanes):
// the kernels run the others as bare multiply-adds.
//
// The common slots are found by a seeded random search over sets of m
// positions; for each set the lanes are packed one after the other by a
// small dynamic program (maximise the entries covered).  A row shorter than
// its run of slots is led by padding slots: A = 0 times a column of the row
// itself, so the sum still starts from +0 and a non-finite value reaches the
// row only if the row multiplies it anyway.  The gathers' bank conflicts,
// which sched::build keeps low, rise to about two wavefronts per half-warp;
// exchanging rows of one length to lower them again measured no gain (the FP64
// unit, not shared memory, bounds these kernels).
#pragma once
#include <algorithm>
#include <array>
#include <vector>

#include "schedule.h"

namespace camp {
namespace sched {

// The entries of every row in their order: row r multiplies the CSR entries
// entry[start[r] .. start[r + 1]), whose columns are col[...].
struct RowChains {
  std::vector<int> start, entry, col;
  int len(int r) const { return start[r + 1] - start[r]; }
};

// A row's place: lane, and the slots [from, to) it may use (the row takes the
// last ones).
struct Place { int lane, from, to; };

inline unsigned next_random(unsigned &s) {
  s = s * 1664525u + 1013904223u;
  return s >> 8;
}

// Pack rows of the given length counts (cnt[l] rows of l entries, l <= longest)
// into Lc lanes whose rows end at slots pos[1..m] (pos[0] = 0).  Returns the
// rows left over; with out, the places by length.
inline int pack_rows(std::vector<int> cnt, int rows, int Lc, const std::vector<int> &pos,
                     std::vector<std::vector<Place>> *out) {
  const int m = (int)pos.size() - 1, longest = (int)cnt.size() - 1;
  std::vector<int> fit(pos[m] + 1), to(m + 1), take(m + 1);
  std::vector<float> value(m + 1);
  for (int lane = 0; lane < Lc && rows > 0; ++lane) {
    int c = 0;
    for (int s = 0; s <= pos[m]; ++s) {
      if (s <= longest && cnt[s]) c = s;
      fit[s] = c;  // the longest row left that fits s slots
    }
    value[m] = 0.0f;
    for (int i = m - 1; i >= 0; --i) {
      value[i] = value[i + 1];
      to[i] = i + 1;
      take[i] = 0;
      for (int j = i + 1; j <= m; ++j) {
        const int room = pos[j] - pos[i], l = fit[room];
        if (l == 0) continue;
        // entries covered, long rows first, less what padding wastes
        const float v = value[j] + l + 0.002f * l * l - 0.3f * (room - l);
        if (v > value[i]) {
          value[i] = v;
          to[i] = j;
          take[i] = l;
        }
        if (room >= longest) break;
      }
    }
    for (int i = 0; i < m; i = to[i]) {
      int l = take[i];
      while (l > 0 && !cnt[l]) --l;  // the lane itself took the last row of that length
      if (l == 0) continue;
      --cnt[l];
      --rows;
      if (out) (*out)[l].push_back(Place{lane, pos[i], pos[to[i]]});
    }
  }
  return rows;
}

// Align the rows of `ch` (n rows) on Lc lanes in at most max_slots slots per
// lane.  On success word and entry receive the slots [slot][lane] (the host
// form of sched::build; padding: entry -1) and the slots per lane are
// returned; 0 if no layout was found (the caller keeps its own).
inline int align(int n, const RowChains &ch, int Lc, int max_slots, std::vector<unsigned> &word,
                 std::vector<int> &entry) {
  int longest = 0;
  for (int r = 0; r < n; ++r) longest = std::max(longest, ch.len(r));
  const int nnz = ch.start[n];
  const int fewest = std::max((nnz + Lc - 1) / Lc, longest);
  // large products gain little from aligned ends, and the search grows
  if (max_slots > 32 * kEndWords || n > 512) return 0;
  std::vector<int> cnt(longest + 1, 0);
  for (int r = 0; r < n; ++r) ++cnt[ch.len(r)];
  unsigned seed = 12345u;
  std::vector<int> found;
  const int m0 = (n + Lc - 1) / Lc;  // rows of a lane
  int tries = 480;  // bounds the search for patterns that have no such layout
  for (int L = fewest; L <= max_slots && found.empty(); ++L)
    for (int m = std::min(L, m0 + 3); m <= std::min(L, m0 + 9) && found.empty(); m += 2) {
      std::vector<int> base, pos;
      int best = n + 1;
      for (int t = 0; t < 40 && found.empty() && tries > 0; ++t, --tries) {
        std::vector<char> is(L + 1, 0);
        if (base.empty() || next_random(seed) % 10 == 0) {
          for (int c = 0; c < m - 1;) {
            const int x = 1 + (int)(next_random(seed) % (unsigned)(L - 1));
            if (!is[x]) {
              is[x] = 1;
              ++c;
            }
          }
        } else {  // move one end by one or two slots
          for (int i = 1; i < m; ++i) is[base[i]] = 1;
          if (m > 1) {
            static const int step[4] = {-2, -1, 1, 2};
            const int i = 1 + (int)(next_random(seed) % (unsigned)(m - 1));
            const int x = base[i] + step[next_random(seed) % 4];
            if (x < 1 || x >= L || is[x]) continue;
            is[base[i]] = 0;
            is[x] = 1;
          }
        }
        pos.assign(1, 0);
        for (int x = 1; x < L; ++x)
          if (is[x]) pos.push_back(x);
        pos.push_back(L);
        const int left = pack_rows(cnt, n, Lc, pos, nullptr);
        if (left <= best) {
          best = left;
          base = pos;
        }
        if (left == 0) found = pos;
      }
    }
  if (found.empty()) return 0;
  const int L = found.back();
  std::vector<std::vector<Place>> places(longest + 1);
  pack_rows(cnt, n, Lc, found, &places);
  std::vector<std::vector<int>> rows(longest + 1);
  for (int r = 0; r < n; ++r) rows[ch.len(r)].push_back(r);
  word.assign((size_t)L * Lc, 0u);
  entry.assign((size_t)L * Lc, -1);
  std::vector<int> used(Lc, 0);
  for (int l = 1; l <= longest; ++l)
    for (size_t i = 0; i < rows[l].size(); ++i) {
      const Place &p = places[l][i];
      const int r = rows[l][i], s = ch.start[r];
      used[p.lane] = std::max(used[p.lane], p.to);
      for (int j = p.from; j < p.to; ++j) {
        const int q = j - (p.to - l);
        const size_t t = (size_t)j * Lc + p.lane;
        word[t] = (unsigned)ch.col[q < 0 ? s : s + q] | ((unsigned)r << 11) |
                  (q == l - 1 ? kEnd : 0u);
        entry[t] = q < 0 ? -1 : ch.entry[s + q];
      }
    }
  // a lane's idle slots before its next row lead that row (its first column);
  // those past its last row read a column another lane reads
  for (int q = 0; q < Lc; ++q) {
    unsigned next = 0u;
    bool have = false;
    for (int j = L - 1; j >= 0; --j) {
      unsigned &w = word[(size_t)j * Lc + q];
      if (entry[(size_t)j * Lc + q] >= 0 || (w >> 11)) {
        next = w & ~kEnd;
        have = true;
      } else if (have) {
        w = next;
      }
    }
    for (int j = used[q]; j < L; ++j)
      for (int x = 0; x < Lc; ++x)
        if (entry[(size_t)j * Lc + x] >= 0) {
          word[(size_t)j * Lc + q] = word[(size_t)j * Lc + x] & 0x7ffu;
          break;
        }
  }
  return L;
}

}  // namespace sched
}  // namespace camp
