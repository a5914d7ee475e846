// Host-side bookkeeping of MergeAndReduce (Algorithm 3): which SoftmaxBalance calls fire,
// where their t input rows live and where their t/2 survivors go.  Pure integer code, no
// CUDA calls, so it can be exercised without a device.
//
// Per stream the arena holds one region per level:
//   level 0      : linear buffer [start0, start0+len0) of uncompressed rows (C^0 + window)
//   level 1..T-1 : 2t rows; the set C^l is empty or holds one half (t/2 rows) at base 0 or t
//   level T      : C^T, appended to for ever
// A batch may contain many consecutive blocks of a stream; survivors that will be consumed
// again inside the same batch travel through two shared ping-pong pools instead of the
// small per-level regions (pool (l & 1) receives level-l survivors, two halves per slot).
#pragma once

#include <algorithm>
#include <climits>
#include <cstdint>
#include <utility>
#include <vector>

#include "common.cuh"

namespace bkv {

struct StreamState {
  int64_t appended = 0;                  // tokens ever appended to C^0
  int64_t pending = 0;                   // tokens appended since the last compress
  int32_t start0 = 0, len0 = 0;          // level-0 segment
  int32_t lvl_len[kMaxLevels + 1] = {};  // rows held at levels 1..T
  int32_t lvl_base[kMaxLevels + 1] = {}; // base (0 or t) of the half held at levels 1..T-1
  int64_t calls_done[kMaxLevels + 1] = {};  // calls run per level (= next call ordinal)
  bool same_as(const StreamState& o) const {
    bool eq = appended == o.appended && pending == o.pending && start0 == o.start0 && len0 == o.len0;
    for (int l = 0; l <= kMaxLevels; ++l)
      eq = eq && lvl_len[l] == o.lvl_len[l] && lvl_base[l] == o.lvl_base[l] && calls_done[l] == o.calls_done[l];
    return eq;
  }
};

struct Layout {
  int32_t t = 0, T = 0, W = 0;
  int64_t R = 0;                          // rows per stream
  int32_t region_off[kMaxLevels + 1] = {};
  int32_t cap0 = 0, capT = 0;
  int64_t pool_row[2] = {0, 0};           // first arena row of each pool
  int64_t pool_pairs = 0;                 // slots (of t rows) per pool
};

struct Plan {
  std::vector<std::vector<CallDesc>> levels;  // [T] calls per level, launch order
  std::vector<MoveDesc> moves;
  std::vector<SegUpdate> segs;
  int max_move_rows = 0;
};

// Blocks of t eligible tokens that are ready in C^0 (the newest W tokens are not eligible).
inline int64_t ready_blocks(const Layout& Lo, const StreamState& S) {
  const int64_t eligible = std::max<int64_t>(0, S.appended - Lo.W);
  return eligible / Lo.t - S.calls_done[0];
}

// Plans every call that `runs` (stream, number of level-0 blocks) triggers, level by level.
// Returns false if a pool would overflow (the caller sizes batches so that it cannot).
inline bool plan_batch(const Layout& Lo, StreamState* st, const std::vector<std::pair<int, int>>& runs, Plan& P) {
  const int t = Lo.t, T = Lo.T, half = t / 2;
  P.levels.assign(T, {});
  P.moves.clear(); P.segs.clear(); P.max_move_rows = 0;
  struct Cur { int stream; std::vector<int64_t> src; };
  std::vector<Cur> cur;
  for (const auto& run : runs) {
    const int s = run.first, nb = run.second;
    if (nb <= 0) continue;
    StreamState& S = st[s];
    Cur c{s, {}};
    const int64_t base = (int64_t)s * Lo.R + Lo.region_off[0] + S.start0;
    for (int k = 0; k < nb; ++k) c.src.push_back(base + (int64_t)k * t);
    S.start0 += nb * t;
    S.len0 -= nb * t;
    cur.push_back(std::move(c));
  }
  for (int l = 0; l < T; ++l) {
    int64_t pool_next = 0;
    std::vector<Cur> nxt;
    for (auto& c : cur) {
      StreamState& S = st[c.stream];
      const int n = (int)c.src.size();
      if (n == 0) continue;
      const int64_t sb = (int64_t)c.stream * Lo.R;
      Cur nc{c.stream, {}};
      if (l + 1 == T) {
        for (int k = 0; k < n; ++k) {
          CallDesc d{};
          d.src_row = c.src[k];
          d.dst_row = sb + Lo.region_off[T] + S.lvl_len[T] + (int64_t)k * half;
          d.dbg_off = -1; d.stream = c.stream; d.ordinal = (int32_t)S.calls_done[l]++;
          P.levels[l].push_back(d);
        }
        S.lvl_len[T] += n * half;
      } else {
        const int h = S.lvl_len[l + 1] ? 1 : 0;     // a half is already waiting in C^{l+1}
        const int slots = h + n, pairs = slots / 2, left = slots % 2;
        const int64_t pers = sb + Lo.region_off[l + 1];
        const int old_base = S.lvl_base[l + 1];
        const int new_base = h ? (old_base ? 0 : t) : 0;
        const int pool_pairs_needed = pairs - (h && pairs > 0 ? 1 : 0);
        if (pool_next + pool_pairs_needed > Lo.pool_pairs) return false;
        for (int k = 0; k < n; ++k) {
          const int j = h + k, pr = j / 2, within = j % 2;
          CallDesc d{};
          d.src_row = c.src[k];
          if (pr < pairs) {
            if (h && pr == 0) d.dst_row = pers + old_base + half;
            else d.dst_row = Lo.pool_row[l & 1] + (pool_next + pr - h) * (int64_t)t + (int64_t)within * half;
          } else {
            d.dst_row = pers + new_base;
          }
          d.dbg_off = -1; d.stream = c.stream; d.ordinal = (int32_t)S.calls_done[l]++;
          P.levels[l].push_back(d);
        }
        for (int pr = 0; pr < pairs; ++pr) {
          if (h && pr == 0) nc.src.push_back(pers + old_base);
          else nc.src.push_back(Lo.pool_row[l & 1] + (pool_next + pr - h) * (int64_t)t);
        }
        pool_next += pool_pairs_needed;
        S.lvl_len[l + 1] = left ? half : 0;
        S.lvl_base[l + 1] = left ? new_base : 0;
      }
      nxt.push_back(std::move(nc));
    }
    cur.swap(nxt);
  }
  for (const auto& run : runs) {
    const int s = run.first;
    if (run.second <= 0) continue;
    StreamState& S = st[s];
    const int64_t r0 = (int64_t)s * Lo.R + Lo.region_off[0];
    if (S.len0 == 0) {
      S.start0 = 0;
    } else if (S.start0 >= S.len0) {
      P.moves.push_back(MoveDesc{r0 + S.start0, r0, s, S.len0});
      P.max_move_rows = std::max(P.max_move_rows, (int)S.len0);
      S.start0 = 0;
    }
    const int32_t sbase = s * (T + 1);
    P.segs.push_back(SegUpdate{sbase, S.start0, S.len0, 0});
    for (int l = 1; l < T; ++l) P.segs.push_back(SegUpdate{sbase + l, S.lvl_base[l], S.lvl_len[l], 0});
    P.segs.push_back(SegUpdate{sbase + T, 0, S.lvl_len[T], 0});
  }
  return true;
}

// The same for lockstep streams -- all of them in state S, each running its nb ready blocks: one CallSet per level in
// place of lists, the state after the batch (S is updated), the move of the remainder (E) and the segments of a stream.
// The caller keeps n_streams * nb within the level-0 calls that the pools are sized for.
inline void plan_lockstep(const Layout& Lo, StreamState& S, int nb, int layer, int first, std::vector<CallSet>& sets,
                          std::vector<int>& n_calls, BatchEnd& E, Seg* seg) {
  const int t = Lo.t, T = Lo.T, half = t / 2;
  sets.assign(T, CallSet{});
  n_calls.assign(T, 0);
  int n = nb, src_rel = Lo.region_off[0] + S.start0, src_held = 0, src_pairs = 0;
  int64_t src_pool = -1;
  S.start0 += nb * t;
  S.len0 -= nb * t;
  for (int l = 0; l < T && n > 0; ++l) {
    CallSet& C = sets[l];
    n_calls[l] = n;
    C.layer = layer; C.first = first; C.per_stream = n; C.ordinal0 = (int32_t)S.calls_done[l];
    C.src_rel = src_rel; C.src_held = src_held; C.src_pool = src_pool; C.src_pairs = src_pairs;
    S.calls_done[l] += n;
    if (l + 1 == T) {
      C.top = 1;
      C.dst_rel = Lo.region_off[T] + S.lvl_len[T];
      S.lvl_len[T] += n * half;
      break;
    }
    const int h = S.lvl_len[l + 1] ? 1 : 0;       // a half is already waiting in C^{l+1}
    const int slots = h + n, pairs = slots / 2, left = slots % 2;
    const int pers = Lo.region_off[l + 1], old_base = S.lvl_base[l + 1];
    const int new_base = h ? (old_base ? 0 : t) : 0;
    C.dst_held = h;
    C.dst_held_rel = pers + old_base + half;
    C.dst_left_rel = pers + new_base;
    C.dst_pairs_all = pairs;
    C.dst_pairs = pairs - (h && pairs > 0 ? 1 : 0);
    C.dst_pool = Lo.pool_row[l & 1];
    src_rel = pers + old_base; src_held = h; src_pool = C.dst_pool; src_pairs = C.dst_pairs;
    n = pairs;
    S.lvl_len[l + 1] = left ? half : 0;
    S.lvl_base[l + 1] = left ? new_base : 0;
  }
  E = BatchEnd{layer, first, 0, 0};
  if (S.len0 == 0) {
    S.start0 = 0;
  } else if (S.start0 >= S.len0) {
    E.move_src = S.start0;
    E.move_rows = S.len0;
    S.start0 = 0;
  }
  seg[0] = Seg{S.start0, S.len0};
  for (int l = 1; l < T; ++l) seg[l] = Seg{S.lvl_base[l], S.lvl_len[l]};
  seg[T] = Seg{0, S.lvl_len[T]};
}

// Streams per batch of n lockstep streams with nb blocks each, at most `most` (>= 1) per batch: the split with the fewest
// waves of `slots` CTAs over all launches (a launch of 6.9 waves takes as long as one of 7).
inline int lockstep_batch(int n, int nb, int T, int most, int slots) {
  auto waves = [&](int streams) {
    int64_t w = 0, calls = (int64_t)streams * nb;
    for (int l = 0; l < T && calls > 0; ++l, calls = (int64_t)streams * (nb >> l)) w += (calls + slots - 1) / slots;
    return w;
  };
  if (n <= most) return n;
  int best = most;
  int64_t best_w = INT64_MAX;
  for (int b = most; b >= std::max(1, most / 2); --b) {
    const int64_t w = (int64_t)(n / b) * waves(b) + (n % b ? waves(n % b) : 0);
    if (w < best_w) { best_w = w; best = b; }
  }
  return best;
}

}  // namespace bkv
