// Work split of the windowed attention: which key tiles of which (stream, head, query-tile pair)
// each worker (a CTA, or a CTA pair) processes, and how the parts of an item that is split along
// its keys find each other.  Pure integer arithmetic, compiled for the host (launch set-up, the
// plan entry point and its CPU tests) and for the device (every role of the kernel walks the same
// sequence).
#pragma once

#include <stdint.h>

#include "common.h"

#if defined(__CUDACC__)
#define UNSTEP_HD __host__ __device__ __forceinline__
#else
#define UNSTEP_HD inline
#endif

namespace unstep {

constexpr int kTileM = 128;                 // queries per tile (two tiles per work item)
constexpr int kTileN = 128;                 // keys per tile
constexpr int kMinStepsPerWorker = 4;       // shortest share of the remainder that may cross items
constexpr int kMaxClusterParts = 8;         // largest portable cluster

struct AttnParams {
  int32_t Hn, L, T, C;
  int32_t q_tiles;          // ceil(L / 128)
  int32_t q_pairs;          // ceil(q_tiles / 2)
  int32_t tiles_per_frame;  // ceil(T / 128)
  int32_t flat;             // 1: key tiles run across frame boundaries inside a slot run
  int32_t n_streams;
  float scale_log2e;        // log2(e) / sqrt(128)
  int32_t items_per_stream; // Hn * q_pairs
  int32_t n_workers;        // workers of the launch (grid size, or clusters)
  int32_t full_rounds;      // whole rounds per stream, n_workers items each
  int32_t leftover;         // items per stream behind the whole rounds: the remainder
  int32_t parts;            // > 0: every item of the remainder is cut into this many parts, one per worker
  int32_t cluster;          // 1: the parts of an item are a cluster (no whole rounds, 2 <= parts <= kMaxClusterParts)
  int32_t n_active;         // parts == 0: workers that take a share of the remainder, >= 1
  int64_t all_steps;        // key tiles of all items of the launch
  int32_t narrow;           // 1: total_steps * n_active fits 32 bits, and so does every index of the shares
  int64_t total_steps;      // remainder: sum over the leftover items of their key tiles
  float* part;              // workspace: partial results of split items, kPartFloats per slot
  int* counters;            // workspace: arrivals per (item, query tile), zero between launches
  int* status;              // status word; with the extents below, for checking builds
  int32_t out_wide;         // 1: `out` is 32-byte aligned
  int64_t extent_out;       // 16-byte vectors of `out` that belong to this launch's streams
  int64_t extent_part;      // floats of `part`
  int64_t extent_counters;  // ints of `counters`
  int32_t sink;             // S: cache slots [0, S) hold frames [0, S) for good, the ring follows
  int32_t first_frame[kMaxStreamsPerLaunch];  // first frame of the recent part of stream b
  int32_t n_sink[kMaxStreamsPerLaunch];       // sink frames attended in front of the recent part
  int32_t tiles[kMaxStreamsPerLaunch];        // key tiles of one item of stream b
  // flat mode: the attended frames are at most three runs of consecutive cache slots (sink
  // prefix, ring up to its end, ring from its start); run r starts at cache row run_row0 and
  // has run_rows keys, its tiles are [run_tile_end[r-1], run_tile_end[r])
  int32_t run_row0[kMaxStreamsPerLaunch][3];
  int32_t run_rows[kMaxStreamsPerLaunch][3];
  int32_t run_tile_end[kMaxStreamsPerLaunch][3];
  int64_t step_base[kMaxStreamsPerLaunch];    // remainder steps of all streams before b
};

// One unit of work of a worker: key tiles [t0, t1) of item (b, h, query-tile pair qp).
struct Seg {
  int b, h, qp, nq, t0, t1;
  int tiles;             // key tiles of the whole item
  int item;              // item index inside the launch
  int64_t item_step0;    // remainder: step index of the item's first tile, with p.parts its first worker
  bool first_in_worker;  // this segment starts the worker's range
};

// Where key tile j of an item of stream b lives and how many of its 128 keys are real.
// Flat mode: tiles are cut from the runs of consecutive ring slots, so only the last tile of
// a run is ragged; it is fetched through the per-frame map, whose zero fill ends it cleanly at
// the end of its frame (a run ends on a frame end, and the ragged tile is shorter than a frame).
// Per-frame mode (frames shorter than a tile): every tile lies inside one frame.
struct TileInfo {
  int valid;      // real keys in the tile, 1..128
  bool framed;    // fetch through the (token, slot) map at (tok0, slot), else the flat map at row
  int row, slot, tok0;
};
UNSTEP_HD TileInfo tile_info(const AttnParams& p, int b, int j) {
  TileInfo t;
  if (p.flat) {
    int r = 0;
    if (j >= p.run_tile_end[b][0]) r = (j >= p.run_tile_end[b][1]) ? 2 : 1;
    const int t_begin = r == 0 ? 0 : p.run_tile_end[b][r - 1];
    const int tt = j - t_begin;
    const int rows = p.run_rows[b][r];
    const int row0 = p.run_row0[b][r];
    const int ntl = p.run_tile_end[b][r] - t_begin;
    const bool last = (tt == ntl - 1);
    t.valid = last ? rows - kTileN * tt : kTileN;
    t.framed = last;
    t.row = row0 + kTileN * tt;
    t.slot = (row0 + rows - 1) / p.T;
    t.tok0 = p.T - t.valid;
  } else {
    const int fi = j / p.tiles_per_frame;
    const int tt = j - fi * p.tiles_per_frame;
    t.valid = (tt == p.tiles_per_frame - 1) ? p.T - kTileN * tt : kTileN;
    t.framed = true;
    t.row = 0;
    // frame list = the attended sink frames, then the recent frames
    const int frame = fi < p.n_sink[b] ? fi : p.first_frame[b] + fi - p.n_sink[b];
    t.slot = frame < p.sink ? frame : p.sink + (frame - p.sink) % p.C;
    t.tok0 = kTileN * tt;
  }
  return t;
}

// Work split.  Items are ordered stream, head, query pair, so neighbouring workers work on the
// same head and share its K/V through L2.
//   1. Whole rounds: while a stream still has at least n_workers items, worker c takes item
//      (round * n_workers + c) whole.  All workers walk the key tiles in step, so a K/V tile is
//      fetched from HBM once and then hit in L2 by the other workers of the head.
//   2. Remainder: the leftover items of all streams (fewer than n_workers per stream), split along
//      their keys in one of two ways (plan_launch chooses):
//      - p.parts > 0: every item is cut into p.parts parts and each worker takes one of them (in a
//        launch without whole rounds the parts of an item may be a cluster of blocks: p.cluster);
//      - p.parts == 0: the items form one sequence of (item, key tile) steps, and each of the first
//        n_active workers takes an equal contiguous share of it (n_active <= total_steps, so no
//        share is empty and the workers that hold parts of an item are exactly those between the
//        owners of its first and last step).
//      The parts of an item are merged by whichever worker finishes last, or by its cluster.
struct Sched {
  int64_t lo, hi, cur;
  int b_round, round;   // position in the whole rounds
  int me;
  const AttnParams& p;
  // (a * b) / c; a 64-bit division takes several hundred clk, a chain of them was 2 us of the
  // epilogue of every part
  UNSTEP_HD static int64_t mul_div(const AttnParams& p, int64_t a, int64_t b, int64_t c) {
    if (p.narrow) return static_cast<uint32_t>(a) * static_cast<uint32_t>(b) / static_cast<uint32_t>(c);
    return a * b / c;
  }
  UNSTEP_HD static int64_t worker_lo(const AttnParams& p, int64_t c) {
    return c >= p.n_active ? p.total_steps : mul_div(p, p.total_steps, c, p.n_active);
  }
  UNSTEP_HD static int worker_of(const AttnParams& p, int64_t step) {
    int64_t c = mul_div(p, step, p.n_active, p.total_steps);
    while (c + 1 < p.n_active && worker_lo(p, c + 1) <= step) ++c;
    while (c > 0 && worker_lo(p, c) > step) --c;
    return static_cast<int>(c);
  }
  UNSTEP_HD Sched(const AttnParams& prm, int worker) : me(worker), p(prm) {
    if (p.parts > 0) {   // cur: the worker's part, hi: one past it
      lo = worker;
      hi = worker < static_cast<int64_t>(p.n_streams) * p.leftover * p.parts ? lo + 1 : lo;
    } else {
      lo = worker_lo(p, worker);
      hi = worker_lo(p, worker + 1);
    }
    cur = lo;
    b_round = 0;
    round = 0;
  }
  UNSTEP_HD void decode(Seg& s, int b, int in_stream) const {
    s.b = b;
    s.tiles = p.tiles[b];
    s.item = b * p.items_per_stream + in_stream;
    s.qp = in_stream % p.q_pairs;
    s.h = in_stream / p.q_pairs;
    s.nq = (2 * s.qp + 1 < p.q_tiles) ? 2 : 1;
  }
  UNSTEP_HD bool next(Seg& s) {
    while (b_round < p.n_streams) {          // whole rounds
      if (round < p.full_rounds) {
        decode(s, b_round, round * p.n_workers + me);
        s.t0 = 0;
        s.t1 = s.tiles;
        s.item_step0 = 0;
        s.first_in_worker = false;
        ++round;
        return true;
      }
      round = 0;
      ++b_round;
    }
    if (cur >= hi) return false;             // remainder
    if (p.parts > 0) {
      const int item = me / p.parts, part = me - item * p.parts;
      const int b = item / p.leftover;
      decode(s, b, p.full_rounds * p.n_workers + item - b * p.leftover);
      s.t0 = s.tiles * part / p.parts;   // remainder_parts keeps the products within 32 bits
      s.t1 = s.tiles * (part + 1) / p.parts;
      s.item_step0 = me - part;
      s.first_in_worker = true;
      cur = hi;
      return true;
    }
    int b = 0;
    while (b + 1 < p.n_streams && p.step_base[b + 1] <= cur) ++b;
    const int tiles = p.tiles[b];
    const int64_t rel = cur - p.step_base[b];
    const int left_item = static_cast<int>(mul_div(p, rel, 1, tiles));
    decode(s, b, p.full_rounds * p.n_workers + left_item);
    s.t0 = static_cast<int>(rel - static_cast<int64_t>(left_item) * tiles);
    const int64_t left = hi - cur;
    s.t1 = (left < tiles - s.t0) ? s.t0 + static_cast<int>(left) : tiles;
    s.item_step0 = cur - s.t0;
    s.first_in_worker = (cur == lo);
    cur += s.t1 - s.t0;
    return true;
  }
};

// Parts of a split item: the workers that own its first and its last step, and the scratch slot
// (0 or 1 of the two a worker has) in which worker c publishes its part of the item that starts
// at global step item_step0.
UNSTEP_HD int first_part_worker(const AttnParams& p, const Seg& s) {
  return p.parts > 0 ? static_cast<int>(s.item_step0) : Sched::worker_of(p, s.item_step0);
}
UNSTEP_HD int last_part_worker(const AttnParams& p, const Seg& s) {
  return p.parts > 0 ? static_cast<int>(s.item_step0) + p.parts - 1 : Sched::worker_of(p, s.item_step0 + s.tiles - 1);
}
UNSTEP_HD int part_slot(const AttnParams& p, int c, int64_t item_step0) {
  return p.parts > 0 || Sched::worker_lo(p, c) >= item_step0 ? 0 : 1;   // 0: the part starts the worker's range
}

// How the remainder (`items` of `least` to `most` key tiles, `steps` in all) is split: the number of
// parts per item, or 0 for `*shares` equal shares across the items.  Parts leave a worker with one
// part of one item; shares give the workers less to do, but each then holds parts of two items, one
// after the other, each with a hand-over, and an item falls into more parts.  The estimates (us)
// are fitted to launches of 2 to 40 items of 6 to 85 key tiles on a B200, with the pipeline of one S per query
// tile (the present one's are in cluster_parts): a step 1.6; a second part
// 3.4, each further one 1.6; shares 6 and 2.2 for each part of an item.  Measured, us: 8 items x 43
// steps 82 whole, 5 parts 33, 6 parts 31, 8 parts 33, 86 shares of 4 steps 35; 40 items x 16 steps 35
// whole, 3 parts 25, 148 shares 36; 80 items x 37 steps behind a whole round: shares.
inline int32_t remainder_parts(int64_t items, int64_t steps, int32_t least, int32_t most, int max_workers,
                               int32_t* shares) {
  int64_t n = steps / kMinStepsPerWorker;
  n = n < 1 ? 1 : (n > max_workers ? max_workers : n);
  *shares = static_cast<int32_t>(n);
  const double share = static_cast<double>((steps + n - 1) / n);
  double lowest = 1.6 * share + 6.0 + 2.2 * (static_cast<double>(steps) / static_cast<double>(items) / share + 1.0);
  int32_t best = 0;
  for (int32_t parts = 1; parts * items <= max_workers && parts <= least; ++parts) {
    if (static_cast<int64_t>(most) * parts > INT32_MAX) break;   // a part's bounds are 32-bit products
    const double cost = 1.6 * ((most + parts - 1) / parts) + (parts > 1 ? 3.4 + 1.6 * (parts - 2) : 0.0);
    if (cost < lowest) {
      lowest = cost;
      best = parts;
    }
  }
  return best;
}

// How many clusters of `parts` blocks a launch may have: all that the device runs at the same time, but of 3 and of 5
// three less (42 of 45, 23 of 26).  A launch that is set up under the kernel in front of it gets the SMs one by one as
// that one leaves, odd clusters are placed where three or five happen to be free, and the last ones found no place
// until the first had ended.  Append and attention of 13 key tiles, us, median: clusters of 3: 41 items 24.3, 42 26.3,
// 43 28.0, 44 35.2, 45 42.3; of 5: 23 20.3, 24 22.9, 25 25.9, 26 24.7.  Over other shapes 42 clusters of 3 are shorter than
// 42 of 2 (by 9 % on average, 6 % longer at worst), 44 longer; 24 and 25 of 5 are longer than those of 4.  Clusters of 2, 4,
// 6 and 8 never did that, up to 148 blocks, nor did those of 7, which are 105 blocks at most.
inline int32_t cluster_limit(const int32_t* clusters, int32_t parts) {
  return parts == 3 || parts == 5 ? clusters[parts] - 3 : clusters[parts];
}

// Parts that form a cluster, which merges them through shared memory: how many, or 0 where the split that
// remainder_parts chose (p.parts, p.n_active) is shorter.  clusters[n]: clusters of n blocks that the device runs at the
// same time (148 SMs: 74, 45, 33, 26, 22, 15, 15 of 2 to 8 blocks).  The estimates (us) are fitted to append and attention
// of 930 launches of 1 to 74 items of 2 to 183 key tiles, each split in every way.  With two query tiles an item, one in
// brackets: a step 1.35 (1.0), in frames of 65 to 127 tokens, whose tiles all take the masked code, 1.9 (1.4), in a cluster
// 4 % more; the merge of a cluster 4.1 (2.5) however many the parts, as each merges a share of the columns; through
// global memory 5.2 (4.1) and 1.3 (1.1) for each part beyond the second; either way 0.024 for each further block.
// Measured, us, global memory, whole or shares -> clusters: 8 items x 41 key tiles 26.0 -> 22.2, 20 x 40 31.6 -> 26.1, 40 x 41
// 42.0 -> 40.5, 52 x 40 45.6 -> 43.4, 2 items of a toy layer 14.1 -> 11.2.  Whole and shorter: 74 x 4 16.1, clusters of 2
// 21.4; 33 x 4 13.3, of 4 16.2; 41 of a toy layer x 3 10.4, of 3 12.6.  Through global memory and shorter, as a long
// part gains little by the merge: 70 x 183 162-186, of 2 174-207; 72 x 123 114-129, 122-142; 64 x 65 67.4, 71.3.  With one
// estimate for all (a step 1.6, a merge 2.5, nothing for a block) 19 % of the launches were slower than without clusters,
// by up to 33 %; 0.8 % are now, by up to 8 %, and all of them take 2 % less on average.
// That is the time of one launch.  The finer cut takes more SMs for it, and launches of several streams side by side
// lose where two no longer fit the device at once: per launch, us, 1 / 2 / 3 streams, parts through global memory
// -> clusters: 20 x 16 21.8 / 12.2 / 9.7 -> 18.4 / 13.9 / 13.7 (80 -> 120 blocks), 24 x 7 20.0 / 10.0 / 6.9 -> 15.4 / 10.0 /
// 9.0 (48 -> 96), 2 x 6 13.1 / 6.7 / 4.7 -> 10.2 / 5.3 / 3.7 (6 -> 12).  Streams that are served together go into one
// launch, so the line is drawn by the single launch.
inline int32_t cluster_parts(const AttnParams& p, int64_t items, int64_t steps, int32_t least, int32_t most,
                             const int32_t* clusters) {
  const bool lone = p.q_tiles == 1, masked = !p.flat && p.T > kTileN / 2;
  const double step = masked ? (lone ? 1.4 : 1.9) : (lone ? 1.0 : 1.35), block = 0.024 * static_cast<double>(items);
  double us;
  if (p.parts > 0) {
    us = step * ((most + p.parts - 1) / p.parts) +
         (p.parts > 1 ? (lone ? 4.1 : 5.2) + (lone ? 1.1 : 1.3) * (p.parts - 2) + block * (p.parts - 1) : 0.0);
  } else {
    const double share = static_cast<double>((steps + p.n_active - 1) / p.n_active);
    us = step * share + 6.0 + 2.2 * (static_cast<double>(steps) / static_cast<double>(items) / share + 1.0);
  }
  int32_t best = 0;
  for (int32_t parts = 2; parts <= kMaxClusterParts && parts <= least; ++parts) {
    if (items > cluster_limit(clusters, parts) || static_cast<int64_t>(most) * parts > INT32_MAX) continue;
    const double cost = 1.04 * step * ((most + parts - 1) / parts) + (lone ? 2.5 : 4.1) + block * (parts - 1);
    if (cost < us) {
      us = cost;
      best = parts;
    }
  }
  return best;
}

// Fills the per-launch part of `p` for streams [b0, b0 + nb): the attended frames of each stream
// cut into runs of consecutive cache slots, the key tiles, and the split of the work over at
// most `max_workers` workers.  The shape-wide fields (Hn, L, T, C, q_tiles, q_pairs,
// tiles_per_frame, flat, items_per_stream, sink) must already be set.  `clusters` as in cluster_parts;
// without it no part is in a cluster.  Host only.
inline int plan_launch(AttnParams& p, const unstep_shape_t* shape, const int32_t* start_frame, int nb,
                       int32_t window_frames, int32_t sink_frames, int32_t sink_attend, int max_workers,
                       const int32_t* clusters = nullptr) {
  p.n_streams = nb;
  for (int i = 0; i < nb; ++i) {
    const int hi = start_frame[i] + shape->chunk_frames;
    const int lo = hi - window_frames > 0 ? hi - window_frames : 0;
    const int n_sink = sink_attend < lo ? sink_attend : lo;   // sink frames not already in the recent part
    p.first_frame[i] = lo;
    p.n_sink[i] = n_sink;
    for (int r = 0; r < 3; ++r) p.run_row0[i][r] = p.run_rows[i][r] = p.run_tile_end[i][r] = 0;
    if (p.flat) {
      // walk the attended frames in order and cut them into runs of consecutive cache slots
      int n_runs = 0, prev_slot = -2;
      for (int k = 0; k < n_sink + hi - lo; ++k) {
        const int frame = k < n_sink ? k : lo + k - n_sink;
        const int slot = frame < sink_frames ? frame : sink_frames + (frame - sink_frames) % shape->ring_frames;
        if (slot != prev_slot + 1) {
          if (n_runs == 3) return UNSTEP_ERR_INVALID_ARG;  // cannot happen: sink, ring end, ring start
          p.run_row0[i][n_runs++] = slot * p.T;
        }
        p.run_rows[i][n_runs - 1] += p.T;
        prev_slot = slot;
      }
      int tiles = 0;
      for (int r = 0; r < 3; ++r) {
        tiles += (p.run_rows[i][r] + kTileN - 1) / kTileN;
        p.run_tile_end[i][r] = tiles;
      }
      p.tiles[i] = tiles;
    } else {
      p.tiles[i] = (n_sink + hi - lo) * p.tiles_per_frame;
    }
  }
  // One worker per SM where there are whole rounds for all of them; a launch of fewer items than
  // that is all remainder, and has the workers that the split asks for.
  const int64_t all_items = static_cast<int64_t>(nb) * p.items_per_stream;
  p.n_workers = max_workers;
  p.full_rounds = all_items > max_workers ? p.items_per_stream / max_workers : 0;
  p.leftover = p.items_per_stream - p.full_rounds * max_workers;
  int64_t steps = 0;
  p.all_steps = 0;
  int32_t least = INT32_MAX, most = 0;
  for (int i = 0; i < nb; ++i) {
    p.step_base[i] = steps;
    p.all_steps += static_cast<int64_t>(p.items_per_stream) * p.tiles[i];
    steps += static_cast<int64_t>(p.leftover) * p.tiles[i];
    least = p.tiles[i] < least ? p.tiles[i] : least;
    most = p.tiles[i] > most ? p.tiles[i] : most;
  }
  p.total_steps = steps;
  p.parts = 0;
  p.cluster = 0;
  p.n_active = 1;
  p.narrow = 1;
  if (steps > 0) {
    const int64_t items = static_cast<int64_t>(nb) * p.leftover;
    p.parts = remainder_parts(items, steps, least, most, max_workers, &p.n_active);
    if (clusters != nullptr && p.full_rounds == 0) {
      const int32_t parts = cluster_parts(p, items, steps, least, most, clusters);
      p.cluster = parts > 0;
      if (p.cluster) p.parts = parts;
    }
    p.narrow = steps * p.n_active <= INT32_MAX;
    if (p.full_rounds == 0) p.n_workers = p.parts > 0 ? static_cast<int32_t>(items) * p.parts : p.n_active;
  }
  return UNSTEP_OK;
}

// Shape-wide fields of the parameter block.
inline void plan_shape(AttnParams& p, const unstep_shape_t* shape, int32_t sink_frames) {
  const int64_t T = static_cast<int64_t>(shape->grid_h) * shape->grid_w;
  const int64_t L = T * shape->chunk_frames;
  p.sink = sink_frames;
  p.Hn = shape->heads;
  p.L = static_cast<int32_t>(L);
  p.T = static_cast<int32_t>(T);
  p.C = shape->ring_frames;
  p.q_tiles = static_cast<int32_t>((L + kTileM - 1) / kTileM);
  p.q_pairs = (p.q_tiles + 1) / 2;
  p.tiles_per_frame = static_cast<int32_t>((T + kTileN - 1) / kTileN);
  p.flat = (T >= kTileN) ? 1 : 0;  // a ragged tile must fit inside one frame
  p.scale_log2e = 1.4426950408889634f / 11.313708498984761f;   // log2(e) / sqrt(128)
  p.items_per_stream = p.Hn * p.q_pairs;
  p.part = nullptr;
  p.counters = nullptr;
  p.status = nullptr;
  p.extent_out = p.extent_part = p.extent_counters = 0;
}

// Argument checks shared by the attention entry points and the plan entry point (no device needed).
inline int check_attn_args(const unstep_shape_t* shape, const int32_t* start_frame, int32_t window_frames,
                           int32_t sink_frames, int32_t sink_attend) {
  const int rc = check_shape(shape, true);
  if (rc != UNSTEP_OK) return rc;
  if (start_frame == nullptr) return UNSTEP_ERR_INVALID_ARG;
  if (window_frames < shape->chunk_frames || window_frames > shape->ring_frames) return UNSTEP_ERR_INVALID_ARG;
  if (sink_frames < 0 || sink_frames > 4096 || sink_attend < 0 || sink_attend > sink_frames)
    return UNSTEP_ERR_INVALID_ARG;
  for (int b = 0; b < shape->batch; ++b)
    if (start_frame[b] < 0 || start_frame[b] > INT32_MAX - shape->chunk_frames) return UNSTEP_ERR_INVALID_ARG;
  const uint64_t C = static_cast<uint64_t>(shape->ring_frames) + sink_frames;
  const uint64_t T = static_cast<uint64_t>(shape->grid_h) * shape->grid_w;
  if (C * T >= (uint64_t(1) << 30)) return UNSTEP_ERR_INVALID_ARG;  // cache rows are 32-bit coordinates
  return UNSTEP_OK;
}

}  // namespace unstep
