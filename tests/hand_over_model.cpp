// Every order in which four softmax warps and their issuing warp can meet the named barriers of the
// attention kernel, with every wait giving up or not: can one of them be left at a barrier for good?
//
//   hand_over_model TILES SEGMENT     key tiles of the group, tiles between two group barriers
//
// prints for each rule: name, reachable states, states in which nobody can go on although not all are done.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <set>
#include <tuple>
#include <vector>

#include "handover.h"

struct Rule {   // which barrier (0 or 1) belongs to a tile, and whether a warp that gave up waits there
  const char* name;
  int (*barrier)(uint32_t tile);
  bool (*waits)(bool gave_up);
};

static const Rule kRules[] = {
    {"kernel",
     [](uint32_t t) { return unstep::p_ready_barrier(0, t) == unstep::p_ready_barrier(0, 0) ? 0 : 1; },
     [](bool g) { return unstep::p_ready_waits(g); }},
    // two that leave somebody behind
    {"one_barrier_arrive", [](uint32_t) { return 0; }, [](bool) { return false; }},
    {"one_barrier_wait", [](uint32_t) { return 0; }, [](bool g) { return g; }}};

enum Stage : int8_t { kWaitS, kAtP, kEpilogue, kAtGroup };   // kAtP, kAtGroup: waiting at a barrier
struct Warp {
  int8_t tile = 0, stage = kWaitS, gave = 0;
  bool operator<(const Warp& o) const { return std::tie(tile, stage, gave) < std::tie(o.tile, o.stage, o.gave); }
};
struct State {
  Warp w[4];
  int8_t tile = 0, at_p = 0, ok = 1;   // issuer: next hand-over, waiting there, no wait gave up yet
  int8_t passed = 0;                   // hand-overs behind which it issued: P V of the tile and the next S
  int8_t count[2] = {0, 0}, group = 0; // arrivals at the barriers
  bool operator<(const State& o) const {
    for (int i = 0; i < 4; ++i)
      if (w[i] < o.w[i] || o.w[i] < w[i]) return w[i] < o.w[i];
    return std::tie(tile, at_p, ok, passed, count[0], count[1], group) <
           std::tie(o.tile, o.at_p, o.ok, o.passed, o.count[0], o.count[1], o.group);
  }
};

static int n_tiles, segment;

static void next_tile(Warp& w) {   // behind the hand-over of a tile: the segment's epilogue, or the next tile
  ++w.tile;
  w.stage = w.tile % segment == 0 || w.tile == n_tiles ? kEpilogue : kWaitS;
}

// One arrival at P barrier b; the fifth completes the phase and lets everybody who waits there go on.
static void arrive(State& s, const Rule& r, int b) {
  if (++s.count[b] < 5) return;
  s.count[b] = 0;
  for (Warp& w : s.w)
    if (w.stage == kAtP && r.barrier(w.tile) == b) next_tile(w);
  if (s.at_p && r.barrier(s.tile) == b) {
    s.at_p = 0;
    if (s.ok) s.passed = s.tile + 1;
    ++s.tile;
  }
}

static std::vector<State> successors(const State& s, const Rule& r) {
  std::vector<State> out;
  for (int i = 0; i < 4; ++i) {
    const Warp& w = s.w[i];
    const bool waiting = (w.stage == kWaitS && w.tile < n_tiles) || w.stage == kEpilogue;
    if (!waiting) continue;
    if (!w.gave) {   // the wait in front of it (S of the tile, the last P V) may always run out
      out.push_back(s);
      out.back().w[i].gave = 1;
    }
    if (w.stage == kWaitS && (w.gave || s.passed >= w.tile)) {
      State t = s;
      const int b = r.barrier(w.tile);
      if (r.waits(w.gave)) t.w[i].stage = kAtP;
      else next_tile(t.w[i]);
      arrive(t, r, b);
      out.push_back(t);
    } else if (w.stage == kEpilogue && (w.gave || s.passed >= w.tile)) {
      State t = s;
      t.w[i].stage = kAtGroup;
      if (++t.group == 4) {
        t.group = 0;
        for (Warp& x : t.w) {
          if (x.stage == kAtGroup) x.stage = kWaitS;
          if (s.w[0].gave || s.w[1].gave || s.w[2].gave || s.w[3].gave) x.gave = 1;   // the group's vote
        }
      }
      out.push_back(t);
    }
  }
  if (s.tile < n_tiles && !s.at_p) {
    if (s.ok) {
      out.push_back(s);
      out.back().ok = 0;
    }
    State t = s;
    t.at_p = 1;
    arrive(t, r, r.barrier(s.tile));
    out.push_back(t);
  }
  for (State& t : out) std::sort(t.w, t.w + 4);   // the four warps are alike
  return out;
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  n_tiles = atoi(argv[1]);
  segment = atoi(argv[2]);
  for (const Rule& r : kRules) {
    std::set<State> seen;
    std::vector<State> todo = {State()};
    seen.insert(State());
    size_t blocked = 0;
    while (!todo.empty()) {
      const State s = todo.back();
      todo.pop_back();
      const std::vector<State> next = successors(s, r);
      bool done = s.tile == n_tiles && s.group == 0;
      for (const Warp& w : s.w) done = done && w.tile == n_tiles && w.stage == kWaitS;
      if (done ? (s.count[0] != 0 || s.count[1] != 0) : next.empty()) ++blocked;
      for (const State& t : next)
        if (seen.insert(t).second) todo.push_back(t);
    }
    printf("%s %zu %zu\n", r.name, seen.size(), blocked);
  }
  return 0;
}
