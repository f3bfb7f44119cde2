// Every order in which the softmax warps and the two issuing warps of the attention kernel can meet the
// named barriers of S and P, with every wait giving up or not: can one of them be left there for good?
//
//   score_hand_over_model TILES SEGMENT GROUPS WARPS   key tiles per group, tiles between two epilogues, groups
//                                                      (query tiles), warps per group (the kernel has four)
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

static int n_tiles, segment, n_groups, n_warps;

struct Rule {
  const char* name;
  bool two;             // two barriers of a kind per group, or one
  bool gave_up_waits;   // a warp that gave up waits at the barriers (the kernel's rule), or only arrives there too
  int s_free(int a, int tile) const { return unstep::s_free_barrier(a, two ? tile : 0); }
  int p_ready(int a, int tile) const { return unstep::p_ready_barrier(a, two ? tile : 0); }
  bool waits(bool gave_up) const { return gave_up_waits && unstep::p_ready_waits(gave_up); }
};

enum Stage : int8_t { kWaitS, kAtS, kWaitPv, kAtP, kEpilogue, kAtGroup };   // kAt*: waiting at a barrier
struct Warp {
  int8_t tile = 0, stage = kWaitS, gave = 0;
  auto key() const { return std::tie(tile, stage, gave); }
  bool operator<(const Warp& o) const { return key() < o.key(); }
};
struct Issuer {   // steps through the (tile, group) pairs; `good`: how many it issued before a wait of its own gave up
  int8_t step = 0, at = 0, ok = 1, good = 0;
  auto key() const { return std::tie(step, at, ok, good); }
};
struct State {
  Warp w[2][4];
  Issuer qk, pv;
  int8_t count[16] = {};
  std::vector<int8_t> flat() const {
    std::vector<int8_t> v;
    for (auto& g : w)
      for (const Warp& x : g) v.insert(v.end(), {x.tile, x.stage, x.gave});
    for (const Issuer* i : {&qk, &pv}) v.insert(v.end(), {i->step, i->at, i->ok, i->good});
    v.insert(v.end(), count, count + 16);
    return v;
  }
};
static int group_of(int step) { return step % n_groups; }
static int tile_of(int step) { return step / n_groups; }
static int step_of(int a, int tile) { return tile * n_groups + a; }
static int steps() { return n_tiles * n_groups; }

static void issue(Issuer& i) {
  if (i.ok) i.good = i.step + 1;
  ++i.step;
}
static void behind_p(Warp& w) {
  ++w.tile;
  w.stage = w.tile % segment == 0 || w.tile == n_tiles ? kEpilogue : kWaitS;
}
static void arrive(State& s, const Rule& r, int b) {
  const bool group = b < unstep::kPReadyBarrier;
  if (++s.count[b] < n_warps + (group ? 0 : 1)) return;
  s.count[b] = 0;
  for (int a = 0; a < n_groups; ++a) {
    bool any = false;
    for (int k = 0; k < n_warps; ++k) any = any || s.w[a][k].gave;
    for (int k = 0; k < n_warps; ++k) {
      Warp& w = s.w[a][k];
      if (w.stage == kAtS && r.s_free(a, w.tile) == b) w.stage = kWaitPv;
      else if (w.stage == kAtP && r.p_ready(a, w.tile) == b) behind_p(w);
      else if (w.stage == kAtGroup && unstep::kGroupBarrier + a == b) {
        w.stage = kWaitS;
        if (any) w.gave = 1;   // the group's vote
      }
    }
  }
  if (s.qk.at && r.s_free(group_of(s.qk.step - 1), tile_of(s.qk.step - 1)) == b) {
    s.qk.at = 0;
    issue(s.qk);   // the next Q K^T, or the end
  } else if (s.pv.at && r.p_ready(group_of(s.pv.step), tile_of(s.pv.step)) == b) {
    s.pv.at = 0;
    issue(s.pv);
  }
}

static std::vector<State> successors(const State& s, const Rule& r) {
  std::vector<State> out;
  for (int a = 0; a < n_groups; ++a)
    for (int k = 0; k < n_warps; ++k) {
      const Warp& w = s.w[a][k];
      if (w.stage == kAtS || w.stage == kAtP || w.stage == kAtGroup || (w.stage == kWaitS && w.tile == n_tiles)) continue;
      if (!w.gave) {   // any wait may run out
        out.push_back(s);
        out.back().w[a][k].gave = 1;
      }
      const bool seen = w.stage == kWaitS ? s.qk.good > step_of(a, w.tile)
                                          : (w.stage == kWaitPv && w.tile % segment == 0) || s.pv.good > step_of(a, w.tile - 1);
      if (!w.gave && !seen) continue;
      State t = s;
      Warp& x = t.w[a][k];
      const bool waits = r.waits(w.gave);
      int b;
      if (w.stage == kWaitS) {
        b = r.s_free(a, w.tile);
        x.stage = waits ? kAtS : kWaitPv;
      } else if (w.stage == kWaitPv) {
        b = r.p_ready(a, w.tile);
        if (waits) x.stage = kAtP;
        else behind_p(x);
      } else {
        b = unstep::kGroupBarrier + a;
        x.stage = kAtGroup;
      }
      arrive(t, r, b);
      out.push_back(t);
    }
  for (int i = 0; i < 2; ++i) {
    const Issuer& x = i == 0 ? s.qk : s.pv;
    if (x.at || x.step >= steps() + (i == 0 ? 1 : 0)) continue;
    if (x.ok) {
      out.push_back(s);
      (i == 0 ? out.back().qk : out.back().pv).ok = 0;
    }
    State t = s;
    if (i == 0 && x.step == 0) {
      issue(t.qk);
    } else {
      (i == 0 ? t.qk : t.pv).at = 1;
      const int step = i == 0 ? x.step - 1 : x.step;
      arrive(t, r, i == 0 ? r.s_free(group_of(step), tile_of(step)) : r.p_ready(group_of(step), tile_of(step)));
    }
    out.push_back(t);
  }
  for (State& t : out)
    for (int a = 0; a < n_groups; ++a) std::sort(t.w[a], t.w[a] + n_warps);   // the warps of a group are alike
  return out;
}

int main(int argc, char** argv) {
  if (argc != 5) return 2;
  n_tiles = atoi(argv[1]), segment = atoi(argv[2]), n_groups = atoi(argv[3]), n_warps = atoi(argv[4]);
  for (const Rule& r : {Rule{"kernel", true, true}, Rule{"one_barrier", false, true}, Rule{"one_barrier_arrive", false, false},
                        Rule{"two_barriers_arrive", true, false}}) {
    std::set<std::vector<int8_t>> seen;
    std::vector<State> todo = {State()};
    seen.insert(State().flat());
    size_t blocked = 0;
    while (!todo.empty()) {
      const State s = todo.back();
      todo.pop_back();
      const std::vector<State> next = successors(s, r);
      bool done = s.qk.step == steps() + 1 && s.pv.step == steps(), left = false;
      for (int a = 0; a < n_groups; ++a)
        for (int k = 0; k < n_warps; ++k) done = done && s.w[a][k].tile == n_tiles && s.w[a][k].stage == kWaitS;
      for (int8_t c : s.count) left = left || c != 0;
      if (done ? left : next.empty()) ++blocked;
      for (const State& t : next)
        if (seen.insert(t.flat()).second) todo.push_back(t);
    }
    printf("%s %zu %zu\n", r.name, seen.size(), blocked);
  }
  return 0;
}
