// The work split of launches whose parts are clusters: cluster_plan HEADS TOKENS_H TOKENS_W CHUNK FRAMES START prints
// cluster, parts and workers of the launch on 148 SMs, then a line per segment: worker, head, pair, first and end tile.
#include <cstdio>
#include <cstdlib>

#include "attn_sched.h"

int main(int argc, char** argv) {
  if (argc != 7) return 2;
  unstep_shape_t sh = {};
  sh.batch = 1, sh.heads = atoi(argv[1]), sh.head_dim = 128, sh.grid_h = atoi(argv[2]), sh.grid_w = atoi(argv[3]);
  sh.chunk_frames = atoi(argv[4]), sh.ring_frames = atoi(argv[5]);
  const int32_t start = atoi(argv[6]);
  const int32_t clusters[unstep::kMaxClusterParts + 1] = {0, 0, 74, 45, 33, 26, 22, 15, 15};
  unstep::AttnParams p;
  unstep::plan_shape(p, &sh, 0);
  if (unstep::plan_launch(p, &sh, &start, 1, sh.ring_frames, 0, 0, 148, clusters) != UNSTEP_OK) return 1;
  printf("%d %d %d\n", p.cluster, p.parts, p.n_workers);
  for (int w = 0; w < p.n_workers; ++w) {
    unstep::Sched sched(p, w);
    unstep::Seg s;
    while (sched.next(s)) printf("%d %d %d %d %d %d\n", w, s.h, s.qp, s.t0, s.t1, s.tiles);
  }
  return 0;
}
