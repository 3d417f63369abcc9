// Runs the tile queue of the guidance distances (sfm_guide_queue.h) on the CPU,
// an atomic operation at a time: CTAs as state machines, a CTA's pushes side by
// side, and a scheduler that holds single ones up for long.  The tiles are a
// ring or a path with a value each, relaxed to its neighbours' + 1.
// Arguments: tiles, CTAs, seed, longest hold-up in steps.  Prints the number of
// steps, "stuck" (the queue lost an entry), or "wrong".
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "sfm_guide_queue.h"

using namespace sfm;

struct Push {
  int tile;
  int at = 0;  // 0 mark, 1 position, 2 publish, 3 done
  unsigned pos = 0;
};
struct Cta {
  enum { kClaim, kTake, kUnmark, kRelax, kPush, kDone, kExit } at = kClaim;
  unsigned pos = 0;
  int tile = -1;
  long held = 0;
  std::vector<Push> push;
};

int main(int argc, char** argv) {
  if (argc != 5) return 2;
  const int n = atoi(argv[1]), nctas = atoi(argv[2]), hold = atoi(argv[4]);
  std::mt19937 rng((unsigned)atoi(argv[3]));
  const bool ring = rng() & 1u;
  std::vector<int> scratch(kGuideQueueInts + kGuideTileInts * n + 2, 0), value(n, 1 << 20);
  int* base = scratch.data();
  if (reinterpret_cast<size_t>(base) & 7) ++base;
  const GuideTiles gt = guide_tiles(base, n);
  auto neighbours = [&](int t) {
    std::vector<int> v;
    for (int d : {-1, 1})
      if (ring)
        v.push_back((t + d + n) % n);
      else if (t + d >= 0 && t + d < n)
        v.push_back(t + d);
    return v;
  };
  // start: every tile in the queue, values from the rightmost tile on
  value[n - 1] = 0;
  for (int t = 0; t < n; ++t)
    if (guide_mark(gt, t) && !guide_publish(gt, guide_position(gt), t)) return 2;
  std::vector<Cta> ctas(nctas);
  long step = 0;
  for (int left = nctas; left > 0; ++step) {
    if (step > 2000000L) {
      puts("stuck");
      return 1;
    }
    Cta& c = ctas[rng() % nctas];
    if (c.at == Cta::kExit) continue;
    if (c.held > 0 && step < c.held) continue;
    if (hold && rng() % 16 == 0) {
      c.held = step + rng() % hold;
      continue;
    }
    switch (c.at) {
      case Cta::kClaim:
        c.pos = guide_claim(gt);
        c.at = Cta::kTake;
        break;
      case Cta::kTake:
        c.tile = guide_take(gt, c.pos);
        if (c.tile >= 0)
          c.at = Cta::kUnmark;
        else if (guide_over(guide_work(gt))) {
          c.at = Cta::kExit;
          --left;
        }
        break;
      case Cta::kUnmark:
        guide_unmark(gt, c.tile);
        c.at = Cta::kRelax;
        break;
      case Cta::kRelax: {
        // a change, or one in three without, queues the neighbours
        int best = value[c.tile];
        for (int t : neighbours(c.tile)) best = value[t] + 1 < best ? value[t] + 1 : best;
        c.push.clear();
        if (best < value[c.tile] || (step < 20000 && rng() % 3 == 0)) {
          value[c.tile] = best;
          for (int t : neighbours(c.tile)) {
            Push p;
            p.tile = t;
            c.push.push_back(p);
          }
        }
        c.at = Cta::kPush;
        break;
      }
      case Cta::kPush: {
        bool open = false;
        for (Push& p : c.push) open = open || p.at != 3;
        if (!open) {
          c.at = Cta::kDone;
          break;
        }
        Push& p = c.push[rng() % c.push.size()];
        if (p.at == 0)
          p.at = guide_mark(gt, p.tile) ? 1 : 3;
        else if (p.at == 1) {
          p.pos = guide_position(gt);
          p.at = 2;
        } else if (p.at == 2 && guide_publish(gt, p.pos, p.tile))
          p.at = 3;
        break;
      }
      case Cta::kDone:
        guide_done(gt);
        c.at = Cta::kClaim;
        break;
      default:
        break;
    }
  }
  for (int t = 0; t < n; ++t) {
    const int want = ring ? (t + 1 < n - 1 - t ? t + 1 : n - 1 - t) : n - 1 - t;
    if (value[t] != want) {
      puts("wrong");
      return 1;
    }
  }
  printf("%ld\n", step);
  return 0;
}
