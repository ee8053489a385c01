// CPU driver for the sizes of the banded solves (csrc/band_plan.h): for each launch read
// from stdin ("n", then n lines "m0 D L", then the doubles of shared memory), the sizes that
// the planner and the launch derive from its tasks, and what the kernel copies.
// Output per launch: stage, side rows; per task: whether the rule admits it, and of both
// passes the largest piece, whether every piece starts and ends on 16 bytes, and the rows
// that the pieces cover.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "band_plan.h"

using namespace fock;

struct T { int m0, D, L; bool twist; };

int main() {
  int n, room;
  while (std::scanf("%d", &n) == 1) {
    std::vector<T> ts(n);
    int step = 0, rows8 = 0, side = 0;
    for (T& t : ts) {
      if (std::scanf("%d %d %d", &t.m0, &t.D, &t.L) != 3) return 1;
      t.twist = t.D > 0 && t.L >= 2 * t.D + 2;   // as the planner
      step = std::max(step, (int)band_step(t.D + 1, t.m0));
      rows8 = std::max(rows8, band_stage_rows8(t.D, t.m0));
      side = std::max(side, band_side_rows(t.D, t.m0, t.twist));
    }
    if (std::scanf("%d", &room) != 1) return 1;
    const int stage = band_stage(step, rows8, side, room);
    std::printf("%d %d", stage, side);
    for (const T& t : ts) {
      const int qc = step <= stage ? t.m0 : band_rows(t.D + 1, t.m0, stage);
      int most = 0, aligned = 1, covered = 0;
      for (int pass = 0; pass < 2 && qc > 0; ++pass) {
        const int nd = t.D + pass, width = nd * t.m0, total = (int)band_step(nd, t.m0);
        for (int h = 0; h * qc < t.m0; ++h) {
          const int c = band_piece(qc, width, total, h);
          most = std::max(most, c + (c & 1));     // copied two at a time
          if ((h * qc * width) % 2 || (c % 2 && h * qc * width + c + 1 > total)) aligned = 0;
          if (pass) covered += std::min(qc, t.m0 - h * qc);
        }
      }
      std::printf(" %d %d %d %d", (int)band_rule(t.L, t.D, t.m0), most, aligned, covered);
    }
    std::printf("\n");
  }
  return 0;
}
