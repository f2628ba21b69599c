// Prints the plan of a step (csrc/lbcad_plan.h) for the boxes on standard input: "split tighter n" (tighter: how many
// times the scratch is made smaller), then n lines "nx ny nz".
#include <cstdio>

#include "lbcad_plan.h"

int main() {
  int split, tighter, n;
  while (std::scanf("%d %d %d", &split, &tighter, &n) == 3) {
    std::vector<lbcad_grid> boxes(n);
    for (lbcad_grid& b : boxes)
      if (std::scanf("%d %d %d", &b.nx, &b.ny, &b.nz) != 3) return 1;
    lbcad::ScratchRule rule;
    for (int i = 0; i < tighter; ++i) rule = rule.tighter();
    const lbcad::StepPlan p = lbcad::plan_step(boxes, split != 0, rule);
    std::printf("%lld %d\n", p.scratch, (int)p.parts.size());
    for (const lbcad::StepPart& s : p.parts)
      std::printf("%d %d %d %d %d %d %d\n", s.first, s.ninst, s.fz, s.fn, s.lz, s.ln, s.sz0);
    for (const lbcad::ScratchPlace& q : p.place) std::printf("%lld %lld\n", q.at, q.sites);
  }
  return 0;
}
