// Prints the plan of a step (csrc/lbcad_plan.h) for the boxes on standard input: "split n", then n lines "nx ny nz".
#include <cstdio>

#include "lbcad_plan.h"

int main() {
  int split, n;
  while (std::scanf("%d %d", &split, &n) == 2) {
    std::vector<lbcad_grid> boxes(n);
    for (lbcad_grid& b : boxes)
      if (std::scanf("%d %d %d", &b.nx, &b.ny, &b.nz) != 3) return 1;
    const lbcad::StepPlan p = lbcad::plan_step(boxes, split != 0);
    std::printf("%lld %d\n", p.scratch, (int)p.parts.size());
    for (const lbcad::StepPart& s : p.parts)
      std::printf("%d %d %d %d %d %d %d\n", s.first, s.ninst, s.fz, s.fn, s.lz, s.ln, s.sz0);
    for (const lbcad::ScratchPlace& q : p.place) std::printf("%lld %lld\n", q.at, q.sites);
  }
  return 0;
}
