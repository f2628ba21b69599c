// How the Euler step of the default path is divided: the groups of instances that a launch holds, the slabs of
// planes a large box is stepped in, and the scratch these need.  Host code without CUDA.
#pragma once

#include <algorithm>
#include <vector>

#include "lbcad.h"

namespace lbcad {

// Instances of one launch (see InstPack).
constexpr int kPackMany = 28;

// The scratch that a launch of the Euler step may take: that of at most `sites` sites (a batch is launched in groups
// of at most that many, a larger box in slabs of planes, with which the fields kernel also works on the planes next to
// them), but of no fewer than `least` planes to a slab.  At 12 values a site 2^26 sites keep it at 3.2 GB in FP32, where
// a scratch for every site would take a sixth of the memory left for boxes as large as the device holds; planes of more
// than 2^26 / 10 sites take ten of them, because a slab of few planes repeats much of the fields kernel's work (1.25
// times at 8 planes, 3 times at one).  Where there is no memory for that, tighter() of it still steps the box, down
// to three planes of the largest box.
struct ScratchRule {
  long long sites = 1LL << 26;
  int least = 8;
  ScratchRule tighter() const {
    ScratchRule r;
    r.sites = std::max(1LL, sites / 4);
    r.least = 1;
    return r;
  }
  bool tightest() const { return sites == 1 && least == 1; }
};

// Planes of the step's slabs of a box (nz: all at once).
inline int slab_planes(const lbcad_grid& b, const ScratchRule& rule) {
  const long long plane = (long long)b.nx * b.ny;
  if (plane * b.nz <= rule.sites) return b.nz;
  const int n = (int)std::max((long long)rule.least, rule.sites / plane - 2);
  return n + 2 < b.nz ? n : b.nz;
}

// Sites of a box that its scratch holds: those of a slab and of the planes next to it, or all.
inline long long scratch_sites(const lbcad_grid& b, const ScratchRule& rule) {
  const int n = slab_planes(b, rule);
  return (long long)b.nx * b.ny * (n < b.nz ? n + 2 : b.nz);
}

// One launch of a step: instances first ... first + ninst - 1.  Of a box that is stepped in slabs the LB kernel
// works on the planes lz ... lz + ln - 1 and the fields kernel on fz ... fz + fn - 1, modulo the height, and plane
// sz0 is the first of the scratch; fn = ln = 0: all planes of every box.
struct StepPart {
  int first = 0, ninst = 0;
  int fz = 0, fn = 0, lz = 0, ln = 0, sz0 = 0;
};

// Where an instance's scratch starts and the sites it holds (in sites of the one scratch that the launches use in turn).
struct ScratchPlace {
  long long at = 0, sites = 0;
};

struct StepPlan {
  std::vector<StepPart> parts;
  std::vector<ScratchPlace> place;  // by instance
  long long scratch = 0;            // sites of the scratch
};

// split (sync coupling, Heun): a scratch of its own for each whole box, so that only kPackMany bounds a group.
// A box that is stepped in slabs is alone in its group: the launches of a slab are of that slab only.
inline StepPlan plan_step(const std::vector<lbcad_grid>& boxes, bool split, const ScratchRule& rule = {}) {
  StepPlan p;
  p.place.resize(boxes.size());
  for (int first = 0; first < (int)boxes.size();) {
    StepPart part;
    part.first = first;
    if (!split && slab_planes(boxes[first], rule) < boxes[first].nz) {
      const lbcad_grid& b = boxes[first];
      part.ninst = 1;
      p.place[first].sites = scratch_sites(b, rule);
      p.scratch = std::max(p.scratch, p.place[first].sites);
      for (int n = slab_planes(b, rule), z = 0; z < b.nz; z += n) {
        part.lz = z;
        part.ln = std::min(n, b.nz - z);
        part.fz = z - 1;
        part.fn = part.ln + 2;
        part.sz0 = (z + b.nz - 1) % b.nz;
        p.parts.push_back(part);
      }
    } else {
      long long used = 0;
      for (int i = first; i < (int)boxes.size() && part.ninst < kPackMany; ++i) {
        if (!split && slab_planes(boxes[i], rule) < boxes[i].nz) break;
        const long long sites = scratch_sites(boxes[i], rule);
        if (!split && part.ninst > 0 && used + sites > rule.sites) break;
        if (!split) p.place[i] = ScratchPlace{used, sites};
        used += sites;
        ++part.ninst;
      }
      if (!split) p.scratch = std::max(p.scratch, used);
      p.parts.push_back(part);
    }
    first += part.ninst;
  }
  return p;
}

}  // namespace lbcad
