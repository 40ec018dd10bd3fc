// Tables of the resident 2D step (host): where a CTA finds the copies and the owner of every
// boundary node of its elements, and what it fetches from other CTAs.  The layouts are those of
// Flow2DArgs.
#pragma once
#include <cstdint>
#include <vector>

#include "selbm_setup.h"

namespace slb {

struct Flow2DTables {
  std::vector<int32_t> u, off, slot, base, rem, rem_off, bas, bas_off;
  int rmax = 0, bmax = 0;
};

// false, with nothing built, when a table's offsets would not fit 32 bits
bool build_flow2d_tables(const Setup &S, int epc, Flow2DTables *t);

}  // namespace slb
