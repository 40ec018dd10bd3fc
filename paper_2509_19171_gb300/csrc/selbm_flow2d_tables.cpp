#include "selbm_flow2d_tables.h"

#include <algorithm>

namespace slb {

bool build_flow2d_tables(const Setup &S, int epc, Flow2DTables *t) {
  const int E = S.E, Nb = S.Nb, row = 9 * Nb;
  // trace offsets run to E 9 Nb
  if ((int64_t)E * row > INT32_MAX) return false;
  const int grid = (E + epc - 1) / epc;
  t->u.assign((size_t)E * Nb, 0);
  t->off.assign((size_t)E * Nb + 1, 0);
  t->base.assign((size_t)E * Nb, 0);
  t->rem_off.assign(1, 0);
  t->bas_off.assign(1, 0);
  std::vector<int32_t> at((size_t)E * Nb, -1), at_u(S.Gb, -1);
  for (int k = 0; k < S.Gb; ++k)
    for (int c = S.bnode_off[k]; c < S.bnode_off[k + 1]; ++c) t->u[S.bnode_slot[c]] = k;
  for (int cta = 0; cta < grid; ++cta) {
    const int e0 = cta * epc, e1 = std::min(E, e0 + epc);
    const size_t rem0 = t->rem.size(), bas0 = t->bas.size();
    for (size_t lb = (size_t)e0 * Nb; lb < (size_t)e1 * Nb; ++lb) {
      t->off[lb] = (int32_t)t->slot.size();
      const int k = t->u[lb];
      for (int c = S.bnode_off[k]; c < S.bnode_off[k + 1]; ++c) {
        const int s = S.bnode_slot[c], e2 = s / Nb;
        if (e2 >= e0 && e2 < e1) {
          t->slot.push_back(-3 - (s - e0 * Nb));
          continue;
        }
        if (at[s] < 0) { at[s] = (int32_t)(t->rem.size() - rem0); t->rem.push_back(e2 * row + s % Nb); }
        t->slot.push_back(at[s]);
      }
      // the first copy owns the node
      const int s = S.bnode_slot[S.bnode_off[k]];
      if ((size_t)s == lb) t->base[lb] = -1;
      else if (s / Nb >= e0 && s / Nb < e1) t->base[lb] = -3 - (s - e0 * Nb);
      else {
        if (at_u[k] < 0) { at_u[k] = (int32_t)(t->bas.size() - bas0); t->bas.push_back(k); }
        t->base[lb] = at_u[k];
      }
    }
    for (size_t r = rem0; r < t->rem.size(); ++r) at[(size_t)(t->rem[r] / row) * Nb + t->rem[r] % row] = -1;
    for (size_t r = bas0; r < t->bas.size(); ++r) at_u[t->bas[r]] = -1;
    t->rem_off.push_back((int32_t)t->rem.size());
    t->bas_off.push_back((int32_t)t->bas.size());
    t->rmax = std::max(t->rmax, (int)(t->rem.size() - rem0));
    t->bmax = std::max(t->bmax, (int)(t->bas.size() - bas0));
  }
  t->off[(size_t)E * Nb] = (int32_t)t->slot.size();
  if (t->rem.empty()) t->rem.push_back(0);
  if (t->bas.empty()) t->bas.push_back(0);
  return true;
}

}  // namespace slb
