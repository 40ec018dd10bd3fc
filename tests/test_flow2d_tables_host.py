"""Host tables of the resident 2D step, compiled with the host compiler: a mesh whose trace offsets
exceed 32 bits is turned down before any of its arrays is read, and the tables of a small mesh lead
every copy of a node to the same node."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_19171_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "selbm_flow2d_tables.h"
using namespace slb;
int main() {
  // counts of a mesh of order N, its arrays left out: 32-bit offsets end at E = 2^31 / (9 Nb)
  const int orders[3] = {2, 7, 14};
  for (int N : orders) {
    Setup S;
    S.dim = 2; S.N = N; S.Nb = 4 * N;
    S.E = (int)((1ll << 31) / (9 * S.Nb)) + 1;
    Flow2DTables t;
    if (build_flow2d_tables(S, (S.E + 151) / 152, &t) || !t.u.empty()) { std::printf("accepted N = %d\n", N); return 1; }
  }
  // a ring of 5 elements of 4 boundary nodes: nodes 2, 3 of element e are nodes 0, 1 of element e + 1
  Setup S;
  S.dim = 2; S.N = 1; S.Nb = 4; S.E = 5; S.Gb = 10;
  S.bnode_off.push_back(0);
  for (int e = 0; e < 5; ++e)
    for (int b = 0; b < 2; ++b) {
      const int prev = (e + 4) % 5;
      const int lo = e < prev ? 4 * e + b : 4 * prev + 2 + b, hi = e < prev ? 4 * prev + 2 + b : 4 * e + b;
      S.bnode_slot.push_back(lo);
      S.bnode_slot.push_back(hi);
      S.bnode_off.push_back((int)S.bnode_slot.size());
    }
  for (int epc = 1; epc <= 5; ++epc) {
    Flow2DTables t;
    if (!build_flow2d_tables(S, epc, &t)) return 2;
    for (int lb = 0; lb < 20; ++lb) {
      const int cta = lb / 4 / epc, k = t.u[lb], nc = S.bnode_off[k + 1] - S.bnode_off[k];
      if (t.off[lb + 1] - t.off[lb] != nc) return 3;
      for (int c = 0; c < nc; ++c) {
        const int want = S.bnode_slot[S.bnode_off[k] + c], s = t.slot[t.off[lb] + c];
        const int got = s >= 0 ? t.rem[t.rem_off[cta] + s] / 36 * 4 + t.rem[t.rem_off[cta] + s] % 36 : -3 - s + cta * epc * 4;
        if (got != want) return 4;
      }
      const int own = S.bnode_slot[S.bnode_off[k]], b = t.base[lb];
      if (b == -1 ? own != lb : b >= 0 ? t.bas[t.bas_off[cta] + b] != k : -3 - b + cta * epc * 4 != own) return 5;
    }
  }
  return 0;
}
"""


def test_tables(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "main.cpp"
    src.write_text(MAIN)
    exe = str(tmp_path / "tables")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(src), os.path.join(CSRC, "selbm_flow2d_tables.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
