// Test-only C shim over the stage kernel's work-item list (csrc/stage_cut.h), compiled with g++ by
// tests/test_stage_cut.py.
#include "../paper_2607_19277_gb300/csrc/stage_cut.h"

using namespace agile;

extern "C" {

// The cut the launch rule chooses: out = n1, a, m, items, whole.
void shim_cut(int nblk, int sms, int fp64, int prims, int source, int ctas, int* out) {
  const StageCut c = stage_cut(nblk, sms, fp64 != 0, prims != 0, source != 0, ctas);
  out[0] = c.n1;
  out[1] = c.a;
  out[2] = c.m;
  out[3] = c.items();
  out[4] = c.whole() ? 1 : 0;
}

// The item list of such a cut: out[item][3] = block, first plane, planes.
void shim_items(int nblk, int n1, int a, int m, int* out) {
  StageCut c;
  c.nblk = nblk;
  c.n1 = n1;
  c.a = a;
  c.m = m;
  c.set_divisor();
  for (int w = 0; w < c.items(); ++w) c.item(w, out[3 * w], out[3 * w + 1], out[3 * w + 2]);
}
}
