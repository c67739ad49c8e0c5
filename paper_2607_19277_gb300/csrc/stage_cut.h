// Work items of the stage kernel's launches: the item list the kernel walks and the rule that
// chooses it. Plain C++ on the host, so that both can be checked without a GPU.
#pragma once
#include "agile_internal.h"

#ifdef __CUDACC__
#define CUT_FN __host__ __device__
#else
#define CUT_FN
#endif

namespace agile {

// Work items of a launch over nblk blocks: the first n1 blocks whole, of the others m items of a
// planes each, then (behind all of those) one of the 16 - m a planes left, if any. Sizes fall
// along the list, so that CTAs taking the next free item end close together.
struct StageCut {
  int nblk = -1;
  int n1 = 0, a = NB, m = 1;
  unsigned long long inv_m = 1ull << 32;   // ceil(2^32 / m): exact for items below 2^28
  void set_divisor() { inv_m = ((1ull << 32) + m - 1) / m; }
  CUT_FN int rest() const { return NB - m * a; }
  CUT_FN int items() const { return n1 + (nblk - n1) * (rest() > 0 ? m + 1 : m); }
  CUT_FN bool whole() const { return n1 == nblk || a == NB; }
  // block (index into the work list), first plane and planes of item w
  CUT_FN void item(int w, int& blk, int& k0, int& nz) const {
    const int nr = nblk - n1;
    if (w < n1) {
      blk = w;
      k0 = 0;
      nz = NB;
    } else if (w - n1 < nr * m) {
      const int v = w - n1, q = (int)((unsigned long long)(unsigned)v * inv_m >> 32);   // v / m
      blk = n1 + q;
      k0 = (v - q * m) * a;
      nz = a;
    } else {
      blk = n1 + (w - n1 - nr * m);
      k0 = m * a;
      nz = rest();
    }
  }
};

// Work items of a launch. A launch of few blocks is cut along z into items of fewer than 16
// planes, so that it fills the SMs (one block per CTA leaves 144 of 152 SMs idle at 8 blocks
// and runs 16 planes in sequence); one of some hundreds is cut where its last blocks would
// leave SMs idle. An item costs its planes and a start c (four more planes loaded and converted,
// one more z-face) of about c = 1.1 planes in FP32, 0.6 where the planes come as primitives
// (SRHD) and 0.5 in FP64, whose faces cost more. Compared is the time of the SM that ends last:
//  - every block into 2^zs equal items, the SM with the most items deciding; few items on an
//    SM run slower per plane than a full one: one alone by 1.4 in FP32 and by 1.12 in FP64 where
//    two CTAs fit, two of three by 1.15 for SRHD in FP32. The smallest count is taken unless
//    another is at least 3% better;
//  - the first n1 blocks whole (none, all full rounds of the SMs or of the CTAs), the others in m
//    items of a planes and one of the rest, each taken by the SM that is free first. That holds
//    only where items are left when all CTAs have one: the first are placed by the hardware
//    (with one CTA launched per SM where two fit, a chained launch finds SMs of the one before it
//    still busy and two CTAs share another: 311 -> 441 us for 64 blocks of HD FP64). The estimate
//    is good to 2% for one CTA per SM and to 5% for more, where 4 <= a <= 8, and the cut kernel
//    of the frozen-field physics is some 6% slower per plane than the whole one.
// The equal cuts so chosen are within 4% of the fastest in 16 sizes x 7 schemes timed (SRHD in
// FP32 within 13%), the uneven ones within 4% of the fastest of 19 n1 and a at 8 sizes in FP64
// and 6 x 4 schemes in FP32. us per stage launch on 152 SMs, whole blocks -> equal cut: HD FP64
// 8 blocks 633 -> 64; MHD FP32 8 blocks 47 -> 13, 64 blocks 48 -> 27, 210 blocks 73 -> 61, 1000
// blocks 230 uncut (242 cut in two). Equal -> uneven: MHD FP64 40 blocks 556 -> 419, 120 blocks
// 1258 -> 1047, 512 blocks 4475 -> 4319; SRHD FP64 60 blocks 486 -> 440; HD FP64 400 blocks
// 1661 -> 1495; MHD FP32 120 blocks 42.0 -> 38.0, 470 blocks 125 -> 110; HD FP32 1250 blocks
// 149 -> 141. Costs: frozen-field FP32 launches of 40 to 215 blocks, mostly in equal items, 2 to 5%.
inline double cut_makespan(int sms, const int* count, const double* cost, int classes) {
  // SMs by load (few distinct ones), each item to a least loaded SM, in list order
  double load[64];
  int num[64];
  int n = 1;
  load[0] = 0.0;
  num[0] = sms;
  for (int c = 0; c < classes; ++c) {
    for (int k = count[c]; k > 0;) {
      int lo = 0;
      for (int i = 1; i < n; ++i)
        if (load[i] < load[lo]) lo = i;
      const int take = k < num[lo] ? k : num[lo];
      const double to = load[lo] + cost[c];
      num[lo] -= take;
      k -= take;
      if (!num[lo]) {
        --n;
        load[lo] = load[n];
        num[lo] = num[n];
      }
      int at = 0;
      while (at < n && !(load[at] > to - 1e-9 && load[at] < to + 1e-9)) ++at;
      if (at == n) {
        if (n == 64) return 1e300;   // (not met: a class adds at most two distinct loads)
        load[n] = to;
        num[n++] = 0;
      }
      num[at] += take;
    }
  }
  double worst = 0.0;
  for (int i = 0; i < n; ++i) worst = load[i] > worst ? load[i] : worst;
  return worst;
}
// ctas_per_sm: those the launch has (an autotuned grid may have fewer than fit: with one per SM all
// items run alone, and a lone one is not slower than others).
inline StageCut stage_cut(int nblk, int sms, bool fp64, bool prims, bool source, int ctas_per_sm) {
  const double c = fp64 ? 0.5 : (prims ? 0.6 : 1.1);
  const double one = ctas_per_sm == 1 ? 1.0 : (fp64 ? 1.12 : 1.4);
  const double two = !fp64 && prims && ctas_per_sm > 2 ? 1.15 : 1.0;
  StageCut best;
  best.nblk = nblk;
  double best_cost = 0.0;
  for (int zs = 0; zs <= 4; ++zs) {
    const long long per_sm = (((long long)nblk << zs) + sms - 1) / sms;
    const double cost = (double)per_sm * ((NB >> zs) + c) * (per_sm == 1 ? one : per_sm == 2 ? two : 1.0);
    if (zs == 0 || cost < 0.97 * best_cost) {
      best.a = NB >> zs;
      best.m = 1 << zs;
      best_cost = cost;
    }
  }
  best_cost *= fp64 ? 0.985 : 0.95;
  if (source && best.whole()) best_cost *= 0.94;
  const int round[3] = {nblk, ctas_per_sm * sms, sms};
  for (int i = 0; i < 3; ++i) {
    const int nr = i == 0 ? nblk : nblk % round[i];
    if (nr == 0 || (i > 0 && nblk < round[1]) || (i == 2 && ctas_per_sm == 1)) continue;
    for (int a = ctas_per_sm == 1 ? 2 : 4; a <= (ctas_per_sm == 1 ? NB - 1 : 8); ++a) {
      StageCut t;
      t.nblk = nblk;
      t.n1 = nblk - nr;
      t.a = a;
      t.m = NB / a;
      if (t.items() <= ctas_per_sm * sms) continue;
      const int count[3] = {t.n1, nr * t.m, t.rest() ? nr : 0};
      const double cost[3] = {NB + c, a + c, t.rest() + c};
      const double span = cut_makespan(sms, count, cost, 3);
      if (span < best_cost) {
        best = t;
        best_cost = span;
      }
    }
  }
  best.set_divisor();
  return best;
}

// The cut of a mesh's or a batch's launches, formed again when what it depends on changes. us per
// first stage launch of autotuned batches with one CTA per SM, with the cut for all CTAs that fit
// -> with their own: HD FP64 64 blocks 311 -> 260 (two per SM 273), 400 blocks 1547 -> 1516; FP32 HD
// 120 blocks at two per SM 24.7 -> 22.6. Launches that hand out items by stride take the same
// items (uneven ones: MHD FP64 120 blocks 993 us, equal ones 1185; MHD FP32 120 blocks 33.0 and 36.8).
struct StageCutCache {
  StageCut cut;
  int ctas_per_sm = 0;
  const StageCut& get(int nblk, int sms, bool fp64, bool prims, bool source, int ctas) {
    if (cut.nblk != nblk || ctas_per_sm != ctas) {
      cut = stage_cut(nblk, sms, fp64, prims, source, ctas);
      ctas_per_sm = ctas;
    }
    return cut;
  }
};

}  // namespace agile
