// Launch of the persistent per-stage update kernel for one physics trait and scheme.
#pragma once
#include "kernels.cuh"
#include "launch.h"

namespace agile {

// CTAs per SM a staging layout allows, by the shared memory of an SM (233472 bytes, 1 KB
// reserved per CTA) and the register budget it implies: FP32 three when three CTAs fit, else
// two; FP64 two when two CTAs fit (hydrodynamics, whose FP64 kernel fits 128 registers), else
// one (its full register budget).
template <template <typename> class PT, typename R, int RAW, int SFB>
constexpr int stage_minb() {
  constexpr size_t SMEM = stage_smem_bytes<PT, R, RAW, SFB>();
  if (sizeof(R) == 8) return 2 * (SMEM + 1024) <= 233472 ? 2 : 1;
  return 3 * (SMEM + 1024) <= 233472 ? 3 : (2 * (SMEM + 1024) <= 233472 ? 2 : 1);
}

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
inline StageCut stage_cut(int nblk, int sms, bool fp64, bool prims, bool source, int ctas_per_sm) {
  const double c = fp64 ? 0.5 : (prims ? 0.6 : 1.1);
  const double one = fp64 ? (ctas_per_sm > 1 ? 1.12 : 1.0) : 1.4;
  const double two = !fp64 && prims ? 1.15 : 1.0;
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
  best.inv_m = ((1ull << 32) + best.m - 1) / best.m;
  return best;
}

// Z_CUT: launches of this layout may cut blocks along z (a kernel of its own: the item bounds
// as variables cost 1.6% on a 256^3 launch of whole blocks, 0.457 -> 0.464 ms for HD FP32).
template <template <typename> class PT, typename R, int LIM, int FLUX, int RAW, int SFB, bool Z_CUT>
static cudaError_t stage_go_layout(const StageArgs& a, cudaStream_t s) {
  constexpr size_t SMEM = stage_smem_bytes<PT, R, RAW, SFB>();
  constexpr int MINB = stage_minb<PT, R, RAW, SFB>();
  auto whole = stage_kernel<PT, R, LIM, FLUX, MINB, RAW, SFB, false>;
  auto cut = stage_kernel<PT, R, LIM, FLUX, MINB, RAW, SFB, Z_CUT>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(whole, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
    if (e == cudaSuccess && Z_CUT)
      e = cudaFuncSetAttribute(cut, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  // persistent grid: as many CTAs as fit on the GPU at once, each looping over work items
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  if (a.nblk <= 0) return cudaSuccess;
  StageArgs args = a;
  args.cut.nblk = a.nblk;
  if constexpr (Z_CUT) {
    if (!a.cut_cache) {
      args.cut = stage_cut(a.nblk, sms, sizeof(R) == 8, prim_pass_of<PT<R>>::value, PT<R>::SOURCE, MINB);
    } else {
      if (a.cut_cache->nblk != a.nblk)
        *a.cut_cache = stage_cut(a.nblk, sms, sizeof(R) == 8, prim_pass_of<PT<R>>::value, PT<R>::SOURCE, MINB);
      args.cut = *a.cut_cache;
    }
  }
  // a tuned persistent grid, else the default
  int grid = a.grid > 0 ? a.grid : MINB * sms;
  if (grid > args.cut.items()) grid = args.cut.items();
  args.ppf.set(a.gamma, 0.0);
  args.ppd.set(a.gamma, 0.0);
  args.fa = (float)a.a;
  args.fb = (float)a.b;
  args.combine = a.a != 0.0 ? 1 : 0;
  const CUtensorMap& tm = *static_cast<const CUtensorMap*>(args.tmap);
  return launch_chained(args.cut.whole() ? whole : cut, dim3(grid), 256, SMEM, s, tm, args);
}

// Staging layouts: STAGE_LAYOUT_RING4 = four raw slots, one flux buffer, two barriers per
// plane; STAGE_LAYOUT_RING5_DB = five raw slots, two flux buffers, one barrier per plane;
// STAGE_LAYOUT_RING3_DB = three raw slots, two flux buffers, one barrier per plane, the update's
// stage input loaded from global memory (L2) ahead of the face work instead of kept in a raw
// slot. The default (layout 0) takes layout 2 where it keeps as many CTAs per SM as layout 1, else
// layout 3 where that keeps two (256^3 MHD launch: layout 1 858 us, layout 3 831; with resistivity
// on 1728 blocks 396 and 388), else layout 1: three CTAs per SM cover the second barrier as well
// as layout 3 saves it (FFHD, 1728 blocks: 195 us either way). FP64 keeps layout 1. Only the
// default layout cuts blocks along z (stage_cut).
template <template <typename> class PT, typename R, int LIM, int FLUX>
static cudaError_t stage_go(const StageArgs& a, cudaStream_t s) {
  if constexpr (sizeof(R) == 8) {
    return stage_go_layout<PT, R, LIM, FLUX, 4, 1, true>(a, s);
  } else {
    constexpr int m1 = stage_minb<PT, R, 4, 1>();
    constexpr int dflt = stage_minb<PT, R, 5, 2>() >= m1             ? STAGE_LAYOUT_RING5_DB
                         : m1 == 2 && stage_minb<PT, R, 3, 2>() == 2 ? STAGE_LAYOUT_RING3_DB
                                                                     : STAGE_LAYOUT_RING4;
    const int lay = a.layout == 0 ? dflt : a.layout;
    if (lay == STAGE_LAYOUT_RING5_DB) return stage_go_layout<PT, R, LIM, FLUX, 5, 2, dflt == STAGE_LAYOUT_RING5_DB>(a, s);
    if (lay == STAGE_LAYOUT_RING3_DB) return stage_go_layout<PT, R, LIM, FLUX, 3, 2, dflt == STAGE_LAYOUT_RING3_DB>(a, s);
    return stage_go_layout<PT, R, LIM, FLUX, 4, 1, dflt == STAGE_LAYOUT_RING4>(a, s);
  }
}

}  // namespace agile
