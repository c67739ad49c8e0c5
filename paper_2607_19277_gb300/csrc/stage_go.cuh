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
  // a tuned persistent grid, else the default
  int grid = a.grid > 0 ? a.grid : MINB * sms;
  if constexpr (Z_CUT) {
    const int ctas = grid / sms < 1 ? 1 : (grid / sms > MINB ? MINB : grid / sms);
    args.cut = a.cut_cache->get(a.nblk, sms, sizeof(R) == 8, prim_pass_of<PT<R>>::value, PT<R>::SOURCE, ctas);
  }
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
// layout 3 where that keeps two (256^3 MHD launch: layout 1 858 us, layout 3 833; with resistivity
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
