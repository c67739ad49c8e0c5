// Non-update kernels: coarse-fine ghost slots (restriction, limited-linear prolongation),
// coarse-fine flux correction, global signal-speed reduction for the CFL step, GLM damping,
// Loehner estimator, regrid prolongation/restriction, state packing and conserved sums.
#include <math.h>

#include <type_traits>

#include "kernels.cuh"
#include "launch.h"

namespace agile {

int phys_nvar(int phys) {
  return phys == PH_MHD ? 9 : (phys == PH_FFHD ? 6 : (phys == PH_FFHD_HTC ? 7 : 5));
}
int phys_naux(int phys) { return phys == PH_SRHD || phys == PH_SRHD_SYNGE ? 2 : 0; }

// ------------------------------------------------------------------------------ helpers
template <typename R>
__device__ __forceinline__ R minmod_(R a, R b) {
  return (a > R(0) && b > R(0)) ? (a < b ? a : b) : ((a < R(0) && b < R(0)) ? (a > b ? a : b) : R(0));
}

// Two neighbouring cells of a row in one access.
template <typename R>
struct pair_of {
  using type = typename std::conditional<sizeof(R) == 4, float2, double2>::type;
};

// Mean of the 8 fine cells from q (the lower corner, x even): x fastest, then y, then z, added
// in that order and scaled by 1/8 (volume-average restriction).
template <typename R>
__device__ __forceinline__ R mean8(const R* __restrict__ q) {
  using V = typename pair_of<R>::type;
  const V a = *reinterpret_cast<const V*>(q), b = *reinterpret_cast<const V*>(q + 16);
  const V c = *reinterpret_cast<const V*>(q + 256), d = *reinterpret_cast<const V*>(q + 272);
  R s = a.x + a.y;
  s = s + b.x;
  s = s + b.y;
  s = s + c.x;
  s = s + c.y;
  s = s + d.x;
  s = s + d.y;
  return s * R(0.125);
}

__device__ __forceinline__ int axis_stride(int d) { return d == 0 ? 1 : (d == 1 ? 16 : 256); }

// Where the neighbour of a cell along one axis is found: its first variable, the distance of
// the variables, and how the value is formed from it.
enum : int { CELL_NONE = -1, CELL_VALUE = 0, CELL_MEAN8 = 1, CELL_REFLECT = 2 };
template <typename R>
struct CellRef {
  const R* p;
  int vs;
  int mode;
};
// Value of variable v through a reference along axis e (CELL_REFLECT: a reflecting wall negates
// the normal vector components).
template <class P, typename R>
__device__ __forceinline__ R cell_value(const CellRef<R>& c, int v, int e) {
  if (c.mode == CELL_MEAN8) return mean8<R>(c.p + (size_t)v * NCELL);
  const R x = c.p[(size_t)v * c.vs];
  const bool neg = c.mode == CELL_REFLECT && ((P::IV >= 0 && v == P::IV + e) || (P::BOFF >= 0 && v == P::BOFF + e));
  return neg ? -x : x;
}
// The neighbour of cell `off` of block C one step up (dir = 1) or down (-1) along axis e: inside
// the block, in a same-level neighbour, a physical boundary image (both kinds mirror the
// block's own edge cell), and across a coarse-fine face, SLOTS: from the filled ghost slot;
// else, where the neighbour is finer, the mean of its cells, and where it is coarser, nothing
// (the prolongation of a ghost slot takes no slope there).
template <class P, typename R, bool SLOTS>
__device__ __forceinline__ CellRef<R> cell_ref(const R* __restrict__ U, const R* __restrict__ G,
                                               const BlockDesc* __restrict__ bd, int C, int off, int e, int dir) {
  constexpr int NT = P::NV + P::NA;
  const int se = axis_stride(e);
  const int pe = (off >> (4 * e)) & 15;
  const R* own = U + (size_t)C * NT * NCELL + off;
  if (dir > 0 ? pe < NB - 1 : pe > 0) return {own + dir * se, NCELL, CELL_VALUE};
  const int f = 2 * e + (dir > 0 ? 1 : 0);
  const int sv = bd[C].src[f];
  if (sv >= 0) return {U + (size_t)sv * NT * NCELL + off - dir * 15 * se, NCELL, CELL_VALUE};
  if (sv == SRC_OUTFLOW) return {own, NCELL, CELL_VALUE};
  if (sv == SRC_REFLECT) return {own, NCELL, CELL_REFLECT};
  const int x = off & 15, y = (off >> 4) & 15, z = off >> 8;
  const int t1 = e == 0 ? y : x, t2 = e == 2 ? y : z;
  if (SLOTS) {
    const int layer = dir > 0 ? 0 : 1;
    return {G + (size_t)(SRC_SLOT0 - sv) * NT * 512 + layer * 256 + t2 * 16 + t1, 512, CELL_VALUE};
  }
  if (bd[C].kind[f] == FK_COARSER) return {own, NCELL, CELL_NONE};
  const int fb = bd[C].nbr[f][(t1 >> 3) + 2 * (t2 >> 3)];
  const int st1 = e == 0 ? 16 : 1, st2 = e == 2 ? 16 : 256;
  const int fo = (dir > 0 ? 0 : NB - 2) * se + 2 * (t1 & 7) * st1 + 2 * (t2 & 7) * st2;
  return {U + (size_t)fb * NT * NCELL + fo, NCELL, CELL_MEAN8};
}

// ------------------------------------------------------------------------------ ghost slots
// One CTA per coarse-fine face of a block. Bound by the latency of dependent reads (task,
// descriptor, cells), so each thread has the loads of all variables in flight: cell offsets
// come from axis strides (an index array would live in local memory), fine cells are read in
// pairs along x. Finer neighbour: one thread per ghost column of two layers. Coarser
// neighbour: the slot's 2 x 16 x 16 fine ghost cells lie in one layer of 8 x 8 coarse cells of
// block C; the value and the three limited slopes of each are formed once (256 threads: 64
// cells x {value, slope along x, y, z}) and shared by its fine cells. A four-level HD blast, FP32:
// 40 -> 20 us a launch against index arrays in local memory and one fine cell per load.
template <template <typename> class PT, typename R>
__global__ void __launch_bounds__(256, 4) ghost_kernel(const R* __restrict__ U, R* __restrict__ G,
                                                        const BlockDesc* __restrict__ bd,
                                                        const GhostTask* __restrict__ tasks) {
  using P = PT<R>;
  constexpr int NT = P::NV + P::NA;
  chain_wait();
  const GhostTask& tk = tasks[blockIdx.x];
  const int d = tk.face >> 1, s = tk.face & 1;
  const int sd = axis_stride(d), st1 = d == 0 ? 16 : 1, st2 = d == 2 ? 16 : 256;
  const int t1 = threadIdx.x & 15, t2 = threadIdx.x >> 4;
  R* g = G + (size_t)tk.slot * NT * 512 + t2 * 16 + t1;
  if (tk.kind == FK_FINER) {                 // CTA-uniform
    const int fb = tk.nbr[(t1 >> 3) + 2 * (t2 >> 3)];
    const R* q = U + (size_t)fb * NT * NCELL + (s ? 0 : NB - 4) * sd + 2 * (t1 & 7) * st1 + 2 * (t2 & 7) * st2;
#pragma unroll
    for (int v = 0; v < NT; ++v) {
      g[(size_t)v * 512] = mean8<R>(q + (size_t)v * NCELL);
      g[(size_t)v * 512 + 256] = mean8<R>(q + (size_t)v * NCELL + 2 * sd);
    }
    return;
  }
  __shared__ R s_uc[NT][64], s_sig[3][NT][64];
  {
    const int cl = threadIdx.x & 63, job = threadIdx.x >> 6;
    const int n = 8 * tk.par[d] + (s ? 0 : 7);              // the coarse layer along d
    const int a1 = 8 * tk.par[d == 0 ? 1 : 0] + (cl & 7), a2 = 8 * tk.par[d == 2 ? 1 : 2] + (cl >> 3);
    const int off = n * sd + a1 * st1 + a2 * st2;
    const int C = tk.nbr[0];
    const R* own = U + (size_t)C * NT * NCELL + off;
    if (job == 0) {
#pragma unroll
      for (int v = 0; v < NT; ++v) s_uc[v][cl] = own[(size_t)v * NCELL];
    } else {
      const int e = job - 1;                                 // the slope's direction
      const CellRef<R> up = cell_ref<P, R, false>(U, (const R*)nullptr, bd, C, off, e, 1);
      const CellRef<R> um = cell_ref<P, R, false>(U, (const R*)nullptr, bd, C, off, e, -1);
      const bool ok = up.mode != CELL_NONE && um.mode != CELL_NONE;
#pragma unroll
      for (int v = 0; v < NT; ++v) {
        const R c = own[(size_t)v * NCELL];
        s_sig[e][v][cl] = ok ? minmod_(cell_value<P, R>(up, v, e) - c, c - cell_value<P, R>(um, v, e)) : R(0);
      }
    }
  }
  __syncthreads();
  // fine ghost cells: u_C + sum_e of the sign of the offset along e times sigma_e / 4 (the
  // layer's parity is that of its coordinate along d)
  const int cl = (t1 >> 1) + 8 * (t2 >> 1);
#pragma unroll
  for (int layer = 0; layer < 2; ++layer) {
    const R sl = layer ? R(1) : R(-1), s1 = (t1 & 1) ? R(1) : R(-1), s2 = (t2 & 1) ? R(1) : R(-1);
    const R sx = d == 0 ? sl : s1, sy = d == 1 ? sl : (d == 0 ? s1 : s2), sz = d == 2 ? sl : s2;
#pragma unroll
    for (int v = 0; v < NT; ++v) {
      R acc = sx * s_sig[0][v][cl];
      acc = acc + sy * s_sig[1][v][cl];
      acc = acc + sz * s_sig[2][v][cl];
      g[(size_t)v * 512 + layer * 256] = s_uc[v][cl] + R(0.25) * acc;
    }
  }
}

// ------------------------------------------------------------------------------ flux fix-up
// U += b dt (+/-)(F_coarse - mean of the 2x2 fine face fluxes) / dx on the cells beside the
// coarse-fine faces of a coarse block: one CTA per face (grid.y), one thread per cell. A cell
// on an edge between such faces belongs to the first of them in the task's order and receives
// their corrections in that order, so no two threads touch a cell and the faces need not wait
// for one another. Latency-bound (task, fluxes, cell); the factors b dt / dx are formed in FP64
// by three threads. Against one CTA per block with its faces in sequence 17 -> 12 us a launch on
// the four-level blast.
template <typename R, int NV, int NT>
__global__ void __launch_bounds__(256) fixup_kernel(R* __restrict__ U, const R* __restrict__ FR,
                                                     const BlockDesc* __restrict__ bd,
                                                     const FixupTask* __restrict__ tasks, double b,
                                                     const double* __restrict__ dtch,
                                                     const int* __restrict__ solve_of) {
  chain_wait();
  const FixupTask& tk = tasks[blockIdx.x];
  const int j = blockIdx.y, nface = tk.nface;
  if (j >= nface) return;                    // CTA-uniform
  __shared__ R s_w[3];
  if (threadIdx.x < 3) {
    const double dt = dtch[2 * (solve_of ? solve_of[tk.blk] : 0)];   // the block's solve
    s_w[threadIdx.x] = R(b * dt / bd[tk.blk].dx[threadIdx.x]);
  }
  const int fj = tk.face[j], dj = fj >> 1;
  const int c1 = threadIdx.x & 15, c2 = threadIdx.x >> 4, cd = (fj & 1) ? NB - 1 : 0;
  const int x = dj == 0 ? cd : c1, y = dj == 1 ? cd : (dj == 0 ? c1 : c2), z = dj == 2 ? cd : c2;
  __syncthreads();
  auto beside = [&](int face) {              // the cell lies beside this face
    const int d = face >> 1;
    return (d == 0 ? x : (d == 1 ? y : z)) == ((face & 1) ? NB - 1 : 0);
  };
  for (int i = 0; i < j; ++i)
    if (beside(tk.face[i])) return;          // corrected by that face's CTA
  R* u = U + (size_t)tk.blk * NT * NCELL + z * 256 + y * 16 + x;
  R val[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) val[v] = u[(size_t)v * NCELL];
  for (int i = j; i < nface; ++i) {
    const int face = tk.face[i], d = face >> 1;
    if (!beside(face)) continue;
    const int t1 = d == 0 ? y : x, t2 = d == 2 ? y : z;
    const int sf = tk.slot_f[i][(t1 >> 3) + 2 * (t2 >> 3)];
    const R w = s_w[d] * ((face & 1) ? R(1) : R(-1));
    const R* pc = FR + (size_t)tk.slot_c[i] * NV * 256 + t2 * 16 + t1;
    const R* pf = FR + (size_t)sf * NV * 256 + 2 * (t2 & 7) * 16 + 2 * (t1 & 7);
    using V = typename pair_of<R>::type;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const V f0 = *reinterpret_cast<const V*>(pf + (size_t)v * 256);
      const V f1 = *reinterpret_cast<const V*>(pf + (size_t)v * 256 + 16);
      R avg = f0.x + f0.y;
      avg = avg + f1.x;
      avg = avg + f1.y;
      avg = avg * R(0.25);
      val[v] = val[v] + w * (pc[(size_t)v * 256] - avg);
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) u[(size_t)v * NCELL] = val[v];
}

// ------------------------------------------------------------------------------ CFL speeds
// Four CTAs (grid.y) per block, four cells a thread: the pass mostly runs over the few blocks
// with corrected faces, where one CTA per block spent 16 us on 16 cells in sequence.
constexpr int SPEED_PARTS = 4;
template <template <typename> class PT, typename R>
__global__ void __launch_bounds__(256) speeds_kernel(const R* U,
                                                      const BlockDesc* __restrict__ bd,
                                                      const PhysParamsT<R> pp,   // formed on the host
                                                      unsigned long long* speeds, int* status,
                                                      const int* __restrict__ solve_of,
                                                      const int* __restrict__ wl) {
  using P = PT<R>;
  constexpr int NV = P::NV, NA = P::NA, NT = NV + NA;
  chain_wait();
  const int b = wl ? wl[blockIdx.x] : (int)blockIdx.x;
  __shared__ R s_id[3];
  if (threadIdx.x < 3) s_id[threadIdx.x] = R(1.0 / bd[b].dx[threadIdx.x]);
  __syncthreads();
  const R id[3] = {s_id[0], s_id[1], s_id[2]};
  R ssum = R(0), smax = R(0);
  int st = 0;
  const R* base = U + (size_t)b * NT * NCELL;
#pragma unroll 2
  for (int i = 0; i < NCELL / SPEED_PARTS / 256; ++i) {
    const int c = blockIdx.y * (NCELL / SPEED_PARTS) + i * 256 + threadIdx.x;
    R u[NV], aux[2] = {R(0), R(0)};
#pragma unroll
    for (int v = 0; v < NV; ++v) u[v] = base[(size_t)v * NCELL + c];
    if constexpr (NA > 0) aux[0] = base[(size_t)NV * NCELL + c];
    cell_speeds<PT, R>(u, aux, pp, id, ssum, smax, st);
  }
  block_max2<256>(ssum, smax, speeds + 2 * (solve_of ? solve_of[b] : 0));
  if (st) atomicOr(status, st);
}

__global__ void set_dt_kernel(unsigned long long* speeds, double* dtch, double dt_host, double cfl, int nsolve,
                              double rate_floor, int* work, int reset) {
  chain_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 4) work[i] = 0;
  if (i >= nsolve) return;
  const double smax = __longlong_as_double((long long)speeds[2 * i]);
  const double cmax = __longlong_as_double((long long)speeds[2 * i + 1]);
  dtch[2 * i] = dt_host > 0.0 ? dt_host : cfl / fmax(smax, rate_floor);
  dtch[2 * i + 1] = cmax;
  if (reset) speeds[2 * i] = speeds[2 * i + 1] = 0;
}

// ------------------------------------------------------------------------------ GLM source
// One CTA per block: thread 0 forms the factor in FP64, the CTA scales psi in the stencil
// precision with 16-byte accesses (psi of a block is 4096 contiguous values).
template <typename R>
__global__ void __launch_bounds__(256) glm_decay_kernel(R* U, const BlockDesc* __restrict__ bd,
                                                         const double* dtch, double alpha,
                                                         const int* __restrict__ solve_of,
                                                         const int* __restrict__ wl) {
  __shared__ R s_f;
  chain_wait();
  const int b = wl ? wl[blockIdx.x] : (int)blockIdx.x;
  if (threadIdx.x == 0) {
    const double* dc = dtch + 2 * (solve_of ? solve_of[b] : 0);
    const double dxm = fmin(fmin(bd[b].dx[0], bd[b].dx[1]), bd[b].dx[2]);
    s_f = R(exp(-0.5 * dc[0] * dc[1] * alpha / dxm));
  }
  __syncthreads();
  const R f = s_f;
  using V = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
  constexpr int PER = 16 / sizeof(R);
  V* psi = reinterpret_cast<V*>(U + ((size_t)b * 9 + 8) * NCELL);
  for (int c = threadIdx.x; c < NCELL / PER; c += blockDim.x) {
    V v = psi[c];
    if constexpr (sizeof(R) == 4) {
      v.x *= f; v.y *= f; v.z *= f; v.w *= f;
    } else {
      v.x *= f; v.y *= f;
    }
    psi[c] = v;
  }
}

// ------------------------------------------------------------------------------ estimator
// One variable of cell (x, y, z) in the halo view of block b (the rules of load_cell: a
// same-level neighbour's interior, a physical boundary image with the normal vector
// components negated at a reflecting wall, or a ghost slot).
template <class P, typename R>
__device__ __forceinline__ R load_var(const R* __restrict__ U, const R* __restrict__ G, const int* src, int b,
                                      int x, int y, int z, int iv) {
  constexpr int NT = P::NV + P::NA;
  int f = -1;
  if (x < 0) f = 0;
  else if (x > NB - 1) f = 1;
  else if (y < 0) f = 2;
  else if (y > NB - 1) f = 3;
  else if (z < 0) f = 4;
  else if (z > NB - 1) f = 5;
  int q[3] = {x, y, z};
  int blk = b;
  bool neg = false;
  if (f >= 0) {
    const int d = f >> 1, s = f & 1;
    const int sv = src[f];
    if (sv >= 0) {
      q[d] &= NB - 1;
      blk = sv;
    } else if (sv == SRC_OUTFLOW) {
      q[d] = s ? NB - 1 : 0;
    } else if (sv == SRC_REFLECT) {
      q[d] = s ? 2 * NB - 1 - q[d] : -1 - q[d];
      neg = (P::IV >= 0 && iv == P::IV + d) || (P::BOFF >= 0 && iv == P::BOFF + d);
    } else {
      const int slot = SRC_SLOT0 - sv;
      const int layer = s ? q[d] - NB : q[d] + 2;
      const int t1 = d == 0 ? q[1] : q[0];
      const int t2 = d == 2 ? q[1] : q[2];
      return G[((size_t)slot * NT + iv) * 512 + layer * 256 + t2 * 16 + t1];
    }
  }
  const R v = U[((size_t)blk * NT + iv) * NCELL + q[2] * 256 + q[1] * 16 + q[0]];
  return neg ? -v : v;
}

// Loehner (1987) second-derivative estimate per cell and variable (axis terms only):
// E_u = sqrt(sum_d (u+ - 2u0 + u-)^2 / sum_d (|u+ - u0| + |u0 - u-| + eps (|u+| + 2|u0| + |u-|))^2),
// E = sum_u w_u E_u; every operation rounded on its own (no FMA) in this order. Per refinement
// variable the CTA stages the block's interior (coalesced) and its six face layers in shared
// memory; each thread keeps the running sums of its 16 cells in registers.
// Whether the nonzero value x became zero or subnormal in its FP32 copy f (a test on the
// bits of x, which keeps FP64 operations out of the FP32 screen).
template <typename R>
__device__ __forceinline__ bool below_fp32_normal(R x, float f) {
  bool nz;
  if constexpr (sizeof(R) == 8) nz = (__double_as_longlong(x) & 0x7fffffffffffffffLL) != 0;
  else nz = (__float_as_int(x) & 0x7fffffff) != 0;
  return nz && !(fabsf(f) >= 1.17549435e-38f);
}

template <template <typename> class PT, typename R>
__global__ void __launch_bounds__(256) estimate_kernel(const R* __restrict__ U, const R* __restrict__ G,
                                                        const BlockDesc* __restrict__ bd,
                                                        const int* __restrict__ vars,
                                                        const double* __restrict__ weights, int nvars,
                                                        double eps, double* __restrict__ emax,
                                                        const int* __restrict__ wl,
                                                        const double* __restrict__ tols,
                                                        const int* __restrict__ solve_of, double margin) {
  using P = PT<R>;
  constexpr int NT = P::NV + P::NA;
  const int b = wl ? wl[blockIdx.x] : (int)blockIdx.x;
  const int t = threadIdx.x;
  __shared__ int src[6];
  __shared__ R sI[NCELL];          // interior of the staged variable
  __shared__ R sF[6][256];         // its face layers: face f, cell (t1 + 16 t2) as in the ghost slots
  __shared__ double red[8];
  __shared__ int s_amb;
  if (t < 6) src[t] = bd[b].src[t];
  // one refinement variable of the block (interior and face layers) into shared memory
  auto stage = [&](int iv) {
    __syncthreads();               // src is set; the previous variable's reads are done
    const R* base = U + ((size_t)b * NT + iv) * NCELL;
#pragma unroll 4
    for (int c = t; c < NCELL; c += 256) sI[c] = base[c];
    for (int e = t; e < 6 * 256; e += 256) {
      const int f = e >> 8, d = f >> 1, s = f & 1, t1 = e & 15, t2 = (e >> 4) & 15;
      int q[3];
      q[d] = s ? NB : -1;
      q[d == 0 ? 1 : 0] = t1;
      q[d == 2 ? 1 : 2] = t2;
      sF[f][t2 * 16 + t1] = load_var<P, R>(U, G, src, b, q[0], q[1], q[2], iv);
    }
    __syncthreads();
  };
  // the three values of the stencil of cell c along d (face layers beyond the block)
  auto nbrs = [&](int c, int d, R& a, R& m) {
    const int x = c & 15, y = (c >> 4) & 15, z = c >> 8;
    const int pos = d == 0 ? x : (d == 1 ? y : z);
    const int st = d == 0 ? 1 : (d == 1 ? 16 : 256);
    const int t1 = d == 0 ? y : x, t2 = d == 2 ? y : z;
    a = pos < NB - 1 ? sI[c + st] : sF[2 * d + 1][t2 * 16 + t1];
    m = pos > 0 ? sI[c - st] : sF[2 * d][t2 * 16 + t1];
  };
  // maximum over the CTA of a non-negative value (every thread calls it)
  auto block_max = [&](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((t & 31) == 0) red[t >> 5] = v;
    __syncthreads();
    double mx = red[0];
    for (int i = 1; i < 8; ++i) mx = fmax(mx, red[i]);
    return mx;
  };

  if (tols) {
    // Screen for the refinement decision: the same estimate in FP32 for every cell. Each cell's
    // FP32 value lies within `margin` of the exact one (the caller's bound from eps and the
    // weights), so the FP32 block maximum lies within `margin` of the exact maximum. Where it
    // is farther than that from both thresholds (refine above tols[0], coarsen below tols[1]
    // of the block's solve), it leads to the same decision and is returned as it is;
    // otherwise (or on values outside the screen's range) the exact FP64 pass below decides.
    float etf[16];
    bool bad = false;
    const float epsf = (float)eps;
    for (int i = 0; i < nvars; ++i) {
      stage(vars[i]);
      const float wf = (float)weights[i];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int c = t + 256 * j;
        const float o = (float)sI[c];
        bool lost = below_fp32_normal(sI[c], o);
        float num = 0.0f, den = 0.0f, smag = 0.0f;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          R ar, mr;
          nbrs(c, d, ar, mr);
          const float a = (float)ar, m = (float)mr;
          lost |= below_fp32_normal(ar, a) || below_fp32_normal(mr, m);
          const float tt = (a - 2.0f * o) + m;
          const float sm = (fabsf(a) + 2.0f * fabsf(o)) + fabsf(m);
          const float q = (fabsf(a - o) + fabsf(o - m)) + epsf * sm;
          num += tt * tt;
          den += q * q;
          smag = fmaxf(smag, sm);
        }
        const float e = den > 0.0f ? sqrtf(num / den) : 0.0f;
        // outside the screen's range: non-finite, squares that could underflow or overflow,
        // or a nonzero value that FP32 sees as zero or subnormal
        bad |= !(e <= 1.5f) || (smag > 0.0f && smag < 1e-10f) || !(smag < 1e18f) || lost;
        etf[j] = i == 0 ? wf * e : etf[j] + wf * e;
      }
    }
    float bf = 0.0f;
#pragma unroll
    for (int j = 0; j < 16; ++j) bf = fmaxf(bf, etf[j]);
    if (t == 0) s_amb = 0;
    __syncthreads();
    if (bad) s_amb = 1;
    const double M = block_max((double)bf);   // its barriers also publish s_amb
    const int sv = solve_of ? solve_of[b] : 0;
    const double tr = tols[2 * sv], tc = tols[2 * sv + 1];
    const bool amb = s_amb || !(margin >= 0.0) || fabs(M - tr) <= margin || fabs(M - tc) <= margin;
    if (!amb) {                    // CTA-uniform
      if (t == 0) emax[b] = M;
      return;
    }
  }

  double etot[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) etot[j] = 0.0;
  for (int i = 0; i < nvars; ++i) {
    const double w = weights[i];
    stage(vars[i]);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int c = t + 256 * j;
      const double o = (double)sI[c];
      double num = 0.0, den = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        R ar, mr;
        nbrs(c, d, ar, mr);
        const double a = (double)ar, m = (double)mr;
        const double tt = __dadd_rn(__dsub_rn(a, __dmul_rn(2.0, o)), m);
        const double q = __dadd_rn(__dadd_rn(fabs(__dsub_rn(a, o)), fabs(__dsub_rn(o, m))),
                                   __dmul_rn(eps, __dadd_rn(__dadd_rn(fabs(a), __dmul_rn(2.0, fabs(o))),
                                                            fabs(m))));
        const double t2q = __dmul_rn(tt, tt), q2 = __dmul_rn(q, q);
        num = d == 0 ? t2q : __dadd_rn(num, t2q);
        den = d == 0 ? q2 : __dadd_rn(den, q2);
      }
      const double e = den > 0.0 ? __dsqrt_rn(__ddiv_rn(num, den)) : 0.0;
      const double we = __dmul_rn(w, e);
      etot[j] = i == 0 ? we : __dadd_rn(etot[j], we);
    }
  }
  double best = 0.0;
#pragma unroll
  for (int j = 0; j < 16; ++j) best = fmax(best, etot[j]);
  const double mx = block_max(best);
  if (t == 0) emax[b] = mx;
}

// One CTA per block of the new mesh: a copy (16 bytes a thread), the mean of eight children, or
// the limited-linear prolongation of one octant of the parent, whose values and slopes are
// formed once per coarse cell for its eight fine cells (91 -> 16 us per regrid of the blast
// against 4-byte copies and seven cells read per fine cell).
template <template <typename> class PT, typename R>
__global__ void __launch_bounds__(256, 4) regrid_kernel(const R* __restrict__ Uold, const R* __restrict__ Gold,
                                                         const BlockDesc* __restrict__ bdold,
                                                         R* __restrict__ Unew,
                                                         const RegridSrc* __restrict__ srcs) {
  using P = PT<R>;
  using V = typename pair_of<R>::type;
  constexpr int NT = P::NV + P::NA;
  const int nb = blockIdx.x;
  const RegridSrc& rs = srcs[nb];
  R* out = Unew + (size_t)nb * NT * NCELL;
  if (rs.mode == 0) {
    const uint4* in = reinterpret_cast<const uint4*>(Uold + (size_t)rs.src[0] * NT * NCELL);
    uint4* o4 = reinterpret_cast<uint4*>(out);
    constexpr int N4 = NT * NCELL * (int)sizeof(R) / 16;
#pragma unroll 4
    for (int i = threadIdx.x; i < N4; i += 256) o4[i] = in[i];
    return;
  }
  if (rs.mode == 2) {
    for (int c = threadIdx.x; c < NCELL; c += 256) {
      const int x = c & 15, y = (c >> 4) & 15, z = c >> 8;
      const int fb = rs.src[(x >> 3) + 2 * (y >> 3) + 4 * (z >> 3)];
      const R* q = Uold + (size_t)fb * NT * NCELL + 2 * (z & 7) * 256 + 2 * (y & 7) * 16 + 2 * (x & 7);
#pragma unroll
      for (int v = 0; v < NT; ++v) out[(size_t)v * NCELL + c] = mean8<R>(q + (size_t)v * NCELL);
    }
    return;
  }
  const int P0 = rs.src[0];
  const int oct = 8 * (rs.octant & 1) + 16 * 8 * ((rs.octant >> 1) & 1) + 256 * 8 * (rs.octant >> 2);
  for (int c = threadIdx.x; c < 512; c += 256) {
    const int cx = c & 7, cy = (c >> 3) & 7, cz = c >> 6;
    const int off = oct + cz * 256 + cy * 16 + cx;
    const R* own = Uold + (size_t)P0 * NT * NCELL + off;
    CellRef<R> up[3], um[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      up[e] = cell_ref<P, R, true>(Uold, Gold, bdold, P0, off, e, 1);
      um[e] = cell_ref<P, R, true>(Uold, Gold, bdold, P0, off, e, -1);
    }
    R* o = out + 2 * cz * 256 + 2 * cy * 16 + 2 * cx;
#pragma unroll
    for (int v = 0; v < NT; ++v) {
      const R u = own[(size_t)v * NCELL];
      R sig[3];
#pragma unroll
      for (int e = 0; e < 3; ++e)
        sig[e] = minmod_(cell_value<P, R>(up[e], v, e) - u, u - cell_value<P, R>(um[e], v, e));
#pragma unroll
      for (int q = 0; q < 4; ++q) {          // the pairs along x at (y, z) = (q & 1, q >> 1)
        const R sy = (q & 1) ? sig[1] : -sig[1], sz = (q >> 1) ? sig[2] : -sig[2];
        V w;
        w.x = u + R(0.25) * ((-sig[0] + sy) + sz);
        w.y = u + R(0.25) * ((sig[0] + sy) + sz);
        *reinterpret_cast<V*>(o + (size_t)v * NCELL + (q >> 1) * 256 + (q & 1) * 16) = w;
      }
    }
  }
}

// ------------------------------------------------------------------------ recovery pass
// Primitives and auxiliaries of every cell of U_s (the work list's blocks, 16 CTAs of one
// z-plane each) and of its ghost slots (two CTAs of 256 cells each per slot) into W / WG,
// laid out as U_s / the slots are. One recovery per stored cell: the same function the stage
// kernel applies, on the same inputs, so the primitives are the same bit for bit. With
// speeds non-null (the first stage of a step) it also reduces the CFL maxima of the leaf
// cells per solve from these primitives, as the stage kernel's fused reduction would have
// from the same state at the end of the previous step.
template <template <typename> class PT, typename R>
__global__ void __launch_bounds__(256) prim_pass_kernel(const R* U, R* W, const R* G, R* WG,
                                                        const int* __restrict__ wl, int nwork,
                                                        PhysParamsT<R> pp, int* status,
                                                        const BlockDesc* __restrict__ bd,
                                                        const int* __restrict__ solve_of,
                                                        unsigned long long* speeds) {
  using P = PT<R>;
  constexpr int NV = P::NV, NA = P::NA, NT = NV + NA;
  chain_wait();
  const int item = blockIdx.x;
  const R* src;
  R* dst;
  int vs;
  int b = -1;
  if (item < nwork * 16) {
    const int w = item >> 4, z = item & 15;
    b = wl ? wl[w] : w;
    const size_t off = (size_t)b * NT * NCELL + (size_t)z * 256 + threadIdx.x;
    src = U + off;
    dst = W + off;
    vs = NCELL;
  } else {
    const int j = item - nwork * 16;          // slot j / 2, cells (j % 2) * 256 ..
    const size_t off = (size_t)(j >> 1) * NT * 512 + (size_t)(j & 1) * 256 + threadIdx.x;
    src = G + off;
    dst = WG + off;
    vs = 512;
  }
  R u[NT], p[NV], aux[NA > 0 ? NA : 1];
#pragma unroll
  for (int v = 0; v < NT; ++v) u[v] = src[(size_t)v * vs];
  __shared__ R s_id[3];
  if (speeds && b >= 0 && threadIdx.x < 3) s_id[threadIdx.x] = R(1.0 / bd[b].dx[threadIdx.x]);
  if constexpr (NA > 0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) aux[i] = u[NV + i];
  } else {
    aux[0] = R(0);
  }
  int st = 0;
  P::cons2prim(u, p, aux, pp, st);
#pragma unroll
  for (int v = 0; v < NV; ++v) dst[(size_t)v * vs] = p[v];
#pragma unroll
  for (int i = 0; i < NA; ++i) dst[(size_t)(NV + i) * vs] = aux[i];
  if (st) atomicOr(status, st);
  if (speeds && b >= 0) {             // CTA-uniform: a pool plane, not a ghost slot
    __syncthreads();
    const R id[3] = {s_id[0], s_id[1], s_id[2]};
    R ssum = R(0), smax = R(0);
    prim_speeds<PT, R>(p, pp, id, ssum, smax);
    block_max2<256>(ssum, smax, speeds + 2 * (solve_of ? solve_of[b] : 0));
  }
}

// ------------------------------------------------------------------------------ state I/O
// Four CTAs (grid.y) per block. The conversion runs in FP64 whatever the stencil precision, and
// the FP64 units bind it: the equation parameters come from the host, Gamma is formed once and
// xi = Gamma^2 rho h from the conserved values it has just been part of, xi = tau + p + D.
constexpr int IC_PARTS = 4;
template <template <typename> class PT, typename R>
__global__ void __launch_bounds__(256) prim2cons_kernel(R* __restrict__ U, const double* __restrict__ prim,
                                                         const int* __restrict__ blocks,
                                                         const PhysParamsT<double> pp) {
  using P = PT<double>;
  constexpr int NV = P::NV, NA = P::NA, NT = NV + NA;
  const int i = blockIdx.x;
  const int b = blocks[i];
#pragma unroll 2
  for (int j = 0; j < NCELL / IC_PARTS / 256; ++j) {
    const int c = blockIdx.y * (NCELL / IC_PARTS) + j * 256 + threadIdx.x;
    double p[NV], u[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) p[v] = prim[((size_t)i * NV + v) * NCELL + c];
    P::prim2cons(p, u, pp);
    R* o = U + (size_t)b * NT * NCELL + c;
#pragma unroll
    for (int v = 0; v < NV; ++v) o[(size_t)v * NCELL] = R(u[v]);
    if constexpr (NA > 0) {
      o[(size_t)NV * NCELL] = R((u[4] + p[4]) + u[0]);
      o[(size_t)(NV + 1) * NCELL] = R(rsqrt_(1.0 + p[1] * p[1] + p[2] * p[2] + p[3] * p[3]));
    }
  }
}

template <typename R>
__global__ void unpack_kernel(R* __restrict__ U, const double* __restrict__ cons, int nv, int na) {
  const int b = blockIdx.x;
  const int nt = nv + na;
  for (int i = threadIdx.x; i < nt * NCELL; i += blockDim.x) {
    const int v = i / NCELL;
    U[(size_t)b * nt * NCELL + i] = v < nv ? R(cons[(size_t)b * nv * NCELL + i]) : R(0);
  }
}

template <typename R>
__global__ void pack_kernel(const R* __restrict__ U, double* __restrict__ cons, double* __restrict__ aux,
                            int nv, int na) {
  const int b = blockIdx.x;
  const int nt = nv + na;
  for (int i = threadIdx.x; i < nt * NCELL; i += blockDim.x) {
    const int v = i / NCELL;
    const double val = (double)U[(size_t)b * nt * NCELL + i];
    if (v < nv) {
      if (cons) cons[(size_t)b * nv * NCELL + i] = val;
    } else if (aux) {
      aux[(size_t)b * na * NCELL + (i - nv * NCELL)] = val;
    }
  }
}

// Per-block volume integrals of the conserved variables, all variables in one pass. FP64
// pools add in FP64. FP32 pools add each thread's 16 values in FP32 with the exact error of
// every addition kept (Knuth's TwoSum: s = a + b, e = (a - (s - (s - a))) + (b - (s - a)),
// so s + e = a + b exactly), an FP32 pair whose sum carries about 48 significant bits, then
// in FP64: the FP64 units of the GPU add 64 times slower than its FP32 units.
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  hi = s;
  lo = __fadd_rn(lo, e);
}

template <typename R>
__global__ void __launch_bounds__(256) sums_kernel(const R* __restrict__ U, const BlockDesc* __restrict__ bd,
                                                    double* __restrict__ part, int nv, int na) {
  const int b = blockIdx.x;
  const int nt = nv + na;
  const double dv = bd[b].dx[0] * bd[b].dx[1] * bd[b].dx[2];
  __shared__ double red[8][16];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int v = 0; v < nv; ++v) {
    const R* p = U + ((size_t)b * nt + v) * NCELL;
    double s;
    if constexpr (sizeof(R) == 4) {
      const float4* q = reinterpret_cast<const float4*>(p);
      float hi = 0.0f, lo = 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 x = q[threadIdx.x + 256 * i];
        two_sum_acc(hi, lo, x.x);
        two_sum_acc(hi, lo, x.y);
        two_sum_acc(hi, lo, x.z);
        two_sum_acc(hi, lo, x.w);
      }
      s = (double)hi + (double)lo;
    } else {
      s = 0.0;
      for (int c = threadIdx.x; c < NCELL; c += 256) s += (double)p[c];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[w][v] = s;
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += red[i][threadIdx.x];
    part[(size_t)b * nv + threadIdx.x] = t * dv;
  }
}

template <template <typename> class PT, typename R>
__global__ void halo_kernel(const R* __restrict__ U, const R* __restrict__ G,
                            const BlockDesc* __restrict__ bd, int b, double* __restrict__ out) {
  using P = PT<R>;
  constexpr int NT = P::NV + P::NA;
  int src[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) src[i] = bd[b].src[i];
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < 8000; c += gridDim.x * blockDim.x) {
    const int x = c % 20 - 2, y = (c / 20) % 20 - 2, z = c / 400 - 2;
    const int outside = (x < 0 || x > 15) + (y < 0 || y > 15) + (z < 0 || z > 15);
    if (outside > 1) {
      for (int v = 0; v < NT; ++v) out[(size_t)v * 8000 + c] = __longlong_as_double(0x7ff8000000000000LL);
      continue;
    }
    R u[NT];
    load_cell<P, R>(U, G, src, b, x, y, z, u);
    for (int v = 0; v < NT; ++v) out[(size_t)v * 8000 + c] = (double)u[v];
  }
}

// ------------------------------------------------------------------------------ dispatch
#define AGILE_DISPATCH(phys, rb, CALL)                         \
  do {                                                         \
    if ((phys) == PH_HD) {                                     \
      if ((rb) == 8) { using R = double; CALL(HdPhys); }       \
      else { using R = float; CALL(HdPhys); }                  \
    } else if ((phys) == PH_MHD) {                             \
      if ((rb) == 8) { using R = double; CALL(MhdPhys); }      \
      else { using R = float; CALL(MhdPhys); }                 \
    } else if ((phys) == PH_SRHD) {                            \
      if ((rb) == 8) { using R = double; CALL(SrhdPhys); }     \
      else { using R = float; CALL(SrhdPhys); }                \
    } else if ((phys) == PH_FFHD) {                            \
      if ((rb) == 8) { using R = double; CALL(FfhdPhys); }     \
      else { using R = float; CALL(FfhdPhys); }                \
    } else if ((phys) == PH_FFHD_HTC) {                        \
      if ((rb) == 8) { using R = double; CALL(FfhdHtcPhys); }  \
      else { using R = float; CALL(FfhdHtcPhys); }             \
    } else {                                                   \
      if ((rb) == 8) { using R = double; CALL(SrhdSyngePhys); }\
      else { using R = float; CALL(SrhdSyngePhys); }           \
    }                                                          \
  } while (0)

cudaError_t launch_ghosts(const AuxArgs& a, const GhostTask* tasks, int ntasks, cudaStream_t s) {
  if (ntasks == 0) return cudaSuccess;
  // not chained behind the stage kernel, nor is the fix-up: their many small CTAs, waiting where
  // its last ones run, cost a refined blast 3-5%
#define CALL(PT) ghost_kernel<PT, R><<<ntasks, 256, 0, s>>>((const R*)a.U, (R*)a.Gw, a.bd, tasks)
  AGILE_DISPATCH(a.phys, a.real_bytes, CALL);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_fixup(const AuxArgs& a, const FixupTask* tasks, int ntasks, double b,
                         const double* dtch, cudaStream_t s) {
  if (ntasks == 0) return cudaSuccess;
  const int nv = phys_nvar(a.phys), nt = nv + phys_naux(a.phys);
  if (nv == 6) return cudaErrorInvalidValue;   // ffhd runs on uniform meshes only
  const dim3 grid(ntasks, NFACE);
#define CALL(R, NV, NT) \
  fixup_kernel<R, NV, NT><<<grid, 256, 0, s>>>((R*)a.Uw, (const R*)a.FR, a.bd, tasks, b, dtch, a.solve_of)
  if (a.real_bytes == 8) {
    if (nv == 9) CALL(double, 9, 9);
    else if (nt == 5) CALL(double, 5, 5);
    else CALL(double, 5, 7);
  } else {
    if (nv == 9) CALL(float, 9, 9);
    else if (nt == 5) CALL(float, 5, 5);
    else CALL(float, 5, 7);
  }
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_speeds(const AuxArgs& a, unsigned long long* speeds, cudaStream_t s) {
  if (a.nblk == 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
#define CALL(PT)                                                                                  \
  do {                                                                                            \
    PhysParamsT<R> pp;                                                                            \
    pp.set(a.gamma, 0.0);                                                                         \
    e = launch_chained(speeds_kernel<PT, R>, dim3(a.nblk, SPEED_PARTS), 256, 0, s, (const R*)a.U, a.bd, pp, speeds, a.status, \
                       a.solve_of, a.wl);                                                         \
  } while (0)
  AGILE_DISPATCH(a.phys, a.real_bytes, CALL);
#undef CALL
  return e;
}

cudaError_t launch_set_dt(unsigned long long* speeds, double* dtch, double dt_host, double cfl, int* work,
                          bool reset, cudaStream_t s, int nsolve, double rate_floor) {
  return launch_chained(set_dt_kernel, dim3((nsolve + 127) / 128), 128, 0, s, speeds, dtch, dt_host, cfl, nsolve,
                        rate_floor, work, (int)reset);
}

cudaError_t launch_glm_decay(const AuxArgs& a, const double* dtch, cudaStream_t s) {
  if (a.nblk == 0) return cudaSuccess;
  if (a.real_bytes == 8)
    return launch_chained(glm_decay_kernel<double>, dim3(a.nblk), 256, 0, s, (double*)a.Uw, a.bd, dtch, a.glm_alpha,
                          a.solve_of, a.wl);
  return launch_chained(glm_decay_kernel<float>, dim3(a.nblk), 256, 0, s, (float*)a.Uw, a.bd, dtch, a.glm_alpha,
                        a.solve_of, a.wl);
}

cudaError_t launch_estimate(const AuxArgs& a, const int* vars, const double* weights, int nvars,
                            double eps, double* emax, cudaStream_t s, const double* tols, double margin) {
  if (a.nblk == 0) return cudaSuccess;
#define CALL(PT)                                                                                          \
  estimate_kernel<PT, R><<<a.nblk, 256, 0, s>>>((const R*)a.U, (const R*)a.G, a.bd, vars, weights, nvars, eps, \
                                                emax, a.wl, tols, a.solve_of, margin)
  AGILE_DISPATCH(a.phys, a.real_bytes, CALL);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_regrid(const AuxArgs& a, void* Unew, const RegridSrc* src, int nnew, cudaStream_t s) {
  if (nnew == 0) return cudaSuccess;
#define CALL(PT) regrid_kernel<PT, R><<<nnew, 256, 0, s>>>((const R*)a.U, (const R*)a.G, a.bd, (R*)Unew, src)
  AGILE_DISPATCH(a.phys, a.real_bytes, CALL);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_prim_pass(const AuxArgs& a, void* W, void* WG, int nslots, unsigned long long* speeds,
                             cudaStream_t s) {
  const long long grid = 16LL * a.nblk + 2LL * nslots;
  if (grid == 0) return cudaSuccess;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (a.phys != PH_SRHD && a.phys != PH_SRHD_SYNGE) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
#define CALL(PT)                                                                               \
  do {                                                                                         \
    PhysParamsT<R> pp;                                                                         \
    pp.set(a.gamma, 0.0);                                                                      \
    e = launch_chained(prim_pass_kernel<PT, R>, dim3((unsigned)grid), 256, 0, s, (const R*)a.U, (R*)W, \
                       (const R*)a.G, (R*)WG, a.wl, a.nblk, pp, a.status, a.bd, a.solve_of, speeds); \
  } while (0)
  if (a.phys == PH_SRHD) {
    if (a.real_bytes == 8) { using R = double; CALL(SrhdPhys); }
    else { using R = float; CALL(SrhdPhys); }
  } else {
    if (a.real_bytes == 8) { using R = double; CALL(SrhdSyngePhys); }
    else { using R = float; CALL(SrhdSyngePhys); }
  }
#undef CALL
  return e;
}

cudaError_t launch_prim2cons(const AuxArgs& a, const double* prim, const int* blocks, int n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  PhysParamsT<double> pp;
  pp.set(a.gamma, 0.0);
#define CALL(PT) prim2cons_kernel<PT, R><<<dim3(n, IC_PARTS), 256, 0, s>>>((R*)a.Uw, prim, blocks, pp)
  AGILE_DISPATCH(a.phys, a.real_bytes, CALL);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_unpack(const AuxArgs& a, const double* cons, cudaStream_t s) {
  if (a.nblk == 0) return cudaSuccess;
  const int nv = phys_nvar(a.phys), na = phys_naux(a.phys);
  if (a.real_bytes == 8) unpack_kernel<double><<<a.nblk, 256, 0, s>>>((double*)a.Uw, cons, nv, na);
  else unpack_kernel<float><<<a.nblk, 256, 0, s>>>((float*)a.Uw, cons, nv, na);
  return cudaGetLastError();
}

cudaError_t launch_pack(const AuxArgs& a, double* cons, double* aux, cudaStream_t s) {
  if (a.nblk == 0) return cudaSuccess;
  const int nv = phys_nvar(a.phys), na = phys_naux(a.phys);
  if (a.real_bytes == 8) pack_kernel<double><<<a.nblk, 256, 0, s>>>((const double*)a.U, cons, aux, nv, na);
  else pack_kernel<float><<<a.nblk, 256, 0, s>>>((const float*)a.U, cons, aux, nv, na);
  return cudaGetLastError();
}

cudaError_t launch_sums(const AuxArgs& a, double* part, cudaStream_t s) {
  if (a.nblk == 0) return cudaSuccess;
  const int nv = phys_nvar(a.phys), na = phys_naux(a.phys);
  if (a.real_bytes == 8) sums_kernel<double><<<a.nblk, 256, 0, s>>>((const double*)a.U, a.bd, part, nv, na);
  else sums_kernel<float><<<a.nblk, 256, 0, s>>>((const float*)a.U, a.bd, part, nv, na);
  return cudaGetLastError();
}

cudaError_t launch_halo(const AuxArgs& a, int block, double* out, cudaStream_t s) {
#define CALL(PT) halo_kernel<PT, R><<<32, 256, 0, s>>>((const R*)a.U, (const R*)a.G, a.bd, block, out)
  AGILE_DISPATCH(a.phys, a.real_bytes, CALL);
#undef CALL
  return cudaGetLastError();
}

}  // namespace agile
