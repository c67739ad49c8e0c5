// Device self-checks of the stencil's arithmetic: its functions evaluated one by one on values the
// caller chooses, so that the stated error bounds can be tested without a solver around them.
#include "agile.h"
#include "physics.cuh"

#include <algorithm>

namespace agile {
namespace {

__global__ void fp64_kernel(int op, const double* a, const double* b, size_t n, double* out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double x = a[i], y = b[i];
    double r = 0.0;
    if (op == AGILE_FP64_SQRT) r = rsqrt_(x);
    else if (op == AGILE_FP64_SQRT_QUOTIENT) r = rsqrt_div(x, y);
    else if (op == AGILE_FP64_MIN) r = rmin(x, y);
    else if (op == AGILE_FP64_MAX) r = rmax(x, y);
    else if (op == AGILE_FP64_POSITIVE) r = rpos(x) ? 1.0 : 0.0;
    else r = rneg(x) ? 1.0 : 0.0;
    out[i] = r;
  }
}

// The relativistic recovery of the FP32 stencil, and whether its last step ran in FP32 pairs.
template <int EOS>
__global__ void recover_kernel(const float* cons, const float* start, size_t n, PhysParamsT<float> pp, float* out) {
  using P = SrhdPhysE<float, EOS>;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    float u[5], p[5], aux[2] = {start[i], 0.0f};
    for (int v = 0; v < 5; ++v) u[v] = cons[5 * i + v];
    float x, lo, hi, s2;
    P::bracket(u, aux[0], pp, x, lo, hi, s2);
    float q[5], qa[2];
    const bool pairs = P::seed_f32(x, u[0], s2, lo, lo, hi, pp) && P::finish_pairs(u, x, lo, hi, q, qa, pp);
    int st = 0;
    P::cons2prim(u, p, aux, pp, st);
    for (int v = 0; v < 5; ++v) out[8 * i + v] = p[v];
    out[8 * i + 5] = aux[0];
    out[8 * i + 6] = aux[1];
    out[8 * i + 7] = st ? -1.0f : (pairs ? 1.0f : 0.0f);
  }
}

// Device copies of host arrays for one check, freed in stream order.
struct Buffers {
  cudaStream_t s;
  cudaError_t e = cudaSuccess;
  void* p[4] = {nullptr, nullptr, nullptr, nullptr};
  explicit Buffers(cudaStream_t s_) : s(s_) {}
  ~Buffers() {
    for (void* q : p)
      if (q) cudaFreeAsync(q, s);
  }
  template <typename T>
  T* get(int i, size_t bytes, const T* from = nullptr) {
    if (e == cudaSuccess) e = cudaMallocAsync(&p[i], bytes, s);
    if (e == cudaSuccess && from) e = cudaMemcpyAsync(p[i], from, bytes, cudaMemcpyHostToDevice, s);
    return static_cast<T*>(p[i]);
  }
  template <typename T>
  void back(T* to, int i, size_t bytes) {
    if (e == cudaSuccess) e = cudaMemcpyAsync(to, p[i], bytes, cudaMemcpyDeviceToHost, s);
  }
};

}  // namespace
}  // namespace agile

extern "C" agile_status agile_selftest_fp64(int op, const double* a, const double* b, size_t n, void* stream,
                                            double* out) {
  using namespace agile;
  if (!a || !b || !out || n == 0 || n > ((size_t)1 << 26) || op < 0 || op > AGILE_FP64_NOT_NONNEGATIVE)
    return AGILE_EINVAL;
  Buffers d((cudaStream_t)stream);
  const size_t bytes = n * sizeof(double);
  const double *da = d.get(0, bytes, a), *db = d.get(1, bytes, b);
  double* dout = d.get<double>(2, bytes);
  if (d.e == cudaSuccess) {
    fp64_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, d.s>>>(op, da, db, n, dout);
    d.e = cudaGetLastError();
  }
  d.back(out, 2, bytes);
  if (d.e == cudaSuccess) d.e = cudaStreamSynchronize(d.s);
  return d.e == cudaSuccess ? AGILE_OK : AGILE_ECUDA;
}

extern "C" agile_status agile_selftest_recover32(int eos, double gamma, const float* cons, const float* start, size_t n,
                                                 void* stream, float* out) {
  using namespace agile;
  if (!cons || !start || !out || n == 0 || n > ((size_t)1 << 26) || !(gamma > 1.0) ||
      (eos != AGILE_EOS_IDEAL && eos != AGILE_EOS_SYNGE))
    return AGILE_EINVAL;
  Buffers d((cudaStream_t)stream);
  const float *dc = d.get(0, 5 * n * sizeof(float), cons), *ds = d.get(1, n * sizeof(float), start);
  float* dout = d.get<float>(2, 8 * n * sizeof(float));
  PhysParamsT<float> pp;
  pp.set(gamma, 0.0);
  if (d.e == cudaSuccess) {
    const unsigned grid = (unsigned)std::min<size_t>((n + 255) / 256, 4096);
    if (eos == AGILE_EOS_SYNGE) recover_kernel<EOS_SYNGE><<<grid, 256, 0, d.s>>>(dc, ds, n, pp, dout);
    else recover_kernel<EOS_IDEAL><<<grid, 256, 0, d.s>>>(dc, ds, n, pp, dout);
    d.e = cudaGetLastError();
  }
  d.back(out, 2, 8 * n * sizeof(float));
  if (d.e == cudaSuccess) d.e = cudaStreamSynchronize(d.s);
  return d.e == cudaSuccess ? AGILE_OK : AGILE_ECUDA;
}
