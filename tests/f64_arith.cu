// f64_arith.cu -- the arithmetic of the FP64 basis kernels (musr_kernels_f64.cuh) on arrays, for
// test_gpu_f64_arith.py: the logarithm, the reciprocals and a thread's time factors.
#include "musr_kernels_f64.cuh"

namespace musr {
namespace kern {
namespace {

__global__ void elementwise(int what, const double* __restrict__ x, double* __restrict__ y, int n) {
  __shared__ double2 tab[kLogTable];
  for (int i = threadIdx.x; i < kLogTable; i += blockDim.x) tab[i] = log_table.t[i];
  __syncthreads();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    y[i] = what == 0 ? ln_tab(x[i], tab) : what == 1 ? recip_any(x[i]) : count_weight(x[i], false);
}

// One CTA through `iters` iterations of kBlock bins of a one-term theory without an envelope: P of
// every bin, cosine and sine part.
template <int SHAPE>
__global__ void __launch_bounds__(kBlock, 1) factors(int kind, double lam, double sigma, double kt, double nu, double dt,
                                                     double t0, int iters, double2* __restrict__ P) {
  __shared__ Smem64 sm;
  __shared__ Job job;
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(Smem64) / 4); i += kBlock) reinterpret_cast<int*>(&sm)[i] = 0;
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(Job) / 4); i += kBlock) reinterpret_cast<int*>(&job)[i] = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    HistSet& hs = sm.hs;
    hs.H = hs.nterms = 1;
    hs.nslots = 7;
    hs.dt_us = dt;
    hs.tile_bins = iters * kBlock;
    CanonTerm& ct = hs.canon[0];
    ct.kind = kind;
    ct.amp_slot = -1;
    ct.nexp = ct.ngauss = 1;
    ct.exp_slot[0] = 2;
    ct.gauss_slot[0] = 3;
    ct.kt_slot = 4;
    ct.nu_slot = 5;
    ct.phi_slot = 6;
    ChunkCache& cc = sm.cc;
    cc.nh = 1;
    cc.nhi = iters * kBlock;
    cc.t0 = t0;
    const double loc[7] = {1.0, 0.0, lam, sigma, kt, nu, 0.0};
    for (int s = 0; s < 7; ++s) cc.loc[0][s] = loc[s];
  }
  __syncthreads();
  load_chunk64<SHAPE>(job, sm.hs, sm);
  TimeFactors<SHAPE> tf;
  double nd = 0.0, t_fresh = 0.0;
  for (int it = 0; it < iters; ++it) {  // as basis64_item
    const int n = it * kBlock + threadIdx.x, step = sm.c.safe ? it & (kRebase - 1) : 0;
    if (step == 0) {
      nd = __dadd_rn(static_cast<double>(n), -sm.cc.t0);
      t_fresh = __dmul_rn(nd, dt);
    }
    double t = t_fresh;
    if (step != 0) t = __dadd_rn(t, sm.c.td[step]);
    double E, Pc[1], Ps[1], dK[1];
    tf.at(job, sm.hs, sm.c, step, iters > 1, nd, t, &E, Pc, Ps, dK);
    P[n] = make_double2(Pc[0], kind == kTermTF ? Ps[0] : 0.0);
  }
}

}  // namespace
}  // namespace kern
}  // namespace musr

using namespace musr;
using namespace musr::kern;

// what: 0 ln x, 1 1 / x, 2 1 / max(x, 1); x, y: host arrays of n values.  Returns a cudaError_t.
extern "C" int f64_elementwise(int what, const double* x, double* y, int n) {
  double* d = nullptr;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&d), 2 * sizeof(double) * n);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    elementwise<<<64, 256>>>(what, d, d + n, n);
    e = cudaMemcpy(y, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  return e;
}

// kind: a TermKind of musr_dev.h; P: host array of iters * 256 (cosine, sine) pairs.
extern "C" int f64_factors(int kind, double lam, double sigma, double kt, double nu, double dt, double t0, int iters,
                           double* P) {
  double2* d = nullptr;
  const size_t bytes = sizeof(double2) * kBlock * iters;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&d), bytes);
  if (e != cudaSuccess) return e;
  if (kind == kTermTF)
    factors<kShapeT1><<<1, kBlock>>>(kind, lam, sigma, kt, nu, dt, t0, iters, d);
  else
    factors<kShapeN1><<<1, kBlock>>>(kind, lam, sigma, kt, nu, dt, t0, iters, d);
  e = cudaMemcpy(P, d, bytes, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e;
}
