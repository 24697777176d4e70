// musr_fftconv.h -- FP64 convolution on the doubled mesh by pruned transforms (musr_fftconv.cu),
// the FP64 path of the particle-mesh Poisson solve (musr_poisson.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace musr {

constexpr int kFftMaxPasses = 12;
constexpr int kFftMaxLen = 4096;  // longest half-transform of an axis (a block holds at least one line)

// One axis: mesh points m, the length mp >= m of its two half transforms (a product of 2, 3, 5 and 7),
// their radices, first pass first, and each pass's sub-transform length.
struct FftAxis {
  int m, mp, npass;
  int radix[kFftMaxPasses], sub[kFftMaxPasses];
  const double2* tw;  // [2 mp] exp(-2 pi i k / (2 mp))
  const int* pos;     // [mp] storage position of frequency k of a half transform
};

struct FftConv {
  FftAxis x, y, z;
  int num_sms = 1;
  int nzc = 0;              // spectrum columns per (x, y) line: mp_z + 1
  double2* a = nullptr;     // [m_x][m_y][nzc]
  double2* b = nullptr;     // [m_x][2 mp_y][nzc]
  double* ghat = nullptr;   // [2 mp_x][2 mp_y][nzc]: the kernel's (real) transform, scaled
  void* tables = nullptr;   // twiddles and positions
};

// Axis lengths for a mesh; false where an axis is too long for these kernels, or long with few lines.
bool fftconv_plan(FftConv* c, int mx, int my, int mz, int num_sms);
// The tables on the device; the buffers of a solve.
cudaError_t fftconv_tables(FftConv* c);
cudaError_t fftconv_buffers(FftConv* c);
void fftconv_free(FftConv* c);
// ghat from the real parts of the kernel's transform hat ([2 mp_x][2 mp_y][mp_z + 1] complex, natural
// order), times `scale` over the transforms' normalisation.
cudaError_t fftconv_set_kernel(FftConv* c, const double2* hat, double scale, cudaStream_t s);
// phi = the convolution of rho with the kernel on the mesh ([m_x][m_y][m_z]); five launches.
cudaError_t fftconv_solve(const FftConv* c, const double* rho, double* phi, cudaStream_t s);

}  // namespace musr
