// musr_fftconv.cu -- convolution of an mx x my x mz density with a kernel known by its transform on
// the doubled mesh, in FP64 (sm_103a).
//
// What binds it: the FP64 pipe (one warp instruction per 16 clocks and SM).  A 3-D library transform
// of the doubled mesh was already there at 86 % of that pipe's peak, but it transforms all eight
// octants forward and back although seven hold zeros going in and are dropped coming out.  Here
// each axis's transform runs on the lines that hold something: 1/4 of the z lines, 1/2 of the y
// lines, all x lines, and each of length 2 mp as two transforms of length mp (Hockney's doubled
// axis: even frequencies are the transform of the mp points, odd ones that of the points times
// exp(-i pi n / mp); going back the two are combined the same way), so that neither the zeros nor
// the dropped half cost an operation.
//
//   z  forward   pairs of real lines as one complex line; the two spectra separated
//   y  forward   [x][my][c] -> [x][2 mp_y][c]
//   x            forward, times the kernel's real transform, inverse, in one kernel
//   y  inverse, z inverse (two real lines at once)
//
// A block holds 2 C half lines (C neighbouring columns, both halves) in shared memory, the column
// fastest, and runs the radix passes in place: forward decimation in frequency leaves the
// frequencies in digit-reversed order, the inverse starts from it, and the kernel's transform is
// stored in that order, so nothing is ever reordered.  Radix 8 with its sqrt(1/2) factors folded
// into multiply-adds takes 6.5 instructions per point and pass, a twiddle 4.
//
// Measured on GB300 (256 x 256 x 128, device arrays): 15.33 -> 6.16 ms a solve (z 0.43 + 0.44, y 0.88 +
// 0.91, x 3.50 ms; 26 FP64 instructions per point of a y transform, 55 per point of the x convolution;
// the pipe 83-86 % of its peak busy; DRAM below 0.5 TB/s).  37 x 44 x 23: 189 -> 64 us.
//
// The half length mp is the product of 2, 3, 5 and 7 at or above m that needs the fewest
// instructions (m itself where it is such a product): the padded circular length 2 mp >= 2 m gives
// the same linear convolution.  Axes whose half length would exceed 4096 stay with the library's
// transform (a block could not hold a line's two halves), as do long axes with few lines (fftconv_plan).
#include "musr_fftconv.h"

#include <cmath>
#include <vector>

namespace musr {
namespace {

constexpr int kThreads = 256;

// -------------------------------------------------------------------------------------------
// Butterflies: y_q = sum_t x_t exp(-+ 2 pi i t q / R), natural order (upper sign: forward).
// -------------------------------------------------------------------------------------------
__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
template <bool INV>
__device__ __forceinline__ double2 rot(double2 a) {  // times -i (forward) or i
  return INV ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}
template <bool CONJ>
__device__ __forceinline__ double2 mul(double2 a, double2 w) {  // a w or a conj(w)
  return CONJ ? make_double2(fma(a.x, w.x, a.y * w.y), fma(a.y, w.x, -(a.x * w.y)))
              : make_double2(fma(a.x, w.x, -(a.y * w.y)), fma(a.y, w.x, a.x * w.y));
}

// cos and sin of 2 pi k / R for the odd radices.
__device__ __forceinline__ constexpr double cos_of(int R, int k) {
  return R == 3   ? (k == 0 ? 1.0 : -0.5)
         : R == 5 ? (k == 0 ? 1.0 : (k == 1 || k == 4) ? 0.30901699437494742410 : -0.80901699437494742410)
                  : (k == 0              ? 1.0
                     : k == 1 || k == 6  ? 0.62348980185873353053
                     : (k == 2 || k == 5) ? -0.22252093395631440429
                                          : -0.90096886790241912624);
}
__device__ __forceinline__ constexpr double sin_of(int R, int k) {
  const int r = 2 * k > R ? R - k : k;
  const double s = R == 3   ? 0.86602540378443864676
                   : R == 5 ? (r == 1 ? 0.95105651629515357212 : 0.58778525229247312917)
                            : (r == 1   ? 0.78183148246802980871
                               : r == 2 ? 0.97492791218182360702
                                        : 0.43388373911755812048);
  return k == 0 ? 0.0 : (2 * k > R ? -s : s);
}

template <int R, bool INV>
struct Butterfly {  // odd R
  static __device__ __forceinline__ void run(double2 (&x)[R]) {
    constexpr int H = R / 2;
    double2 t[H], s[H], y0 = x[0];
#pragma unroll
    for (int k = 1; k <= H; ++k) {
      t[k - 1] = add(x[k], x[R - k]);
      s[k - 1] = sub(x[k], x[R - k]);
      y0 = add(y0, t[k - 1]);
    }
#pragma unroll
    for (int j = 1; j <= H; ++j) {
      double2 m = x[0], n = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 1; k <= H; ++k) {
        const double c = cos_of(R, (j * k) % R), w = sin_of(R, (j * k) % R);
        m = make_double2(fma(c, t[k - 1].x, m.x), fma(c, t[k - 1].y, m.y));
        n = k == 1 ? make_double2(w * s[0].x, w * s[0].y)
                   : make_double2(fma(w, s[k - 1].x, n.x), fma(w, s[k - 1].y, n.y));
      }
      const double2 r = rot<INV>(n);
      x[j] = add(m, r);
      x[R - j] = sub(m, r);  // x[j], x[R - j] are read only through t and s
    }
    x[0] = y0;
  }
};
template <bool INV>
struct Butterfly<2, INV> {
  static __device__ __forceinline__ void run(double2 (&x)[2]) {
    const double2 a = x[0];
    x[0] = add(a, x[1]);
    x[1] = sub(a, x[1]);
  }
};
template <bool INV>
struct Butterfly<4, INV> {
  static __device__ __forceinline__ void run(double2 (&x)[4]) {
    const double2 a = add(x[0], x[2]), b = sub(x[0], x[2]), c = add(x[1], x[3]), d = rot<INV>(sub(x[1], x[3]));
    x[0] = add(a, c);
    x[1] = add(b, d);
    x[2] = sub(a, c);
    x[3] = sub(b, d);
  }
};
template <bool INV>
struct Butterfly<8, INV> {
  static __device__ __forceinline__ void run(double2 (&x)[8]) {
    constexpr double h = 0.70710678118654752440;
    const double2 a0 = add(x[0], x[4]), a4 = sub(x[0], x[4]), a1 = add(x[1], x[5]), a5 = sub(x[1], x[5]);
    const double2 a2 = add(x[2], x[6]), a6 = rot<INV>(sub(x[2], x[6])), a3 = add(x[3], x[7]), a7 = sub(x[3], x[7]);
    const double2 b0 = add(a0, a2), b2 = sub(a0, a2), b1 = add(a1, a3), b3 = rot<INV>(sub(a1, a3));
    x[0] = add(b0, b1);
    x[4] = sub(b0, b1);
    x[2] = add(b2, b3);
    x[6] = sub(b2, b3);
    // the odd half: a5 and a7 rotated by an eighth turn are h (a5 + rot a5) and h (rot a7 - a7)
    const double2 p = add(a5, rot<INV>(a5)), q = sub(rot<INV>(a7), a7);
    const double2 e = add(a4, a6), f = sub(a4, a6), s = add(p, q), d = rot<INV>(sub(p, q));
    x[1] = make_double2(fma(h, s.x, e.x), fma(h, s.y, e.y));
    x[5] = make_double2(fma(-h, s.x, e.x), fma(-h, s.y, e.y));
    x[3] = make_double2(fma(h, d.x, f.x), fma(h, d.y, f.y));
    x[7] = make_double2(fma(-h, d.x, f.x), fma(-h, d.y, f.y));
  }
};

// One radix pass over L lines of length mp in buf ([mp][L]): sub-transforms of length s.  TW: whether
// the pass has twiddles (the one with s = 1 has none; decided at compile time, since as a run-time
// test the compiler predicates the multiplications and they go through the FP64 pipe all the same:
// 3 of 29 instructions per point of a transform of 256).
template <int R, bool INV, bool TW, int L>
__device__ __forceinline__ void radix_pass(double2* buf, int mp, int s, const double2* __restrict__ tw) {
  const int n = R * s, tstep = 2 * mp / n, total = mp / R * L;
  for (int b = threadIdx.x; b < total; b += kThreads) {
    const int line = b % L, r = b / L, blk = TW ? r / s : r, j = TW ? r - blk * s : 0;
    double2* p = buf + (blk * n + j) * L + line;
    double2 x[R];
#pragma unroll
    for (int q = 0; q < R; ++q) x[q] = p[q * s * L];
    if (INV && TW) {
#pragma unroll
      for (int q = 1; q < R; ++q) x[q] = mul<true>(x[q], __ldg(tw + q * j * tstep));
    }
    Butterfly<R, INV>::run(x);
    if (!INV && TW) {
#pragma unroll
      for (int q = 1; q < R; ++q) x[q] = mul<false>(x[q], __ldg(tw + q * j * tstep));
    }
#pragma unroll
    for (int q = 0; q < R; ++q) p[q * s * L] = x[q];
  }
  __syncthreads();
}

template <bool INV, bool TW, int L>
__device__ __forceinline__ void radix_pass_of(int R, double2* buf, int mp, int s, const double2* __restrict__ tw) {
  switch (R) {
    case 2:
      radix_pass<2, INV, TW, L>(buf, mp, s, tw);
      break;
    case 3:
      radix_pass<3, INV, TW, L>(buf, mp, s, tw);
      break;
    case 4:
      radix_pass<4, INV, TW, L>(buf, mp, s, tw);
      break;
    case 5:
      radix_pass<5, INV, TW, L>(buf, mp, s, tw);
      break;
    case 7:
      radix_pass<7, INV, TW, L>(buf, mp, s, tw);
      break;
    default:
      radix_pass<8, INV, TW, L>(buf, mp, s, tw);
      break;
  }
}

// All passes of the half transforms of one axis, in place (the caller synchronises before).
template <bool INV, int L>
__device__ void transform(double2* buf, const FftAxis& ax) {
  const int last = ax.npass - 1;  // the pass without twiddles: last going forward, first going back
  if (INV && last >= 0) radix_pass_of<INV, false, L>(ax.radix[last], buf, ax.mp, 1, ax.tw);
  for (int i = 0; i < last; ++i) {
    const int p = INV ? last - 1 - i : i;
    radix_pass_of<INV, true, L>(ax.radix[p], buf, ax.mp, ax.sub[p], ax.tw);
  }
  if (!INV && last >= 0) radix_pass_of<INV, false, L>(ax.radix[last], buf, ax.mp, 1, ax.tw);
}

// Storage: buf[n][half][column], 2 C lines.
template <int C>
__device__ __forceinline__ void put_halves(double2* buf, int n, int c, double2 v, const double2* __restrict__ tw) {
  buf[(n * 2) * C + c] = v;
  buf[(n * 2 + 1) * C + c] = mul<false>(v, __ldg(tw + n));
}
template <int C>
__device__ __forceinline__ double2 join_halves(const double2* buf, int n, int c, const double2* __restrict__ tw) {
  const double2 o = mul<true>(buf[(n * 2 + 1) * C + c], __ldg(tw + n));
  return add(buf[(n * 2) * C + c], o);
}

extern __shared__ double2 fft_smem[];

// z forward: real rows 2 i and 2 i + 1 of rho as one complex line, separated into the spectra of
// both (times 2: folded into the kernel's scale).  Column u of a row: frequency 2 u for
// u <= mp / 2, then the odd ones.
template <int C>
__global__ void __launch_bounds__(kThreads) z_forward(const double* __restrict__ rho, double2* __restrict__ a, int64_t rows,
                                                      FftAxis ax, int nzc) {
  double2* buf = fft_smem;
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * (2 * C);
  const int m = ax.m, mp = ax.mp;
  for (int i = threadIdx.x; i < 2 * C * mp; i += kThreads) {  // row by row: coalesced
    const int row = i / mp, n = i - row * mp;
    double v = 0.0;
    if (n < m && r0 + row < rows) v = __ldg(rho + (r0 + row) * m + n);
    double* d = reinterpret_cast<double*>(buf + (n * 2) * C + (row >> 1));
    d[row & 1] = v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < C * mp; i += kThreads) {
    const int n = i / C, c = i % C;
    buf[(n * 2 + 1) * C + c] = mul<false>(buf[(n * 2) * C + c], __ldg(ax.tw + n));
  }
  __syncthreads();
  transform<false, 2 * C>(buf, ax);
  const int ne = mp / 2 + 1;
  for (int i = threadIdx.x; i < C * nzc; i += kThreads) {
    const int c = i / nzc, u = i - c * nzc;
    const int half = u >= ne, k = half ? u - ne : u, kc = half ? mp - 1 - k : (k ? mp - k : 0);
    const double2 p = buf[(__ldg(ax.pos + k) * 2 + half) * C + c], q = buf[(__ldg(ax.pos + kc) * 2 + half) * C + c];
    const int64_t r = r0 + 2 * c;
    if (r < rows) a[r * nzc + u] = make_double2(p.x + q.x, p.y - q.y);
    if (r + 1 < rows) a[(r + 1) * nzc + u] = make_double2(p.y + q.y, q.x - p.x);
  }
}

template <int C>
__global__ void __launch_bounds__(kThreads) z_inverse(const double2* __restrict__ a, double* __restrict__ phi, int64_t rows,
                                                      FftAxis ax, int nzc) {
  double2* buf = fft_smem;
  const int64_t r0 = static_cast<int64_t>(blockIdx.x) * (2 * C);
  const int m = ax.m, mp = ax.mp, ne = mp / 2 + 1;
  for (int i = threadIdx.x; i < C * nzc; i += kThreads) {
    const int c = i / nzc, u = i - c * nzc;
    const int half = u >= ne, k = half ? u - ne : u, kc = half ? mp - 1 - k : (k ? mp - k : 0);
    const int64_t r = r0 + 2 * c;
    double2 p = make_double2(0.0, 0.0), q = p;
    if (r < rows) p = a[r * nzc + u];
    if (r + 1 < rows) q = a[(r + 1) * nzc + u];
    buf[(__ldg(ax.pos + k) * 2 + half) * C + c] = make_double2(p.x - q.y, p.y + q.x);
    if (kc != k) buf[(__ldg(ax.pos + kc) * 2 + half) * C + c] = make_double2(p.x + q.y, q.x - p.y);
  }
  __syncthreads();
  transform<true, 2 * C>(buf, ax);
  for (int i = threadIdx.x; i < C * m; i += kThreads) {
    const int n = i / C, c = i % C;
    buf[(n * 2) * C + c] = join_halves<C>(buf, n, c, ax.tw);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * C * m; i += kThreads) {
    const int row = i / m, n = i - row * m;
    if (r0 + row < rows)
      phi[(r0 + row) * m + n] = reinterpret_cast<const double*>(buf + (n * 2) * C + (row >> 1))[row & 1];
  }
}

// y forward: CTA (i, x) takes C columns of plane x.
template <int C>
__global__ void __launch_bounds__(kThreads) y_forward(const double2* __restrict__ a, double2* __restrict__ b, FftAxis ax,
                                                      int nzc) {
  double2* buf = fft_smem;
  const int m = ax.m, mp = ax.mp, c0 = blockIdx.x * C;
  a += static_cast<int64_t>(blockIdx.y) * m * nzc;
  b += static_cast<int64_t>(blockIdx.y) * 2 * mp * nzc;
  for (int i = threadIdx.x; i < mp * C; i += kThreads) {
    const int n = i / C, c = i % C;
    double2 v = make_double2(0.0, 0.0);
    if (n < m && c0 + c < nzc) v = __ldg(a + static_cast<int64_t>(n) * nzc + c0 + c);
    put_halves<C>(buf, n, c, v, ax.tw);
  }
  __syncthreads();
  transform<false, 2 * C>(buf, ax);
  for (int i = threadIdx.x; i < mp * 2 * C; i += kThreads) {
    const int c = i % C, half = (i / C) & 1, n = i / (2 * C);
    if (c0 + c < nzc) b[(static_cast<int64_t>(half) * mp + n) * nzc + c0 + c] = buf[i];
  }
}

template <int C>
__global__ void __launch_bounds__(kThreads) y_inverse(const double2* __restrict__ b, double2* __restrict__ a, FftAxis ax,
                                                      int nzc) {
  double2* buf = fft_smem;
  const int m = ax.m, mp = ax.mp, c0 = blockIdx.x * C;
  a += static_cast<int64_t>(blockIdx.y) * m * nzc;
  b += static_cast<int64_t>(blockIdx.y) * 2 * mp * nzc;
  for (int i = threadIdx.x; i < mp * 2 * C; i += kThreads) {
    const int c = i % C, half = (i / C) & 1, n = i / (2 * C);
    buf[i] = c0 + c < nzc ? b[(static_cast<int64_t>(half) * mp + n) * nzc + c0 + c] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  transform<true, 2 * C>(buf, ax);
  for (int i = threadIdx.x; i < m * C; i += kThreads) {
    const int n = i / C, c = i % C;
    if (c0 + c < nzc) a[static_cast<int64_t>(n) * nzc + c0 + c] = join_halves<C>(buf, n, c, ax.tw);
  }
}

// x: forward, times the kernel's transform, inverse; in place on C of the ncols columns.
template <int C>
__global__ void __launch_bounds__(kThreads) x_convolve(double2* __restrict__ b, const double* __restrict__ ghat, FftAxis ax,
                                                       int64_t ncols) {
  double2* buf = fft_smem;
  const int m = ax.m, mp = ax.mp;
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * C;
  for (int i = threadIdx.x; i < mp * C; i += kThreads) {
    const int n = i / C, c = i % C;
    double2 v = make_double2(0.0, 0.0);
    if (n < m && c0 + c < ncols) v = b[n * ncols + c0 + c];
    put_halves<C>(buf, n, c, v, ax.tw);
  }
  __syncthreads();
  transform<false, 2 * C>(buf, ax);
  for (int i = threadIdx.x; i < mp * 2 * C; i += kThreads) {
    const int c = i % C, half = (i / C) & 1, n = i / (2 * C);
    const double g = c0 + c < ncols ? __ldg(ghat + (static_cast<int64_t>(half) * mp + n) * ncols + c0 + c) : 0.0;
    const double2 v = buf[i];
    buf[i] = make_double2(v.x * g, v.y * g);
  }
  __syncthreads();
  transform<true, 2 * C>(buf, ax);
  for (int i = threadIdx.x; i < m * C; i += kThreads) {
    const int n = i / C, c = i % C;
    if (c0 + c < ncols) b[n * ncols + c0 + c] = join_halves<C>(buf, n, c, ax.tw);
  }
}

// ghat in the storage order of the spectra, from the transform in natural order.
__global__ void store_kernel(const double2* __restrict__ hat, double* __restrict__ ghat, FftAxis x, FftAxis y, FftAxis z,
                             int nzc, double scale) {
  const int64_t total = 4LL * x.mp * y.mp * nzc;
  for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {  // e: frequencies (kx, ky, column u)
    const int u = static_cast<int>(e % nzc);
    const int64_t r = e / nzc;
    const int ky = static_cast<int>(r % (2 * y.mp)), kx = static_cast<int>(r / (2 * y.mp));
    const int ne = z.mp / 2 + 1, kz = u < ne ? 2 * u : 2 * (u - ne) + 1;
    const int64_t px = static_cast<int64_t>(kx & 1) * x.mp + x.pos[kx >> 1];
    const int64_t py = static_cast<int64_t>(ky & 1) * y.mp + y.pos[ky >> 1];
    ghat[(px * (2 * y.mp) + py) * nzc + u] = hat[(static_cast<int64_t>(kx) * (2 * y.mp) + ky) * (z.mp + 1) + kz].x * scale;
  }
}

// FP64 instructions per point of the half transforms of length n, first pass first; appends the
// radices.  Radix 8 while it divides, then the rest.
double pass_cost(int n, std::vector<int>* radices) {
  static const int kR[] = {8, 7, 5, 4, 3, 2};
  static const double kCost[] = {6.5, 9.5, 7.2, 4.0, 4.0, 2.0};
  double cost = 0.0;
  radices->clear();
  for (int i = 0; i < 6; ++i)
    while (n % kR[i] == 0) {
      n /= kR[i];
      cost += kCost[i] + (n > 1 ? 4.0 * (kR[i] - 1) / kR[i] : 0.0);
      radices->push_back(kR[i]);
    }
  return n == 1 ? cost : -1.0;
}

bool plan_axis(FftAxis* ax, int m) {
  std::vector<int> best, r;
  double best_cost = 0.0;
  int best_n = 0;
  const int top = m < 8 ? 8 : m + m / 3;
  for (int n = m; n <= top && n <= kFftMaxLen; ++n) {
    const double c = pass_cost(n, &r);
    if (c < 0.0 || static_cast<int>(r.size()) > kFftMaxPasses) continue;
    const double t = n * (c + 6.0);  // and what every point costs beside the passes
    if (!best_n || t < best_cost) best_n = n, best_cost = t, best = r;
  }
  if (!best_n) return false;
  ax->m = m;
  ax->mp = best_n;
  ax->npass = static_cast<int>(best.size());
  int s = best_n;
  for (int p = 0; p < ax->npass; ++p) {
    ax->radix[p] = best[p];
    s /= best[p];
    ax->sub[p] = s;
  }
  ax->tw = nullptr;
  ax->pos = nullptr;
  return true;
}

// Columns per block: 64 KB of shared memory at most where that leaves one (three blocks per SM), fewer where
// `sets` sets of n columns would leave SMs without a block.
// Measured: a solve of 1 x 1 x 300 91 -> 52 us, 73 with the library's transforms.
int columns_of(int mp, int64_t n, int64_t sets, int num_sms) {
  int c = mp <= 256 ? 8 : mp <= 512 ? 4 : mp <= 1024 ? 2 : 1;
  while (c > 1 && (n + c - 1) / c * sets < num_sms) c /= 2;
  return c;
}

template <class K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  return bytes > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes))
                           : cudaSuccess;
}

template <int C>
cudaError_t run_z(const FftConv* c, const double* rho, double* phi, bool forward, cudaStream_t s) {
  const size_t bytes = sizeof(double2) * 2 * C * c->z.mp;
  const int64_t rows = static_cast<int64_t>(c->x.m) * c->y.m, blocks = (rows + 2 * C - 1) / (2 * C);
  cudaError_t e = forward ? allow_smem(z_forward<C>, bytes) : allow_smem(z_inverse<C>, bytes);
  if (e != cudaSuccess) return e;
  if (forward)
    z_forward<C><<<static_cast<unsigned>(blocks), kThreads, bytes, s>>>(rho, c->a, rows, c->z, c->nzc);
  else
    z_inverse<C><<<static_cast<unsigned>(blocks), kThreads, bytes, s>>>(c->a, phi, rows, c->z, c->nzc);
  return cudaGetLastError();
}
template <int C>
cudaError_t run_y(const FftConv* c, bool forward, cudaStream_t s) {
  const size_t bytes = sizeof(double2) * 2 * C * c->y.mp;
  const dim3 grid((c->nzc + C - 1) / C, c->x.m);
  cudaError_t e = forward ? allow_smem(y_forward<C>, bytes) : allow_smem(y_inverse<C>, bytes);
  if (e != cudaSuccess) return e;
  if (forward)
    y_forward<C><<<grid, kThreads, bytes, s>>>(c->a, c->b, c->y, c->nzc);
  else
    y_inverse<C><<<grid, kThreads, bytes, s>>>(c->b, c->a, c->y, c->nzc);
  return cudaGetLastError();
}
template <int C>
cudaError_t run_x(const FftConv* c, cudaStream_t s) {
  const size_t bytes = sizeof(double2) * 2 * C * c->x.mp;
  const int64_t ncols = 2LL * c->y.mp * c->nzc;
  cudaError_t e = allow_smem(x_convolve<C>, bytes);
  if (e != cudaSuccess) return e;
  x_convolve<C><<<static_cast<unsigned>((ncols + C - 1) / C), kThreads, bytes, s>>>(c->b, c->ghat, c->x, ncols);
  return cudaGetLastError();
}

#define MUSR_BY_COLUMNS(columns, f, ...)  \
  [&] {                                   \
    switch (columns) {                    \
      case 8:                             \
        return f<8>(__VA_ARGS__);         \
      case 4:                             \
        return f<4>(__VA_ARGS__);         \
      case 2:                             \
        return f<2>(__VA_ARGS__);         \
      default:                            \
        return f<1>(__VA_ARGS__);         \
    }                                     \
  }()

}  // namespace

// tw[k] = exp(-i pi k / mp), k < 2 mp, each rounded from long double.  One eighth of the circle is evaluated (a
// quarter for odd mp) and the rest is its images: long double is software on Arm, 0.3 us a value, and the whole
// circle made creating a solver with an axis of 4096 points 4.8 ms longer.
static void fill_twiddles(double2* tw, int mp) {
  const long double pi = 3.14159265358979323846264338327950288L;
  std::vector<double2> arc(mp / 2 + 1);  // (cos, sin) of pi j / (2 mp)
  for (int j = 0; j <= mp / 2; j += mp % 2 ? 1 : 2) {
    const long double a = pi * j / (2 * mp);
    arc[j] = make_double2(static_cast<double>(cosl(a)), static_cast<double>(sinl(a)));
  }
  for (int k = 0; k < 2 * mp; ++k) {
    const int j = k <= mp ? k : 2 * mp - k;     // sine of the other sign beyond mp
    const int q = 2 * (2 * j <= mp ? j : mp - j);  // cosine of the other sign beyond mp / 2; at most mp
    const double2 e = 2 * q <= mp ? arc[q] : make_double2(arc[mp - q].y, arc[mp - q].x);
    tw[k] = make_double2(2 * j <= mp ? e.x : -e.x, k <= mp ? -e.y : e.y);
  }
}

bool fftconv_plan(FftConv* c, int mx, int my, int mz, int num_sms) {
  c->num_sms = num_sms;
  // grid limits: the y kernels' planes are a grid's second dimension
  if (mx > 65535 || !plan_axis(&c->x, mx) || !plan_axis(&c->y, my) || !plan_axis(&c->z, mz)) return false;
  c->nzc = c->z.mp + 1;
  // A block holds a line of a long axis by itself and takes 26 (y, z) or 55 (x) FP64 instructions per point of
  // it, 60 us at 2048 points and 250 us at 4096 over a solve's kernels, however few the lines; the library splits
  // a line.  Measured, one solve with its wait, ours and the library's: 2048 x 4 x 4 159 / 136 us, 2048 x 8 x 8
  // 215 / 250, 4096 x 2 x 2 267 / 107, 4096 x 4 x 4 283 / 203, 4096 x 8 x 8 395 / 470, 1500 x 1 x 1 116 / 155.
  const int longest = c->x.mp > c->y.mp ? (c->x.mp > c->z.mp ? c->x.mp : c->z.mp) : (c->y.mp > c->z.mp ? c->y.mp : c->z.mp);
  const int64_t lines = static_cast<int64_t>(c->x.mp) * c->y.mp * c->z.mp / longest;
  if (longest > 1536 && lines < 32) return false;
  return 8.0 * c->x.mp * c->y.mp * c->z.mp < 4294967296.0;
}

cudaError_t fftconv_tables(FftConv* c) {
  FftAxis* axes[3] = {&c->x, &c->y, &c->z};
  size_t bytes = 0;
  for (FftAxis* ax : axes) bytes += sizeof(double2) * 2 * ax->mp + sizeof(double2) * ((sizeof(int) * ax->mp + 15) / 16);
  std::vector<char> host(bytes, 0);
  cudaError_t e = cudaMalloc(&c->tables, bytes);
  if (e != cudaSuccess) return e;
  size_t off = 0;
  for (FftAxis* ax : axes) {
    double2* tw = reinterpret_cast<double2*>(host.data() + off);
    fill_twiddles(tw, ax->mp);
    ax->tw = reinterpret_cast<const double2*>(static_cast<char*>(c->tables) + off);
    off += sizeof(double2) * 2 * ax->mp;
    int* pos = reinterpret_cast<int*>(host.data() + off);
    for (int p = 0; p < ax->mp; ++p) {  // digits of position p, most significant first, are k's, least first
      int rest = p, k = 0, w = 1;
      for (int i = 0; i < ax->npass; ++i) {
        k += rest / ax->sub[i] * w;
        rest %= ax->sub[i];
        w *= ax->radix[i];
      }
      pos[k] = p;
    }
    ax->pos = reinterpret_cast<const int*>(static_cast<char*>(c->tables) + off);
    off += sizeof(double2) * ((sizeof(int) * ax->mp + 15) / 16);
  }
  return cudaMemcpy(c->tables, host.data(), bytes, cudaMemcpyHostToDevice);
}

cudaError_t fftconv_buffers(FftConv* c) {
  const size_t line = static_cast<size_t>(c->x.m) * c->nzc;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&c->a), sizeof(double2) * line * c->y.m);
  if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&c->b), sizeof(double2) * line * 2 * c->y.mp);
  return e;
}

void fftconv_free(FftConv* c) {
  cudaFree(c->a);
  cudaFree(c->b);
  cudaFree(c->ghat);
  cudaFree(c->tables);
  c->a = c->b = nullptr;
  c->ghat = nullptr;
  c->tables = nullptr;
}

cudaError_t fftconv_set_kernel(FftConv* c, const double2* hat, double scale, cudaStream_t s) {
  const int64_t total = 4LL * c->x.mp * c->y.mp * c->nzc;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&c->ghat), sizeof(double) * total);
  if (e != cudaSuccess) return e;
  const int64_t blocks = (total + 255) / 256;
  // the inverse transforms' normalisation, and the 2 of the separated pairs
  const double norm = 2.0 * (2.0 * c->x.mp) * (2.0 * c->y.mp) * (2.0 * c->z.mp);
  store_kernel<<<static_cast<unsigned>(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(hat, c->ghat, c->x, c->y, c->z, c->nzc,
                                                                                   scale / norm);
  return cudaGetLastError();
}

cudaError_t fftconv_solve(const FftConv* c, const double* rho, double* phi, cudaStream_t s) {
  const int64_t rows = static_cast<int64_t>(c->x.m) * c->y.m;
  const int cz = columns_of(c->z.mp, (rows + 1) / 2, 1, c->num_sms), cy = columns_of(c->y.mp, c->nzc, c->x.m, c->num_sms);
  const int cx = columns_of(c->x.mp, 2LL * c->y.mp * c->nzc, 1, c->num_sms);
  cudaError_t e = MUSR_BY_COLUMNS(cz, run_z, c, rho, phi, true, s);
  if (e == cudaSuccess) e = MUSR_BY_COLUMNS(cy, run_y, c, true, s);
  if (e == cudaSuccess) e = MUSR_BY_COLUMNS(cx, run_x, c, s);
  if (e == cudaSuccess) e = MUSR_BY_COLUMNS(cy, run_y, c, false, s);
  if (e == cudaSuccess) e = MUSR_BY_COLUMNS(cz, run_z, c, rho, phi, false, s);
  return e;
}

}  // namespace musr
