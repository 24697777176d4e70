// musr_kernels_f64.cuh -- the FP64 path of theories with a basis form (sm_103a).
//
// What binds it: the FP64 pipe.  An SM issues one FP64 warp instruction per 16 clocks (2 lanes
// per clock), 64 issue slots of everything else beside it, so the kernel's time is its number
// of FP64 instructions (ncu on the term-list kernel it replaces: pipe 80-86 % of its peak busy,
// issue slots 9 %).  The term-list kernel (fp64_item) spends 130 of them per (histogram, bin) on
// the cost of a one-term theory and 400 on the cost and gradient of a two-term one, most in
// exp, sincospi, log and the divisions of CUDA's library, evaluated per histogram and bin.  Here
//   * the model is the linear combination of time-only basis functions that the SPLIT path
//     uses (musr_dev.h), in FP64: a chunk of up to 8 histograms that share t0 and every
//     time-dependent parameter evaluates the time factors once per bin, and a (histogram, bin)
//     pair costs M multiply-adds for N, the cost term and 2 M + 1 for the gradient;
//   * a thread's bins are 256 apart: each factor exp(-L t - S t^2 / 2) cos(2 pi nu t) is evaluated
//     at one bin in kRebase, its phase reduced in double-double arithmetic, and taken from there
//     to the others by one complex multiplication with the chunk's table of the factor over i
//     steps (i < kRebase; a Gaussian's cross term exp(-S t i D) by one more, a running product);
//   * 1/N and 1/max(d,1) are an approximate reciprocal and one third-order Newton step, the
//     logarithm of d/N a table of 1024 intervals and a fourth-degree series;
//   * comparisons, selections and the widening of FP32 counts run on the integer pipe.
// What is left per pair (M = 3, -2lnL with gradient): N 3, residual 1, 1/N 3, u 1, d/N 1,
// logarithm 6, cost 2, G and W 4, V 3 = 24 instructions, and an eighth of the per-bin work.
//
// Measured (GB300, 8 x 65536 bins, -2lnL, two cosine terms): see eval64_kernel below.
#pragma once

#include "musr_kernels.cuh"

namespace musr {
namespace kern {
namespace {

constexpr int kRebase = 32;      // bins of a thread between two fresh evaluations of the time factors
constexpr int kLogTable = 1024;  // intervals of the logarithm's table
constexpr int kRatioHi = 0x3eb00000;  // high word of 2^-20

// One chunk's constants for the FP64 basis kernels.
struct Chunk64 {
  double gam[kGroupMax][kGamStride];   // [Nbkg, Gam_0 .. Gam_{M-1}] of each histogram
  double gdot[kGroupMax][kGamStride];  // their directional derivatives (Gauss-Newton products)
  int kinds[kMaxTerms];
  int dkt_src[kMaxTerms];
  double bamp[kMaxTerms];              // amplitude carried by the basis (merged shapes), else 1
  double lam[kMaxTerms], S[kMaxTerms]; // exponent: lam t + S t^2 / 2 (lam includes 1 / tau)
  double kt[kMaxTerms];                // Kubo-Toyabe width Delta, or the Lorentzian's rate a
  double st_hi[kMaxTerms], st_lo[kMaxTerms];  // phase step per bin nu dt (turns) as a double-double
  double dlam[kMaxTerms], dsig[kMaxTerms], dnu[kMaxTerms], ddel[kMaxTerms];  // along a direction
  double rate;      // decay envelope: 1 / tau (or 0)
  // over i steps of 256 bins from time zero: each term's factor (cosine and sine part), its
  // Kubo-Toyabe exponential, the envelope
  double2 q[kMaxTerms][kRebase];
  double qk[kMaxTerms][kRebase], qe[kRebase];
  double td[kRebase];  // i steps of 256 bins as a time
  int safe;         // the products neither overflow nor start from an underflowed value
};

struct Smem64 {
  // idle staging space of chunk_finalize ([columns][segments] doubles, at most kBlock of them)
  alignas(16) float stage[1][1][2 * kBlock];
  Job job;
  double x[kHeadParams];
  HistSet hs;
  const HistSet* hs_src;
  ChunkCache cc;
  TileState ts;
  Finish fin;
  Chunk64 c;
  double red[kWarps][64];
  double tot[kMaxChan + 1];
  double2 logtab[kLogTable];  // (c, -ln c) per interval
  int flag;
};

// ---------------------------------------------------------------------------------------------
// Arithmetic
// ---------------------------------------------------------------------------------------------

// Whether x > 0 and x > 1 (x not a NaN): doubles order like their bits for positive values.
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool above_one(double x) { return __double_as_longlong(x) > 0x3ff0000000000000LL; }

// 1/x from PTX's approximate reciprocal y (relative error e0 about 2^-20) by the third-order
// Newton (Householder) step y + y (e + e^2), e = 1 - x y: the error left is e0^3, below the
// rounding of the last operation.  x neither 0 nor subnormal (rcp's result would be infinite) nor
// above 2^1022 (it would be flushed to 0): recip_range(x).
__device__ __forceinline__ bool recip_range(double x) {  // x in [2^-1022, 2^1022)
  return static_cast<unsigned>(__double2hiint(x) - 0x00100000) < 0x7fc00000u;
}
__device__ __forceinline__ double recip(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = __fma_rn(-x, y, 1.0);
  e = __fma_rn(e, e, e);
  return __fma_rn(y, e, y);
}
// The division of values outside that range.  A call: inlined, its instructions are predicated into the
// loop over bins, and one that is predicated off takes the FP64 pipe all the same.
__device__ __noinline__ double divide(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ double recip_any(double x) { return recip_range(x) ? recip(x) : divide(1.0, x); }
// 1 / max(d, 1); only FP64 stores (f32 false) can hold counts above recip's range.
__device__ __forceinline__ double count_weight(double d, bool f32) {
  if (!f32 && __double2hiint(d) >= 0x7fd00000) return divide(1.0, d);
  return above_one(d) ? recip(d) : 1.0;
}

// d / N^2: 0 where N^2 overflows (N from 2^512), as the quotient itself.
__device__ __forceinline__ double likelihood_weight(double d, double N) {
  const double y = recip_any(N);
  return static_cast<unsigned>(__double2hiint(N) - 0x5ff00000) < 0x20000000u ? 0.0 : d * y * y;
}

// ln x by table and series (Tang's method, ACM TOMS 16 (1990) 378): x = 2^k m with m in
// [0.70, 1.41); c of m's interval (1/1024 of an octave's mantissa range) approximates 1/m, so
// that ln x = k ln 2 - ln c + ln(1 + r), r = m c - 1, |r| < h = 2^-11, the last by its series to r^4 with
// r^5 / 5 folded into the cubic term as (3/20) h^2 r^3: what is left is below 2^-59 on [-h, h] and odd, so
// that it does not add up over a sum of bins.  One interval holds 1 (h/2 below it, h above) with c = 1, so
// that ln is exactly 0 there and the absolute error near it stays at 2^-53 |ln x| + 2^-57 (elsewhere three
// roundings: 2.2 x 2^-53 |ln x| at most).  Over 65536 Poisson bins of 1e5 / 1e6 / 1e7 counts a -2lnL's relative
// error is 2.3e-14 / 4.7e-13 / 2.9e-12 (a model of these operations on the host), that of log(d / N) itself; with
// an interval from 1 to 2^-10 above it and c = 1, where r leaves [-h, h], and the plain series it was 4.5e-13 /
// 1.1e-11 / 4.3e-11.  Arguments outside [2^-1000, 2^1000] (or not positive numbers) take CUDA's log.
constexpr int kLogOff = 0x3fe6a200;  // high word of the table's lower end
__device__ __forceinline__ double ln_tab(double x, const double2* tab) {
  const int hi = __double2hiint(x);
  if (static_cast<unsigned>(hi - 0x01700000) > 0x7d000000u) return log(x);
  const int tmp = hi - kLogOff, k = tmp >> 20;
  const double2 t = tab[(tmp >> 10) & (kLogTable - 1)];
  const double m = __hiloint2double(hi - (k << 20), __double2loint(x));
  const double r = __fma_rn(m, t.x, -1.0);
  double q = __fma_rn(r, -0.25, 1.0 / 3.0 + 3.0 / 20.0 / 4194304.0);
  q = __fma_rn(r, q, -0.5);
  double l = __dadd_rn(__fma_rn(__dmul_rn(r, r), q, r), t.y);
  if (k != 0) l = __fma_rn(static_cast<double>(k), 0.69314718055994530942, l);
  return l;
}

// The table, computed when the library is compiled (a logarithm per thread at every launch would
// cost it 2 us): c = 1 / (midpoint of the interval) in 24 bits or fewer (1 for the interval that
// holds 1), and -ln c of that c by the series of atanh,
// ln c = 2 (z + z^3/3 + ...), z = (c - 1)/(c + 1), |z| < 0.18, summed from its smallest term.
struct LogTable {
  double2 t[kLogTable];
};
constexpr double neg_ln(double c) {
  const double z = (c - 1.0) / (c + 1.0), z2 = z * z;
  double s = 0.0;
  for (int k = 25; k >= 3; k -= 2) s = (s + 1.0 / k) * z2;
  return -2.0 * (z + z * s);
}
constexpr LogTable make_log_table() {
  LogTable r{};
  for (int i = 0; i < kLogTable; ++i) {
    // high words from kLogOff in steps of 0x400: mantissa 1 + w / 2^20, below 1 at half the scale
    const int lo = kLogOff + (i << 10), up = lo + 0x400;
    auto value = [](int hi) {
      const double m = 1.0 + (hi & 0xfffff) / 1048576.0;
      return (hi >> 20) == 0x3ff ? m : 0.5 * m;
    };
    const double mid = 0.5 * (value(lo) + value(up));
    const bool one = lo <= 0x3ff00000 && 0x3ff00000 < up;
    const double c = one ? 1.0 : static_cast<double>(static_cast<float>(1.0 / mid));
    r.t[i].x = c;
    r.t[i].y = one ? 0.0 : neg_ln(c);
  }
  return r;
}
__device__ const LogTable log_table = make_log_table();

// ---------------------------------------------------------------------------------------------
// Chunk set-up
// ---------------------------------------------------------------------------------------------

// Directional derivatives of a histogram's coefficients (see coef_row) along a Gauss-Newton
// direction with local components dir(slot).
template <int SHAPE, class Slot, class Dir>
__device__ void dcoef_row64(const HistSet& hs, Slot slot, Dir dir, const double* cph, const double* sph, double* gd) {
  using Bs = Basis<SHAPE>;
  constexpr double kDeg = kTwoPi / 360.0;
  const double N0 = slot(0), vN0 = dir(0);
  gd[0] = dir(1);
  gd[1] = hs.envelope ? vN0 : 0.0;
  if (Bs::MERGED) {
    const double vph = dir(hs.canon[0].phi_slot) * kDeg;
    gd[2] = vN0 * cph[0] - N0 * sph[0] * vph;
    gd[3] = -vN0 * sph[0] - N0 * cph[0] * vph;
  } else {
#pragma unroll
    for (int k = 0; k < Bs::NT; ++k) {
      if (k >= hs.nterms) break;
      const CanonTerm& ct = hs.canon[k];
      const double a = ct.amp_slot >= 0 ? slot(ct.amp_slot) : 1.0, va = ct.amp_slot >= 0 ? dir(ct.amp_slot) : 0.0;
      const double dNa = vN0 * a + N0 * va;
      if (ct.kind == kTermTF) {
        const double vph = dir(ct.phi_slot) * kDeg;
        gd[1 + Bs::bc(k)] = dNa * cph[k] - N0 * a * sph[k] * vph;
        gd[1 + Bs::bs(k)] = -dNa * sph[k] - N0 * a * cph[k] * vph;
      } else {
        gd[1 + Bs::bc(k)] = dNa;
      }
    }
  }
}

// After load_chunk (header, slot values, row pointers): the FP64 coefficients and constants.
template <int SHAPE, class SM>
__device__ void load_chunk64(const Job& job, const HistSet& hs, SM& sm) {
  using Bs = Basis<SHAPE>;
  ChunkCache& cc = sm.cc;
  Chunk64& c = sm.c;
  const int tid = threadIdx.x, nh = cc.nh;
  const double D = kBlock * hs.dt_us;  // length of one step of a thread
  static_assert(kGroupMax * kMaxTerms == 32, "one lane per (histogram, term)");
  if (tid < 32) {  // cosine and sine of every phase
    const int hl = tid / kMaxTerms, k = tid - hl * kMaxTerms;
    double cp = 1.0, sp = 0.0;
    if (hl < nh && k < hs.nterms && hs.canon[k].kind == kTermTF) {
      const double x = cc.loc[hl][hs.canon[k].phi_slot] * (1.0 / 360.0);
      sincospi(2.0 * (x - rint(x)), &sp, &cp);
    }
    cc.cph[hl][k] = cp;
    cc.sph[hl][k] = sp;
  } else if (tid < 32 + kMaxTerms) {
    const int k = tid - 32;
    int kind = kTermNone, src = -1;
    double lam = hs.envelope ? 1.0 / kTauMuUs : 0.0, S = 0.0, kt = 0.0, nu = 0.0, bamp = 1.0;
    double dl = 0.0, ds = 0.0, dn = 0.0, dd = 0.0;
    if (k < hs.nterms) {
      const CanonTerm& ct = hs.canon[k];
      kind = ct.kind;
      for (int i = 0; i < ct.nexp; ++i) {
        lam += cc.loc[0][ct.exp_slot[i]];
        dl += cc.ldir[0][ct.exp_slot[i]];
      }
      for (int i = 0; i < ct.ngauss; ++i) {
        const double g = cc.loc[0][ct.gauss_slot[i]];
        S = fma(g, g, S);
        ds = fma(g, cc.ldir[0][ct.gauss_slot[i]], ds);
      }
      // finite rates whose sum or square overflows: the largest double, so that 0 times it (time zero) is 0
      constexpr double kBig = 1.7976931348623157e308;
      bool finite = true;
      for (int i = 0; i < ct.nexp; ++i) finite = finite && isfinite(cc.loc[0][ct.exp_slot[i]]);
      for (int i = 0; i < ct.ngauss; ++i) finite = finite && isfinite(cc.loc[0][ct.gauss_slot[i]]);
      if (finite && !isfinite(lam)) lam = lam > 0.0 ? kBig : -kBig;
      if (finite && !isfinite(S)) S = kBig;
      if (Bs::MERGED && ct.amp_slot >= 0) bamp = cc.loc[0][ct.amp_slot];
      if (kind == kTermKT || kind == kTermLKT || kind == kTermDKT) {
        kt = cc.loc[0][ct.kt_slot];
        dd = cc.ldir[0][ct.kt_slot] * (kind == kTermKT ? 2.0 / 3.0 * kt : (kind == kTermLKT ? 2.0 / 3.0 : 1.0));
      }
      if (kind == kTermTF) nu = cc.loc[0][ct.nu_slot];
      if (kind == kTermTF || kind == kTermDKT) dn = cc.ldir[0][ct.nu_slot];
      if (kind == kTermDKT) {
        src = hs.dkt_of[(static_cast<int64_t>(cc.row[0]) * kMaxTerms + ct.dkt_term) * kMaxPrims + ct.dkt_prim];
        if (!dbg_ok(job.dbg, src >= 0 && src < hs.ndkt, kDbgDkt)) src = -1;
      }
    }
    c.kinds[k] = kind;
    c.dkt_src[k] = src;
    c.bamp[k] = bamp;
    c.lam[k] = lam;
    c.S[k] = S;
    c.kt[k] = kt;
    c.dlam[k] = dl;
    c.dsig[k] = ds;
    c.dnu[k] = dn;
    c.ddel[k] = dd;
    c.st_hi[k] = nu * hs.dt_us;
    c.st_lo[k] = fma(nu, hs.dt_us, -c.st_hi[k]);
  } else if (tid == 64) {
    c.rate = hs.envelope ? 1.0 / kTauMuUs : 0.0;
  }
  __syncthreads();
  // The tables: a warp per term, a lane per number of steps (the envelope's by another warp),
  // beside the coefficients of the histograms.
  static_assert(kRebase == 32 && kWarps > kMaxTerms + 1, "one lane per table entry");
  const int wp = tid >> 5, i = tid & 31;
  const bool many = hs.tile_bins > kBlock;  // an item of one iteration needs no table
  if (many && wp >= 2 && wp < 2 + kMaxTerms) {
    const int k = wp - 2;
    if (k < hs.nterms && k < Bs::NT) {
      const double ti = i * D, z = c.kt[k] * ti;
      const double X = exp(-(fma(0.5 * c.S[k], ti, c.lam[k]) * ti));
      double s = 0.0, co = 1.0;
      if (c.kinds[k] == kTermTF) {
        const double ni = i * kBlock, p = c.st_hi[k] * ni;
        sincospi(2.0 * ((p - rint(p)) + fma(c.st_lo[k], ni, fma(c.st_hi[k], ni, -p))), &s, &co);
      }
      c.q[k][i] = make_double2(X * co, X * s);
      if (c.kinds[k] == kTermKT || c.kinds[k] == kTermLKT)
        c.qk[k][i] = exp(c.kinds[k] == kTermKT ? -(0.5 * z * z) : -z);
    }
  } else if (many && wp == 2 + kMaxTerms) {
    c.qe[i] = exp(-c.rate * (i * D));
    c.td[i] = i * D;
  }
  if (tid < nh) {
    double g[kGamStride], gd[kGamStride];
#pragma unroll
    for (int i = 0; i < kGamStride; ++i) g[i] = gd[i] = 0.0;
    const double N0 = cc.loc[tid][0];
    g[0] = cc.loc[tid][1];
    g[1] = hs.envelope ? N0 : 0.0;
    if (Bs::MERGED) {
      g[2] = N0 * cc.cph[tid][0];
      g[3] = -N0 * cc.sph[tid][0];
    } else {
#pragma unroll
      for (int k = 0; k < Bs::NT; ++k) {
        if (k >= hs.nterms) break;
        const CanonTerm& ct = hs.canon[k];
        const double a = ct.amp_slot >= 0 ? cc.loc[tid][ct.amp_slot] : 1.0;
        if (ct.kind == kTermTF) {
          g[1 + Bs::bc(k)] = N0 * a * cc.cph[tid][k];
          g[1 + Bs::bs(k)] = -N0 * a * cc.sph[tid][k];
        } else {
          g[1 + Bs::bc(k)] = N0 * a;
        }
      }
    }
    if (job.dir)
      dcoef_row64<SHAPE>(hs, [&](int q) { return cc.loc[tid][q]; }, [&](int q) { return cc.ldir[tid][q]; },
                         cc.cph[tid], cc.sph[tid], gd);
#pragma unroll
    for (int i = 0; i < kGamStride; ++i) {
      c.gam[tid][i] = g[i];
      c.gdot[tid][i] = gd[i];
    }
  } else if (tid == 32) {
    // The products hold where no factor of them overflows and nothing grows from an underflowed value: every
    // exponent within +-600 over the fit's times and the steps from a fresh bin (up to len further), or terms
    // that decay after time zero and whose fresh value and cross term exp(-S t i D) before it stay within
    // that.  (Otherwise, and for NaN parameters, every bin is evaluated afresh.)
    const double t1 = (cc.nlo - 4 - cc.t0) * hs.dt_us, t2 = (cc.nhi - cc.t0) * hs.dt_us;
    const double len = fmin(kRebase * D, t2 - t1 + D);
    const double T = fmax(fabs(t1), fabs(t2)) + D + len, T0 = fmax(-t1, 0.0);  // T0: the stretch before time zero
    int ok = T0 * c.rate <= 600.0;
    for (int k = 0; k < hs.nterms && k < kMaxTerms; ++k) {
      const double kt = c.kt[k], S = c.S[k] + (c.kinds[k] == kTermKT ? kt * kt : 0.0);
      const double lam = fabs(c.lam[k]) + (c.kinds[k] == kTermLKT ? fabs(kt) : 0.0);
      const bool small = lam * T + S * T * T <= 600.0;
      const bool decays = c.lam[k] >= 0.0 && (c.kinds[k] != kTermLKT || kt >= 0.0) && lam < 1e150 && S < 1e150 &&
                          lam * T0 + S * T0 * (T0 + len) <= 600.0;
      if (!(small || decays)) ok = 0;
    }
    c.safe = ok;
  }
  __syncthreads();
}

// A thread's time factors, its bins kBlock apart.  at() gives the pieces of the bin at time t (nd bins
// from time zero), `step` steps after the last bin evaluated afresh (0: evaluates this one; the steps
// are taken in order, and many says whether any follow): the envelope E, per term P with its cosine
// and sine parts, and a Kubo-Toyabe term's derivative factors dK (along Delta) and, in Ps, dynamic
// Kubo-Toyabe's along nu.
template <int SHAPE>
struct TimeFactors {
  using Bs = Basis<SHAPE>;
  static constexpr int NT = Bs::NT;
  // Per term at the last fresh bin: the factor a exp(-L t - S t^2/2) with its cosine and sine
  // parts (fc, fs), a Gaussian's cross ratio of one step 1 + w (already in fc, fs for the steps made),
  // and the same of a Kubo-Toyabe term's own exponential (fk, wk); the envelope (fE).  The ratio is
  // kept as its difference from 1: rounded to a double it would add its own error at every step, with
  // one sign along a thread (root mean square of a factor over 32768 bins, sigma 0.05: 6.2e-16 against
  // 1.5e-16; at sigma 0.3 7.1e-16 against 4.0e-16, 4.5e-16 for the factor evaluated in every bin).
  double fE, fc[NT], fs[NT], w[NT], fk[NT], wk[NT];

  __device__ __forceinline__ TimeFactors() {
    fE = 0.0;
#pragma unroll
    for (int k = 0; k < NT; ++k) fc[k] = fs[k] = fk[k] = w[k] = wk[k] = 0.0;
  }

  __device__ __forceinline__ void at(const Job& job, const HistSet& hs, const Chunk64& c, int step, bool many, double nd,
                                     double t, double* E, double (&Pc)[NT], double (&Ps)[NT], double (&dK)[NT]) {
    const int nterms = Bs::NTF < 0 ? min(hs.nterms, NT) : NT;
    if (step == 0) {
      fE = exp(-__dmul_rn(c.rate, t));
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        if (k >= nterms) continue;
        const double S = c.S[k];
        fc[k] = __dmul_rn(c.bamp[k], exp(-__dmul_rn(__fma_rn(__dmul_rn(0.5, S), t, c.lam[k]), t)));
        if (S != 0.0 && many) w[k] = expm1(-__dmul_rn(__dmul_rn(S, t), kBlock * hs.dt_us));
        if (Bs::tf(c.kinds, k)) {
          const double p = __dmul_rn(c.st_hi[k], nd);  // phase in turns, as a double-double
          const double pl = __fma_rn(c.st_lo[k], nd, __fma_rn(c.st_hi[k], nd, -p));
          double s, co;
          sincospi(__dmul_rn(2.0, __dadd_rn(__dadd_rn(p, -rint(p)), pl)), &s, &co);
          fs[k] = __dmul_rn(fc[k], s);
          fc[k] = __dmul_rn(fc[k], co);
        } else if (c.kinds[k] == kTermKT) {
          const double z = __dmul_rn(c.kt[k], t);
          fk[k] = exp(-__dmul_rn(__dmul_rn(0.5, z), z));
          if (many) wk[k] = expm1(-__dmul_rn(__dmul_rn(__dmul_rn(c.kt[k], c.kt[k]), t), kBlock * hs.dt_us));
        } else if (c.kinds[k] == kTermLKT) {
          fk[k] = exp(-__dmul_rn(c.kt[k], t));
        }
      }
    }
    *E = fE;
    double xc[NT], xs[NT], kg[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) xc[k] = fc[k], xs[k] = fs[k], kg[k] = fk[k];
    if (step != 0) {
      *E = __dmul_rn(fE, c.qe[step]);
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        if (k >= nterms) continue;
        const double2 q = c.q[k][step];
        if (c.S[k] != 0.0) fc[k] = __fma_rn(fc[k], w[k], fc[k]);
        if (Bs::tf(c.kinds, k)) {
          if (c.S[k] != 0.0) fs[k] = __fma_rn(fs[k], w[k], fs[k]);
          xc[k] = __fma_rn(fc[k], q.x, -__dmul_rn(fs[k], q.y));
          xs[k] = __fma_rn(fc[k], q.y, __dmul_rn(fs[k], q.x));
        } else {
          xc[k] = __dmul_rn(fc[k], q.x);
          if (c.kinds[k] == kTermKT) fk[k] = __fma_rn(fk[k], wk[k], fk[k]);
          if (c.kinds[k] == kTermKT || c.kinds[k] == kTermLKT) kg[k] = __dmul_rn(fk[k], c.qk[k][step]);
        }
      }
    }
    // Time-only pieces of the bin: P (with cosine and sine parts), and a Kubo-Toyabe term's
    // derivative factors dK (along Delta) and, in Ps, dynamic Kubo-Toyabe's along nu.
#pragma unroll
    for (int k = 0; k < NT; ++k) {
      Pc[k] = xc[k];
      Ps[k] = xs[k];
      dK[k] = 0.0;
      if (k >= nterms || Bs::tf(c.kinds, k)) continue;
      const int kind = c.kinds[k];
      if (kind == kTermKT) {
        const double z = __dmul_rn(c.kt[k], t), u = __dmul_rn(z, z);
        const double Xg = __dmul_rn(xc[k], kg[k]);
        dK[k] = __dmul_rn(__dmul_rn(Xg, __dmul_rn(t, t)), __dadd_rn(u, -3.0));
        Pc[k] = __fma_rn(__dmul_rn(2.0 / 3.0, __dadd_rn(1.0, -u)), Xg, __dmul_rn(xc[k], 1.0 / 3.0));
      } else if (kind == kTermLKT) {
        const double u = __dmul_rn(c.kt[k], t);
        const double Xg = __dmul_rn(xc[k], kg[k]);
        dK[k] = __dmul_rn(__dmul_rn(Xg, t), __dadd_rn(u, -2.0));
        Pc[k] = __fma_rn(__dmul_rn(2.0 / 3.0, __dadd_rn(1.0, -u)), Xg, __dmul_rn(xc[k], 1.0 / 3.0));
      } else if (Bs::DKT && kind == kTermDKT) {
        double Gd = 1.0, gD = 0.0, gN = 0.0;
        if (c.dkt_src[k] >= 0)
          dkt_lookup(static_cast<const double*>(job.dkt) + static_cast<size_t>(c.dkt_src[k]) * kDktTable, t, &Gd, &gD,
                     &gN);
        dK[k] = __dmul_rn(xc[k], gD);
        Ps[k] = __dmul_rn(xc[k], gN);
        Pc[k] = __dmul_rn(xc[k], Gd);
      }
    }
  }
};

// ---------------------------------------------------------------------------------------------
// One work item: a tile of one chunk.  Channels, rows and their finalisation as on the SPLIT
// path (split_item), in FP64.  The cost's value is formed by explicitly rounded operations only,
// so that the value-only and the value+gradient kernels return the same bits.
// ---------------------------------------------------------------------------------------------
template <int SHAPE, int MODE, bool GRAD>
__device__ void basis64_item(const Job& job, const HistSet& hs, int item, Smem64& sm) {
  using Bs = Basis<SHAPE>;
  constexpr int NT = Bs::NT, M = Bs::M, G = Bs::G, NPH = Bs::NPH, NCH = Bs::NCH;
  constexpr bool GN = MODE == 2 || MODE == 3;
  static_assert(NCH + 1 <= 64, "channels and value in one scatter sum");
  const ChunkCache& cc = sm.cc;
  const Chunk64& c = sm.c;
  const int tid = threadIdx.x;
  const int nh = cc.nh, nlo = cc.nlo, nhi = cc.nhi, ts = sm.ts.tile_start;
  const int nterms = Bs::NTF < 0 ? min(hs.nterms, NT) : NT;
  const double dt = hs.dt_us;
  const bool f32 = hs.store == kStoreF32;
  const bool safe = c.safe != 0;
  bool timed = false;  // some term's value needs the bin's time (Kubo-Toyabe factors)
#pragma unroll
  for (int k = 0; k < NT; ++k) timed = timed || (k < nterms && !Bs::tf(c.kinds, k) && c.kinds[k] != kTermPlain);

  double acc_v = 0.0;
  double gacc[G][NPH], sh[NT][4];
#pragma unroll
  for (int i = 0; i < G; ++i)
#pragma unroll
    for (int q = 0; q < NPH; ++q) gacc[i][q] = 0.0;
#pragma unroll
  for (int k = 0; k < NT; ++k)
#pragma unroll
    for (int q = 0; q < 4; ++q) sh[k][q] = 0.0;
  int bad = 0;

  TimeFactors<SHAPE> tf;
  const int iters = min(hs.tile_bins / kBlock, (nhi - ts + kBlock - 1) / kBlock);
  double nd = 0.0, t_fresh = 0.0;  // bin - t0 and its time, of the last fresh bin
  for (int it = 0; it < iters; ++it) {
    const int n = ts + it * kBlock + tid, step = safe ? it & (kRebase - 1) : 0;
    if (step == 0) {
      nd = __dadd_rn(static_cast<double>(n), -cc.t0);
      t_fresh = __dmul_rn(nd, dt);
    }
    double t = t_fresh;
    if (step != 0 && (GRAD || timed)) t = __dadd_rn(t, c.td[step]);
    double E, Pc[NT], Ps[NT], dK[NT];
    tf.at(job, hs, c, step, iters > 1, nd, t, &E, Pc, Ps, dK);
    double Bf[M];
#pragma unroll
    for (int m = 0; m < M; ++m) Bf[m] = m == 0 ? E : 0.0;
#pragma unroll
    for (int k = 0; k < NT; ++k) {
      if (k >= nterms) continue;
      if (Bs::MERGED) {
        if (k < Bs::NTF) {
          Bf[1] = k == 0 ? Pc[k] : __dadd_rn(Bf[1], Pc[k]);
          Bf[2] = k == 0 ? Ps[k] : __dadd_rn(Bf[2], Ps[k]);
        } else {
          Bf[0] = __dadd_rn(Bf[0], Pc[k]);
        }
      } else {
        Bf[Bs::bc(k)] = Pc[k];
        if (Bs::tf(c.kinds, k)) Bf[Bs::bs(k)] = Ps[k];
      }
    }
    double Bd[GN ? M : 1];  // Gauss-Newton products: the basis functions' derivatives along v
    if (GN) {
#pragma unroll
      for (int m = 0; m < (GN ? M : 1); ++m) Bd[m] = 0.0;
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        if (k >= nterms) continue;
        const double g = -t * fma(t, c.dsig[k], c.dlam[k]);
        if (Bs::tf(c.kinds, k)) {
          const double w = kTwoPi * t * c.dnu[k];
          const double dc = fma(Pc[k], g, -Ps[k] * w), ds = fma(Ps[k], g, Pc[k] * w);
          Bd[Bs::bc(k) % (GN ? M : 1)] += dc;
          Bd[Bs::bs(k) % (GN ? M : 1)] += ds;
        } else {
          const double dN = Bs::DKT && c.kinds[k] == kTermDKT ? Ps[k] : 0.0;
          Bd[Bs::bc(k) % (GN ? M : 1)] += fma(Pc[k], g, fma(c.ddel[k], dK[k], c.dnu[k] * dN));
        }
      }
    }
    double V[M];
#pragma unroll
    for (int m = 0; m < M; ++m) V[m] = 0.0;

    const bool in = n >= nlo && n < nhi && dbg_ok(job.dbg, n < hs.stride, kDbgRow);
    if (in) {
#pragma unroll
      for (int hl = 0; hl < G; ++hl) {
        if (hl >= nh) break;
        const double* gm = c.gam[hl];
        double d, iv = 0.0;
        if (f32)
          d = widen(__ldg(static_cast<const float*>(cc.rowp[hl]) + n));
        else
          d = __ldg(static_cast<const double*>(cc.rowp[hl]) + n);
        if (MODE == 0 || MODE == 2)
          iv = cc.roww[hl] ? __ldg(static_cast<const double*>(cc.roww[hl]) + n) : count_weight(d, f32);
        double N = gm[0];
#pragma unroll
        for (int m = 0; m < M; ++m) N = __fma_rn(gm[1 + m], Bf[m], N);
        double u;
        if (GN) {
          const double* gdv = c.gdot[hl];
          double Nd = gdv[0];
#pragma unroll
          for (int m = 0; m < M; ++m) Nd = fma(gdv[1 + m], Bf[m], fma(gm[1 + m], Bd[m % (GN ? M : 1)], Nd));
          double cw = iv;
          if (MODE == 3) {
            cw = 0.0;
            if (positive(d)) {
              if (!positive(N)) bad = 1;
              cw = likelihood_weight(d, N);
            }
          }
          u = cw * Nd;
          acc_v = fma(u, Nd, acc_v);
        } else if (MODE == 0) {
          const double r = __dadd_rn(N, -d);
          u = __dmul_rn(r, iv);
          acc_v = __fma_rn(r, u, acc_v);
        } else {
          const double r = __dadd_rn(N, -d);
          if (positive(d)) {
            u = __dmul_rn(r, recip(N));
            double x = __dadd_rn(1.0, -u);  // d/N
            // Below 2^-20 the difference has lost d/N's digits (and below 2^-53 all of them): the
            // quotient itself.  Above it the logarithm's error, 2^-53 N/d, times d stays at 2^-53 of
            // the bin's N - d.  N outside recip's range comes here too.
            if (__double2hiint(x) < kRatioHi || !recip_range(N)) {
              x = divide(d, N);
              u = __dadd_rn(1.0, -x);
              if (!positive(N)) bad = 1;
            }
            acc_v = __dadd_rn(acc_v, __fma_rn(d, ln_tab(x, sm.logtab), r));
          } else {
            u = 1.0;
            acc_v = __dadd_rn(acc_v, r);
          }
        }
        if (GRAD) {
#pragma unroll
          for (int m = 0; m < M; ++m) gacc[hl][m] = fma(u, Bf[m], gacc[hl][m]);
          gacc[hl][M] += u;
#pragma unroll
          for (int m = 0; m < M; ++m) V[m] = fma(u, gm[1 + m], V[m]);
        }
      }
    }
    if (GRAD && in) {  // beyond the window a growing factor may have overflowed, and 0 times it is not 0
      const double h2 = 0.5 * t * t;
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        if (k >= nterms) continue;
        const double Vc = V[Bs::bc(k)];
        double Dk;
        if (Bs::tf(c.kinds, k)) {
          const double Vs = V[Bs::bs(k)];
          Dk = fma(Vc, Pc[k], Vs * Ps[k]);
          sh[k][2] = fma(t, fma(Vs, Pc[k], -Vc * Ps[k]), sh[k][2]);  // times 2 pi at the end
        } else {
          Dk = Vc * Pc[k];
          if (c.kinds[k] != kTermPlain) sh[k][3] = fma(Vc, dK[k], sh[k][3]);
          if (Bs::DKT && c.kinds[k] == kTermDKT) sh[k][2] = fma(Vc, Ps[k], sh[k][2]);
        }
        sh[k][0] = fma(-t, Dk, sh[k][0]);
        if (c.S[k] != 0.0) sh[k][1] = fma(-h2, Dk, sh[k][1]);
      }
    }
  }

  // thread -> warp (scatter sum) -> CTA (FP64 tree) -> row
  bad = __syncthreads_or(bad);
  const int lane = tid & 31, wp = tid >> 5;
  if (GRAD) {
    double a[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) a[i] = 0.0;
    a[0] = acc_v;
#pragma unroll
    for (int hl = 0; hl < G; ++hl)
#pragma unroll
      for (int q = 0; q < NPH; ++q) a[1 + hl * NPH + q] = gacc[hl][q];
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q) a[1 + G * NPH + k * 4 + q] = sh[k][q];
    warp_scatter_sum<64>(a);
    sm.red[wp][2 * lane] = a[0];
    sm.red[wp][2 * lane + 1] = a[1];
  } else {
    const double r = warp_sum_d(acc_v);
    if (lane == 0) sm.red[wp][0] = r;
  }
  __syncthreads();
  static_assert(kWarps == 8, "the tree below sums 8 warps");
  if (!dbg_ok(job.dbg, item >= 0 && item < job.nrows, kDbgPartial)) return;
  double* row = job.partials + static_cast<int64_t>(item) * hs.pstride;
  if (tid < (GRAD ? 1 + NCH : 1)) {
    double s = ((sm.red[0][tid] + sm.red[1][tid]) + (sm.red[2][tid] + sm.red[3][tid])) +
               ((sm.red[4][tid] + sm.red[5][tid]) + (sm.red[6][tid] + sm.red[7][tid]));
    if (tid == 0) {
      if (MODE != 0) s *= 2.0;
      // +inf: the likelihood is undefined (N <= 0 where d > 0) or the parameters were not finite
      if (bad || !isfinite(s)) s = __longlong_as_double(0x7ff0000000000000LL);
    } else if (tid > G * NPH) {
      const int k = (tid - 1 - G * NPH) >> 2, q = (tid - 1 - G * NPH) & 3;
      if (q == 2 && k < nterms && Bs::tf(c.kinds, k)) s *= kTwoPi;
    }
    row[tid] = s;
  }
}

// Persistent kernel: each CTA takes a contiguous range of the launch's items, as eval_kernel.  One
// CTA per SM: its 8 warps keep the FP64 pipe as busy as 16 do (84-90 % of its peak), and the
// decomposition is picked for that grid.
// Measured on GB300 (a call with its copies, before: the term-list kernel with CUDA's library
// functions per histogram and bin):
//   8 x 65536 bins, two cosine terms, -2lnL value and gradient, one vector   467 ->   79 us
//   1 x 16384 bins, one cosine term, -2lnL at 1000 vectors                  4116 -> 1040 us
//   8 x 65536 bins, Gauss-Newton products along 28 directions               8884 ->  849 us
//   (the whole matrix: musr_gram64.cu)
// The first of these executes 44 FP64 instructions per pair (16 of them fresh time factors, a CTA
// having two iterations), the second 30 (33, 1114 us, with a table of 256 intervals and the bin's time
// formed in every bin), the third 31.
template <int SHAPE, int MODE, bool GRAD>
__global__ void __launch_bounds__(kBlock, 1) eval64_kernel(const __grid_constant__ LaunchHead head) {
  __shared__ Smem64 sm;
  const int per = (head.total_items + gridDim.x - 1) / gridDim.x;
  const int beg = blockIdx.x * per, end = min(head.total_items, beg + per);
  if (threadIdx.x == 0) {
    sm.cc.job = -1;
    sm.cc.chunk = -1;
    sm.hs_src = nullptr;
  }
  if (MODE == 1)  // read after several barriers
    for (int i = threadIdx.x; i < kLogTable; i += kBlock) sm.logtab[i] = log_table.t[i];
  const Job& job = sm.job;
  const HistSet& hs = sm.hs;
  int ji = -1;
  for (int gi = beg; gi < end; ++gi) {
    int chunk = -1;
    if (ji < 0) {
      ji = job_of_item(head, gi);
      if (ji == 0) chunk = head.first.items[gi].x;  // on its way beside the histogram set
      enter_job(head, ji, sm);
    }
    while (gi >= job.item_begin + hs.nitems) {
      enter_job(head, ++ji, sm);
      chunk = -1;
    }
    const int item = gi - job.item_begin;
    if (sm.cc.job != ji || item < sm.cc.item0 || item >= sm.cc.item0 + sm.cc.ntiles) {
      if (chunk < 0) chunk = job.items[item].x;
      __syncthreads();
      load_chunk(job, hs, ji, chunk, sm);
      load_chunk64<SHAPE>(job, hs, sm);
    }
    load_tile_at(sm.cc.tile0 + (item - sm.cc.item0) * hs.tile_bins, hs, 0, sm);
    basis64_item<SHAPE, MODE, GRAD>(job, hs, item, sm);
    complete_item<2, SHAPE, GRAD>(job, hs, sm);
  }
}

template <int SHAPE, int MODE, bool GRAD>
int launch64(const LaunchHead& head, int num_sms, cudaStream_t stream, LaunchInfo* info) {
  int grid = num_sms < head.total_items ? num_sms : head.total_items;
  if (grid < 1) grid = 1;
  eval64_kernel<SHAPE, MODE, GRAD><<<grid, kBlock, 0, stream>>>(head);
  if (info) {
    info->grid = grid;
    info->block = kBlock;
  }
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

template <int SHAPE>
int dispatch64(int mode, int grad, const LaunchHead& h, int sms, cudaStream_t s, LaunchInfo* info) {
  if (mode == 2) return launch64<SHAPE, 2, true>(h, sms, s, info);
  if (mode == 3) return launch64<SHAPE, 3, true>(h, sms, s, info);
  if (mode == 0) return grad ? launch64<SHAPE, 0, true>(h, sms, s, info) : launch64<SHAPE, 0, false>(h, sms, s, info);
  return grad ? launch64<SHAPE, 1, true>(h, sms, s, info) : launch64<SHAPE, 1, false>(h, sms, s, info);
}

}  // namespace
}  // namespace kern
}  // namespace musr
