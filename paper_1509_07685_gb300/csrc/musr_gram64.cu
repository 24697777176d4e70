// musr_gram64.cu -- the Gauss-Newton matrix of a theory with a basis form in one pass over the data
// (FP64): per histogram the sums over bins of (d^2 cost / dN^2) J_i J_j over its local slots, which
// the host adds up into parameters through the map.
//
// The matrix by products with unit vectors is P evaluations: 31 FP64 instructions per (histogram,
// bin) pair and parameter, 862 for 28 parameters, and the FP64 pipe was 91 % busy with them.  A
// histogram has few local slots (7 there), so its own triangle of 28 sums, with the 13 multiply-adds
// that form J, the reciprocal and the weight, is 57 per pair (90 executed, with the
// time functions, the set-up and the sums).
// The CTA's threads first evaluate the time functions of 256 bins (the basis functions, and P t,
// P t^2 and the Kubo-Toyabe derivatives of each term) into shared memory, a bin each; then each
// warp takes one histogram of the chunk (several warps one histogram where the chunk has fewer than
// 8) and a lane a bin, with the triangle in registers; so one kernel per shape serves every theory,
// J's coefficients being data.  A CTA keeps its sums over all its tiles of a chunk and writes one row.
// Measured on GB300 (8 x 65536 bins, 28 parameters, -2lnL, the whole call): 8.88 ms with the term-list
// kernel's products, 0.85 ms with the basis kernel's, 0.134 ms here.
// Up to 12 local slots (78 sums fill the registers); theories with more, and dynamic Kubo-Toyabe factors,
// whose tables are solved for a job on the device, keep the products, as do theories with a primitive on
// N0's slot.
#include "musr_kernels_f64.cuh"

namespace musr {
namespace kern {
namespace {

template <int SHAPE>
struct GramSmem {
  static constexpr int F = Basis<SHAPE>::M + 6 * Basis<SHAPE>::NT;
  Job job;
  double x[kHeadParams];
  HistSet hs;
  const HistSet* hs_src;
  ChunkCache cc;
  TileState ts;
  Chunk64 c;
  double phi[F][kBlock];
  double coef[kGroupMax][kGramEntries];
  double red[kWarps][96];
};

// Coefficient of an entry for chunk histogram hl.
template <int SHAPE>
__device__ double gram_coef(const HistSet& hs, const ChunkCache& cc, const Chunk64& c, int hl, GramEntry e) {
  using Bs = Basis<SHAPE>;
  constexpr double kDeg = kTwoPi / 360.0;
  const int k = e.term;
  const double N0 = cc.loc[hl][0], co = cc.cph[hl][k], sn = cc.sph[hl][k];
  const double a = !Bs::MERGED && k < hs.nterms && hs.canon[k].amp_slot >= 0 ? cc.loc[hl][hs.canon[k].amp_slot] : 1.0;
  const double gc = c.gam[hl][1 + Bs::bc(k)], gs = c.gam[hl][1 + Bs::bs(k)];
  switch (e.coef) {
    case kGOne:
      return 1.0;
    case kGN0C:
      return a * co;
    case kGN0S:
      return -a * sn;
    case kGN0P:
      return a;
    case kGAmpC:
      return N0 * co;
    case kGAmpS:
      return -N0 * sn;
    case kGAmpP:
      return N0;
    case kGPhiC:
      return -N0 * a * kDeg * sn;
    case kGPhiS:
      return -N0 * a * kDeg * co;
    case kGLamC:
      return -gc;
    case kGLamS:
      return -gs;
    case kGSigC:
      return -cc.loc[0][e.slot] * gc;
    case kGSigS:
      return -cc.loc[0][e.slot] * gs;
    case kGNuC:
      return kTwoPi * gs;
    case kGNuS:
      return -kTwoPi * gc;
    case kGDel:
      return (2.0 / 3.0) * cc.loc[0][e.slot] * gc;
    case kGLkt:
      return (2.0 / 3.0) * gc;
    default:
      return gc;
  }
}

// NJ: the slots at most (8 or 12); the triangle's NJ (NJ + 1) / 2 sums per thread in registers.
template <int SHAPE, int NJ>
__global__ void __launch_bounds__(kBlock, 1) gram64_kernel(const __grid_constant__ LaunchHead head,
                                                           const __grid_constant__ GramPlan gp, double* __restrict__ rows) {
  using Bs = Basis<SHAPE>;
  constexpr int NT = Bs::NT, M = Bs::M, NE = NJ * (NJ + 1) / 2, NP = (NE + 31) / 32 * 32;
  extern __shared__ __align__(16) unsigned char gram_smem[];
  GramSmem<SHAPE>& sm = *reinterpret_cast<GramSmem<SHAPE>*>(gram_smem);
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int per = (head.total_items + gridDim.x - 1) / gridDim.x;
  const int beg = blockIdx.x * per, end = min(head.total_items, beg + per);
  if (tid == 0) sm.hs_src = nullptr;
  const Job& job = sm.job;
  const HistSet& hs = sm.hs;
  const ChunkCache& cc = sm.cc;
  if (beg >= end) return;
  enter_job(head, 0, sm);
  const int nj = gp.nj;
  double acc[NP];
  int bad = 0, cur = -1;

  auto flush = [&] {  // the CTA's sums of the current chunk: one row per histogram
    const int any = __syncthreads_or(bad);
    warp_scatter_sum<NP>(acc);
#pragma unroll
    for (int i = 0; i < NP / 32; ++i) sm.red[wp][lane * (NP / 32) + i] = acc[i];
    __syncthreads();
    const int nh = cc.nh, parts = kWarps / nh;
    double* row = rows + (static_cast<int64_t>(blockIdx.x) + cur) * (kGroupMax * NE);
    for (int i = tid; i < nh * NE; i += kBlock) {
      const int hl = i / NE, e = i - hl * NE;
      double v = 0.0;
      for (int p = 0; p < parts; ++p) v += sm.red[hl * parts + p][e];
      row[i] = any ? __longlong_as_double(0x7ff0000000000000LL) : v;  // the likelihood is undefined
    }
    __syncthreads();
  };

  for (int gi = beg; gi < end; ++gi) {
    const int chunk = job.items[gi].x;
    if (chunk != cur) {
      if (cur >= 0) flush();
      cur = chunk;
      bad = 0;
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[i] = 0.0;
      load_chunk(job, hs, 0, chunk, sm);
      load_chunk64<SHAPE>(job, hs, sm);
      const int ne = gp.ptr[nj];
      for (int i = tid; i < cc.nh * ne; i += kBlock) {
        const int hl = i / ne, e = i - hl * ne;
        sm.coef[hl][e] = gram_coef<SHAPE>(hs, cc, sm.c, hl, gp.e[e]);
      }
      __syncthreads();
    }
    const int ts = cc.tile0 + (gi - cc.item0) * hs.tile_bins;
    const int iters = min(hs.tile_bins / kBlock, (cc.nhi - ts + kBlock - 1) / kBlock);
    const int nterms = Bs::NTF < 0 ? min(hs.nterms, NT) : NT;
    const int parts = kWarps / cc.nh, hl = wp / parts, part = wp - hl * parts;
    const bool busy = hl < cc.nh, f32 = hs.store == kStoreF32;
    TimeFactors<SHAPE> tf;
    double nd = static_cast<double>(ts + tid) - cc.t0;
    for (int it = 0; it < iters; ++it, nd += static_cast<double>(kBlock)) {
      {
        const double t = nd * hs.dt_us;
        double E, Pc[NT], Ps[NT], dK[NT];
        tf.at(job, hs, sm.c, sm.c.safe ? it & (kRebase - 1) : 0, iters > 1, nd, t, &E, Pc, Ps, dK);
        double Bf[M];
#pragma unroll
        for (int m = 0; m < M; ++m) Bf[m] = m == 0 ? E : 0.0;
#pragma unroll
        for (int k = 0; k < NT; ++k) {
          if (k >= nterms) continue;
          const bool cosine = Bs::tf(sm.c.kinds, k);
          Bf[Bs::bc(k)] = Bs::MERGED ? Bf[Bs::bc(k)] + Pc[k] : Pc[k];
          if (cosine) Bf[Bs::bs(k)] = Bs::MERGED ? Bf[Bs::bs(k)] + Ps[k] : Ps[k];
          sm.phi[M + 6 * k][tid] = t * Pc[k];
          if (cosine) sm.phi[M + 6 * k + 1][tid] = t * Ps[k];
          if (sm.c.S[k] != 0.0) {
            sm.phi[M + 6 * k + 2][tid] = t * (t * Pc[k]);
            if (cosine) sm.phi[M + 6 * k + 3][tid] = t * (t * Ps[k]);
          } else {  // a width of 0: its derivative's coefficient is 0 too
            sm.phi[M + 6 * k + 2][tid] = sm.phi[M + 6 * k + 3][tid] = 0.0;
          }
          if (!cosine) sm.phi[M + 6 * k + 4][tid] = dK[k];
        }
#pragma unroll
        for (int m = 0; m < M; ++m) sm.phi[m][tid] = Bf[m];
      }
      __syncthreads();
      if (busy) {
        const double Nbkg = cc.loc[hl][1], N0 = cc.loc[hl][0];
        for (int r = part; r < kBlock / 32; r += parts) {
          const int b = r * 32 + lane, n = ts + it * kBlock + b;
          if (n < cc.nlo || n >= cc.nhi || !dbg_ok(job.dbg, n < hs.stride, kDbgRow)) continue;
          const double d = f32 ? widen(__ldg(static_cast<const float*>(cc.rowp[hl]) + n))
                               : __ldg(static_cast<const double*>(cc.rowp[hl]) + n);
          double J[NJ];
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            J[j] = 0.0;
            if (j >= nj) continue;
            const int e1 = gp.ptr[j + 1];
            for (int e = gp.ptr[j]; e < e1; ++e) {
              const int fn = gp.e[e].func;
              const double v = sm.coef[hl][e];
              J[j] = fn == 255 ? J[j] + v : fma(v, sm.phi[fn][b], J[j]);
            }
          }
          const double N = fma(N0, J[0], Nbkg);
          double w;
          if (gp.mode == 2) {
            w = 2.0 * (cc.roww[hl] ? __ldg(static_cast<const double*>(cc.roww[hl]) + n) : count_weight(d, f32));
          } else {
            w = 0.0;  // without a count: 0 times a derivative that is not finite is not 0
            if (positive(d)) {
              if (!positive(N)) bad = 1;
              w = 2.0 * likelihood_weight(d, N);
            }
          }
#pragma unroll
          for (int i = 0; i < NJ; ++i) {
            if (i >= nj) break;
            const double wj = w * J[i];
#pragma unroll
            for (int j = 0; j <= i; ++j) acc[i * (i + 1) / 2 + j] = fma(wj, J[j], acc[i * (i + 1) / 2 + j]);
          }
        }
      }
      __syncthreads();
    }
  }
  flush();
}

// Sums the rows of a chunk's histogram in CTA order: block (hl, chunk), kSeg threads per value.
constexpr int kSeg = 8;
__global__ void gram_sum_kernel(const HistSet* __restrict__ hsp, const double* __restrict__ rows, double* __restrict__ sums,
                                int ne, int per) {
  __shared__ double seg[kSeg][78];
  const int hl = blockIdx.x, chunk = blockIdx.y, e = threadIdx.x % ne, k = threadIdx.x / ne;
  const Chunk& ch = hsp->chunks[chunk];
  if (hl >= ch.nh) return;
  const int b0 = ch.item0 / per, n = (ch.item0 + ch.ntiles - 1) / per - b0 + 1;
  double v = 0.0;
  for (int b = n * k / kSeg; b < n * (k + 1) / kSeg; ++b)
    v += rows[(static_cast<int64_t>(b0 + b + chunk) * kGroupMax + hl) * ne + e];
  seg[k][e] = v;
  __syncthreads();
  if (k == 0) {
    v = 0.0;
    for (int q = 0; q < kSeg; ++q) v += seg[q][e];
    sums[(static_cast<int64_t>(chunk) * kGroupMax + hl) * ne + e] = v;
  }
}

template <int SHAPE, int NJ>
int launch_gram_of(const GramPlan& plan, const LaunchHead& head, int nchunks, double* rows, double* sums, int num_sms,
                   cudaStream_t s) {
  constexpr int NE = NJ * (NJ + 1) / 2;
  auto kernel = gram64_kernel<SHAPE, NJ>;
  constexpr int bytes = static_cast<int>(sizeof(GramSmem<SHAPE>));
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return -1;
  const int grid = num_sms < head.total_items ? num_sms : head.total_items;
  kernel<<<grid, kBlock, bytes, s>>>(head, plan, rows);
  if (cudaPeekAtLastError() != cudaSuccess) return -1;
  const int per = (head.total_items + grid - 1) / grid;
  gram_sum_kernel<<<dim3(kGroupMax, nchunks), kSeg * NE, 0, s>>>(head.first.hs, rows, sums, NE, per);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

// The entries of one shape.
template <int SHAPE>
bool plan_of(const HistSet& hs, const bool* active, GramPlan* p) {
  using Bs = Basis<SHAPE>;
  int nj = 0, ne = 0;
  bool fits = true;
  auto put = [&](int func, int coef, int term, int slot) {
    if (ne == kGramEntries) {
      fits = false;
      return;
    }
    p->e[ne++] = {static_cast<unsigned char>(func), static_cast<unsigned char>(coef), static_cast<unsigned char>(term),
                  static_cast<unsigned char>(slot)};
  };
  auto fn = [](int k, int q) { return Bs::M + 6 * k + q; };
  // The kernel forms N from slot 0's derivative (N = N0 J_0 + Nbkg), which is N / N0's only where nothing
  // but N0 reads the slot; a theory whose primitives read it too keeps the products.
  for (int i = hs.slot_ptr[0]; i < hs.slot_ptr[1]; ++i)
    if (hs.contrib[hs.slot_list[i]].kind != kCN0) return false;
  for (int s = 0; s < hs.nslots && fits; ++s) {
    if (s != 0 && (!active[s] || hs.slot_ptr[s] == hs.slot_ptr[s + 1])) continue;
    if (nj == kGramSlots) return false;
    p->slot[nj] = static_cast<unsigned char>(s);
    p->ptr[nj++] = static_cast<unsigned char>(ne);
    for (int i = hs.slot_ptr[s]; i < hs.slot_ptr[s + 1]; ++i) {
      const Contrib c = hs.contrib[hs.slot_list[i]];
      const int k = c.term;
      const bool cosine = hs.canon[k].kind == kTermTF;
      const int bc = Bs::bc(k), bs = Bs::bs(k);
      switch (c.kind) {
        case kCN0:
          if (hs.envelope) put(0, kGOne, 0, s);
          for (int q = 0; q < (Bs::MERGED ? 1 : hs.nterms); ++q) {
            if (hs.canon[q].kind == kTermTF) {
              put(Bs::bc(q), kGN0C, q, s);
              put(Bs::bs(q), kGN0S, q, s);
            } else if (!Bs::MERGED) {
              put(Bs::bc(q), kGN0P, q, s);
            }
          }
          break;
        case kCBkg:
          put(255, kGOne, 0, s);
          break;
        case kCAmp:
          put(bc, cosine ? kGAmpC : kGAmpP, k, s);
          if (cosine) put(bs, kGAmpS, k, s);
          break;
        case kCPhi:
          put(bc, kGPhiC, k, s);
          put(bs, kGPhiS, k, s);
          break;
        case kCLam:
          put(fn(k, 0), kGLamC, k, s);
          if (cosine) put(fn(k, 1), kGLamS, k, s);
          break;
        case kCSig:
          put(fn(k, 2), kGSigC, k, s);
          if (cosine) put(fn(k, 3), kGSigS, k, s);
          break;
        case kCNu:
          put(fn(k, 0), kGNuC, k, s);
          put(fn(k, 1), kGNuS, k, s);
          break;
        case kCDel:
          put(fn(k, 4), kGDel, k, s);
          break;
        case kCLkt:
          put(fn(k, 4), kGLkt, k, s);
          break;
        default:
          return false;  // dynamic Kubo-Toyabe: its tables need a job on the device
      }
    }
  }
  p->nj = nj;
  for (int j = nj; j <= kGramSlots; ++j) p->ptr[j] = static_cast<unsigned char>(ne);
  return fits && nj > 0;
}

}  // namespace
}  // namespace kern

#define MUSR_BY_SHAPE(shape, CALL) \
  switch (shape) {                 \
    CALL(kShapeGeneric)            \
    CALL(kShapeT1)                 \
    CALL(kShapeN1)                 \
    CALL(kShapeT1N1)               \
    CALL(kShapeT2)                 \
    CALL(kShapeT2N1)               \
    CALL(kShapeT2m)                \
    CALL(kShapeT2N1m)              \
  }

bool gram_plan(const HistSet& hs, const bool* active, int mode, GramPlan* plan) {
  plan->mode = mode;
#define MUSR_CALL(S) \
  case S:            \
    return kern::plan_of<S>(hs, active, plan);
  MUSR_BY_SHAPE(hs.shape, MUSR_CALL)
#undef MUSR_CALL
  return false;
}

int64_t gram_rows(const GramPlan& plan, int nchunks, int num_sms) {
  return (static_cast<int64_t>(num_sms) + nchunks) * kGroupMax * gram_values(plan.nj);
}

int launch_gram(int shape, const GramPlan& plan, const LaunchHead& head, int nchunks, double* rows, double* sums,
                int num_sms, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
#define MUSR_CALL(S)                                                                             \
  case S:                                                                                        \
    return plan.nj <= 8 ? kern::launch_gram_of<S, 8>(plan, head, nchunks, rows, sums, num_sms, s) \
                        : kern::launch_gram_of<S, 12>(plan, head, nchunks, rows, sums, num_sms, s);
  MUSR_BY_SHAPE(shape, MUSR_CALL)
#undef MUSR_CALL
  return -1;
}

}  // namespace musr
