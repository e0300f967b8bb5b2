// Data movers of the contraction path and of fuse / unfuse (Sec. II.B: the
// "permutes, reshapes, and copies" that fill the fused storage), plus the trace.
//
// One launch runs every piece of a phase. A CTA takes one work item: up to 32
// pieces (see CopyJob) with at most 4096 elements in all, staged whole in
// shared memory. The dense side of each piece (a contiguous range of its
// block) is moved linearly; the strided side is visited in its own order, so
// that consecutive threads touch consecutive addresses along its innermost
// dim. Index arithmetic per element is one multiply-high division per dim; the
// reads are asynchronous copies into shared memory, a whole item in flight.
// HBM-bound: every element is read once and written once.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.hpp"

namespace ytn {

namespace {

constexpr int kThreads = 256;
constexpr int kJobWords = (int)(sizeof(CopyJob) / 4);

__device__ __forceinline__ void cp_async8(double *smem_dst, const double *gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
               "l"(gsrc)
               : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// Negation by the sign bit (an integer operation: this GPU's FP64 pipe is far
// slower than its memory system); exact, and it keeps NaN payloads.
constexpr unsigned long long kSignBit = 0x8000000000000000ull;

__device__ __forceinline__ double flip(double x, unsigned long long mask) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)mask);
}

// The parameters of one piece, in registers: the last ND of its dim slots.
template <int ND>
struct Piece {
  int64_t g_off, d_off;
  int p;       // the piece's start in the staging buffer
  int negmode; // 0: as is; 1: negated (fermionic swap gate); 2: odd source offsets
               // negated (imaginary parts of interleaved complex data: conj)
  int ext[ND], gstr[ND], lstr[ND], shf[ND];
  uint32_t mag[ND];

  __device__ __forceinline__ void load(const CopyJob &J) {
    g_off = J.g_off;
    d_off = J.d_off;
    p = J.p;
    negmode = J.negate;
#pragma unroll
    for (int i = 0; i < ND; i++) {
      const int k = kMaxCopyDims - ND + i;
      ext[i] = J.ext[k];
      gstr[i] = J.gstr[k];
      lstr[i] = J.lstr[k];
      mag[i] = J.mag[k];
      shf[i] = J.shf[k];
    }
  }

  // Element l of the piece (in strided-side order): its offsets on the strided
  // side (global, from g_off) and on the dense side (from the piece's start).
  __device__ __forceinline__ void offsets(uint32_t l, int64_t &go, int &lo) const {
    go = 0;
    lo = 0;
#pragma unroll
    for (int i = ND - 1; i > 0; i--) {
      const uint32_t q = (l + __umulhi(l, mag[i])) >> shf[i];
      const int r = (int)(l - q * (uint32_t)ext[i]);
      go += (int64_t)r * gstr[i];
      lo += r * lstr[i];
      l = q;
    }
    go += (int64_t)l * gstr[0];
    lo += (int)l * lstr[0];
  }
};

// Calls body(P, l, e) for every element e of the item's flat range
// [w0, w1) of this warp: lanes take consecutive elements of one piece at a time
// (l: the element's index in its piece), so that a warp's accesses to the
// strided side follow that side's innermost dim. A piece's parameters are read
// from shared memory once per warp and piece.
template <int ND, class Body>
__device__ __forceinline__ void for_warp_range(const CopyJob *Js, int nj, int w0, int w1, Body body) {
  if (w0 >= w1) return;
  const int lane = threadIdx.x & 31;
  // first piece: the last one starting at or before w0
  int j = 31 - __clz(__ballot_sync(0xffffffffu, lane < nj && Js[lane].p <= w0));
  for (int e0 = w0; e0 < w1; j++) {
    Piece<ND> P;
    P.load(Js[j]);
    const int seg_end = min(w1, P.p + Js[j].size);
#pragma unroll 4
    for (int e = e0 + lane; e < seg_end; e += 32) body(P, e - P.p, e);
    e0 = seg_end;
  }
}

// DENSE_SRC (mode 2): read linearly, write in destination order; else
// (mode 3) read in source order, write linearly. The reads are asynchronous
// copies straight into shared memory, all of an item's in flight at once.
// Each warp takes one eighth of the item's elements in both phases.
template <int ND, bool DENSE_SRC>
__device__ __forceinline__ void stage_item(const CopyJob *Js, int nj, int total, const double *src,
                                           double *__restrict__ dst, double *stage) {
  constexpr int kWarps = kThreads / 32;
  const int per_warp = (total + kWarps - 1) / kWarps;
  const int w0 = min(total, (int)(threadIdx.x >> 5) * per_warp), w1 = min(total, w0 + per_warp);
  if (DENSE_SRC) {
    for_warp_range<ND>(Js, nj, w0, w1, [&](const Piece<ND> &P, int l, int e) {
      cp_async8(stage + e, src + P.d_off + l);
    });
  } else {
    for_warp_range<ND>(Js, nj, w0, w1, [&](const Piece<ND> &P, int l, int e) {
      int64_t go;
      int lo;
      P.offsets((uint32_t)l, go, lo);
      const int at = P.p + lo;
      if ((unsigned)at < (unsigned)total) cp_async8(stage + at, src + P.g_off + go);
    });
  }
  cp_async_wait_all();
  __syncthreads();
  if (DENSE_SRC) {
    for_warp_range<ND>(Js, nj, w0, w1, [&](const Piece<ND> &P, int l, int e) {
      int64_t go;
      int lo;
      P.offsets((uint32_t)l, go, lo);
      const int at = P.p + lo;
      const bool neg = P.negmode == 1 || (P.negmode == 2 && ((P.d_off + lo) & 1));
      if ((unsigned)at < (unsigned)total) dst[P.g_off + go] = flip(stage[at], neg ? kSignBit : 0ull);
    });
  } else {
    for_warp_range<ND>(Js, nj, w0, w1, [&](const Piece<ND> &P, int l, int e) {
      dst[P.d_off + l] = flip(stage[e], P.negmode == 1 ? kSignBit : 0ull);
    });
  }
}

template <int ND>
__device__ __forceinline__ void stage_dispatch(bool dense_src, const CopyJob *Js, int nj, int total,
                                               const double *src, double *dst, double *stage) {
  if (dense_src) stage_item<ND, true>(Js, nj, total, src, dst, stage);
  else stage_item<ND, false>(Js, nj, total, src, dst, stage);
}

// One work item: its pieces' parameters into shared memory, then the staged move.
// MAXND: the most dims an item of the launch has (the host reads it from the job
// table). Instantiated for at most 4 dims the kernel needs 48 registers instead
// of 64 and fits five CTAs per SM instead of four.
template <int MAXND>
__device__ __forceinline__ void run_item(const CopyJob *__restrict__ jobs, const CopyItem &it,
                                         const double *src, double *__restrict__ dst, CopyJob *Js,
                                         double *stage) {
  const int nj = it.njobs, total = it.total, nd = it.kind & 255, mode = it.kind >> 8;
  // the planner never makes other items, and the host never launches an item with
  // more dims than MAXND
  if (nj < 1 || nj > kStageJobs || total < 1 || total > kStageElems || nd < 1 || nd > MAXND) return;
  {
    const int32_t *s = reinterpret_cast<const int32_t *>(jobs + it.job);
    int32_t *d = reinterpret_cast<int32_t *>(Js);
    for (int w = threadIdx.x; w < nj * kJobWords; w += kThreads) d[w] = s[w];
  }
  __syncthreads();
  const bool dense_src = mode == 2;
  switch (nd) {
    case 1: stage_dispatch<1>(dense_src, Js, nj, total, src, dst, stage); break;
    case 2: stage_dispatch<2>(dense_src, Js, nj, total, src, dst, stage); break;
    case 3: stage_dispatch<3>(dense_src, Js, nj, total, src, dst, stage); break;
    case 4: stage_dispatch<4>(dense_src, Js, nj, total, src, dst, stage); break;
    default:
      if constexpr (MAXND > 4) {
        switch (nd) {
          case 5: stage_dispatch<5>(dense_src, Js, nj, total, src, dst, stage); break;
          case 6: stage_dispatch<6>(dense_src, Js, nj, total, src, dst, stage); break;
          case 7: stage_dispatch<7>(dense_src, Js, nj, total, src, dst, stage); break;
          default: stage_dispatch<8>(dense_src, Js, nj, total, src, dst, stage); break;
        }
      }
      break;
  }
}

template <int MAXND>
__global__ void __launch_bounds__(kThreads, MAXND <= 4 ? 5 : 4) copy_kernel(const CopyJob *__restrict__ jobs,
                                                                           const CopyItem *__restrict__ items,
                                                                           unsigned first,
                                                                           const double *src,
                                                                           double *__restrict__ dst,
                                                                           const double *src2,
                                                                           double *__restrict__ dst2) {
  __shared__ CopyJob Js[kStageJobs];
  __shared__ double stage[kStageElems];
  after_previous_kernel();
  const bool one = blockIdx.x < first;
  run_item<MAXND>(jobs, items[blockIdx.x], one ? src : src2, one ? dst : dst2, Js, stage);
}

// Gathers of the sectors that the split path's accuracy check flagged (FP64
// fallback): a persistent grid, even CTAs for A and odd ones for B, walks the flagged
// sectors' work items (each sector's items are [first[q], first[q] + count), the
// running counts over the flagged sectors in item_end). With no flagged sector every
// CTA returns at once.
struct FlaggedGather {
  const CopyItem *items;
  const int32_t *item_end;
  const double *src;
  double *dst;
};

__global__ void __launch_bounds__(kThreads, 4) copy_flagged_kernel(const CopyJob *__restrict__ jobs,
                                                                   const SplitSector *__restrict__ sectors,
                                                                   const int32_t *flagged,
                                                                   const SplitRecord *rec,
                                                                   FlaggedGather ga, FlaggedGather gb) {
  __shared__ CopyJob Js[kStageJobs];
  __shared__ double stage[kStageElems];
  after_previous_kernel();
  const int nflag = rec->nfallback;
  if (nflag <= 0) return;
  const bool isA = (blockIdx.x & 1) == 0;
  const FlaggedGather g = isA ? ga : gb;
  const int total = g.item_end[nflag - 1];
  for (int t = blockIdx.x >> 1; t < total; t += gridDim.x >> 1) {
    int lo = 0, hi = nflag - 1;   // first flagged sector whose items end after t
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (g.item_end[mid] > t) hi = mid;
      else lo = mid + 1;
    }
    const SplitSector &sc = sectors[flagged[lo]];
    const int first = isA ? sc.ga0 : sc.gb0;
    const int local = t - (lo > 0 ? g.item_end[lo - 1] : 0);
    __syncthreads();   // the previous item's shared memory is no longer read
    run_item<kMaxCopyDims>(jobs, g.items[first + local], g.src, g.dst, Js, stage);
  }
}

// Zero fill of the flagged sectors' FP64 sector matrices (partially populated
// operands) before their gathers.
__global__ void __launch_bounds__(kThreads) zero_flagged_kernel(const SectorDev *__restrict__ sectors,
                                                                const int32_t *flagged,
                                                                const SplitRecord *rec, double *wa,
                                                                double *wb, int zero_a, int zero_b) {
  after_previous_kernel();
  const int nflag = rec->nfallback;
  for (int k = blockIdx.x; k < nflag; k += gridDim.x) {
    const SectorDev s = sectors[flagged[k]];
    const int64_t na = zero_a ? (int64_t)s.M * s.K : 0, nb = zero_b ? (int64_t)s.K * s.N : 0;
    for (int64_t e = threadIdx.x; e < na; e += kThreads) wa[s.a_off + e] = 0.0;
    for (int64_t e = threadIdx.x; e < nb; e += kThreads) wb[s.b_off + e] = 0.0;
  }
}

// Where element e of an output block starts in a contribution: its rest dims' part.
struct TraceIndex {
  int idx[kMaxCopyDims];
  __device__ __forceinline__ void start(const TraceOut &o, int e) {
#pragma unroll
    for (int i = kMaxCopyDims - 1; i >= 0; i--)
      if (i < o.nrd) {
        idx[i] = e % o.rext[i];
        e /= o.rext[i];
      }
  }
  __device__ __forceinline__ int64_t base(const TraceOut &o, const TraceContrib &tc) const {
    int64_t off = tc.src_off;
#pragma unroll
    for (int i = 0; i < kMaxCopyDims; i++)
      if (i < o.nrd) off += (int64_t)idx[i] * tc.rstr[i];
    return off;
  }
};

// sum + the diagonal terms [t, end) of a contribution whose element starts at base.
__device__ __forceinline__ double trace_terms(const TraceContrib &tc, const double *src, int64_t base, int64_t t,
                                              int64_t end, double sum) {
  if (tc.ndiag == 1) {   // one pair: the terms lie a constant stride apart
    const int64_t st = tc.dstr[0];
    const double *q = src + base + t * st;
#pragma unroll 8
    for (; t < end; t++, q += st) sum += *q;
    return sum;
  }
  for (; t < end; t++) {
    int rem = (int)t;
    int64_t off = base;
    for (int k = tc.ndiag - 1; k >= 0; k--) {
      const int dk = rem % tc.dext[k];
      rem /= tc.dext[k];
      off += (int64_t)dk * tc.dstr[k];
    }
    sum += src[off];
  }
  return sum;
}

// Trace with few terms per output element (trace_flat): a thread per element, which sums its
// terms in order, kTraceFlatElems of them per CTA. Bound by the loads' latency, or HBM on large
// outputs: 3.2e6 elements of one term 35 us, 1070 us with the kernel below, 65 us with a CTA
// per output block.
__global__ void __launch_bounds__(kTraceFlatElems) trace_flat_kernel(const TraceChunk *__restrict__ chunks,
                                                                       const TraceOut *__restrict__ outs,
                                                                       const TraceContrib *__restrict__ contribs,
                                                                       const double *src, double *__restrict__ dst) {
  after_previous_kernel();
  const TraceChunk ch = chunks[blockIdx.x];
  const TraceOut &o = outs[ch.out];
  const int e = threadIdx.x;
  if (e >= o.nrest - ch.e0) return;
  TraceIndex ix;
  ix.start(o, ch.e0 + e);
  double sum = 0.0;
  for (int c = 0; c < o.ncontrib; c++) {
    const TraceContrib &tc = contribs[o.first + c];
    const int64_t terms = (c + 1 < o.ncontrib ? contribs[o.first + c + 1].term0 : o.nterms) - tc.term0;
    sum = trace_terms(tc, src, ix.base(o, tc), 0, terms, sum);
  }
  dst[o.dst_off + ch.e0 + e] = sum;
}

// Trace: a CTA takes kTraceElems elements of one output block. Its threads are
// `wide` lanes over the elements (32, or the power of two that holds a smaller
// block) times kTraceThreads / wide workers, each summing an equal contiguous share
// of the block's terms (the diagonal elements of its contributing blocks in order);
// the workers' sums are added in a fixed order, so repeated calls give the same
// bits. Latency-bound: the terms are single elements far apart in memory, so the
// time is a thread's chain of loads, eight in flight, and before them its search through
// the contributions, which are read into shared memory together when they fit. The D =
// 16 environment's partial trace (61 output blocks, about 256 terms each): 769 us with a
// thread per output element and a CTA per block, 24 us with the terms over 512 threads,
// 17 us with the contributions in shared memory.
constexpr int kTraceThreads = 512;
constexpr int kTraceStage = 64;   // contributions kept in shared memory

__global__ void __launch_bounds__(kTraceThreads) trace_kernel(const TraceChunk *__restrict__ chunks,
                                                              const TraceOut *__restrict__ outs,
                                                              const TraceContrib *__restrict__ contribs,
                                                              const double *src,
                                                              double *__restrict__ dst) {
  __shared__ double part[kTraceThreads];
  __shared__ TraceContrib staged[kTraceStage];
  after_previous_kernel();
  const TraceChunk ch = chunks[blockIdx.x];
  const TraceOut &o = outs[ch.out];
  const TraceContrib *cs = contribs + o.first;
  if (o.ncontrib <= kTraceStage) {
    const int64_t *from = reinterpret_cast<const int64_t *>(cs);
    for (int w = threadIdx.x; w < o.ncontrib * (int)(sizeof(TraceContrib) / 8); w += kTraceThreads)
      reinterpret_cast<int64_t *>(staged)[w] = from[w];
    cs = staged;
    __syncthreads();
  }
  const int ne = min(kTraceElems, o.nrest - ch.e0);
  int wide = kTraceElems;
  while (wide / 2 >= ne) wide >>= 1;
  const int lane = threadIdx.x & (wide - 1), worker = threadIdx.x / wide, nworkers = kTraceThreads / wide;
  double sum = 0.0;
  if (lane < ne) {
    const int64_t nterms = o.nterms;
    const int64_t t0 = nterms * worker / nworkers, t1 = nterms * (worker + 1) / nworkers;
    if (t0 < t1) {
      TraceIndex ix;
      ix.start(o, ch.e0 + lane);
      // first contribution: the last one whose terms start at or before t0
      int lo = 0, hi = o.ncontrib - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cs[mid].term0 <= t0) lo = mid;
        else hi = mid - 1;
      }
      int64_t t = t0;
      for (int c = lo; t < t1; c++) {
        const TraceContrib &tc = cs[c];
        const int64_t end = c + 1 < o.ncontrib ? min(t1, cs[c + 1].term0) : t1;
        sum = trace_terms(tc, src, ix.base(o, tc), t - tc.term0, end - tc.term0, sum);
        t = end;
      }
    }
  }
  part[threadIdx.x] = sum;
  __syncthreads();
  // the workers' sums, halved in a fixed tree
  for (int h = nworkers / 2; h > 0; h >>= 1) {
    if (worker < h) part[worker * wide + lane] += part[(worker + h) * wide + lane];
    __syncthreads();
  }
  if (worker == 0 && lane < ne) dst[o.dst_off + ch.e0 + lane] = part[lane];
}

// x with -0 as +0, as a sum that starts from +0 gives it (an FP64 addition more per element
// cost 1 us of the 10 of the D = 8 run's scatter).
__device__ __forceinline__ double plus_zero(double x) {
  const long long b = __double_as_longlong(x);
  return __longlong_as_double(b == (long long)kSignBit ? 0ll : b);
}

// Scatter-combine of a complex product: the doubled real C_q holds the four
// real products in quadrants; a CTA writes kCScatterElems elements of one C block,
// re = P00 - P11 and im = P01 + P10 (absent quadrants, from a real operand, count as
// zero), as interleaved complex elements. HBM-bound: 32 bytes read and 16 written
// per element; reads run along rows of C_q, writes are consecutive 16-byte pairs,
// four elements (sixteen loads) in flight per thread. One CTA per block with a
// division per dim took 428 us on 489 blocks of 1500 elements on average (most of
// the GPU idle behind the largest blocks); chunks of 1024 take 9.8 us.
__global__ void __launch_bounds__(256) cscatter_kernel(const CScatterJob *__restrict__ jobs,
                                                       const CScatterChunk *__restrict__ chunks,
                                                       const double *P, double *__restrict__ C) {
  after_previous_kernel();
  const CScatterChunk ch = chunks[blockIdx.x];
  const CScatterJob J = jobs[ch.job];
  double2 *out = reinterpret_cast<double2 *>(C) + J.dst;
  const double *src = P + J.src;
  const bool h01 = J.q01 >= 0, h10 = J.q10 >= 0, h11 = J.q11 >= 0;
  constexpr int kPer = kCScatterElems / 256;
  double r0[kPer], r1[kPer], i0[kPer], i1[kPer];
#pragma unroll
  for (int u = 0; u < kPer; u++) {
    const uint32_t e = (uint32_t)ch.e0 + threadIdx.x + 256 * u;
    const bool in = e < (uint32_t)J.n;
    const uint32_t i = (e + __umulhi(e, J.mag)) >> J.shf, j = e - i * (uint32_t)J.nj;
    const double *p = src + (int64_t)i * J.ld + j;
    r0[u] = in ? p[0] : 0.0;
    r1[u] = in && h11 ? p[J.q11] : 0.0;
    i0[u] = in && h01 ? p[J.q01] : 0.0;
    i1[u] = in && h10 ? p[J.q10] : 0.0;
  }
#pragma unroll
  for (int u = 0; u < kPer; u++) {
    const uint32_t e = (uint32_t)ch.e0 + threadIdx.x + 256 * u;
    if (e < (uint32_t)J.n) out[e] = make_double2(r0[u] - r1[u], plus_zero(i0[u] + i1[u]));
  }
}

}  // namespace

cudaError_t launch_cscatter(const CScatterJob *jobs, const CScatterChunk *chunks, int64_t nchunks, const double *wc,
                            double *c, cudaStream_t stream) {
  if (nchunks <= 0) return cudaSuccess;
  if (nchunks > INT32_MAX) return cudaErrorInvalidValue;
  return launch_chained(cscatter_kernel, (unsigned)nchunks, 256, 0, stream, jobs, chunks, wc, c);
}

cudaError_t launch_copy(const CopyJob *jobs, const CopyItem *items, int64_t first, int64_t nitems, const double *src,
                        double *dst, const double *src2, double *dst2, cudaStream_t stream, int max_nd) {
  if (nitems <= 0) return cudaSuccess;
  if (nitems > INT32_MAX || max_nd < 1 || max_nd > kMaxCopyDims) return cudaErrorInvalidValue;
  return launch_chained(max_nd <= 4 ? copy_kernel<4> : copy_kernel<kMaxCopyDims>, (unsigned)nitems, kThreads, 0, stream,
                        jobs, items, (unsigned)first, src, dst, src2, dst2);
}

cudaError_t launch_trace(const TraceChunk *chunks, int64_t nsplit, int64_t nflat, const TraceOut *outs,
                         const TraceContrib *contribs, const double *src, double *dst, cudaStream_t stream) {
  if (nsplit > INT32_MAX || nflat > INT32_MAX) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  if (nsplit > 0)
    e = launch_chained(trace_kernel, (unsigned)nsplit, kTraceThreads, 0, stream, chunks, outs, contribs, src, dst);
  if (e == cudaSuccess && nflat > 0)
    e = launch_chained(trace_flat_kernel, (unsigned)nflat, kTraceFlatElems, 0, stream, chunks + nsplit, outs, contribs,
                       src, dst);
  return e;
}

cudaError_t launch_gather_flagged(const CopyJob *jobs, const CopyItem *items_a, const CopyItem *items_b,
                                  const SplitSector *sp_sectors, const SectorDev *sectors, const int32_t *flagged,
                                  const int32_t *item_end_a, const int32_t *item_end_b, const SplitRecord *rec,
                                  const double *a, const double *b, double *wa, double *wb, bool zero_a, bool zero_b,
                                  int num_sms, cudaStream_t stream) {
  const unsigned grid = (unsigned)std::max(1, num_sms) * 4;
  cudaError_t e = cudaSuccess;
  if (zero_a || zero_b)
    e = launch_chained(zero_flagged_kernel, grid, kThreads, 0, stream, sectors, flagged, rec, wa, wb, (int)zero_a,
                       (int)zero_b);
  if (e == cudaSuccess)
    e = launch_chained(copy_flagged_kernel, grid, kThreads, 0, stream, jobs, sp_sectors, flagged, rec,
                       FlaggedGather{items_a, item_end_a, a, wa}, FlaggedGather{items_b, item_end_b, b, wb});
  return e;
}

}  // namespace ytn
