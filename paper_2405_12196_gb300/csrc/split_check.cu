// Accuracy check of the split-precision products, with its FP64 fallback.
//
// The split GEMM rounds each operand row (a row of A_q, a column of B_q) to the
// digits kept at its power-of-two scale 2^e, drops the digit products of order
// >= s and rounds the FP32 accumulator of the orders >= 3. Every one of these
// errors is a small multiple of the product of the two scales, 2^(e_i + f_j),
// per element of C_q, and grows like sqrt(K) over the contraction (independent
// roundings). So the absolute error of C_q is estimated, per element, by
// eta sqrt(K) 2^(e_i + f_j), and its relative Frobenius error by
//     est_q = eta sqrt(K_q sum_i 4^(e_i) sum_j 4^(f_j)) / ||C_q||_F,
// which sees the data through the scales and the result: when a row holds one
// large element and the rest far below it, or when the products cancel, the
// scales are large against |c_ij| and the estimate grows with that ratio.
//
// A CTA sums the scales of kCheckRows rows of one sector's operands (both taken relative
// to the operands' largest exponents, so nothing overflows): FP64 additions are slow on
// this GPU, two a clock and SM, so the rows of a large sector are shared out (one CTA
// per sector took 83 us for two sectors of 133,000 rows and columns). The sums are added
// in a fixed order, within a CTA and over a sector's CTAs. The last CTA to
// finish, from these and the ||C_q||^2 that the GEMM epilogue summed, with one division
// per sector and the lists only when a sector is flagged (a chain of latencies: square
// roots and four prefix sums per sector made it 17 to 24 us, now 13 to 14):
//   - lists the sectors with est_q > rtol, in sector order, with the running
//     counts of their 64 x 64 tiles and of their gather work items (the FP64
//     recomputation reads these lists);
//   - writes the call's record: the relative error of the whole result before
//     and after the fallback (sectors weighted by their norms), the largest
//     per-sector estimate, the number of recomputed sectors and their FLOPs;
//   - raises the tolerance flag in the context's status word when even the
//     result after the fallback is estimated above rtol.
// Everything runs on the device, so a call stays asynchronous and can be
// recorded into a graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include "kernels.hpp"

namespace ytn {

namespace {

constexpr int kThreads = 256;

// 4^k for k <= 0 as an FP64 value built from its bits (0 below the normal range).
__device__ __forceinline__ double pow4(int k) {
  return k >= -511 ? __longlong_as_double((long long)(1023 + 2 * k) << 52) : 0.0;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The warp's sums of a (in lanes 0..15) and b (in lanes 16..31), with half the additions of
// two sums: an FP64 addition takes a warp 16 clocks of the SM's FP64 pipe.
__device__ __forceinline__ double warp_sum2(double a, double b) {
  const bool upper = (threadIdx.x & 16) != 0;
  double v = upper ? b : a;
  v += __shfl_xor_sync(0xffffffffu, upper ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// This thread's share of the sum of 4^(e[i] - E) over rows [lo, hi).
__device__ __forceinline__ double scale_sum(const int32_t *e, uint32_t lo, uint32_t hi, int E) {
  double s = 0.0;
  uint32_t i = lo + 4 * threadIdx.x;
#pragma unroll 4
  for (; i + 4 <= hi; i += 4 * kThreads) {   // rows start on multiples of 128
    const int4 x = *reinterpret_cast<const int4 *>(e + i);
    s += (pow4(x.x - E) + pow4(x.y - E)) + (pow4(x.z - E) + pow4(x.w - E));
  }
  for (; i < hi; i++) s += pow4(e[i] - E);   // the one thread whose four rows meet hi
  return s;
}

// Exclusive prefix sum over the block (one value per thread); returns the
// thread's offset and the block total in *total.
__device__ __forceinline__ int block_scan(int v, int *red, int *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) red[warp] = x;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; w++) {
    if (w < warp) before += red[w];
    all += red[w];
  }
  *total = all;
  return before + x - v;
}

__global__ void __launch_bounds__(kThreads) split_check_kernel(
    const SplitSector *__restrict__ sectors, int nsec, const SplitCheckChunk *__restrict__ chunks,
    const int32_t *ea, const int32_t *eb, const int32_t *emax, const float *normsq, double *secv,
    int32_t *__restrict__ flagged, int32_t *__restrict__ tile_end, int32_t *__restrict__ item_end_a,
    int32_t *__restrict__ item_end_b, SplitRecord *rec, double eta_split, double eta_fp64, double rtol, int slices,
    int *status) {
  __shared__ double dred[4][kThreads / 32];
  __shared__ int ired[kThreads / 32];
  __shared__ int is_last;
  after_previous_kernel();
  // a chunk per sector: the tables need no look (0.5 us on the D = 10 run)
  const bool single = nsec == (int)gridDim.x;
  const SplitCheckChunk ch = single ? SplitCheckChunk{(int)blockIdx.x, 0} : chunks[blockIdx.x];
  const int q = ch.sector, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  {
    const SplitSector sc = sectors[q];
    // rows of A, then of B from align4(M) on
    const int64_t lo = (int64_t)ch.idx * kCheckRows, hi = lo + kCheckRows, mb = ((int64_t)sc.M + 3) & ~(int64_t)3;
    double se = 0.0, sf = 0.0;
    if (lo < sc.M) se = scale_sum(ea + sc.ea_off, lo, min((int64_t)sc.M, hi), emax[2 * q]);
    if (hi > mb && lo - mb < sc.N)
      sf = scale_sum(eb + sc.eb_off, max((int64_t)0, lo - mb), min((int64_t)sc.N, hi - mb), emax[2 * q + 1]);
    const double v = warp_sum2(se, sf);
    if ((lane & 15) == 0) dred[lane >> 4][warp] = v;
    __syncthreads();
  }
  // the last CTA to get here sees every sector's sums (one thread writes and fences: all
  // 256 of them fencing took 0.8 us more on the D = 9 environment)
  if (tid == 0) {
    double se = 0.0, sf = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; w++) {
      se += dred[0][w];
      sf += dred[1][w];
    }
    *reinterpret_cast<double2 *>(secv + 2 * (int64_t)blockIdx.x) = make_double2(se, sf);
    __threadfence();
    is_last = atomicAdd(&rec->done_blocks, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();

  // the sums of sectors of several chunks into their first chunk's place, a warp per sector
  if (!single) {
    for (int base = 32 * warp; base < nsec; base += kThreads) {
      int c0 = 0, n = 0;
      if (base + lane < nsec) {
        c0 = sectors[base + lane].chk0;
        n = sectors[base + lane].chk1 - c0;
      }
      for (uint32_t many = __ballot_sync(0xffffffffu, n > 1); many; many &= many - 1) {
        const int b = __ffs(many) - 1;
        const int from = __shfl_sync(0xffffffffu, c0, b), to = from + __shfl_sync(0xffffffffu, n, b);
        double se = 0.0, sf = 0.0;
        for (int c = from + lane; c < to; c += 32) {
          se += __ldcg(secv + 2 * c);
          sf += __ldcg(secv + 2 * c + 1);
        }
        const double v = warp_sum2(se, sf);
        if ((lane & 15) == 0) __stcg(secv + 2 * from + (lane >> 4), v);
      }
    }
    __syncthreads();
  }
  // K_q sum_i 4^(e_i - emax_A) sum_j 4^(f_j - emax_B): 0 for a zero operand
  auto value = [&](int s) {
    if (emax[2 * s] <= 0 || emax[2 * s + 1] <= 0) return 0.0;
    const double *v = secv + 2 * (single ? s : sectors[s].chk0);
    return (double)sectors[s].K * __ldcg(v) * __ldcg(v + 1);
  };
  // reference exponent: the largest emax_A + emax_B among sectors with data
  int g = INT_MIN;
  for (int s = tid; s < nsec; s += kThreads)
    if (normsq[s] > 0.0f || value(s) > 0.0) g = max(g, emax[2 * s] + emax[2 * s + 1]);
  g = __reduce_max_sync(0xffffffffu, g);
  if (lane == 0) ired[warp] = g;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kThreads / 32; w++) g = max(g, ired[w]);
  const double split2 = eta_split * eta_split, after2 = eta_fp64 * eta_fp64, limit = rtol * rtol;
  double norm = 0.0, err_split = 0.0, err_after = 0.0, worst = 0.0;   // squares
  int nflag = 0, ntile = 0, nia = 0, nib = 0;
  for (int base = 0; base < nsec; base += kThreads) {
    const int s = base + tid;
    int flag = 0;
    if (s < nsec) {
      const double v = value(s), n2 = (double)normsq[s];
      double est = 0.0;   // squared
      if (v > 0.0) est = n2 > 0.0 ? split2 * (v / n2) : INFINITY;
      flag = est > limit;
      worst = fmax(worst, est);
      if (g != INT_MIN) {
        const double w = pow4(emax[2 * s] + emax[2 * s + 1] - g);
        norm += n2 * w;
        err_split += split2 * v * w;
        err_after += (flag ? after2 : split2) * v * w;
      }
    }
    if (!__syncthreads_or(flag)) continue;
    // the lists of the FP64 recomputation
    int tiles = 0, ia = 0, ib = 0;
    if (flag) {
      const SplitSector t = sectors[s];
      tiles = ((t.M + 63) / 64) * ((t.N + 63) / 64);
      ia = t.ga1 - t.ga0;
      ib = t.gb1 - t.gb0;
      atomicAdd(&rec->fallback_flops, 2.0 * (double)t.M * (double)t.N * (double)t.K);
    }
    int total_flag, total_tiles, total_ia, total_ib;
    const int pos = block_scan(flag, ired, &total_flag);
    const int tpos = block_scan(tiles, ired, &total_tiles);
    const int apos = block_scan(ia, ired, &total_ia);
    const int bpos = block_scan(ib, ired, &total_ib);
    if (flag) {
      flagged[nflag + pos] = s;
      tile_end[nflag + pos] = ntile + tpos + tiles;
      item_end_a[nflag + pos] = nia + apos + ia;
      item_end_b[nflag + pos] = nib + bpos + ib;
    }
    nflag += total_flag;
    ntile += total_tiles;
    nia += total_ia;
    nib += total_ib;
  }
  if (32 * warp < nsec) {   // the others looked at no sector
    norm = warp_sum(norm);
    err_split = warp_sum(err_split);
    err_after = warp_sum(err_after);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  }
  if (lane == 0) {
    dred[0][warp] = norm;
    dred[1][warp] = err_split;
    dred[2][warp] = err_after;
    dred[3][warp] = worst;
  }
  __syncthreads();
  if (tid == 0) {
    norm = err_split = err_after = worst = 0.0;
    for (int w = 0; w < kThreads / 32; w++) {
      norm += dred[0][w];
      err_split += dred[1][w];
      err_after += dred[2][w];
      worst = fmax(worst, dred[3][w]);
    }
    auto rel = [&](double e2) { return e2 > 0.0 ? (norm > 0.0 ? sqrt(e2 / norm) : INFINITY) : 0.0; };
    const double after = rel(err_after);
    rec->err_est = after;
    rec->split_err_est = rel(err_split);
    rec->max_sector_est = sqrt(worst);
    rec->rtol = rtol;
    rec->nsectors = nsec;
    rec->nfallback = nflag;
    rec->within = after <= rtol;
    rec->slices = slices;
    __threadfence();
    rec->valid = 1;
    if (!(after <= rtol)) atomicCAS(status + 1, 0, 1);
  }
}

}  // namespace

cudaError_t launch_split_check(const SplitSector *sectors, int64_t nsec, const SplitCheckChunk *chunks,
                               int64_t nchunks, const int32_t *ea, const int32_t *eb, const int32_t *emax,
                               const float *normsq, double *secv, int32_t *flagged, int32_t *tile_end,
                               int32_t *item_end_a, int32_t *item_end_b, SplitRecord *rec, double eta_split,
                               double eta_fp64, double rtol, int slices, int *status, cudaStream_t stream) {
  if (nsec <= 0) return cudaSuccess;
  if (nchunks < nsec || nchunks > INT32_MAX) return cudaErrorInvalidValue;
  return launch_chained(split_check_kernel, (unsigned)nchunks, kThreads, 0, stream, sectors, (int)nsec, chunks, ea, eb,
                        emax, normsq, secv, flagged, tile_end, item_end_a, item_end_b, rec, eta_split, eta_fp64, rtol,
                        slices, status);
}

}  // namespace ytn
