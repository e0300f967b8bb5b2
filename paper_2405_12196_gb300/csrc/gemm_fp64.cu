// Grouped FP64 GEMM over the charge sectors of a contraction (Sec. II.B: the
// fused matrices are multiplied sector by sector, C_q = A_q B_q), on the FP64
// tensor cores (DMMA, mma.sync m8n8k4 f64).
//
// One launch covers every sector: the grid is the host-built tile list
// (sector, m-tile, n-tile), largest tiles first so that long ones start early.
// Each CTA computes one tile of C_q over the full K (no split-K), so every
// output element has one fixed summation order: results do not depend on the
// schedule, the tile edge or on what else runs on the GPU. The tile edge (64, 32 or
// 16) is chosen per sector by the planner so that the work spreads over the SMs.
//
// On GB300 the FP64 rate (DMMA and DFMA alike, about 1 TFLOP/s for the whole GPU: two
// multiply-adds per clock and SM) is low enough that this kernel is bound by the FP64
// pipe at every tile edge; operands are staged through padded shared memory with a
// register prefetch of the next K step. So no padding is multiplied: DMMA blocks
// outside the sector are skipped, K advances in steps of 4 to its end, and sectors
// with K <= 2 (double layers contracted over a physical leg: one element per charge)
// take plain multiply-adds, one per K, instead of a DMMA step of 4. The Z2 D = 8
// double layer (2 sectors of 2048 x 2048 x 1) took 260 us with K padded to 16 and
// takes 38 us (gemm_outer_kernel).
//
// The epilogue writes C's blocks directly through the planner's row, column and block
// tables (OutView), or the dense C_q of the workspace when a scatter follows.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.hpp"

namespace ytn {

namespace {

constexpr int BK = 16, PAD = 4;
constexpr int kThreads = 128;

__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}

// Load one BK-slice of the A (or B) tile into registers: T x 16 elements, T/8 per
// thread. kmajor: element (r, k) at base[r * ld + k]; else at base[k * ld + r].
template <int T>
__device__ __forceinline__ void load_tile(double (&v)[T / 8], const double *base, int ld, bool kmajor,
                                          int rows, int r0, int k0, int K) {
  const int t = threadIdx.x;
  if (kmajor) {
    const int k = t & 15;
#pragma unroll
    for (int i = 0; i < T / 8; i++) {
      const int r = (t >> 4) + 8 * i;
      const int gr = r0 + r, gk = k0 + k;
      v[i] = (gr < rows && gk < K) ? base[(int64_t)gr * ld + gk] : 0.0;
    }
  } else {
    const int r = t & (T - 1);
#pragma unroll
    for (int i = 0; i < T / 8; i++) {
      const int k = t / T + (kThreads / T) * i;
      const int gr = r0 + r, gk = k0 + k;
      v[i] = (gr < rows && gk < K) ? base[(int64_t)gk * ld + gr] : 0.0;
    }
  }
}

template <int T>
__device__ __forceinline__ void store_tile(double (*s)[64 + PAD], const double (&v)[T / 8], bool kmajor) {
  const int t = threadIdx.x;
  if (kmajor) {
    const int k = t & 15;
#pragma unroll
    for (int i = 0; i < T / 8; i++) s[k][(t >> 4) + 8 * i] = v[i];
  } else {
    const int r = t & (T - 1);
#pragma unroll
    for (int i = 0; i < T / 8; i++) s[t / T + (kThreads / T) * i][r] = v[i];
  }
}

// A warp's accumulators (8 x 8 DMMA blocks; the thread's elements are rows m + 8 i,
// columns n + 8 j and the next one) into C.
template <int NB>
__device__ __forceinline__ void store_tile_out(const SectorDev &s, int sector, const OutView &out,
                                               const double (&acc)[NB][NB][2], int m, int n) {
  if (!out.sec) {   // the dense C_q
    double *C = out.c + s.c_off;
#pragma unroll
    for (int i = 0; i < NB; i++) {
      if (m + 8 * i >= s.M) continue;
      double *row = C + (int64_t)(m + 8 * i) * s.N;
#pragma unroll
      for (int j = 0; j < NB; j++)
#pragma unroll
        for (int h = 0; h < 2; h++)
          if (n + 8 * j + h < s.N) row[n + 8 * j + h] = acc[i][j][h];
    }
    return;
  }
  const SectorOut so = out.sec[sector];
  OutCol col[NB][2];
#pragma unroll
  for (int j = 0; j < NB; j++)
#pragma unroll
    for (int h = 0; h < 2; h++)
      if (n + 8 * j + h < s.N) col[j][h] = out.cols[so.cols + n + 8 * j + h];
#pragma unroll
  for (int i = 0; i < NB; i++) {
    if (m + 8 * i >= s.M) continue;
    const OutRow row = out.rows[so.rows + m + 8 * i];
    const int64_t *base = out.base + so.base + (int64_t)row.blk * so.ncb;
#pragma unroll
    for (int j = 0; j < NB; j++)
#pragma unroll
      for (int h = 0; h < 2; h++)
        if (n + 8 * j + h < s.N) {
          const int64_t b = __ldg(base + col[j][h].blk);
          if (b >= 0) out.c[b + (int64_t)row.idx * col[j][h].len + col[j][h].idx] = acc[i][j][h];
        }
  }
}

// One T x T tile of C_q (T = 64, 32 or 16): four warps of (T/2) x (T/2), each a grid
// of (T/16) x (T/16) DMMA 8x8 blocks.
template <int T>
__device__ __forceinline__ void gemm_tile(const SectorDev &s, const GemmTile &tl, const double *wa,
                                          const double *wb, const OutView &out,
                                          double (*As)[BK][64 + PAD], double (*Bs)[BK][64 + PAD]) {
  constexpr int NB = T / 16;
  const int M = s.M, N = s.N, K = s.K;
  const int m0 = tl.mt * T, n0 = tl.nt * T;
  const double *A = wa + s.a_off;
  const double *B = wb + s.b_off;
  const int lda = s.a_kmajor ? K : M;
  const int ldb = s.b_kmajor ? K : N;
  const bool akm = s.a_kmajor != 0, bkm = s.b_kmajor != 0;

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp >> 1) * (T / 2), wn = (warp & 1) * (T / 2);
  double acc[NB][NB][2];
#pragma unroll
  for (int i = 0; i < NB; i++)
#pragma unroll
    for (int j = 0; j < NB; j++) acc[i][j][0] = acc[i][j][1] = 0.0;

  // DMMA blocks of this warp that meet the sector (the same for the whole warp)
  const int nbm = (M - m0 - wm + 7) >> 3, nbn = (N - n0 - wn + 7) >> 3;
  double ra[T / 8], rb[T / 8];
  const int nk = (K + BK - 1) / BK;
  if (nk > 0) {
    load_tile<T>(ra, A, lda, akm, M, m0, 0, K);
    load_tile<T>(rb, B, ldb, bkm, N, n0, 0, K);
    store_tile<T>(As[0], ra, akm);
    store_tile<T>(Bs[0], rb, bkm);
  }
  __syncthreads();
  for (int kt = 0; kt < nk; kt++) {
    const int cur = kt & 1;
    const bool more = kt + 1 < nk;
    if (more) {
      load_tile<T>(ra, A, lda, akm, M, m0, (kt + 1) * BK, K);
      load_tile<T>(rb, B, ldb, bkm, N, n0, (kt + 1) * BK, K);
    }
    const int kend = min(BK, K - kt * BK);   // steps of 4 beyond K hold zeros only
#pragma unroll
    for (int kk = 0; kk < BK; kk += 4) {
      if (kk >= kend) break;
      double af[NB], bf[NB];
#pragma unroll
      for (int i = 0; i < NB; i++) af[i] = As[cur][kk + (lane & 3)][wm + i * 8 + (lane >> 2)];
#pragma unroll
      for (int j = 0; j < NB; j++) bf[j] = Bs[cur][kk + (lane & 3)][wn + j * 8 + (lane >> 2)];
#pragma unroll
      for (int i = 0; i < NB; i++)
#pragma unroll
        for (int j = 0; j < NB; j++)
          if (i < nbm && j < nbn) dmma(acc[i][j], af[i], bf[j]);
    }
    if (more) {
      store_tile<T>(As[cur ^ 1], ra, akm);
      store_tile<T>(Bs[cur ^ 1], rb, bkm);
    }
    __syncthreads();
  }
  store_tile_out<NB>(s, tl.sector, out, acc, m0 + wm + (lane >> 2), n0 + wn + 2 * (lane & 3));
}

// Sectors with K <= 2: one tile of 64 rows x COLS columns by 2 COLS threads, thread t the
// rows of its half (t / COLS, every second one) at column t % COLS, so that the stores of
// a warp run along the columns. The products are summed in the order of k, as the DMMA
// steps do.
constexpr int kOuterK = 2;

template <int COLS>
__device__ __forceinline__ void outer_tile(const SectorDev &s, const GemmTile &tl, const double *wa,
                                           const double *wb, const OutView &out, double (*As)[64],
                                           OutRow *rows) {
  const int M = s.M, N = s.N, K = s.K, t = threadIdx.x;
  const int m0 = tl.mt * 64, n = tl.nt * COLS + (t & (COLS - 1));
  const int nr = min(64, M - m0);
  const bool direct = out.sec != nullptr;
  const SectorOut so = direct ? out.sec[tl.sector] : SectorOut{};
  for (int e = t; e < nr * K; e += 2 * COLS) {
    const int r = e / K, k = e - r * K;
    As[k][r] = wa[s.a_off + (s.a_kmajor ? (int64_t)(m0 + r) * K + k : (int64_t)k * M + m0 + r)];
  }
  if (t < nr) rows[t] = direct ? out.rows[so.rows + m0 + t] : OutRow{0, m0 + t};
  double b[kOuterK];
  OutCol col{0, n, N, 0};
  if (n < N) {
#pragma unroll
    for (int k = 0; k < kOuterK; k++)
      b[k] = k < K ? wb[s.b_off + (s.b_kmajor ? (int64_t)n * K + k : (int64_t)k * N + n)] : 0.0;
    if (direct) col = out.cols[so.cols + n];
  }
  __syncthreads();
  if (n >= N) return;
  int blk = direct ? -1 : 0;
  int64_t base = s.c_off;
#pragma unroll 4
  for (int r = t / COLS; r < nr; r += 2) {
    const OutRow row = rows[r];
    if (row.blk != blk) {
      blk = row.blk;
      base = __ldg(out.base + so.base + (int64_t)blk * so.ncb + col.blk);
    }
    double v = fma(As[0][r], b[0], 0.0);   // a sum from +0, as the DMMA steps': no -0 from a zero factor
    if (K > 1) v = fma(As[1][r], b[1], v);
    if (base >= 0) out.c[base + (int64_t)row.idx * col.len + col.idx] = v;
  }
}

// Plans of such sectors only (tiles of 64 x 128, 128 the tile's size). The Z2 D = 8 double
// layer (8.4e6 elements, 67 MB) takes 38 us, 50 us as 64 x 64 tiles among the DMMA kernel's.
// Neither the FP64 multiplications (16 clocks a warp and SM: 14 us) nor the stores (10 us at
// the copy peak) bound it: 48 registers let five CTAs share an SM, so that its 1024 CTAs
// are 1.35 waves, and each begins with a chain of loads (tile, sector, tables, operands).
__global__ void __launch_bounds__(256) gemm_outer_kernel(const SectorDev *__restrict__ sectors,
                                                         const GemmTile *__restrict__ tiles,
                                                         const double *wa, const double *wb, OutView out) {
  __shared__ double As[kOuterK][64];
  __shared__ OutRow rows[64];
  after_previous_kernel();
  const GemmTile tl = tiles[blockIdx.x];
  const SectorDev s = sectors[tl.sector];
  outer_tile<128>(s, tl, wa, wb, out, As, rows);
}

__global__ void __launch_bounds__(kThreads) gemm_fp64_kernel(const SectorDev *__restrict__ sectors,
                                                             const GemmTile *__restrict__ tiles,
                                                             const double *wa,
                                                             const double *wb, OutView out) {
  __shared__ double As[2][BK][64 + PAD];
  __shared__ double Bs[2][BK][64 + PAD];
  after_previous_kernel();
  const GemmTile tl = tiles[blockIdx.x];
  const SectorDev s = sectors[tl.sector];
  if (tl.size == 16) gemm_tile<16>(s, tl, wa, wb, out, As, Bs);
  else if (tl.size == 32) gemm_tile<32>(s, tl, wa, wb, out, As, Bs);
  else if (s.K <= kOuterK)
    outer_tile<64>(s, tl, wa, wb, out, reinterpret_cast<double(*)[64]>(&As[0][0][0]),
               reinterpret_cast<OutRow *>(&Bs[0][0][0]));
  else gemm_tile<64>(s, tl, wa, wb, out, As, Bs);
}

// FP64 recomputation of the sectors that the split path's accuracy check
// flagged: a persistent grid walks the flagged sectors' 64 x 64 tiles, whose list
// the check wrote on the device (tile_end: running tile counts per flagged
// sector). With no flagged sector every CTA returns at once.
__global__ void __launch_bounds__(kThreads) gemm_fp64_redo_kernel(const SectorDev *__restrict__ sectors,
                                                                  const int32_t *flagged,
                                                                  const int32_t *tile_end,
                                                                  const SplitRecord *rec,
                                                                  const double *wa,
                                                                  const double *wb, OutView out) {
  __shared__ double As[2][BK][64 + PAD];
  __shared__ double Bs[2][BK][64 + PAD];
  after_previous_kernel();
  const int nflag = rec->nfallback;
  if (nflag <= 0) return;
  const int total = tile_end[nflag - 1];
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    int lo = 0, hi = nflag - 1;   // first flagged sector whose tiles end after t
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (tile_end[mid] > t) hi = mid;
      else lo = mid + 1;
    }
    const int local = t - (lo > 0 ? tile_end[lo - 1] : 0);
    const SectorDev s = sectors[flagged[lo]];
    const int nt = (s.N + 63) / 64;
    const GemmTile tl{flagged[lo], local / nt, local % nt, 64};
    gemm_tile<64>(s, tl, wa, wb, out, As, Bs);
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_gemm_fp64_redo(const SectorDev *sectors, const int32_t *flagged, const int32_t *tile_end,
                                  const SplitRecord *rec, const double *wa, const double *wb, const OutView &out,
                                  int num_sms, cudaStream_t stream) {
  return launch_chained(gemm_fp64_redo_kernel, (unsigned)std::max(1, num_sms) * 4, kThreads, 0, stream, sectors, flagged,
                        tile_end, rec, wa, wb, out);
}

cudaError_t launch_gemm_fp64(const SectorDev *sectors, const GemmTile *tiles, int64_t ntiles,
                             const double *wa, const double *wb, const OutView &out, bool outer, cudaStream_t stream) {
  if (ntiles <= 0) return cudaSuccess;
  if (ntiles > INT32_MAX) return cudaErrorInvalidValue;
  if (outer) return launch_chained(gemm_outer_kernel, (unsigned)ntiles, 256, 0, stream, sectors, tiles, wa, wb, out);
  return launch_chained(gemm_fp64_kernel, (unsigned)ntiles, kThreads, 0, stream, sectors, tiles, wa, wb, out);
}

}  // namespace ytn
