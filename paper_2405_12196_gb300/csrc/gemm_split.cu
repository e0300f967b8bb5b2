// Split-precision grouped GEMM over the charge sectors of a contraction on the
// 5th-generation tensor cores (tcgen05, accumulators in tensor memory, operands
// fed by bulk TMA copies), with FP64 results.
//
// Operands are the BF16 slices written by split_kernels.cu: A_q = 2^(e_i - 8)
// sum_p A_p and B_q = 2^(f_j - 8) sum_q B_q (up to the rounding of the last digit),
// with slice p a signed digit of magnitude <= 2^7 times 2^{-8p}.
// C_q = 2^(e_i + f_j - 16) sum_{p + q <= s - 1} A_p B_q^T, where s is the number of
// slices used (products of order p + q >= s are dropped, as in the Ozaki scheme).
//
// Accumulation, per 128 x 128 output tile:
//   E2 = A_0 B_0                     order 0, exact in FP32 per K chunk of 256
//   E3 = A_0 B_1 + A_1 B_0           order 1, exact (an integer times 2^-8)
//   E4 = A_0 B_2 + A_1 B_1 + A_2 B_0 order 2, exact (an integer times 2^-16)
//   R  = every kept product of order >= 3, FP32 per K chunk of 256
// A digit product is at most 2^14 in magnitude, so over a chunk of 256 the three
// exact accumulators stay within 3 * 256 * 2^14 < 2^24 units of their lowest bit
// and FP32 holds them exactly; after each chunk the epilogue warps read all four
// from tensor memory and add them into a 64-bit fixed-point accumulator (units
// of 2^-24 of the order-0 product). Only R, about 2^-24 of the result per K, is
// rounded in FP32, and only over 256 of K at a time (the tensor cores' FP32
// accumulation of mixed-magnitude products is not round-to-nearest, so its error
// grows with the number of additions). The result is converted to FP64 and
// scaled by 2^(e_i + f_j - 40). Tensor memory: E2 [0,128), E3 [128,256),
// E4 [256,384), R [384,512).
//
// Tiles and roles. A pair of CTAs (a cluster of two, one CTA per SM, persistent over
// the host-ordered tile list) computes one 256 x 128 tile with cta_group::2 MMAs: each
// CTA holds 128 rows of the P operand and half (64 rows) of the 128-row Q operand, the
// tensor cores of both SMs read the two Q halves, and each CTA accumulates its 128 P
// rows x 128 Q rows. P is B (tensor-memory lanes are columns of C, so that the stores of
// a warp run along C's rows) and Q is A, except in the tiles of a sector with 64-wide
// column tails, where P is A and Q is B. Against one CTA per 128 x 128 tile an SM reads
// 6 KB instead of 8 KB of shared memory per 128 x 128 x 16 MMA and fetches 12 KB per
// slice and stage instead of 16 KB, which leaves room for deeper rings.
//   warp 0     (both CTAs) bulk-copy producer: per K stage of 32 the CTA's P slices and
//              its half of the Q slices into two rings (see Ring);
//   warp 1     (leader CTA) MMA issuer: M = 256, N = 128, K = 16. The exact products
//              and the R products are two queues over the stages, the exact ones' chunks
//              ending two stages before R's; the queue whose chunk ends first goes
//              ahead, as far as its ring allows, and while its accumulators are drained
//              the other one has stages left to multiply. The whole warp runs the loop
//              on uniform values, so that the MMA operands come from uniform registers,
//              and its barriers are tested with the default (CTA) scope: with
//              cluster-scope acquires a test cost 500 clocks and the issue loop, not
//              the tensor cores, set the pace;
//              (peer CTA) relays its "stage loaded" signals to the leader;
//   warps 2-17 (both CTAs) epilogue: chunk drains and the FP64 output (four warps per
//              32-lane quarter of tensor memory, 32 columns each; warp 2 also
//              allocates and frees tensor memory), whose 32 64-bit accumulators per
//              lane take most of the 96 registers that a 576-thread CTA leaves a thread
//              (the output, which needs tables and places beside them, spills 108 bytes
//              of stores and 172 of loads; with 64-wide tails 200 and 384), and writes
//              C's blocks (OutView) or the dense C_q.
// Bound by the tensor cores, and on large contractions by power. An MMA takes 64 clocks
// per SM, a stage of five slices 1920. On the D = 20 environment (15 slice products of
// 1.86e12 FLOPs) a stage took 2940 clocks with one CTA per 128 x 128 tile (18.1 ms, and
// 0.9 ms for the scatter of C) and takes 2180 (15.6 ms with C written, at 1.77 instead
// of 1.95 GHz: the power limit now takes part of the gain); D = 12 (30 GFLOP): 416 + 45
// us -> 320 us.
// Every wait is bounded; on expiry the kernel records a status code, stops
// issuing work, waits (bounded, whatever the abort flag says: mbar_drain) for its own
// copies and MMAs and frees tensor memory before returning.
#include <cuda_runtime.h>

#include "kernels.hpp"

namespace ytn {

namespace {

constexpr int kThreads = 576;     // 18 warps
constexpr int kFirstEpiWarp = 2;  // warps 2..17: epilogue
constexpr int kEpiWarps = 16;
constexpr int kHalfBytes = kSliceBytes / 2;   // a CTA's half of a Q slice
constexpr uint32_t kColE2 = 0, kColE3 = 128, kColE4 = 256, kColR = 384;
constexpr uint32_t kMaxPolls = 1u << 26;
constexpr uint32_t kDrainPolls = 1u << 18;
constexpr int kOutGroup = 8;    // rows of Q converted without a look at C's blocks in between
constexpr int kMaxStarts = 4;   // blocks of C among a warp's 32 rows with places read ahead

// Shared memory of one CTA: two rings, since the exact products read slices 0..2 of a
// stage only and the R products all of them. The lead ring holds slices 0..2 (per
// stage the P slices, then the Q halves), a slot free once both queues are past the
// stage; the rest ring slices 3..S-1, free once the R queue is. While one queue waits
// for a drain the other runs ahead by the depth of its rings: four stages in 216 KB with
// five slices, where one ring of whole stages held three (17.0 against 15.9 ms on the
// D = 20 environment).
template <int S>
struct Ring {
  static constexpr int kRest = S - 3;
  static constexpr int kLeadSlot = 3 * (kSliceBytes + kHalfBytes), kRestSlot = kRest * (kSliceBytes + kHalfBytes);
  static constexpr int kLeadStages = S == 6 ? 3 : 4, kRestStages = S == 4 ? 4 : 3;
  static constexpr int kLeadBytes = kLeadStages * kLeadSlot, kBytes = kLeadBytes + kRestStages * kRestSlot;
  static constexpr int kSmem = kBytes + 1024 + 256;
};

// The last K stage of the chunk that stage st of ks belongs to, for R (stages 7, 15, ...)
// and for the exact accumulators (E: 5, 13, ... when the tile has more than one chunk;
// where they end does not change the result); at most eight stages each, and both end at
// the last stage.
__device__ __forceinline__ int e_end(int st, int ks) { return ks > 8 ? min(((st + 2) | 7) - 2, ks - 1) : ks - 1; }
__device__ __forceinline__ int r_end(int st, int ks) { return min(st | 7, ks - 1); }

// instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major, M = 256; the
// N field (bits 17..22, N / 8) is set per tile: 128, or 64 for the narrow tiles
constexpr uint32_t kIdescBase = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 4) << 24);
__device__ __forceinline__ uint32_t idesc_for(int bn) { return kIdescBase | ((uint32_t)(bn >> 3) << 17); }

// lead ring full / empty, rest ring full / empty (up to four slots each), drains, end
enum Bar { kFull0 = 0, kEmpty0 = 4, kRestFull0 = 8, kRestEmpty0 = 12, kEFull = 16, kEEmpty, kRFull, kREmpty, kDone, kNumBars };

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The leader CTA's copy of a shared-memory location, as a cluster address.
__device__ __forceinline__ uint32_t leader_addr(uint32_t addr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Whether the phase of parity `parity` has completed (no waiting).
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Raises the abort flag of both CTAs of the pair.
__device__ __forceinline__ void abort_pair(volatile int *abort_flag) {
  const uint32_t mine = smem_u32(const_cast<int *>(abort_flag));
#pragma unroll
  for (int c = 0; c < 2; c++)
    asm volatile("{\n\t.reg .u32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.u32 [a], %2;\n\t}" ::"r"(
                     mine),
                 "r"(c), "r"(1)
                 : "memory");
}

// Bounded wait for the phase of parity `parity` to complete. Returns false (and
// records `code` in the status word and the CTA's abort flag) when the bound is
// reached or another role has aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status,
                                          int code) {
  for (uint32_t i = 0; i < kMaxPolls; i++) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 63) == 63 && *abort_flag) return false;
  }
  abort_pair(abort_flag);
  atomicCAS(status, 0, code);
  return false;
}

// A last look at a phase that mbar_wait gave up on: the bulk copies and MMAs already issued
// go on after an abort, and a CTA keeps its shared and tensor memory until they have
// ended. They end within microseconds; kDrainPolls tests take a few milliseconds (a slot
// of the leader whose peer stopped before its copy never completes: then the bound ends it).
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < kDrainPolls && !mbar_test(bar, parity); i++) {}
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// Shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512 B apart.
// Its upper word is the same for every operand; the lower one holds the address in
// 16-byte units.
constexpr uint32_t kDescHi = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | (1u << 16); }

__device__ __forceinline__ void umma(uint32_t tmem_d, uint32_t da, uint32_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n\t}\n" ::"r"(tmem_d),
      "r"(da), "r"(db), "r"(idesc), "r"(accumulate), "r"(kDescHi));
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok));
  return ok != 0;
}

// Arrives on the barrier of the given offset in both CTAs once every MMA issued so far
// has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// acc += a * b in 64 bits, one multiply-add.
__device__ __forceinline__ void mad_wide(long long &acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// One element's exact accumulators over a chunk into the fixed-point sum (unit 2^-24).
__device__ __forceinline__ void add_exact(long long &acc, float e2, float e3, float e4) {
  // order 0: |E2| <= 256 * 2^14 = 2^22, read from the bit pattern of E2 + 1.5 * 2^23
  // (exact on the closed range: the pattern is linear in the integer up to and
  // including 2^24)
  const int x2 = __float_as_int(e2 + 12582912.0f) - 0x4B400000;
  // order 1: |E3 * 2^8| <= 2 * 256 * 2^14 = 2^23
  const int x3 = __float2int_rn(e3 * 256.0f);
  // order 2: |E4 * 2^16| <= 3 * 256 * 2^14 < 2^24
  const int x4 = __float2int_rn(e4 * 65536.0f);
  // |x2 * 2^8 + x3| <= 2^30 + 2^23 < 2^31
  mad_wide(acc, x2 * 256 + x3, 65536);
  mad_wide(acc, x4, 256);
}

// R over a chunk, at most 256 (4 * 2^14 * 2^-24 + 5 * 2^14 * 2^-32 + 6 * 2^14 * 2^-40)
// < 1.02, so R * 2^24 fits 32 bits.
__device__ __forceinline__ void add_rest(long long &acc, float r) {
  acc += (long long)__float2int_rn(r * 16777216.0f);
}

// The bits of (1.f) 2^(be - 1023) below the normal range (be < 1, rounded to nearest
// even) or above it (infinity); n: the significand with its leading one at bit 52.
__device__ __noinline__ unsigned long long out_of_range_bits(unsigned long long n, int be) {
  if (be > 2046) return 0x7FF0000000000000ull;
  const int sh = 1 - be;
  if (sh > 54) return 0;
  const unsigned long long q = n >> sh, r = n & ((1ull << sh) - 1), half = 1ull << (sh - 1);
  return q + ((r > half || (r == half && (q & 1))) ? 1 : 0);
}

// acc 2^e as an FP64 value for any |acc| < 2^53 and any e: exact in the normal range.
// rel: |acc| 2^r in FP32, rounded to nearest (0 below its normal range).
__device__ __noinline__ double scaled_any(long long acc, int e, int r, float &rel) {
  const unsigned long long sign = acc < 0 ? 1ull << 63 : 0;
  const unsigned long long m = acc < 0 ? (unsigned long long)(-acc) : (unsigned long long)acc;
  rel = 0.0f;
  if (m == 0) return 0.0;
  const int lz = __clzll((long long)m), be = 63 - lz + e + 1023, re = 63 - lz + r + 127;
  const unsigned long long n = m << (lz - 11);   // leading one at bit 52
  if (re >= 1) rel = __uint_as_float((uint32_t)((n + (1ull << 28)) >> 29) + ((uint32_t)(re - 1) << 23));
  const unsigned long long bits = be >= 1 && be <= 2046 ? n + ((unsigned long long)(be - 1) << 52) : out_of_range_bits(n, be);
  return __longlong_as_double((long long)(bits | sign));
}

// The same for |acc| < 2^51, results certain to be normal, e = f + t and r = t - 40 >= -120,
// by one FP64 addition (the bits of 1.5 2^52 + acc, less 1.5 2^52: exact) and integer
// operations on the exponents: f20 and t20 are f and t in the place of a double's exponent,
// and what rel and the result share is added once (rel's field is taken modulo 2^9, which
// holds it: 127 + r + 51 at most). rel is cut to FP32's 24 bits, not rounded (two additions
// more per element, 5% of the Z2 edge): kCutSquare times its square is as close as with
// rounding (rel off by 2^-24 at most).
constexpr float kCutSquare = 1.0f + 0x1p-23f;
__device__ __forceinline__ double scaled_add(long long acc, uint32_t f20, uint32_t t20, float &rel) {
  const double c = __longlong_as_double(acc + 0x4338000000000000ll) - 6755399441055744.0;
  const uint32_t h = (uint32_t)__double2hiint(c), l = (uint32_t)__double2loint(c);   // 0 for zero
  const uint32_t g = h + t20;
  rel = h != 0 ? __uint_as_float((__funnelshift_l(l, g, 3) - (936u << 23)) & 0x7fffffffu) : 0.0f;
  return __hiloint2double(h != 0 ? (int)(g + f20) : 0, (int)l);
}

// The same with integer operations only.
__device__ __forceinline__ double scaled_int(long long acc, uint32_t f20, uint32_t t20, float &rel) {
  const uint32_t s = (uint32_t)((int)((unsigned long long)acc >> 32) >> 31);   // all ones when negative
  const unsigned long long m = ((unsigned long long)acc ^ (((unsigned long long)s << 32) | s)) - (long long)(int)s;
  const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
  const int lz = mh ? __clz((int)mh) : 32 + __clz((int)ml);   // 64 for zero; at least 11
  const int sh = lz - 11;
  uint32_t nh = __funnelshift_l(ml, mh, sh), nl = ml << (sh & 31);   // leading one at bit 52
  if (sh >= 32) {
    nh = nl;
    nl = 0;
  }
  const uint32_t g = nh + t20 - ((uint32_t)lz << 20);
  rel = nh != 0 ? __uint_as_float(__funnelshift_l(nl, g, 3) + (149u << 23)) : 0.0f;
  const uint32_t hi = (g + f20 + (1085u << 20)) | (s & 0x80000000u);
  return __hiloint2double((int)(nh != 0 ? hi : 0u), (int)nl);
}

// Where the element of the tile's P row p and Q row q lies (null: nowhere; have: p is a
// row of the sector), and the row length len of its block (of C_q, when dense).
__device__ __noinline__ double *place_in_c(const OutView &out, const SplitTile *t, bool swap, bool have, int p, int q,
                                           int &len) {
  const int pi = t->pt * 2 * kSplitBM + p, qi = t->q_first + q;
  OutRow r{0, swap ? pi : qi};
  OutCol c{0, swap ? qi : pi, t->ld, 0};
  int64_t at = t->c_off;
  if (!have) return nullptr;
  if (out.sec) {
    r = out.rows[swap ? t->p_rec + p : t->q_rec + q];
    c = out.cols[swap ? t->q_rec + q : t->p_rec + p];
    at = __ldg(out.base + t->base + (int64_t)r.blk * t->ncb + c.blk);
  }
  len = c.len;
  return at >= 0 ? out.c + at + (int64_t)r.idx * c.len + c.idx : nullptr;
}

// 2^k as an FP32 value for k <= 0 (0 below the normal range).
__device__ __forceinline__ float pow2f(int k) { return k >= -126 ? __int_as_float((k + 127) << 23) : 0.0f; }

// Descriptor offsets in the 16-byte units of the start-address field: one slice of P
// (8 KB) and one K step of 16 (32 bytes); the Q halves lie 4 KB apart in a 128-wide
// tile and 2 KB apart in a 64-wide one (qsu). The shared-memory footprint stays below
// 256 KB, so additions never carry out of the 14-bit field.
constexpr uint32_t kSliceU = kSliceBytes >> 4, kStepU = 2;

// Descriptors of the slices of one stage: P slices and Q halves 0..2 in the lead slot,
// the others in the rest slot.
struct StageDesc {
  uint32_t pl, ql, pr, qr, qsu;
  __device__ __forceinline__ uint32_t p(int i) const { return i < 3 ? pl + i * kSliceU : pr + (i - 3) * kSliceU; }
  __device__ __forceinline__ uint32_t q(int i) const { return i < 3 ? ql + i * qsu : qr + (i - 3) * qsu; }
};

// The product of A's slice i and B's slice j (K step ks), wherever they lie (swap: P is
// A): the products of one accumulator are issued in the order of A's slices either way,
// so that its rounding does not depend on the operands' roles.
__device__ __forceinline__ void product(uint32_t d, const StageDesc &s, int i, int j, int ks, bool swap, uint32_t idesc,
                                        uint32_t acc) {
  umma(d, (swap ? s.p(i) : s.p(j)) + ks * kStepU, (swap ? s.q(j) : s.q(i)) + ks * kStepU, idesc, acc);
}

// Orders 0, 1, 2 of one 32-wide K stage into the exact accumulators; `fresh`
// starts a new chunk.
__device__ __forceinline__ void issue_exact(uint32_t tmem, const StageDesc &s, bool fresh, uint32_t idesc, bool swap) {
#pragma unroll
  for (int ks = 0; ks < 2; ks++) {
    const uint32_t acc = (fresh && ks == 0) ? 0u : 1u;
    product(tmem + kColE2, s, 0, 0, ks, swap, idesc, acc);
    product(tmem + kColE3, s, 0, 1, ks, swap, idesc, acc);
    product(tmem + kColE3, s, 1, 0, ks, swap, idesc, 1u);
    product(tmem + kColE4, s, 0, 2, ks, swap, idesc, acc);
    product(tmem + kColE4, s, 1, 1, ks, swap, idesc, 1u);
    product(tmem + kColE4, s, 2, 0, ks, swap, idesc, 1u);
  }
}

// Orders 3 .. S-1 of one stage into R; `fresh` starts a new chunk.
template <int S>
__device__ __forceinline__ void issue_rest(uint32_t tmem, const StageDesc &s, bool fresh, uint32_t idesc, bool swap) {
#pragma unroll
  for (int ks = 0; ks < 2; ks++) {
#pragma unroll
    for (int L = 3; L <= S - 1; L++) {
#pragma unroll
      for (int i = 0; i <= L; i++) {
        const uint32_t acc = (fresh && ks == 0 && L == 3 && i == 0) ? 0u : 1u;
        product(tmem + kColR, s, i, L - i, ks, swap, idesc, acc);
      }
    }
  }
}

// A slot of a ring and the parity of its current use.
struct Slot {
  int i = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next(int n) {
    if (++i == n) {
      i = 0;
      phase ^= 1;
    }
  }
  __device__ __forceinline__ void back(int n) {
    if (--i < 0) {
      i = n - 1;
      phase ^= 1;
    }
  }
};

// A position in the sequence of K stages over the CTA pair's tiles: stage st of the ks
// stages of tile t, and the stage's places in the rings. The same in every lane of the
// warp (the tile's fields are broadcast), so that the issue loop's values can live in
// uniform registers, which tcgen05.mma takes its operands from. The next tile's fields
// are loaded a tile ahead.
struct Cursor {
  int t, st, ks;
  uint32_t form, g;   // form: bn | swap << 16; g: stages passed
  Slot lead, rest;
  int next_ks;
  uint32_t next_form;

  __device__ __forceinline__ void fetch(const SplitTile *tiles, int i, int ntiles) {
    if (i < ntiles) {
      next_ks = tiles[i].ks;
      next_form = (uint32_t)tiles[i].bn | ((uint32_t)tiles[i].swap << 16);
    }
  }
  __device__ __forceinline__ void take() {
    ks = __shfl_sync(0xffffffffu, next_ks, 0);
    form = __shfl_sync(0xffffffffu, next_form, 0);
  }
  __device__ __forceinline__ void start(const SplitTile *tiles, int first, int step, int ntiles) {
    t = first;
    st = 0;
    g = 0;
    next_ks = 0;
    next_form = 0;
    fetch(tiles, first, ntiles);
    take();
    fetch(tiles, first + step, ntiles);
  }
  __device__ __forceinline__ void advance(const SplitTile *tiles, int step, int ntiles, int lead_stages,
                                          int rest_stages) {
    g++;
    lead.next(lead_stages);
    rest.next(rest_stages);
    if (++st == ks) {
      st = 0;
      t += step;
      take();
      fetch(tiles, t + step, ntiles);
    }
  }
};

// MIX: the tile list may hold 64-wide tiles and tiles whose P operand is A; without it
// every tile is 128 wide with P = B, and both are constants.
template <int S, bool MIX>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    gemm_split_kernel(const SplitSector *__restrict__ sectors, const SplitTile *__restrict__ tiles, int ntiles,
                      const uint8_t *sa, const uint8_t *sb, const int32_t *ea,
                      const int32_t *eb, const int32_t *emax, float *__restrict__ normsq,
                      OutView out, int *status) {
  using RG = Ring<S>;
  constexpr int kLeadP = 3 * kSliceBytes, kRestP = RG::kRest * kSliceBytes;   // P bytes of a slot
  extern __shared__ uint8_t smem_raw[];
  after_previous_kernel();
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + RG::kBytes);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kNumBars);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank(), pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  auto bar = [&](int i) { return smem_u32(&bars[i]); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; i++) {
      mbar_init(bar(kFull0 + i), rank == 0 ? 2 : 1);   // the leader's: its own copies and the peer's relay
      mbar_init(bar(kEmpty0 + i), 1);
      mbar_init(bar(kRestFull0 + i), rank == 0 ? 2 : 1);
      mbar_init(bar(kRestEmpty0 + i), 1);
    }
    mbar_init(bar(kEFull), 1);
    mbar_init(bar(kEEmpty), 2 * kEpiWarps);   // used in the leader: the epilogue warps of both CTAs
    mbar_init(bar(kRFull), 1);
    mbar_init(bar(kREmpty), 2 * kEpiWarps);
    mbar_init(bar(kDone), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // barriers initialised and tensor memory allocated in both CTAs
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      Slot lead, rest;
      uint32_t nlead = 0, nrest = 0;   // slots loaded
      bool ok = true;
      for (int t = pair; t < ntiles && ok; t += npairs) {
        const SplitTile tl = tiles[t];
        const SplitSector sc = sectors[tl.sector];
        const bool swap = MIX && tl.swap, narrow = MIX && tl.bn == 64;
        const int pt = 2 * tl.pt + rank;
        const bool have = pt * kSplitBM < (swap ? sc.M : sc.N);   // else this CTA's lanes hold no output
        const uint8_t *pblk = (swap ? sa + sc.sa_off : sb + sc.sb_off) + (int64_t)pt * sc.ks * kBlockBytes;
        // this CTA's half of the Q tile: 64 rows of a 128-row block, or 32 of a 64-row half
        const uint8_t *qblk = (swap ? sb + sc.sb_off : sa + sc.sa_off) +
                              (int64_t)(narrow ? tl.qt >> 1 : tl.qt) * sc.ks * kBlockBytes +
                              (narrow ? (tl.qt & 1) * kHalfBytes + rank * (kHalfBytes / 2) : rank * kHalfBytes);
        const uint32_t qbytes = narrow ? kHalfBytes / 2 : kHalfBytes;
        for (int kt = 0; kt < sc.ks; kt++, pblk += kBlockBytes, qblk += kBlockBytes) {
          // n slices from slice p0 on into the slot at dst: P slices, then Q halves
          auto load = [&](int full, int empty, const Slot &sl, uint32_t dst, int p0, int n) {
            ok = mbar_wait(bar(empty + sl.i), sl.phase ^ 1, abort_flag, status, 1);
            if (!ok) return;
            const uint32_t fb = bar(full + sl.i), pbytes = (uint32_t)n * kSliceBytes;
            mbar_expect_tx(fb, (have ? pbytes : 0) + n * qbytes);
            if (have) bulk_g2s(dst, pblk + p0 * kSliceBytes, pbytes, fb);
            for (int p = 0; p < n; p++)
              bulk_g2s(dst + pbytes + p * qbytes, qblk + (p0 + p) * kSliceBytes, qbytes, fb);
          };
          load(kFull0, kEmpty0, lead, smem_u32(smem) + lead.i * RG::kLeadSlot, 0, 3);
          if (!ok) break;
          nlead++;
          lead.next(RG::kLeadStages);
          load(kRestFull0, kRestEmpty0, rest, smem_u32(smem) + RG::kLeadBytes + rest.i * RG::kRestSlot, 3, RG::kRest);
          if (!ok) break;
          nrest++;
          rest.next(RG::kRestStages);
        }
      }
      // no copy, and no arrival of a "slot free" commit, may still be in flight when
      // the CTA exits (after an abort some slots are never freed: those waits end with
      // the flag, and the commits that were issued are waited for through kDone)
      auto finish = [&](Slot &sl, uint32_t n, int stages, int full, int empty) {
        for (uint32_t k = 0; k < min(n, (uint32_t)stages); k++) {
          sl.back(stages);
          if (!mbar_wait(bar(full + sl.i), sl.phase, abort_flag, status, 2)) mbar_drain(bar(full + sl.i), sl.phase);
          mbar_wait(bar(empty + sl.i), sl.phase, abort_flag, status, 10);
        }
      };
      finish(lead, nlead, RG::kLeadStages, kFull0, kEmpty0);
      finish(rest, nrest, RG::kRestStages, kRestFull0, kRestEmpty0);
    }
  } else if (warp == 1 && rank == 1) {
    // --------------------------------------------------------- relay (peer CTA)
    if (lane == 0) {
      Slot lead, rest;
      bool ok = true;
      for (int t = pair; t < ntiles && ok; t += npairs) {
        const int ks = tiles[t].ks;
        for (int kt = 0; kt < ks && ok; kt++) {
          ok = mbar_wait(bar(kFull0 + lead.i), lead.phase, abort_flag, status, 9);
          if (!ok) break;
          mbar_arrive_cluster(leader_addr(bar(kFull0 + lead.i)));
          ok = mbar_wait(bar(kRestFull0 + rest.i), rest.phase, abort_flag, status, 9);
          if (!ok) break;
          mbar_arrive_cluster(leader_addr(bar(kRestFull0 + rest.i)));
          lead.next(RG::kLeadStages);
          rest.next(RG::kRestStages);
        }
      }
      // the leader's MMAs read this CTA's shared memory and their commits arrive here
      if (!mbar_wait(bar(kDone), 0, abort_flag, status, 6)) mbar_drain(bar(kDone), 0);
    }
  } else if (warp == 1) {
    // --------------------------------------------------------- MMA issuer (leader)
    // The whole warp runs the loop on uniform values; one elected lane issues.
    const uint32_t slot_base = smem_u32(smem), bar_base = bar(0);
    auto ready = [&](int i, uint32_t parity) { return __all_sync(0xffffffffu, mbar_test(bar_base + 8 * i, parity)); };
    Cursor e, r;   // next stage of the exact products and of the R products
    e.start(tiles, pair, npairs, ntiles);
    r.start(tiles, pair, npairs, ntiles);
    uint32_t loaded = 0;                 // stages whose lead slices are known to have arrived
    uint32_t ne = 0, nr = 0;             // chunks committed
    bool ewait = false, rwait = false;   // the accumulators still hold a chunk to be drained
    bool e_fresh = true, r_fresh = true;   // the next stage starts a chunk
    uint32_t idle = 0;
    auto lead_ready = [&](const Cursor &c) {
      if (c.g < loaded) return true;
      if (!ready(kFull0 + c.lead.i, c.lead.phase)) return false;
      loaded = c.g + 1;
      return true;
    };
    auto stage = [&](const Cursor &c, bool narrow) {
      const uint32_t l = slot_base + c.lead.i * RG::kLeadSlot, r2 = slot_base + RG::kLeadBytes + c.rest.i * RG::kRestSlot;
      return StageDesc{desc_lo(l), desc_lo(l + kLeadP), desc_lo(r2), desc_lo(r2 + kRestP),
                       (uint32_t)(narrow ? kHalfBytes / 2 : kHalfBytes) >> 4};
    };
    while (e.t < ntiles || r.t < ntiles) {
      // the queue whose chunk ends at the earlier stage goes first, so that the other one
      // has stages left to multiply while that chunk is drained; the other one when it
      // is blocked (by its drain, or the depth of the ring)
      const uint32_t ge = e.g + (e_end(e.st, e.ks) - e.st), gr = r.g + (r_end(r.st, r.ks) - r.st);
      bool did = false, exact = e.t < ntiles && (ge <= gr || r.t >= ntiles);
#pragma unroll 1
      for (int turn = 0; turn < 2 && !did; turn++, exact = !exact) {
        if (exact) {
          if (e.t >= ntiles || !lead_ready(e)) continue;
          if (ewait) {
            if (!ready(kEEmpty, (ne - 1) & 1)) continue;
            ewait = false;
          }
          tc_fence_after();
          const bool narrow = MIX && (e.form & 0xffff) == 64, swap = MIX && (e.form >> 16);
          const bool ends = e.st == e_end(e.st, e.ks), free_slot = r.g > e.g;   // R is past this stage
          const StageDesc sd = stage(e, narrow);
          if (elect_one()) {
            issue_exact(tmem, sd, e_fresh, idesc_for(narrow ? 64 : 128), swap);
            if (ends) umma_commit(bar_base + 8 * kEFull);
            if (free_slot) umma_commit(bar_base + 8 * (kEmpty0 + e.lead.i));
          }
          __syncwarp();
          if (ends) {
            ne++;
            ewait = true;
          }
          e_fresh = ends;
          e.advance(tiles, npairs, ntiles, RG::kLeadStages, RG::kRestStages);
        } else {
          if (r.t >= ntiles || !lead_ready(r) || !ready(kRestFull0 + r.rest.i, r.rest.phase)) continue;
          if (rwait) {
            if (!ready(kREmpty, (nr - 1) & 1)) continue;
            rwait = false;
          }
          tc_fence_after();
          const bool narrow = MIX && (r.form & 0xffff) == 64, swap = MIX && (r.form >> 16);
          const bool ends = r.st == r_end(r.st, r.ks), free_slot = e.g > r.g;
          const StageDesc sd = stage(r, narrow);
          if (elect_one()) {
            issue_rest<S>(tmem, sd, r_fresh, idesc_for(narrow ? 64 : 128), swap);
            if (ends) umma_commit(bar_base + 8 * kRFull);
            if (free_slot) umma_commit(bar_base + 8 * (kEmpty0 + r.lead.i));
            umma_commit(bar_base + 8 * (kRestEmpty0 + r.rest.i));
          }
          __syncwarp();
          if (ends) {
            nr++;
            rwait = true;
          }
          r_fresh = ends;
          r.advance(tiles, npairs, ntiles, RG::kLeadStages, RG::kRestStages);
        }
        did = true;
      }
      if (did) {
        idle = 0;
      } else {
        idle++;
        const bool late = idle >= kMaxPolls;
        if (late || ((idle & 63) == 63 && __any_sync(0xffffffffu, *abort_flag != 0))) {
          if (late && lane == 0) {
            abort_pair(abort_flag);
            atomicCAS(status, 0, 3);
          }
          break;
        }
      }
    }
    // every issued MMA has completed before tensor memory is released
    __syncwarp();
    if (elect_one()) umma_commit(bar(kDone));
    __syncwarp();
    if (lane == 0 && !mbar_wait(bar(kDone), 0, abort_flag, status, 6)) mbar_drain(bar(kDone), 0);
  } else if (warp >= kFirstEpiWarp) {
    // ---------------------------------------------------------------- epilogue
    // four warps per 32-lane quarter of tensor memory; columns [c0, c0 + w) with
    // w = 32 in a 128-wide tile and 16 in a 64-wide one
    const int quarter = warp & 3, part = (warp - kFirstEpiWarp) >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t e_empty = leader_addr(bar(kEEmpty)), r_empty = leader_addr(bar(kREmpty));
    uint32_t ce = 0, cr = 0;   // chunks drained
    bool ok = true;
    for (int t = pair; t < ntiles && ok; t += npairs) {
      const struct { int sector, ks, bn, swap; } tl = {tiles[t].sector, tiles[t].ks, tiles[t].bn, tiles[t].swap};
      const bool narrow = MIX && tl.bn == 64, swap = MIX && tl.swap;
      const int c0 = narrow ? part * 16 : part * 32;   // first column
      const int ngroups = narrow ? 4 : 8;              // groups of 4 columns
      // the tables that the output needs, into L1 while the first chunk is multiplied
      const SplitTile *tp = tiles + t;
      const int p0 = rank * kSplitBM + quarter * 32;   // the warp's first row of P in the tile
      if (p0 + lane < tp->np) {
        prefetch_l1((swap ? ea : eb) + tp->p_exp + p0 + lane);
        if (out.sec) {
          if (swap) prefetch_l1(out.rows + tp->p_rec + p0 + lane);
          else prefetch_l1(out.cols + tp->p_rec + p0 + lane);
        }
      }
      if (c0 + lane < tp->nq) {
        prefetch_l1((swap ? eb : ea) + tp->q_exp + c0 + lane);
        if (out.sec) {
          if (swap) prefetch_l1(out.cols + tp->q_rec + c0 + lane);
          else prefetch_l1(out.rows + tp->q_rec + c0 + lane);
        }
      }
      long long acc[32];
#pragma unroll
      for (int j = 0; j < 32; j++) acc[j] = 0;
      auto drain_r = [&]() {
        ok = mbar_wait(bar(kRFull), cr & 1, abort_flag, status, 8);
        if (!ok) return;
        cr++;
        tc_fence_after();
#pragma unroll
        for (int g = 0; g < 4; g++) {
          if (g < ngroups / 2) {
            uint32_t vr[8];
            tmem_ld8(lane_addr + kColR + c0 + g * 8, vr);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; i++) add_rest(acc[g * 8 + i], __uint_as_float(vr[i]));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(r_empty);
      };
      // The tile's place in C: a lane holds one row of P, its accumulators 32 rows of Q.
      // The lanes read the places and exponents of those 32 rows, one each. Inside a block
      // of C consecutive rows of Q lie a constant step apart, so an element costs the
      // conversion, an addition and the store. Read before the last chunk's drains, with
      // the places of the first kMaxStarts blocks (most often all there are), so that the
      // chain of loads ends while the last chunk is multiplied.
      const bool direct = out.sec != nullptr;
      const bool in = p0 + lane < tp->np;
      const int nq = min(tp->nq - c0, ngroups * 4);   // valid rows of Q
      int ep = 0, uq = 0;        // exponents of the lane's row of P, of row `lane` of the 32
      uint32_t starts = 0;       // rows that enter a block of C
      int len = 0;               // columns of the lane's block
      double *places[kMaxStarts];   // the lane's places at the first starts
      auto place = [&](int j) { return place_in_c(out, tp, swap, in, p0 + lane, c0 + j, len); };
      auto find_places = [&]() {
        int lblk = 0, lidx = tp->pt * 2 * kSplitBM + p0 + lane;   // the lane's row of P in C
        int ublk = 0, uidx = tp->q_first + c0 + lane;             // row `lane` of the 32
        len = tp->ld;
        if (in) {
          ep = (swap ? ea : eb)[tp->p_exp + p0 + lane];
          if (direct && swap) {
            const OutRow x = out.rows[tp->p_rec + p0 + lane];
            lblk = x.blk;
            lidx = x.idx;
          } else if (direct) {
            const OutCol x = out.cols[tp->p_rec + p0 + lane];
            lblk = x.blk;
            lidx = x.idx;
            len = x.len;
          }
        }
        if (lane < nq) {
          uq = (swap ? eb : ea)[tp->q_exp + c0 + lane];
          if (direct && swap) {
            const OutCol x = out.cols[tp->q_rec + c0 + lane];
            ublk = x.blk;
            uidx = x.idx;
            len = x.len;   // of this lane's column: read through the lane that starts a block
          } else if (direct) {
            const OutRow x = out.rows[tp->q_rec + c0 + lane];
            ublk = x.blk;
            uidx = x.idx;
          }
        }
        const int before = __shfl_up_sync(0xffffffffu, ublk, 1);
        starts = __ballot_sync(0xffffffffu, lane < nq && (lane == 0 || ublk != before));
        const int64_t *base = out.base + tp->base + (swap ? (int64_t)lblk * tp->ncb : (int64_t)lblk);
        const int64_t bstep = swap ? 1 : tp->ncb;
        int64_t at[kMaxStarts];
        uint32_t m = starts;
#pragma unroll
        for (int k = 0; k < kMaxStarts; k++, m &= m - 1) {
          const int b = __shfl_sync(0xffffffffu, ublk, m ? __ffs(m) - 1 : 0);
          at[k] = tp->c_off;
          if (direct) at[k] = in && m ? __ldg(base + bstep * b) : -1;
        }
        m = starts;
#pragma unroll
        for (int k = 0; k < kMaxStarts; k++, m &= m - 1) {
          const int j = m ? __ffs(m) - 1 : 0;
          const int x = __shfl_sync(0xffffffffu, uidx, j);
          const int l = MIX && swap ? __shfl_sync(0xffffffffu, len, j) : len;
          places[k] = in && at[k] >= 0 ? out.c + at[k] + (swap ? (int64_t)lidx * l + x : (int64_t)x * l + lidx) : nullptr;
        }
      };
      // drains in the order in which their chunks end; the last one, of R, comes below
      int se = e_end(0, tl.ks), sr = r_end(0, tl.ks);   // last stages of the next chunks
#pragma unroll 1
      while (ok && (se < tl.ks || sr < tl.ks - 1)) {
        if (se <= sr) {
          if (se == tl.ks - 1) find_places();
          ok = mbar_wait(bar(kEFull), ce & 1, abort_flag, status, 7);
          if (!ok) break;
          ce++;
          tc_fence_after();
#pragma unroll
          for (int g = 0; g < 8; g++) {
            if (g < ngroups) {
              uint32_t v2[4], v3[4], v4[4];
              tmem_ld4(lane_addr + kColE2 + c0 + g * 4, v2);
              tmem_ld4(lane_addr + kColE3 + c0 + g * 4, v3);
              tmem_ld4(lane_addr + kColE4 + c0 + g * 4, v4);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 4; i++)
                add_exact(acc[g * 4 + i], __uint_as_float(v2[i]), __uint_as_float(v3[i]), __uint_as_float(v4[i]));
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(e_empty);
          se = se == tl.ks - 1 ? tl.ks : min(se + 8, tl.ks - 1);
        } else {
          drain_r();
          sr = min(sr + 8, tl.ks - 1);
        }
      }
      if (!ok) break;
      drain_r();
      if (!ok) break;
      // C = acc * 2^(e_i + f_j - 40); beside it, the tile's share of the sector's
      // ||C_q||^2 relative to 4^(emax_A + emax_B) for the accuracy check, in FP32
      // (relative to the largest of the Q row exponents inside the sum, so that the
      // additions to exponents stay small, and of the P rows outside). Half of the
      // elements are converted by an FP64 addition, half by integer operations: the
      // FP64 unit takes 16 clocks per warp, about what the integers of the other half
      // take, and nothing branches in between: 11,000 clocks for the CTA's 128 x 128
      // elements, against 16,000 with integers and a range check per element. The MMA
      // issuer waits for what exceeds the first chunk of the next tile.
      const int pref = emax[2 * tl.sector + (swap ? 0 : 1)], qref = emax[2 * tl.sector + (swap ? 1 : 0)];
      const int64_t step = swap ? 1 : len;
      const int e0 = ep + qref - 2 * kExpBias - 40;
      uq = max(uq - qref, -4096);
      // few blocks, every result normal and every sum below 2^51? (Rows past the sector have
      // zero slices and sums; a warp at the sector's edge took the general way at first,
      // and the whole tile waited for it.)
      const int umin = __reduce_min_sync(0xffffffffu, lane < nq ? uq : 0);
      const int lo = __reduce_min_sync(0xffffffffu, in ? e0 : 0), hi = __reduce_max_sync(0xffffffffu, in ? e0 : 0);
      const bool plain = umin >= -80 && lo + umin > -900 && hi < 900 && tl.ks <= 252 && __popc(starts) <= kMaxStarts;
      float ss = 0.0f;
      double *ptr = nullptr;
      if (plain) {
        const double *const *next = places;
        bool put = false;
        const uint32_t u20 = (uint32_t)uq << 20, e20 = (uint32_t)e0 << 20;
        auto element = [&](int j) {
          const uint32_t t20 = __shfl_sync(0xffffffffu, u20, j);
          float rel;
          const double d = j & 1 ? scaled_int(acc[j], e20, t20, rel) : scaled_add(acc[j], e20, t20, rel);
          if (put && j < nq) *ptr = d;
          ptr += step;
          ss = fmaf(rel, rel, ss);
        };
#pragma unroll
        for (int h = 0; h < 32; h += kOutGroup) {
          if (h >= nq) break;
          // a block starts at the group's first row or not at all, most often: then its
          // elements follow one another without a branch and overlap
          if (starts >> h & 1) {
            ptr = const_cast<double *>(*next++);
            put = ptr != nullptr;
          }
          if (!(starts >> h & ((1u << kOutGroup) - 2))) {
#pragma unroll
            for (int i = 0; i < kOutGroup; i++) element(h + i);
          } else {
#pragma unroll
            for (int i = 0; i < kOutGroup; i++) {
              if (i > 0 && (starts >> (h + i) & 1)) {
                ptr = const_cast<double *>(*next++);
                put = ptr != nullptr;
              }
              element(h + i);
            }
          }
        }
        ss = in ? ss * kCutSquare : 0.0f;
      } else {
#pragma unroll
        for (int j = 0; j < 32; j++) {
          const int t = __shfl_sync(0xffffffffu, uq, j);
          if (j < nq) {
            if (starts >> j & 1) ptr = place(j);
            float rel;
            const double d = scaled_any(acc[j], e0 + t, t - 40, rel);
            if (ptr) {
              *ptr = d;
              ptr += step;
              ss = fmaf(rel, rel, ss);
            }
          }
        }
      }
      ss *= pow2f(2 * (ep - pref));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      if (lane == 0 && ss > 0.0f) atomicAdd(normsq + tl.sector, ss);
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // neither CTA's shared or tensor memory is in use any more
  tc_fence_after();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  cluster_sync();
}

template <int S, bool MIX>
cudaError_t configure_one() {
  cudaError_t e = cudaFuncSetAttribute(gemm_split_kernel<S, MIX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Ring<S>::kSmem);
  if (e != cudaSuccess) return e;
  // all of the SM's unified memory as shared memory, so that a slicing CTA of the
  // pipelined split fits beside this kernel's CTA (the L1 share it leaves unused
  // is not read by this kernel: operands arrive by bulk copies)
  return cudaFuncSetAttribute(gemm_split_kernel<S, MIX>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              cudaSharedmemCarveoutMaxShared);
}

}  // namespace

// Opt the kernels in to their shared-memory size; once per device (a context
// does it at creation), so that launches stay free of non-stream calls.
cudaError_t configure_split_gemm() {
  for (cudaError_t (*configure)() : {configure_one<4, false>, configure_one<5, false>, configure_one<6, false>,
                                     configure_one<4, true>, configure_one<5, true>, configure_one<6, true>}) {
    cudaError_t e = configure();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_gemm_split(const SplitSector *sectors, const SplitTile *tiles, int64_t ntiles, const uint8_t *sa,
                              const uint8_t *sb, const int32_t *ea, const int32_t *eb, const int32_t *emax,
                              float *normsq, const OutView &out, int slices, int *status, int num_sms,
                              bool mixed_widths, cudaStream_t stream) {
  if (ntiles <= 0) return cudaSuccess;
  if (ntiles > INT32_MAX || slices < 4 || slices > kSlices) return cudaErrorInvalidValue;
  const int64_t pairs = std::min<int64_t>(ntiles, std::max(1, num_sms / 2));
  cudaError_t e = cudaSuccess;
  auto launch = [&](auto kernel, int smem) {
    e = launch_chained(kernel, (unsigned)(2 * pairs), kThreads, (size_t)smem, stream, sectors, tiles, (int)ntiles, sa, sb,
                       ea, eb, emax, normsq, out, status);
  };
  switch (slices + (mixed_widths ? 8 : 0)) {
    case 4: launch(gemm_split_kernel<4, false>, Ring<4>::kSmem); break;
    case 5: launch(gemm_split_kernel<5, false>, Ring<5>::kSmem); break;
    case 6: launch(gemm_split_kernel<6, false>, Ring<6>::kSmem); break;
    case 12: launch(gemm_split_kernel<4, true>, Ring<4>::kSmem); break;
    case 13: launch(gemm_split_kernel<5, true>, Ring<5>::kSmem); break;
    default: launch(gemm_split_kernel<6, true>, Ring<6>::kSmem); break;
  }
  return e;
}

}  // namespace ytn
