// FP64 fast-diagonalization apply on the tensor cores, for n_k <= 256 (in
// directions whose U_k has rows of very different sizes on the FP64 pipe, see
// kRowRange).
//
// GB300 issues two FP64 FMAs per clock per SM (1.26 TFLOP/s in all), so the
// 12 n^4 FLOP of the six mode products take 2.6 ms at n = 128 on the FP64
// pipe however they are arranged (the SIMT kernel of fd.cu measured 3.10 ms).
// Here each FP64 operand is split into six 10-bit integer digits (the
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with
// integer digits), and the products of digits run on the tensor cores:
//
//   a_mi = 2^(ea_m - 1080) sum_s da[s]_mi 1024^(5 - s),   |da[0]| <= 256,
//   b_ji = 2^(eb_j - 1080) sum_t db[t]_ji 1024^(5 - t),   |da[s]| <= 512
//   sum_i a_mi b_ji = 2^(ea_m + eb_j - 2160) sum_g 1024^(10 - g) G_g,
//   G_g = sum_{s + t = g} sum_i da[s]_mi db[t]_ji
//
// with ea_m the largest exponent field of row m and eb_j that of row j of B
// (U_k^T or U_k, split at set-up). Digits are exact in FP16; the FP32
// accumulators of tcgen05.mma hold the integers of groups 0 to 3 exactly,
// whatever the digits (split_plan.h). Groups g <= 5 are kept (21 digit
// products); their accumulators are summed as 64-bit integers and rounded to
// FP64 once. A product's error is relative to the largest entries of its row
// and column: in units of 2^-53 of their norms 0.1-0.2 for rows along an
// eigenvector of degree 1 (an FP64 chain: 6-9), 18 for one large entry among
// 127 equal ones that are smaller by any factor (chain: 47). The divide by
// D_1 (+) D_2 (+) D_3 multiplies the integer result before that rounding. The
// digits' path executes no FP64 instruction (each would issue at the
// 2-per-clock rate).
//
// Measured: 212 us per apply at n = 128 (SIMT: 3.10 ms), 110 us at (95, 61, 77)
// (SIMT: 0.98 ms), 1.41 ms at n = 192 (SIMT: 13.8 ms). A pass at n = 128 takes the
// phases of its one tile per SM in turn, nothing beside them: reading and
// splitting the rows (6 us), the MMAs with the summation of their accumulators
// (the MMAs alone 5 us), the last rounding (2.5 us), and about 6 us between two
// launches. A profile shows 23 % of the issue slots and 10 % of the tensor pipe
// in use; waiting for instructions is the largest stall (the unrolled steps
// miss the instruction cache), but the steps of a group as a loop took as long.
// With groups 1 to 3 in fewer, larger sums (eight instead of fifteen steps at
// K = 128) an apply took 172 and 94 us, but rows whose digits add up with one
// sign passed 2^24 and lost up to 3000 units of 2^-53.
//
// A CTA takes 128 rows (the other directions' indices) and up to 128 columns.
// A's digits live in tensor memory (6 slices of K/2 columns: 384 of 512 at
// K = 128), where each thread writes the digits of its own row; B's digits
// lie in shared memory (6 x 32 KB at n = 128); two accumulators of 64 columns
// take the rest of tensor memory: the products of a step go into one while the
// previous one is read.
//
// Directions are contracted in the order 3, 2, 1 and back 1, 3, 2: in four of
// the six products (three of four in 2D) the row index is then contiguous in
// memory and rows map to lanes without a transposition; the other two read
// rows that are contiguous in the contracted direction through a
// warp-private transposition. The divide's table inv_lam is stored in the
// layout the third product writes, [j1][j3][j2].
#include "common.cuh"
#include "split_plan.h"

#include <atomic>
#include <cstdlib>
#include <type_traits>

#include <cuda_fp16.h>

namespace {

using namespace igafd_split;

constexpr int kM = 128;                 // rows per CTA (MMA M, TMEM lanes)
constexpr int kThreads = 512;           // 4 warps per lane quarter
constexpr int kWarps = kThreads / 32;
constexpr int kSpin = kWaitPolls;    // bounded waits
// X + kBias = sum_s (digit_s + 512) 1024^(5-s): every 10-bit field is then the
// digit plus 512
constexpr unsigned long long kBias = 512ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) +
                                               (1ull << 40) + (1ull << 50));

struct SplitArgs {
  const double *in;
  double *out;
  long long M;            // rows
  int F;                  // rows m = hi F + lo
  long long in_hi, in_lo, in_k, out_hi, out_lo, out_n;   // element strides
  int K, Kp;              // contracted length, padded to a multiple of 32 (the kernel's KP)
  int N, Np, NT;          // columns, padded to 16; columns per CTA (multiple of 16)
  const unsigned char *img;   // digits of B: [slice][64-wide K chunk][Np][128 B], swizzled
  const int *eb;              // exponent field of each row of B
  const int *range;           // largest and smallest exponent field of the rows of U_k
  const double *U;            // U_k, B's element (column j, term k) at j u_j + k u_k
  int u_j, u_k;
  const double *inv_lam;      // divide table, indexed like out (null: none)
  const double *done;
  int *err;
  int polls;              // of a wait before it gives up
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// K-major, 128-byte swizzle (8-row groups of 1024 B)
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(16 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Bounded wait, given up early once another thread's wait ran out.
__device__ __forceinline__ bool wait_on(uint64_t *bar, uint32_t parity, const int *failed,
                                        int polls = kSpin) {
  for (int it = 0; it < polls; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 255) == 255 && *(volatile const int *)failed) return false;
  }
  return false;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// shifts by 32 or more give 0
__device__ __forceinline__ uint32_t shr_clamp(uint32_t v, uint32_t s) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
  return r;
}

// The exponent field of a double given its high word: 1 for zero and
// subnormals (whose mantissa has no hidden bit), 0x7ff for infinities and NaN.
__device__ __forceinline__ int exp_field(uint32_t hi) {
  const int e = (int)((hi >> 20) & 0x7ffu);
  return e > 1 ? e : 1;
}

// X + kBias with X = d 2^(1022 + kBits - ea) rounded down, |X| <= 2^kBits, as
// its upper and lower 30 bits (junk above bit 30 of the lower word); d's
// exponent field lowered by s (0 or a column scaling of U_k).
__device__ __forceinline__ void biased_fixed(double d, int ea, uint32_t &w1, uint32_t &w0, int s = 0) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  // mantissa with the hidden bit at bit 63 (its place holds the exponent's
  // lowest bit, which is 0 where there is no hidden bit)
  const uint32_t mh = __funnelshift_l(lo, hi, 11) | ((hi & 0x7ff00000u) ? 0x80000000u : 0u);
  const uint32_t ml = lo << 11;
  const uint32_t sh = (uint32_t)(ea + 64 - kBits - exp_field(hi) + s);
  const uint32_t s1 = min(sh, 32u);
  uint32_t xh = shr_clamp(mh, s1);
  uint32_t xl = shr_clamp(__funnelshift_rc(ml, mh, s1), sh - s1);
  const uint32_t sg = (uint32_t)((int)hi >> 31);
  const unsigned long long x =
      (((unsigned long long)(xh ^ sg) << 32) | (xl ^ sg)) + kBias;
  w0 = (uint32_t)x;
  w1 = __funnelshift_r(w0, (uint32_t)(x >> 32), 30);
}

// digit at bit 10 POS of the words of two elements, as packed FP16 (element 0
// in the low half): fields 0..1023 become 1024 + field by their bits, minus 1536
template <int POS> __device__ __forceinline__ uint32_t digit2(uint32_t a, uint32_t b) {
  uint32_t w;
  if (POS == 0) w = __byte_perm(a, b, 0x5410);
  else if (POS == 1) w = __byte_perm(a, b, 0x6521) >> 2;
  else w = __byte_perm(a, b, 0x7632) >> 4;
  w = (w & 0x03ff03ffu) | 0x64006400u;
  const __half2 h = __hsub2(*reinterpret_cast<__half2 *>(&w), __half2half2(__ushort_as_half(0x6600)));
  return *reinterpret_cast<const uint32_t *>(&h);
}

// T 2^E lam for what round_fixed leaves out (noinline: rare)
__device__ __noinline__ double round_slow(long long T, int E, double lam) {
  return ldexp((double)T, E) * lam;
}

// T 2^E (times lam with LAM) rounded to FP64 with integer instructions; slow
// is set, and the value undefined, for results outside the normal range and
// for lam that is not a positive normal number
template <bool LAM>
__device__ __forceinline__ double round_fixed(long long T, int E, double lam, bool &slow) {
  const int sg = (int)(T >> 63);
  const unsigned long long u = (unsigned long long)(T ^ (long long)sg) - (unsigned long long)(long long)sg;
  uint32_t h = (uint32_t)(u >> 32), l = (uint32_t)u;
  int e = E + 1085 + 1;                             // exponent field of the result minus 1, and 1
  if (h == 0u) { h = l; l = 0u; e -= 32; }
  const int lz = __clz((int)h);
  h = __funnelshift_l(l, h, lz);
  l = l << (lz & 31);
  e -= lz;                                          // (h l) in [2^63, 2^64), or 0
  if (LAM) {
    const uint32_t lh = (uint32_t)__double2hiint(lam), ll = (uint32_t)__double2loint(lam);
    slow = slow || lh - 0x00100000u >= 0x7fe00000u;
    // the upper half of the 128-bit product, but for the carry of its lower half (2^-63)
    const uint32_t Lh = __funnelshift_l(ll, lh, 11) | 0x80000000u, Ll = ll << 11;
    const unsigned long long p = (unsigned long long)h * Lh + __umulhi(h, Ll) + __umulhi(l, Lh);
    h = (uint32_t)(p >> 32);
    l = (uint32_t)p;
    const int n = (int)(~h >> 31);                  // one more shift
    h = __funnelshift_l(l, h, n);
    l <<= n;
    e += (int)(lh >> 20) - 1022 - n;
  }
  // 53 bits and the rounding bit; a carry runs into the exponent field
  const unsigned long long q =
      (((unsigned long long)(h >> 11) << 32) | __funnelshift_r(l, h, 11)) + ((l >> 10) & 1u) +
      ((unsigned long long)(uint32_t)(e - 1) << 52);
  const bool zero = T == 0;
  slow = slow || (!zero && (uint32_t)(e - 2) >= 2043u);
  return __hiloint2double(zero ? 0 : (int)((uint32_t)(q >> 32) | ((uint32_t)sg & 0x80000000u)),
                          zero ? 0 : (int)(uint32_t)q);
}

// Columns per accumulator and CTAs per SM: with K <= 64 two CTAs fit (256 TMEM
// columns and half the shared memory each), so one's MMAs and the start of the
// next launch overlap the other's integer work.
constexpr int acc_cols(int KP) { return KP > 64 ? 64 : 32; }
// With K > 128 a CTA takes at most 64 columns, so that B's digits of both
// parts fit.
constexpr int b_rows(int KP) { return KP > 128 ? 64 : kM; }
constexpr int ctas_per_sm(int KP) { return KP > 64 ? 1 : 2; }
// doubles per row of a transposition buffer, and its bytes for all warps
constexpr int trans_cols(int KP) { return KP > 128 ? 8 : 17; }
constexpr int trans_bytes(int KP) { return 16 * 32 * trans_cols(KP) * 8; }
// f(0), f(1), ... f(N - 1), as constants
template <typename F, int... I>
__device__ __forceinline__ void each_of(F &&f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F> __device__ __forceinline__ void each_step(F &&f) {
  each_of(f, std::make_integer_sequence<int, N>{});
}

// Largest difference between the exponents of the rows of U_k (by their largest
// entries) up to which the digits are used: a right-hand side that meets a
// small row multiplies entries that lost as many bits of the 58 as the row is
// smaller than the columns' largest. Uniform knots have at most 3 (n <= 256,
// every degree), spans graded by up to 50 have 4, span scalings 4 for a
// standard deviation of 1 of their logarithms. Largest errors of P^{-1} r in 2D
// over random, constant and single-entry right-hand sides (60 graded and scaled
// pencils), digits against FP64 chains: 0.9 and 2.5 x 1e-15 up to 4, 2.5 and
// 2.0 at 5, 19 and 1.5 at 8.
constexpr int kRowRange = 4;

// The mode product of this CTA's rows and columns as FP64 chains, for
// pencils beyond that range and for U_k that is not finite: on the FP64 pipe,
// rows and columns as below, U_k from L1 (n = 128: 3.1 ms per apply, as the
// SIMT kernel; (95, 61, 77): 0.70 ms). Decided by what the set-up left on the
// device, so that captured launches follow a new set-up.
template <bool LAM>
__device__ __forceinline__ void chain_rows(const SplitArgs &a, int n0, int cols) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long m = (long long)blockIdx.x * kM + (warp & 3) * 32 + lane;
  if (m >= a.M) return;
  const long long hi = m / a.F, lo = m - hi * a.F;
  const double *src = a.in + hi * a.in_hi + lo * a.in_lo;
  const long long ob = hi * a.out_hi + lo * a.out_lo;
  constexpr int C = 8;                                     // columns at a time
  for (int c = C * (warp >> 2); c < cols; c += C * (kWarps / 4)) {
    double acc[C];
    const double *u[C];
#pragma unroll
    for (int t = 0; t < C; ++t) {
      acc[t] = 0.0;
      u[t] = a.U + (size_t)min(n0 + c + t, a.N - 1) * a.u_j;
    }
    for (int k = 0; k < a.K; ++k) {
      const double x = __ldg(src + (long long)k * a.in_k);
#pragma unroll
      for (int t = 0; t < C; ++t) acc[t] = fma(x, __ldg(u[t] + (size_t)k * a.u_k), acc[t]);
    }
#pragma unroll
    for (int t = 0; t < C; ++t)
      if (c + t < cols && n0 + c + t < a.N) {
        const long long o = ob + (long long)(n0 + c + t) * a.out_n;
        a.out[o] = LAM ? acc[t] * __ldg(a.inv_lam + o) : acc[t];
      }
  }
}

template <int KP, bool LAM>
__global__ void __launch_bounds__(kThreads, ctas_per_sm(KP)) split_pass_kernel(SplitArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sB = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bar_b[2], bar_full[2], bar_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ unsigned short s_ea[4][kM];
  __shared__ short s_eb[kM];
  __shared__ int s_fail, s_issued[2];     // commits on bar_full
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n0 = (int)blockIdx.y * a.NT;
  const int NTc = a.Np - n0 < a.NT ? a.Np - n0 : a.NT;     // columns of this CTA
  constexpr int nkc = (KP + 63) / 64;                      // 64-wide K chunks
  constexpr int KA = part_terms(KP);                       // terms of the first part
  constexpr int KR = KP - KA;                              // and of the second
  constexpr int scols = KA / 2;                            // TMEM columns per slice of A
  constexpr int dbase = kSlices * scols;                   // two accumulators follow
  constexpr int kNS = acc_cols(KP), kFirst = first_slices(KP);
  constexpr int kTmem = dbase + 2 * kNS > 256 ? 512 : 256; // allocated columns
  // B in shared memory: [slice][chunk][128 (64) rows][128 B] (row strides fixed, so
  // that descriptors are constants apart from the column block)
  constexpr int kChunk = b_rows(KP) * 128;
  constexpr int slice_bytes = nkc * kChunk;
  const int nsub = (NTc + kNS - 1) / kNS;

  // Already converged when this launch begins (the flag only rises within a
  // solve): leave before TMEM and B's digits are taken, still in stream order.
  if (a.done) {
    if (tid == 0) s_fail = *(volatile const double *)a.done != 0.0;
    __syncthreads();
    if (s_fail) {
      pdl_wait();
      pdl_trigger();
      return;
    }
    __syncthreads();
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar_b[i], 1);
      mbar_init(&bar_full[i], 1);
      mbar_init(&bar_empty[i], kWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = s_issued[0] = s_issued[1] = 0;
  }
  auto load_slices = [&](int s0, int s1, uint64_t *bar) {   // one thread
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"((uint32_t)((s1 - s0) * nkc * NTc * 128))
                 : "memory");
    for (int s = s0; s < s1; ++s)
      for (int c = 0; c < nkc; ++c)
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                smem_u32(sB + (size_t)s * slice_bytes + (size_t)c * kChunk)),
            "l"(a.img + ((size_t)(s * nkc + c) * a.Np + n0) * 128), "r"((uint32_t)(NTc * 128)),
            "r"(smem_u32(bar))
            : "memory");
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "n"(kTmem));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    if (lane == 0) load_slices(0, kFirst, &bar_b[0]);
  }
  const int rows_hi = a.range[0], rows_lo = a.range[1];
  for (int n = tid; n < NTc; n += kThreads)
    s_eb[n] = (short)(n0 + n < a.N ? a.eb[n0 + n] : 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  // barriers, TMEM and the first digits of B overlap the previous kernel's tail
  pdl_wait();
  pdl_trigger();
  if (a.done && *a.done != 0.0) {                          // uniform
    if (tid == 0) wait_on(&bar_b[0], 0, &s_fail);
    __syncthreads();
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmem));
    return;
  }

  if (rows_hi - rows_lo > kRowRange || rows_hi == 0x7ff) {  // uniform
    chain_rows<LAM>(a, n0, NTc);
    if (tid == 0) wait_on(&bar_b[0], 0, &s_fail);
    __syncthreads();
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmem));
    return;
  }

  // ---- A: this thread's row (lane 32 q + lane) and K range [kq KQ, kq KQ + KQ)
  // of a part ----
  const int q = warp & 3, kq = warp >> 2;
  constexpr int KQ = KA / 4;                               // 8, 16, 24 or 32
  const int lrow = q * 32 + lane;
  const long long m = (long long)blockIdx.x * kM + lrow;
  const bool row_ok = m < a.M;
  const long long hi = row_ok ? m / a.F : 0, lo = row_ok ? m - hi * a.F : 0;
  const int k0 = kq * KQ;
  const uint32_t lanes = (uint32_t)(q * 32) << 16;
  auto load_row = [&](int kb, double (&x)[KQ]) {           // terms kb + k0 ..
    if (a.in_k != 1) {
      const double *src = a.in + hi * a.in_hi + lo * a.in_lo + (long long)(kb + k0) * a.in_k;
#pragma unroll
      for (int i = 0; i < KQ; ++i)
        x[i] = (row_ok && kb + k0 + i < a.K) ? __ldg(src + (long long)i * a.in_k) : 0.0;
    } else {
      // rows contiguous in K: a warp reads runs of several rows at a time and
      // transposes through its own buffer (up to K = 128 in the part of shared
      // memory that the later digits of B take afterwards)
      constexpr int PW = KP > 128 ? 8 : 16;                // elements of a row per piece
      constexpr int TC = trans_cols(KP), HP = (KQ + PW - 1) / PW, RW = 32 / PW;
      double *buf = reinterpret_cast<double *>(sB + (size_t)kFirst * slice_bytes) + warp * 32 * TC;
      const long long base = row_ok ? hi * a.in_hi + lo * a.in_lo : -1;
      const int cc = lane % PW;
      // the 8-wide buffer is unpadded: its columns are exchanged by row instead
      auto at = [&](int r, int c) { return r * TC + (TC == 8 ? c ^ (r & 7) : c); };
      double y[HP][PW];
#pragma unroll
      for (int h = 0; h < HP; ++h) {
#pragma unroll
        for (int t = 0; t < PW; ++t) {
          const int k = kb + k0 + PW * h + cc;
          const long long b = __shfl_sync(0xffffffffu, base, RW * t + lane / PW);
          const bool ok = b >= 0 && PW * h + cc < KQ && k < a.K;
          y[h][t] = ok ? __ldg(a.in + b + k) : 0.0;
        }
      }
#pragma unroll
      for (int h = 0; h < HP; ++h) {
        __syncwarp();
#pragma unroll
        for (int t = 0; t < PW; ++t) buf[at(RW * t + lane / PW, cc)] = y[h][t];
        __syncwarp();
#pragma unroll
        for (int t = 0; t < PW; ++t)
          if (PW * h + t < KQ) x[PW * h + t] = buf[at(lane, t)];
      }
      __syncwarp();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
  };
  auto largest = [&](const double (&x)[KQ], int em) {
#pragma unroll
    for (int i = 0; i < KQ; ++i) em = max(em, exp_field((uint32_t)__double2hiint(x[i])));
    return em;
  };
  // the digits of a part into TMEM
  auto put_digits = [&](const double (&x)[KQ], int ea) {
    uint32_t w1[KQ], w0[KQ];
#pragma unroll
    for (int i = 0; i < KQ; ++i) biased_fixed(x[i], ea, w1[i], w0[i]);
    auto put = [&](int s, auto pos, const uint32_t *w) {
      constexpr int POS = decltype(pos)::value;
#pragma unroll
      for (int b = 0; b < KQ / 8; ++b)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                         tmem + lanes + (uint32_t)(s * scols + (k0 >> 1) + 4 * b)),
                     "r"(digit2<POS>(w[8 * b], w[8 * b + 1])),
                     "r"(digit2<POS>(w[8 * b + 2], w[8 * b + 3])),
                     "r"(digit2<POS>(w[8 * b + 4], w[8 * b + 5])),
                     "r"(digit2<POS>(w[8 * b + 6], w[8 * b + 7]))
                     : "memory");
    };
    put(0, std::integral_constant<int, 2>{}, w1);
    put(1, std::integral_constant<int, 1>{}, w1);
    put(2, std::integral_constant<int, 0>{}, w1);
    put(3, std::integral_constant<int, 2>{}, w0);
    put(4, std::integral_constant<int, 1>{}, w0);
    put(5, std::integral_constant<int, 0>{}, w0);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  };
  int ea;
  {
    double x[KQ];
    int em = 1;
    if constexpr (KR > 0) {                                // the second part's exponents too
      load_row(KA, x);
      em = largest(x, em);
    }
    load_row(0, x);
    if (LAM && row_ok && (lane & 15) == 0) {               // the divide's table, used last
      const double *t = a.inv_lam + hi * a.out_hi + lo * a.out_lo + (long long)n0 * a.out_n;
      for (int n = kq; n < NTc && n0 + n < a.N; n += 4)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(t + (long long)n * a.out_n));
    }
    s_ea[kq][lrow] = (unsigned short)largest(x, em);
    __syncthreads();
    if (kFirst < kSlices && tid == 0) load_slices(kFirst, kSlices, &bar_b[1]);
    ea = max(max((int)s_ea[0][lrow], (int)s_ea[1][lrow]), max((int)s_ea[2][lrow], (int)s_ea[3][lrow]));
    put_digits(x, ea);
  }

  // ---- digit products. A step's MMAs are issued by one elected lane of warp
  // step mod 16, while the others sum the step before. (Elected by elect.sync,
  // so that descriptors stay in uniform registers: an MMA then issues in its
  // execution time, 31 clocks, instead of 45-120 from a lane picked by index;
  // a seventeenth warp for the issue alone would leave 96 registers a thread
  // and spill.) ----
  const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
  const uint64_t b0 = sw128_desc(smem_u32(sB));
  bool ok = true;
  // K terms of part `part` (KT of them, from chunk c0), group and chunks of step i
  auto issue = [&](auto part, auto step, int sub, int st) {   // one warp
    constexpr int i = decltype(step)::value, part_ = decltype(part)::value;
    constexpr int KT = part_ ? KR : KA, kc0 = part_ ? KA / 64 : 0;
    constexpr Step p = Steps<KT>::at(i);
    const int buf = st & 1;
    if (sub == 0) {                                        // (a poll each once they have arrived)
      constexpr unsigned waits = step_waits(KP, p.g);
      if (waits & 1u) ok = ok && wait_on(&bar_b[0], 0, &s_fail, a.polls);
      if (waits & 2u) ok = ok && wait_on(&bar_b[1], 0, &s_fail, a.polls);
    }
    if (st >= 2) ok = ok && wait_on(&bar_empty[buf], (uint32_t)(((st >> 1) - 1) & 1), &s_fail, a.polls);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) return;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int nc = NTc - sub * kNS < kNS ? NTc - sub * kNS : kNS;
    const uint32_t idesc = (1u << 4) | ((uint32_t)(nc >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
    const uint32_t d = tm + (uint32_t)(dbase + buf * kNS);
    uint32_t elected;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(elected));
    const uint64_t bsub = b0 + (uint32_t)(sub * kNS * 128 >> 4);   // (descriptor steps of 16 bytes)
    if (elected) {
#pragma unroll
      for (int sl = 0; sl <= p.g; ++sl) {
        if (!(p.prods >> sl & 1u)) continue;
        const uint64_t bs = bsub + (uint32_t)((p.g - sl) * slice_bytes >> 4);
#pragma unroll
        for (int ks = p.k0; ks < p.k1; ++ks) {
          const uint32_t acc = (p.prods & ((1u << sl) - 1u)) == 0u && ks == p.k0 ? 0u : 1u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
              "r"(tm + (uint32_t)(sl * scols + ks * 8)),
              "l"(bs + (uint64_t)(((ks >> 2) + kc0) * (kChunk >> 4) + (ks & 3) * 2)), "r"(idesc), "r"(acc));
        }
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              smem_u32(&bar_full[buf]))
          : "memory");
      s_issued[buf] = (st >> 1) + 1;
    }
    __syncwarp();
  };
  // ---- accumulators to integers, rounded once ----
  constexpr int C = kNS / 4;                               // columns per thread in a block
  const bool bad_row = ea == 0x7ff;
  const long long ob = hi * a.out_hi + lo * a.out_lo;
  constexpr int kTop = KR > 0 ? 38 : 39;                   // weight of group 0 in T
  int st = 0;
  if (warp == 0) issue(std::integral_constant<int, 0>{}, std::integral_constant<int, 0>{}, 0, 0);
  for (int sub = 0; sub < nsub; ++sub) {
    long long T[C] = {};
    auto sum = [&](auto part, auto step) {
      constexpr int i = decltype(step)::value, part_ = decltype(part)::value;
      constexpr int KT = part_ ? KR : KA, per = Steps<KT>::kCount;
      constexpr int g = Steps<KT>::at(i).g;
      const int buf = st & 1;
      if (warp == ((st + 1) & (kWarps - 1)) && (i + 1 < per || (KR == 0 && sub + 1 < nsub)))
        issue(part, std::integral_constant<int, (i + 1) % per>{}, i + 1 < per ? sub : sub + 1, st + 1);
      ok = ok && wait_on(&bar_full[buf], (uint32_t)((st >> 1) & 1), &s_fail, a.polls);
      ok = __all_sync(0xffffffffu, ok);
      ++st;
      if (!ok) {
        s_fail = 1;
        return;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t v[C];
      const uint32_t dv = tmem + lanes + (uint32_t)(dbase + buf * kNS + kq * C);
      if constexpr (C == 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                       "=r"(v[6]), "=r"(v[7])
                     : "r"(dv));
      else
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
            "%14,%15}, [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
              "=r"(v[14]), "=r"(v[15])
            : "r"(dv));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_empty[buf]);
      // T in units of 2^11 (2^12 with two parts) of group 5: |G_0| 2^kTop <=
      // 2^62; what is dropped of groups 4 and 5 is of the order of the groups
      // not computed
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const int G = __float2int_rn(__uint_as_float(v[c]));
        constexpr int w = kTop - 10 * g;                   // 2^w: the group's weight
        if (g == 0) T[c] = (part_ ? T[c] : 0) + ((long long)G << kTop);
        else if (w >= 0) T[c] += (long long)G * (1 << (w >= 0 && w < 31 ? w : 0));
        else T[c] += (long long)((G + (1 << (w < 0 ? -w - 1 : 0))) >> (w < 0 ? -w : 0));
      }
    };
    auto sum_part = [&](auto part) {
      each_step<Steps<decltype(part)::value ? KR : KA>::kCount>([&](auto step) { sum(part, step); });
    };
    sum_part(std::integral_constant<int, 0>{});
    if constexpr (KR > 0) {                                // (one column block)
      constexpr std::integral_constant<int, 1> second{};
      double x[KQ];
      load_row(KA, x);
      __syncthreads();                                     // every MMA on the first digits is done
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      put_digits(x, ea);
      if (warp == (st & (kWarps - 1))) issue(second, std::integral_constant<int, 0>{}, 0, st);
      sum_part(second);
    }
    if (!row_ok) continue;
    const int nl0 = sub * kNS + kq * C;                  // this thread's first column, and how many
    const int ncol = min(C, min(NTc - nl0, a.N - n0 - nl0));
    const long long o0 = ob + (long long)(n0 + nl0) * a.out_n;
    double lam[C];
#pragma unroll
    for (int c = 0; c < C; ++c) lam[c] = LAM && c < ncol ? __ldg(a.inv_lam + o0 + c * a.out_n) : 1.0;
    const bool bad = bad_row || !ok;                     // !ok: NaN, never what the buffer held before
    bool slow = bad;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const double y = round_fixed<LAM>(T[c], ea + (int)s_eb[(nl0 + c) & (kM - 1)] - 2060 - kTop, lam[c], slow);
      if (c < ncol) a.out[o0 + c * a.out_n] = y;
    }
    if (slow) {                                          // rare: again, one by one
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (c < ncol)
          a.out[o0 + c * a.out_n] =
              bad ? __longlong_as_double(0x7ff8000000000000ll)
                      : round_slow(T[c], ea + (int)s_eb[nl0 + c] - 2060 - kTop, lam[c]);
    }
  }
  if (!ok) s_fail = 1;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && s_fail) {
    atomicExch(a.err, (int)IGAFD_ERR_TIMEOUT);
    // a wait ran out: give the copies and MMAs in flight a bounded chance to
    // finish before shared memory and TMEM are released
    const int none = 0;
    wait_on(&bar_b[0], 0, &none);
    if (kFirst < kSlices) wait_on(&bar_b[1], 0, &none);
    for (int i = 0; i < 2; ++i)
      if (s_issued[i]) wait_on(&bar_full[i], (uint32_t)((s_issued[i] - 1) & 1), &none);
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmem));
}

// Digits of B = U_k^T (transpose) or U_k as the shared-memory images of the
// pass kernel, and the exponent field of each row: one CTA per (row, image).
// U_k's columns are brought to one size by powers of two s_j first (outlier
// eigenvectors are large at the ends, 2^4.4 times the others at n = 128, p = 3,
// and would take those bits from the rest of a row): the forward product's
// column j is raised by s_j, U_k's lowered; between the two only the range of
// the intermediate values moves, by 2^4 or so. Without it constant right-hand
// sides at n = 120, p = 7 were off by 1.2e-14 (FP64 chains 1.8e-15, now 0.4e-15).
// The forward images are made first.
struct ImgJob {
  const double *U;
  int n, Np, Kp, transpose;
  unsigned char *img;
  int *eb;
  int *col;       // s_j, set by the forward image
  int *range;     // largest and smallest exponent field of U_k's rows
};
struct ImgBatch {
  ImgJob j[3];
};
__global__ void __launch_bounds__(256) split_image_kernel(ImgBatch b) {
  const ImgJob J = b.j[blockIdx.y];
  const int r = blockIdx.x, k = threadIdx.x;
  if (r >= J.Np) return;
  __shared__ int s_e[2][8];
  const int nkc = (J.Kp + 63) >> 6;
  double d = 0.0;
  int s = 0;
  if (r < J.n && k < J.n) {
    d = J.transpose ? J.U[(size_t)k * J.n + r] : J.U[(size_t)r * J.n + k];
    if (!J.transpose) s = J.col[k];
  }
  int raw = exp_field((uint32_t)__double2hiint(d)), e = raw - s;
  for (int o = 16; o > 0; o >>= 1) {
    raw = max(raw, __shfl_xor_sync(0xffffffffu, raw, o));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  }
  if ((k & 31) == 0) {
    s_e[0][k >> 5] = raw;
    s_e[1][k >> 5] = e;
  }
  __syncthreads();
  for (int w = 0; w < 8; ++w) {
    raw = max(raw, s_e[0][w]);
    e = max(e, s_e[1][w]);
  }
  if (k == 0 && J.transpose) {
    const int up = r < J.n ? max(-64, min(64, e - 1023)) : 0;
    if (r < J.n) J.col[r] = up;
    J.eb[r] = e + up;
    if (r == 0) {
      J.range[0] = 0;
      J.range[1] = 0x7ff;
    }
  } else if (k == 0) {
    J.eb[r] = e;
    if (r < J.n) {
      atomicMax(&J.range[0], raw);
      atomicMin(&J.range[1], raw);
    }
  }
  if (k >= nkc * 64) return;
  uint32_t w1, w0;
  biased_fixed(d, e, w1, w0, s);
  const int kb = (k & 63) * 2;
  unsigned char *at = J.img + ((size_t)(k >> 6) * J.Np + r) * 128 + ((((kb >> 4) ^ (r & 7)) << 4) | (kb & 15));
  const size_t slice = (size_t)nkc * J.Np * 128;
  auto put = [&](int i, uint32_t w) { *reinterpret_cast<unsigned short *>(at + i * slice) = (unsigned short)w; };
  put(0, digit2<2>(w1, w1));
  put(1, digit2<1>(w1, w1));
  put(2, digit2<0>(w1, w1));
  put(3, digit2<2>(w0, w0));
  put(4, digit2<1>(w0, w0));
  put(5, digit2<0>(w0, w0));
}

int pad(int n, int to) { return (n + to - 1) / to * to; }

size_t pass_smem(int Kp) {
  const size_t slice = (size_t)((Kp + 63) / 64) * b_rows(Kp) * 128;
  const size_t a = kSlices * slice, b = first_slices(Kp) * slice + trans_bytes(Kp);
  return 1024 + (a > b ? a : b);
}

}  // namespace

struct FDSplit {
  unsigned char *mem;         // one allocation for all below
  unsigned char *img[3][2];   // [direction][0: U_k^T, 1: U_k]
  int *eb[3][2];
  int *col[3];                // column scalings of U_k (exponents), then its rows' range (2)
};

bool igafd_fd_split_shape(const igafd_patch *P) {
  for (int k = 0; k < P->dim; ++k)
    if (P->n[k] > 256) return false;
  return true;
}

// Digit images of U_k^T and U_k. Allocates on the first call; later calls (a
// re-setup of P) refill the same buffers. Enqueues two kernels.
igafd_status igafd_fd_split_init(igafd_patch *P, cudaStream_t s) {
  if (!igafd_fd_split_shape(P)) return IGAFD_OK;
  if (!P->split) {
    P->split = (FDSplit *)calloc(1, sizeof(FDSplit));
    if (!P->split) return IGAFD_ERR_OOM;
  }
  FDSplit &S = *P->split;
  if (!S.mem) {
    // sizes first, then addresses, each on a 256-byte boundary
    for (int set = 0; set < 2; ++set) {
      size_t at = 0;
      auto take = [&](size_t bytes) {
        unsigned char *q = S.mem + (set ? at : 0);
        at += (bytes + 255) / 256 * 256;
        return q;
      };
      for (int k = 0; k < P->dim; ++k) {
        const int n = P->n[k], Np = pad(n, 16), Kp = pad(n, 32);
        S.col[k] = (int *)take((n + 2) * sizeof(int));
        for (int d = 0; d < 2; ++d) {
          S.img[k][d] = take((size_t)kSlices * ((Kp + 63) / 64) * Np * 128);
          S.eb[k][d] = (int *)take(Np * sizeof(int));
        }
      }
      if (!set && cudaMalloc(&S.mem, at) != cudaSuccess) {
        cudaGetLastError();
        S.mem = nullptr;
        return IGAFD_ERR_OOM;
      }
    }
  }
  ImgBatch b[2] = {};
  int rows = 0;
  for (int k = 0; k < P->dim; ++k)
    for (int d = 0; d < 2; ++d) {
      ImgJob &J = b[d].j[k];
      J.U = P->U[k]; J.n = P->n[k]; J.Np = pad(J.n, 16); J.Kp = pad(J.n, 32);
      J.transpose = d == 0;
      J.img = S.img[k][d];
      J.eb = S.eb[k][d];
      J.col = S.col[k];
      J.range = J.col + J.n;
      rows = J.Np > rows ? J.Np : rows;
    }
  for (int d = 0; d < 2; ++d) split_image_kernel<<<dim3(rows, P->dim), 256, 0, s>>>(b[d]);
  IGAFD_LAUNCHED(2);
  IGAFD_CUDA(cudaGetLastError());
  return IGAFD_OK;
}

void igafd_fd_split_free(igafd_patch *P) {
  if (!P || !P->split) return;
  cudaFree(P->split->mem);
  free(P->split);
  P->split = nullptr;
}

// One mode product: rows m = hi F + lo at in + hi in_hi + lo in_lo + k in_k.
static igafd_status launch_pass(igafd_patch *P, int k, int dir, SplitArgs a, cudaStream_t s) {
  a.K = a.N = P->n[k];
  a.Kp = pad(a.K, 32);
  a.Np = pad(a.N, 16);
  a.img = P->split->img[k][dir];
  a.eb = P->split->eb[k][dir];
  a.range = P->split->col[k] + P->n[k];
  a.U = P->U[k];
  a.u_j = dir == 0 ? 1 : a.N;
  a.u_k = dir == 0 ? a.N : 1;
  a.err = P->err_flag;
  a.polls = P->wait_polls;
  // Column split: with fewer 128-row tiles than SMs, a CTA's columns are
  // halved while all CTAs still fit one wave (a CTA's time is about half the
  // splitting of its rows, which every column part repeats, and half the
  // digit products, which shrink with the columns).
  const long long tiles = (a.M + kM - 1) / kM;
  int parts = 1;
  while (parts < 8 && tiles * parts * 2 <= P->num_sms && pad(a.Np, 32 * parts) / parts > 16) parts *= 2;
  if (a.Kp > 128) parts = parts < (a.Np + 63) / 64 ? (a.Np + 63) / 64 : parts;
  a.NT = pad((a.Np + parts - 1) / parts, 16);
  parts = (a.Np + a.NT - 1) / a.NT;
  const size_t smem = pass_smem(a.Kp);
  using Kern = void (*)(SplitArgs);
#define IGAFD_SPLIT(K) {split_pass_kernel<K, false>, split_pass_kernel<K, true>}
  static const Kern kerns[8][2] = {IGAFD_SPLIT(32),  IGAFD_SPLIT(64),  IGAFD_SPLIT(96),  IGAFD_SPLIT(128),
                                   IGAFD_SPLIT(160), IGAFD_SPLIT(192), IGAFD_SPLIT(224), IGAFD_SPLIT(256)};
#undef IGAFD_SPLIT
  static std::atomic<unsigned long long> attr_set{0};
  const unsigned long long bit = 1ull << (P->dev & 63);
  if (!(attr_set.load() & bit)) {
    for (int i = 0; i < 16; ++i)
      IGAFD_CUDA(cudaFuncSetAttribute(kerns[i / 2][i % 2], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)pass_smem(32 * (i / 2 + 1))));
    attr_set.fetch_or(bit);
  }
  IGAFD_CUDA(igafd_launch(kerns[a.Kp / 32 - 1][a.inv_lam ? 1 : 0], dim3((unsigned)tiles, (unsigned)parts),
                          dim3(kThreads), smem, s, a));
  IGAFD_LAUNCHED(1);
  return IGAFD_OK;
}

// z = P^{-1} r. 3D: [i3][i2][i1] -> [j3][i2][i1] -> [j3][j2][i1] ->
// [j1][j3][j2] (divided) -> [i1][j3][j2] -> [i1][i3][j2] -> [i3][i2][i1];
// 2D: [i2][i1] -> [j2][i1] -> [j1][j2] (divided) -> [i1][j2] -> [i2][i1].
igafd_status igafd_fd_split_apply(igafd_patch *P, const double *r, double *z, cudaStream_t s,
                                  double *done_flag) {
  if (!P->split) return IGAFD_ERR_ARG;
  const long long n1 = P->n[0], n2 = P->n[1], n3 = P->dim == 3 ? P->n[2] : 1;
  const long long n12 = n1 * n2, n23 = n2 * n3;
  double *t1 = P->fd_a, *t2 = P->fd_b;
  SplitArgs a{};
  a.done = done_flag;
  auto pass = [&](int k, int dir, const double *in, double *out, long long M, long long F,
                  long long in_hi, long long in_lo, long long in_k, long long out_hi,
                  long long out_lo, long long out_n, const double *inv_lam) {
    a.in = in; a.out = out; a.M = M; a.F = (int)F;
    a.in_hi = in_hi; a.in_lo = in_lo; a.in_k = in_k;
    a.out_hi = out_hi; a.out_lo = out_lo; a.out_n = out_n;
    a.inv_lam = inv_lam;
    return launch_pass(P, k, dir, a, s);
  };
  if (P->dim == 3) {
    IGAFD_TRY(pass(2, 0, r, t1, n12, n12, 0, 1, n12, 0, 1, n12, nullptr));
    IGAFD_TRY(pass(1, 0, t1, t2, n1 * n3, n1, n12, 1, n1, n12, 1, n1, nullptr));
    IGAFD_TRY(pass(0, 0, t2, t1, n23, n23, 0, n1, 1, 0, 1, n23, P->inv_lam));
    IGAFD_TRY(pass(0, 1, t1, t2, n23, n23, 0, 1, n23, 0, 1, n23, nullptr));
    IGAFD_TRY(pass(2, 1, t2, t1, n12, n2, n23, 1, n2, n23, 1, n2, nullptr));
    // rows m = i3 n1 + i1 of [i1][i3][j2], contiguous in j2
    return pass(1, 1, t1, z, n1 * n3, n1, n2, n23, 1, n12, 1, n1, nullptr);
  }
  IGAFD_TRY(pass(1, 0, r, t1, n1, n1, 0, 1, n1, 0, 1, n1, nullptr));
  IGAFD_TRY(pass(0, 0, t1, t2, n2, n2, 0, n1, 1, 0, 1, n2, P->inv_lam));
  IGAFD_TRY(pass(0, 1, t2, t1, n2, n2, 0, 1, n2, 0, 1, n2, nullptr));
  return pass(1, 1, t1, z, n1, n1, 0, n2, 1, 0, 1, n1, nullptr);
}
