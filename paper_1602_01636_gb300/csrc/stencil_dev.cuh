// Device code shared by the single-problem and batched stencil kernels:
// the stencil layout, the arguments, the per-CTA pipeline and the ring set-up.
#pragma once
// y = A x with A stored as a (2p+1)^d-point FP64 stencil, offset-major:
// S[o][row] with row stride Np (N rounded up to kTile), o = sum_k
// (delta_k + p)(2p+1)^(k-1) (Section 2.1: an interior row of A couples to
// (2p+1)^d columns). Also r = b - A x (true residual).
//
// On GB300 the 343 FP64 FMAs of a p = 3 row take longer on the FP64 pipe
// (2 FMA/clk/SM) than its 2.7 KB of coefficients take to stream from HBM, so
// the kernel is built to keep the FP64 pipe fed from shared memory: a
// persistent grid of CTAs walks tiles of 64 to 256 rows (tile_rows); for every
// (delta_2, delta_3) group a producer warp brings the 2p+1 coefficient runs of
// the tile (contiguous) and the contiguous window of x they multiply into a
// shared-memory ring with bulk asynchronous copies (cp.async.bulk, completion
// on mbarriers), several groups ahead of the eight compute warps. x is read
// from a copy with a zero halo of p planes on both ends, and couplings that
// leave the index box are stored as 0, so every row runs the same
// branch-free (2p+1)^d FMAs and no read leaves the allocation. Every
// mbarrier wait is bounded: on timeout the kernel records an error, waits
// (bounded) for its own copies and returns. Optional fused dot with a
// deterministic last-block reduction.
#include "common.cuh"

#include <atomic>
#include <cstring>

namespace {

constexpr int kTile = 256;                        // rows per tile at most (StencilArgs::tile in use)
constexpr int kSolveTile = 128;                   // and at least in a solve (tile_rows)
// ring depths (offset groups in flight per CTA) the kernel is built for; the
// autotuner picks one per (dimension, degree, sizes), default kStagesDefault
constexpr int kStagesDefault = 4;
constexpr long long kSpin = 1ll << 26;   // mbarrier poll limit (~seconds)

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Bounded wait; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
  for (long long i = 0; i < kSpin; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// Last block of a grid-stride reduction: returns true in every thread of the
// block that finished last (all partials visible).
__device__ __forceinline__ bool last_block(unsigned int *counter, unsigned blocks) {
  __shared__ bool am_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned t = atomicAdd(counter, 1u);
    am_last = (t == blocks - 1);
  }
  __syncthreads();
  return am_last;
}

__device__ double sum_partials(const double *part, int n, double *sh32) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += ((volatile const double *)part)[i];
  return block_sum(v, sh32);
}

struct StencilArgs {
  const double *S;    // [n_off][Np]
  const double *x;    // interior pointer of a zero-padded vector (halo H)
  double *y;
  const double *b;    // MODE 1
  const double *z;    // MODE 1, optional: also (y, z) -> scal[S_RZOLD] (flexible beta)
  int n1, n2, n3;
  long long N, Np;
  long long pad;      // rows the stencil arrays hold (N rounded up to kTile)
  int tile;           // rows per tile (a multiple of 64 with two rows per thread, else of 32)
  long long ntiles;
  double *partial;    // null: no dot
  unsigned *counter;
  double *scal;       // PCG scalars (pcg != 0)
  int pcg;
  const double *done; // skip when *done != 0
  int *err;           // set on an mbarrier timeout
  int every;          // > 0: run only when scal[S_ITER] is a multiple of every
  unsigned long long *tstat;  // optional device timing (see igafd_patch::tstat)
  // half-stored stencil (the HALF kernels): S is [(n_off + 1) / 2][Np] with
  // Np the row stride, offsets from oc (the centre) up, row i at shH + i
  int oc;
  long long shH;
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

template <int P, bool HALF = false>
struct Geom {
  static constexpr int W = 2 * P + 1;
  // coefficient run stride in a ring stage: a tile, or (half-stored stencil)
  // a tile and two rows, so that a mirrored run can start one row early
  static constexpr int RS = HALF ? kTile + 2 : kTile;
  static constexpr int XW = (kTile + 2 * P + 2 + 1) & ~1;   // x window (even count)
  static constexpr int STAGE = W * RS + XW;                  // doubles per ring stage
};

// Warp-specialised pipeline: the compute warps take R consecutive rows per
// thread (R = 1: warps 0..7, one row each; R = 2: warps 0..3, two rows each,
// reading both rows' coefficients and the shared x values with 16-byte
// shared-memory loads, which halves the load instructions per FMA); the next
// warp (one elected lane) streams, for every (delta_2, delta_3) group, the
// 2p+1 coefficient runs of the tile and the x window they multiply into a
// ring of kStages shared-memory stages (full/empty mbarriers). The FP64 FMAs
// read both operands from shared memory.
//
// MODE 0: y = A x, dot (x, y) -> alpha = rho / (x, y) when pcg.
// MODE 1: y = b - A x, dot (y, y) -> true (r, r) when pcg; with z given also
// (y, z) -> (r, z_old) of the flexible beta, so that a recomputed residual
// replaces the recurrence one in every scalar that uses it.
// One CTA's share of the product, as CTA vb of a grid of vgrid CTAs: tiles
// vb, vb + vgrid, ..., the fused dot, and (in the CTA that finishes last) the
// dot's fixed-order sum over the vgrid partial sums. The ring's barriers are
// initialised by the caller; gstage counts the ring stages this CTA has
// passed through so far, so a persistent CTA can keep its ring across calls.
//
// HALF: the stencil is stored by its symmetry (offsets from the centre up).
// The run of a stored offset o is S[o - oc][shH + row0 ...]; the run of an
// offset o below the centre (delta < 0) is the mirrored offset's run shifted
// by off(delta) rows, S[mirror(o) - oc][shH + row0 + off ...], fetched from
// the even row at or before its start so that every bulk copy is 16-byte
// aligned; every run is two rows longer than the tile (RS = kTile + 2 apart in
// shared memory) and the compute warps read a mirrored run one row later when
// its start was odd.
template <int DIM, int P, int MODE, int kStages, int R, bool HALF = false>
__device__ __forceinline__ void stencil_cta(const StencilArgs &a, long long vb, long long vgrid,
                                            double *ring, uint64_t *full, uint64_t *empty,
                                            long long &gstage, volatile int *s_abort) {
  using Gm = Geom<P, HALF>;
  constexpr int W = Gm::W;
  constexpr int RS = Gm::RS;
  constexpr int NOFF = DIM == 3 ? W * W * W : W * W;
  constexpr int G = DIM == 3 ? W * W : W;        // (delta_2, delta_3) groups per tile
  constexpr int kCompute = kTile / R;            // compute threads
  constexpr int NV = ((W + 1) / 2 + 1) * 2;      // x values a two-row thread holds
  static_assert(R == 1 || R == 2, "one or two rows per thread");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int my_tiles = (int)(a.ntiles > vb ? (a.ntiles - 1 - vb) / vgrid + 1 : 0);
  const long long total = (long long)my_tiles * G;
  const long long n12 = (long long)a.n1 * a.n2;
  const long long g0 = gstage;                   // global index of this call's first stage
  const int h = a.tile;
  // ring position, advanced step by step (a step: one (delta_2, delta_3)
  // group of one tile): slot, and how often the ring has come round
  int slot = (int)(g0 % kStages);
  uint32_t turn = (uint32_t)(g0 / kStages);
  constexpr int D3 = DIM == 3 ? W : 1;           // delta_3 values

  double dot = 0.0, dot2 = 0.0;
  if (warp == kCompute / 32) {
    // ---------------- producer warp ----------------
    if (lane == 0) {
      long long issued = 0;
      bool ok = true;
      const uint32_t xrun = (uint32_t)(((h + 2 * P + 3) & ~1) * sizeof(double));
      long long row0 = vb * h;
      for (int t = 0; t < my_tiles && ok; ++t, row0 += vgrid * h) {
        // the last tile's rows end with the arrays (both multiples of 32)
        const int rows = (int)(a.pad - row0 < h ? a.pad - row0 : h);
        const uint32_t run = (uint32_t)((HALF ? rows + 2 : rows) * sizeof(double));
        int ob = 0;                                        // first offset of the group
#pragma unroll 1
        for (int d3 = 0; d3 < D3 && ok; ++d3) {
          const long long off3 = DIM == 3 ? (d3 - P) * n12 : 0;
#pragma unroll 1
          for (int d2 = 0; d2 < W; ++d2, ob += W) {
            if (turn > 0) {
              long long it = 0;
              while (!mbar_try_wait(&empty[slot], (turn - 1) & 1)) {
                if (*s_abort || ++it > kSpin) { ok = false; break; }
              }
              if (!ok) break;
            }
            const long long off23 = off3 + (long long)(d2 - P) * a.n1;
            long long x0 = row0 + off23 - P;
            x0 -= (x0 & 1);                                // 16-byte aligned start
            double *st = ring + (size_t)slot * Gm::STAGE;
            uint64_t *bar = &full[slot];
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive_tx(bar, W * run + xrun);
            if constexpr (!HALF) {
              const double *src = a.S + (size_t)ob * a.Np + row0;
#pragma unroll
              for (int d1 = 0; d1 < W; ++d1) bulk_g2s(st + d1 * kTile, src + (size_t)d1 * a.Np, run, bar);
            } else {
              for (int d1 = 0; d1 < W; ++d1) {
                const int o = ob + d1;
                long long start = a.shH + row0;
                int arr = o - a.oc;
                if (o < a.oc) {                            // delta < 0: the mirrored run
                  arr = NOFF - 1 - o - a.oc;
                  start += (d1 - P) + off23;
                }
                start -= (start & 1);
                bulk_g2s(st + d1 * RS, a.S + (size_t)arr * a.Np + start, run, bar);
              }
            }
            bulk_g2s(st + W * RS, a.x + x0, xrun, bar);
            ++issued;
            if (++slot == kStages) { slot = 0; ++turn; }
          }
        }
      }
      if (!ok) {
        *s_abort = 1;
        atomicExch(a.err, (int)IGAFD_ERR_TIMEOUT);
      }
      // never leave with copies in flight: wait (bounded) for the last stages issued
      for (long long q = issued - kStages > 0 ? issued - kStages : 0; q < issued; ++q)
        mbar_wait(&full[(g0 + q) % kStages], (uint32_t)(((g0 + q) / kStages) & 1));
    }
  } else {
    // ---------------- compute warps ----------------
    // Two accumulators per row (even and odd offsets of a run): the FMA
    // chains of a warp are then short enough that a CTA alone on its SM (the
    // last tiles, small patches) is not held up by the FMA latency.
    bool ok = true;
    const int t0 = R * tid;                      // first of this thread's R rows in the tile
    long long row0 = vb * h;
    for (int t = 0; t < my_tiles && ok; ++t, row0 += vgrid * h) {
      const long long row = row0 + t0;
      double acc[R][2];
      bool live[R];
      // bit d of v2, v3: (i_2 + d - P, i_3 + d' - P) inside the box
      uint32_t v2[R], v3[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r][0] = acc[r][1] = 0.0;
        live[r] = t0 + r < h && row + r < a.N;
        const uint32_t j = (uint32_t)(row + r) / (uint32_t)a.n1;
        const int i2 = (int)(j % (uint32_t)a.n2), i3 = DIM == 3 ? (int)(j / (uint32_t)a.n2) : 0;
        v2[r] = v3[r] = 0u;
#pragma unroll
        for (int d = 0; d < W; ++d) {
          if (live[r] && (unsigned)(i2 + d - P) < (unsigned)a.n2) v2[r] |= 1u << d;
          if (live[r] && (DIM == 2 || (unsigned)(i3 + d - P) < (unsigned)a.n3)) v3[r] |= 1u << d;
        }
      }
      const int odd0 = (int)((row0 - P) & 1), odd1 = a.n1 & 1, odd12 = (int)(n12 & 1);
      int ob = 0;
#pragma unroll 1
      for (int d3 = 0; d3 < D3 && ok; ++d3) {
#pragma unroll 1
        for (int d2 = 0; d2 < W; ++d2, ob += W) {
          long long it = 0;
          while (!mbar_try_wait(&full[slot], turn & 1)) {
            if (*s_abort || ++it > kSpin) { ok = false; break; }
          }
          if (!ok) {
            *s_abort = 1;
            atomicExch(a.err, (int)IGAFD_ERR_TIMEOUT);
            break;
          }
          // the x window starts sh elements before row0 + off(0, d2, d3) - P
          const int sh = odd0 ^ ((d2 - P) & odd1 & 1) ^ (DIM == 3 ? (d3 - P) & odd12 & 1 : 0);
          const double *st = ring + (size_t)slot * Gm::STAGE;
          // rows whose (i_2 + delta_2, i_3 + delta_3) leaves the box have only
          // zero coefficients in this group; skip when the whole warp is out
          bool in23 = false;
#pragma unroll
          for (int r = 0; r < R; ++r) in23 = in23 || ((v2[r] >> d2) & (DIM == 3 ? v3[r] >> d3 : 1u) & 1u);
          // the slot is free once the group's operands are in registers
          auto release = [&]() {
            __syncwarp();
            if (lane == 0)
              asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[slot])) : "memory");
          };
          if (!__any_sync(0xffffffffu, in23)) {
            release();
          } else {
            // HALF: a mirrored run is read one row late when its start row was odd
            if constexpr (R == 1) {
              const double *cf = st + t0;
              const double *xw = st + W * RS + t0 + sh;       // xw[j] = x[row + off - P + j]
              double c[W], x[W];
#pragma unroll
              for (int j = 0; j < W; ++j) {
                const int hs = HALF && ob + j < a.oc ? (int)((a.shH & 1) ^ sh ^ (j & 1)) : 0;
                c[j] = cf[j * RS + hs];
                x[j] = xw[j];
              }
              release();
#pragma unroll
              for (int j = 0; j < W; ++j) acc[0][j & 1] = fma(c[j], x[j], acc[0][j & 1]);
            } else if constexpr (HALF) {
              // rows row, row + 1: two 8-byte loads per run (no branch on the
              // shift); x[row + off - P + j] = xv[j + sh], of the next row xv[j + 1 + sh]
              const double *cf = st + t0;
              const double2 *xb = reinterpret_cast<const double2 *>(st + W * RS + t0);
              double xv[NV];
#pragma unroll
              for (int m = 0; m < NV / 2; ++m) { const double2 v = xb[m]; xv[2 * m] = v.x; xv[2 * m + 1] = v.y; }
              double c0[W], c1[W];
#pragma unroll
              for (int j = 0; j < W; ++j) {
                const int hs = ob + j < a.oc ? (int)((a.shH & 1) ^ sh ^ (j & 1)) : 0;
                c0[j] = cf[j * RS + hs];
                c1[j] = cf[j * RS + hs + 1];
              }
              release();
#pragma unroll
              for (int j = 0; j < W; ++j) {
                const double xa = sh ? xv[j + 1] : xv[j], xc = sh ? xv[j + 2] : xv[j + 1];
                acc[0][j & 1] = fma(c0[j], xa, acc[0][j & 1]);
                acc[1][j & 1] = fma(c1[j], xc, acc[1][j & 1]);
              }
            } else {
              // rows row, row + 1: coefficients c[j] = (S[o_j][row], S[o_j][row + 1]);
              // x[row + off - P + j] = xv[j + sh], x[row + 1 + off - P + j] = xv[j + 1 + sh]
              const double2 *cf = reinterpret_cast<const double2 *>(st + t0);
              const double2 *xb = reinterpret_cast<const double2 *>(st + W * kTile + t0);
              double xv[NV];
#pragma unroll
              for (int m = 0; m < NV / 2; ++m) { const double2 v = xb[m]; xv[2 * m] = v.x; xv[2 * m + 1] = v.y; }
              if (sh == 0) {
#pragma unroll
                for (int j = 0; j < W; ++j) {
                  const double2 c = cf[j * (kTile / 2)];
                  acc[0][j & 1] = fma(c.x, xv[j], acc[0][j & 1]);
                  acc[1][j & 1] = fma(c.y, xv[j + 1], acc[1][j & 1]);
                }
              } else {
#pragma unroll
                for (int j = 0; j < W; ++j) {
                  const double2 c = cf[j * (kTile / 2)];
                  acc[0][j & 1] = fma(c.x, xv[j + 1], acc[0][j & 1]);
                  acc[1][j & 1] = fma(c.y, xv[j + 2], acc[1][j & 1]);
                }
              }
              release();
            }
          }
          if (++slot == kStages) { slot = 0; ++turn; }
        }
      }
      if (!ok) break;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!live[r]) continue;
        const double ax = acc[r][0] + acc[r][1];
        if (MODE == 0) {
          a.y[row + r] = ax;
          dot = fma(a.x[row + r], ax, dot);
        } else {
          const double rr = a.b[row + r] - ax;
          a.y[row + r] = rr;
          dot = fma(rr, rr, dot);
          if (a.z) dot2 = fma(rr, a.z[row + r], dot2);
        }
      }
    }
  }
  gstage = g0 + total;
  __syncthreads();
  if (*s_abort) {
    if (tid == 0 && a.pcg) {
      a.scal[S_STATUS] = (double)IGAFD_ERR_TIMEOUT;
      a.scal[S_DONE] = 1.0;
    }
    return;
  }
  if (!a.partial) return;
  __shared__ double sh32[32];
  const double bs = block_sum(dot, sh32);
  const double bs2 = (MODE == 1 && a.z) ? block_sum(dot2, sh32) : 0.0;
  if (tid == 0) {
    a.partial[vb] = bs;
    if (MODE == 1 && a.z) a.partial[vgrid + vb] = bs2;
  }
  if (!last_block(a.counter, (unsigned)vgrid)) return;
  const double tot = sum_partials(a.partial, (int)vgrid, sh32);
  const double tot2 = (MODE == 1 && a.z) ? sum_partials(a.partial + vgrid, (int)vgrid, sh32) : 0.0;
  if (tid == 0) {
    *a.counter = 0u;
    if (a.tstat) {   // this block finished last: launch duration = now - first start
      a.tstat[1] += global_ns() - a.tstat[0];
      a.tstat[2] += 1ull;
      a.tstat[0] = ~0ull;
    }
    if (a.pcg) {
      double *scal = a.scal;
      if (MODE == 0) {
        scal[S_PQ] = tot;
        const double alpha = scal[S_RHO] / tot;
        if (!(tot > 0.0) || !isfinite(alpha)) {
          scal[S_STATUS] = (double)IGAFD_ERR_BREAKDOWN;
          scal[S_DONE] = 1.0;
        }
        scal[S_ALPHA] = alpha;
      } else {
        scal[S_TRUE_RR] = tot;
        scal[S_RR] = tot;
        if (a.z) scal[S_RZOLD] = tot2;
      }
    }
  }
}

// Initialise the ring's full/empty barriers of a CTA (thread 0; the caller syncs).
template <int kStages, int kCompute>
__device__ __forceinline__ void ring_init(uint64_t *full, uint64_t *empty) {
  for (int s = 0; s < kStages; ++s) {
    mbar_init(&full[s], 1);
    mbar_init(&empty[s], kCompute / 32);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Resident CTAs per SM of a kernel with `smem` bytes of dynamic shared
// memory: the attribute and the occupancy are per device, set and measured
// once per device.
template <typename Kern>
igafd_status per_sm_of(Kern kern, int block, size_t smem, std::atomic<unsigned long long> &set,
                       std::atomic<int> *per_sm, int *out) {
  int dev = 0;
  IGAFD_CUDA(cudaGetDevice(&dev));
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(set.load() & bit)) {
    IGAFD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int nb = 0;
    IGAFD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, block, smem));
    per_sm[dev & 63].store(nb > 0 ? nb : 1);
    set.fetch_or(bit);
  }
  *out = per_sm[dev & 63].load();
  return IGAFD_OK;
}

// Rows per tile for N rows on `sms` SMs with `per_sm` resident CTAs each. The
// CTAs of an SM share its FP64 pipe and every CTA walks its tiles in turn, so
// the product takes as many rounds as the CTA with most tiles, each as long as
// the rows in flight on an SM in a round (and some per round), or as one
// tile's latency (measured at p = 3: 117 clocks per FMA of a chain with 2
// warps on the SM, 139 with 7, where the pipe takes 16 per warp). With 256-row
// tiles only, the last round of a mid-sized patch ran on few CTAs and a small
// patch on few SMs: (61, 90, 47) at p = 4 took 373 us, now 319 (299 us of FP64
// work); (20, 20, 20) at p = 3 took 35 us, now 24. Ties go to the larger tile.
// The products of a solve take tiles of kSolveTile rows or more: a batch runs the
// same tiles (its results are the single solves' bit for bit) for many problems
// at once, where the SMs are never idle and small tiles only cost (12 problems
// of 16 to 48 functions per direction, one group each, BF16: 6.34 ms with tiles
// down to 64 rows, 5.95 with 128, 5.77 with 256 only; the same problems one by
// one 13.4, 13.6 and 14.1 ms).
inline int tile_rows(long long N, int sms, int per_sm, int step, int lowest) {
  int best = kTile;
  double cost = -1.0;
  for (int h = kTile; h >= lowest; h -= step) {
    const long long tiles = (N + h - 1) / h, ctas = (long long)sms * per_sm;
    const long long rounds = (tiles + ctas - 1) / ctas;
    const double rows = (double)h * (rounds > 1 ? per_sm : (double)((tiles + sms - 1) / sms));
    const double w = rows + 48.0 > 215.0 + 0.3 * rows ? rows + 48.0 : 215.0 + 0.3 * rows;
    if (cost < 0.0 || rounds * w < cost) {
      cost = rounds * w;
      best = h;
    }
  }
  return best;
}

}  // namespace
