// Stiffness stencil of a 3D patch by sum factorisation over the whole patch.
//
//   A[i, i + delta] = sum_{r,s} sum_q d_r B_i(q) Q_rs(q) d_s B_{i+delta}(q)
//
// is contracted one direction at a time, direction 3 first, over all points
// of the other two, so that the elements a pair (i_k, i_k + delta_k) shares
// are summed once per direction (per element the same sums would be formed
// for every pair of local functions: about 110,000 FP64 FMAs per dof at p = 3
// against 20,000 here):
//
//   points_kernel   Q at the quadrature points of a range of element layers of
//                   direction 3, times the weights; the geometry map by sum
//                   factorisation along rows of points; min det J and the
//                   extreme eigenvalues of Q
//   dir3_kernel     T1[8][i3][delta3][q2][q1]: the eight products of Q's
//                   entries with (value, derivative) pairs of direction 3
//   dir2_kernel     T2[4][i3][delta3][delta2][i2][q1]: by the (value,
//                   derivative) pair direction 1 still has to apply
//   dir1_kernel     the stencil entries, one thread per row
//
// Only delta3 >= 0 is computed; a full stencil gets delta3 < 0 from the
// symmetry A_ij = A_ji (entry -delta of row i + off(delta)). No atomics and
// no read-modify-write: an entry is written once, in an order of summation
// that does not depend on the launch. i3 is taken in batches (and i2 in
// chunks) whose T1 and T2 stay near L2's size; the layers of Q that a batch needs are
// kept in a ring.
//
// Bound: the FP64 pipe (2 FMA/clk/SM), 629 G FMA/s. At n = 56, p = 3 the
// contractions take 3.3 G FMA (5.3 ms; measured 1.6 + 2.7 + 2.8 ms for
// directions 3, 2, 1) and the points about 160 operations each (2.7 ms;
// measured 4.4 ms): 11.5 ms, where one block per element, with its local
// matrix and a read-modify-write of the stencil in 64 colour classes, took
// 155 ms. The load vector takes 4.9 ms (element blocks: 22 ms).
#include "common.cuh"
#include "geom.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <vector>

namespace {

using namespace igafd_geom;

constexpr int kThr = 128;
constexpr int kLoad = 64;       // points of direction 1 per block of load_kernel
constexpr int kRows = 64;       // rows per block of dir1_kernel (small patches fill more of it)
constexpr int kMaxSmem = 200 * 1024;   // dynamic shared memory that a kernel may ask for

// Lets a kernel ask for up to kMaxSmem, once per device: the attribute belongs
// to the kernel, not to a launch, and other host threads launch it too.
template <typename Kern> igafd_status allow_smem(Kern kern, std::atomic<unsigned long long> &set) {
  int dev = 0;
  IGAFD_CUDA(cudaGetDevice(&dev));
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(set.load() & bit)) {
    IGAFD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    set.fetch_or(bit);
  }
  return IGAFD_OK;
}

// order-preserving map of doubles to unsigned integers
__host__ __device__ __forceinline__ unsigned long long key_of(double d) {
#ifdef __CUDA_ARCH__
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
#else
  unsigned long long b;
  memcpy(&b, &d, 8);
#endif
  return (b >> 63) ? ~b : b | (1ull << 63);
}
__host__ __device__ __forceinline__ double of_key(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? k & ~(1ull << 63) : ~k;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

struct AsmArgs {
  PV v;
  const int2 *sup[3];       // per function (full index): first element of its support, and how many
  int T1;                   // quadrature points along direction 1
  int q2lo, C2;             // points of direction 2 held: [q2lo, q2lo + C2)
  int i2lo, c2;             // kept functions of direction 2 of this chunk
  int i3lo, c3;             // kept functions of direction 3 of this batch
  int ring;                 // element layers of direction 3 in the ring of Q
  double *Q;                // [6][ring * nq][C2][T1]
  double *t1;               // [8][c3][p + 1][C2][T1]
  double *t2;               // [4][c3][p + 1][2p + 1][c2][T1]
  unsigned long long *best; // keys of min det J, min lambda_min, max lambda_max
  double *S;                // the stencil, row i of offset o at (o - o_min) ld + H + i
  long long ld, H;
  int o_min;
};

// One row (q2, q3) of points per block: the geometry's control net contracted
// in directions 2 and 3 into rows over direction 1's control points (values,
// and derivatives in directions 2 and 3), then per point along direction 1.
// ROWS false: nets whose rows do not fit in shared memory (more than about 2800
// control points of direction 1, far more than the points), each point's map
// straight from the net.
template <bool ROWS>
__global__ void __launch_bounds__(kThr) points_kernel(AsmArgs a, int e3lo) {
  extern __shared__ double sm[];
  const PV &v = a.v;
  const int gp = v.gp, ga = gp + 1, gm = v.gm[0], nq = v.nq;
  const int ql = blockIdx.x, q2 = a.q2lo + ql, q3 = e3lo * nq + blockIdx.y;
  double *row = sm;                         // [3 coordinates][vv, dv, vd][gm]
  double *krow = sm + 9 * gm;               // [km]
  if constexpr (ROWS) {
    const double *v2 = v.gv[1] + (size_t)q2 * ga, *d2 = v.gd[1] + (size_t)q2 * ga;
    const double *v3 = v.gv[2] + (size_t)q3 * ga, *d3 = v.gd[2] + (size_t)q3 * ga;
    const int g2 = v.gspan[1][q2] - gp, g3 = v.gspan[2][q3] - gp;
    for (int t = threadIdx.x; t < 3 * gm; t += kThr) {
      const int c = t / gm, g1 = t - c * gm;
      double s0 = 0.0, s2 = 0.0, s3 = 0.0;
      for (int a3 = 0; a3 < ga; ++a3) {
        double r0 = 0.0, r2 = 0.0;
        const double *C = v.ctrl + (((size_t)c * v.gm[2] + g3 + a3) * v.gm[1] + g2) * gm + g1;
        for (int a2 = 0; a2 < ga; ++a2) {
          const double x = C[(size_t)a2 * gm];
          r0 = fma(x, v2[a2], r0);
          r2 = fma(x, d2[a2], r2);
        }
        s0 = fma(r0, v3[a3], s0);
        s2 = fma(r2, v3[a3], s2);
        s3 = fma(r0, d3[a3], s3);
      }
      row[(c * 3 + 0) * gm + g1] = s0;
      row[(c * 3 + 1) * gm + g1] = s2;
      row[(c * 3 + 2) * gm + g1] = s3;
    }
    if (v.kctrl) {
      const int kp = v.kp, ka = kp + 1, km = v.km[0];
      const double *k2 = v.kv[1] + (size_t)q2 * ka, *k3 = v.kv[2] + (size_t)q3 * ka;
      const int s2 = v.kspan[1][q2] - kp, s3 = v.kspan[2][q3] - kp;
      for (int k1 = threadIdx.x; k1 < km; k1 += kThr) {
        double s = 0.0;
        for (int a3 = 0; a3 < ka; ++a3) {
          double r = 0.0;
          for (int a2 = 0; a2 < ka; ++a2)
            r = fma(v.kctrl[((size_t)(s3 + a3) * v.km[1] + s2 + a2) * km + k1], k2[a2], r);
          s = fma(r, k3[a3], s);
        }
        krow[k1] = s;
      }
    }
  }
  __syncthreads();
  double mdet = 1e300, lmin = 1e300, lmax = -1e300;
  // extremes found so far by any block: points that cannot pass them are left
  // out of the eigenvalue evaluation (below)
  const double seen_min = of_key(((volatile unsigned long long *)a.best)[1]);
  const double seen_max = of_key(((volatile unsigned long long *)a.best)[2]);
  const double w23 = v.w[1][q2] * v.w[2][q3];
  const size_t plane = (size_t)a.C2 * a.T1;
  const int slot = (q3 / nq) % a.ring * nq + q3 % nq;
  double *out = a.Q + (size_t)slot * plane + (size_t)ql * a.T1;
  const size_t comp = (size_t)a.ring * nq * plane;
  for (int q1 = threadIdx.x; q1 < a.T1; q1 += kThr) {
    double J[3][3] = {}, kap = v.kappa;
    if constexpr (ROWS) {
      const double *v1 = v.gv[0] + (size_t)q1 * ga, *d1 = v.gd[0] + (size_t)q1 * ga;
      const int g1 = v.gspan[0][q1] - gp;
      for (int i = 0; i < ga; ++i) {
        const double x = v1[i], d = d1[i];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          J[c][0] = fma(row[(c * 3 + 0) * gm + g1 + i], d, J[c][0]);
          J[c][1] = fma(row[(c * 3 + 1) * gm + g1 + i], x, J[c][1]);
          J[c][2] = fma(row[(c * 3 + 2) * gm + g1 + i], x, J[c][2]);
        }
      }
      if (v.kctrl) {
        const int ka = v.kp + 1, k1 = v.kspan[0][q1] - v.kp;
        double s = 0.0;
        for (int i = 0; i < ka; ++i) s = fma(krow[k1 + i], v.kv[0][(size_t)q1 * ka + i], s);
        kap *= s;
      }
    } else {
      const int t[3] = {q1, q2, q3};
      double x[3];
      geo_eval<3>(v, t, x, J);
      kap = kappa_eval<3>(v, t);
    }
    // Q = kappa |det| J^-1 J^-T = kappa / |det| (adj J)(adj J)^T; B row r of the adjugate
    double B[3][3];
    B[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    B[1][0] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    B[2][0] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    B[0][1] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
    B[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
    B[2][1] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
    B[0][2] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
    B[1][2] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
    B[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double det = J[0][0] * B[0][0] + J[0][1] * B[1][0] + J[0][2] * B[2][0];
    mdet = fmin(mdet, det);
    const double sc = kap / fabs(det);
    double Q[6];                            // 00, 11, 22, 01, 02, 12
    const int rr[6] = {0, 1, 2, 0, 0, 1}, ss[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
    for (int q = 0; q < 6; ++q)
      Q[q] = sc * (B[rr[q]][0] * B[ss[q]][0] + B[rr[q]][1] * B[ss[q]][1] + B[rr[q]][2] * B[ss[q]][2]);
    // eigenvalues lie within 2 sqrt(p2 / 6) of the mean q (p2 the squared
    // Frobenius norm of Q - q I): the closed form is evaluated only where
    // that interval reaches past the extremes known so far (by more than the
    // closed form's own rounding)
    const double tr = (Q[0] + Q[1] + Q[2]) * (1.0 / 3.0);
    const double x0 = Q[0] - tr, x1 = Q[1] - tr, x2 = Q[2] - tr;
    const double p4 = (x0 * x0 + x1 * x1 + x2 * x2 + 2.0 * (Q[3] * Q[3] + Q[4] * Q[4] + Q[5] * Q[5])) *
                          (2.0 / 3.0) * (1.0 + 1e-9);
    const double eps = 4e-15 * tr;
    const double up = fmax(lmax, seen_max) - tr + eps, dn = tr - fmin(lmin, seen_min) + eps;
    if (!(up > 0.0 && p4 < up * up && dn > 0.0 && p4 < dn * dn)) {
      double l0, l1;
      sym_eig_extremes<3>(Q, &l0, &l1);
      lmin = fmin(lmin, l0);
      lmax = fmax(lmax, l1);
    }
    const double wt = w23 * v.w[0][q1];
#pragma unroll
    for (int q = 0; q < 6; ++q) out[q * comp + q1] = Q[q] * wt;
  }
  for (int o = 16; o > 0; o >>= 1) {
    mdet = fmin(mdet, __shfl_xor_sync(0xffffffffu, mdet, o));
    lmin = fmin(lmin, __shfl_xor_sync(0xffffffffu, lmin, o));
    lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (mdet < of_key(a.best[0])) atomicMin(&a.best[0], key_of(mdet));
    if (lmin < of_key(a.best[1])) atomicMin(&a.best[1], key_of(lmin));
    if (lmax > of_key(a.best[2])) atomicMax(&a.best[2], key_of(lmax));
  }
}

// T1 of one i3: thread per point (q1, q2). The products of direction 3's
// functions are the same for the whole block. Arrays: vv Q11, vv Q22, vv Q12,
// dv Q13, dv Q23, vd Q13, vd Q23, dd Q33 (first letter: row function).
template <int P>
__global__ void __launch_bounds__(kThr) dir3_kernel(AsmArgs a) {
  constexpr int A = P + 1, NQ = P + 1;
  __shared__ double2 pr[A * NQ][A][2];      // (vv, dv), (vd, dd) per point and delta3
  __shared__ int s_plane[A * NQ], s_n[A * NQ];
  const PV &v = a.v;
  const int i3 = a.i3lo + blockIdx.z, I = i3 + v.ds;
  const int2 sp = a.sup[2][I];
  const int np = sp.y * NQ;
  for (int t = threadIdx.x; t < np; t += kThr) {
    const int e = sp.x + t / NQ, g = t % NQ, la = I - (v.span[2][e] - P);
    const double *bv = v.bv[2] + (size_t)(e * NQ + g) * A, *bd = v.bd[2] + (size_t)(e * NQ + g) * A;
    s_plane[t] = e % a.ring * NQ + g;
    s_n[t] = A - la;                        // delta3 < A - la: a shared function exists
#pragma unroll
    for (int d = 0; d < A; ++d) {
      const double g0 = la + d <= P ? bv[la + d] : 0.0, g1 = la + d <= P ? bd[la + d] : 0.0;
      pr[t][d][0] = make_double2(bv[la] * g0, bd[la] * g0);
      pr[t][d][1] = make_double2(bv[la] * g1, bd[la] * g1);
    }
  }
  __syncthreads();
  const int q1 = blockIdx.x * kThr + threadIdx.x, ql = blockIdx.y;
  if (q1 >= a.T1) return;
  const size_t plane = (size_t)a.C2 * a.T1, comp = (size_t)a.ring * NQ * plane;
  const double *Q = a.Q + (size_t)ql * a.T1 + q1;
  double acc[A][8];
#pragma unroll
  for (int d = 0; d < A; ++d)
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[d][k] = 0.0;
  for (int t = 0; t < np; ++t) {
    const double *x = Q + (size_t)s_plane[t] * plane;
    const double q11 = x[0], q22 = x[comp], q33 = x[2 * comp], q12 = x[3 * comp], q13 = x[4 * comp],
                 q23 = x[5 * comp];
    const int n = s_n[t];
#pragma unroll
    for (int d = 0; d < A; ++d) {
      if (d >= n) break;                    // uniform
      const double2 b = pr[t][d][0], c = pr[t][d][1];
      acc[d][0] = fma(b.x, q11, acc[d][0]);
      acc[d][1] = fma(b.x, q22, acc[d][1]);
      acc[d][2] = fma(b.x, q12, acc[d][2]);
      acc[d][3] = fma(b.y, q13, acc[d][3]);
      acc[d][4] = fma(b.y, q23, acc[d][4]);
      acc[d][5] = fma(c.x, q13, acc[d][5]);
      acc[d][6] = fma(c.x, q23, acc[d][6]);
      acc[d][7] = fma(c.y, q33, acc[d][7]);
    }
  }
  const size_t arr = (size_t)a.c3 * A * plane;
  double *out = a.t1 + ((size_t)blockIdx.z * A * a.C2 + ql) * a.T1 + q1;
#pragma unroll
  for (int d = 0; d < A; ++d)
#pragma unroll
    for (int k = 0; k < 8; ++k) out[k * arr + d * plane] = acc[d][k];
}

// T2 of one (i3, delta3, i2): thread per q1. With the row function's value f
// and derivative f' applied first, a point costs 9 + 6 operations per column
// function instead of 9 products each. Arrays: dd, dv, vd, vv of direction 1.
template <int P>
__global__ void __launch_bounds__(kThr) dir2_kernel(AsmArgs a) {
  constexpr int A = P + 1, NQ = P + 1, W = 2 * P + 1;
  __shared__ double2 s_b[A * NQ][A];        // (value, derivative) of the element's functions
  __shared__ int s_a[A * NQ];
  const PV &v = a.v;
  const int i2 = a.i2lo + blockIdx.y, I = i2 + v.ds;
  const int2 sp = a.sup[1][I];
  const int np = sp.y * NQ;
  for (int t = threadIdx.x; t < np; t += kThr) {
    const int e = sp.x + t / NQ;
    const size_t at = (size_t)(sp.x * NQ + t) * A;
    s_a[t] = I - (v.span[1][e] - P);
#pragma unroll
    for (int b = 0; b < A; ++b) s_b[t][b] = make_double2(v.bv[1][at + b], v.bd[1][at + b]);
  }
  __syncthreads();
  const int q1 = blockIdx.x * kThr + threadIdx.x, z = blockIdx.z;   // z = i3 A + delta3
  if (q1 >= a.T1) return;
  const size_t plane = (size_t)a.C2 * a.T1, arr = (size_t)a.c3 * A * plane;
  const double *x = a.t1 + (size_t)z * plane + (size_t)(sp.x * NQ - a.q2lo) * a.T1 + q1;
  double acc[W][4];
#pragma unroll
  for (int d = 0; d < W; ++d)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[d][k] = 0.0;
  for (int t = 0; t < np; ++t, x += a.T1) {
    const int la = s_a[t];
    const double2 f = s_b[t][la];
    const double t0 = x[0], t1 = x[arr], t2 = x[2 * arr], t3 = x[3 * arr], t4 = x[4 * arr],
                 t5 = x[5 * arr], t6 = x[6 * arr], t7 = x[7 * arr];
    const double c0 = f.x * t0, c1 = f.x * t5, c2 = fma(f.y, t2, f.x * t3), c3 = fma(f.y, t6, f.x * t7);
    const double d1 = f.x * t2, d3 = fma(f.y, t1, f.x * t4);
#pragma unroll
    for (int d = 0; d < W; ++d) {
      const int b = la + d - P;
      if (b >= 0 && b <= P) {               // uniform
        const double2 g = s_b[t][b];
        acc[d][0] = fma(g.x, c0, acc[d][0]);
        acc[d][1] = fma(g.x, c1, fma(g.y, d1, acc[d][1]));
        acc[d][2] = fma(g.x, c2, acc[d][2]);
        acc[d][3] = fma(g.x, c3, fma(g.y, d3, acc[d][3]));
      }
    }
  }
  const size_t line = (size_t)a.c2 * a.T1, arr2 = (size_t)a.c3 * A * W * line;
  double *out = a.t2 + (size_t)z * W * line + (size_t)blockIdx.y * a.T1 + q1;
#pragma unroll
  for (int d = 0; d < W; ++d)
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k * arr2 + d * line] = acc[d][k];
}

// The entries of one (i3, delta3, i2, delta2): thread per row i1.
template <int P>
__global__ void __launch_bounds__(kRows) dir1_kernel(AsmArgs a) {
  constexpr int A = P + 1, NQ = P + 1, W = 2 * P + 1;
  extern __shared__ double sm[];            // [4][points of this block's rows]
  const PV &v = a.v;
  const int z = blockIdx.z, d2i = z % W, d3 = (z / W) % A, b3 = z / (W * A);
  const int i3 = a.i3lo + b3, i2 = a.i2lo + blockIdx.y, d2 = d2i - P;
  if (i3 + d3 >= v.n[2] || i2 + d2 < 0 || i2 + d2 >= v.n[1]) return;   // outside the box
  const int ob = ((d3 + P) * W + d2i) * W;
  if (ob + W <= a.o_min) return;                                       // not stored
  const int first = blockIdx.x * kRows, last = min(first + kRows, v.n[0]) - 1;
  const int2 s0 = a.sup[0][first + v.ds], s1 = a.sup[0][last + v.ds];
  const int qa = s0.x * NQ, nqp = (s1.x + s1.y) * NQ - qa;
  const size_t line = (size_t)a.c2 * a.T1, arr2 = (size_t)a.c3 * A * W * line;
  const double *src = a.t2 + (size_t)z * line + (size_t)blockIdx.y * a.T1 + qa;
  for (int k = 0; k < 4; ++k)
    for (int t = threadIdx.x; t < nqp; t += kRows) sm[k * nqp + t] = src[k * arr2 + t];
  __syncthreads();
  const int i1 = first + threadIdx.x;
  if (i1 > last) return;
  const int I = i1 + v.ds;
  const int2 sp = a.sup[0][I];
  double acc[W];
#pragma unroll
  for (int d = 0; d < W; ++d) acc[d] = 0.0;
  for (int j = 0; j < sp.y; ++j) {
    const int e = sp.x + j, la = I - (v.span[0][e] - P);
    const double *bv = v.bv[0] + (size_t)e * NQ * A, *bd = v.bd[0] + (size_t)e * NQ * A;
    const double *t = sm + (e * NQ - qa);
    double u[NQ], w[NQ];                    // factors of the column function's value and derivative
#pragma unroll
    for (int g = 0; g < NQ; ++g) {
      const double f = bv[g * A + la], fd = bd[g * A + la];
      u[g] = fma(fd, t[nqp + g], f * t[3 * nqp + g]);
      w[g] = fma(fd, t[g], f * t[2 * nqp + g]);
    }
#pragma unroll
    for (int d = 0; d < W; ++d) {
      const int b = la + d - P;
      if (b >= 0 && b <= P) {
#pragma unroll
        for (int g = 0; g < NQ; ++g)
          acc[d] = fma(bv[g * A + b], u[g], fma(bd[g * A + b], w[g], acc[d]));
      }
    }
  }
  const long long n1 = v.n[0], n12 = n1 * v.n[1];
  const long long row = i1 + n1 * i2 + n12 * i3;
  const long long off23 = n1 * d2 + n12 * d3;
  const int top = W * W * W - 1;
#pragma unroll
  for (int d = 0; d < W; ++d) {
    const int d1 = d - P, o = ob + d;
    if (i1 + d1 < 0 || i1 + d1 >= v.n[0] || o < a.o_min) continue;
    a.S[(size_t)(o - a.o_min) * a.ld + a.H + row] = acc[d];
    if (d3 > 0 && a.o_min == 0) a.S[(size_t)(top - o) * a.ld + a.H + row + off23 + d1] = acc[d];
  }
}

// Load vector b_i = sum_q f(x_q) B_i(zeta_q) |det J(zeta_q)| w_q of a 3D
// patch, f from fq (order of igafd_quad_points) or, with fq null, f = 3 pi^2
// prod sin(pi x_k). A block takes one element of directions 2 and 3 (a colour
// class: no two blocks of a launch share a function) and a tile of elements of
// direction 1 (every other tile); groups of threads share the element's rows
// (q2, q3), each thread summing its points q1 into the (p + 1)^2 local
// functions of those directions, with the geometry contracted along rows of points as in points_kernel;
// direction 1 is contracted last, in shared memory. (ROWS as in points_kernel.)
template <int P, int RG, bool ROWS>
__global__ void __launch_bounds__(kLoad * RG) load_kernel(PV v, int c2, int c3, int ne2, int par,
                                                    const double *fq, double *b) {
  constexpr int A = P + 1, NQ = P + 1, TE = kLoad / NQ;
  extern __shared__ double sm[];
  const int gp = v.gp, ga = gp + 1;
  const int e2 = c2 + A * ((int)blockIdx.x % ne2), e3 = c3 + A * ((int)blockIdx.x / ne2);
  const int el0 = (2 * (int)blockIdx.y + par) * TE;
  if (el0 >= v.nel[0]) return;
  const int ne = min(TE, v.nel[0] - el0), np = ne * NQ, t = threadIdx.x % kLoad, grp = threadIdx.x / kLoad,
            q1 = el0 * NQ + t;
  const int glo = v.gspan[0][el0 * NQ] - gp, G = v.gspan[0][el0 * NQ + np - 1] - glo + 1;
  const long long T0 = (long long)v.nel[0] * NQ, T1 = (long long)v.nel[1] * NQ;
  double acc[A][A];
#pragma unroll
  for (int i = 0; i < A; ++i)
#pragma unroll
    for (int j = 0; j < A; ++j) acc[i][j] = 0.0;
  double *row = sm + (size_t)grp * 9 * G;
  for (int r = 0; r < NQ * NQ; r += RG) {
    const int g = min(r + grp, NQ * NQ - 1);    // (a group without a row of its own adds nothing)
    const int q2 = e2 * NQ + g % NQ, q3 = e3 * NQ + g / NQ;
    const double *v2 = v.gv[1] + (size_t)q2 * ga, *d2 = v.gd[1] + (size_t)q2 * ga;
    const double *v3 = v.gv[2] + (size_t)q3 * ga, *d3 = v.gd[2] + (size_t)q3 * ga;
    const int g2 = v.gspan[1][q2] - gp, g3 = v.gspan[2][q3] - gp;
    __syncthreads();
    for (int k = t; ROWS && k < 3 * G; k += kLoad) {
      const int c = k / G, g1 = k - c * G;
      double s0 = 0.0, s2 = 0.0, s3 = 0.0;
      for (int a3 = 0; a3 < ga; ++a3) {
        double r0 = 0.0, r2 = 0.0;
        const double *C = v.ctrl + (((size_t)c * v.gm[2] + g3 + a3) * v.gm[1] + g2) * v.gm[0] + glo + g1;
        for (int a2 = 0; a2 < ga; ++a2) {
          const double x = C[(size_t)a2 * v.gm[0]];
          r0 = fma(x, v2[a2], r0);
          r2 = fma(x, d2[a2], r2);
        }
        s0 = fma(r0, v3[a3], s0);
        s2 = fma(r2, v3[a3], s2);
        s3 = fma(r0, d3[a3], s3);
      }
      row[(c * 3 + 0) * G + g1] = s0;
      row[(c * 3 + 1) * G + g1] = s2;
      row[(c * 3 + 2) * G + g1] = s3;
    }
    __syncthreads();
    if (t < np && r + grp < NQ * NQ) {
      double J[3][3] = {}, X[3] = {};
      if constexpr (ROWS) {
        const double *v1 = v.gv[0] + (size_t)q1 * ga, *d1 = v.gd[0] + (size_t)q1 * ga;
        const int g1 = v.gspan[0][q1] - gp - glo;
        for (int i = 0; i < ga; ++i) {
          const double x = v1[i], d = d1[i];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const double y = row[(c * 3 + 0) * G + g1 + i];
            X[c] = fma(y, x, X[c]);
            J[c][0] = fma(y, d, J[c][0]);
            J[c][1] = fma(row[(c * 3 + 1) * G + g1 + i], x, J[c][1]);
            J[c][2] = fma(row[(c * 3 + 2) * G + g1 + i], x, J[c][2]);
          }
        }
      } else {
        const int at[3] = {q1, q2, q3};
        geo_eval<3>(v, at, X, J);
      }
      const double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) +
                         J[0][1] * (J[1][2] * J[2][0] - J[1][0] * J[2][2]) +
                         J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
      const double f = fq ? fq[q1 + T0 * (q2 + T1 * q3)]
                          : 3.0 * M_PI * M_PI * (sinpi(X[0]) * sinpi(X[1]) * sinpi(X[2]));
      const double fw = f * fabs(det) * (v.w[0][q1] * v.w[1][q2] * v.w[2][q3]);
#pragma unroll
      for (int i = 0; i < A; ++i) {
        const double h = fw * v.bv[2][(size_t)q3 * A + i];
#pragma unroll
        for (int j = 0; j < A; ++j) acc[i][j] = fma(h, v.bv[1][(size_t)q2 * A + j], acc[i][j]);
      }
    }
  }
  for (int r = 0; r < RG; ++r) {            // the groups' sums, in order
    __syncthreads();
    if (grp != r) continue;
#pragma unroll
    for (int i = 0; i < A; ++i)
#pragma unroll
      for (int j = 0; j < A; ++j) {
        double *x = sm + (i * A + j) * kLoad + t;
        *x = r ? *x + acc[i][j] : acc[i][j];
      }
  }
  __syncthreads();
  const int I0 = v.span[0][el0] - P, F = v.span[0][el0 + ne - 1] - I0 + 1;
  for (int k = threadIdx.x; k < F * A * A; k += kLoad * RG) {
    const int I = I0 + k % F, j = (k / F) % A, i = k / (F * A);
    const int I2 = v.span[1][e2] - P + j, I3 = v.span[2][e3] - P + i;
    if (I < v.ds || I >= v.ds + v.n[0] || I2 < v.ds || I2 >= v.ds + v.n[1] || I3 < v.ds ||
        I3 >= v.ds + v.n[2])
      continue;
    const double *r = sm + (i * A + j) * kLoad;
    double s = 0.0;
    for (int e = 0; e < ne; ++e) {
      const int la = I - (v.span[0][el0 + e] - P);
      if (la < 0 || la > P) continue;
      for (int g = 0; g < NQ; ++g)
        s = fma(v.bv[0][(size_t)((el0 + e) * NQ + g) * A + la], r[e * NQ + g], s);
    }
    b[(I - v.ds) + (long long)v.n[0] * ((I2 - v.ds) + (long long)v.n[1] * (I3 - v.ds))] += s;
  }
}

// RG groups of rows at once; a net too fine for their shared memory takes one
// (a block's rows reach over at most all its control points of direction 1),
// and one too fine for that the map point by point.
template <int P, int RG = (P <= 3 ? 4 : 2), bool ROWS = true>
igafd_status load_p(const PV &v, const double *fq, double *b, cudaStream_t s) {
  constexpr int A = P + 1, TE = kLoad / A;
  const size_t smem = sizeof(double) * std::max(ROWS ? (size_t)9 * v.gm[0] * RG : 0, (size_t)A * A * kLoad);
  if constexpr (ROWS)
    if (smem > kMaxSmem) return load_p<P, 1, (RG > 1)>(v, fq, b, s);
  static std::atomic<unsigned long long> smem_set{0};
  IGAFD_TRY(allow_smem(load_kernel<P, RG, ROWS>, smem_set));
  const int tiles = (v.nel[0] + TE - 1) / TE;
  for (int c3 = 0; c3 < std::min(A, v.nel[2]); ++c3)
    for (int c2 = 0; c2 < std::min(A, v.nel[1]); ++c2)
      for (int par = 0; par < std::min(2, tiles); ++par) {
        const int ne2 = (v.nel[1] - c2 + A - 1) / A, ne3 = (v.nel[2] - c3 + A - 1) / A;
        load_kernel<P, RG, ROWS><<<dim3(ne2 * ne3, (tiles - par + 1) / 2), kLoad * RG, smem, s>>>(v, c2, c3, ne2, par, fq, b);
        IGAFD_LAUNCHED(1);
        IGAFD_CUDA(cudaGetLastError());
      }
  return IGAFD_OK;
}

__global__ void init_best_kernel(unsigned long long *best) {
  best[0] = key_of(1e300);
  best[1] = key_of(1e300);
  best[2] = key_of(-1e300);
}

template <int P>
igafd_status contract(const AsmArgs &a, size_t smem1, cudaStream_t s) {
  constexpr int A = P + 1, W = 2 * P + 1;
  const unsigned tx = (unsigned)((a.T1 + kThr - 1) / kThr);
  dir3_kernel<P><<<dim3(tx, a.C2, a.c3), kThr, 0, s>>>(a);
  dir2_kernel<P><<<dim3(tx, a.c2, a.c3 * A), kThr, 0, s>>>(a);
  dir1_kernel<P><<<dim3((unsigned)((a.v.n[0] + kRows - 1) / kRows), a.c2, a.c3 * A * W), kRows, smem1, s>>>(a);
  IGAFD_LAUNCHED(3);
  IGAFD_CUDA(cudaGetLastError());
  return IGAFD_OK;
}

igafd_status contract_p(int p, const AsmArgs &a, size_t smem1, cudaStream_t s) {
  switch (p) {
    case 1: return contract<1>(a, smem1, s);
    case 2: return contract<2>(a, smem1, s);
    case 3: return contract<3>(a, smem1, s);
    case 4: return contract<4>(a, smem1, s);
    case 5: return contract<5>(a, smem1, s);
    default: return contract<6>(a, smem1, s);
  }
}

// One run over the patch with i2 in chunks of `chunk` functions and i3 in
// batches of `batch` (scratch allocated here; OOM leaves it to the caller to
// try smaller ones).
struct Runner {
  igafd_patch *P;
  cudaStream_t s;
  std::vector<int> span[3];
  std::vector<int2> sup[3];
  int2 *dsup;
  unsigned long long *best;
  std::vector<void *> held;

  // elements of kept functions [a, b) of direction k
  void elements(int k, int a, int b, int *lo, int *hi) const {
    *lo = 1 << 30;
    *hi = 0;
    for (int i = a; i < b; ++i) {
      const int2 q = sup[k][i + P->dshift];
      *lo = std::min(*lo, q.x);
      *hi = std::max(*hi, q.x + q.y);
    }
  }
  size_t need(int chunk, int batch, int *C2, int *ring) const {
    const int p = P->p, nq = p + 1, A = p + 1, W = 2 * p + 1;
    int lo, hi;
    *C2 = 0;
    for (int i = 0; i < P->n[1]; i += chunk) {
      elements(1, i, std::min(i + chunk, P->n[1]), &lo, &hi);
      *C2 = std::max(*C2, (hi - lo) * nq);
    }
    *ring = 0;
    for (int i = 0; i < P->n[2]; i += batch) {
      elements(2, i, std::min(i + batch, P->n[2]), &lo, &hi);
      *ring = std::max(*ring, hi - lo);
    }
    const size_t T1 = (size_t)P->nel[0] * nq;
    return 8 * T1 * ((size_t)6 * *ring * nq * *C2 + (size_t)8 * batch * A * *C2 +
                     (size_t)4 * batch * A * W * chunk);
  }
  igafd_status run(int chunk, int batch) {
    const int p = P->p, nq = p + 1, A = p + 1;
    AsmArgs a{};
    a.v = make_view(P);
    for (int k = 0, at = 0; k < 3; ++k) {
      a.sup[k] = dsup + at;
      at += (int)sup[k].size();
    }
    a.T1 = P->nel[0] * nq;
    int C2 = 0;
    const size_t bytes = need(chunk, batch, &C2, &a.ring);
    double *w = nullptr;
    if (cudaMalloc((void **)&w, bytes) != cudaSuccess) {
      cudaGetLastError();
      return IGAFD_ERR_OOM;
    }
    held.push_back(w);
    a.best = best;
    a.S = P->stencil;
    a.o_min = P->stencil_half ? P->n_off / 2 : 0;
    a.ld = P->stencil_half ? P->sh_ld : P->Np;
    a.H = P->stencil_half ? P->sh_H : 0;
    const int km = P->kctrl ? P->dir[0].km : 0;
    size_t smem0 = (size_t)(9 * P->dir[0].gm + km) * sizeof(double);
    const bool rows = smem0 <= kMaxSmem;
    if (!rows) smem0 = 0;
    static std::atomic<unsigned long long> smem_set{0};
    IGAFD_TRY(allow_smem(points_kernel<true>, smem_set));
    const auto points = rows ? points_kernel<true> : points_kernel<false>;
    size_t smem1 = 0;                       // rows' points of a dir1 block
    for (int i = 0; i < P->n[0]; i += kRows) {
      int lo, hi;
      elements(0, i, std::min(i + kRows, P->n[0]), &lo, &hi);
      smem1 = std::max(smem1, (size_t)4 * (hi - lo) * nq * sizeof(double));
    }
    for (int i2 = 0; i2 < P->n[1]; i2 += chunk) {
      int e2lo, e2hi;
      a.i2lo = i2;
      a.c2 = std::min(chunk, P->n[1] - i2);
      elements(1, i2, i2 + a.c2, &e2lo, &e2hi);
      a.q2lo = e2lo * nq;
      a.C2 = (e2hi - e2lo) * nq;
      a.Q = w;
      a.t1 = a.Q + (size_t)6 * a.ring * nq * C2 * a.T1;
      a.t2 = a.t1 + (size_t)8 * batch * A * C2 * a.T1;
      int have = 0;                         // element layers of direction 3 evaluated so far
      for (int i3 = 0; i3 < P->n[2]; i3 += batch) {
        int lo, hi;
        a.i3lo = i3;
        a.c3 = std::min(batch, P->n[2] - i3);
        elements(2, i3, i3 + a.c3, &lo, &hi);
        have = std::max(have, lo);
        if (hi > have) {
          points<<<dim3(a.C2, (hi - have) * nq), kThr, smem0, s>>>(a, have);
          IGAFD_LAUNCHED(1);
          have = hi;
        }
        IGAFD_TRY(contract_p(p, a, smem1, s));
      }
    }
    return IGAFD_OK;
  }
};

}  // namespace

// Geometry diagnostics (min det J, the Prop. 1 estimate) and the stiffness
// stencil of a 3D patch, p <= 6. The entries not computed (couplings that
// leave the box, the halos of a half-stored stencil) are 0.
igafd_status igafd_assemble3(igafd_patch *P, cudaStream_t s) {
  const int p = P->p;
  if (p > 6) return IGAFD_ERR_ARG;
  Runner R{};
  R.P = P;
  R.s = s;
  size_t funcs = 0;
  for (int k = 0; k < 3; ++k) {
    R.span[k].resize(P->nel[k]);
    IGAFD_CUDA(cudaMemcpyAsync(R.span[k].data(), P->dir[k].span, P->nel[k] * sizeof(int),
                               cudaMemcpyDeviceToHost, s));
  }
  IGAFD_CUDA(cudaStreamSynchronize(s));
  std::vector<int2> all;
  for (int k = 0; k < 3; ++k) {
    R.sup[k].assign(P->dir[k].m, make_int2(0, 0));
    for (int e = 0; e < P->nel[k]; ++e)
      for (int a = 0; a <= p; ++a) {
        int2 &q = R.sup[k][R.span[k][e] - p + a];
        if (q.y++ == 0) q.x = e;
      }
    all.insert(all.end(), R.sup[k].begin(), R.sup[k].end());
    funcs += R.sup[k].size();
  }
  const int o_min = P->stencil_half ? P->n_off / 2 : 0;
  const long long ld = P->stencil_half ? P->sh_ld : P->Np;
  IGAFD_CUDA(cudaMemsetAsync(P->stencil, 0, (size_t)(P->n_off - o_min) * ld * sizeof(double), s));
  igafd_status st = IGAFD_ERR_OOM;
  double h[3] = {};
  if (cudaMalloc((void **)&R.dsup, funcs * sizeof(int2)) == cudaSuccess) R.held.push_back(R.dsup);
  if (cudaMalloc((void **)&R.best, 3 * sizeof(unsigned long long)) == cudaSuccess) R.held.push_back(R.best);
  if (R.held.size() == 2) {
    st = cudaMemcpyAsync(R.dsup, all.data(), funcs * sizeof(int2), cudaMemcpyHostToDevice, s) == cudaSuccess
             ? IGAFD_OK : IGAFD_ERR_CUDA;
    init_best_kernel<<<1, 1, 0, s>>>(R.best);
    // i2 whole and one i3 at a time if that takes at most 1 GB of scratch,
    // else i2 in chunks; then as many i3 per batch as keep T1, T2 and Q near
    // L2's size (fewer launches, and enough blocks for small patches)
    int chunk = P->n[1], batch = 1, C2, ring;
    while (chunk > 1 && R.need(chunk, 1, &C2, &ring) > (size_t)1 << 30) chunk = (chunk + 1) / 2;
    while (batch < P->n[2] && 2 * batch * (p + 1) * (2 * p + 1) <= 65535 &&
           R.need(chunk, 2 * batch, &C2, &ring) <= (size_t)192 << 20)
      batch *= 2;
    if (batch > P->n[2]) batch = P->n[2];
    if (st == IGAFD_OK) st = R.run(chunk, batch);
    while (st == IGAFD_ERR_OOM && (chunk > 1 || batch > 1)) {   // little memory left: smaller pieces
      if (batch > 1) batch = (batch + 1) / 2; else chunk = (chunk + 1) / 2;
      st = R.run(chunk, batch);
    }
    unsigned long long key[3] = {};
    if (st == IGAFD_OK &&
        (cudaMemcpyAsync(key, R.best, sizeof(key), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
         cudaStreamSynchronize(s) != cudaSuccess))
      st = IGAFD_ERR_CUDA;
    for (int i = 0; i < 3; ++i) h[i] = of_key(key[i]);
  } else {
    cudaGetLastError();
  }
  cudaStreamSynchronize(s);
  for (void *q : R.held) cudaFree(q);
  if (st != IGAFD_OK) return st;
  P->min_detJ = h[0];
  P->q_bound = h[2] / h[1];
  return h[0] > 0.0 ? IGAFD_OK : IGAFD_ERR_FOLDED;
}

// b += the load vector (b zeroed by the caller); see load_kernel.
igafd_status igafd_load3(igafd_patch *P, const double *fq, double *b, cudaStream_t s) {
  const PV v = make_view(P);
  switch (P->p) {
    case 1: return load_p<1>(v, fq, b, s);
    case 2: return load_p<2>(v, fq, b, s);
    case 3: return load_p<3>(v, fq, b, s);
    case 4: return load_p<4>(v, fq, b, s);
    case 5: return load_p<5>(v, fq, b, s);
    case 6: return load_p<6>(v, fq, b, s);
    default: return load_p<7>(v, fq, b, s);
  }
}
