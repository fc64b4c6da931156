// Setup of the compressed operator, all in FP64 on the device:
//   assembly of a defining tensor (eqs. (5)-(6)) directly in its circulant
//   embedding (Section V.A), 3-D FFT, and truncated HOSVD (Algorithm 1).
//
// HOSVD on the weighted octant.  The spectrum A of every component obeys
// A[.., P-k, ..] = s A[.., k, ..] along each axis (s = +-1), so row P-k of a
// mode unfolding is s times row k.  With E the P x H map that copies the H =
// P/2 + 1 distinct rows into all P rows (with signs) and D = diag(w),
// w_k = sqrt(2) for 0 < k < P/2 and 1 otherwise (E^H E = D^2):
//   * the unfolding of A has the same singular values as that of the
//     weighted octant A_w = A[0:H1, 0:H2, 0:H3] x1 D1 x2 D2 x3 D3;
//   * its left singular vectors are U = E D^-1 Y, Y those of A_w;
//   * the core A x1 U1^* x2 U2^* x3 U3^* equals A_w x1 Y1^* x2 Y2^* x3 Y3^*.
// So Algorithm 1 runs on an (P/2+1)^3 tensor, exactly, and only the H_q
// rows D^-1 Y of each factor are stored (the others follow by the sign).
//
// The singular vectors come from the Hermitian Gram matrix of each
// unfolding, diagonalised by parallel cyclic Jacobi.  Because forming the
// Gram matrix squares the singular values, a second pass re-forms the Gram
// matrix of Y^* A_w^(q) (rows nearly orthogonal, norms sigma_j) and
// diagonalises it again; Jacobi on that graded, nearly diagonal matrix
// gives the small singular values to high relative accuracy, which the
// 1e-8 truncation threshold needs.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <vector>

#include <cooperative_groups.h>

#include "vie_internal.cuh"
#include "stages.cuh"

namespace {

constexpr double kPi = 3.14159265358979323846;

// One component of h^3 (k0^2 delta_ab + d_a d_b) g at the voxel-centre offset
// (o1, o2, o3) h, or the equivalent-sphere self term at zero offset.
__device__ double2 dyadic_entry(int ca, int cb, int o1, int o2, int o3, double h, double k0, double2 self) {
  if (o1 == 0 && o2 == 0 && o3 == 0) return ca == cb ? self : make_double2(0.0, 0.0);
  const double R[3] = {o1 * h, o2 * h, o3 * h};
  const double r = sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]);
  double sn, cs;
  sincos(k0 * r, &sn, &cs);
  const double inv4pir = 1.0 / (4.0 * kPi * r);
  const double2 g = make_double2(cs * inv4pir, -sn * inv4pir);   // exp(-i k0 r)/(4 pi r)
  const double ir = 1.0 / r;
  const double2 diag = make_double2(k0 * k0 - ir * ir, -k0 * ir);
  const double2 dyad = make_double2(-k0 * k0 + 3.0 * ir * ir, 3.0 * k0 * ir);
  const double Ra = ca == 0 ? R[0] : (ca == 1 ? R[1] : R[2]), Rb = cb == 0 ? R[0] : (cb == 1 ? R[1] : R[2]);
  const double rr = (Ra * ir) * (Rb * ir);
  double2 f = make_double2(dyad.x * rr, dyad.y * rr);
  if (ca == cb) f = f + diag;
  return (h * h * h) * (g * f);
}

// One component at every circulant index.  Each entry is evaluated once, at its
// non-negative offsets, and written to its up to eight mirror images (an odd
// coordinate flips the sign, exactly); index n of an axis holds zeros.  The
// evaluation is bound by FP64 arithmetic (a sincos, a square root and two
// divisions), so an eighth of the evaluations is an eighth of the time.
__global__ void assemble_kernel(double2* out, int ca, int cb, int n1, int n2, int n3, int P1,
                                int P2, int P3, double h, double k0, double2 self) {
  const unsigned total = (unsigned)(n1 + 1) * (n2 + 1) * (n3 + 1);
  const double s1 = ((ca == 0) != (cb == 0)) ? -1.0 : 1.0, s2 = ((ca == 1) != (cb == 1)) ? -1.0 : 1.0,
               s3 = ((ca == 2) != (cb == 2)) ? -1.0 : 1.0;
  for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    const int o3 = (int)(idx % (unsigned)(n3 + 1)), q = (int)(idx / (unsigned)(n3 + 1));
    const int o2 = q % (n2 + 1), o1 = q / (n2 + 1);
    double2 v = make_double2(0.0, 0.0);
    if (o1 < n1 && o2 < n2 && o3 < n3) v = dyadic_entry(ca, cb, o1, o2, o3, h, k0, self);
    const int m1 = (o1 == 0 || o1 == n1) ? 1 : 2, m2 = (o2 == 0 || o2 == n2) ? 1 : 2,
              m3 = (o3 == 0 || o3 == n3) ? 1 : 2;
    for (int a = 0; a < m1; ++a)
      for (int b = 0; b < m2; ++b)
        for (int c = 0; c < m3; ++c) {
          const int i1 = a ? P1 - o1 : o1, i2 = b ? P2 - o2 : o2, i3 = c ? P3 - o3 : o3;
          const double sg = (a ? s1 : 1.0) * (b ? s2 : 1.0) * (c ? s3 : 1.0);
          out[((long long)i1 * P2 + i2) * P3 + i3] = sg * v;
        }
  }
}

// max |A[mirror] - s A|^2 and max |A|^2 over the tensor (non-negative doubles
// compare like their bit patterns; no square root per entry).
__global__ void parity_check_kernel(const double2* A, int P1, int P2, int P3, int s1, int s2, int s3,
                                    unsigned long long* out) {
  const long long total = (long long)P1 * P2 * P3;
  double dev = 0.0, mx = 0.0;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int i3 = (int)(idx % P3);
    const int i2 = (int)((idx / P3) % P2);
    const int i1 = (int)(idx / ((long long)P2 * P3));
    const double2 a = A[idx];
    const double s = (double)(s1 * s2 * s3);
    const int m1 = (P1 - i1) % P1, m2 = (P2 - i2) % P2, m3 = (P3 - i3) % P3;
    const double2 b = A[((long long)m1 * P2 + m2) * P3 + m3];
    dev = fmax(dev, abs2(b - s * a));
    mx = fmax(mx, abs2(a));
    // single-axis mirrors
    const double2 bx = A[((long long)m1 * P2 + i2) * P3 + i3];
    dev = fmax(dev, abs2(bx - (double)s1 * a));
    const double2 by = A[((long long)i1 * P2 + m2) * P3 + i3];
    dev = fmax(dev, abs2(by - (double)s2 * a));
  }
  for (int o = 16; o > 0; o >>= 1) {
    dev = fmax(dev, __shfl_down_sync(0xffffffffu, dev, o));
    mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out, __double_as_longlong(dev));
    atomicMax(out + 1, __double_as_longlong(mx));
  }
}

__global__ void octant_kernel(const double2* A, double2* Aw, int P1, int P2, int P3, int H1, int H2,
                              int H3) {
  const long long total = (long long)H1 * H2 * H3;
  const double r2 = 1.41421356237309504880;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int k3 = (int)(idx % H3);
    const int k2 = (int)((idx / H3) % H2);
    const int k1 = (int)(idx / ((long long)H2 * H3));
    double w = 1.0;
    if (k1 != 0 && 2 * k1 != P1) w *= r2;
    if (k2 != 0 && 2 * k2 != P2) w *= r2;
    if (k3 != 0 && 2 * k3 != P3) w *= r2;
    Aw[idx] = w * A[((long long)k1 * P2 + k2) * P3 + k3];
  }
}

// Factor-wise route (Section V.A): the weighted octant of the Toeplitz defining
// tensor itself, T_w[i1, i2, i3] = w(i1) w(i2) w(i3) T_ab(i1 h, i2 h, i3 h) for
// offsets 0 <= i_q < n_q, w(0) = 1, w(i > 0) = sqrt(2) (offsets +i and -i
// hold the same entry up to the component's parity sign).
__global__ void toeplitz_octant_kernel(double2* out, int ca, int cb, int n1, int n2, int n3, double h,
                                       double k0, double2 self) {
  const long long total = (long long)n1 * n2 * n3;
  const double r2 = 1.41421356237309504880;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const int o3 = (int)(idx % n3);
    const int o2 = (int)((idx / n3) % n2);
    const int o1 = (int)(idx / ((long long)n2 * n3));
    const double2 v = dyadic_entry(ca, cb, o1, o2, o3, h, k0, self);
    double w = 1.0;
    if (o1 != 0) w *= r2;
    if (o2 != 0) w *= r2;
    if (o3 != 0) w *= r2;
    out[idx] = w * v;
  }
}

// Rows k = 0 .. P/2 of the embedded, DFT'd factor, normalised to orthonormal
// columns: out[k][j] = P^-1/2 sum_{|i| < n} U[i][j] exp(-2 pi i k i / P), with
// U[-i] = s U[i] and the stored rows U[i], i = 0..n-1 (Uh [n][r]):
//   out[k][j] = P^-1/2 (U[0][j] + sum_{i >= 1} U[i][j] (w^{ki} + s conj(w^{ki}))).
__global__ void factor_dft_kernel(const double2* Uh, double2* out, const double2* roots, int n, int P,
                                  int r, int s) {
  const int total = (P / 2 + 1) * r;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    const int k = idx / r, j = idx % r;
    double2 acc = Uh[j];
    for (int i = 1; i < n; ++i) {
      const double2 w = roots[(int)(((long long)k * i) % P)];
      const double2 c = make_double2(w.x + s * w.x, w.y - s * w.y);
      acc = cmadd(Uh[(long long)i * r + j], c, acc);
    }
    const double sc = 1.0 / sqrt((double)P);
    out[idx] = make_double2(sc * acc.x, sc * acc.y);
  }
}

__global__ void to_c64_kernel(const double2* a, float2* b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    b[i] = make_float2((float)a[i].x, (float)a[i].y);
}

// element (i, m) of the mode-q unfolding of a D0 x D1 x D2 tensor (at most 513^3
// entries: 32-bit indices)
__device__ __forceinline__ unsigned unfold_index(int q, unsigned i, unsigned m, unsigned D1, unsigned D2) {
  if (q == 0) return i * D1 * D2 + m;
  if (q == 1) return (m / D2) * D1 * D2 + i * D2 + m % D2;
  return m * D2 + i;
}

// Partial Gram matrices part[z] = X_z X_z^* of the mode-q unfolding X (Dq x M),
// X_z its z-th range of columns: one 16 x 16 tile of the upper triangle per CTA
// and range.  FP64 arithmetic bounds it (2 fused multiply-adds per clock and SM),
// so the column ranges are there to occupy every SM: with one CTA per tile and no
// ranges, 25 CTAs of a 65^3 octant took 1.9 ms per mode.
__global__ void __launch_bounds__(256) gram_kernel(const double2* __restrict__ X, double2* part, int q, int D0,
                                                   int D1, int D2, int ntile, unsigned chunk) {
  __shared__ double2 Ai[16][17], Aj[16][17];
  const unsigned Dq = q == 0 ? D0 : (q == 1 ? D1 : D2);
  const unsigned M = (unsigned)D0 * D1 * D2 / Dq;
  int ti = 0, tj = blockIdx.x;                          // tile row ti <= tj
  while (tj >= ntile - ti) {
    tj -= ntile - ti;
    ++ti;
  }
  tj += ti;
  const unsigned tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const unsigned i0 = ti * 16, j0 = tj * 16;
  const unsigned mlo = blockIdx.y * chunk, mhi = min(M, mlo + chunk);
  // consecutive threads read consecutive addresses: along m, or along i for mode 3
  const unsigned li = q == 2 ? tx : ty, lm = q == 2 ? ty : tx;
  double2 acc = make_double2(0.0, 0.0);
  for (unsigned m0 = mlo; m0 < mhi; m0 += 16) {
    const unsigned m = m0 + lm;
    Ai[li][lm] = (i0 + li < Dq && m < mhi) ? X[unfold_index(q, i0 + li, m, D1, D2)] : make_double2(0, 0);
    Aj[li][lm] = (j0 + li < Dq && m < mhi) ? X[unfold_index(q, j0 + li, m, D1, D2)] : make_double2(0, 0);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const double2 u = Ai[ty][k], v = Aj[tx][k];       // acc += u conj(v)
      acc.x = fma(u.x, v.x, fma(u.y, v.y, acc.x));
      acc.y = fma(u.y, v.x, fma(-u.x, v.y, acc.y));
    }
    __syncthreads();
  }
  if (i0 + ty < Dq && j0 + tx < Dq)
    part[((size_t)blockIdx.y * Dq + i0 + ty) * Dq + j0 + tx] = acc;
}

// G = sum of the partial Gram matrices, in order; the lower triangle is the
// conjugate of the upper one, the diagonal real
__global__ void gram_sum_kernel(const double2* part, double2* G, int D, int nz) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < D * D; idx += gridDim.x * blockDim.x) {
    const int i = idx / D, j = idx % D;
    const bool up = i <= j;
    const int src = up ? idx : j * D + i;
    // tiles hold their whole 16 x 16 square, so (i, j) with i > j inside a diagonal
    // tile exists too; the upper entry is used for both
    double2 s = make_double2(0.0, 0.0);
    for (int z = 0; z < nz; ++z) s = s + part[(size_t)z * D * D + src];
    if (i == j) s.y = 0.0;
    G[idx] = up ? s : conjg(s);
  }
}

// out = in x_q M with M(i, t) = Mat[t * ld + i] (conjugated if cj):
// out[p, i, r] = sum_t in[p, t, r] M(i, t); in is Dpre x Dm x Dpost.
__global__ void mode_product_kernel(const double2* in, double2* out, const double2* Mat, int ld,
                                    int cj, long long Dpre, int Dm, long long Dpost, int Rm) {
  const long long total = Dpre * Rm * Dpost;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long r = idx % Dpost;
    const int i = (int)((idx / Dpost) % Rm);
    const long long p = idx / (Dpost * Rm);
    const double2* src = in + p * Dm * Dpost + r;
    double2 acc = make_double2(0.0, 0.0);
    for (int t = 0; t < Dm; ++t) {
      double2 mv = Mat[(long long)t * ld + i];
      if (cj) mv = conjg(mv);
      acc = cmadd(src[(long long)t * Dpost], mv, acc);
    }
    out[idx] = acc;
  }
}

struct JacobiJob {
  double2* A;     // m x m Hermitian, overwritten (diagonal = eigenvalues)
  double2* V;     // m x m eigenvectors (columns)
  int m;
};

// One rotation of a Jacobi step: columns p < q (q < 0: the index left over when m
// is odd), new p' = c p - conj(s) q, q' = s p + c q; np, nq the rotated diagonal.
struct JacobiRot {
  double c, np, nq;
  double2 s;
  int p, q;
};

constexpr int kJacobiCtas = 8;        // CTAs (one cluster) per matrix
constexpr int kJacobiThreads = 256;
constexpr int kJacobiMaxPairs = 257;

// Parallel cyclic Jacobi (round-robin pairing, all disjoint rotations of a step
// applied at once), one cluster of eight CTAs per matrix, every matrix of a group
// of components in one launch.  A pair (p, q) is rotated when |a_pq|^2 > tol^2
// |a_pp a_qq|; the sweep loop stops after a sweep without rotations or after
// max_sweeps (status -1).
//
// A step is bound by FP64 issue (a warp instruction occupies its SM quarter for 64
// clocks, with one lane or 32), so it is spread over the cluster's 32 quarters, warp
// by warp, with full warps:
//   1. the first warp of every CTA forms the rotations of its pairs and writes them
//      into every CTA's shared memory, while the warps of the other quarters apply
//      the previous step's rotations to V;
//   2. each 2 x 2 block (pair i, pair j > i) of A is rotated from both sides by one
//      thread, which also writes its mirror image.
// One cluster barrier after each.  A and V change hands between SMs through L2.
// Eighteen 65 x 65 matrices: about 8 ms a pass (14.3 ms with the rotations' square
// roots and divisions taken one by one, V in a third phase and half-empty warps; 20
// ms for three of them with one CTA each).
__global__ void __launch_bounds__(kJacobiThreads) jacobi_kernel(const JacobiJob* jobs, int max_sweeps,
                                                                double tol, int* rotated, int* status) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int jobid = blockIdx.x / kJacobiCtas;
  const JacobiJob job = jobs[jobid];
  const int m = job.m, mm = m + (m & 1), M = mm - 1, npair = mm / 2;
  double2* A = job.A;
  double2* V = job.V;
  __shared__ JacobiRot rots[2][kJacobiMaxPairs];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kWarps = kJacobiThreads / 32;
  const int gt = (warp * kJacobiCtas + rank) * 32 + lane, gn = kJacobiCtas * kJacobiThreads;
  // V's warps: those off the first quarter (warps 0 and 4 share it)
  const int vwarp = warp < 4 ? warp - 1 : warp - 2, vn = (kWarps - 2) * kJacobiCtas * 32;
  const bool on_v = (warp & 3) != 0;
  const int nblk = npair * (npair - 1) / 2;
  const double tol2 = tol * tol;
  for (int e = gt; e < m * m; e += gn) V[e] = make_double2((e / m) == (e % m) ? 1.0 : 0.0, 0.0);
  cluster.sync();
  auto update_v = [&](const JacobiRot* rot) {            // V <- V J
    if (!on_v) return;
    for (int it = (vwarp * kJacobiCtas + rank) * 32 + lane; it < npair * m; it += vn) {
      const int k = it / npair, bj = it - k * npair;
      const JacobiRot& rj = rot[bj];
      if (rj.q < 0 || (rj.s.x == 0.0 && rj.s.y == 0.0)) continue;
      const double2 vp = __ldcg(&V[k * m + rj.p]), vq = __ldcg(&V[k * m + rj.q]);
      V[k * m + rj.p] = conj_madd(make_double2(-rj.s.x, -rj.s.y), vq, rj.c * vp);
      V[k * m + rj.q] = cmadd(rj.s, vp, rj.c * vq);
    }
  };
  int sweep = 0, buf = 0;
  bool done = (m <= 1), pending = false;
  for (; sweep < max_sweeps && !done; ++sweep) {
    int* flag = rotated + jobid * max_sweeps + sweep;
    for (int step = 0; step < M; ++step, buf ^= 1) {
      JacobiRot* rot = rots[buf];
      if (warp == 0) {
        // this CTA's pairs: rank, rank + 8, ...
        for (int i = rank + kJacobiCtas * lane; i < npair; i += 32 * kJacobiCtas) {
          int p, q;
          if (i == 0) { p = 0; q = 1 + step; }
          else { p = 1 + (step + i) % M; q = 1 + (step - i + M) % M; }
          if (p > q) { int t = p; p = q; q = t; }
          JacobiRot r;
          r.c = 1.0;
          r.np = r.nq = 0.0;
          r.s = make_double2(0.0, 0.0);
          r.p = p;
          r.q = q < m ? q : -1;
          if (q < m) {
            const double app = __ldcg(&A[p * m + p]).x, aqq = __ldcg(&A[q * m + q]).x;
            const double2 apq = __ldcg(&A[p * m + q]);
            const double a2 = abs2(apq);
            if (a2 > tol2 * fabs(app * aqq) && a2 > 0.0) {
              const double rmag = rsqrt(a2), mag = a2 * rmag;
              const double th = 0.5 * (aqq - app) * rmag, ath = fabs(th);
              const double u = fma(th, th, 1.0);
              // t = sign(th) / (|th| + sqrt(th^2 + 1))
              const double t = copysign(1.0 / (ath + (ath > 1e9 ? ath : u * rsqrt(u))), th);
              r.c = rsqrt(fma(t, t, 1.0));
              const double sm = t * r.c * rmag;
              r.s = make_double2(sm * apq.x, sm * apq.y);          // s e^{i phi}
              r.np = fma(-t, mag, app);                             // rotated diagonal
              r.nq = fma(t, mag, aqq);
              *flag = 1;
            }
          }
          for (int k = 0; k < kJacobiCtas; ++k) cluster.map_shared_rank(rot, k)[i] = r;
        }
      } else if (pending) {
        update_v(rots[buf ^ 1]);
      }
      pending = true;
      cluster.sync();
      // A <- J^* A J: the diagonal blocks, then the blocks (i, j > i) and their mirror
      // images (the index runs along the rows of the strict upper triangle)
      for (int it = gt; it < nblk + npair; it += gn) {
        if (it >= nblk) {
          // the rotation annihilates a_pq exactly and moves t|a_pq| between a_pp and
          // a_qq; writing those values (instead of the rounded updates) lets the
          // relative stopping test be met on graded matrices
          const JacobiRot& ri = rot[it - nblk];
          if (ri.s.x == 0.0 && ri.s.y == 0.0) continue;
          A[ri.p * m + ri.p] = make_double2(ri.np, 0.0);
          A[ri.q * m + ri.q] = make_double2(ri.nq, 0.0);
          A[ri.p * m + ri.q] = make_double2(0.0, 0.0);
          A[ri.q * m + ri.p] = make_double2(0.0, 0.0);
          continue;
        }
        // row bi starts at bi (2 npair - bi - 1) / 2
        const float w = 2 * npair - 1;
        int bi = (int)(0.5f * (w - sqrtf(w * w - 8.f * it)));
        bi = max(0, min(bi, npair - 2));
        while (bi > 0 && bi * (2 * npair - bi - 1) / 2 > it) --bi;
        while (bi < npair - 2 && (bi + 1) * (2 * npair - bi - 2) / 2 <= it) ++bi;
        const int bj = it - bi * (2 * npair - bi - 1) / 2 + bi + 1;
        const JacobiRot& ri = rot[bi];
        const JacobiRot& rj = rot[bj];
        const bool zi = ri.s.x == 0.0 && ri.s.y == 0.0, zj = rj.s.x == 0.0 && rj.s.y == 0.0;
        if (zi && zj) continue;
        const double2 z = make_double2(0.0, 0.0);
        const bool hi = ri.q >= 0, hj = rj.q >= 0;
        double2 pp = __ldcg(&A[ri.p * m + rj.p]), pq = hj ? __ldcg(&A[ri.p * m + rj.q]) : z;
        double2 qp = hi ? __ldcg(&A[ri.q * m + rj.p]) : z, qq = hi && hj ? __ldcg(&A[ri.q * m + rj.q]) : z;
        if (!zi) {                                      // rows: p' = c p - s q, q' = conj(s) p + c q
          const double2 ns = make_double2(-ri.s.x, -ri.s.y);
          const double2 u = cmadd(ns, qp, ri.c * pp), v = conj_madd(ri.s, pp, ri.c * qp);
          const double2 u2 = cmadd(ns, qq, ri.c * pq), v2 = conj_madd(ri.s, pq, ri.c * qq);
          pp = u; qp = v; pq = u2; qq = v2;
        }
        if (!zj) {                                      // columns: p' = c p - conj(s) q, q' = s p + c q
          const double2 ns = make_double2(-rj.s.x, -rj.s.y);
          const double2 u = conj_madd(ns, pq, rj.c * pp), v = cmadd(rj.s, pp, rj.c * pq);
          const double2 u2 = conj_madd(ns, qq, rj.c * qp), v2 = cmadd(rj.s, qp, rj.c * qq);
          pp = u; pq = v; qp = u2; qq = v2;
        }
        A[ri.p * m + rj.p] = pp;
        A[rj.p * m + ri.p] = conjg(pp);
        if (hj) {
          A[ri.p * m + rj.q] = pq;
          A[rj.q * m + ri.p] = conjg(pq);
        }
        if (hi) {
          A[ri.q * m + rj.p] = qp;
          A[rj.p * m + ri.q] = conjg(qp);
        }
        if (hi && hj) {
          A[ri.q * m + rj.q] = qq;
          A[rj.q * m + ri.q] = conjg(qq);
        }
      }
      cluster.sync();
    }
    done = __ldcg(flag) == 0;            // the same for every CTA: set before the last barrier
  }
  if (pending) update_v(rots[buf ^ 1]);
  if (rank == 0 && threadIdx.x == 0) status[jobid] = done ? sweep : -1;
}

int grid_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  if (b < 1) b = 1;
  return (int)b;
}

void make_roots(int N, std::vector<double2>& r64, std::vector<float2>& r32) {
  r64.resize(N);
  r32.resize(N);
  for (int m = 0; m < N; ++m) {
    const double a = -2.0 * kPi * (double)m / (double)N;
    r64[m] = make_double2(std::cos(a), std::sin(a));
    r32[m] = make_float2((float)r64[m].x, (float)r64[m].y);
  }
}

template <typename P> int dalloc(P** p, size_t bytes) {
  cudaError_t e = cudaMalloc((void**)p, bytes ? bytes : 16);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("device allocation of %zu bytes failed", bytes);
    return VIE_ERR_OOM;
  }
  return VIE_OK;
}

// Scratch of a setup that compresses `comps` components at a time; the arrays [6]
// are indexed by the component's place in its group.
struct DeviceBuffers {
  int comps = 0;
  double2* full = nullptr;       // P1 P2 P3
  double2* aw[6] = {};           // H1 H2 H3: the group's weighted octants
  double2* tmp = nullptr;        // H1 H2 H3
  double2* gram[6][3] = {};      // Hq x Hq
  double2* vec[6][3] = {};       // Hq x Hq
  double2* vec2[6][3] = {};      // Hq x Hq
  double2* ytr = nullptr;        // truncated Y, max Hq x Hq
  double2* part = nullptr;       // partial Gram matrices: in `full` where they fit, the
  double2* part_own = nullptr;   // spectrum being out of use by then, else here
  size_t part_entries = 0;
  JacobiJob* jobs = nullptr;     // [18]
  int* jstatus = nullptr;        // [18], then the sweeps' rotation flags [18][kJacobiSweeps]
  unsigned long long* red = nullptr;   // [6][2]
  void release_group() {
    for (int i = 0; i < 6; ++i) {
      cudaFree(aw[i]);
      aw[i] = nullptr;
      for (int q = 0; q < 3; ++q) {
        for (double2** p : {&gram[i][q], &vec[i][q], &vec2[i][q]}) {
          cudaFree(*p);
          *p = nullptr;
        }
      }
    }
  }
  ~DeviceBuffers() {
    cudaFree(full); cudaFree(tmp); cudaFree(ytr); cudaFree(part_own);
    release_group();
    cudaFree(jobs); cudaFree(jstatus); cudaFree(red);
  }
};

constexpr int kJacobiSweeps = 60;

// Components compressed at a time.  All six together keep the eigen-solver's SMs
// busy, but hold six octants and 54 matrices: at 256^3 2.2 s with 4.1 GB of scratch
// (factor-wise route, which is there to do without the 2.1 GB spectrum: 1.9 s, 1.95
// GB), one by one 3.9 s with 2.7 GB (3.5 s, 0.55 GB).  So a group may hold
// kSetupExtra more than one component's scratch: six together up to about 100^3
// (96^3: 88 ms), three at 128^3 (258 ms; six 217 ms), one from about 200^3.
constexpr size_t kSetupExtra = 128u << 20;
int setup_group(size_t comp_bytes) {
  for (int g : {6, 3, 2})
    if ((g - 1) * comp_bytes <= kSetupExtra) return g;
  return 1;
}

// upper-triangle 16 x 16 tiles of a D x D Gram matrix, and its column ranges: enough
// CTAs for about four per SM
int gram_tiles(int D) {
  const int n = (D + 15) / 16;
  return n * (n + 1) / 2;
}
int gram_ranges(int D, long long M) {
  const long long want = (4LL * device_sms() + gram_tiles(D) - 1) / gram_tiles(D);
  return (int)std::max<long long>(1, std::min<long long>(want, (M + 255) / 256));
}

}  // namespace

// 3-D FFT of a P1 x P2 x P3 FP64 array in place (three line stages).
static void fft3d_f64(const vie_op* op, double2* a, cudaStream_t s) {
  const long long P1 = op->P[0], P2 = op->P[1], P3 = op->P[2];
  for (int axis = 0; axis < 3; ++axis) {
    LineArgs<double> L = {};
    L.in = a;
    L.out = a;
    L.roots = op->roots64[axis];
    L.plan = op->plan[axis];
    L.lin = L.lout = op->P[axis];
    L.scale = 1.0;
    L.nbatch = 1;
    L.batch_per_rhs = 1;
    L.prof_family = PF_SETUP;
    if (axis == 0) {          // lines along x, columns z, other y
      L.nother = (int)P2; L.ncol = (int)P3;
      L.in_os = L.out_os = P3; L.in_ls = L.out_ls = P2 * P3; L.in_cs = L.out_cs = 1;
    } else if (axis == 1) {   // lines along y, columns z, other x
      L.nother = (int)P1; L.ncol = (int)P3;
      L.in_os = L.out_os = P2 * P3; L.in_ls = L.out_ls = P3; L.in_cs = L.out_cs = 1;
    } else {                  // lines along z (contiguous), columns y, other x
      L.nother = (int)P1; L.ncol = (int)P2;
      L.in_os = L.out_os = P2 * P3; L.in_ls = L.out_ls = 1; L.in_cs = L.out_cs = P3;
    }
    launch_line_fft<double>(L, s);
  }
}

// (2/3)(1 + i k0 a) exp(-i k0 a) - 1 (or without the -1/3 part), a = h (3/4pi)^(1/3)
static double2 self_term_value(const vie_op* op) {
  const double h = op->grid.h, k0 = op->k0;
  const double a = h * std::cbrt(3.0 / (4.0 * kPi));
  const double ca_ = std::cos(k0 * a), sa_ = std::sin(k0 * a);
  double2 self = make_double2((2.0 / 3.0) * (ca_ + k0 * a * sa_) - 1.0,
                              (2.0 / 3.0) * (k0 * a * ca_ - sa_));
  if (op->flags & VIE_SELF_TERM_PV) self.x += 1.0 / 3.0;
  return self;
}

int assemble_spectrum(const vie_op* op, int c, double2* out, cudaStream_t s) {
  int ca, cb;
  component_axes(c, &ca, &cb);
  const double h = op->grid.h, k0 = op->k0;
  const double2 self = self_term_value(op);
  const long long total = (long long)op->P[0] * op->P[1] * op->P[2];
  assemble_kernel<<<grid_for(total), 256, 0, s>>>(out, ca, cb, op->n[0], op->n[1], op->n[2],
                                                   op->P[0], op->P[1], op->P[2], h, k0, self);
  fft3d_f64(op, out, s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_status(e, "assemble/fft");
  return VIE_OK;
}

static int init_tables(vie_op* op) {
  VIE_TRY(line_fft_init_attributes());
  VIE_TRY(fused_init_attributes());
  VIE_TRY(multi_init_attributes());
  VIE_TRY(tp_init_attributes());
  VIE_TRY(umma_init_attributes());
  VIE_TRY(plane_init_attributes());
  for (int q = 0; q < 3; ++q) {
    const int N = op->P[q];
    if (!make_plan(N, &op->plan[q])) {
      set_error("padded size %d has a prime factor above 7", N);
      return VIE_ERR_ARG;
    }
    std::vector<double2> r64;
    std::vector<float2> r32;
    make_roots(N, r64, r32);
    VIE_TRY(dalloc(&op->roots64[q], N * sizeof(double2)));
    VIE_TRY(dalloc(&op->roots32[q], N * sizeof(float2)));
    VIE_CUDA(cudaMemcpy(op->roots64[q], r64.data(), N * sizeof(double2), cudaMemcpyHostToDevice));
    VIE_CUDA(cudaMemcpy(op->roots32[q], r32.data(), N * sizeof(float2), cudaMemcpyHostToDevice));
    VIE_TRY(plan_prepare(N));
  }
  return VIE_OK;
}

// Gram matrix of the mode-q unfolding of an H[0] x H[1] x H[2] tensor
static void launch_gram(DeviceBuffers& d, const double2* X, double2* G, int q, const int* H, cudaStream_t s) {
  const int D = H[q], n = (D + 15) / 16;
  const long long M = (long long)H[0] * H[1] * H[2] / D;
  const int nz = gram_ranges(D, M);
  const unsigned chunk = (unsigned)(((M + nz - 1) / nz + 15) / 16 * 16);
  gram_kernel<<<dim3(gram_tiles(D), nz), 256, 0, s>>>(X, d.part, q, H[0], H[1], H[2], n, chunk);
  gram_sum_kernel<<<grid_for((long long)D * D), 256, 0, s>>>(d.part, G, D, nz);
}

// Diagonalise the Gram matrices of the group's components (first: c0; 3 modes each)
// in one launch.
static int run_jacobi(DeviceBuffers& d, int c0, double2* (&V)[6][3], const int* H, cudaStream_t s) {
  constexpr int kMaxJobs = 18;
  const int njobs = 3 * d.comps;
  JacobiJob jobs[kMaxJobs];
  for (int j = 0; j < njobs; ++j) jobs[j] = JacobiJob{d.gram[j / 3][j % 3], V[j / 3][j % 3], H[j % 3]};
  int* flags = d.jstatus + kMaxJobs;
  VIE_CUDA(cudaMemcpyAsync(d.jobs, jobs, njobs * sizeof(JacobiJob), cudaMemcpyHostToDevice, s));
  VIE_CUDA(cudaMemsetAsync(flags, 0, njobs * kJacobiSweeps * sizeof(int), s));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(njobs * kJacobiCtas);
  cfg.blockDim = dim3(kJacobiThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kJacobiCtas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  VIE_CUDA(cudaLaunchKernelEx(&cfg, jacobi_kernel, (const JacobiJob*)d.jobs, (int)kJacobiSweeps, 1e-15, flags,
                              d.jstatus));
  int st[kMaxJobs];
  VIE_CUDA(cudaMemcpyAsync(st, d.jstatus, njobs * sizeof(int), cudaMemcpyDeviceToHost, s));
  VIE_CUDA(cudaStreamSynchronize(s));
  for (int j = 0; j < njobs; ++j) {
    if (st[j] < 0) {
      set_error("Jacobi eigen-solver did not converge (component %d, matrix %d, size %d)", c0 + j / 3, j % 3,
                H[j % 3]);
      return VIE_ERR_NUMERIC;
    }
  }
  return VIE_OK;
}

static size_t rank_from_sigma2(const std::vector<double>& s2, double tol, int rule, double norm2) {
  const size_t H = s2.size();
  if (H == 0 || s2[0] <= 0.0) return 1;
  if (rule == VIE_RANK_SIGMA_MAX) {
    const double thr = tol / std::sqrt(3.0) * std::sqrt(s2[0]);
    size_t r = 0;
    for (size_t j = 0; j < H; ++j)
      if (std::sqrt(s2[j]) >= thr) ++r;
    return std::max<size_t>(r, 1);
  }
  const double bound = tol / std::sqrt(3.0) * std::sqrt(norm2);
  std::vector<double> tail(H + 1, 0.0);
  for (size_t j = H; j-- > 0;) tail[j] = tail[j + 1] + s2[j];
  for (size_t r = 1; r <= H; ++r)
    if (std::sqrt(tail[r]) <= bound) return r;
  return H;
}

// Compression of the six components (op->comp).  Spectrum route: Algorithm 1 on
// the weighted octant of the FFT'd circulant component.  Factor-wise route
// (VIE_SETUP_FACTORWISE, Section V.A): Algorithm 1 on the weighted octant of
// the Toeplitz defining tensor, then the embedding and DFT of each factor
// column; F_q E_q / sqrt(P_q) is an isometry, so both routes give the same
// ranks and the same truncated model (core scaled by sqrt(P1 P2 P3)).
// The components of a group go through each stage together, so that the eigen-solver,
// a long chain on few SMs per matrix, runs once per pass on all their matrices.

// dimensions of the weighted octant the HOSVD runs on
static void octant_dims(const vie_op* op, bool factorwise, int* H) {
  for (int q = 0; q < 3; ++q) H[q] = factorwise ? op->n[q] : op->H[q];
}

// weighted octant of component c into aw; its parity check into d.red[2 c]
static int component_octant(vie_op* op, int c, double2* aw, DeviceBuffers& d, cudaStream_t s, bool factorwise) {
  const int P1 = op->P[0], P2 = op->P[1], P3 = op->P[2];
  int H[3];
  octant_dims(op, factorwise, H);
  const long long full = (long long)P1 * P2 * P3;
  const long long oct = (long long)H[0] * H[1] * H[2];
  TuckerComp& tc = op->comp[c];
  for (int q = 0; q < 3; ++q) tc.s[q] = component_parity(c, q);
  if (!factorwise || op->spec64 != nullptr) {
    VIE_TRY(assemble_spectrum(op, c, d.full, s));
    // the symmetry every later step relies on
    parity_check_kernel<<<grid_for(full), 256, 0, s>>>(d.full, P1, P2, P3, tc.s[0], tc.s[1], tc.s[2],
                                                        d.red + 2 * c);
    if (op->spec64) {
      VIE_CUDA(cudaMemcpyAsync(op->spec64 + c * full, d.full, full * sizeof(double2),
                               cudaMemcpyDeviceToDevice, s));
      to_c64_kernel<<<grid_for(full), 256, 0, s>>>(d.full, op->spec32 + c * full, full);
    }
  }
  if (!factorwise) {
    octant_kernel<<<grid_for(oct), 256, 0, s>>>(d.full, aw, P1, P2, P3, H[0], H[1], H[2]);
  } else {
    int ca, cb;
    component_axes(c, &ca, &cb);
    toeplitz_octant_kernel<<<grid_for(oct), 256, 0, s>>>(aw, ca, cb, H[0], H[1], H[2], op->grid.h,
                                                          op->k0, self_term_value(op));
  }
  VIE_CUDA(cudaGetLastError());
  return VIE_OK;
}

// Both eigen-solver passes of the components [c0, c0 + d.comps): d.vec and d.vec2
// hold the eigenvectors Y and V2, the diagonals of d.gram the squared singular values.
static int component_eigenvectors(vie_op* op, int c0, DeviceBuffers& d, cudaStream_t s, bool factorwise) {
  int H[3];
  octant_dims(op, factorwise, H);
  const long long oct = (long long)H[0] * H[1] * H[2];
  VIE_CUDA(cudaMemsetAsync(d.red, 0, 12 * sizeof(unsigned long long), s));
  // pass 1: Gram matrices of the three unfoldings and their eigenvectors Y
  for (int i = 0; i < d.comps; ++i) {
    VIE_TRY(component_octant(op, c0 + i, d.aw[i], d, s, factorwise));
    for (int q = 0; q < 3; ++q) launch_gram(d, d.aw[i], d.gram[i][q], q, H, s);
  }
  VIE_CUDA(cudaGetLastError());
  if (!factorwise || op->spec64 != nullptr) {
    unsigned long long red[12];
    VIE_CUDA(cudaMemcpyAsync(red, d.red, sizeof(red), cudaMemcpyDeviceToHost, s));
    VIE_CUDA(cudaStreamSynchronize(s));
    for (int c = c0; c < c0 + d.comps; ++c) {
      double dev, mx;
      std::memcpy(&dev, &red[2 * c], 8);
      std::memcpy(&mx, &red[2 * c + 1], 8);
      dev = std::sqrt(dev);
      mx = std::sqrt(mx);
      if (!(dev <= 1e-9 * mx + 1e-300) || !std::isfinite(mx)) {
        set_error("component %d spectrum breaks its mirror symmetry (%.3e of %.3e)", c, dev, mx);
        return VIE_ERR_NUMERIC;
      }
    }
  }
  VIE_TRY(run_jacobi(d, c0, d.vec, H, s));
  // pass 2: Gram of Y^* A_w^(q), eigenvectors V2; final vectors Y V2
  for (int i = 0; i < d.comps; ++i) {
    for (int q = 0; q < 3; ++q) {
      const long long Dpre = q == 0 ? 1 : (q == 1 ? H[0] : (long long)H[0] * H[1]);
      const long long Dpost = q == 0 ? (long long)H[1] * H[2] : (q == 1 ? H[2] : 1);
      mode_product_kernel<<<grid_for(oct), 256, 0, s>>>(d.aw[i], d.tmp, d.vec[i][q], H[q], 1, Dpre, H[q],
                                                        Dpost, H[q]);
      launch_gram(d, d.tmp, d.gram[i][q], q, H, s);
    }
  }
  VIE_CUDA(cudaGetLastError());
  return run_jacobi(d, c0, d.vec2, H, s);
}

// Ranks, core and stored factors of component c from its eigenvectors (place i).
static int compress_component(vie_op* op, int c, int i, double tol, int rule, DeviceBuffers& d,
                              cudaStream_t s, bool factorwise) {
  const int P1 = op->P[0], P2 = op->P[1], P3 = op->P[2];
  int H[3];
  octant_dims(op, factorwise, H);
  TuckerComp& tc = op->comp[c];

  // sort pass-2 eigenvalues, pick ranks, form Y V2 restricted to the kept columns
  double norm2 = 0.0;
  std::vector<double2> Ytr[3];
  for (int q = 0; q < 3; ++q) {
    const int h = H[q];
    std::vector<double2> G2(h), YV((size_t)h * h);             // G2: the diagonal
    VIE_CUDA(cudaMemcpy2DAsync(G2.data(), sizeof(double2), d.gram[i][q], (h + 1) * sizeof(double2),
                               sizeof(double2), h, cudaMemcpyDeviceToHost, s));
    // Y V2: view Y as [h][h][1] and contract its second index with V2
    mode_product_kernel<<<grid_for((long long)h * h), 256, 0, s>>>(d.vec[i][q], d.ytr, d.vec2[i][q], h,
                                                                   0, h, h, 1, h);
    VIE_CUDA(cudaGetLastError());
    VIE_CUDA(cudaMemcpyAsync(YV.data(), d.ytr, YV.size() * sizeof(double2), cudaMemcpyDeviceToHost,
                             s));
    VIE_CUDA(cudaStreamSynchronize(s));
    std::vector<double> lam(h);
    for (int j = 0; j < h; ++j) lam[j] = std::max(G2[j].x, 0.0);
    std::vector<int> order(h);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return lam[a] > lam[b]; });
    std::vector<double> s2(h);
    for (int j = 0; j < h; ++j) s2[j] = lam[order[j]];
    double sum = 0.0;
    for (double v : s2) sum += v;
    if (q == 0) norm2 = sum;
    // singular values of the spectrum's unfolding (P_q / 2 + 1 of them); the
    // factor-wise route has those of the Toeplitz tensor's, sqrt(P1 P2 P3) times smaller
    const double sig_scale = factorwise ? std::sqrt((double)P1 * P2 * P3) : 1.0;
    tc.sigma[q].assign(op->H[q], 0.0);
    for (int j = 0; j < h && j < op->H[q]; ++j) tc.sigma[q][j] = sig_scale * std::sqrt(s2[j]);
    // every mode sees the same ||A||_F; use mode 1's sum for all three
    const int r = (int)rank_from_sigma2(s2, tol, rule, norm2);
    tc.r[q] = r;
    Ytr[q].resize((size_t)h * r);
    for (int i = 0; i < h; ++i)
      for (int j = 0; j < r; ++j) Ytr[q][(size_t)i * r + j] = YV[(size_t)i * h + order[j]];
  }
  if (!(norm2 > 0.0) || !std::isfinite(norm2)) {
    set_error("component %d has zero or non-finite norm", c);
    return VIE_ERR_NUMERIC;
  }

  // core = A_w x1 Y1^* x2 Y2^* x3 Y3^*  (the truncated Y's go to d.vec2)
  const int r1 = tc.r[0], r2 = tc.r[1], r3 = tc.r[2];
  for (int q = 0; q < 3; ++q)
    VIE_CUDA(cudaMemcpy(d.vec2[i][q], Ytr[q].data(), Ytr[q].size() * sizeof(double2),
                        cudaMemcpyHostToDevice));
  mode_product_kernel<<<grid_for((long long)r1 * H[1] * H[2]), 256, 0, s>>>(
      d.aw[i], d.tmp, d.vec2[i][0], r1, 1, 1, H[0], (long long)H[1] * H[2], r1);
  mode_product_kernel<<<grid_for((long long)r1 * r2 * H[2]), 256, 0, s>>>(
      d.tmp, d.aw[i], d.vec2[i][1], r2, 1, r1, H[1], H[2], r2);
  mode_product_kernel<<<grid_for((long long)r1 * r2 * r3), 256, 0, s>>>(
      d.aw[i], d.tmp, d.vec2[i][2], r3, 1, (long long)r1 * r2, H[2], 1, r3);
  VIE_CUDA(cudaGetLastError());
  const size_t ncore = (size_t)r1 * r2 * r3;
  VIE_TRY(dalloc(&tc.core64, ncore * sizeof(double2)));
  VIE_TRY(dalloc(&tc.core32, ncore * sizeof(float2)));
  if (factorwise) {
    // the spectrum's core: the Toeplitz tensor's times sqrt(P1 P2 P3)
    const double sc = std::sqrt((double)P1 * P2 * P3);
    std::vector<double2> hc(ncore);
    VIE_CUDA(cudaMemcpyAsync(hc.data(), d.tmp, ncore * sizeof(double2), cudaMemcpyDeviceToHost, s));
    VIE_CUDA(cudaStreamSynchronize(s));
    for (auto& v : hc) v = make_double2(sc * v.x, sc * v.y);
    VIE_CUDA(cudaMemcpy(d.tmp, hc.data(), ncore * sizeof(double2), cudaMemcpyHostToDevice));
  }
  VIE_CUDA(cudaMemcpyAsync(tc.core64, d.tmp, ncore * sizeof(double2), cudaMemcpyDeviceToDevice, s));
  to_c64_kernel<<<grid_for(ncore), 256, 0, s>>>(tc.core64, tc.core32, (long long)ncore);

  // stored factor rows: U_half = D^-1 Y (rows 0..P/2 of the full factor); on the
  // factor-wise route D^-1 Y are the Toeplitz factor's rows at offsets 0..n-1, which
  // are embedded and DFT'd into rows 0..P/2 of the spectrum's factor
  for (int q = 0; q < 3; ++q) {
    const int h = op->H[q], r = tc.r[q];
    std::vector<double2> u64((size_t)h * r);
    std::vector<float2> u32((size_t)h * r);
    if (!factorwise) {
      for (int i = 0; i < h; ++i) {
        const double w = (i == 0 || 2 * i == op->P[q]) ? 1.0 : 1.0 / std::sqrt(2.0);
        for (int j = 0; j < r; ++j) {
          const double2 v = Ytr[q][(size_t)i * r + j];
          u64[(size_t)i * r + j] = make_double2(w * v.x, w * v.y);
        }
      }
    } else {
      const int n = op->n[q];
      std::vector<double2> ut((size_t)n * r);
      for (int i = 0; i < n; ++i) {
        const double w = i == 0 ? 1.0 : 1.0 / std::sqrt(2.0);
        for (int j = 0; j < r; ++j) {
          const double2 v = Ytr[q][(size_t)i * r + j];
          ut[(size_t)i * r + j] = make_double2(w * v.x, w * v.y);
        }
      }
      VIE_CUDA(cudaMemcpy(d.ytr, ut.data(), ut.size() * sizeof(double2), cudaMemcpyHostToDevice));
      factor_dft_kernel<<<grid_for((long long)h * r), 256, 0, s>>>(d.ytr, d.tmp, op->roots64[q], n,
                                                                    op->P[q], r, tc.s[q]);
      VIE_CUDA(cudaGetLastError());
      VIE_CUDA(cudaMemcpyAsync(u64.data(), d.tmp, u64.size() * sizeof(double2), cudaMemcpyDeviceToHost, s));
      VIE_CUDA(cudaStreamSynchronize(s));
    }
    for (size_t i = 0; i < u64.size(); ++i) u32[i] = make_float2((float)u64[i].x, (float)u64[i].y);
    VIE_TRY(dalloc(&tc.U64[q], u64.size() * sizeof(double2)));
    VIE_TRY(dalloc(&tc.U32[q], u32.size() * sizeof(float2)));
    VIE_CUDA(cudaMemcpy(tc.U64[q], u64.data(), u64.size() * sizeof(double2), cudaMemcpyHostToDevice));
    VIE_CUDA(cudaMemcpy(tc.U32[q], u32.data(), u32.size() * sizeof(float2), cudaMemcpyHostToDevice));
    if (q == 2) {
      // transposed copy: a warp rebuilding consecutive k3 reads consecutive addresses
      std::vector<float2> t((size_t)r * h);
      for (int i = 0; i < h; ++i)
        for (int j = 0; j < r; ++j) t[(size_t)j * h + i] = u32[(size_t)i * r + j];
      VIE_TRY(dalloc(&tc.U3t32, t.size() * sizeof(float2)));
      VIE_CUDA(cudaMemcpy(tc.U3t32, t.data(), t.size() * sizeof(float2), cudaMemcpyHostToDevice));
    }
  }
  VIE_CUDA(cudaStreamSynchronize(s));
  return VIE_OK;
}

static int finish_operator(vie_op* op) {
  for (int q = 0; q < 3; ++q) {
    op->rmax[q] = 1;
    for (int c = 0; c < 6; ++c) op->rmax[q] = std::max(op->rmax[q], op->comp[c].r[q]);
  }
  op->slab_stride = (size_t)op->H[0] * op->rmax[1] * op->rmax[2];
  VIE_TRY(dalloc(&op->slab32, 6 * op->slab_stride * sizeof(float2)));
  VIE_TRY(dalloc(&op->slab64, 6 * op->slab_stride * sizeof(double2)));
  CompMeta<float> m32[6];
  CompMeta<double> m64[6];
  for (int c = 0; c < 6; ++c) {
    const TuckerComp& tc = op->comp[c];
    m32[c] = CompMeta<float>{tc.U32[1], tc.U32[2], tc.U3t32, op->slab32 + c * op->slab_stride,
                             tc.r[1], tc.r[2], tc.s[0], tc.s[1], tc.s[2]};
    m64[c] = CompMeta<double>{tc.U64[1], tc.U64[2], nullptr, op->slab64 + c * op->slab_stride,
                              tc.r[1], tc.r[2], tc.s[0], tc.s[1], tc.s[2]};
  }
  static_assert(sizeof(CompMeta<float>) == sizeof(CompMeta<double>), "meta layout");
  VIE_TRY(dalloc(&op->dev_err, sizeof(int)));
  VIE_CUDA(cudaMemset(op->dev_err, 0, sizeof(int)));
  VIE_TRY(dalloc((char**)&op->meta, sizeof(m32) + sizeof(m64)));
  VIE_CUDA(cudaMemcpy(op->meta, m32, sizeof(m32), cudaMemcpyHostToDevice));
  VIE_CUDA(cudaMemcpy(static_cast<char*>(op->meta) + sizeof(m32), m64, sizeof(m64),
                      cudaMemcpyHostToDevice));
  // slab cores S_c[k1] = core_c x1 U1_c[k1, :]: the first stage of eq. (13), fixed
  // for the operator, so formed once here rather than at every matvec
  VIE_TRY(launch_slab_cores<float>(op, 0));
  VIE_TRY(launch_slab_cores<double>(op, 0));
  // FP32 scratch for the per-matvec rebuild of the half fibres (planned z edges):
  // whole k1 planes of [H2][6][H3], as many as fit in kOctBudget
  if (vie::plan_exists(op->P[2]) && octant_smem_bytes(op->rmax[1], op->rmax[2]) <= kOctantSmemMax) {
    constexpr size_t kOctBudget = 64u << 20;
    const size_t plane = (size_t)op->H[1] * 6 * op->H[2] * sizeof(float2);
    op->oct_k1 = (int)std::max<size_t>(1, std::min<size_t>(op->H[0], kOctBudget / plane));
    const int st = dalloc(&op->oct32, (size_t)op->oct_k1 * plane);
    if (st != VIE_OK && lane_fft_edge(op->P[2])) return st;
    if (st != VIE_OK) {                    // the z stage of other edges does without
      clear_error();
      op->oct32 = nullptr;
      op->oct_k1 = 0;
    }
  }
  if (op->oct32 != nullptr) {
    VIE_CUDA(cudaStreamCreateWithFlags(&op->rb_stream, cudaStreamNonBlocking));
    VIE_CUDA(cudaEventCreateWithFlags(&op->rb_fork, cudaEventDisableTiming));
    VIE_CUDA(cudaEventCreateWithFlags(&op->rb_join, cudaEventDisableTiming));
    if ((op->flags & VIE_REBUILD_TCGEN05) && !(op->flags & VIE_REBUILD_SIMT) && lane_fft_edge(op->P[2]) &&
        umma_rebuild_eligible(op)) {
      op->umma = true;
    } else if (tc_rebuild_eligible(op)) {
      tc_layout(op->rmax[2], op->H[2], &op->tc_ks, &op->tc_nsplit, &op->tc_ntc);
    }
    if (op->tc_ks > 0 && tc_rebuild_fits(op)) {
      VIE_TRY(dalloc(&op->u3frag, 6ull * op->tc_nsplit * op->tc_ks * op->tc_ntc * 32 * sizeof(uint4)));
      VIE_TRY(launch_u3_fragments(op, 0));
    }
  }
  VIE_CUDA(cudaDeviceSynchronize());
  return VIE_OK;
}

int op_tables(vie_op* op) { return init_tables(op); }

int build_operator(const vie_grid* grid, double tol, int rank_rule, int flags, cudaStream_t s,
                   vie_op** out) {
  vie_op* op = new (std::nothrow) vie_op();
  if (!op) {
    set_error("host allocation failed");
    return VIE_ERR_OOM;
  }
  op->grid = *grid;
  op->flags = flags;
  op->k0 = wavenumber(grid->freq_hz);
  const int nn[3] = {grid->n1, grid->n2, grid->n3};
  for (int q = 0; q < 3; ++q) {
    op->n[q] = nn[q];
    op->P[q] = 2 * nn[q];
    op->H[q] = nn[q] + 1;
  }
  int st = init_tables(op);
  if (st != VIE_OK) { vie_destroy(op); return st; }
  const long long full = (long long)op->P[0] * op->P[1] * op->P[2];
  if (flags & VIE_STORE_UNCOMPRESSED) {
    if ((st = dalloc(&op->spec64, 6 * full * sizeof(double2))) != VIE_OK ||
        (st = dalloc(&op->spec32, 6 * full * sizeof(float2))) != VIE_OK) {
      vie_destroy(op);
      return st;
    }
  }
  {
    DeviceBuffers d;
    const int hmax = std::max(op->H[0], std::max(op->H[1], op->H[2]));
    const bool factorwise = (flags & VIE_SETUP_FACTORWISE) != 0;
    // the P1 P2 P3 spectrum is formed only on the spectrum route or to be stored
    const bool need_full = !factorwise || (flags & VIE_STORE_UNCOMPRESSED);
    int H[3];
    octant_dims(op, factorwise, H);
    const size_t aw = (size_t)H[0] * H[1] * H[2];
    size_t mats = 0;                                   // Gram matrix, Y and V2 of every mode
    for (int q = 0; q < 3; ++q) {
      mats += 3 * (size_t)H[q] * H[q];
      d.part_entries = std::max(d.part_entries, (size_t)gram_ranges(H[q], aw / H[q]) * H[q] * H[q]);
    }
    const size_t tmp = std::max(aw, (size_t)hmax * hmax);
    const bool part_in_full = need_full && (size_t)full >= d.part_entries;
    const size_t fixed = (need_full ? (size_t)full : 0) + tmp + (size_t)hmax * hmax +
                         (part_in_full ? 0 : d.part_entries);
    if ((need_full && (st = dalloc(&d.full, full * sizeof(double2))) != VIE_OK) ||
        (st = dalloc(&d.tmp, tmp * sizeof(double2))) != VIE_OK ||
        (st = dalloc(&d.ytr, (size_t)hmax * hmax * sizeof(double2))) != VIE_OK ||
        (!part_in_full && (st = dalloc(&d.part_own, d.part_entries * sizeof(double2))) != VIE_OK) ||
        (st = dalloc(&d.jobs, 18 * sizeof(JacobiJob))) != VIE_OK ||
        (st = dalloc(&d.jstatus, 18 * (1 + kJacobiSweeps) * sizeof(int))) != VIE_OK ||
        (st = dalloc(&d.red, 12 * sizeof(unsigned long long))) != VIE_OK) {
      vie_destroy(op);
      return st;
    }
    d.part = part_in_full ? d.full : d.part_own;
    auto alloc_group = [&](int g) {
      d.comps = g;
      for (int i = 0; i < g; ++i) {
        VIE_TRY(dalloc(&d.aw[i], aw * sizeof(double2)));
        for (int q = 0; q < 3; ++q) {
          const size_t hh = (size_t)H[q] * H[q] * sizeof(double2);
          VIE_TRY(dalloc(&d.gram[i][q], hh));
          VIE_TRY(dalloc(&d.vec[i][q], hh));
          VIE_TRY(dalloc(&d.vec2[i][q], hh));
        }
      }
      return (int)VIE_OK;
    };
    st = alloc_group(setup_group((aw + mats) * sizeof(double2)));
    if (st == VIE_ERR_OOM && d.comps > 1) {            // one component at a time may still fit
      d.release_group();
      clear_error();
      st = alloc_group(1);
    }
    op->setup_scratch_bytes = (fixed + d.comps * (aw + mats)) * sizeof(double2);
    for (int c0 = 0; c0 < 6 && st == VIE_OK; c0 += d.comps) {
      st = component_eigenvectors(op, c0, d, s, factorwise);
      for (int i = 0; i < d.comps && st == VIE_OK; ++i)
        st = compress_component(op, c0 + i, i, tol, rank_rule, d, s, factorwise);
    }
    if (st == VIE_OK) {
      cudaError_t e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) st = cuda_status(e, "compress");
    }
  }
  if (st == VIE_OK) st = finish_operator(op);
  if (st != VIE_OK) {
    vie_destroy(op);
    return st;
  }
  *out = op;
  return VIE_OK;
}
