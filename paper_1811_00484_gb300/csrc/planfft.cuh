// Matvec stages for every padded edge N = 2n with a factor plan: x / y line
// stages (zero-padded forward, cropped inverse) and the fused z stage (forward
// transform, voxel-wise product, inverse transform), in FP32 (planfft64.cuh:
// FP64).  All lengths, strides in shared memory and radices are compile-time
// constants, so the only index arithmetic left is one multiply-add per access.
//
// What bounds them: the line stages the memory (96^3, 16 right-hand sides: x 192,
// y 371, inverse y 319 and inverse x 168 us, 5.3 to 6.4 TB/s of their bytes; 363,
// 701, 501 and 260 us with radices as uneven as 24 x 8), on small grids the latency of
// one load, exchange and store; the z stage shared-memory wavefronts (60 to 70 % of
// the peak) and issue (60 %) together (96^3, 16 right-hand sides: 983 us against
// 1421 us for a four-step transform of one component per warp).
//
// Line stage, N = Q1 Q2, thread (col, t): columns are adjacent in memory.
// With n = a + Q2 b, k = c + Q1 h,
//   X[c + Q1 h] = sum_a w_{Q2}^{a h} w_N^{a c} sum_b x[a + Q2 b] w_{Q1}^{b c}:
//   pass 1 (thread a): DFT of length Q1 over b, twiddle, X1[c][a][col] to shared
//   pass 2 (thread c): DFT of length Q2 over a, rows c + Q1 h to global memory.
// One shared-memory exchange and one barrier per line.  The padding (b >= Q1/2
// are zero; Q1 even forward) and the crop (only h < Q2/2 are kept; Q2 even
// inverse) are pruned out of the butterflies.
//
// Fused stage, N = R1 R2 R3 (R3 = 1: two passes), S threads per z-line, up to
// four mirror lines of one (k1, k2) group per CTA.  n = a + M1 b (M1 = R2 R3),
// a = e + R3 f, k = c + R1 g + R1 R2 h:
//   pass 1 (thread a):      DFT-R1 over b, twiddle w_N^{a c}
//   pass 2 (thread (c, e)): DFT-R2 over f, twiddle w_{R2 R3}^{e g}
//   pass 3 (thread (c, g)): DFT-R3 over e, frequencies c + R1 g + R1 R2 h
// Every pass reads and writes the same addresses in the same thread, so each of
// the three Cartesian components keeps one buffer and a barrier is needed only
// between passes (two per right-hand side with two passes, four with three).
// The thread ends with the three components of its frequencies in registers,
// forms Y = D G D J there (mirror signs folded into G's off-diagonal entries)
// and runs the passes backwards in place.
//
// The half fibre G[6][N/2+1] of the group is copied from the FP32 rebuild
// scratch, read from the stored spectra (only the octant k <= P/2: the rest is
// its mirror image, an eighth of the bytes), or rebuilt by the CTA (ranks beyond
// the rebuild kernels').
#pragma once

#include "regdft.cuh"
#include "stages.cuh"

namespace vie {
namespace plan {

// one set of plan_table.h (plan_set.cuh); false when the edge is not in it
template <typename T, int K> bool line_set(const LineArgs<T>& a, cudaStream_t s);
template <typename T, int K> bool fused_set(const FusedArgs<T>& a, int k10, int nk1, cudaStream_t s);
template <typename T, int K> cudaError_t prepare_set(int N);

__host__ __device__ constexpr int imax(int a, int b) { return a > b ? a : b; }
__host__ __device__ constexpr int imin(int a, int b) { return a < b ? a : b; }

// ---------------------------------------------------------------------------
// line stage
// ---------------------------------------------------------------------------
// Threads per column: the smaller radix when it divides the larger (every thread
// then has the same work in both passes; with 16 threads for 16 x 8 half of them
// waited at the barrier through pass 1), else the larger.  An inverse stage waits
// for its loads, twice the forward one's: one thread per first-pass butterfly up
// to radix 16 (N = 128, 8 right-hand sides: 58 us with 8 threads, 52 us with 16; N
// = 512, 32 x 16: 921 us with 16 threads, 1096 us with 32).
__host__ __device__ constexpr int line_slots(int Q1, int Q2, bool inv) {
  const int big = imax(Q1, Q2), small = imin(Q1, Q2);
  return inv && Q2 >= Q1 && Q2 <= 16 ? Q2 : (big % small == 0 ? small : big);
}
// columns per CTA: 128 bytes of a row, fewer when a line needs more than 16 threads
__host__ __device__ constexpr int line_cols(int S) { return S <= 16 ? 16 : 8; }
// registers a thread may use: the larger radix's values, its DFT's temporaries
// and the addresses.  Radices 12 to 16 with 12 to 16 threads per line run at 64
// (four CTAs of 256 threads; 192 x 96 x 96 lines, 16 right-hand sides: 395 us at
// 80 registers, 373 us at 64); with 8 threads doing two butterflies they spill there.
__host__ __device__ constexpr int line_regs(int R, int S) {
  return R <= 8 ? 48 : R <= 10 ? 56 : R <= 16 ? (S >= 12 ? 64 : 80) : R <= 21 ? 96 : 128;
}
__host__ __device__ constexpr int line_blocks(int Q1, int Q2, bool inv) {
  const int S = line_slots(Q1, Q2, inv), th = line_cols(S) * S;
  const int b = 65536 / (line_regs(imax(Q1, Q2), S) * ((th + 31) / 32 * 32));
  return b < 1 ? 1 : (b > 24 ? 24 : b);
}

template <int Q1, int Q2, bool INV>
__global__ void __launch_bounds__(line_cols(line_slots(Q1, Q2, INV)) * line_slots(Q1, Q2, INV), line_blocks(Q1, Q2, INV))
    plan_line_kernel(const LineArgs<float> a) {
  using C = float2;
  constexpr int S = line_slots(Q1, Q2, INV);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* X = reinterpret_cast<C*>(smem_raw);               // [Q1][Q2][CW]
  const int CW = blockDim.x, col = threadIdx.x, t0 = threadIdx.y;
  const int c0 = blockIdx.x * CW + col, o = blockIdx.y, bb = blockIdx.z;
  if (a.early) pdl_trigger();
  pdl_wait();
  if (a.active != nullptr && a.active[bb / a.batch_per_rhs] == 0) return;   // block-uniform
  if (a.prof != nullptr && blockIdx.x == 0 && o == 0 && col == 0 && t0 == 0)
    atomicAdd(a.prof, a.prof_batch_bytes);
  const bool col_ok = c0 < a.ncol;
  const float rs = (a.flags & (PRO_RSCALE | EPI_RSCALE))
                   ? (float)a.rscale[(long long)(bb / a.batch_per_rhs) * a.rscale_stride]
                   : 1.f;
  // offsets inside one batch entry fit 32 bits (checked at launch)
  const unsigned ils = (unsigned)a.in_ls, ols = (unsigned)a.out_ls, hls = (unsigned)a.chi_ls;
  const unsigned hoff = (unsigned)(o * a.chi_os) + (unsigned)c0;
  {
    const C* in = a.in + bb * a.in_bs;
    const unsigned ioff = (unsigned)(o * a.in_os) + (unsigned)c0;
#pragma unroll
    for (int i = 0; i < (Q2 + S - 1) / S; ++i) {
      const int t = t0 + i * S;
      if (Q2 % S != 0 && t >= Q2) break;
      C v[Q1];
      if constexpr (!INV) {
        C x[Q1 / 2];
#pragma unroll
        for (int m = 0; m < Q1 / 2; ++m) x[m] = col_ok ? in[ioff + (t + Q2 * m) * ils] : czero<C>();
        if (a.flags & (PRO_RSCALE | PRO_CONJ | PRO_CHI)) {
#pragma unroll
          for (int m = 0; m < Q1 / 2; ++m) {
            if (a.flags & PRO_RSCALE) x[m] = rs * x[m];
            if (a.flags & PRO_CONJ) x[m] = conjg(x[m]);
            if ((a.flags & PRO_CHI) && col_ok) x[m] = a.chi[hoff + (t + Q2 * m) * hls] * x[m];
          }
        }
        dft_half_in<Q1, false>(x, v);
      } else {
#pragma unroll
        for (int m = 0; m < Q1; ++m) v[m] = col_ok ? in[ioff + (t + Q2 * m) * ils] : czero<C>();
        dft_reg<Q1, true>(v);
      }
#pragma unroll
      for (int c = 1; c < Q1; ++c) {
        const C w = __ldg(a.roots + t * c);
        v[c] = v[c] * (INV ? conjg(w) : w);
      }
#pragma unroll
      for (int c = 0; c < Q1; ++c) X[(c * Q2 + t) * CW + col] = v[c];
    }
  }
  __syncthreads();
  if (!col_ok) return;
  C* out = a.out + bb * a.out_bs;
  const unsigned ooff = (unsigned)(o * a.out_os) + (unsigned)c0;
#pragma unroll
  for (int i = 0; i < (Q1 + S - 1) / S; ++i) {
    const int t = t0 + i * S;
    if (Q1 % S != 0 && t >= Q1) break;
    C u[Q2];
#pragma unroll
    for (int f = 0; f < Q2; ++f) u[f] = X[(t * Q2 + f) * CW + col];
    if constexpr (!INV) {
      dft_reg<Q2, false>(u);
#pragma unroll
      for (int h = 0; h < Q2; ++h) out[ooff + (t + Q1 * h) * ols] = u[h];
    } else {
      C y[Q2 / 2];
      dft_half_out<Q2, true>(u, y);
#pragma unroll
      for (int h = 0; h < Q2 / 2; ++h) y[h] = a.scale * y[h];
      if (a.flags & (EPI_CONJ | EPI_SUB | EPI_ADD)) {
        const C* add = a.addend + bb * a.out_bs;
#pragma unroll
        for (int h = 0; h < Q2 / 2; ++h) {
          C x = y[h];
          if (a.flags & EPI_CONJ) x = conjg(x);
          if (a.flags & (EPI_SUB | EPI_ADD)) {
            if (a.flags & EPI_CHI) x = a.chi[hoff + (t + Q1 * h) * hls] * x;
            C w = add[ooff + (t + Q1 * h) * ols];
            if (a.flags & EPI_RSCALE) w = rs * w;
            x = (a.flags & EPI_SUB) ? (w - x) : (w + x);
          }
          y[h] = x;
        }
      }
#pragma unroll
      for (int h = 0; h < Q2 / 2; ++h) out[ooff + (t + Q1 * h) * ols] = y[h];
    }
  }
}

// kernel of the pass order Q1, Q2 (forward: Q1 even; inverse: Q2 even)
template <int Q1, int Q2, bool INV> void launch_plan_line_order(LineArgs<float> a, cudaStream_t s) {
  constexpr int S = line_slots(Q1, Q2, INV), CMAX = line_cols(S);
  // lines whose columns are adjacent across `o` too (the x stages) form one run
  if (a.in_os == a.ncol && a.out_os == a.ncol && (a.chi == nullptr || a.chi_os == a.ncol) &&
      (long long)a.ncol * a.nother < (1LL << 30)) {
    a.ncol *= a.nother;
    a.nother = 1;
  }
  // equal column groups: 50 columns are 4 groups of 13, not 3 of 16 and one of 2
  // (vie_autotune may have chosen smaller CTAs than the default)
  const int cmax = a.threads > 0 ? imin(CMAX, imax(4, a.threads / S)) : CMAX;
  const int tiles = (a.ncol + cmax - 1) / cmax;
  const int cw = (a.ncol + tiles - 1) / tiles;
  a.prof = prof_bytes(a.prof_family);
  ProfScope ps(a.prof_family, s);
  const dim3 grid((unsigned)tiles, (unsigned)a.nother, (unsigned)a.nbatch), block((unsigned)cw, S);
  launch_pdl(plan_line_kernel<Q1, Q2, INV>, grid, block, (size_t)Q1 * Q2 * cw * sizeof(float2), s, a);
}

// Q1 is even: forward Q1 x Q2, inverse Q2 x Q1 (the even radix where the half is)
template <int Q1, int Q2> void launch_plan_line(const LineArgs<float>& a, cudaStream_t s) {
  static_assert(Q1 % 2 == 0, "the pruned radix is even");
  if (a.inverse) launch_plan_line_order<Q2, Q1, true>(a, s);
  else launch_plan_line_order<Q1, Q2, false>(a, s);
}

template <int Q1, int Q2> cudaError_t prepare_plan_line(float) {
  constexpr size_t smem = (size_t)Q1 * Q2 * 16 * sizeof(float2);       // at most 16 columns
  if constexpr (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(plan_line_kernel<Q1, Q2, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(plan_line_kernel<Q2, Q1, true>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// fused z stage
// ---------------------------------------------------------------------------
// Threads per line: one per slot of the widest pass, or, where that makes a group
// one warp (eight butterflies a line, radix 12 and up) or the first radix is so
// large that registers limit the threads anyway, only the M1 butterflies of the
// first pass, later passes looping over their slots (N = 128 with 8 right-hand
// sides: 16 threads 171 us, 8 threads 165 us; N = 112: 37 and 30 us; N = 216: 357
// and 295 us; but N = 160: 97 and 122 us, N = 80: 8.4 and 11.5 us).
__host__ __device__ constexpr int fused_slots(int R1, int R2, int R3) {
  const int M1 = R2 * R3, wide = imax(imax(M1, R1 * R3), R3 > 1 ? R1 * R2 : R1);
  return R3 == 1 && ((M1 == 8 && R1 >= 12) || R1 >= 18) ? M1 : wide;
}

template <int R1, int R2, int R3> struct FusedPlan {
  static constexpr int N = R1 * R2 * R3, M1 = R2 * R3, H3 = N / 2 + 1;
  static constexpr int HL = R3 > 1 ? R3 : R2;               // frequencies per slot of the last pass
  static constexpr int TL = R3 > 1 ? R1 * R2 : R1;          // slots of the last pass
  static constexpr int S = fused_slots(R1, R2, R3);         // threads per line
  static constexpr int PR = R3 > 1 ? (R3 | 1) : 1;          // padded run of e
  static constexpr int LD = (R3 > 1 ? R2 * PR : R2) | 1;    // row c of a line's buffer (odd)
  static constexpr int LS = R1 * LD;                        // one line of one component
  // lines S (mod 16) entries apart: consecutive threads of neighbouring lines
  // fall in different 8-byte banks, in the rows of pass 1 and (LD odd) the
  // columns of pass 2
  static constexpr int LSTR = 3 * LS + ((S - 3 * LS) % 16 + 16) % 16;
  static constexpr int NL = (R1 + 1) / 2;                   // inputs that can be nonzero
  // small groups share a CTA (and its twiddle tables)
  static constexpr int GP = 4 * S >= 64 ? 1 : (64 + 4 * S - 1) / (4 * S);
  static constexpr int threads = 4 * S * GP;
  static constexpr int GH = 6 * H3 + (6 * H3 & 1);          // half fibres, 16-byte multiple
  static constexpr int T1 = R1 * M1, T2 = R3 > 1 ? R2 * R3 : 0;   // twiddles [c][a], [g][e]
  static constexpr int XS = 4 * LSTR;
  static constexpr int fixed = GP * (GH + XS) + T1 + T2;    // shared entries
  static __host__ __device__ constexpr int inner(int a) {   // X1 column of a = e + R3 f
    return R3 > 1 ? (a / R3) * PR + a % R3 : a;
  }
};
template <int R1, int R2, int R3> __host__ __device__ constexpr int fused_blocks() {
  using P = FusedPlan<R1, R2, R3>;
  // live at the peak: three components of HL frequencies and a half fibre
  // entry, or two components' inputs, one transform and its temporaries
  const int live = imax(6 * P::HL + 60, 4 * P::NL + 3 * R1 + 36);
  const int regs = live < 64 ? 64 : live > 168 ? 168 : live;
  const int wt = (P::threads + 31) / 32 * 32;
  const int by_regs = 65536 / (((regs + 7) / 8 * 8) * wt);
  const int by_smem = (int)((size_t)227 * 1024 / (P::fixed * sizeof(float2) + 1024));
  const int b = by_regs < by_smem ? by_regs : by_smem;
  return b < 1 ? 1 : (b > 16 ? 16 : b);
}

template <int R1, int R2, int R3>
__global__ void __launch_bounds__(FusedPlan<R1, R2, R3>::threads, fused_blocks<R1, R2, R3>())
    plan_fused_kernel(const FusedArgs<float> a, int k10) {
  using C = float2;
  using P = FusedPlan<R1, R2, R3>;
  constexpr int N = P::N, S = P::S, H3 = P::H3, HL = P::HL, LD = P::LD, NL = P::NL, M1 = P::M1;
  constexpr bool kEven = R1 % 2 == 0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sm = reinterpret_cast<C*>(smem_raw);
  const int gp = threadIdx.x / (4 * S), lt = threadIdx.x % (4 * S);
  const int l = lt / S, t = lt % S;
  C* G = sm + gp * P::GH;                                          // [6][H3]
  C* X = sm + P::GP * P::GH + gp * P::XS + l * P::LSTR;            // [3][R1][LD]
  C* tw1 = sm + P::GP * (P::GH + P::XS);                           // w_N^{a c} at [c][a]
  C* tw2 = tw1 + P::T1;                                            // w_{R2 R3}^{e g} at [g][e]
  const int k1 = k10 + blockIdx.y, k2 = blockIdx.x * P::GP + gp;
  const bool group = k2 < a.H2;
  const int nx = (k1 == 0 || 2 * k1 == a.P1) ? 1 : 2;
  const int ny = (k2 == 0 || 2 * k2 == a.P2) ? 1 : 2;
  const bool valid = group && l < nx * ny;
  const int ix = valid ? l / ny : 0, iy = valid ? l % ny : 0;
  const int kx = ix ? a.P1 - k1 : k1, ky = iy ? a.P2 - k2 : k2;
  C* line0 = a.data + ((long long)kx * a.P2 + ky) * (N / 2) + t;
  // lines exchange nothing with one another: a line inside one warp, or of whole
  // warps, needs no barrier of the CTA
  auto sync = [&]() {
    if constexpr (32 % S == 0) {
      __syncwarp();
    } else if constexpr (S % 32 == 0) {
      asm volatile("bar.sync %0, %1;" ::"r"(1 + gp * 4 + l), "n"(S) : "memory");
    } else {
      __syncthreads();
    }
  };
  // no rebuilt half fibres to copy (ranks beyond the rebuild kernels'):
  // eq. (13) for this group here, W_c = U2_c[k2, :] S_c[k1], G_c[k3] = W_c . U3_c[k3, :]
  const bool here = a.spec == nullptr && a.octant == nullptr;
  if (here) {
    C* W = sm + P::fixed + gp * 6 * a.r3max;
    if (group) {
      for (int it = lt; it < 6 * a.r3max; it += 4 * S) {
        const int c = it / a.r3max, q = it - c * a.r3max;
        const CompMeta<float>& m = a.meta[c];
        C acc = czero<C>();
        if (q < m.r3) {
          const C* sl = m.slab + (long long)k1 * a.r2max * a.r3max + q;
          const C* u2 = m.U2 + (long long)k2 * m.r2;
          for (int b = 0; b < m.r2; ++b) acc = cmadd(u2[b], sl[b * a.r3max], acc);
        }
        W[it] = acc;
      }
    }
    __syncthreads();
    if (group) {
      for (int it = lt; it < 6 * H3; it += 4 * S) {
        const int c = it / H3, kk = it - c * H3;
        const int r3 = a.meta[c].r3;
        const C* u3 = a.meta[c].U3 + (long long)kk * r3;
        C acc = czero<C>();
        for (int q = 0; q < r3; ++q) acc = cmadd(W[c * a.r3max + q], u3[q], acc);
        G[it] = acc;
      }
    }
  }
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && blockIdx.x == 0 && k1 == 0 && threadIdx.x == 0) {
    unsigned long long nb = 0;
    for (int b = 0; b < a.B; ++b) nb += (a.active == nullptr || a.active[b]) ? 1 : 0;
    atomicAdd(a.prof, nb * a.prof_rhs_bytes + a.prof_launch_bytes);
  }
  auto next_active = [&](int b) {
    if (a.active != nullptr)
      while (b < a.B && a.active[b] == 0) ++b;
    return b;
  };
  // the three components' inputs in flight together
  C x[3][NL];
  auto load = [&](int b) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const C* src = line0 + (long long)(b * 3 + q) * a.comp_stride;
#pragma unroll
      for (int m = 0; m < NL; ++m)
        x[q][m] = (valid && (S == M1 || t < M1) && (kEven || t + M1 * m < N / 2)) ? src[M1 * m] : czero<C>();
    }
  };
  int b = next_active(0);
  if (b < a.B) load(b);
  // tables and half fibres while those are under way
  for (int i = threadIdx.x; i < P::T1; i += P::threads) tw1[i] = a.roots[(i / M1) * (i % M1)];
  if constexpr (R3 > 1)
    for (int i = threadIdx.x; i < P::T2; i += P::threads) tw2[i] = a.roots[R1 * (i / R3) * (i % R3)];
  if (group) {
    if (a.spec != nullptr) {
      const C* src = a.spec + ((long long)k1 * a.P2 + k2) * N;
      for (int it = lt; it < 6 * H3; it += 4 * S) {
        const int c = it / H3, kk = it - c * H3;
        G[it] = src[c * a.spec_stride + kk];
      }
    } else if (!here) {
      const float4* src = reinterpret_cast<const float4*>(
          a.octant + ((long long)(k1 - a.oct_k1a) * a.H2 + k2) * 6 * H3);
      float4* dst = reinterpret_cast<float4*>(G);
      for (int it = lt; it < 3 * H3; it += 4 * S) dst[it] = src[it];
    }
  }
  const float sx = ix ? -1.f : 1.f, sy = iy ? -1.f : 1.f;
  __syncthreads();                                     // tables and half fibres
  for (bool first = true; b < a.B; b = next_active(b + 1), first = false) {   // block-uniform
    if (!first) load(b);
    if (S == M1 || t < M1) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        C v[R1];
        if constexpr (kEven) {
          dft_half_in<R1, false>(x[q], v);
        } else {
#pragma unroll
          for (int m = 0; m < R1; ++m) v[m] = m < NL ? x[q][m < NL ? m : 0] : czero<C>();
          dft_reg<R1, false>(v);
        }
        C* row = X + q * P::LS + P::inner(t);
        row[0] = v[0];
#pragma unroll
        for (int c = 1; c < R1; ++c) row[c * LD] = v[c] * tw1[c * M1 + t];
      }
    }
    sync();
    if constexpr (R3 > 1) {
#pragma unroll 1
      for (int sl = t; sl < R1 * R3; sl += S) {          // slot (c, e)
        C* p = X + (sl % R1) * LD + sl / R1;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          C u[R2];
#pragma unroll
          for (int f = 0; f < R2; ++f) u[f] = p[q * P::LS + f * P::PR];
          dft_reg<R2, false>(u);
          p[q * P::LS] = u[0];
#pragma unroll
          for (int g = 1; g < R2; ++g) p[q * P::LS + g * P::PR] = u[g] * tw2[g * R3 + sl / R1];
        }
      }
      sync();
    }
#pragma unroll 1
    for (int sl = t; sl < P::TL; sl += S) {              // slot (c, g)
      C s[3][HL];
      C* own = X + (sl % R1) * LD + (R3 > 1 ? (sl / R1) * P::PR : 0);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
#pragma unroll
        for (int e = 0; e < HL; ++e) s[q][e] = own[q * P::LS + e];
        dft_reg<HL, false>(s[q]);
      }
      // Y = D G D J at f = sl + TL h
#pragma unroll
      for (int h = 0; h < HL; ++h) {
        const int f = sl + P::TL * h;
        const bool zm = 2 * f > N;
        const C* gf = G + (zm ? N - f : f);
        const float sz = zm ? -1.f : 1.f;
        const C gxx = gf[0], gyy = gf[3 * H3], gzz = gf[5 * H3];
        const C gxy = (sx * sy) * gf[H3], gxz = (sx * sz) * gf[2 * H3], gyz = (sy * sz) * gf[4 * H3];
        const C jx = s[0][h], jy = s[1][h], jz = s[2][h];
        s[0][h] = cmadd(gxx, jx, cmadd(gxy, jy, gxz * jz));
        s[1][h] = cmadd(gxy, jx, cmadd(gyy, jy, gyz * jz));
        s[2][h] = cmadd(gxz, jx, cmadd(gyz, jy, gzz * jz));
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        dft_reg<HL, true>(s[q]);
#pragma unroll
        for (int e = 0; e < HL; ++e) own[q * P::LS + e] = s[q][e];
      }
    }
    sync();
    if constexpr (R3 > 1) {
#pragma unroll 1
      for (int sl = t; sl < R1 * R3; sl += S) {
        C* p = X + (sl % R1) * LD + sl / R1;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          C u[R2];
          u[0] = p[q * P::LS];
#pragma unroll
          for (int g = 1; g < R2; ++g) u[g] = p[q * P::LS + g * P::PR] * conjg(tw2[g * R3 + sl / R1]);
          dft_reg<R2, true>(u);
#pragma unroll
          for (int f = 0; f < R2; ++f) p[q * P::LS + f * P::PR] = u[f];
        }
      }
      sync();
    }
    if (S == M1 || t < M1) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        C v[R1];
        const C* row = X + q * P::LS + P::inner(t);
        v[0] = row[0];
#pragma unroll
        for (int c = 1; c < R1; ++c) v[c] = row[c * LD] * conjg(tw1[c * M1 + t]);
        C* dst = line0 + (long long)(b * 3 + q) * a.comp_stride;
        if constexpr (kEven) {
          C y[R1 / 2];
          dft_half_out<R1, true>(v, y);
          if (valid) {
#pragma unroll
            for (int m = 0; m < R1 / 2; ++m) dst[M1 * m] = y[m];
          }
        } else {
          dft_reg<R1, true>(v);
          if (valid) {
#pragma unroll
            for (int m = 0; m < NL; ++m)
              if (t + M1 * m < N / 2) dst[M1 * m] = v[m];
          }
        }
      }
    }
  }
}

template <int R1, int R2, int R3>
constexpr size_t fused_smem_fixed() {
  return (size_t)FusedPlan<R1, R2, R3>::fixed * sizeof(float2);
}

// groups k1 in [k10, k10 + nk1), every k2
template <int R1, int R2, int R3>
void launch_plan_fused(const FusedArgs<float>& a, int k10, int nk1, cudaStream_t s) {
  using P = FusedPlan<R1, R2, R3>;
  size_t smem = fused_smem_fixed<R1, R2, R3>();
  if (a.spec == nullptr && a.octant == nullptr) smem += (size_t)P::GP * 6 * a.r3max * sizeof(float2);
  launch_pdl(plan_fused_kernel<R1, R2, R3>, dim3((unsigned)((a.H2 + P::GP - 1) / P::GP), (unsigned)nk1),
             dim3(P::threads), smem, s, a, k10);
}

constexpr size_t kFusedSmemMax = 200 * 1024;

template <int R1, int R2, int R3> cudaError_t prepare_plan_fused(float) {
  return cudaFuncSetAttribute(plan_fused_kernel<R1, R2, R3>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmemMax);
}

}  // namespace plan
}  // namespace vie
