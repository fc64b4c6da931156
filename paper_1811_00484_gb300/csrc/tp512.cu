// Length-512 transforms of the matvec (Section V.B) for 256-voxel grid edges
// (P = 512): the fused z stage (zero-padded forward z-FFT, voxel-wise product
// with the rebuilt or stored spectra, cropped inverse z-FFT) and the FP64 x and y
// line stages.  The FP32 line stages are the planned 32 x 16 kernels: with eight
// 256^3 right-hand sides x 2.0, y 3.9, inverse y 3.5 and inverse x 2.6 ms with its
// epilogue, against 2.4, 4.2, 3.9 and 4.1 ms for persistent three-pass kernels
// fed by TMA tiles, which one exchange and one barrier per line beat.
//
// Three radix-8 passes, 64 threads per line, 8 values per thread.  With
// n = a + 64 b (a < 64, b < 8), a = e + 8 f and k = c + 8 g + 64 h,
//   X[c + 8g + 64h] = sum_e w8^{eh} w64^{eg} sum_f w8^{fg} w512^{ac}
//                     sum_b w8^{bc} x[a + 64 b],
// so
//   pass 1 (thread a):      DFT-8 over b, twiddle w512^{a c}, store X1[c][a]
//   pass 2 (thread (c, e)): DFT-8 over f (a = e + 8f), twiddle w64^{e g},
//                           store X2[c][g][e]
//   pass 3 (thread (c, g)): DFT-8 over e, giving X[c + 8g + 64h] in register h.
// The inverse runs the three passes backwards (inverse DFT-8s, conjugate
// twiddles), from the register layout where the forward one ends to the
// layout where it starts, so a forward / product / inverse sequence never
// reorders data.  Zero padding (x[n] = 0 for n >= 256: b >= 4) and cropping
// (outputs n < 256) prune the first and last passes.
//
// Exchange layouts (float2 units): X1[c][a] at c LA + a, X2[c][g][e] at
// c 72 + 9 g + e.  Each half-warp's 64-bit accesses of every pass fall in 16
// different bank pairs (checked for both thread layouts below).
#include <algorithm>

#include "stages.cuh"
#include "mbar.cuh"

namespace vie {

namespace tp {

constexpr int kN = 512;
constexpr int kM = 64;            // threads per line
constexpr int kX2 = 576;          // 8 x 72 per line

template <typename C>
__device__ __forceinline__ C root(const C* roots, int e, bool inv) {
  const C w = __ldg(roots + e);
  return inv ? conjg(w) : w;
}

template <typename C> struct RealOf;
template <> struct RealOf<float2> { using type = float; };
template <> struct RealOf<double2> { using type = double; };

// DFT-8 of x[0..3] with x[4..7] = 0: X[2k] = DFT4(x)[k], X[2k+1] = DFT4(x_n w8^n)[k]
template <typename C>
__device__ __forceinline__ void dft8_half_in(C* v, bool inv) {
  using T = typename RealOf<C>::type;
  const T r = (T)0.70710678118654752440;
  C e0 = v[0], e1 = v[1], e2 = v[2], e3 = v[3];
  C o0 = v[0], o1, o2, o3;
  if (!inv) {
    o1 = mk(r * (v[1].x + v[1].y), r * (v[1].y - v[1].x));
    o2 = mul_mi(v[2]);
    o3 = mk(r * (v[3].y - v[3].x), -r * (v[3].x + v[3].y));
  } else {
    o1 = mk(r * (v[1].x - v[1].y), r * (v[1].x + v[1].y));
    o2 = mul_i(v[2]);
    o3 = mk(-r * (v[3].x + v[3].y), r * (v[3].x - v[3].y));
  }
  dft4(e0, e1, e2, e3, inv);
  dft4(o0, o1, o2, o3, inv);
  v[0] = e0; v[2] = e1; v[4] = e2; v[6] = e3;
  v[1] = o0; v[3] = o1; v[5] = o2; v[7] = o3;
}

// pass 1 in thread a: v[b] = x[a + 64 b]  ->  X1[c][a]
template <bool INV, bool HALF_IN, typename C>
__device__ __forceinline__ void pass1(C (&v)[8], int a, const C* roots, C* x1, int la) {
  if (HALF_IN) dft8_half_in(v, INV); else dft8<C, typename RealOf<C>::type>(v, INV);
#pragma unroll
  for (int c = 1; c < 8; ++c) v[c] = v[c] * root(roots, a * c, INV);
#pragma unroll
  for (int c = 0; c < 8; ++c) x1[c * la + a] = v[c];
}

// pass 3 in thread (c, g): X2[c][g][e]  ->  w[h] = X[c + 8 g + 64 h]
template <bool INV, typename C>
__device__ __forceinline__ void pass3(int c, int g, const C* x2, C (&w)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) w[e] = x2[c * 72 + 9 * g + e];
  dft8<C, typename RealOf<C>::type>(w, INV);
}

// inverse of pass 1 in thread a: X1[c][a]  ->  v[b] = 512 x[a + 64 b]
__device__ __forceinline__ void ipass1(int a, const float2* x1, int la, float2 (&v)[8]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = x1[c * la + a];
  dft8<float2, float>(v, true);
}

// Per-slot twiddle table in shared memory, [22][64] (row j, slot t):
//   rows 0..6   w512^{t c},             c = 1..7        (pass 1)
//   rows 7..13  w64^{(t mod 8) x},      x = 1..7        (pass 2, inverse pass 3)
//   rows 14..21 w512^{(t mod 8 + 8 f) (t div 8)}, f = 0..7   (inverse pass 2)
// The same for every line, tile and right-hand side a thread handles.
constexpr int kTwRows = 22;
__device__ __forceinline__ void fill_twiddles(float2* tw, const float2* roots, int tid, int nth) {
  for (int i = tid; i < kTwRows * kM; i += nth) {
    const int j = i / kM, t = i % kM;
    int e;
    if (j < 7) e = t * (j + 1);
    else if (j < 14) e = 8 * (t & 7) * (j - 6);
    else e = ((t & 7) + 8 * (j - 14)) * (t >> 3);
    tw[i] = roots[e];
  }
}
__device__ __forceinline__ float2 twv(const float2* tw, int row, int t, bool inv) {
  const float2 w = tw[row * kM + t];
  return inv ? conjg(w) : w;
}

template <bool INV, bool HALF_IN>
__device__ __forceinline__ void pass1t(float2 (&v)[8], int a, const float2* tw, float2* x1, int la) {
  if (HALF_IN) dft8_half_in(v, INV); else dft8<float2, float>(v, INV);
#pragma unroll
  for (int c = 1; c < 8; ++c) v[c] = v[c] * twv(tw, c - 1, a, INV);
#pragma unroll
  for (int c = 0; c < 8; ++c) x1[c * la + a] = v[c];
}

// pass 2 up to its twiddles (the caller stores u[g] at X2[c][g][e]); slot t = 8 c + e
template <bool INV>
__device__ __forceinline__ void pass2t_load(float2 (&u)[8], int t, const float2* x1, int la,
                                            const float2* tw) {
  const int c = t >> 3, e = t & 7;
#pragma unroll
  for (int f = 0; f < 8; ++f) u[f] = x1[c * la + e + 8 * f];
  dft8<float2, float>(u, INV);
#pragma unroll
  for (int g = 1; g < 8; ++g) u[g] = u[g] * twv(tw, 6 + g, t, INV);
}

// inverse of pass 3 in slot t = 8 c + g
__device__ __forceinline__ void ipass3t(int t, float2 (&w)[8], float2* x2, const float2* tw) {
  const int c = t >> 3, g = t & 7;
  dft8<float2, float>(w, true);
#pragma unroll
  for (int e = 1; e < 8; ++e) w[e] = w[e] * twv(tw, 6 + e, t, true);
#pragma unroll
  for (int e = 0; e < 8; ++e) x2[c * 72 + 9 * g + e] = w[e];
}

// inverse of pass 2 in slot t = 8 c + e
__device__ __forceinline__ void ipass2t(int t, const float2* x2, float2* x1, int la, const float2* tw) {
  const int c = t >> 3, e = t & 7;
  float2 u[8];
#pragma unroll
  for (int g = 0; g < 8; ++g) u[g] = x2[c * 72 + 9 * g + e];
  dft8<float2, float>(u, true);
#pragma unroll
  for (int f = 0; f < 8; ++f) x1[c * la + e + 8 * f] = u[f] * twv(tw, 14 + f, t, true);
}

// ---------------------------------------------------------------------------
// FP64 line stage (the refinement residuals): 4 adjacent columns per CTA, 64
// threads per column (col = tid & 3, slot t = tid >> 2; a warp's global
// accesses are 8 rows x 64 contiguous bytes), one exchange buffer per column
// used as X1 and then X2, twiddles read from the root table.  Bound by FP64
// arithmetic.
// ---------------------------------------------------------------------------
constexpr int kCols64 = 4;
constexpr int kX64 = 580;
constexpr size_t kLine64Smem = (size_t)kCols64 * kX64 * sizeof(double2);

template <bool INV, bool HALF>
__global__ void __launch_bounds__(256, 3) line_tp64_kernel(const LineArgs<double> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, col = tid & 3, t = tid >> 2;
  double2* x = reinterpret_cast<double2*>(smem_raw) + col * kX64;
  const int c0 = blockIdx.x * kCols64, o = blockIdx.y, bb = blockIdx.z;
  if (a.early) pdl_trigger();
  pdl_wait();
  if (a.active != nullptr && a.active[bb / a.batch_per_rhs] == 0) return;   // block-uniform
  const bool col_ok = c0 + col < a.ncol;
  const double rs = (a.flags & (PRO_RSCALE | EPI_RSCALE))
                        ? a.rscale[(long long)(bb / a.batch_per_rhs) * a.rscale_stride]
                        : 1.0;
  const double2* in = a.in + bb * a.in_bs + o * a.in_os + (long long)(c0 + col);
  double2 v[8];
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const int p = t + kM * b;
    double2 xv = make_double2(0.0, 0.0);
    if ((INV || !HALF || b < 4) && col_ok && p < a.lin) {
      xv = in[(long long)p * a.in_ls];
      if (!INV) {
        if (a.flags & PRO_RSCALE) xv = rs * xv;
        if (a.flags & PRO_CONJ) xv = conjg(xv);
        if (a.flags & PRO_CHI) xv = a.chi[o * a.chi_os + (long long)p * a.chi_ls + (long long)(c0 + col)] * xv;
      }
    }
    v[b] = xv;
  }
  pass1<INV, !INV && HALF>(v, t, a.roots, x, 64);
  __syncthreads();
  const int c = t >> 3, g = t & 7;
  {
    double2 u[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) u[f] = x[c * 64 + g + 8 * f];
    dft8<double2, double>(u, INV);
#pragma unroll
    for (int q = 1; q < 8; ++q) u[q] = u[q] * root(a.roots, 8 * g * q, INV);
    __syncthreads();                       // X1 read: X2 overwrites the same buffer
#pragma unroll
    for (int q = 0; q < 8; ++q) x[c * 72 + 9 * q + g] = u[q];
  }
  __syncthreads();
  pass3<INV>(c, g, x, v);
  if (!col_ok) return;
  double2* out = a.out + bb * a.out_bs + o * a.out_os + (long long)(c0 + col);
#pragma unroll
  for (int h = 0; h < 8; ++h) {
    if (INV && HALF && h >= 4) continue;
    const int p = c + 8 * g + kM * h;
    if (p >= a.lout) continue;
    double2 xv = v[h];
    if (INV) {
      xv = a.scale * xv;
      if (a.flags & EPI_CONJ) xv = conjg(xv);
      if (a.flags & (EPI_SUB | EPI_ADD)) {
        if (a.flags & EPI_CHI) xv = a.chi[o * a.chi_os + (long long)p * a.chi_ls + (long long)(c0 + col)] * xv;
        double2 w = a.addend[bb * a.out_bs + o * a.out_os + (long long)(c0 + col) + (long long)p * a.out_ls];
        if (a.flags & EPI_RSCALE) w = rs * w;
        xv = (a.flags & EPI_SUB) ? (w - xv) : (w + xv);
      }
    }
    out[(long long)p * a.out_ls] = xv;
  }
}

// ---------------------------------------------------------------------------
// Fused z stage: one CTA of 256 threads per (k1, k2) mirror group, 64 threads
// per mirror line (thread tid: line l = tid >> 6, slot t = tid & 63).  Each
// thread carries the three Cartesian components of its line through the
// forward passes (one after another, sharing the line's exchange buffers),
// holds their spectra at the eight frequencies c + 8g + 64h in registers,
// forms Y = D G D J there (G the rebuilt or stored half fibre with mirror signs
// D), and runs the inverse passes.  The line's 256 outputs
// overwrite its 256 inputs.
// ---------------------------------------------------------------------------
constexpr int kGS = 256 + 32 + 1;     // ghalf_slot(256) + 1
constexpr int kLA = 72;               // X1 row stride of the fused layout
constexpr size_t kFusedSmem = (size_t)(6 * kGS + 4 * kX2 + 4 * kX2 + kTwRows * kM) * sizeof(float2);

__global__ void __launch_bounds__(256, 3) fused_tp_kernel(const FusedArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* ghalf = reinterpret_cast<float2*>(smem_raw);   // [6][kGS]
  const int tid = threadIdx.x, l = tid >> 6, t = tid & 63;
  float2* x1 = ghalf + 6 * kGS + l * kX2;
  float2* x2 = ghalf + 6 * kGS + 4 * kX2 + l * kX2;
  float2* tw = ghalf + 6 * kGS + 8 * kX2;
  const int grp = a.g0 + blockIdx.x;
  const int k1 = grp / a.H2, k2 = grp % a.H2;
  const int nx = (k1 == 0 || 2 * k1 == a.P1) ? 1 : 2;
  const int ny = (k2 == 0 || 2 * k2 == a.P2) ? 1 : 2;
  const bool valid = l < nx * ny;                          // warp-uniform
  const int ix = valid ? l / ny : 0, iy = valid ? l % ny : 0;
  const int kx = ix ? a.P1 - k1 : k1, ky = iy ? a.P2 - k2 : k2;
  const long long line_off = ((long long)kx * a.P2 + ky) * a.n3;
  const int n3 = a.n3;
  fill_twiddles(tw, a.roots, tid, 256);
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && grp == 0 && tid == 0) {
    unsigned long long nb = 0;
    for (int b = 0; b < a.B; ++b) nb += (a.active == nullptr || a.active[b]) ? 1 : 0;
    atomicAdd(a.prof, nb * a.prof_rhs_bytes + a.prof_launch_bytes);
  }
  {
    // the group's half fibre: rebuilt for this matvec into the scratch, or the
    // octant k <= P/2 of the stored spectra (the rest is its mirror image)
    constexpr int H3 = kN / 2 + 1;
    const bool stored = a.spec != nullptr;
    const float2* src = stored ? a.spec + ((long long)k1 * a.P2 + k2) * kN
                               : a.octant + ((long long)(k1 - a.oct_k1a) * a.H2 + k2) * 6 * H3;
    const long long cs = stored ? a.spec_stride : H3;
    for (int it = tid; it < 6 * H3; it += 256) {
      const int cc = it / H3, kk = it - cc * H3;
      ghalf[cc * kGS + ghalf_slot(kk)] = src[cc * cs + kk];
    }
  }
  const float sx = ix ? -1.f : 1.f, sy = iy ? -1.f : 1.f;
  const int c = t >> 3, g = t & 7;
  __syncthreads();
  // a line's 64 threads (two warps) exchange values only among themselves: a named
  // barrier per line instead of the CTA's
  auto line_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + l) : "memory"); };
  for (int b = 0; b < a.B; ++b) {
    if (a.active != nullptr && a.active[b] == 0) continue;   // block-uniform
    float2 s[3][8];
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
      const float2* line = a.data + (long long)(b * 3 + comp) * a.comp_stride + line_off;
      float2 v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int p = t + kM * m;
        v[m] = (m < 4 && valid && p < n3) ? line[p] : make_float2(0.f, 0.f);
      }
      pass1t<false, true>(v, t, tw, x1, kLA);
      line_sync();
      {
        float2 u[8];
        pass2t_load<false>(u, t, x1, kLA, tw);
#pragma unroll
        for (int q = 0; q < 8; ++q) x2[c * 72 + 9 * q + (t & 7)] = u[q];
      }
      line_sync();
      pass3<false>(c, g, x2, s[comp]);
    }
    // Y = D G D J at f = c + 8 g + 64 h
#pragma unroll
    for (int h = 0; h < 8; ++h) {
      const int f = c + 8 * g + kM * h;
      float2 G[6];
      const bool zm = 2 * f > kN;
      const int fold = zm ? kN - f : f;
      const float sz = zm ? -1.f : 1.f;
      const float2* gp = ghalf + ghalf_slot(fold);
#pragma unroll
      for (int q = 0; q < 6; ++q) G[q] = gp[q * kGS];
      // D G D with the mirror signs folded into the off-diagonal entries
      const float sxy = sx * sy, sxz = sx * sz, syz = sy * sz;
      const float2 gxy = sxy * G[1], gxz = sxz * G[2], gyz = syz * G[4];
      const float2 jx = s[0][h], jy = s[1][h], jz = s[2][h];
      s[0][h] = cmadd(G[0], jx, cmadd(gxy, jy, gxz * jz));
      s[1][h] = cmadd(gxy, jx, cmadd(G[3], jy, gyz * jz));
      s[2][h] = cmadd(gxz, jx, cmadd(gyz, jy, G[5] * jz));
    }
    // inverse passes: the first writes X1 (in the X2 layout), which the forward
    // passes last read before the barrier that preceded pass 3, the second
    // reads X1 and writes X2 (layout of X1), the third reads X2
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
      float2* line = a.data + (long long)(b * 3 + comp) * a.comp_stride + line_off;
      ipass3t(t, s[comp], x1, tw);
      line_sync();
      ipass2t(t, x1, x2, kLA, tw);
      line_sync();
      float2 v[8];
      ipass1(t, x2, kLA, v);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int p = t + kM * m;
        if (valid && p < n3) line[p] = v[m];
      }
    }
    // the next right-hand side's pass 1 writes X1, last read by the inverse pass
    // 2 above before the barrier that preceded the inverse pass 1
  }
}

}  // namespace tp

// FP64 x / y stage of a length-512 line (columns contiguous in memory)
bool launch_line_tp64(LineArgs<double> a, cudaStream_t s) {
  if (a.plan.N != tp::kN || a.in_cs != 1 || a.out_cs != 1) return false;
  if ((a.flags & (PRO_CHI | EPI_CHI)) && a.chi_cs != 1) return false;
  if (a.nother > 65535 || a.nbatch > 65535) return false;
  const bool half = a.inverse ? (2 * a.lout == tp::kN) : (2 * a.lin == tp::kN);
  dim3 grid((a.ncol + tp::kCols64 - 1) / tp::kCols64, a.nother, a.nbatch);
  a.prof = nullptr;
  ProfScope ps(a.prof_family, s);
  if (a.inverse)
    launch_pdl(half ? tp::line_tp64_kernel<true, true> : tp::line_tp64_kernel<true, false>, grid,
               dim3(256), tp::kLine64Smem, s, a);
  else
    launch_pdl(half ? tp::line_tp64_kernel<false, true> : tp::line_tp64_kernel<false, false>, grid,
               dim3(256), tp::kLine64Smem, s, a);
  return true;
}

// fused z stage over the mirror groups [a.g0, a.g0 + groups) (P3 = 512, n3 <= 256)
bool fused_tp_supported(const FusedArgs<float>& a) {
  return a.P3 == tp::kN && 2 * a.n3 <= tp::kN && (a.spec != nullptr || a.octant != nullptr);
}

void launch_fused_tp(const FusedArgs<float>& a, int groups, cudaStream_t s) {
  launch_pdl(tp::fused_tp_kernel, dim3(groups), dim3(256), tp::kFusedSmem, s, a);
}

}  // namespace vie

int tp_init_attributes() {
  cudaError_t e = cudaSuccess;
  const int fs = (int)vie::tp::kFusedSmem;
  e = e != cudaSuccess ? e : cudaFuncSetAttribute(vie::tp::fused_tp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, fs);
  return e == cudaSuccess ? VIE_OK : cuda_status(e, "length-512 kernel attributes");
}

// ---------------------------------------------------------------------------
// Self-test of the bounded wait: one thread waits on a shared-memory mbarrier
// for at most `limit_ns`; with arrive = 1 the barrier's single arrival is
// made first (the wait completes), with arrive = 0 nothing arrives and the
// wait must give up.  status: 1 completed, 2 gave up.
// ---------------------------------------------------------------------------
namespace vie {
__global__ void bounded_wait_selftest_kernel(int arrive, unsigned long long limit_ns, int* status) {
  __shared__ __align__(8) uint64_t bar;
  mbar_init(&bar, 1);
  mbar_fence_init();
  if (arrive) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
  *status = mbar_wait_bounded(&bar, 0, limit_ns) ? 1 : 2;
}
}  // namespace vie

int grid_barrier_selftest(bool all_arrive, double seconds, cudaStream_t s);

extern "C" int vie_selftest_bounded_wait(int arrive, double seconds, void* stream) {
  clear_error();
  if (seconds <= 0.0 || seconds > 10.0 || arrive < 0 || arrive > 3) {
    set_error("wait limit %g s outside (0, 10] or unknown kind %d", seconds, arrive);
    return VIE_ERR_ARG;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (arrive >= 2) return grid_barrier_selftest(arrive == 3, seconds, s);
  int* d = nullptr;
  VIE_CUDA(cudaMalloc(&d, sizeof(int)));
  int h = 0;
  vie::bounded_wait_selftest_kernel<<<1, 1, 0, s>>>(arrive ? 1 : 0,
                                                      (unsigned long long)(seconds * 1e9), d);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(d);
  if (e != cudaSuccess) return cuda_status(e, "bounded-wait self-test");
  if (h == 2) {
    set_error("the bounded wait gave up after %g s", seconds);
    return VIE_ERR_TIMEOUT;
  }
  return h == 1 ? VIE_OK : VIE_ERR_CUDA;
}
