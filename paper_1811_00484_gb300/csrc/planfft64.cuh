// The planned matvec stages (planfft.cuh: same passes, same addresses) in FP64.
//
// What bounds them is FP64 arithmetic alone (82 to 90 % of its pipe at 64^3): GB300
// retires 2 FP64 multiply-adds per clock and SM, a warp instruction occupies its
// quarter of the SM for 64 clocks, and shared memory, barriers and loads are free
// beside that.  So every pass is a flat loop over (line, butterfly) items by all
// threads of the CTA: warps are full except for one per pass, whatever the radices,
// and lines of mirror groups that do not exist are skipped.  With threads tied to a
// line as in FP32, a 36-thread group or five butterflies for eight threads left up to
// half of the issue slots to idle lanes: products of 20^3 143 -> 97 us, 36^3 with 8
// right-hand sides 2537 -> 1515 us, 64^3 1281 -> 1173 us (every kernel started early).
//
// For the same reason a kernel here does not let the next one start beside it (but
// see make_line_stages and matvec_run): the SMs that get most of the early CTAs decide
// when the next kernel ends.
#pragma once

#include "planfft.cuh"

namespace vie {
namespace plan {

constexpr int kThreads64 = 128;
constexpr int kCols64 = 16;

template <int R> constexpr int regs64() { return R <= 8 ? 80 : R <= 10 ? 104 : R <= 16 ? 128 : 255; }
template <int R> constexpr int blocks64() { return 65536 / (regs64<R>() * kThreads64); }

template <int Q1, int Q2, bool INV>
__global__ void __launch_bounds__(kThreads64, blocks64<imax(Q1, Q2)>())
    plan_line64_kernel(const LineArgs<double> a, int CW) {
  using C = double2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* X = reinterpret_cast<C*>(smem_raw);               // [Q1][Q2][CW]
  const int c00 = blockIdx.x * CW, o = blockIdx.y, bb = blockIdx.z;
  if (a.early) pdl_trigger();
  pdl_wait();
  if (a.active != nullptr && a.active[bb / a.batch_per_rhs] == 0) return;   // block-uniform
  const int cw = min(CW, a.ncol - c00);
  const double rs = (a.flags & (PRO_RSCALE | EPI_RSCALE))
                        ? a.rscale[(long long)(bb / a.batch_per_rhs) * a.rscale_stride]
                        : 1.0;
  const unsigned ils = (unsigned)a.in_ls, ols = (unsigned)a.out_ls, hls = (unsigned)a.chi_ls;
  const C* in = a.in + bb * a.in_bs + o * a.in_os + c00;
  const C* chi = a.chi + o * a.chi_os + c00;
  for (int it = threadIdx.x; it < Q2 * cw; it += kThreads64) {
    const int t = it / cw, col = it - t * cw;
    C v[Q1];
    if constexpr (!INV) {
      C x[Q1 / 2];
#pragma unroll
      for (int m = 0; m < Q1 / 2; ++m) x[m] = in[(t + Q2 * m) * ils + col];
      if (a.flags & (PRO_RSCALE | PRO_CONJ | PRO_CHI)) {
#pragma unroll
        for (int m = 0; m < Q1 / 2; ++m) {
          if (a.flags & PRO_RSCALE) x[m] = rs * x[m];
          if (a.flags & PRO_CONJ) x[m] = conjg(x[m]);
          if (a.flags & PRO_CHI) x[m] = chi[(t + Q2 * m) * hls + col] * x[m];
        }
      }
      dft_half_in<Q1, false>(x, v);
    } else {
#pragma unroll
      for (int m = 0; m < Q1; ++m) v[m] = in[(t + Q2 * m) * ils + col];
      dft_reg<Q1, true>(v);
    }
    X[t * cw + col] = v[0];
#pragma unroll
    for (int c = 1; c < Q1; ++c) {
      const C w = __ldg(a.roots + t * c);
      X[(c * Q2 + t) * cw + col] = v[c] * (INV ? conjg(w) : w);
    }
  }
  __syncthreads();
  const long long obase = bb * a.out_bs + o * a.out_os + c00;
  C* out = a.out + obase;
  for (int it = threadIdx.x; it < Q1 * cw; it += kThreads64) {
    const int t = it / cw, col = it - t * cw;
    C u[Q2];
#pragma unroll
    for (int f = 0; f < Q2; ++f) u[f] = X[(t * Q2 + f) * cw + col];
    if constexpr (!INV) {
      dft_reg<Q2, false>(u);
#pragma unroll
      for (int h = 0; h < Q2; ++h) out[(t + Q1 * h) * ols + col] = u[h];
    } else {
      C y[Q2 / 2];
      dft_half_out<Q2, true>(u, y);
      const C* add = a.addend + obase;
#pragma unroll
      for (int h = 0; h < Q2 / 2; ++h) {
        C x = a.scale * y[h];
        if (a.flags & EPI_CONJ) x = conjg(x);
        if (a.flags & (EPI_SUB | EPI_ADD)) {
          if (a.flags & EPI_CHI) x = chi[(t + Q1 * h) * hls + col] * x;
          C w = add[(t + Q1 * h) * ols + col];
          if (a.flags & EPI_RSCALE) w = rs * w;
          x = (a.flags & EPI_SUB) ? (w - x) : (w + x);
        }
        out[(t + Q1 * h) * ols + col] = x;
      }
    }
  }
}

// Q1 is even: forward Q1 x Q2, inverse Q2 x Q1
template <int Q1, int Q2> void launch_plan_line(LineArgs<double> a, cudaStream_t s) {
  if (a.in_os == a.ncol && a.out_os == a.ncol && (a.chi == nullptr || a.chi_os == a.ncol) &&
      (long long)a.ncol * a.nother < (1LL << 30)) {
    a.ncol *= a.nother;
    a.nother = 1;
  }
  const int tiles = (a.ncol + kCols64 - 1) / kCols64;
  const int cw = (a.ncol + tiles - 1) / tiles;
  a.prof = nullptr;
  ProfScope ps(a.prof_family, s);
  const dim3 grid((unsigned)tiles, (unsigned)a.nother, (unsigned)a.nbatch);
  const size_t smem = (size_t)Q1 * Q2 * cw * sizeof(double2);
  if (a.inverse) launch_pdl(plan_line64_kernel<Q2, Q1, true>, grid, dim3(kThreads64), smem, s, a, cw);
  else launch_pdl(plan_line64_kernel<Q1, Q2, false>, grid, dim3(kThreads64), smem, s, a, cw);
}

template <int Q1, int Q2> cudaError_t prepare_plan_line(double) {
  constexpr size_t smem = (size_t)Q1 * Q2 * kCols64 * sizeof(double2);
  if constexpr (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(plan_line64_kernel<Q1, Q2, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(plan_line64_kernel<Q2, Q1, true>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e;
  }
  return cudaSuccess;
}

// shared entries: half fibres [6][H3], lines [12][LS]; then W [6][r3max] (rebuilt)
template <int R1, int R2, int R3> constexpr int fused64_entries() {
  using P = FusedPlan<R1, R2, R3>;
  return 6 * P::H3 + 12 * P::LS;
}

template <int R1, int R2, int R3>
__global__ void __launch_bounds__(kThreads64, blocks64<imax(R1, imax(R2, R3))>())
    plan_fused64_kernel(const FusedArgs<double> a, int k10, int bchunk) {
  using C = double2;
  using P = FusedPlan<R1, R2, R3>;
  constexpr int N = P::N, H3 = P::H3, HL = P::HL, LD = P::LD, NL = P::NL, M1 = P::M1, LS = P::LS, TL = P::TL;
  constexpr bool kEven = R1 % 2 == 0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* G = reinterpret_cast<C*>(smem_raw);               // [6][H3]
  C* X = G + 6 * H3;                                   // [line][component][R1][LD]
  const int tid = threadIdx.x;
  const int k1 = k10 + blockIdx.y, k2 = blockIdx.x;
  const int nx = (k1 == 0 || 2 * k1 == a.P1) ? 1 : 2;
  const int ny = (k2 == 0 || 2 * k2 == a.P2) ? 1 : 2;
  const int nl = nx * ny;
  if (a.spec == nullptr) {
    // eq. (13) for this group, W_c = U2_c[k2, :] S_c[k1], G_c[k3] = W_c . U3_c[k3, :]
    C* W = X + 12 * LS;
    for (int it = tid; it < 6 * a.r3max; it += kThreads64) {
      const int c = it / a.r3max, q = it - c * a.r3max;
      const CompMeta<double>& m = a.meta[c];
      C acc = czero<C>();
      if (q < m.r3) {
        const C* sl = m.slab + (long long)k1 * a.r2max * a.r3max + q;
        const C* u2 = m.U2 + (long long)k2 * m.r2;
        for (int b = 0; b < m.r2; ++b) acc = cmadd(u2[b], sl[b * a.r3max], acc);
      }
      W[it] = acc;
    }
    __syncthreads();
    for (int it = tid; it < 6 * H3; it += kThreads64) {
      const int c = it / H3, kk = it - c * H3;
      const int r3 = a.meta[c].r3;
      const C* u3 = a.meta[c].U3 + (long long)kk * r3;
      C acc = czero<C>();
      for (int q = 0; q < r3; ++q) acc = cmadd(W[c * a.r3max + q], u3[q], acc);
      G[it] = acc;
    }
  } else {
    const C* src = a.spec + ((long long)k1 * a.P2 + k2) * N;
    for (int it = tid; it < 6 * H3; it += kThreads64) {
      const int c = it / H3, kk = it - c * H3;
      G[it] = src[c * a.spec_stride + kk];
    }
  }
  pdl_wait();
  // line lc = 3 l + component
  auto line = [&](int b, int lc) {
    const int l = lc / 3, q = lc - 3 * l;
    const int kx = l / ny ? a.P1 - k1 : k1, ky = l % ny ? a.P2 - k2 : k2;
    return a.data + (long long)(b * 3 + q) * a.comp_stride + ((long long)kx * a.P2 + ky) * (N / 2);
  };
  const int b1 = min(a.B, (int)(blockIdx.z + 1) * bchunk);
  for (int b = blockIdx.z * bchunk; b < b1; ++b) {
    if (a.active != nullptr && a.active[b] == 0) continue;   // block-uniform
    for (int it = tid; it < nl * 3 * M1; it += kThreads64) {
      const int lc = it / M1, t = it - lc * M1;
      const C* src = line(b, lc) + t;
      C v[R1];
      if constexpr (kEven) {
        C x[NL];
#pragma unroll
        for (int m = 0; m < NL; ++m) x[m] = src[M1 * m];
        dft_half_in<R1, false>(x, v);
      } else {
#pragma unroll
        for (int m = 0; m < R1; ++m) v[m] = (m < NL && t + M1 * m < N / 2) ? src[M1 * m] : czero<C>();
        dft_reg<R1, false>(v);
      }
      C* row = X + lc * LS + P::inner(t);
      row[0] = v[0];
#pragma unroll
      for (int c = 1; c < R1; ++c) row[c * LD] = v[c] * __ldg(a.roots + t * c);
    }
    __syncthreads();
    if constexpr (R3 > 1) {
      for (int it = tid; it < nl * 3 * R1 * R3; it += kThreads64) {
        const int lc = it / (R1 * R3), sl = it - lc * (R1 * R3), e = sl / R1;
        C* p = X + lc * LS + (sl % R1) * LD + e;
        C u[R2];
#pragma unroll
        for (int f = 0; f < R2; ++f) u[f] = p[f * P::PR];
        dft_reg<R2, false>(u);
        p[0] = u[0];
#pragma unroll
        for (int g = 1; g < R2; ++g) p[g * P::PR] = u[g] * __ldg(a.roots + R1 * e * g);
      }
      __syncthreads();
    }
    for (int it = tid; it < nl * 3 * TL; it += kThreads64) {
      const int lc = it / TL, sl = it - lc * TL;
      C* own = X + lc * LS + (sl % R1) * LD + (R3 > 1 ? (sl / R1) * P::PR : 0);
      C s[HL];
#pragma unroll
      for (int e = 0; e < HL; ++e) s[e] = own[e];
      dft_reg<HL, false>(s);
#pragma unroll
      for (int e = 0; e < HL; ++e) own[e] = s[e];
    }
    __syncthreads();
    // Y = D G D J at f = sl + TL h
    for (int it = tid; it < nl * N; it += kThreads64) {
      const int l = it / N, f = it - l * N, sl = f % TL, h = f / TL;
      C* p = X + 3 * l * LS + (sl % R1) * LD + (R3 > 1 ? (sl / R1) * P::PR : 0) + h;
      const bool xm = l / ny != 0, ym = l % ny != 0, zm = 2 * f > N;
      const C* gf = G + (zm ? N - f : f);
      const C gxx = gf[0], gyy = gf[3 * H3], gzz = gf[5 * H3];
      const double sxy = xm == ym ? 1.0 : -1.0, sxz = xm == zm ? 1.0 : -1.0, syz = ym == zm ? 1.0 : -1.0;
      const C gxy = sxy * gf[H3], gxz = sxz * gf[2 * H3], gyz = syz * gf[4 * H3];
      const C jx = p[0], jy = p[LS], jz = p[2 * LS];
      p[0] = cmadd(gxx, jx, cmadd(gxy, jy, gxz * jz));
      p[LS] = cmadd(gxy, jx, cmadd(gyy, jy, gyz * jz));
      p[2 * LS] = cmadd(gxz, jx, cmadd(gyz, jy, gzz * jz));
    }
    __syncthreads();
    for (int it = tid; it < nl * 3 * TL; it += kThreads64) {
      const int lc = it / TL, sl = it - lc * TL, c = sl % R1, g = sl / R1;
      C* own = X + lc * LS + c * LD + (R3 > 1 ? g * P::PR : 0);
      C s[HL];
#pragma unroll
      for (int e = 0; e < HL; ++e) s[e] = own[e];
      dft_reg<HL, true>(s);
      own[0] = s[0];
#pragma unroll
      for (int e = 1; e < HL; ++e) own[e] = s[e] * conjg(__ldg(a.roots + (R3 > 1 ? R1 * e * g : e * c)));
    }
    __syncthreads();
    if constexpr (R3 > 1) {
      for (int it = tid; it < nl * 3 * R1 * R3; it += kThreads64) {
        const int lc = it / (R1 * R3), sl = it - lc * (R1 * R3), c = sl % R1, e = sl / R1;
        C* p = X + lc * LS + c * LD + e;
        C u[R2];
#pragma unroll
        for (int g = 0; g < R2; ++g) u[g] = p[g * P::PR];
        dft_reg<R2, true>(u);
#pragma unroll
        for (int f = 0; f < R2; ++f) p[f * P::PR] = u[f] * conjg(__ldg(a.roots + (e + R3 * f) * c));
      }
      __syncthreads();
    }
    // the next right-hand side's first pass writes what the same thread reads here
    for (int it = tid; it < nl * 3 * M1; it += kThreads64) {
      const int lc = it / M1, t = it - lc * M1;
      const C* row = X + lc * LS + P::inner(t);
      C v[R1];
#pragma unroll
      for (int c = 0; c < R1; ++c) v[c] = row[c * LD];
      C* dst = line(b, lc) + t;
      if constexpr (kEven) {
        C y[R1 / 2];
        dft_half_out<R1, true>(v, y);
#pragma unroll
        for (int m = 0; m < R1 / 2; ++m) dst[M1 * m] = y[m];
      } else {
        dft_reg<R1, true>(v);
#pragma unroll
        for (int m = 0; m < NL; ++m)
          if (t + M1 * m < N / 2) dst[M1 * m] = v[m];
      }
    }
  }
}

// groups k1 in [k10, k10 + nk1), every k2; where the groups are fewer than four CTAs
// per SM the right-hand sides are shared out too (each share rebuilds the fibre)
template <int R1, int R2, int R3>
void launch_plan_fused(const FusedArgs<double>& a, int k10, int nk1, cudaStream_t s) {
  const int groups = a.H2 * nk1, shares = imin(a.B, (4 * device_sms() + groups - 1) / groups);
  const int bchunk = (a.B + shares - 1) / shares;
  const size_t smem = ((size_t)fused64_entries<R1, R2, R3>() + (a.spec == nullptr ? 6 * a.r3max : 0)) *
                      sizeof(double2);
  launch_pdl(plan_fused64_kernel<R1, R2, R3>,
             dim3((unsigned)a.H2, (unsigned)nk1, (unsigned)((a.B + bchunk - 1) / bchunk)), dim3(kThreads64), smem, s,
             a, k10, bchunk);
}

template <int R1, int R2, int R3> cudaError_t prepare_plan_fused(double) {
  return cudaFuncSetAttribute(plan_fused64_kernel<R1, R2, R3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kFusedSmemMax);
}

}  // namespace plan
}  // namespace vie
