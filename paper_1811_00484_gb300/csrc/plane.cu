// The y and z stages of a small grid in one launch: one CTA per plane kx of the
// x-transformed currents (and right-hand side) takes the padded y transform, the
// padded z transform, the product with the plane's Green's entries, and both
// cropped inverse transforms, all in shared memory, T1 in place.
//
// A product on a small grid is bound by its launches: at 16^3 the five stages,
// the rebuild on its side stream and the four event calls between the streams
// take the host about 30 us, the kernels 3 to 5 us each.  With this kernel a
// product is three launches on one stream, and the rebuild of eq. (13), which
// reads only tables, is done by each CTA before it waits for the x stage.
//
// Passes as in planfft.cuh (n = a + Q2 b, k = c + Q1 h) and in place: a pass
// writes the addresses its thread has read.  The y transform leaves frequency
// c + Q1 h in row c Q2 + h, and the z lines of a row do not care; the inverse
// starts from that order.
#include <algorithm>

#include "plan_table.h"
#include "regdft.cuh"
#include "stages.cuh"

namespace vie {
namespace plane {

constexpr int kThreads = 256;
constexpr size_t kSmemMax = 200 * 1024;

template <typename T> struct PlaneArgs {
  cx<T>* data;                      // T1 [B][3][P1][n2][n3]
  const cx<T>* ry;                  // P2-th and P3-th roots
  const cx<T>* rz;
  int n2, n3, P1, P2, P3, H2, H3;
  int y1, y2, z1, z2;               // P2 = y1 y2, P3 = z1 z2, y1 and z1 even
  const CompMeta<T>* meta;
  int r2max, r3max;
  const cx<T>* spec;                // stored spectra (nullptr: rebuild)
  long long spec_stride;
  unsigned long long* prof;
  unsigned long long prof_rhs_bytes;
};

__host__ __device__ constexpr int odd(int v) { return v | 1; }

// shared entries: A [3][P2][n3], X [3][P2][z1 odd(z2)], G [6][H2][H3]
inline size_t plane_entries(int P2, int n3, int z1, int z2, int H2, int H3) {
  return (size_t)3 * P2 * n3 + (size_t)3 * P2 * z1 * odd(z2) + (size_t)6 * H2 * H3;
}

template <typename F> __device__ __forceinline__ void even_radix(int r, F&& f) {
  switch (r) {
    case 4: f(Int<4>()); break;
    case 6: f(Int<6>()); break;
    default: f(Int<8>()); break;
  }
}
template <typename F> __device__ __forceinline__ void any_radix(int r, F&& f) {
  switch (r) {
    case 3: f(Int<3>()); break;
    case 4: f(Int<4>()); break;
    case 5: f(Int<5>()); break;
    case 6: f(Int<6>()); break;
    default: f(Int<7>()); break;
  }
}
static bool radices_ok(int q1, int q2) {
  return (q1 == 4 || q1 == 6 || q1 == 8) && q2 >= 3 && q2 <= 7;
}

// resident CTAs per SM that the registers are held to (FP32: 80; without the limit
// 89 allowed two, and 14 x 20 x 16 with 16 right-hand sides took two waves)
constexpr int kPerSm = 3;

template <typename T>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? kPerSm : 1) plane_kernel(const PlaneArgs<T> a) {
  using C = cx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x;
  const int kx = blockIdx.x, b = blockIdx.y;
  const int n2 = a.n2, n3 = a.n3, P2 = a.P2, P3 = a.P3, H2 = a.H2, H3 = a.H3;
  const int y1 = a.y1, y2 = a.y2, z1 = a.z1, z2 = a.z2;
  const int LD = odd(z2), XP = z1 * LD;
  C* A = reinterpret_cast<C*>(smem_raw);           // [3][P2][n3]
  C* X = A + 3 * P2 * n3;                          // [3][P2][z1][LD]
  C* G = X + 3 * P2 * XP;                          // [6][H2][H3]
  const bool xm = 2 * kx > a.P1;
  const int k1 = xm ? a.P1 - kx : kx;
  if (a.spec != nullptr) {
    const C* src = a.spec + (long long)k1 * P2 * P3;
    for (int it = tid; it < 6 * H2 * H3; it += kThreads) {
      const int kk = it % H3, r = it / H3, k2 = r % H2, c = r / H2;
      G[it] = src[c * a.spec_stride + (long long)k2 * P3 + kk];
    }
  } else {
    // eq. (13): W_c[k2] = U2_c[k2, :] S_c[k1] (in A, not yet in use), G = W U3^T
    const int rm = a.r3max;
    for (int it = tid; it < 6 * H2 * rm; it += kThreads) {
      const int q = it % rm, r = it / rm, k2 = r % H2, c = r / H2;
      const CompMeta<T>& m = a.meta[c];
      C acc = czero<C>();
      if (q < m.r3) {
        const C* sl = m.slab + (long long)k1 * a.r2max * rm + q;
        const C* u2 = m.U2 + (long long)k2 * m.r2;
        for (int i = 0; i < m.r2; ++i) acc = cmadd(u2[i], sl[i * rm], acc);
      }
      A[it] = acc;
    }
    __syncthreads();
    for (int it = tid; it < 6 * H2 * H3; it += kThreads) {
      const int kk = it % H3, r = it / H3, c = r / H2;
      const int r3 = a.meta[c].r3;
      const C* u3 = a.meta[c].U3 + (long long)kk * r3;
      const C* w = A + r * rm;
      C acc = czero<C>();
      for (int q = 0; q < r3; ++q) acc = cmadd(w[q], u3[q], acc);
      G[it] = acc;
    }
    __syncthreads();
  }
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && kx == 0 && tid == 0) atomicAdd(a.prof, a.prof_rhs_bytes);
  const long long cs = (long long)a.P1 * n2 * n3;
  C* plane0 = a.data + (long long)b * 3 * cs + (long long)kx * n2 * n3;

  // y, pass 1: rows a + y2 m (m < y1 / 2), column z
  even_radix(y1, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < 3 * y2 * n3; it += kThreads) {
      const int z = it % n3, r = it / n3, t = r % y2, c = r / y2;
      const C* src = plane0 + c * cs + z;
      C x[Q / 2], v[Q];
#pragma unroll
      for (int m = 0; m < Q / 2; ++m) x[m] = src[(t + y2 * m) * n3];
      dft_half_in<Q, false>(x, v);
      C* dst = A + (c * P2 + t) * n3 + z;
      dst[0] = v[0];
#pragma unroll
      for (int k = 1; k < Q; ++k) dst[k * y2 * n3] = v[k] * __ldg(a.ry + t * k);
    }
  });
  __syncthreads();
  // y, pass 2
  any_radix(y2, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < 3 * y1 * n3; it += kThreads) {
      const int z = it % n3, r = it / n3;               // r = c y1 + slot
      C* p = A + r * Q * n3 + z;
      C u[Q];
#pragma unroll
      for (int f = 0; f < Q; ++f) u[f] = p[f * n3];
      dft_reg<Q, false>(u);
#pragma unroll
      for (int f = 0; f < Q; ++f) p[f * n3] = u[f];
    }
  });
  __syncthreads();
  // z, pass 1
  even_radix(z1, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < 3 * P2 * z2; it += kThreads) {
      const int t = it % z2, r = it / z2;               // r = c P2 + row
      const C* src = A + r * n3 + t;
      C x[Q / 2], v[Q];
#pragma unroll
      for (int m = 0; m < Q / 2; ++m) x[m] = src[z2 * m];
      dft_half_in<Q, false>(x, v);
      C* dst = X + r * XP + t;
      dst[0] = v[0];
#pragma unroll
      for (int k = 1; k < Q; ++k) dst[k * LD] = v[k] * __ldg(a.rz + t * k);
    }
  });
  __syncthreads();
  // z, pass 2, Y = D G D J at frequencies slot + z1 h, inverse pass 1
  const T sx = xm ? (T)-1 : (T)1;
  any_radix(z2, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < P2 * z1; it += kThreads) {
      const int slot = it % z1, row = it / z1;
      const int ky = row / y2 + y1 * (row % y2);
      const bool ym = 2 * ky > P2;
      const C* gk = G + (ym ? P2 - ky : ky) * H3;
      const T sy = ym ? (T)-1 : (T)1;
      C* own = X + row * XP + slot * LD;
      C s[3][Q];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
#pragma unroll
        for (int f = 0; f < Q; ++f) s[q][f] = own[q * P2 * XP + f];
        dft_reg<Q, false>(s[q]);
      }
#pragma unroll
      for (int h = 0; h < Q; ++h) {
        const int f = slot + z1 * h;
        const bool zm = 2 * f > P3;
        const C* gf = gk + (zm ? P3 - f : f);
        const T sz = zm ? (T)-1 : (T)1;
        const int gs = H2 * H3;
        const C gxx = gf[0], gyy = gf[3 * gs], gzz = gf[5 * gs];
        const C gxy = (sx * sy) * gf[gs], gxz = (sx * sz) * gf[2 * gs], gyz = (sy * sz) * gf[4 * gs];
        const C jx = s[0][h], jy = s[1][h], jz = s[2][h];
        s[0][h] = cmadd(gxx, jx, cmadd(gxy, jy, gxz * jz));
        s[1][h] = cmadd(gxy, jx, cmadd(gyy, jy, gyz * jz));
        s[2][h] = cmadd(gxz, jx, cmadd(gyz, jy, gzz * jz));
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        dft_reg<Q, true>(s[q]);
        own[q * P2 * XP] = s[q][0];
#pragma unroll
        for (int f = 1; f < Q; ++f) own[q * P2 * XP + f] = s[q][f] * conjg(__ldg(a.rz + slot * f));
      }
    }
  });
  __syncthreads();
  // z, inverse pass 2, cropped
  even_radix(z1, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < 3 * P2 * z2; it += kThreads) {
      const int t = it % z2, r = it / z2;
      const C* src = X + r * XP + t;
      C v[Q], y[Q / 2];
#pragma unroll
      for (int k = 0; k < Q; ++k) v[k] = src[k * LD];
      dft_half_out<Q, true>(v, y);
#pragma unroll
      for (int m = 0; m < Q / 2; ++m) A[r * n3 + t + z2 * m] = y[m];
    }
  });
  __syncthreads();
  // y, inverse pass 1
  any_radix(y2, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < 3 * y1 * n3; it += kThreads) {
      const int z = it % n3, r = it / n3, slot = r % y1;
      C* p = A + r * Q * n3 + z;
      C u[Q];
#pragma unroll
      for (int f = 0; f < Q; ++f) u[f] = p[f * n3];
      dft_reg<Q, true>(u);
      p[0] = u[0];
#pragma unroll
      for (int f = 1; f < Q; ++f) p[f * n3] = u[f] * conjg(__ldg(a.ry + slot * f));
    }
  });
  __syncthreads();
  // y, inverse pass 2, cropped
  even_radix(y1, [&](auto R) {
    constexpr int Q = decltype(R)::v;
    for (int it = tid; it < 3 * y2 * n3; it += kThreads) {
      const int z = it % n3, r = it / n3, t = r % y2, c = r / y2;
      const C* src = A + (c * P2 + t) * n3 + z;
      C v[Q], y[Q / 2];
#pragma unroll
      for (int k = 0; k < Q; ++k) v[k] = src[k * y2 * n3];
      dft_half_out<Q, true>(v, y);
      C* dst = plane0 + c * cs + z;
#pragma unroll
      for (int m = 0; m < Q / 2; ++m) dst[(t + y2 * m) * n3] = y[m];
    }
  });
}

// line radices of a planned edge this kernel has (padded edges 16 to 48, and 56)
static bool radices(int N, int* q1, int* q2) {
  switch (N) {
#define VIE_X(N, Q1, Q2, ...) \
  case N: *q1 = Q1; *q2 = Q2; return radices_ok(Q1, Q2);
    VIE_PLAN_SET_0(VIE_X) VIE_PLAN_SET_1(VIE_X) VIE_PLAN_SET_2(VIE_X) VIE_PLAN_SET_3(VIE_X)
    VIE_PLAN_SET_4(VIE_X) VIE_PLAN_SET_5(VIE_X) VIE_PLAN_SET_6(VIE_X) VIE_PLAN_SET_7(VIE_X)
    VIE_PLAN_SET_8(VIE_X) VIE_PLAN_SET_9(VIE_X)
#undef VIE_X
    default: return false;
  }
}

}  // namespace plane

// Small enough for the planes: y and z edges of 8 to 24 or 28 voxels with P2 P3 <= 48^2,
// no rebuild kernel chosen by flag, and few enough planes (each CTA rebuilds its
// plane's entries, so waves of CTAs repeat that).  Where three planes fit an SM two
// waves still win (against the separate stages: 16 x 10 x 16 with 16 right-hand sides
// 22 against 43 us, 16^3 35 against 44, 40 x 8 x 28 with 8 38 against 38); where two do,
// one (20^3 17 against 24 us with one or two right-hand sides, 26 against 26 with four;
// 8 x 28 x 20 22 against 25 with one to four, 35 against 48 with 16; but 20 x 28 x 20
// with four 34 against 28); where one does, half a wave (24^3 25 against 23 us, 12 x 24
// x 24 22 against 25; with stored spectra 14 against 19 and 15 against 20).
// FP64 arithmetic is so slow that few CTAs lose more than the launches cost: there
// only up to 9 x 9 (or 8 x 10) voxels (8^3: 24 us against 20 us, 8 right-hand sides 29 us against
// 42 us; 12^3: 45 us against 30 us).
template <typename T> bool plane_eligible(const vie_op* op, int B) {
  int q, z1, z2;
  if (op->flags & (VIE_REBUILD_SIMT | VIE_REBUILD_TCGEN05)) return false;
  if (!plane::radices(op->P[1], &q, &q) || !plane::radices(op->P[2], &z1, &z2)) return false;
  if (op->P[1] * op->P[2] > (sizeof(T) == 8 ? 18 * 18 : 48 * 48)) return false;
  // W [6][H2][r3max] lies in A and X during the rebuild
  const size_t all = plane::plane_entries(op->P[1], op->n[2], z1, z2, op->H[1], op->H[2]);
  if ((size_t)6 * op->H[1] * (op->rmax[2] + op->H[2]) > all) return false;
  const size_t smem = all * sizeof(cx<T>);
  if (smem > plane::kSmemMax) return false;
  const long long per_sm = std::min<long long>(sizeof(T) == 4 ? plane::kPerSm : 1, (227 * 1024) / (smem + 1024));
  const int planes = sizeof(T) == 8 ? device_sms()
                     : per_sm >= 3  ? 6 * device_sms()
                     : per_sm == 2  ? 2 * device_sms()
                                    : device_sms() / 2;
  return (long long)op->P[0] * B <= planes;
}

template <typename T>
void launch_plane(const vie_op* op, cx<T>* T1, int B, bool stored, cudaStream_t s) {
  plane::PlaneArgs<T> a = {};
  a.data = T1;
  if constexpr (sizeof(T) == 4) {
    a.ry = op->roots32[1];
    a.rz = op->roots32[2];
    a.spec = stored ? op->spec32 : nullptr;
    a.meta = reinterpret_cast<const CompMeta<T>*>(op->meta);
  } else {
    a.ry = op->roots64[1];
    a.rz = op->roots64[2];
    a.spec = stored ? op->spec64 : nullptr;
    a.meta = reinterpret_cast<const CompMeta<T>*>(static_cast<char*>(op->meta) + 6 * sizeof(CompMeta<float>));
  }
  a.n2 = op->n[1];
  a.n3 = op->n[2];
  a.P1 = op->P[0];
  a.P2 = op->P[1];
  a.P3 = op->P[2];
  a.H2 = op->H[1];
  a.H3 = op->H[2];
  plane::radices(a.P2, &a.y1, &a.y2);
  plane::radices(a.P3, &a.z1, &a.z2);
  a.r2max = op->rmax[1];
  a.r3max = op->rmax[2];
  a.spec_stride = (long long)a.P1 * a.P2 * a.P3;
  const int fam = sizeof(T) == 8 ? PF_MATVEC64 : (stored ? PF_FUSED_STORED : PF_FUSED_TUCKER);
  a.prof = sizeof(T) == 8 ? nullptr : prof_bytes(fam);
  a.prof_rhs_bytes = 12ull * a.P1 * a.P2 * a.n3 * sizeof(cx<T>);     // 48 B per padded voxel
  const size_t smem = plane::plane_entries(a.P2, a.n3, a.z1, a.z2, a.H2, a.H3) * sizeof(cx<T>);
  ProfScope ps(fam, s);
  launch_pdl(plane::plane_kernel<T>, dim3((unsigned)a.P1, (unsigned)B), dim3(plane::kThreads), smem, s, a);
}

template bool plane_eligible<float>(const vie_op*, int);
template bool plane_eligible<double>(const vie_op*, int);
template void launch_plane<float>(const vie_op*, float2*, int, bool, cudaStream_t);
template void launch_plane<double>(const vie_op*, double2*, int, bool, cudaStream_t);

}  // namespace vie

int plane_init_attributes() {
  cudaError_t e = cudaFuncSetAttribute(vie::plane::plane_kernel<float>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vie::plane::kSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(vie::plane::plane_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)vie::plane::kSmemMax);
  return e == cudaSuccess ? VIE_OK : cuda_status(e, "plane kernel attributes");
}
