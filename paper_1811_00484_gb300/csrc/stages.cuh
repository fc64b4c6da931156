// Arguments of the matvec's stages, and the device bodies of the multi-grid
// kernels (multi.cu, edges N = 32 R): one x/y line tile, one fused z-line group;
// one slab-core block.
#pragma once

#include "warpfft.cuh"

namespace vie {

// sign of component c (xx, xy, xz, yy, yz, zz) under k_q -> P_q - k_q: the
// dyad (k0^2 delta_ab + d_a d_b) g is odd in coordinate q once per index equal to q
__device__ __forceinline__ int parity_sign(int c, int axis) {
  const int a = c < 3 ? 0 : (c < 5 ? 1 : 2);
  const int b = c == 0 ? 0 : (c == 1 || c == 3) ? 1 : 2;
  return (((a == axis) + (b == axis)) & 1) ? -1 : 1;
}

template <typename T> struct SlabArgs {
  const cx<T>* core[6];
  const cx<T>* U1[6];
  int r1[6], r2[6], r3[6];
  cx<T>* slab;
  long long slab_stride;
  int r2max, r3max;
  unsigned long long* prof;
  unsigned long long prof_launch_bytes;
};

template <typename T> struct FusedArgs {
  cx<T>* data;                 // [B*3][P1][P2][n3], transformed in place
  const cx<T>* roots;          // P3-th roots of unity
  FftPlan plan;
  int n3, P1, P2, P3, H1, H2, H3;
  int B;
  long long comp_stride;       // P1 * P2 * n3
  const CompMeta<T>* meta;     // [6] (Tucker)
  int r2max, r3max;
  const cx<T>* spec;           // [6][P1][P2][P3] (stored)
  long long spec_stride;       // P1 * P2 * P3
  const int* active;           // per RHS, nullptr = all
  const cx<T>* octant;         // rebuilt half fibres [k1 - oct_k1a][H2][6][H3] (nullptr: rebuild here)
  int oct_k1a;                 // first k1 held in `octant`
  int oct_chunk;               // k1 values per fill of `octant`
  bool oct_first_ready;        // host: chunk 0 already rebuilt on the side stream (joined)
  const vie_op* op;            // host: the operator (rebuild launches of later chunks)
  bool oct_cp;                 // host: rebuild from the Tucker+CP model (eq. (17))
  int g0;                      // group of the first CTA (k1 chunks)
  int lines_per_round;         // z-lines (x3 components) held in shared memory at once
  int ld;                      // shared-memory line stride
  unsigned long long* prof;    // profiler byte counter (nullptr = off)
  unsigned long long prof_rhs_bytes, prof_launch_bytes;
};

// S_c[k1] = core_c x1 U1_c[k1, :] for one (k1, c): the first stage of eq. (13)
template <typename T>
__device__ __forceinline__ void slab_core_block(const SlabArgs<T>& a, int k1, int c) {
  using C = cx<T>;
  const int r1 = a.r1[c], r2 = a.r2[c], r3 = a.r3[c];
  const C* core = a.core[c];
  const C* u1 = a.U1[c] + (long long)k1 * r1;
  C* S = a.slab + c * a.slab_stride + (long long)k1 * a.r2max * a.r3max;
  for (int it = threadIdx.x; it < r2 * r3; it += blockDim.x) {
    const int b = it / r3, g = it % r3;
    C acc = czero<C>();
    for (int al = 0; al < r1; ++al) acc = cmadd(u1[al], core[(al * r2 + b) * r3 + g], acc);
    S[b * a.r3max + g] = acc;
  }
}

// Tile slot of element (row p, column c): rows of 16 columns with the
// column index XOR-swizzled by (p ^ p>>4 ^ p>>6) mod 16.  Row-wise loads and
// stores stay conflict-free (a permutation within the row), and so do the
// warps' column accesses at natural rows lane + 32 j and at bit-reversed rows
// k1 + R brev5(lane) for every power-of-two R (at most 3-way otherwise).
__device__ __forceinline__ int tile_slot(int p, int c) {
  return p * 16 + (c ^ ((p ^ (p >> 4) ^ (p >> 6)) & 15));
}

constexpr int kLineTile = 16;      // columns per line tile

__host__ __device__ constexpr size_t line_warp_smem(int R) {
  return (size_t)(32 * R * kLineTile + 32 * R) * sizeof(float2);
}

// One tile of 16 contiguous columns of strided lines (an x or y stage), for
// batch index bb and outer index o.  The CTA stages the tile in shared
// memory (coalesced rows), each warp pulls whole columns into registers,
// transforms them with the lane FFT and writes them back; forward transforms
// (from N/2 loaded points) write the bit-reversed lane layout to natural rows,
// inverse transforms (cropped to N/2 stored points) read it from natural rows.
// Every thread of the block must call it.
template <int R>
__device__ __forceinline__ void line_warp_tile(const LineArgs<float>& a, int c0, int o, int bb,
                                               float2* smem) {
  using C = float2;
  constexpr int N = 32 * R;
  constexpr int TW = kLineTile;
  C* tile = smem;                  // element (row p, column c) at tile_slot(p, c)
  C* roots = smem + N * TW;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nth >> 5;
  // prologue (tables only), then the preceding kernel's results
  for (int m = tid; m < N; m += nth) roots[m] = a.roots[m];
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && c0 == 0 && o == 0 && tid == 0) atomicAdd(a.prof, a.prof_batch_bytes);
  const int ncols = min(TW, a.ncol - c0);
  const C* in = a.in + bb * a.in_bs + o * a.in_os + (long long)c0;
  for (int e = tid; e < a.lin * TW; e += nth) {
    const int c = e % TW, p = e / TW;
    if (c < ncols) tile[tile_slot(p, c)] = in[p * a.in_ls + c];
  }
  __syncthreads();

  const int br = brev5(lane);
  LaneConsts<C, float, R> lc;
  lc.init(lane, roots, N);
  for (int c = warp; c < ncols; c += nwarp) {
    C v[R];
    if (!a.inverse) {
#pragma unroll
      for (int j = 0; j < (R + 1) / 2; ++j) {
        const int p = lane + 32 * j;
        v[j] = p < a.lin ? tile[tile_slot(p, c)] : make_float2(0.f, 0.f);
      }
      warp_fft_fwd<C, float, R>(v, lc, roots, N);
#pragma unroll
      for (int k1 = 0; k1 < R; ++k1) {
        const int p = k1 + R * br;
        if (p < a.lout) tile[tile_slot(p, c)] = v[k1];
      }
    } else {
#pragma unroll
      for (int k1 = 0; k1 < R; ++k1) v[k1] = tile[tile_slot(k1 + R * br, c)];
      warp_fft_inv<C, float, R>(v, lane, lc, roots, N);
#pragma unroll
      for (int j = 0; j < (R + 1) / 2; ++j) {
        const int p = lane + 32 * j;
        if (p < a.lout) tile[tile_slot(p, c)] = v[j];
      }
    }
  }
  __syncthreads();

  C* out = a.out + bb * a.out_bs + o * a.out_os + (long long)c0;
  for (int e = tid; e < a.lout * TW; e += nth) {
    const int c = e % TW, p = e / TW;
    if (c < ncols) out[p * a.out_ls + c] = a.scale * tile[tile_slot(p, c)];
  }
}

// Columns per warp of the register-direct line stage: four c64 columns are one
// 32-byte sector of a row.
constexpr int kRegCols = 4;

// One group of kRegCols adjacent columns of strided lines (an x or y stage),
// transformed by one warp straight from and to global memory, no shared
// memory: lane l holds rows l + 32 j (natural order) of every column, or rows
// k1 + R brev5(l) (the lane FFT's bit-reversed order) on the frequency side.
// Each row access moves the group's 32 contiguous bytes, two 16-byte accesses
// when `vec` (the caller has checked that every row of the group starts on a
// 16-byte boundary), one 8-byte access per column otherwise.  Forward from N/2
// loaded points, inverse cropped to N/2 stored points.
template <int R>
__device__ __forceinline__ void line_reg_group(const LineArgs<float>& a, int c0, int o, int bb,
                                               bool vec, int lane) {
  using C = float2;
  constexpr int N = 32 * R;
  constexpr int NC = kRegCols;
  constexpr int NH = (R + 1) / 2;                // natural-order rows held per lane
  // prologue (tables only), then the preceding kernel's results
  LaneConsts<C, float, R> lc;
  lc.init(lane, a.roots, N);
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && c0 == 0 && o == 0 && lane == 0) atomicAdd(a.prof, a.prof_batch_bytes);
  const int ncols = min(NC, a.ncol - c0);
  const bool v4 = vec && ncols == NC;
  const int br = brev5(lane);
  C v[NC][R];
  const C* in = a.in + bb * a.in_bs + o * a.in_os + (long long)c0;
  C* out = a.out + bb * a.out_bs + o * a.out_os + (long long)c0;
  auto load_row = [&](int p, int j) {
    const C* src = in + (long long)p * a.in_ls;
    if (v4) {
      const float4 x0 = *reinterpret_cast<const float4*>(src);
      const float4 x1 = *reinterpret_cast<const float4*>(src + 2);
      v[0][j] = make_float2(x0.x, x0.y);
      v[1][j] = make_float2(x0.z, x0.w);
      v[2][j] = make_float2(x1.x, x1.y);
      v[3][j] = make_float2(x1.z, x1.w);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) v[c][j] = c < ncols ? src[c] : make_float2(0.f, 0.f);
    }
  };
  auto store_row = [&](int p, int j) {
    C* dst = out + (long long)p * a.out_ls;
    if (v4) {
      *reinterpret_cast<float4*>(dst) = make_float4(v[0][j].x, v[0][j].y, v[1][j].x, v[1][j].y);
      *reinterpret_cast<float4*>(dst + 2) = make_float4(v[2][j].x, v[2][j].y, v[3][j].x, v[3][j].y);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (c < ncols) dst[c] = v[c][j];
    }
  };
  if (!a.inverse) {
#pragma unroll
    for (int j = 0; j < NH; ++j) {
      const int p = lane + 32 * j;
      if (p < a.lin) {
        load_row(p, j);
      } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c][j] = make_float2(0.f, 0.f);
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) warp_fft_fwd<C, float, R>(v[c], lc, a.roots, N);
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) {
      const int p = k1 + R * br;
      if (p < a.lout) store_row(p, k1);
    }
  } else {
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) load_row(k1 + R * br, k1);
#pragma unroll
    for (int c = 0; c < NC; ++c) warp_fft_inv<C, float, R>(v[c], lane, lc, a.roots, N);
#pragma unroll
    for (int j = 0; j < NH; ++j) {
      const int p = lane + 32 * j;
      if (p < a.lout) {
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c][j] = a.scale * v[c][j];
        store_row(p, j);
      }
    }
  }
}

// Two-pass (four-step) variant for N = 8 V, V a multiple of 8: a warp owns
// kRegCols adjacent columns and eight lanes per column, lane = 4 j + c.
//   pass 1 (registers): lane (j, c) holds x[j + 8 m], m < V, of column c, takes
//          the length-V DFT over m and multiplies by w_N^{j k1};
//   exchange (shared memory, one write and one read per value);
//   pass 2 (registers): for k1 = j + 8 t, the length-8 DFT over j gives
//          X[k1 + V k2], k2 < 8.
// The inverse runs the same steps with conjugate roots (unscaled).  For a
// fixed register index the warp's 32 lanes touch 8 rows x 4 columns, i.e.
// whole 32-byte sectors.  No shuffles.  Forward from x[n < N/2] (m < V/2
// nonzero), inverse cropped to n < N/2 (k2 < 4).
// Exchange layout per warp: [c][j][k1], row stride V+1, column stride
// 8(V+1)+4 (both passes conflict-free within each half-warp).
__host__ __device__ constexpr int fs_col_stride(int V) { return 8 * (V + 1) + 4; }
__host__ __device__ constexpr size_t line_fs_smem(int V, int warps) {
  return (size_t)warps * kRegCols * fs_col_stride(V) * sizeof(float2);
}

template <int V>
__device__ __forceinline__ void line_fs_group(const LineArgs<float>& a, int c0, int o, int bb,
                                              int lane, float2* xs) {
  using C = float2;
  constexpr int N = 8 * V;
  constexpr int S = fs_col_stride(V);
  const int j = lane >> 2, c = lane & 3;
  C* xc = xs + c * S;
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && c0 == 0 && o == 0 && lane == 0) atomicAdd(a.prof, a.prof_batch_bytes);
  const bool col_ok = c0 + c < a.ncol;
  const C* in = a.in + bb * a.in_bs + o * a.in_os + (long long)(c0 + c);
  C* out = a.out + bb * a.out_bs + o * a.out_os + (long long)(c0 + c);
  const bool inv = a.inverse != 0;
  C v[V];
  // pass 1: rows j + 8 m
  constexpr int M1 = V / 2;                    // forward: rows loaded (the rest is padding)
#pragma unroll
  for (int m = 0; m < V; ++m) {
    const int p = j + 8 * m;
    C x = make_float2(0.f, 0.f);
    if ((inv || m < M1) && col_ok && p < a.lin) x = in[(long long)p * a.in_ls];
    v[m] = x;
  }
  if (!inv) {
#pragma unroll
    for (int m = M1; m < V; ++m) v[m] = make_float2(0.f, 0.f);   // zero padding, compile-time
  }
  reg_dft<C, float, V>(v, a.roots, N, inv);
#pragma unroll
  for (int k1 = 1; k1 < V; ++k1) {
    const C w = a.roots[j * k1];
    v[k1] = v[k1] * (inv ? conjg(w) : w);
  }
  // exchange: [c][j][k1]
#pragma unroll
  for (int k1 = 0; k1 < V; ++k1) xc[j * (V + 1) + k1] = v[k1];
  __syncwarp();
  // pass 2: k1 = j + 8 t, DFT over the eight j
#pragma unroll
  for (int t = 0; t < V / 8; ++t) {
    const int k1 = j + 8 * t;
    C u[8];
#pragma unroll
    for (int l = 0; l < 8; ++l) u[l] = xc[l * (V + 1) + k1];
    reg_dft<C, float, 8>(u, a.roots, N, inv);
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) {
      if (inv && k2 >= 4) continue;              // cropped to N/2
      const int p = k1 + V * k2;
      if (!col_ok || p >= a.lout) continue;
      out[(long long)p * a.out_ls] = inv ? a.scale * u[k2] : u[k2];
    }
  }
}

// Slot of z-frequency k in a row of the rebuilt half fibre: one padding slot
// every 8 entries, so the lanes' folded, bit-reversed frequencies (stride R)
// fall in different banks (at most 2-way for the radices used, 4-way at R=10).
__device__ __forceinline__ int ghalf_slot(int k) { return k + (k >> 3); }

__host__ __device__ constexpr size_t fused_warp_smem(int R, int H3, int r2max, int r3max) {
  (void)r2max;
  return (size_t)(32 * R + 6 * ((H3 - 1) + ((H3 - 1) >> 3) + 1) + 6 * r3max) * sizeof(float2);
}

// One (k1, k2) mirror group of the fused stage on the register path (P3 = 32 R):
// the four warps of the CTA take one mirror z-line each, hold the three
// components of every right-hand side in registers, and do the forward lane
// FFT, the voxel-wise product with the rebuilt components in the
// bit-reversed lane layout, and the inverse lane FFT.  The rebuild of the
// half fibre (k3 <= P3/2) is shared by the CTA.  Every thread must call it.
template <int R>
__device__ __forceinline__ void fused_warp_group(const FusedArgs<float>& a, int g, float2* smem) {
  using C = float2;
  constexpr int P3 = 32 * R;
  constexpr int NLOAD = (R + 1) / 2;               // points lane + 32 j < P3 / 2 + 16
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int n3 = a.n3, H3 = a.H3;
  const int k1 = g / a.H2, k2 = g % a.H2;
  const int nx = (k1 == 0 || 2 * k1 == a.P1) ? 1 : 2;
  const int ny = (k2 == 0 || 2 * k2 == a.P2) ? 1 : 2;
  const int nl = nx * ny;
  const bool has_line = warp < nl;                 // this warp's mirror line
  const int ix = has_line ? warp / ny : 0, iy = has_line ? warp % ny : 0;
  const int kx = ix ? a.P1 - k1 : k1, ky = iy ? a.P2 - k2 : k2;
  const long long line_off = ((long long)kx * a.P2 + ky) * n3;

  const int GS = ghalf_slot(H3 - 1) + 1;   // padded row length of the half fibre
  C* roots = smem;
  C* ghalf = roots + P3;               // [6][GS]
  C* wv = ghalf + 6 * GS;              // [6][r3max]
  // prologue: tables and factors only (no earlier kernel writes them)
  for (int m = tid; m < P3; m += nth) roots[m] = a.roots[m];
  const bool rebuild_here = a.octant == nullptr;
  if (rebuild_here) {
    for (int it = tid; it < 6 * a.r3max; it += nth) {
      const int c = it / a.r3max, gm = it % a.r3max;
      const CompMeta<float> m = a.meta[c];
      C acc = make_float2(0.f, 0.f);
      if (gm < m.r3) {
        const C* S = m.slab + (long long)k1 * a.r2max * a.r3max;
        const C* u2 = m.U2 + (long long)k2 * m.r2;
        for (int b = 0; b < m.r2; ++b) acc = cmadd(u2[b], S[b * a.r3max + gm], acc);
      }
      wv[it] = acc;
    }
    __syncthreads();
    for (int it = tid; it < 6 * H3; it += nth) {
      const int c = it / H3, kk = it % H3;
      const CompMeta<float>& m = a.meta[c];
      const C* u3t = m.U3t + kk;              // U3_c[kk, q] at u3t[q * H3]: coalesced
      const C* w = wv + c * a.r3max;
      C acc = make_float2(0.f, 0.f);
#pragma unroll 4
      for (int q = 0; q < m.r3; ++q) acc = cmadd(w[q], u3t[(long long)q * H3], acc);
      ghalf[c * GS + ghalf_slot(kk)] = acc;
    }
  }
  pdl_trigger();
  pdl_wait();

  if (a.prof != nullptr && g == 0 && tid == 0) atomicAdd(a.prof, a.B * a.prof_rhs_bytes + a.prof_launch_bytes);
  // the first right-hand side's lines are loaded before the half fibres are copied,
  // so the two latencies overlap
  C v[3][R];
  auto load_lines = [&](int b) {
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
      const C* src = a.data + (long long)(b * 3 + comp) * a.comp_stride + line_off;
#pragma unroll
      for (int j = 0; j < NLOAD; ++j) {
        const int p = lane + 32 * j;
        v[comp][j] = p < n3 ? src[p] : make_float2(0.f, 0.f);
      }
    }
  };
  if (has_line) load_lines(0);
  if (!rebuild_here) {
    // the group's half fibres, rebuilt for this matvec into the scratch
    const C* src = a.octant + ((long long)(k1 - a.oct_k1a) * a.H2 + k2) * 6 * H3;
    for (int it = tid; it < 6 * H3; it += nth) {
      const int c = it / H3, kk = it - c * H3;
      ghalf[c * GS + ghalf_slot(kk)] = src[it];
    }
  }
  __syncthreads();
  if (!has_line) return;                   // no block barrier follows

  const int br = brev5(lane);
  LaneConsts<C, float, R> lc;
  lc.init(lane, roots, P3);
  // mirror signs: the component (a, b) of the spectrum at the mirror point is
  // s_a s_b times its half-fibre value, s_q = -1 along each mirrored axis, so
  // Y = D G D J with D = diag(s_x, s_y, s_z)
  const float sx = ix ? -1.f : 1.f, sy = iy ? -1.f : 1.f;
  for (int b = 0; b < a.B; ++b) {
    if (b != 0) load_lines(b);
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) warp_fft_fwd<C, float, R>(v[comp], lc, roots, P3);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int kk = q + R * br;                       // z-frequency held in register q
      C gc[6];
      C jx = v[0][q], jy = v[1][q], jz = v[2][q];
      const bool zm = 2 * kk > P3;
      const int fold = zm ? P3 - kk : kk;
      const float sz = zm ? -1.f : 1.f;
      const C* gp = ghalf + ghalf_slot(fold);
#pragma unroll
      for (int c = 0; c < 6; ++c) gc[c] = gp[c * GS];
      jx = sx * jx;
      jy = sy * jy;
      jz = sz * jz;
      // Y_a = sum_b G_ab J_b with G symmetric: xx xy xz / xy yy yz / xz yz zz
      const C yx = gc[0] * jx + gc[1] * jy + gc[2] * jz;
      const C yy = gc[1] * jx + gc[3] * jy + gc[4] * jz;
      const C yz = gc[2] * jx + gc[4] * jy + gc[5] * jz;
      v[0][q] = sx * yx;
      v[1][q] = sy * yy;
      v[2][q] = sz * yz;
    }
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
      warp_fft_inv<C, float, R>(v[comp], lane, lc, roots, P3);
      C* dst = a.data + (long long)(b * 3 + comp) * a.comp_stride + line_off;
#pragma unroll
      for (int j = 0; j < NLOAD; ++j) {
        const int p = lane + 32 * j;
        if (p < n3) dst[p] = v[comp][j];
      }
    }
  }
}

// Fused z stage with the four-step transform (P3 = 8 V): one CTA of three warps
// per (k1, k2) mirror group, warp = Cartesian component of J and Y, lane =
// 4 j + l with l the mirror line (up to four) and j the eighth of the line.
//   forward: pass 1 / exchange / pass 2 as in line_fs_group, then the
//            component's spectrum goes to a shared buffer spec[comp][l][f];
//   product: each lane forms Y_comp[l][f] = s_comp sum_b G_comp,b[fold f] s_b J_b[l][f]
//            (D G D, with G the rebuilt half fibre) for the frequencies f = j + 8 m
//            its inverse pass 1 needs;
//   inverse: pass 1 / exchange / pass 2 cropped to n3 outputs, written in place.
// Every thread must call it.
__host__ __device__ constexpr int fused_fs_spec_stride(int V) { return 8 * V + 4; }
__host__ __device__ constexpr size_t fused_fs_smem(int V, int H3) {
  return (size_t)(6 * ((H3 - 1) + ((H3 - 1) >> 3) + 1) + 3 * 4 * fused_fs_spec_stride(V) +
                  3 * kRegCols * fs_col_stride(V)) *
         sizeof(float2);
}

template <int V>
__device__ __forceinline__ void fused_fs_group(const FusedArgs<float>& a, int g, float2* smem) {
  using C = float2;
  constexpr int N = 8 * V;                     // P3
  constexpr int XS = fs_col_stride(V);
  constexpr int SS = fused_fs_spec_stride(V);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int lane = tid & 31, comp = tid >> 5;  // three warps (a fourth, if any, only helps copy)
  const bool act = comp < 3;
  const int j = lane >> 2, ln = lane & 3;
  const int n3 = a.n3, H3 = a.H3;
  const int k1 = g / a.H2, k2 = g % a.H2;
  const int nx = (k1 == 0 || 2 * k1 == a.P1) ? 1 : 2;
  const int ny = (k2 == 0 || 2 * k2 == a.P2) ? 1 : 2;
  const bool valid = ln < nx * ny;
  const int ix = valid ? ln / ny : 0, iy = valid ? ln % ny : 0;
  const int kx = ix ? a.P1 - k1 : k1, ky = iy ? a.P2 - k2 : k2;
  const long long line_off = ((long long)kx * a.P2 + ky) * n3;
  const int GS = ghalf_slot(H3 - 1) + 1;
  C* ghalf = smem;                              // [6][GS]
  C* spec = ghalf + 6 * GS;                     // [3][4][SS]
  C* xw = spec + 3 * 4 * SS + (act ? comp : 0) * kRegCols * XS;   // this warp's exchange buffer
  C* xc = xw + ln * XS;
  pdl_trigger();
  pdl_wait();
  if (a.prof != nullptr && g == 0 && tid == 0) atomicAdd(a.prof, a.B * a.prof_rhs_bytes + a.prof_launch_bytes);
  {
    // the group's half fibres, rebuilt for this matvec into the scratch
    const C* src = a.octant + ((long long)(k1 - a.oct_k1a) * a.H2 + k2) * 6 * H3;
    for (int it = tid; it < 6 * H3; it += nth) {
      const int c = it / H3, kk = it - c * H3;
      ghalf[c * GS + ghalf_slot(kk)] = src[it];
    }
  }
  // rows of G used by this warp's component: x: xx xy xz, y: xy yy yz, z: xz yz zz
  const int g0 = comp == 0 ? 0 : (comp == 1 ? 1 : 2);
  const int g1 = comp == 0 ? 1 : (comp == 1 ? 3 : 4);
  const int g2 = comp == 0 ? 2 : (comp == 1 ? 4 : 5);
  const float sx = ix ? -1.f : 1.f, sy = iy ? -1.f : 1.f;
  const float sc = comp == 0 ? sx : (comp == 1 ? sy : 1.f);
  __syncthreads();
  for (int b = 0; b < a.B; ++b) {
    C* line = a.data + (long long)(b * 3 + (act ? comp : 0)) * a.comp_stride + line_off;
    C v[V];
    if (act) {
      // forward pass 1: x[j + 8 m], m < V/2 (the rest is zero padding)
#pragma unroll
      for (int m = 0; m < V; ++m) {
        const int p = j + 8 * m;
        v[m] = (m < V / 2 && valid && p < n3) ? line[p] : make_float2(0.f, 0.f);
      }
      reg_dft<C, float, V>(v, a.roots, N, false);
#pragma unroll
      for (int q = 1; q < V; ++q) v[q] = v[q] * a.roots[j * q];
#pragma unroll
      for (int q = 0; q < V; ++q) xc[j * (V + 1) + q] = v[q];
      __syncwarp();
      // forward pass 2 -> spec[comp][ln][q + V k2]
      C* sp = spec + (comp * 4 + ln) * SS;
#pragma unroll
      for (int t = 0; t < V / 8; ++t) {
        const int q = j + 8 * t;
        C u[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) u[l] = xc[l * (V + 1) + q];
        reg_dft<C, float, 8>(u, a.roots, N, false);
#pragma unroll
        for (int k = 0; k < 8; ++k) sp[q + V * k] = u[k];
      }
    }
    __syncthreads();
    if (act) {
      // product at f = j + 8 m, straight into the inverse pass 1 registers
      const C* s0 = spec + (0 * 4 + ln) * SS;
      const C* s1 = spec + (1 * 4 + ln) * SS;
      const C* s2 = spec + (2 * 4 + ln) * SS;
#pragma unroll
      for (int m = 0; m < V; ++m) {
        const int f = j + 8 * m;
        const bool zm = 2 * f > N;
        const int fold = zm ? N - f : f;
        const float sz = zm ? -1.f : 1.f;
        const C* gp = ghalf + ghalf_slot(fold);
        const C G0 = gp[g0 * GS], G1 = gp[g1 * GS], G2 = gp[g2 * GS];
        C y = G0 * (sx * s0[f]) + G1 * (sy * s1[f]) + G2 * (sz * s2[f]);
        y = (comp == 2 ? sz : sc) * y;
        v[m] = y;
      }
      // inverse pass 1 (exchange buffer free: pass 2 read it before the barrier)
      reg_dft<C, float, V>(v, a.roots, N, true);
#pragma unroll
      for (int q = 1; q < V; ++q) v[q] = v[q] * conjg(a.roots[j * q]);
#pragma unroll
      for (int q = 0; q < V; ++q) xc[j * (V + 1) + q] = v[q];
      __syncwarp();
      // inverse pass 2, cropped: n = q + V k2 < N / 2
#pragma unroll
      for (int t = 0; t < V / 8; ++t) {
        const int q = j + 8 * t;
        C u[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) u[l] = xc[l * (V + 1) + q];
        reg_dft<C, float, 8>(u, a.roots, N, true);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int n = q + V * k;
          if (valid && n < n3) line[n] = u[k];
        }
      }
    }
    __syncthreads();                           // spec and xw reused by the next right-hand side
  }
}

// Length-512 kernels (tp512.cu): FP64 x / y line stages and the fused z stage
bool launch_line_tp64(LineArgs<double> a, cudaStream_t s);
bool fused_tp_supported(const FusedArgs<float>& a);
void launch_fused_tp(const FusedArgs<float>& a, int groups, cudaStream_t s);
// every edge with a factor plan (plan.cu): false when the launch is not one of theirs
bool plan_exists(int N);
template <typename T> bool launch_plan_line(const LineArgs<T>& a, cudaStream_t s);
// y and z stages of a small grid's planes in one launch, T1 in place (plane.cu)
template <typename T> bool plane_eligible(const vie_op* op, int B);
template <typename T>
void launch_plane(const vie_op* op, cx<T>* T1, int B, bool stored, cudaStream_t s);
template <typename T> bool launch_plan_fused(const FusedArgs<T>& a, int k10, int nk1, cudaStream_t s);

}  // namespace vie
