// Dispatch of the planned matvec stages (planfft.cuh) over the sets of plan_table.h.
#include "plan_table.h"
#include "stages.cuh"

namespace vie {
namespace plan {

// defined in the sets' own translation units
template <typename T, int K> bool line_set(const LineArgs<T>& a, cudaStream_t s);
template <typename T, int K> bool fused_set(const FusedArgs<T>& a, int k10, int nk1, cudaStream_t s);
template <typename T, int K> cudaError_t prepare_set(int N);

#define VIE_SETS(X) X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9)
#define VIE_DECL_T(T, K)                                                              \
  template <> bool line_set<T, K>(const LineArgs<T>&, cudaStream_t);                  \
  template <> bool fused_set<T, K>(const FusedArgs<T>&, int, int, cudaStream_t);      \
  template <> cudaError_t prepare_set<T, K>(int);
#define VIE_DECL(K) VIE_DECL_T(float, K) VIE_DECL_T(double, K)
VIE_SETS(VIE_DECL)
#undef VIE_DECL
#undef VIE_DECL_T

static int set_of(int N) {
  switch (N) {
#define VIE_X0(N, ...) case N: return 0;
#define VIE_X1(N, ...) case N: return 1;
#define VIE_X2(N, ...) case N: return 2;
#define VIE_X3(N, ...) case N: return 3;
#define VIE_X4(N, ...) case N: return 4;
#define VIE_X5(N, ...) case N: return 5;
#define VIE_X6(N, ...) case N: return 6;
#define VIE_X7(N, ...) case N: return 7;
#define VIE_X8(N, ...) case N: return 8;
#define VIE_X9(N, ...) case N: return 9;
#define VIE_SIZES(K) VIE_PLAN_SET_##K(VIE_X##K)
    VIE_SETS(VIE_SIZES)
    default: return -1;
  }
}

}  // namespace plan

bool plan_exists(int N) { return plan::set_of(N) >= 0; }

// Line stage of a planned length: the matvec's half-length transforms (forward
// from N / 2 points, inverse cropped to N / 2) of adjacent columns.  Everything
// else is left to the general kernel.
template <typename T> bool launch_plan_line(const LineArgs<T>& a, cudaStream_t s) {
  const int N = a.plan.N;
  if (a.in_cs != 1 || a.out_cs != 1) return false;
  if ((a.flags & (PRO_CHI | EPI_CHI)) && a.chi_cs != 1) return false;
  if (a.inverse ? (a.lin != N || 2 * a.lout != N) : (2 * a.lin != N || a.lout != N)) return false;
  if (a.nother > 65535 || a.nbatch > 65535) return false;
  // 32-bit element offsets inside one batch entry
  const long long lim = 1LL << 31;
  if (a.in_bs >= lim || a.out_bs >= lim) return false;
  switch (plan::set_of(N)) {
#define VIE_CASE(K) \
  case K: return plan::line_set<T, K>(a, s);
    VIE_SETS(VIE_CASE)
#undef VIE_CASE
    default: return false;
  }
}

// Fused z stage of the groups k1 in [k10, k10 + nk1), every k2
template <typename T> bool launch_plan_fused(const FusedArgs<T>& a, int k10, int nk1, cudaStream_t s) {
  if (2 * a.n3 != a.P3 || nk1 > 65535) return false;
  switch (plan::set_of(a.P3)) {
#define VIE_CASE(K) \
  case K: return plan::fused_set<T, K>(a, k10, nk1, s);
    VIE_SETS(VIE_CASE)
#undef VIE_CASE
    default: return false;
  }
}

template bool launch_plan_line<float>(const LineArgs<float>&, cudaStream_t);
template bool launch_plan_line<double>(const LineArgs<double>&, cudaStream_t);
template bool launch_plan_fused<float>(const FusedArgs<float>&, int, int, cudaStream_t);
template bool launch_plan_fused<double>(const FusedArgs<double>&, int, int, cudaStream_t);

}  // namespace vie

// Shared-memory limits of the kernels for padded edge N (before any launch or
// graph capture)
int plan_prepare(int N) {
  cudaError_t e = cudaSuccess;
  switch (vie::plan::set_of(N)) {
#define VIE_CASE(K) \
  case K:                                                  \
    e = vie::plan::prepare_set<float, K>(N);               \
    if (e == cudaSuccess) e = vie::plan::prepare_set<double, K>(N); \
    break;
    VIE_SETS(VIE_CASE)
#undef VIE_CASE
    default: break;
  }
  return e == cudaSuccess ? VIE_OK : cuda_status(e, "planned kernel attributes");
}
