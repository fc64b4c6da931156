// One set of plan_table.h in one precision: the including file defines VIE_SET
// (the set's number), VIE_SET_SIZES (its list) and VIE_SET_T (float or double).
#include "plan_table.h"
#include "planfft64.cuh"

namespace vie {
namespace plan {

template <> bool line_set<VIE_SET_T, VIE_SET>(const LineArgs<VIE_SET_T>& a, cudaStream_t s) {
  switch (a.plan.N) {
#define VIE_X(N, Q1, Q2, R1, R2, R3) \
  case N: launch_plan_line<Q1, Q2>(a, s); return true;
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return false;
  }
}

template <>
bool fused_set<VIE_SET_T, VIE_SET>(const FusedArgs<VIE_SET_T>& a, int k10, int nk1, cudaStream_t s) {
  switch (a.P3) {
#define VIE_X(N, Q1, Q2, R1, R2, R3) \
  case N: launch_plan_fused<R1, R2, R3>(a, k10, nk1, s); return true;
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return false;
  }
}

template <> cudaError_t prepare_set<VIE_SET_T, VIE_SET>(int N) {
  cudaError_t e = cudaSuccess;
  switch (N) {
#define VIE_X(N, Q1, Q2, R1, R2, R3)                                                   \
  case N:                                                                              \
    e = prepare_plan_line<Q1, Q2>(VIE_SET_T());                                        \
    return e != cudaSuccess ? e : prepare_plan_fused<R1, R2, R3>(VIE_SET_T());
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return e;
  }
}

}  // namespace plan
}  // namespace vie
