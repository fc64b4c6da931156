// One set of plan_table.h in one precision: the including file defines VIE_SET
// (the set's number), VIE_SET_SIZES (its list) and VIE_SET_T (float or double).
#include "plan_table.h"
#include "planfft64.cuh"

namespace vie {
namespace plan {

// FP64 lines of length 512 have a kernel of their own (tp512.cu: 256 x 100 x 100, 14.1
// ms a product, 14.2 ms with the planned x stages; 100 x 256 x 100 13.9 and 14.4 ms)
static constexpr bool has_line(int N) { return sizeof(VIE_SET_T) == 4 || N != 512; }

template <> bool line_set<VIE_SET_T, VIE_SET>(const LineArgs<VIE_SET_T>& a, cudaStream_t s) {
  switch (a.plan.N) {
#define VIE_X(N, Q1, Q2, R1, R2, R3)                           \
  case N:                                                      \
    if constexpr (has_line(N)) launch_plan_line<Q1, Q2>(a, s); \
    return has_line(N);
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
    if constexpr (has_line(N)) e = prepare_plan_line<Q1, Q2>(VIE_SET_T());             \
    return e != cudaSuccess ? e : prepare_plan_fused<R1, R2, R3>(VIE_SET_T());
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return e;
  }
}

}  // namespace plan
}  // namespace vie
