// One set of plan_table.h: the including file defines VIE_SET (the set's number)
// and VIE_SET_SIZES (its list).
#include "plan_table.h"
#include "planfft.cuh"

#define VIE_CAT2(a, b) a##b
#define VIE_CAT(a, b) VIE_CAT2(a, b)

namespace vie {
namespace plan {

template <typename T> static bool set_line(const LineArgs<T>& a, cudaStream_t s) {
  switch (a.plan.N) {
#define VIE_X(N, Q1, Q2, R1, R2, R3) \
  case N: launch_plan_line<T, Q1, Q2>(a, s); return true;
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return false;
  }
}

template <typename T> static bool set_fused(const FusedArgs<T>& a, int k10, int nk1, cudaStream_t s) {
  switch (a.P3) {
#define VIE_X(N, Q1, Q2, R1, R2, R3) \
  case N: launch_plan_fused<T, R1, R2, R3>(a, k10, nk1, s); return true;
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return false;
  }
}

template <typename T> static bool set_prepare(int N, cudaError_t* e) {
  switch (N) {
#define VIE_X(N, Q1, Q2, R1, R2, R3)                                          \
  case N:                                                                     \
    *e = prepare_plan_line<T, Q1, Q2>();                                      \
    if (*e == cudaSuccess) *e = prepare_plan_fused<T, R1, R2, R3>();          \
    return true;
    VIE_SET_SIZES(VIE_X)
#undef VIE_X
    default: return false;
  }
}

bool VIE_CAT(line_set, VIE_SET)(const LineArgs<float>& a, cudaStream_t s) { return set_line<float>(a, s); }
bool VIE_CAT(fused_set, VIE_SET)(const FusedArgs<float>& a, int k10, int nk1, cudaStream_t s) {
  return set_fused<float>(a, k10, nk1, s);
}
bool VIE_CAT(prepare_set, VIE_SET)(int N, cudaError_t* e) { return set_prepare<float>(N, e); }

}  // namespace plan
}  // namespace vie
