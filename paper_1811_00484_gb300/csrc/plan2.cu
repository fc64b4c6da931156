// Matvec stages of the edges in VIE_PLAN_SET_2 (plan_table.h), FP32.
#define VIE_SET 2
#define VIE_SET_T float
#define VIE_SET_SIZES VIE_PLAN_SET_2
#include "plan_set.cuh"
