// Matvec stages of the edges in VIE_PLAN_SET_6 (plan_table.h), FP64.
#define VIE_SET 6
#define VIE_SET_T double
#define VIE_SET_SIZES VIE_PLAN_SET_6
#include "plan_set.cuh"
