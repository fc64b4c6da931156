// Matvec stages of the edges in VIE_PLAN_SET_9 (plan_table.h), FP64.
#define VIE_SET 9
#define VIE_SET_T double
#define VIE_SET_SIZES VIE_PLAN_SET_9
#include "plan_set.cuh"
