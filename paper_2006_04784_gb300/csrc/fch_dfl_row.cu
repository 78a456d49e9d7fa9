// Double-float (FP32 pair) row passes (FCH_FP32X2).
#define FCH_T fch::df
#define FCH_SUFFIX dfl
#define FCH_NO_COL
#include "fch_launch.cuh"
