// FP32 with start columns: the trace kernel, every strip height (1..16).
#include "sdtw_kernels.cuh"

HARU_SDTW_TRACE_INSTANCE(3)
