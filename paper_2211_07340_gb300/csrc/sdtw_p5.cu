// int16 groups with codes too large for the half-code cell: the scheduled sweep kernel, every strip height (1..16).
#include "sdtw_kernels.cuh"

HARU_SDTW_SWEEP_INSTANCE(5)
