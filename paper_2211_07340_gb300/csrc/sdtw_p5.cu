// int16 with both cells (half codes, and larger codes): the scheduled sweep kernel, every strip height (1..16).
#include "sdtw_kernels.cuh"

HARU_SDTW_SWEEP_INSTANCE(5)
