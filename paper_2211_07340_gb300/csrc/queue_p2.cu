// int16 inputs, wide accumulation: the queue's sweep kernel, every strip height (1..16).
#include "sdtw_kernels.cuh"

HARU_SDTW_QUEUE_INSTANCE(2)
